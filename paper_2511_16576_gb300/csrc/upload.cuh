// upload.cuh -- which uploads read the caller's vertices in place (api.cu): host code only.
#pragma once

#include <stdint.h>

constexpr int kPointerOnDevice = 2;  // cudaMemoryTypeDevice

// A device upload's preparation kernel loads the caller's vertices itself, and copies them on
// the way, if they are plain memory of the context's own GPU (`memory_type` and
// `pointer_device` as cudaPointerGetAttributes reports them) at an int2's alignment.  Any other
// address that a copy accepts -- another GPU's, pinned or managed memory -- is copied first: a kernel
// may not be able to load from it.
inline bool pmh_reads_in_place(int memory_type, int pointer_device, int device, uintptr_t address)
{
    return memory_type == kPointerOnDevice && pointer_device == device && address % 8 == 0;
}
