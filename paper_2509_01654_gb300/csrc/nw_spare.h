// nw_spare.h -- device blocks that finished calls gave back, kept for the next
// calls.
//
// cudaMalloc and cudaFree map and unmap pages and wait for the device: 3.3 GB of
// candidate buffers cost 2.7 ms of an 8.1 ms call for 100,000 rows, and sixteen small
// buffers 200 us of a 290 us query.  A call that has synchronised its stream
// therefore gives its buffers here, and the next allocations take them, of any context
// and on any stream; a context with a memory budget takes its own only, which count
// against it.  The list is bounded for a device as a whole (two contexts that call in
// turn use the same blocks).  It is released when an allocation fails for want of
// device memory, before that is refused; by nw_trim; and with the device's last
// context (a program that makes a context for each piece of work keeps the blocks:
// the first candidate lists of 100,003 rows 5.4 ms, 6.7 where the context before had
// freed them).
#pragma once

#include <stddef.h>

namespace nw {

constexpr size_t kSpareBytes = (size_t)4 << 30;  // of a device, over all contexts
constexpr size_t kSpareBlocks = 64;              // of a context

// the smallest block of the device (with an owner: of its own) of `bytes` to `most`
// bytes; its size in *have
void* spare_take(const void* owner, int device, size_t bytes, size_t most, size_t* have);
// keeps a block that no work in flight uses; older blocks of the device make room
void spare_give(const void* owner, int device, void* p, size_t bytes);
size_t spare_held(const void* owner);
// frees the oldest of the owner's blocks, or all of a device: false if there is none
bool spare_drop_oldest(const void* owner);
bool spare_drop_device(int device);
// a context of the device comes, and goes: its blocks stay for the others
void spare_open(int device);
void spare_close(const void* owner, int device);

}  // namespace nw
