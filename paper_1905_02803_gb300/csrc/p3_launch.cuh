// Overlap of a stage's launch with the end of the stage before it
// (programmatic dependent launch): the next stage's launch latency, prologue
// and first instruction fetches run while the last blocks of this one leave
// and their writes become visible.  Forward + inverse without and with it, on
// a stream: 64^3 FP32 37.0 -> 22.1 us, 32^3 FP64 48.2 -> 30.3, 256^3 FP32 169.2
// -> 152.5, 384^3 701 -> 680; in a replayed graph, whose launches are cheaper,
// 24.5 -> 21.8, 31.8 -> 30.5, 155.5 -> 151.8, 685 -> 679 us.
//
// No stage lets the next one in before its blocks leave
// (griddepcontrol.launch_dependents): the blocks let in early go to the SMs
// with room, not evenly, and then run there one after another, while other
// SMs idle.  Measured with that call before each stage's stores: 64 x 64 x 256
// FP32 24.5 -> 38.1 us, 64 x 64 x 512 34.2 -> 48.7, 112^3 FP64 XYZ 89 -> 102,
// 1024 x 1024 x 3 XYZ 78 -> 95; it gained 1 to 3 us on cubes of 40, 80 and 135
// points (41.4 -> 39.1 us), and over 444 calls it lost 5 % in FP32, 3 % in FP64.
#pragma once

namespace p3 {

// Before a stage kernel's first access to memory another kernel may write or
// read: waits until every kernel before it in the stream has finished and its
// writes are visible.
__device__ __forceinline__ void stage_begin()
{
#if P3_PDL
    asm volatile("griddepcontrol.wait;" ::: "memory");
#endif
}

}  // namespace p3
