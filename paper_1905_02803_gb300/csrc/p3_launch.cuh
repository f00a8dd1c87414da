// Overlap of a stage's launch with the end of the stage before it
// (programmatic dependent launch): the next stage's launch latency, prologue
// and first instruction fetches run while the last blocks of this one store
// their results.  Measured, forward + inverse: 64^3 FP32 34.8 -> 26.6 us, 32^3
// FP64 45.2 -> 30.8 us, 256^3 FP32 171 -> 156 us, 24 mixed grids over 16 streams
// 2.08 -> 1.91 ms, 384^3 731 -> 720 us.  Letting the next blocks in from the
// start of a stage instead parks them on SMs that other streams' stages, or the
// stage's own last blocks, could use (128^3: 44 us against 38).
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
// From here on (each block's outputs are computed) the next stage's blocks may
// take free slots of the SMs, where they wait in stage_begin().
__device__ __forceinline__ void stage_ending()
{
#if P3_PDL
    asm volatile("griddepcontrol.launch_dependents;");
#endif
}

}  // namespace p3
