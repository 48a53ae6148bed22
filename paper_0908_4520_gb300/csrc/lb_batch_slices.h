// The groups of the batch kernel and their slices of a CTA's dynamic shared memory (plain
// arithmetic, for the kernel and for a host compiler).
#pragma once

#ifdef __CUDACC__
#define LB_SLICE_FN __host__ __device__ __forceinline__
#else
#define LB_SLICE_FN inline
#endif

namespace lbk {

// The work queues, by the width of the group of warps that advances an instance.
enum BatchKind : int { kBatchCluster = 0, kBatchCta = 1, kBatchQuad = 2, kBatchWarp = 3, kBatchQueues = 4 };

struct BatchSlice {
    int offset, bytes;
};

// warps of a group of that kind in a CTA of nwarp
LB_SLICE_FN int batch_group_warps(int kind, int nwarp) { return kind <= kBatchCta ? nwarp : (kind == kBatchQuad ? 4 : 1); }

// The slice of the group whose first warp is `first`, 16-byte aligned.  A four-warp group that finds
// its queue empty parts into single warps while its neighbours still step theirs, so the slices of
// these two widths must not overlap across groups: one warp's slice is rounded down once, and a
// four-warp group has those of its own four warps.  (Each width's slice rounded by itself put warp 12
// up to 144 bytes inside the third four-warp group's.)  The group of the whole CTA has the whole
// budget: every warp has left it before the first narrower group forms.
LB_SLICE_FN BatchSlice batch_slice(int kind, int first, int smem_cap, int nwarp) {
    if (kind <= kBatchCta) return {0, smem_cap & ~15};
    const int warp = smem_cap / nwarp & ~15;
    return {first * warp, batch_group_warps(kind, nwarp) * warp};
}

}  // namespace lbk

#undef LB_SLICE_FN
