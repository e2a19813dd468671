// FP32 gravity walk kernels for isolated BCs (see ts_walk.cu, and ts_walk_split.cuh for meshes of few cells).
#include "ts_walk_kernels.cuh"
#include "ts_walk_split.cuh"

cudaError_t walk_launch_f32_iso(ts_ctx* c, const WalkParams& P, int mac, bool rel, int T) {
    // The choice depends on the mesh alone, so that walks of parts of it (ranges, block updates) run the
    // kernel of the whole walk and give its bits.  The grids of a batch keep the paired walk: side by side
    // they fill the chip, where it needs fewer instructions (16 grids of 32^3 on 8 streams: 576 us a run, 879 us
    // with the split walk; 64 of 16^3 684 and 490 us), and the batch's two forms then give the same bits.
    if (T == 1 && !P.batched && mac != TS_MAC_MPE && (int64_t)c->nleaf * 16 <= SPLIT_MAX_WARPS) {
        if (mac == TS_MAC_BH) return launch_split<TS_MAC_BH, false>(c, P);
        return rel ? launch_split<TS_MAC_APE, true>(c, P) : launch_split<TS_MAC_APE, false>(c, P);
    }
    return dispatch_bck<float, 0>(c, P, mac, rel, T);
}
