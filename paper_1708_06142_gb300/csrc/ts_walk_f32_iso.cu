// FP32 gravity walk kernels for isolated BCs (see ts_walk.cu, and ts_walk_split.cuh for meshes of few cells).
#include "ts_walk_kernels.cuh"
#include "ts_walk_split.cuh"

cudaError_t walk_launch_f32_iso(ts_ctx* c, const WalkParams& P, int mac, bool rel, int T) {
    // The choice depends on the mesh alone, so that walks of parts of it (ranges, block updates) run the
    // kernel of the whole walk and give its bits.
    if (T == 1 && mac != TS_MAC_MPE && (int64_t)c->nleaf * 16 <= SPLIT_MAX_WARPS) {
        if (mac == TS_MAC_BH) return launch_split<TS_MAC_BH, false>(c, P);
        return rel ? launch_split<TS_MAC_APE, true>(c, P) : launch_split<TS_MAC_APE, false>(c, P);
    }
    return dispatch_bck<float, 0>(c, P, mac, rel, T);
}
