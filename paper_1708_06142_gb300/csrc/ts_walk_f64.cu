// FP64 gravity walk kernels (see ts_walk.cu, and ts_walk64.cuh for the isolated walk with one target per
// lane).
#include "ts_walk64.cuh"
#include "ts_walk_kernels.cuh"

cudaError_t walk_launch_f64(ts_ctx* c, const WalkParams& P, int bck, int mac, bool rel, int T) {
    // isolated BH and APE walks with one target per lane have their own kernel; MPE, periodic and mixed
    // BCs and the other groupings run the scalar one
    if (bck == 0 && T == 1 && mac != TS_MAC_MPE) {
        if (mac == TS_MAC_BH) return launch_walk64<TS_MAC_BH, false>(c, P);
        return rel ? launch_walk64<TS_MAC_APE, true>(c, P) : launch_walk64<TS_MAC_APE, false>(c, P);
    }
    return bck ? dispatch_bck<double, 1>(c, P, mac, rel, T) : dispatch_bck<double, 0>(c, P, mac, rel, T);
}
