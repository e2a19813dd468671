// Isolated FP32 walk for meshes of few cells (BH and APE MACs): 8 targets per warp, 4 lanes each.
//
// The paired walk of ts_walk_dev.cuh gives a warp 32 targets, and each pop then runs 4 pairs of children one
// after the other on every lane.  A 32^3 mesh has 1,024 such warps for 608 schedulers: the launch lasts as
// long as one warp's chain of ~320 pops, with most issue slots empty.  Here lane 8 s + t handles pair s of the
// 8 children for target t, so there are 4 times the warps, a pop is shorter, and 8 targets open fewer groups
// than 32.  It costs more instructions a target (the bookkeeping of a pop serves 8 targets instead of 32), so
// it is used only while the paired walk would leave the chip idle.  Walk alone, BH, paired -> split: 16^3 cells
// (128 warps) theta = 0.5 70 -> 44 us; 32^3 (1,024) theta = 0.4 / 0.5 / 0.8 145 -> 116, 108 -> 79, 51 -> 38 us; 36,352
// cells (1,136) 145 -> 131, 108 -> 88, 53 -> 43 us; 47,104 (1,472) 188 -> 176, 129 -> 116, 59 -> 55 us; but 61,440
// (1,920) theta = 0.5 159 -> 178 us and 64^3 (8,192) 384 -> 608 us.  The line, two warps per scheduler, lies below where
// the two meet.
// Every MAC decision is the paired walk's.
#pragma once
#include "ts_walk_dev.cuh"

#define SPLIT_MAX_WARPS 1216   // warps of 32 targets of the whole mesh: two per scheduler

// error-free sum: s + e = a + b
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
    s = __fadd_rn(a, b);
    const float v = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, v)), __fsub_rn(b, v));
}

template <int MAC, bool REL, bool SUB>
__global__ void __launch_bounds__(32 * TS_WALK_WARPS) k_walk_split(const __grid_constant__ WalkParams P) {
    __shared__ uint2 s_stack[TS_WALK_WARPS][TS_WALK_STACK];
    __shared__ float s_half[TS_MAX_DEPTH + 1][3], s_h2[TS_MAX_DEPTH + 1];
    for (int t = threadIdx.x; t <= TS_MAX_DEPTH; t += blockDim.x) {
        s_half[t][0] = P.geom->half32[t][0]; s_half[t][1] = P.geom->half32[t][1];
        s_half[t][2] = P.geom->half32[t][2]; s_h2[t] = P.geom->hmax2_32[t];
    }
    __syncthreads();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int tg = lane & 7, sub = lane >> 3;
    // gw: quarter (8 targets) of a warp of the other walks' lists
    int64_t gw = (int64_t)blockIdx.x * TS_WALK_WARPS + warp;
    if (P.warp_list) {                           // a subset of warps (Adaptive Block Update)
        if ((gw >> 2) >= *P.nwarp_dev) return;
        gw = 4 * (int64_t)P.warp_list[gw >> 2] + (gw & 3);
    } else if (P.targets) {                      // a list of single targets
        if (gw * 8 >= P.ntargets) return;
    } else {                                     // the cells of leaf-blocks [leaf_begin, leaf_end)
        gw += P.leaf_begin * 64;
        if (gw * 8 >= P.leaf_end * 512) return;
    }
    const float4* ncen = (const float4*)P.ncen;
    const int64_t me = P.targets ? P.targets[gw * 8 + tg] : gw * 8 + tg;
    const float* g0 = (const float*)(P.cell_soa + 8 * (me >> 3)) + (int)(me & 7);
    const float rx = g0[0], ry = g0[8], rz = g0[16];
    const int ml = (int)(me & 511);
    const int q = ml >> 6, o = (ml >> 3) & 7, o2 = ml & 7;
    const int ci = 4 * (q & 1) + 2 * (o & 1) + (o2 & 1);
    const int cj = 4 * ((q >> 1) & 1) + 2 * ((o >> 1) & 1) + ((o2 >> 1) & 1);
    const int ck = 4 * (q >> 2) + 2 * (o >> 2) + (o2 >> 2);
    const int64_t nat = (me >> 9) * 512 + ck * 64 + cj * 8 + ci;
    const float theta2 = (float)P.theta2, eta = (float)P.eta, G = (float)P.G;
    const float alim = REL ? (float)P.eps_rel * (float)P.a_old[nat] : (float)P.a_lim;
    const float ith2 = (float)(1.0 / P.theta2);
    const float2 nrx = make_float2(-rx, -rx), nry = make_float2(-ry, -ry), nrz = make_float2(-rz, -rz);
    float2 k01 = make_float2(0.f, 0.f), k23 = k01, c01 = k01, c23 = k01;   // compensated (phi, a_x), (a_y, a_z)
    unsigned n_int = 0, n_mac = 0, n_pop = 0, n_lanes = 0, root_lanes = 0;  // warp-uniform, in targets

    int sp = 0;
    bool overflow = false;
    {   // the root is tested like any node (its sums by the lanes of pair 0)
        const float4 c0 = ((const float4*)P.ncom)[0], gc = ncen[0];
        const float dx = rx - c0.x, dy = ry - c0.y, dz = rz - c0.z;
        const float d2 = dx * dx + dy * dy + dz * dz;
        const bool outside = fabsf(rx - gc.x) > eta * s_half[0][0] || fabsf(ry - gc.y) > eta * s_half[0][1] ||
                             fabsf(rz - gc.z) > eta * s_half[0][2];
        const bool mac = MAC == TS_MAC_BH ? s_h2[0] < theta2 * d2 : G * c0.w * s_h2[0] < alim * d2 * d2;
        const bool accept = outside && mac;
        if (accept && sub == 0) {
            const float inv = rsqrtf(d2), g3 = c0.w * inv * inv * inv;
            k01 = make_float2(c0.w * inv, -g3 * dx);
            k23 = make_float2(-g3 * dy, -g3 * dz);
        }
        const uint32_t om = __ballot_sync(0xffffffffu, !accept) & 0xffu;
        root_lanes = (unsigned)__popc(om);
        n_int = 8u - root_lanes;
        if (om) {
            if (lane == 0) s_stack[warp][0] = make_uint2(__float_as_uint(gc.w), om);
            sp = 1;
        }
    }
    __syncwarp();

    while (sp > 0 && !overflow) {
        const uint2 e = s_stack[warp][--sp];
        const uint32_t cw = e.x, m0 = e.y;   // m0: targets that opened the node
        const bool act = (m0 >> tg) & 1u, leaf = (cw & TS_CW_CELLS) != 0;
        const int first = (int)(cw & TS_CW_INDEX_MASK);
        const unsigned nt = (unsigned)__popc(m0);
        ++n_pop;
        n_lanes += nt;
        // this lane's pair of children
        const float2* sx = (const float2*)(leaf ? P.cell_soa + 8 * (first >> 3) : P.ncom_soa + 8 * ((first - 1) >> 3)) + sub;
        const float2 cx = __ldg(sx), cy = __ldg(sx + 4), cz = __ldg(sx + 8), m = __ldg(sx + 12);
        float2 dx, dy, dz, d2, s = make_float2(0.f, 0.f), ax = s, ay = s, az = s;
        pk_sep(cx, cy, cz, nrx, nry, nrz, dx, dy, dz, d2);
        if (leaf) {
            // ---- 8 leaf cells: every active target takes all of them except its own cell
            const unsigned self = (unsigned)me - (unsigned)first;
            n_int += 8u * nt - (unsigned)__popc(__ballot_sync(0xffffffffu, act && self < 8u) & 0xffu);
            pk_interact_m<SUB>(dx, dy, dz, d2, m, self != 2u * sub, self != 2u * sub + 1u, s, ax, ay, az);
        } else {
            // ---- 8 internal nodes
            const int dep = (int)(cw >> TS_CW_DEPTH_SHIFT);
            n_mac += 8u * nt;
            const float h2 = s_h2[dep];
            const uint32_t ccw = lane < 8 ? __float_as_uint(ncen[first + lane].w) : 0u;
            bool a0, a1;
            if constexpr (MAC == TS_MAC_BH) {
                const float hb = act ? h2 * ith2 : __int_as_float(0x7f800000);
                a0 = d2.x > hb; a1 = d2.y > hb;
            } else {
                const float2 hh = make_float2(h2, h2), gg = make_float2(G, G), al = make_float2(alim, alim);
                const float2 lhs = __fmul2_rn(__fmul2_rn(gg, m), hh), rhs = __fmul2_rn(__fmul2_rn(al, d2), d2);
                a0 = act && lhs.x < rhs.x; a1 = act && lhs.y < rhs.y;
            }
            if ((P.sb_depths >> dep) & 1u) {   // safe box of this lane's two children (x octants 0 and 1)
                const float4 gc = ncen[first];   // child 0; child (ox, oy, oz) lies at + 2 h (ox, oy, oz)
                const float hx = s_half[dep][0], hy = s_half[dep][1], hz = s_half[dep][2];
                const float qx = rx - gc.x, qy = ry - gc.y, qz = rz - gc.z;
                const bool y = fabsf(sub & 1 ? qy - 2 * hy : qy) <= eta * hy, z = fabsf(sub & 2 ? qz - 2 * hz : qz) <= eta * hz;
                a0 = a0 && !(y && z && fabsf(qx) <= eta * hx);
                a1 = a1 && !(y && z && fabsf(qx - 2 * hx) <= eta * hx);
            }
            const uint32_t b0 = __ballot_sync(0xffffffffu, a0), b1 = __ballot_sync(0xffffffffu, a1);
            pk_interact_m<SUB>(dx, dy, dz, d2, m, a0, a1, s, ax, ay, az);
            // push the opened children in one compacted write: lane j < 8 owns child j, whose accepting targets
            // are byte j / 2 of the ballot of its half of the pairs
            const uint32_t om = lane < 8 ? m0 & ~(((lane & 1 ? b1 : b0) >> (8 * (lane >> 1))) & 0xffu) : 0u;
            const unsigned nz = __ballot_sync(0xffffffffu, om != 0u);
            const int npush = __popc(nz);
            if (sp + npush > TS_WALK_STACK - 8) {   // (the stack limit of the other walks)
                overflow = true;
            } else {
                if (om) s_stack[warp][sp + __popc(nz & ((1u << lane) - 1u))] = make_uint2(ccw, om);
                sp += npush;
            }
        }
        if (act) {
            kahan_add2(k01, c01, make_float2(s.x + s.y, ax.x + ax.y));
            kahan_add2(k23, c23, make_float2(ay.x + ay.y, az.x + az.y));
        }
        __syncwarp();
    }
    if (overflow && lane == 0) atomicOr(P.status, TS_DEV_STACK_OVERFLOW);
    // the four lanes of a target: compensated sum of their sums
    float hi[4] = {k01.x, k01.y, k23.x, k23.y}, lo[4] = {-c01.x, -c01.y, -c23.x, -c23.y};
#pragma unroll
    for (int off = 8; off < 32; off <<= 1)
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const float h = __shfl_xor_sync(0xffffffffu, hi[k], off), l = __shfl_xor_sync(0xffffffffu, lo[k], off);
            float r, er;
            two_sum(hi[k], h, r, er);
            hi[k] = r;
            lo[k] = (lo[k] + l) + er;
        }
    const float phi = -G * (hi[0] + lo[0]), ax = G * (hi[1] + lo[1]), ay = G * (hi[2] + lo[2]), az = G * (hi[3] + lo[3]);
    if (sub == 0) {
        const int64_t oi = P.targets ? gw * 8 + tg : nat;
        ((float*)P.pot)[oi] = phi;
        float* acc = (float*)P.acc + 3 * oi;
        acc[0] = ax; acc[1] = ay; acc[2] = az;
        if (!isfinite(phi) || !isfinite(ax) || !isfinite(ay) || !isfinite(az)) atomicOr(P.status, TS_DEV_NONFINITE);
    }
    if (lane == 0) {
        // every opened (target, child) pair is popped once, so the accepted internal ones are the rest
        const unsigned wi = n_int + n_mac - (n_lanes - root_lanes);
        atomicAdd(&P.counters[0], (unsigned long long)wi);
        atomicAdd(&P.counters[1], (unsigned long long)(n_mac + 8u));
        atomicAdd(&P.counters[2], (unsigned long long)n_pop);
        atomicAdd(&P.counters[3], (unsigned long long)(4u * n_lanes));
        if (P.blk_counts && !P.targets) atomicAdd(&P.blk_counts[gw >> 6], (unsigned long long)wi);
    }
}

template <int MAC, bool REL, bool SUB = false>
static cudaError_t launch_split(ts_ctx* c, const WalkParams& P) {
    if constexpr (!SUB)   // (see rsq)
        if (P.tiny) return launch_split<MAC, REL, true>(c, P);
    const int64_t nwarps = P.targets ? P.ntargets / 8 : (P.leaf_end - P.leaf_begin) * 64;
    if (nwarps <= 0) return cudaSuccess;
    k_walk_split<MAC, REL, SUB><<<(int)((nwarps + TS_WALK_WARPS - 1) / TS_WALK_WARPS), 32 * TS_WALK_WARPS, 0, c->stream>>>(P);
    return cudaGetLastError();
}
