// FP64 gravity walk of isolated meshes, one target per lane, BH and APE MACs (eqs. pot / accel, bhmac, ape).
//
// Bound by the FP64 pipe: GB300 runs one FP64 warp instruction in the time of 64 FP32 or integer ones,
// so the kernel spends those freely to save FP64 ones.  The scalar walk of ts_walk_dev.cuh spends 24 of
// them per (32 lanes, child), many on lanes that do not take the child.  Here
//   - MAC and safe-box tests run in FP32 with a guard band wider than the FP32 rounding of the
//     coordinates; only a lane inside the band decides in FP64, by the same expressions as the scalar
//     walk, so every decision is the FP64 one;
//   - d^2, m / |d| and m / |d|^3 are formed by 64-bit integer arithmetic on the mantissas (pair64): an
//     interaction takes 7 FP64 instructions (separation 3, sums 4);
//   - a leaf-cell group opened by at most 16 lanes (the mean is 11) spreads each target's 8 cells over
//     2, 4 or 8 lanes, in a summation order that does not depend on how many lanes that is, so a
//     target's result does not depend on the other targets of its warp.
// 806,912-cell Plummer mesh, theta = 0.5: 67.4 ms with the scalar walk, 45.9 ms with FP64 reciprocal square
// roots (18 instructions an interaction), 27.6 ms with those in integers (10), 20.9 ms with d^2 too (7); the FP64
// pipe is 87 % busy.  The integer forms are also the more precise ones: m / |d| and m / |d|^3 are within 0.56 units
// in the last place (1/2 for the rounding; the truncated products of d^2 and of the last Newton step add up to
// 7.5 2^-60 relative), where the FP64 instructions give up to 4.5.
// The gain is smaller where FP32 decides less or an argument takes the FP64 instructions (348,160-cell mesh, 9.0 ms
// in lengths of order 1, 28.4 ms with the scalar walk): lengths of 1e18 17.9 ms (nothing is accepted in FP32 from
// h^2 / theta^2 = 1e30 on), half of the blocks massless 14.7 ms, nine tenths 19.4 ms.
#pragma once
#include <float.h>

#include "ts_walk_dev.cuh"

#define W64_GROUPED 16   // most active lanes of a cell group whose cells are spread over lanes

// A positive value q 2^e (q with its leading bit at 62, bits below it to be rounded off) as an FP64 bit
// pattern: biased exponent E for a mantissa in [1, 2), rounded to nearest (a carry moves into E).
__device__ __forceinline__ double pack64(unsigned long long q, int E) {
    return __longlong_as_double((long long)(((q + 512ull) >> 10) + ((unsigned long long)(unsigned)(E - 1) << 52)));
}

// |v| as a 64-bit fixed-point number F 2^(E - 1085) at the common biased exponent E >= that of v (F < 2^63; bits
// below 2^-62 of the scale are dropped; zero and subnormal v count as 0)
__device__ __forceinline__ unsigned long long fixed64(double v, int E) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(v);
    const int e = (int)(b >> 52) & 0x7ff;
    const unsigned long long M = ((b & ((1ull << 52) - 1)) | 1ull << 52) << 10;
    return e ? M >> min(E - e, 63) : 0ull;
}

// mi = m / |d| and g3 = m / |d|^3 to FP64 rounding, without the FP64 pipe.  |d|^2 is summed in 64-bit fixed
// point at the scale of the largest component: X 2^(2k - 62), X in [2^62, 2^64).  An FP32 seed of
// 1 / sqrt(X 2^-62) is refined twice, y (1 + e / 2) with e = 1 - X y^2 from fixed-point products: 2^-22 -> 2^-43 ->
// 2^-60 (Newton's iteration; the products' truncation is the last term).  The mantissa of m is multiplied
// the same way.  Arguments whose exponents come near the ends of the FP64 range (zero, infinite or NaN ones
// among them) take the FP64 instructions.
__device__ __forceinline__ void pair64(double dx, double dy, double dz, double m, double& mi, double& g3) {
    const int E = max(max((__double2hiint(dx) >> 20) & 0x7ff, (__double2hiint(dy) >> 20) & 0x7ff),
                      (__double2hiint(dz) >> 20) & 0x7ff);
    const unsigned long long mb = (unsigned long long)__double_as_longlong(m);
    const int em = (int)(mb >> 52) & 0x7ff;
    const unsigned long long one = 1ull << 52;
    const unsigned long long fx = fixed64(dx, E), fy = fixed64(dy, E), fz = fixed64(dz, E);
    const unsigned long long S = __umul64hi(fx, fx) + __umul64hi(fy, fy) + __umul64hi(fz, fz);   // in [2^60, 3 2^62)
    const int sh = S >> 62 ? 0 : 2;
    const unsigned long long X = S << sh;
    const int k = E - 1022 - (sh >> 1);
    float f;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(f) : "f"((float)(unsigned)(X >> 32) * 9.31322574615478515625e-10f));   // 2^-30
    const unsigned y0 = min(__float2uint_rn(f * 2147483648.f), 0x80000000u);                                        // 2^31 y
    const unsigned long long U = 1ull << 60;
    const int r0 = (int)((long long)(U - __umul64hi(X, (unsigned long long)y0 * y0)) >> 10);                         // 2^50 e
    const unsigned long long y1 = ((unsigned long long)y0 << 32) + (unsigned long long)(((long long)(int)(y0 >> 1) * r0) >> 18);
    const int r1 = (int)(long long)(U - __umul64hi(X, __umul64hi(y1, y1)));                                          // 2^60 e
    const unsigned long long y = y1 + (unsigned long long)(((long long)(int)(y1 >> 33) * r1) >> 28);                 // 2^63 y
    const unsigned long long y3 = __umul64hi(__umul64hi(y, y) << 1, y);                                              // 2^62 y^3
    const unsigned long long M = ((mb & (one - 1)) | one) << 11;
    const unsigned long long h1 = __umul64hi(M, y), h3 = __umul64hi(M, y3);
    const int s1 = __clzll((long long)h1), s3 = __clzll((long long)h3);
    const int E1 = 1 - s1 + em - k, E3 = 2 - s3 + em - 3 * k;
    if ((unsigned)(E - 64) < 1960u && (unsigned)(em - 1) < 2046u && (unsigned)(E1 - 2) < 2044u && (unsigned)(E3 - 2) < 2044u) {
        mi = pack64(h1 << (s1 - 1), E1);
        g3 = pack64(h3 << (s3 - 1), E3);
        if ((long long)mb < 0) { mi = -mi; g3 = -g3; }
    } else {
        const double inv = rsqrt(dx * dx + dy * dy + dz * dz);
        mi = m * inv;
        g3 = mi * (inv * inv);
    }
}

struct Sum64 {
    double p, x, y, z;   // sum of m / |d| and of m d / |d|^3, d = child - target
};

// one child: the terms (mi, g3 d); zero where the lane does not take it
__device__ __forceinline__ void terms64(bool take, double dx, double dy, double dz, double m, double& mi, double& g3) {
    pair64(take ? dx : 1.0, dy, dz, take ? m : 1.0, mi, g3);   // (1: keeps its own cell's zero off the slow branch)
    if (!take) mi = g3 = 0.0;
}

__device__ __forceinline__ void add64(Sum64& s, bool take, double dx, double dy, double dz, double m) {
    double mi, g3;
    terms64(take, dx, dy, dz, m, mi, g3);
    s.p += mi;
    s.x = fma(g3, dx, s.x);
    s.y = fma(g3, dy, s.y);
    s.z = fma(g3, dz, s.z);
}

__device__ __forceinline__ Sum64 operator+(const Sum64& a, const Sum64& b) {
    return Sum64{a.p + b.p, a.x + b.x, a.y + b.y, a.z + b.z};
}

__device__ __forceinline__ Sum64 shfl_xor64(const Sum64& a, int off) {
    return Sum64{__shfl_xor_sync(0xffffffffu, a.p, off), __shfl_xor_sync(0xffffffffu, a.x, off),
                 __shfl_xor_sync(0xffffffffu, a.y, off), __shfl_xor_sync(0xffffffffu, a.z, off)};
}

template <int MAC, bool REL>
__global__ void __launch_bounds__(32 * TS_WALK_WARPS) k_walk64(const __grid_constant__ WalkParams P) {
    __shared__ __align__(32) dbl4 s_com[TS_WALK_WARPS][8];
    __shared__ uint2 s_stack[TS_WALK_WARPS][TS_WALK_STACK];
    __shared__ double s_pos[TS_WALK_WARPS][3][32];
    __shared__ __align__(32) dbl4 s_res[TS_WALK_WARPS][W64_GROUPED];
    __shared__ int s_id[TS_WALK_WARPS][32], s_list[TS_WALK_WARPS][W64_GROUPED];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int64_t gw = (int64_t)blockIdx.x * TS_WALK_WARPS + warp;
    if (P.warp_list) {                           // a subset of warps (Adaptive Block Update)
        if (gw >= *P.nwarp_dev) return;
        gw = P.warp_list[gw];
    } else if (P.targets) {                      // a list of single targets
        if (gw * 32 >= P.ntargets) return;
    } else {                                     // the cells of leaf-blocks [leaf_begin, leaf_end)
        gw += P.leaf_begin * 16;
        if (gw * 32 >= P.leaf_end * 512) return;
    }
    const dbl4* ncom = (const dbl4*)P.ncom;
    const dbl4* ncen = (const dbl4*)P.ncen;
    const dbl4* cell = (const dbl4*)P.cell;
    const int64_t me = P.targets ? P.targets[gw * 32 + lane] : gw * 32 + lane;
    const dbl4 mine = cell[me];
    const double rx = mine.x, ry = mine.y, rz = mine.z;
    const int ml = (int)(me & 511);
    const int q = ml >> 6, o = (ml >> 3) & 7, o2 = ml & 7;
    const int ci = 4 * (q & 1) + 2 * (o & 1) + (o2 & 1);
    const int cj = 4 * ((q >> 1) & 1) + 2 * ((o >> 1) & 1) + ((o2 >> 1) & 1);
    const int ck = 4 * (q >> 2) + 2 * (o >> 2) + (o2 >> 2);
    const int64_t nat = (me >> 9) * 512 + ck * 64 + cj * 8 + ci;
    const double theta2 = P.theta2, eta = P.eta, G = P.G;
    const double alim = REL ? P.eps_rel * (double)P.a_old[nat] : P.a_lim;
    const float frx = (float)rx, fry = (float)ry, frz = (float)rz;
    const float2 nrx = make_float2(-frx, -frx), nry = make_float2(-fry, -fry), nrz = make_float2(-frz, -frz);
    const float fal = (float)alim, fG = (float)G, feta = (float)eta;
    // APE: a side of the test keeps its relative error only if its factors, and G m, are normal numbers
    // (a subnormal one met by a large h^2 or d^4 gives a wrong result of ordinary size)
    const bool ape32 = fabsf(fG) >= FLT_MIN && fal >= FLT_MIN;
    s_pos[warp][0][lane] = rx; s_pos[warp][1][lane] = ry; s_pos[warp][2][lane] = rz;
    s_id[warp][lane] = (int)me;
    Sum64 S{0, 0, 0, 0};
    unsigned n_int = 0, n_mac = 0, n_pop = 0, n_lanes = 0, root_lanes = 0;   // warp-uniform
    unsigned n_root = 0;

    // the exact decision for one child: eqs. bhmac / ape on FP64 separations
    auto mac64 = [&](const dbl4& c, double h2) -> bool {
        const double dx = rx - c.x, dy = ry - c.y, dz = rz - c.z;
        const double d2 = dx * dx + dy * dy + dz * dz;
        return MAC == TS_MAC_BH ? h2 < theta2 * d2 : G * c.w * h2 < alim * d2 * d2;
    };

    int sp = 0;
    bool overflow = false;
    {   // the root is tested like any node
        const dbl4 c0 = ncom[0], g0 = ncen[0];
        const double* hf = P.geom->half64[0];
        const bool outside = fabs(rx - g0.x) > eta * hf[0] || fabs(ry - g0.y) > eta * hf[1] || fabs(rz - g0.z) > eta * hf[2];
        const bool accept = outside && mac64(c0, P.geom->hmax2_64[0]);
        if (accept) {
            const double dx = c0.x - rx, dy = c0.y - ry, dz = c0.z - rz;
            add64(S, true, dx, dy, dz, c0.w);
        }
        const uint32_t om = __ballot_sync(0xffffffffu, !accept);
        root_lanes = (unsigned)__popc(om);
        n_root = 32u - root_lanes;
        if (om) {
            if (lane == 0) s_stack[warp][0] = make_uint2((uint32_t)g0.w, om);
            sp = 1;
        }
    }
    __syncwarp();

    while (sp > 0 && !overflow) {
        const uint2 e = s_stack[warp][--sp];
        const uint32_t cw = e.x, m0 = e.y;
        const bool act = (m0 >> lane) & 1u;
        const int lanes = __popc(m0);
        const int first = (int)(cw & TS_CW_INDEX_MASK);
        const int dep = (int)(cw >> TS_CW_DEPTH_SHIFT);
        ++n_pop;
        n_lanes += (unsigned)lanes;
        if (cw & TS_CW_CELLS) {
            // ---- 8 leaf cells: every active target takes all of them except its own cell
            if (lane < 8) s_com[warp][lane] = cell[first + lane];
            const int myrank = __popc(m0 & ((1u << lane) - 1u));
            if (lanes <= W64_GROUPED && act) s_list[warp][myrank] = lane;
            __syncwarp();
            n_int += 8u * (unsigned)lanes - (unsigned)__popc(__ballot_sync(0xffffffffu, act && (unsigned)((int)me - first) < 8u));
            // The group's sum is ((c0 + c1) + (c2 + c3)) with c_s = cell s, then cell s + 4 added by fma.
            if (lanes > W64_GROUPED) {
                const int self = (int)me - first;
                Sum64 g{0, 0, 0, 0}, h{0, 0, 0, 0};   // the sum of the first two chains; the chain before
#pragma unroll 1
                for (int s = 0; s < 4; ++s) {
                    Sum64 T{0, 0, 0, 0};
#pragma unroll 1
                    for (int j = s; j < 8; j += 4) {
                        const dbl4 c = s_com[warp][j];
                        add64(T, act && j != self, c.x - rx, c.y - ry, c.z - rz, c.w);
                    }
                    if (s == 1) g = h + T;
                    if (s == 3) g = g + (h + T);
                    h = T;
                }
                if (act) S = S + g;
            } else {
                // 2^sh lanes per target, lane r 2^sh + s of target r: one cell each (sh = 3), the cells s and
                // s + 4 (sh = 2), or those of s and s + 2 (sh = 1)
                const int sh = lanes <= 4 ? 3 : lanes <= 8 ? 2 : 1;
                const int r = lane >> sh, sub = lane & ((1 << sh) - 1);
                const bool valid = r < lanes;
                const int ow = s_list[warp][valid ? r : 0];
                const double ox = s_pos[warp][0][ow], oy = s_pos[warp][1][ow], oz = s_pos[warp][2][ow];
                const int self = s_id[warp][ow] - first;
                Sum64 T{0, 0, 0, 0};
                if (sh == 3) {
                    // cell sub: lanes 0..3 of a target take the terms of cells 4..7 from lanes 4..7
                    const dbl4 c = s_com[warp][sub];
                    const double dx = c.x - ox, dy = c.y - oy, dz = c.z - oz;
                    double mi, g3;
                    terms64(valid && sub != self, dx, dy, dz, c.w, mi, g3);
                    const double mj = __shfl_down_sync(0xffffffffu, mi, 4), h3 = __shfl_down_sync(0xffffffffu, g3, 4);
                    const double ex = __shfl_down_sync(0xffffffffu, dx, 4), ey = __shfl_down_sync(0xffffffffu, dy, 4),
                                 ez = __shfl_down_sync(0xffffffffu, dz, 4);
                    T = Sum64{mi + mj, fma(h3, ex, g3 * dx), fma(h3, ey, g3 * dy), fma(h3, ez, g3 * dz)};
                } else {
#pragma unroll 1
                    for (int j = sub; j < 8; j += 4) {
                        const dbl4 c = s_com[warp][j];
                        add64(T, valid && j != self, c.x - ox, c.y - oy, c.z - oz, c.w);
                    }
                }
                T = T + shfl_xor64(T, 1);
                if (sh >= 2) {
                    T = T + shfl_xor64(T, 2);
                } else {   // the other two chains
                    Sum64 V{0, 0, 0, 0};
#pragma unroll 1
                    for (int j = sub + 2; j < 8; j += 4) {
                        const dbl4 c = s_com[warp][j];
                        add64(V, valid && j != self, c.x - ox, c.y - oy, c.z - oz, c.w);
                    }
                    V = V + shfl_xor64(V, 1);
                    T = T + V;
                }
                if (valid && sub == 0) s_res[warp][r] = dbl4{T.p, T.x, T.y, T.z};
                __syncwarp();
                const dbl4 v = s_res[warp][act ? myrank : 0];
                if (act) S = S + Sum64{v.x, v.y, v.z, v.w};
            }
        } else {
            // ---- 8 internal nodes
            if (lane < 8) s_com[warp][lane] = ncom[first + lane];
            n_mac += 8u * (unsigned)lanes;
            const bool sbd = (P.sb_depths >> dep) & 1u;
            // FP32 decisions: bit j of sure / may: child j passes the MAC for certain / possibly
            unsigned sure = 0u, may = 0u;
            const float4* sx = P.ncom_soa + 8 * ((first - 1) >> 3);
            const float tlo = P.thr[dep], thi = P.thr_hi[dep], h2f = P.geom->hmax2_32[dep];
            const bool dep32 = ape32 && h2f >= FLT_MIN;
            if constexpr (MAC == TS_MAC_APE) __syncwarp();   // (s_com)
            // exactly massless (a mass below the FP32 range is 0 there too)
            auto massless = [&](int j) { return (unsigned long long)__double_as_longlong(s_com[warp][j].w) << 1 == 0ull; };
#pragma unroll
            for (int qq = 0; qq < 2; ++qq) {
                const float4 X = __ldg(sx + qq), Y = __ldg(sx + 2 + qq), Z = __ldg(sx + 4 + qq), M = __ldg(sx + 6 + qq);
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    float2 cx, cy, cz, m, dx, dy, dz, d2;
                    pk_pair(X, Y, Z, M, h, cx, cy, cz, m);
                    pk_sep(cx, cy, cz, nrx, nry, nrz, dx, dy, dz, d2);
#pragma unroll
                    for (int u = 0; u < 2; ++u) {
                        const int j = 4 * qq + 2 * h + u;
                        const float v = u ? d2.y : d2.x;
                        bool s, y;
                        if constexpr (MAC == TS_MAC_BH) {
                            s = v > thi;
                            y = !(v <= tlo);
                        } else {
                            // |d2 - v| <= 2 t v + s0 (t = 1e-5 and the cross term of the coordinate errors)
                            const float lo = fmaxf(fmaf(v, 1.f - 2e-5f, -P.ape_s0), 0.f), hi = fmaf(v, 1.f + 2e-5f, P.ape_s0);
                            const float mm = u ? m.y : m.x, gm = fG * mm;
                            const float lhs = gm * h2f, rl = fal * lo * lo, rh = fal * hi * hi;
                            const bool ok = dep32 && (fminf(fabsf(mm), fabsf(gm)) >= FLT_MIN || (mm == 0.f && massless(4 * qq + 2 * h + u)));
                            // (a left side below 1e-30 may have underflowed: it counts as 1e-30)
                            s = ok && lhs >= 0.f && rl < 1e30f && fmaxf(lhs, 1e-30f) * 1.000002f < rl;
                            y = !(ok && lhs > 1e-30f && lhs < 1e30f && lhs * 0.999998f >= rh);
                        }
                        sure |= (s ? 1u : 0u) << j;
                        may |= (y ? 1u : 0u) << j;
                    }
                }
            }
            if (sbd) {   // safe box: children's centres at c0 + 2 h (ox, oy, oz); bits inside for certain / possibly
                const float4 g0 = P.ncen32[first];
                unsigned in[2];
#pragma unroll
                for (int w = 0; w < 2; ++w) {
                    const float tol = w ? P.box_tol : -P.box_tol;
                    auto bits = [&](float qv, float hv, unsigned b0, unsigned b1) {
                        const float ev = fmaf(feta * hv, w ? 1.000002f : 0.999998f, tol);
                        const float q1 = qv - 2.f * hv;   // (a NaN is possibly inside, not certainly)
                        return w ? (!(fabsf(qv) > ev) ? b0 : 0u) | (!(fabsf(q1) > ev) ? b1 : 0u)
                                 : (fabsf(qv) <= ev ? b0 : 0u) | (fabsf(q1) <= ev ? b1 : 0u);
                    };
                    in[w] = bits(frx - g0.x, P.geom->half32[dep][0], 0x55u, 0xAAu) &
                            bits(fry - g0.y, P.geom->half32[dep][1], 0x33u, 0xCCu) &
                            bits(frz - g0.z, P.geom->half32[dep][2], 0x0Fu, 0xF0u);
                }
                sure &= ~in[1];
                may &= ~in[0];
            }
            unsigned amb = act ? may & ~sure : 0u;
            __syncwarp();
            if (__any_sync(0xffffffffu, amb)) {
                const dbl4 g0 = ncen[first];
                const double hx = P.geom->half64[dep][0], hy = P.geom->half64[dep][1], hz = P.geom->half64[dep][2];
                const double h2 = P.geom->hmax2_64[dep];
                while (amb) {   // (lanes diverge: the band is narrow)
                    const int j = __ffs((int)amb) - 1;
                    amb &= amb - 1u;
                    const bool inside = sbd && fabs(rx - g0.x - (j & 1 ? 2 * hx : 0.0)) <= eta * hx &&
                                        fabs(ry - g0.y - (j & 2 ? 2 * hy : 0.0)) <= eta * hy &&
                                        fabs(rz - g0.z - (j & 4 ? 2 * hz : 0.0)) <= eta * hz;
                    if (!inside && mac64(s_com[warp][j], h2)) sure |= 1u << j;
                }
                __syncwarp();
            }
            if (!act) sure = 0u;
            uint32_t my_om = 0;   // lane j < 8: the lanes that open child j
            Sum64 g{0, 0, 0, 0};
#pragma unroll 1
            for (int j = 0; j < 8; ++j) {
                const bool take = (sure >> j) & 1u;
                const uint32_t b = __ballot_sync(0xffffffffu, take);
                if (lane == j) my_om = m0 & ~b;
                if (b) {
                    const dbl4 c = s_com[warp][j];
                    add64(g, take, c.x - rx, c.y - ry, c.z - rz, c.w);
                }
            }
            if (sure) S = S + g;
            // push the opened children in one compacted write: lane j < 8 owns child j
            const unsigned nz = __ballot_sync(0xffffffffu, my_om != 0u);
            const int npush = __popc(nz);
            if (sp + npush > TS_WALK_STACK - 8) {   // (the stack limit of the other walks)
                overflow = true;
            } else {
                if (my_om)
                    s_stack[warp][sp + __popc(nz & ((1u << lane) - 1u))] =
                        make_uint2(__float_as_uint(P.ncen32[first + lane].w), my_om);
                sp += npush;
            }
        }
        __syncwarp();
    }
    if (overflow && lane == 0) atomicOr(P.status, TS_DEV_STACK_OVERFLOW);
    const int64_t oi = P.targets ? gw * 32 + lane : nat;
    const double phi = -G * S.p, ax = G * S.x, ay = G * S.y, az = G * S.z;
    ((double*)P.pot)[oi] = phi;
    double* acc = (double*)P.acc + 3 * oi;
    acc[0] = ax; acc[1] = ay; acc[2] = az;
    if (!isfinite(phi) || !isfinite(ax) || !isfinite(ay) || !isfinite(az)) atomicOr(P.status, TS_DEV_NONFINITE);
    if (lane == 0) {
        // every opened (lane, child) pair is popped once, so the accepted internal ones are the rest
        const unsigned wi = n_root + n_int + n_mac - (n_lanes - root_lanes);
        atomicAdd(&P.counters[0], (unsigned long long)wi);
        atomicAdd(&P.counters[1], (unsigned long long)(n_mac + 32u));
        atomicAdd(&P.counters[2], (unsigned long long)n_pop);
        atomicAdd(&P.counters[3], (unsigned long long)n_lanes);
        if (P.blk_counts && !P.targets) atomicAdd(&P.blk_counts[gw >> 4], (unsigned long long)wi);
    }
}

template <int MAC, bool REL>
static cudaError_t launch_walk64(ts_ctx* c, const WalkParams& P) {
    const int64_t nwarps = P.targets ? P.ntargets / 32 : (P.leaf_end - P.leaf_begin) * 16;
    if (nwarps <= 0) return cudaSuccess;
    k_walk64<MAC, REL><<<(int)((nwarps + TS_WALK_WARPS - 1) / TS_WALK_WARPS), 32 * TS_WALK_WARPS, 0, c->stream>>>(P);
    return cudaGetLastError();
}
