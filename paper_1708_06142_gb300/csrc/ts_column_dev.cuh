// Device code of the column-density walk shared by k_column_walk (ts_column.cu) and the batched
// persistent kernel (ts_batch.cu).  See ts_column.cu for the design.
#pragma once
#include <math.h>

#include "ts_internal.cuh"
#include "ts_pair.cuh"

struct ColParams {
    const float4* ncom;
    const float4* ncen;
    const float4* cell;
    int64_t ncell;
    float theta2, eta, max_dist2;    // max_dist2: infinite if unlimited
    const WalkGeom* geom;
    int npix, nth, nph;
    float nthf, nphf, nth1, nph1, nps1;   // bin counts, and the last bins
    int tiny;                        // 1: squared separations can be subnormal in FP32 (see rsq)
    float thr[TS_MAX_DEPTH + 1];     // BH MAC: accept iff d^2 > thr[depth] (h^2 < theta^2 d^2 in FP32)
    uint32_t sb_depths;              // bit d: the safe-box test can change a MAC decision at depth d
    float psi_lmin, psi_lscale;      // log2(psi_min), nps / log2(psi_max / psi_min)
    float inv_omega;                 // 1 / Omega_pix = N_PIX / (4 pi), times 1 / nsub^3 (see nr_pairs)
    const double* leaf_size;
    // node-ray table: one 32-byte record per entry (see ColHit), psi slowest, phi fastest (the lanes of a
    // warp see a node under similar angular sizes and neighbouring directions), nr_rec biased (see
    // col_bin2); the rows of more than four pixels continue in records of nr_more (record 0 unused).  A
    // weight is its sub-cube count over nsub^3 (the divisor is folded into inv_omega).
    const float4* nr_rec;
    const float4* nr_more;
    float* out;
    int* status;
    unsigned long long* counters;
    // extra mapped quantities (Sec. 2.3, l_q = 1 + nq maps): masses of up to 2 quantities per cell
    // (Morton order) and per internal node; maps and output rows are [l_q][npix]
    const float2* qcell;
    const float2* qnode;
};

// Children are binned two at a time with packed f32x2 arithmetic: direction, angles, bins and weight
// factors, then the loads of their node-ray records, then the scatters into the lane's own pixel map.  A
// record is 32 bytes, read by one 256-bit load (see ld_rec): the FP32 sub-cube counts of up to four pixels,
// their map offsets as 16-bit halves, and the record that continues a longer row.  128^3 box, N_PIX = 48:
// 27.3 ms child by child with 16-byte records of packed integers, 21.8 ms so, 20.0 ms with phi as the
// table's fastest index and rows continued by records instead of single pixels; the maps are the same bit
// for bit.
// cell_pairs, node_pairs: pairs of leaf cells and of internal children whose record loads are in flight
// together.  With the total map alone one of each at 6 CTAs of 4 warps per SM is fastest (128^3: 20.0 ms; two
// pairs of cells 21.4, two of children 20.8).  With extra quantities the maps in shared memory leave few warps
// on an SM, so CTAs of 2 warps, which waste less of it (10 resident warps instead of 8 with 3 maps of 48
// pixels), and two pairs in flight pay (64^3, 3 maps: 4.86 ms with 4 warps and one pair of children, 4.48 with
// 2 warps, 4.33 with two pairs as well).  One extra quantity takes the same: 64^3, 2 maps of 48 pixels 3.04 ms,
// 3.07 with 4 warps, 3.18 with one pair of each; of 12 pixels 2.42, 2.43, 2.35.
template <int NQ>
struct ColTune {
    static constexpr int cell_pairs = NQ == 0 ? 1 : 2, node_pairs = NQ == 0 ? 1 : 2;
    static constexpr int min_ctas = NQ == 0 ? 6 : 1, warps = NQ == 0 ? TS_WALK_WARPS : 2;
};

// Direction angles of the bins.  theta = acos u_z and phi = atan2(y, x) come from polynomials, not
// from acosf / atan2f (which cost a quarter of the walk): least-squares fits at Chebyshev nodes on
// [0, 1] of acos x = sqrt(1 - x) Q(x) (Q of degree 6, |error| < 4.1e-7 rad evaluated in FP32) and of
// atan a = a R(a^2) (R of degree 7, |error| < 1.4e-7 rad), extended to [-1, 1] and to the four
// quadrants by the angle identities (pi - acos|u|; pi/2 - atan, pi - phi, 2 pi - phi), each adding
// one FP32 rounding (at most 6.2e-7 rad in all).  These errors are of the order of the FP32 library
// functions' own, and so is the rate of bin decisions that differ from those of the FP64 angles (a
// few per 10^6 directions).  Zero components follow the signed-zero conventions of atan2: phi = pi
// for x = -0, y = +-0 (the direction straight along z from a node, where phi is undefined), 0 for
// x = +0.
#define COL_F2(c) make_float2(c, c)

__device__ __forceinline__ float col_acos(float u) {
    const float x = fabsf(u), om = 1.f - x;
    const float q = fmaf(fmaf(fmaf(fmaf(fmaf(fmaf(0.0025606194976717234f, x, -0.01186282653361559f), x,
                                             0.027619101107120514f), x, -0.04913029447197914f), x,
                                   0.0888218879699707f), x, -0.21459004282951355f), x, 1.570796251296997f);
    const float a = q * (om * rsqrtf(fmaxf(om, 1e-30f)));   // sqrt(1 - x), 0 at x = 1
    return u < 0.f ? (float)M_PI - a : a;
}

__device__ __forceinline__ float col_phi(float y, float x) {   // atan2(y, x) wrapped to [0, 2 pi)
    const float ax = fabsf(x), ay = fabsf(y), mx = fmaxf(ax, ay);
    const float a = mx > 0.f ? __fdividef(fminf(ax, ay), mx) : 0.f;
    const float s = a * a;
    float p = a * fmaf(fmaf(fmaf(fmaf(fmaf(fmaf(fmaf(-0.004073309246450663f, s, 0.021946610882878304f), s,
                                                -0.056063175201416016f), s, 0.09656256437301636f), s,
                                      -0.13915802538394928f), s, 0.19948509335517883f), s,
                            -0.3333010673522949f), s, 0.999999463558197f);
    if (ay > ax) p = (float)(0.5 * M_PI) - p;
    if (signbit(x)) p = (float)M_PI - p;
    if (y < 0.f) p = (float)(2.0 * M_PI) - p;
    return p;
}

// The same for two directions at once, with the instructions that flush subnormal numbers (the scalar
// functions above serve the meshes where separations can be subnormal; normal arguments give the same
// bits in both).
__device__ __forceinline__ float col_ratio(float a, float b) {   // a / b
    float y;
    asm("div.approx.ftz.f32 %0, %1, %2;" : "=f"(y) : "f"(a), "f"(b));
    return y;
}

// acos of u with |u| = x for two directions; neg: u < 0
__device__ __forceinline__ float2 col_acos2(float2 x, bool neg0, bool neg1) {
    const float2 om = __ffma2_rn(x, COL_F2(-1.f), COL_F2(1.f));
    float2 q = __ffma2_rn(COL_F2(0.0025606194976717234f), x, COL_F2(-0.01186282653361559f));
    q = __ffma2_rn(q, x, COL_F2(0.027619101107120514f));
    q = __ffma2_rn(q, x, COL_F2(-0.04913029447197914f));
    q = __ffma2_rn(q, x, COL_F2(0.0888218879699707f));
    q = __ffma2_rn(q, x, COL_F2(-0.21459004282951355f));
    q = __ffma2_rn(q, x, COL_F2(1.570796251296997f));
    // sqrt(1 - x), 0 at x = 1
    const float2 r = __fmul2_rn(om, make_float2(rsq<false>(fmaxf(om.x, 1e-30f)), rsq<false>(fmaxf(om.y, 1e-30f))));
    const float2 a = __fmul2_rn(q, r), b = __ffma2_rn(a, COL_F2(-1.f), COL_F2((float)M_PI));
    return make_float2(neg0 ? b.x : a.x, neg1 ? b.y : a.y);
}

// atan2(-dy, -dx) wrapped to [0, 2 pi) for two directions
__device__ __forceinline__ float2 col_phi2(float2 dy, float2 dx) {
    float r[2];
    const float ax[2] = {fabsf(dx.x), fabsf(dx.y)}, ay[2] = {fabsf(dy.x), fabsf(dy.y)};
#pragma unroll
    for (int u = 0; u < 2; ++u) {
        const float mx = fmaxf(ax[u], ay[u]);
        r[u] = mx > 0.f ? col_ratio(fminf(ax[u], ay[u]), mx) : 0.f;
    }
    const float2 a = make_float2(r[0], r[1]), s = __fmul2_rn(a, a);
    float2 p = __ffma2_rn(COL_F2(-0.004073309246450663f), s, COL_F2(0.021946610882878304f));
    p = __ffma2_rn(p, s, COL_F2(-0.056063175201416016f));
    p = __ffma2_rn(p, s, COL_F2(0.09656256437301636f));
    p = __ffma2_rn(p, s, COL_F2(-0.13915802538394928f));
    p = __ffma2_rn(p, s, COL_F2(0.19948509335517883f));
    p = __ffma2_rn(p, s, COL_F2(-0.3333010673522949f));
    p = __ffma2_rn(p, s, COL_F2(0.999999463558197f));
    p = __fmul2_rn(a, p);
    float2 q = __ffma2_rn(p, COL_F2(-1.f), COL_F2((float)(0.5 * M_PI)));
    p = make_float2(ay[0] > ax[0] ? q.x : p.x, ay[1] > ax[1] ? q.y : p.y);
    q = __ffma2_rn(p, COL_F2(-1.f), COL_F2((float)M_PI));
    p = make_float2(signbit(dx.x) ? p.x : q.x, signbit(dx.y) ? p.y : q.y);
    q = __ffma2_rn(p, COL_F2(-1.f), COL_F2((float)(2.0 * M_PI)));
    return make_float2(dy.x > 0.f ? q.x : p.x, dy.y > 0.f ? q.y : p.y);
}

template <bool SUB>
__device__ __forceinline__ float col_log2(float x) {
    if constexpr (SUB) return __log2f(x);
    float y;
    asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

template <int NQ>
struct ColHit {
    float4 w;      // sub-cube counts of up to four pixels (0: unused, at a pixel of its own)
    float4 o;      // bits: their map offsets (bytes) in 16-bit halves of .x and .y; .z: 0 or the next record in nr_more
    float f, f1, f2;
};

// Bins and weight factors of two nodes for this lane; a node it does not take (acc false: outside the
// popped entry's mask, its own cell, or beyond max_dist) gets weight factors 0, so its scatter adds zeros
// and leaves the map unchanged.  d: separations target minus node; s: h / |d| uses h of the group.  A bin
// index is the floor of a coordinate clamped to the table (also a NaN), formed by adding 2^23 rounded
// down: its bits are 0x4b000000 + bin, and nr_rec points as many records before the table as the constant
// parts add up to (their sum has its low 24 bits zero and the table is shorter than 2^24).
template <int NQ, bool SUB>
__device__ __forceinline__ void col_bin2(const ColParams& P, bool acc0, bool acc1, float2 m, float2 qa, float2 qb,
                                         float2 dx, float2 dy, float2 dz, float2 d2, float h, ColHit<NQ>* hit) {
    constexpr float M23 = 8388608.f;
    acc0 = acc0 && !(d2.x > P.max_dist2);
    acc1 = acc1 && !(d2.y > P.max_dist2);
    const float2 inv = make_float2(rsq<SUB>(d2.x), rsq<SUB>(d2.y));
    // direction from the target to the node is -d
    const float2 uz = __fmul2_rn(dz, inv);
    float2 th, ph;
    if constexpr (SUB) {
        th = make_float2(col_acos(fminf(1.f, fmaxf(-1.f, -uz.x))), col_acos(fminf(1.f, fmaxf(-1.f, -uz.y))));
        ph = make_float2(col_phi(-dy.x, -dx.x), col_phi(-dy.y, -dx.y));
    } else {
        th = col_acos2(make_float2(fminf(1.f, fabsf(uz.x)), fminf(1.f, fabsf(uz.y))), uz.x > 0.f, uz.y > 0.f);
        ph = col_phi2(dy, dx);
    }
    const float2 psi = __fmul2_rn(COL_F2(h), inv);
    const float2 vt = __fmul2_rn(__fmul2_rn(th, COL_F2((float)(1.0 / M_PI))), COL_F2(P.nthf));
    const float2 vp = __fmul2_rn(__fmul2_rn(ph, COL_F2((float)(0.5 / M_PI))), COL_F2(P.nphf));
    const float2 vs = __fmul2_rn(__fadd2_rn(make_float2(col_log2<SUB>(psi.x), col_log2<SUB>(psi.y)), COL_F2(-P.psi_lmin)),
                                 COL_F2(P.psi_lscale));
    const float2 g = __fmul2_rn(__fmul2_rn(COL_F2(P.inv_omega), inv), inv);
    const float2 fm = __fmul2_rn(m, g);
    const float2 fa = NQ >= 1 ? __fmul2_rn(qa, g) : g, fb = NQ >= 2 ? __fmul2_rn(qb, g) : g;
#pragma unroll
    for (int u = 0; u < 2; ++u) {
        const float X = __fadd_rd(fminf(u ? vt.y : vt.x, P.nth1), M23);
        const float Y = __fadd_rd(fminf(u ? vp.y : vp.x, P.nph1), M23);
        const float Z = __fadd_rd(fminf(fmaxf(u ? vs.y : vs.x, 0.f), P.nps1), M23);
        const uint32_t e = (__float_as_uint(Z) * (uint32_t)P.nth + __float_as_uint(X)) * (uint32_t)P.nph + __float_as_uint(Y);
        ld_rec(P.nr_rec + 2 * (size_t)e, hit[u].w, hit[u].o);
        const bool acc = u ? acc1 : acc0;
        hit[u].f = acc ? (u ? fm.y : fm.x) : 0.f;
        if constexpr (NQ >= 1) hit[u].f1 = acc ? (u ? fa.y : fa.x) : 0.f;
        if constexpr (NQ >= 2) hit[u].f2 = acc ? (u ? fb.y : fb.x) : 0.f;
    }
}

// Scatter of one node into this lane's pixel map and its quantity masses into the following maps
// (map stride npix * 32).  The four slots of a record are added without a test (an unused slot adds 0 to
// a pixel of its own), which keeps the lanes of a warp on one path; the four pixels are distinct, so all
// are read before the first is written.  A longer row continues in further records.  map: the lane's
// column of the map.
template <int NQ>
__device__ __forceinline__ void col_scatter(const ColParams& P, float* map, const ColHit<NQ>& hit) {
    const int ms = P.npix * 32;
    auto add4 = [&](const float4& w4, const float4& o4) {
        const uint32_t a = __float_as_uint(o4.x), b = __float_as_uint(o4.y);
        const uint32_t off[4] = {a & 0xffffu, a >> 16, b & 0xffffu, b >> 16};
        const float w[4] = {w4.x, w4.y, w4.z, w4.w};
#pragma unroll
        for (int k = 0; k <= NQ; ++k) {
            const float f = k == 0 ? hit.f : k == 1 ? hit.f1 : hit.f2;
            float v[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) v[i] = *(const float*)((const char*)(map + k * ms) + off[i]);
#pragma unroll
            for (int i = 0; i < 4; ++i) *(float*)((char*)(map + k * ms) + off[i]) = fmaf(f, w[i], v[i]);
        }
    };
    add4(hit.w, hit.o);
    for (uint32_t more = __float_as_uint(hit.o.z); more;) {
        float4 w, o;
        ld_rec(P.nr_more + 2 * (size_t)more, w, o);
        add4(w, o);
        more = __float_as_uint(o.z);
    }
}

// One warp's column walk: warp gw of the grid described by P (32 Morton-consecutive targets), the
// same shared depth-first traversal as the gravity walk: a stack entry is the child word of an
// opened node and the mask of the lanes that opened it; a pop stages the 8 children in shared
// memory, each lane applies the BH MAC (with the safe box, evaluated once per group as an 8-bit
// mask) to each child, and the children opened by any lane are pushed in one compacted write.
// map: this warp's [1 + NQ][npix][32] pixel maps in shared memory; s_q_w: staging of the children's
// quantity masses (NQ > 0).
template <int NQ = 0, bool SUB = false>
__device__ __forceinline__ void col_walk_warp(const ColParams& P, int64_t gw, int lane, float* map, float4* s_com_w,
                                              float4* s_cen_w, uint2* s_stack_w, const float (*s_half)[3],
                                              const float* s_h2, float2* s_q_w = nullptr) {
    const int npix = P.npix;
    for (int p = 0; p < (1 + NQ) * npix; ++p) map[p * 32 + lane] = 0.f;
    float* mapl = map + lane;
    const float2 zq = make_float2(0.f, 0.f);
    const int64_t me = gw * 32 + lane;
    const float4 mine = P.cell[me];
    const float rx = mine.x, ry = mine.y, rz = mine.z;
    const int ml = (int)(me & 511);
    const int q = ml >> 6, o = (ml >> 3) & 7, o2 = ml & 7;
    const int ci = 4 * (q & 1) + 2 * (o & 1) + (o2 & 1);
    const int cj = 4 * ((q >> 1) & 1) + 2 * ((o >> 1) & 1) + ((o2 >> 1) & 1);
    const int ck = 4 * (q >> 2) + 2 * (o >> 2) + (o2 >> 2);
    const int64_t nat = (me >> 9) * 512 + ck * 64 + cj * 8 + ci;
    const int px = P.geom->pbc[0], py = P.geom->pbc[1], pz = P.geom->pbc[2];
    const float Lx = (float)P.geom->L[0], Ly = (float)P.geom->L[1], Lz = (float)P.geom->L[2];
    const float iLx = (float)P.geom->invL[0], iLy = (float)P.geom->invL[1], iLz = (float)P.geom->invL[2];
    const bool per = px || py || pz;
    const float2 ilx = COL_F2(px ? iLx : 0.f), ily = COL_F2(py ? iLy : 0.f), ilz = COL_F2(pz ? iLz : 0.f);
    const float2 nlx = COL_F2(-Lx), nly = COL_F2(-Ly), nlz = COL_F2(-Lz);
    unsigned n_int = 0, n_mac = 0, n_lanes = 0, root_lanes = 0;   // warp-uniform
    auto mi = [](float d, int per, float L, float iL) { return per ? d - L * rintf(d * iL) : d; };
    // minimum-image separations (target minus child) of two staged children and their squares
    auto sep2 = [&](const float4& a, const float4& b, float2& dx, float2& dy, float2& dz, float2& d2) {
        dx = __ffma2_rn(make_float2(a.x, b.x), COL_F2(-1.f), COL_F2(rx));
        dy = __ffma2_rn(make_float2(a.y, b.y), COL_F2(-1.f), COL_F2(ry));
        dz = __ffma2_rn(make_float2(a.z, b.z), COL_F2(-1.f), COL_F2(rz));
        if (per) {
            dx = pk_image(dx, ilx, nlx);
            dy = pk_image(dy, ily, nly);
            dz = pk_image(dz, ilz, nlz);
        }
        d2 = __ffma2_rn(dz, dz, __ffma2_rn(dx, dx, __fmul2_rn(dy, dy)));
    };

    int sp = 0;
    bool overflow = false;
    {   // the root is tested like any node (opened unless the target sees the whole domain small)
        const float4 c0 = P.ncom[0];
        const float4 g0 = P.ncen[0];
        float2 dx, dy, dz, d2;
        sep2(c0, c0, dx, dy, dz, d2);
        const float gx = mi(rx - g0.x, px, Lx, iLx), gy = mi(ry - g0.y, py, Ly, iLy), gz = mi(rz - g0.z, pz, Lz, iLz);
        const bool outside = fabsf(gx) > P.eta * s_half[0][0] || fabsf(gy) > P.eta * s_half[0][1] ||
                             fabsf(gz) > P.eta * s_half[0][2];
        const bool accept = outside && d2.x > P.thr[0];
        if (accept) {
            ColHit<NQ> hit[2];
            const float2 q0 = NQ ? P.qnode[0] : zq;
            col_bin2<NQ, SUB>(P, true, false, COL_F2(c0.w), COL_F2(q0.x), COL_F2(q0.y), dx, dy, dz, d2, sqrtf(s_h2[0]), hit);
            col_scatter<NQ>(P, mapl, hit[0]);
        }
        const unsigned om = __ballot_sync(0xffffffffu, !accept);
        root_lanes = (unsigned)__popc(om);
        n_int = 32u - root_lanes;
        if (om) {
            if (lane == 0) s_stack_w[0] = make_uint2(__float_as_uint(g0.w), om);
            sp = 1;
        }
    }
    __syncwarp();
    while (sp > 0 && !overflow) {
        const uint2 e = s_stack_w[--sp];
        const uint32_t cw = e.x, mask = e.y;
        const int first = (int)(cw & TS_CW_INDEX_MASK);
        const int dep = (int)(cw >> TS_CW_DEPTH_SHIFT);
        const bool active = (mask >> lane) & 1u;
        n_lanes += (unsigned)__popc(mask);
        __syncwarp();
        if (cw & TS_CW_CELLS) {
            // ---- 8 leaf cells: every active target accepts all of them except its own cell; binned and
            // scattered by every lane of the warp (weights 0 in lanes that do not take them)
            if (lane < 8) s_com_w[lane] = P.cell[first + lane];
            if constexpr (NQ > 0) if (lane >= 16 && lane < 24) s_q_w[lane - 16] = P.qcell[first + lane - 16];
            const int self = (int)(me - first);
            n_int += 8u * (unsigned)__popc(mask) - (unsigned)__popc(__ballot_sync(0xffffffffu, active && (unsigned)self < 8u));
            __syncwarp();
            const float h = sqrtf(s_h2[dep]);
            constexpr int PAIRS = ColTune<NQ>::cell_pairs;
#pragma unroll 1
            for (int j0 = 0; j0 < 8; j0 += 2 * PAIRS) {
                ColHit<NQ> hit[2 * PAIRS];
#pragma unroll
                for (int u = 0; u < PAIRS; ++u) {
                    const int j = j0 + 2 * u;
                    const float4 a = s_com_w[j], b = s_com_w[j + 1];
                    const float2 p0 = NQ ? s_q_w[j] : zq, p1 = NQ ? s_q_w[j + 1] : zq;
                    float2 dx, dy, dz, d2;
                    sep2(a, b, dx, dy, dz, d2);
                    col_bin2<NQ, SUB>(P, active && j != self, active && j + 1 != self, make_float2(a.w, b.w),
                                      make_float2(p0.x, p1.x), make_float2(p0.y, p1.y), dx, dy, dz, d2, h, hit + 2 * u);
                }
#pragma unroll
                for (int u = 0; u < 2 * PAIRS; ++u) col_scatter<NQ>(P, mapl, hit[u]);
            }
        } else {
            // ---- 8 internal nodes
            if (lane < 8) s_com_w[lane] = P.ncom[first + lane];
            else if (lane < 16) s_cen_w[lane - 8] = P.ncen[first + lane - 8];
            else if (NQ > 0 && lane < 24) s_q_w[lane - 16] = P.qnode[first + lane - 16];
            __syncwarp();
            const float hx = s_half[dep][0], hy = s_half[dep][1], hz = s_half[dep][2];
            const float h = sqrtf(s_h2[dep]);
            // safe box once per group (children centres at c0 + 2 h (ox, oy, oz)); skipped where no
            // target inside it can pass the MAC
            unsigned inside = 0u;
            if ((P.sb_depths >> dep) & 1u) {
                const float4 g0 = s_cen_w[0];
                const float qx = rx - g0.x, qy = ry - g0.y, qz = rz - g0.z;
                const float ex = P.eta * hx, ey = P.eta * hy, ez = P.eta * hz;
                const bool x0 = fabsf(mi(qx, px, Lx, iLx)) <= ex, x1 = fabsf(mi(qx - 2 * hx, px, Lx, iLx)) <= ex;
                const bool y0 = fabsf(mi(qy, py, Ly, iLy)) <= ey, y1 = fabsf(mi(qy - 2 * hy, py, Ly, iLy)) <= ey;
                const bool z0 = fabsf(mi(qz, pz, Lz, iLz)) <= ez, z1 = fabsf(mi(qz - 2 * hz, pz, Lz, iLz)) <= ez;
                inside = ((x0 ? 0x55u : 0u) | (x1 ? 0xAAu : 0u)) & ((y0 ? 0x33u : 0u) | (y1 ? 0xCCu : 0u)) &
                         ((z0 ? 0x0Fu : 0u) | (z1 ? 0xF0u : 0u));
            }
            n_mac += 8u * (unsigned)__popc(mask);
            const float thr = active ? P.thr[dep] : __int_as_float(0x7f800000);
            // per NP pairs of children: MACs, bins and record loads, then the scatters
            constexpr int NP = ColTune<NQ>::node_pairs;
#pragma unroll 1
            for (int j0 = 0; j0 < 8; j0 += 2 * NP) {
                float2 dx[NP], dy[NP], dz[NP], d2[NP], m[NP];
                bool a0[NP], a1[NP], any = false;
#pragma unroll
                for (int u = 0; u < NP; ++u) {
                    const int j = j0 + 2 * u;
                    const float4 a = s_com_w[j], b = s_com_w[j + 1];
                    sep2(a, b, dx[u], dy[u], dz[u], d2[u]);
                    m[u] = make_float2(a.w, b.w);
                    a0[u] = d2[u].x > thr && !((inside >> j) & 1u);
                    a1[u] = d2[u].y > thr && !((inside >> (j + 1)) & 1u);
                    const unsigned b0 = __ballot_sync(0xffffffffu, a0[u]), b1 = __ballot_sync(0xffffffffu, a1[u]);
                    if (lane == 0) {   // the accepting lanes, parked above the stack top
                        s_stack_w[TS_WALK_STACK - 8 + j].y = b0;
                        s_stack_w[TS_WALK_STACK - 7 + j].y = b1;
                    }
                    any = any || a0[u] || a1[u];
                }
                if (any) {
                    ColHit<NQ> hit[2 * NP];
#pragma unroll
                    for (int u = 0; u < NP; ++u) {
                        const int j = j0 + 2 * u;
                        const float2 p0 = NQ ? s_q_w[j] : zq, p1 = NQ ? s_q_w[j + 1] : zq;
                        col_bin2<NQ, SUB>(P, a0[u], a1[u], m[u], make_float2(p0.x, p1.x), make_float2(p0.y, p1.y), dx[u], dy[u],
                                          dz[u], d2[u], h, hit + 2 * u);
                    }
#pragma unroll
                    for (int u = 0; u < 2 * NP; ++u) col_scatter<NQ>(P, mapl, hit[u]);
                }
            }
            __syncwarp();
            // push the opened children in one compacted write: lane j < 8 owns child j
            const uint32_t my_om = lane < 8 ? mask & ~s_stack_w[TS_WALK_STACK - 8 + lane].y : 0u;
            const unsigned nz = __ballot_sync(0xffffffffu, my_om != 0u);
            const int npush = __popc(nz);
            if (sp + npush > TS_WALK_STACK - 8) {   // the top 8 slots park the accept masks
                overflow = true;
            } else {
                if (my_om) s_stack_w[sp + __popc(nz & ((1u << lane) - 1u))] =
                    make_uint2(__float_as_uint(s_cen_w[lane].w), my_om);
                sp += npush;
            }
        }
        __syncwarp();
    }
    if (overflow && lane == 0) atomicOr(P.status, TS_DEV_STACK_OVERFLOW);
    // own cell: rho dx / 2 = m / (2 dy dz), cell edges dy = Ly_block / 8, dz = Lz_block / 8
    __syncwarp();
    const int64_t leaf = me >> 9;
    const double own_f = 32.0 / (P.leaf_size[3 * leaf + 1] * P.leaf_size[3 * leaf + 2]);
    float* out = P.out + nat * (1 + NQ) * npix;
#pragma unroll
    for (int k = 0; k <= NQ; ++k) {
        const float mk = k == 0 ? mine.w : (k == 1 ? P.qcell[me].x : P.qcell[me].y);
        const float own = (float)((double)mk * own_f);
        for (int p = 0; p < npix; ++p) out[k * npix + p] = map[(k * npix + p) * 32 + lane] + own;
    }
    if (lane == 0) {
        // every opened (lane, child) pair is popped once: the accepted internal ones are the rest
        atomicAdd(&P.counters[0], (unsigned long long)(n_int + n_mac - (n_lanes - root_lanes)));
        atomicAdd(&P.counters[1], (unsigned long long)(n_mac + 32u));
    }
}
