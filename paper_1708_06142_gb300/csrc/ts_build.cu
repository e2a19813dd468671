// Tree build (Sec. 2.1): cell masses and bottom-up FP64 node moments, one kernel.
//
// k_blocktree: one CTA of 512 threads per leaf-block.  Each thread reads one density value
// (coalesced, natural cell order), forms m = rho dV and the cell centre in FP64, and stores them
// in shared memory at the cell's Morton slot.  The 64 level-2 nodes, 8 level-1 nodes and the
// leaf-block node are then summed in shared memory, children in octant order, one thread per node
// and component (mass, and mass times each coordinate).  Products and sums use explicitly rounded
// FP64 operations (no FMA contraction), so masses and centres of mass are reproducible bit for bit by
// any implementation that sums in the same order.
// The amr-tree follows in the same launch: the CTA that completes the last of 8 sibling blocks (an
// atomic count per sibling group, put back to 0 by that CTA) sums their parent from the stored records
// and goes on to the parent's group.  No CTA waits for another, and each sum is over all 8 children in
// octant order whoever forms it.
// It also writes the FP32 records of every group of 8 siblings structure-of-arrays (x[8], y[8],
// z[8], m[8]) for the paired FP32 walk: cell group g = cells 8g..8g+7, node group g = nodes
// 1+8g..8+8g (node ids are breadth-first, so every child group starts at 1 mod 8).
// With the FP64 records switched off (ts_tree_fp64_records) the FP64 cell records and the FP64
// records of the nodes inside leaf-blocks are not written; those of the leaf-block and amr-tree
// nodes are (the amr sums read them).
//
// Roofline: bound by GB300's FP64 rate (1/64 of FP32; HBM-bound only once that arithmetic is
// cheap), and by latency on meshes of few blocks.  Per cell it reads 8 B of density and writes a 16 B
// FP32 record, its 16 B sibling-group copy and a 32 B FP64 record (none with the FP64 records off); per
// leaf-block 72 + 1 internal records of 16 + 16 + 32 B (16 + 16 B for the 72 with the FP64 records off).
// 2,097,152 cells, FP64 records off: 126 us and 40 us of a second kernel for the amr-tree before, 103 us so
// (one thread per component; the level-1 and leaf-block sums used 8 and 1 of 32 lanes); 32^3 cells: 23 us
// and 12.5 us.
#include <algorithm>

#include "ts_internal.cuh"

__device__ __forceinline__ int morton_of(int i, int j, int k) {
    // cell (i,j,k) in [0,8)^3 -> 64 q + 8 o + o2 with octant bits (x, y, z) at each level
    int q = (i >> 2) | ((j >> 2) << 1) | ((k >> 2) << 2);
    int o = ((i >> 1) & 1) | (((j >> 1) & 1) << 1) | (((k >> 1) & 1) << 2);
    int o2 = (i & 1) | ((j & 1) << 1) | ((k & 1) << 2);
    return 64 * q + 8 * o + o2;
}

// node nid >= 1 is sibling (nid - 1) % 8 of node group (nid - 1) / 8; the root belongs to none
__device__ __forceinline__ void store_soa(float* soa, int64_t g, int j, float x, float y, float z, float m) {
    float* q = soa + 32 * g + j;
    q[0] = x; q[8] = y; q[16] = z; q[24] = m;
}

// Component k (0: mass, 1..3: x, y, z) of a node's sums over its 8 children in octant order
__device__ __forceinline__ double mom_step(double a, int k, double m, double x) {
    return __dadd_rn(a, k ? __dmul_rn(m, x) : m);
}

// ... and of its record: the mass, or the centre of mass (of an empty node: the geometric centre)
__device__ __forceinline__ double mom_value(double a, int k, double m, const dbl4& cen) {
    if (k == 0) return m;
    if (m > 0) return __ddiv_rn(a, m);
    return k == 1 ? cen.x : k == 2 ? cen.y : cen.z;
}

// stores component k of node nid's records (mass last in each)
__device__ __forceinline__ void store_comp(float4* n32, dbl4* n64, float* soa, int nid, int k, double v, bool w64) {
    const int f = (k + 3) & 3;
    if (w64) ((double*)&n64[nid])[f] = v;
    ((float*)&n32[nid])[f] = (float)v;
    if (nid > 0) soa[32 * (int64_t)((nid - 1) >> 3) + 8 * f + ((nid - 1) & 7)] = (float)v;
}

struct AmrDev {
    const int* parent;   // [group] node id of the parent of sibling group g (nodes 1 + 8 g .. 8 + 8 g)
    unsigned* count;     // [group] blocks of the group completed in this build
};

__global__ void __launch_bounds__(512) k_blocktree(const double* __restrict__ rho, const double* __restrict__ leaf_lo,
                                                   const double* __restrict__ leaf_size, const int* __restrict__ leaf_nid,
                                                   const dbl4* __restrict__ ncen64, int nb, float4* __restrict__ cell32,
                                                   dbl4* __restrict__ cell64, float4* __restrict__ ncom32,
                                                   dbl4* ncom64, float* __restrict__ cellsoa,
                                                   float* __restrict__ ncomsoa, int full64, AmrDev amr) {
    // [component: m, x, y, z][cell or node], padded by one per 8 so that the threads that each sum 8
    // consecutive entries hit different banks
    __shared__ double sc[4][576], l2[4][72], l1[4][8];
    __shared__ double s_cc[3][8], s_dv;
    const int n = blockIdx.x, t = threadIdx.x;
    const int i = t & 7, j = (t >> 3) & 7, k = t >> 6;
    // The 8 cell-centre coordinates per axis and the cell volume, computed once per leaf-block (the
    // kernel is bound by GB300's FP64 rate).  x / 8 and x * 0.125 are the same exact scaling by a
    // power of two, so the results are bit-identical to lo + (i + 1/2) e / 8 and (e/8)^3.
    const double r0 = rho[(size_t)n * TS_NCB + t];
    if (t < 24) {
        const int a = t >> 3, c = t & 7;
        s_cc[a][c] = __dadd_rn(leaf_lo[3 * n + a], __dmul_rn(__dmul_rn(c + 0.5, leaf_size[3 * n + a]), 0.125));
    } else if (t == 32) {
        const double ex = leaf_size[3 * n], ey = leaf_size[3 * n + 1], ez = leaf_size[3 * n + 2];
        s_dv = __dmul_rn(__dmul_rn(__dmul_rn(ex, 0.125), __dmul_rn(ey, 0.125)), __dmul_rn(ez, 0.125));
    }
    __syncthreads();
    {
        const int mt = morton_of(i, j, k), at = mt + (mt >> 3);
        sc[0][at] = __dmul_rn(r0, s_dv);
        sc[1][at] = s_cc[0][i]; sc[2][at] = s_cc[1][j]; sc[3][at] = s_cc[2][k];
    }
    __syncthreads();
    const int base = nb + 72 * n;
    const int g2 = t & 63, k2 = t >> 6;   // level-2 node 8 q + o and component of this thread
    double a2 = 0;
    if (t < 256) {
#pragma unroll
        for (int c = 0; c < 8; ++c) a2 = mom_step(a2, k2, sc[0][9 * g2 + c], sc[k2][9 * g2 + c]);
        if (k2 == 0) l2[0][g2 + (g2 >> 3)] = a2;
    }
    // cell records in Morton order (coalesced)
    {
        const size_t id = (size_t)n * TS_NCB + t;
        const int at = t + (t >> 3);
        const double x = sc[1][at], y = sc[2][at], z = sc[3][at], m = sc[0][at];
        if (full64) cell64[id] = dbl4{x, y, z, m};
        cell32[id] = make_float4((float)x, (float)y, (float)z, (float)m);
        store_soa(cellsoa, (int64_t)(id >> 3), t & 7, (float)x, (float)y, (float)z, (float)m);
    }
    __syncthreads();
    if (t < 256) {
        const int nid = base + 8 + g2;
        const double v = mom_value(a2, k2, l2[0][g2 + (g2 >> 3)], ncen64[nid]);
        if (k2) l2[k2][g2 + (g2 >> 3)] = v;
        store_comp(ncom32, ncom64, ncomsoa, nid, k2, v, full64);
    }
    __syncthreads();
    if (t >= 32) return;
    // one warp from here on: lane 4 q + k takes component k of level-1 node q
    const int kk = t & 3, q = t >> 2;
    double a = 0;
#pragma unroll
    for (int c = 0; c < 8; ++c) a = mom_step(a, kk, l2[0][9 * q + c], l2[kk][9 * q + c]);
    double v = mom_value(a, kk, __shfl_sync(0xffffffffu, a, t & ~3), ncen64[base + q]);
    l1[kk][q] = v;
    store_comp(ncom32, ncom64, ncomsoa, base + q, kk, v, full64);
    __syncwarp();
    a = 0;   // the leaf-block node (every 4 lanes form it, lanes 0..3 store it)
#pragma unroll
    for (int c = 0; c < 8; ++c) a = mom_step(a, kk, l1[0][c], l1[kk][c]);
    int nid = leaf_nid[n];
    v = mom_value(a, kk, __shfl_sync(0xffffffffu, a, t & ~3), ncen64[nid]);
    if (t < 4) store_comp(ncom32, ncom64, ncomsoa, nid, kk, v, true);
    // amr ancestors completed by this block
    while (nid > 0) {
        const int g = (nid - 1) >> 3;
        __syncwarp();
        int done = 0;
        if (t == 0) {
            // the barrier orders lanes 0..3's stores before this lane's fence, and the fence before its count
            __threadfence();
            done = (int)atomicInc(&amr.count[g], 7u);   // (the last arrival puts it back to 0 for the next build)
            __threadfence();   // ... and orders the other blocks' stores, seen by its count, before the warp's loads
        }
        if (__shfl_sync(0xffffffffu, done, 0) != 7) return;
        __syncwarp();
        const double* ch = (const double*)&ncom64[1 + 8 * g];   // the 8 siblings' records (x, y, z, m)
        double m[8], x[8];
#pragma unroll
        for (int c = 0; c < 8; ++c) {   // (through L2: other CTAs wrote them)
            m[c] = __ldcg(ch + 4 * c + 3);
            x[c] = __ldcg(ch + 4 * c + ((kk + 3) & 3));
        }
        a = 0;
#pragma unroll
        for (int c = 0; c < 8; ++c) a = mom_step(a, kk, m[c], x[c]);
        nid = amr.parent[g];
        v = mom_value(a, kk, __shfl_sync(0xffffffffu, a, t & ~3), ncen64[nid]);
        if (t < 4) store_comp(ncom32, ncom64, ncomsoa, nid, kk, v, true);
    }
}

cudaError_t launch_tree_build(ts_ctx* c, const double* density) {
    k_blocktree<<<c->nleaf, 512, 0, c->stream>>>(density, c->d_leaf_lo, c->d_leaf_size, c->d_leaf_nid, c->d_ncen64,
                                                 c->nb, c->d_cell32, c->d_cell64, c->d_ncom32, c->d_ncom64,
                                                 (float*)c->d_cellsoa, (float*)c->d_ncomsoa, c->rec64 ? 1 : 0,
                                                 AmrDev{c->d_amr_parent, (unsigned*)c->d_amr_count});
    return cudaGetLastError();
}

// ------------------------------------------------------------------------------ MPE moments
// B_p = sum_i m_i |r_i - r_a|^p (p = 2, 3) over the cells of a node (Sec. 2.2.1, eq. mpe).
// One CTA per leaf-block: each thread holds one cell (Morton order) and adds its terms about the
// centre of mass of each of its ancestors: its level-2 node (8 consecutive threads), level-1 node
// (64), the leaf-block node (512, stored) and every amr ancestor (512 per leaf-block, FP64 atomics
// onto zeroed accumulators).  R is the arithmetic of the terms and of the sums within the CTA:
// double for the FP64 walk; float for the FP32 walk, whose MAC compares the moments in FP32 anyway
// (the FP64 pipe runs at 1/64 of the FP32 rate, and these terms need an FP64 square root each).
template <typename R> struct BM;
template <> struct BM<double> { typedef dbl4 V; typedef double2 P; };
template <> struct BM<float> { typedef float4 V; typedef float2 P; };

__device__ __forceinline__ double2 bterm(const dbl4& cell, const dbl4& ra) {
    const double dx = __dsub_rn(cell.x, ra.x), dy = __dsub_rn(cell.y, ra.y), dz = __dsub_rn(cell.z, ra.z);
    const double u = __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz));
    const double b2 = __dmul_rn(cell.w, u);
    return make_double2(b2, __dmul_rn(b2, sqrt(u)));
}

__device__ __forceinline__ float2 bterm(const float4& cell, const float4& ra) {
    const float dx = cell.x - ra.x, dy = cell.y - ra.y, dz = cell.z - ra.z;
    const float u = fmaf(dz, dz, fmaf(dy, dy, dx * dx));
    const float b2 = cell.w * u;
    return make_float2(b2, b2 * sqrtf(u));
}

template <typename P>
__device__ __forceinline__ P warp_sum2(P v, int width) {
    for (int o = width / 2; o; o >>= 1) {
        v.x += __shfl_xor_sync(0xffffffffu, v.x, o);
        v.y += __shfl_xor_sync(0xffffffffu, v.y, o);
    }
    return v;
}

// block-wide sum of 512 threads (16 warps), valid in thread 0; every thread must call it
template <typename P>
__device__ P block_sum2(P v, P* sm) {
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    v = warp_sum2(v, 32);
    __syncthreads();
    if (l == 0) sm[w] = v;
    __syncthreads();
    if (w == 0) {
        v = l < 16 ? sm[l] : P{0, 0};
        v = warp_sum2(v, 16);
    }
    return v;
}

template <typename R>
__global__ void __launch_bounds__(512) k_bmoments(const typename BM<R>::V* __restrict__ cell,
                                                  const typename BM<R>::V* __restrict__ ncom,
                                                  const int* __restrict__ leaf_nid, const int* __restrict__ anc,
                                                  int anc_max, int nb, double2* __restrict__ bm) {
    typedef typename BM<R>::P P;
    __shared__ P sm[16];
    __shared__ P l1[8][2];
    const int n = blockIdx.x, t = threadIdx.x;
    const typename BM<R>::V c = cell[(size_t)n * TS_NCB + t];
    const int base = nb + 72 * n;
    // level-2 node g = t / 8
    P v = warp_sum2(bterm(c, ncom[base + 8 + (t >> 3)]), 8);
    if ((t & 7) == 0) bm[base + 8 + (t >> 3)] = make_double2(v.x, v.y);
    // level-1 node q = t / 64: two warps
    v = warp_sum2(bterm(c, ncom[base + (t >> 6)]), 32);
    if ((t & 31) == 0) l1[t >> 6][(t >> 5) & 1] = v;
    __syncthreads();
    if (t < 8) bm[base + t] = make_double2((double)l1[t][0].x + (double)l1[t][1].x, (double)l1[t][0].y + (double)l1[t][1].y);
    // the leaf-block node
    const int leaf = leaf_nid[n];
    v = block_sum2(bterm(c, ncom[leaf]), sm);
    if (t == 0) bm[leaf] = make_double2(v.x, v.y);
    // amr ancestors
    for (int a = 0; a < anc_max; ++a) {
        const int id = anc[(size_t)n * anc_max + a];
        if (id < 0) break;   // uniform across the CTA
        v = block_sum2(bterm(c, ncom[id]), sm);
        if (t == 0) {
            atomicAdd(&bm[id].x, (double)v.x);
            atomicAdd(&bm[id].y, (double)v.y);
        }
    }
}

__global__ void k_bmoments_f32(const double2* __restrict__ bm, int nint, float2* __restrict__ out) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < nint; i += gridDim.x * blockDim.x)
        out[i] = make_float2((float)bm[i].x, (float)bm[i].y);
}

cudaError_t launch_bmoments(ts_ctx* c, bool fp64) {
    cudaError_t e = cudaMemsetAsync(c->d_bmom64, 0, sizeof(double2) * c->nb, c->stream);   // amr accumulators
    if (e != cudaSuccess) return e;
    if (fp64)
        k_bmoments<double><<<c->nleaf, 512, 0, c->stream>>>(c->d_cell64, c->d_ncom64, c->d_leaf_nid, c->d_leaf_anc,
                                                            c->anc_max, c->nb, c->d_bmom64);
    else
        k_bmoments<float><<<c->nleaf, 512, 0, c->stream>>>(c->d_cell32, c->d_ncom32, c->d_leaf_nid, c->d_leaf_anc,
                                                           c->anc_max, c->nb, c->d_bmom64);
    k_bmoments_f32<<<std::min((c->nint + 255) / 256, 152 * 8), 256, 0, c->stream>>>(c->d_bmom64, c->nint, c->d_bmom32);
    return cudaGetLastError();
}
