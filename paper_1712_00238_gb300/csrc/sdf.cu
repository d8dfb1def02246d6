// Skeletal density function of a solid from oriented boundary samples (Section 4).
//
// Pass 1 (per query point p_i): |xi| = min_j ||p_i - q_j|| (Eq. 10A; ties go to the
// lowest j, which does not change the value) and the generalised winding number
// w = sum_j a_j (q_j - p).n_j / (S ||q_j - p||^d), S = 2 pi (2D) or 4 pi (3D); the
// point is inside (pmc = -1) when w > 1/2, a membership derived from the
// consistent outward orientation of the samples.
// Pass 2: rho(p_i) = sum_j phi(zeta_ij) cos(theta_ij) a_j (Eq. 13 as a midpoint
// sum) with zeta = xi + i eta (Eq. 11), cos(theta) = (p - q).n / eta (Eq. 12a),
// phi = lambda / sqrt(2 pi) zeta^-2 g_sigma(eta/|xi| - 1) (Eq. 15),
// lambda = +lambda1 outside / -lambda2 inside (Eq. 16c), and only samples with
// eta/|xi| - 1 <= eps (Eq. 17t).  In 2D every element is weighted by its planar
// angle over 2 pi, i.e. the 3D summand times 2 eta.
// Over all pairs, both stage boundary tiles in shared memory; one query point per thread.
// A block of queries may split its boundary tiles across several CTAs (grid
// y), each writing a partial (nearest distance and winding sum; rho); a
// finishing kernel combines the partials in a fixed order, so the results do
// not depend on how many CTAs shared the work's scheduling.
// In 3D both passes walk the boundary as a two-level tree instead (256-sample tiles
// of 32-sample sub-tiles, the Morton order's own hierarchy): see k_sdf_tree; small
// builds' distances and memberships take all pairs (sdf_tree_pays).
#include <float.h>
#include <math.h>

#include <algorithm>

#include "kernels.cuh"

namespace sd {

// Queries are processed in Morton order (perm_q) and the boundary samples are
// pre-sorted the same way, so a CTA's 256 queries and a tile's 256 samples are
// each spatially compact.  Pass 2 skips every tile whose bounding box lies
// farther than (1 + eps) max|xi| from the CTA's box: all its pairs would fail
// the truncation test of Eq. 17t anyway (the restriction to eps-approximate
// nearest neighbours of Section 4), so the sum is unchanged.

template <typename T>
__device__ __forceinline__ T recip(T x) { return T(1) / x; }
template <>
__device__ __forceinline__ float recip<float>(float x) { return __frcp_rn(x); }

// Every pair: 2D, and 3D builds too small for the tree (sdf_tree_pays).
template <typename T, int D>
__global__ void __launch_bounds__(SDF_TILE) k_sdf_nearest(SdfArgs<T> a, int tiles_per_split, T* part_d2, T* part_w) {
    __shared__ vec4<T> sq[SDF_TILE];
    __shared__ vec4<T> sn[SDF_TILE];  // normal with the area in .w
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const bool live = i < a.m;
    const int64_t src = live ? (a.perm_q ? (int64_t)a.perm_q[i] : i) : 0;
    vec4<T> p;
    if (live) p = a.qry[src];
    else { p.x = p.y = p.z = p.w = T(0); }
    T dmin = INFINITY;
    T wind = T(0);
    const int64_t t_lo = (int64_t)blockIdx.y * tiles_per_split * SDF_TILE;
    const int64_t t_hi = min(a.n_b, t_lo + (int64_t)tiles_per_split * SDF_TILE);
    for (int64_t t0 = t_lo; t0 < t_hi; t0 += SDF_TILE) {
        const int64_t j = t0 + threadIdx.x;
        if (j < a.n_b) {
            sq[threadIdx.x] = a.bnd[j];
            sn[threadIdx.x] = a.nrm[j];
        }
        __syncthreads();
        const int cnt = live ? (int)min((int64_t)SDF_TILE, a.n_b - t0) : 0;
        for (int k = 0; k < cnt; ++k) {
            const vec4<T> q = sq[k];
            const vec4<T> nn = sn[k];
            const T dx = q.x - p.x, dy = q.y - p.y, dz = D == 3 ? q.z - p.z : T(0);
            const T d2 = dx * dx + dy * dy + dz * dz;
            dmin = d2 < dmin ? d2 : dmin;
            const T dot = dx * nn.x + dy * nn.y + dz * nn.z;
            if (D == 3) {
                const T r = rsqrt(d2);
                wind += nn.w * dot * r * r * r;
            } else {
                wind += nn.w * dot * recip(d2);
            }
        }
        __syncthreads();
    }
    if (!live) return;
    part_d2[(int64_t)blockIdx.y * a.m + i] = dmin;
    part_w[(int64_t)blockIdx.y * a.m + i] = wind;
}

// Nearest distance (the smallest partial) and membership (the partial winding
// sums added in split order) of each query.
template <typename T, int D>
__global__ void k_sdf_nearest_finish(SdfArgs<T> a, int splits, const T* part_d2, const T* part_w) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= a.m) return;
    T dmin = INFINITY, wind = T(0);
    for (int k = 0; k < splits; ++k) {
        const T d = part_d2[(int64_t)k * a.m + i];
        dmin = d < dmin ? d : dmin;
        wind += part_w[(int64_t)k * a.m + i];
    }
    const T S = D == 3 ? T(4.0 * M_PI) : T(2.0 * M_PI);
    a.xi_abs[i] = sqrt(dmin);
    int8_t m = (wind > T(0.5) * S) ? int8_t(-1) : int8_t(1);
    if (a.pmc_override) {
        const int64_t src = a.perm_q ? (int64_t)a.perm_q[i] : i;
        m = a.pmc_override[src] < 0 ? int8_t(-1) : int8_t(1);
    }
    a.pmc[i] = m;
}

// ---------------------------------------------------------------------------
// 3D: nearest distance and membership over the two-level boundary tree
// ---------------------------------------------------------------------------
//
// Over all pairs both are O(m n_b) (5,000 spheres: 6.4e10 pairs, 45.7 ms, issue
// bound).  The tree leaves a query a few hundred pairs:
//   nearest    a tile or sub-tile whose box is farther from the warp's 32 queries than
//              every lane's nearest so far holds no nearer sample: the minimum over
//              the rest is the minimum over all;
//   membership the sign of w - S/2.  A node seen from R = c - p, |R| >= beta rho (c its
//              centre, rho the radius of its samples about c), contributes
//              sum_j N_j.(R + d_j) / |R + d_j|^3, N_j = a_j n_j, expanded in d_j to second
//              order.  The term of order k of the gradient of 1/|R + d| is at most
//              (k + 1) |d|^k / |R|^(k+2), so what is dropped is at most
//              sum_{k>=3} (k+1) sum_j |N_j| |d_j|^k / |R|^(k+2) <= g(1/beta) B3 / |R|^5,
//              B3 = sum_j |N_j| |d_j|^3, g(x) = 4/(1-x) + x/(1-x)^2.
//              The bounds add up to E; a query with |w - S/2| <= E (plus a margin for
//              rounding, 0.01 S + 1e-4 of the summed solid angles) is summed again over
//              every sample (k_sdf_wind_list), so the membership is that of the full
//              sum.  Closed solids sampled at their own resolution sit near w = 0 or S:
//              E stays below 0.6 of S/2 at beta = 2.5 on the sphere packings and
//              below 0.15 on the cylinder, and no query was left over.
constexpr int NODE = 28;  // centre (3), rho | N (3), A | M sym (6), B3, V_x | V_y, V_z, cubic (10)
constexpr float TREE_BETA = 2.5f;

// Moments of every tile and sub-tile about their box centres (one CTA per tile;
// nodes: n_tiles of tiles, then n_tiles * SDF_TILE / 32 of sub-tiles; rho < 0: empty).
template <typename T>
__device__ __forceinline__ void node_terms(T* v, const T d[3], const T N[3]) {
    const T A = sqrt(N[0] * N[0] + N[1] * N[1] + N[2] * N[2]);
    const T d2 = d[0] * d[0] + d[1] * d[1] + d[2] * d[2];
    const T xx = d[0] * d[0], yy = d[1] * d[1], zz = d[2] * d[2], xy = d[0] * d[1], xz = d[0] * d[2], yz = d[1] * d[2];
    const T nd = N[0] * d[0] + N[1] * d[1] + N[2] * d[2];
    v[0] = N[0]; v[1] = N[1]; v[2] = N[2]; v[3] = A;
    v[4] = N[0] * d[0]; v[5] = N[1] * d[1]; v[6] = N[2] * d[2];
    v[7] = N[0] * d[1] + N[1] * d[0]; v[8] = N[0] * d[2] + N[2] * d[0]; v[9] = N[1] * d[2] + N[2] * d[1];
    v[10] = A * d2 * sqrt(d2);
    // V_c = 2 sum_a T_a,ac + sum_b T_c,bb with T_a,bc = N_a d_b d_c
    v[11] = T(2) * nd * d[0] + N[0] * d2;
    v[12] = T(2) * nd * d[1] + N[1] * d2;
    v[13] = T(2) * nd * d[2] + N[2] * d2;
    // T_a,bc R_a R_b R_c by monomial: xxx xxy xxz yyx yyy yyz zzx zzy zzz xyz
    v[14] = N[0] * xx; v[15] = N[1] * xx + T(2) * N[0] * xy; v[16] = N[2] * xx + T(2) * N[0] * xz;
    v[17] = N[0] * yy + T(2) * N[1] * xy; v[18] = N[1] * yy; v[19] = N[2] * yy + T(2) * N[1] * yz;
    v[20] = N[0] * zz + T(2) * N[2] * xz; v[21] = N[1] * zz + T(2) * N[2] * yz; v[22] = N[2] * zz;
    v[23] = T(2) * (N[0] * yz + N[1] * xz + N[2] * xy);
}

// FP32 samples by twos for the paired instructions of the tree's direct sums: x0 x1
// y0 y1 | z0 z1 Nx0 Nx1 | Ny0 Ny1 Nz0 Nz1, N = area times normal.  A pair past the end
// repeats its last sample with N = 0.
constexpr int PAIR = 12;

template <typename T>
__global__ void __launch_bounds__(SDF_TILE) k_sdf_nodes(const vec4<T>* bnd, const vec4<T>* nrm, int64_t n_b,
                                                        const float* tile_box, const float* sub_box, T* nodes,
                                                        int64_t n_tiles, float* pairs) {
    constexpr int NW = SDF_TILE / 32, NV = NODE - 4;
    __shared__ T part[NW][NV + 1];
    const int64_t i = (int64_t)blockIdx.x * SDF_TILE + threadIdx.x;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const bool live = i < n_b;
    vec4<T> q, nn;
    q.x = q.y = q.z = nn.x = nn.y = nn.z = nn.w = T(0);
    if (live) {
        q = bnd[i];
        nn = nrm[i];
    }
    const T N[3] = {nn.x * nn.w, nn.y * nn.w, nn.z * nn.w};
    if constexpr (sizeof(T) == 4) {
        if (i < (n_b + 1) / 2 * 2) {
            const float4 pos = live ? q : bnd[n_b - 1];
            float* w = pairs + (i >> 1) * PAIR + (i & 1);
            w[0] = pos.x; w[2] = pos.y; w[4] = pos.z;
            w[6] = N[0]; w[8] = N[1]; w[10] = N[2];
        }
    }
    for (int level = 0; level < 2; ++level) {
        const float* box = level ? sub_box + ((int64_t)blockIdx.x * NW + warp) * 6 : tile_box + (int64_t)blockIdx.x * 6;
        T c[3], d[3], v[NV], rho = T(0);
        for (int k = 0; k < 3; ++k) c[k] = box[k] <= box[3 + k] ? T(0.5f * (box[k] + box[3 + k])) : T(0);
        if (live) {
            d[0] = q.x - c[0]; d[1] = q.y - c[1]; d[2] = q.z - c[2];
            node_terms<T>(v, d, N);
            rho = sqrt(d[0] * d[0] + d[1] * d[1] + d[2] * d[2]);
        } else {
            for (int k = 0; k < NV; ++k) v[k] = T(0);
        }
        for (int off = 16; off > 0; off >>= 1) {
            for (int k = 0; k < NV; ++k) v[k] += __shfl_down_sync(0xffffffffu, v[k], off);
            const T o = __shfl_down_sync(0xffffffffu, rho, off);
            rho = o > rho ? o : rho;
        }
        const bool empty = level && !__any_sync(0xffffffffu, live);
        if (level) {
            T* nd = nodes + (n_tiles + (int64_t)blockIdx.x * NW + warp) * NODE;
            if (lane == 0) {
                nd[0] = c[0]; nd[1] = c[1]; nd[2] = c[2];
                nd[3] = empty ? T(-1) : rho * T(1.00001);
                for (int k = 0; k < NV; ++k) nd[4 + k] = v[k];
            }
        } else {
            if (lane == 0) {
                for (int k = 0; k < NV; ++k) part[warp][k] = v[k];
                part[warp][NV] = rho;
            }
            __syncthreads();
            T* nd = nodes + (int64_t)blockIdx.x * NODE;
            if (threadIdx.x <= NV) {
                T r = part[0][threadIdx.x];
                for (int w = 1; w < NW; ++w) {
                    const T o = part[w][threadIdx.x];
                    r = threadIdx.x < NV ? r + o : (o > r ? o : r);
                }
                nd[threadIdx.x < NV ? 4 + threadIdx.x : 3] = threadIdx.x < NV ? r : r * T(1.00001);
            }
            if (threadIdx.x < 3) nd[threadIdx.x] = c[threadIdx.x];
        }
    }
}

__device__ __forceinline__ float4 load4(const float* p) { return __ldg(reinterpret_cast<const float4*>(p)); }
__device__ __forceinline__ double4_32a load4(const double* p) { return *reinterpret_cast<const double4_32a*>(p); }
__device__ __forceinline__ float4 sample4(const float4* p) { return __ldg(p); }
__device__ __forceinline__ double4_32a sample4(const double4_32a* p) { return *p; }

// Reciprocal square root; a denormal squared distance (coinciding points) counts as zero.
__device__ __forceinline__ float rsqrt_(float x) {
    float r;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ double rsqrt_(double x) { return rsqrt(x); }

// A far node's winding sum at the lane's Q points, its dropped part's bound (over g)
// and its solid angle's magnitude.
template <typename T, int Q>
__device__ __forceinline__ void node_eval(const T* nd, const vec4<T> (&p)[Q], T (&wind)[Q], T (&err)[Q], T (&mag)[Q]) {
    const vec4<T> n0 = load4(nd), n1 = load4(nd + 4), n2 = load4(nd + 8), n3 = load4(nd + 12), n4 = load4(nd + 16),
                  n5 = load4(nd + 20), n6 = load4(nd + 24);
    const T tr = n2.x + n2.y + n2.z;
#pragma unroll
    for (int q = 0; q < Q; ++q) {
        const T x = n0.x - p[q].x, y = n0.y - p[q].y, z = n0.z - p[q].z;
        const T xx = x * x, yy = y * y, zz = z * z, xy = x * y;
        const T ri = rsqrt_(xx + yy + zz);
        const T r2 = ri * ri, r3 = r2 * ri, r5 = r3 * r2;
        const T M = n2.x * xx + n2.y * yy + n2.z * zz + n2.w * xy + z * (n3.x * x + n3.y * y);
        const T VR = n3.w * x + n4.x * y + n4.y * z;
        const T C = xx * (n4.z * x + n4.w * y + n5.x * z) + yy * (n5.y * x + n5.z * y + n5.w * z) +
                    zz * (n6.x * x + n6.y * y + n6.z * z) + xy * z * n6.w;
        wind[q] += r3 * (n1.x * x + n1.y * y + n1.z * z + tr) + r5 * (T(7.5) * r2 * C - T(3) * M - T(1.5) * VR);
        err[q] += n3.z * r5;
        mag[q] += n1.w * r2;
    }
}

// The warp's box of query points (lo[3], hi[3]), in float, widened for the rounding.
template <typename T, int Q>
__device__ __forceinline__ void warp_box(const vec4<T> (&p)[Q], float lo[3], float hi[3]) {
    for (int d = 0; d < 3; ++d) {
        lo[d] = INFINITY;
        hi[d] = -INFINITY;
        for (int q = 0; q < Q; ++q) {
            const float v = (float)(d == 0 ? p[q].x : (d == 1 ? p[q].y : p[q].z));
            lo[d] = fminf(lo[d], v);
            hi[d] = fmaxf(hi[d], v);
        }
        for (int off = 16; off > 0; off >>= 1) {
            lo[d] = fminf(lo[d], __shfl_xor_sync(0xffffffffu, lo[d], off));
            hi[d] = fmaxf(hi[d], __shfl_xor_sync(0xffffffffu, hi[d], off));
        }
        lo[d] -= 1e-6f * (fabsf(lo[d]) + 1.f);
        hi[d] += 1e-6f * (fabsf(hi[d]) + 1.f);
    }
}
// Squared distance between two boxes (b: lo[3], hi[3]).
__device__ __forceinline__ float box_gap2(const float* b, const float lo[3], const float hi[3]) {
    float g2 = 0.f;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        const float g = fmaxf(0.f, fmaxf(b[d] - hi[d], lo[d] - b[3 + d]));
        g2 = fmaf(g, g, g2);
    }
    return g2;
}
// The same from one point: a warp whose 32 queries straddle a fold of the Morton
// curve has a box full of nothing, so what its box lets through is put to a vote.
template <typename T>
__device__ __forceinline__ float point_gap2(const float* b, const vec4<T>& p) {
    const float v[3] = {(float)p.x, (float)p.y, (float)p.z};
    float g2 = 0.f;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        const float m = 1e-6f * (fabsf(v[d]) + 1.f);
        const float g = fmaxf(0.f, fmaxf(b[d] - v[d], v[d] - b[3 + d]) - m);
        g2 = fmaf(g, g, g2);
    }
    return g2;
}
// Whether a node is far enough from every point of the box for its expansion.
template <typename T>
__device__ __forceinline__ bool node_far(const T* nd, const float lo[3], const float hi[3]) {
    float g2 = 0.f;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        const float c = (float)nd[d];
        const float g = fmaxf(0.f, fmaxf(c - hi[d], lo[d] - c));
        g2 = fmaf(g, g, g2);
    }
    const float need = TREE_BETA * (float)nd[3];
    return g2 >= need * need * 1.0001f;
}

// One CTA per 32 Q Morton-consecutive queries (Q per lane of each of its 8 warps).
// Lanes test 32 tiles at a time; the warps share the far tiles, and each takes one
// of a near tile's 8 sub-tiles, so they finish together.  Nodes and samples are
// broadcast loads, four wavefronts per 16 bytes: the L1 data pipe is what bounds the
// kernel (88 % at one query a lane), and two queries a lane halve them.  FP32 samples
// are read and evaluated by twos (pairs) with paired instructions.  5,000 spheres
// (199,433 queries, 320,000 samples): 3.0 ms, issuing on 70 % of cycles; the
// cylinder (50,342, 20,000) 0.17 ms.
constexpr int TREE_NW = 8;
// Two queries a lane where that still gives every SM two CTAs.
constexpr int64_t TREE_PAIR_MIN = 64 * 2 * GPU_SMS;

template <typename T, int Q>
__global__ void __launch_bounds__(32 * TREE_NW, sizeof(T) == 4 ? 4 : 0) k_sdf_tree(SdfArgs<T> a, const T* nodes, const float* tile_box,
                                                           const float* sub_box, const float* pairs, int* list,
                                                           int* list_n) {
    constexpr int SUB = SDF_TILE / 32;
    static_assert(SUB == TREE_NW, "a tile's sub-tiles go to the warps");
    __shared__ T sh[3][TREE_NW][32 * Q];
    __shared__ float best_gap[TREE_NW];
    __shared__ int best_tile[TREE_NW];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t i0 = (int64_t)blockIdx.x * (32 * Q) + lane;
    vec4<T> p[Q];
#pragma unroll
    for (int q = 0; q < Q; ++q) {
        const int64_t i = min(i0 + 32 * q, a.m - 1);  // the last group's spare places repeat a query
        p[q] = a.qry[a.perm_q ? (int64_t)a.perm_q[i] : i];
    }
    const int n_tiles = (int)a.n_tiles;
    float lo[3], hi[3];
    warp_box<T, Q>(p, lo, hi);

    // nearest sample: a first bound from the nearest tile
    float gap = INFINITY;
    int tile0 = 0;
    for (int t = threadIdx.x; t < n_tiles; t += 32 * TREE_NW) {
        const float g = box_gap2(tile_box + (int64_t)t * 6, lo, hi);
        if (g < gap) { gap = g; tile0 = t; }
    }
    for (int off = 16; off > 0; off >>= 1) {
        const float g = __shfl_xor_sync(0xffffffffu, gap, off);
        const int o = __shfl_xor_sync(0xffffffffu, tile0, off);
        if (g < gap || (g == gap && o < tile0)) { gap = g; tile0 = o; }
    }
    if (lane == 0) { best_gap[warp] = gap; best_tile[warp] = tile0; }
    __syncthreads();
    gap = best_gap[0];
    tile0 = best_tile[0];
    for (int w = 1; w < TREE_NW; ++w)
        if (best_gap[w] < gap) { gap = best_gap[w]; tile0 = best_tile[w]; }
    T dmin[Q];
#pragma unroll
    for (int q = 0; q < Q; ++q) dmin[q] = INFINITY;
    float2 nx[Q], ny[Q], nz[Q];  // FP32: the negated points, doubled
#pragma unroll
    for (int q = 0; q < Q; ++q) {
        nx[q] = make_float2(-(float)p[q].x, -(float)p[q].x);
        ny[q] = make_float2(-(float)p[q].y, -(float)p[q].y);
        nz[q] = make_float2(-(float)p[q].z, -(float)p[q].z);
    }
    auto scan_sub = [&](int64_t j0) {  // the samples of one sub-tile
        const int cnt = (int)min((int64_t)32, a.n_b - j0);
        if constexpr (sizeof(T) == 4) {
            const float* b = pairs + (j0 >> 1) * PAIR;
#pragma unroll 4
            for (int k = 0; k < cnt; k += 2, b += PAIR) {
                const float4 u = load4(b);
                const float2 z = __ldg(reinterpret_cast<const float2*>(b + 4));
#pragma unroll
                for (int q = 0; q < Q; ++q) {
                    const float2 dx = __fadd2_rn(make_float2(u.x, u.y), nx[q]), dy = __fadd2_rn(make_float2(u.z, u.w), ny[q]),
                                 dz = __fadd2_rn(z, nz[q]);
                    const float2 d2 = __ffma2_rn(dz, dz, __ffma2_rn(dy, dy, __fmul2_rn(dx, dx)));
                    dmin[q] = fminf(dmin[q], fminf(d2.x, d2.y));
                }
            }
            return;
        }
        const vec4<T>* b = a.bnd + j0;
#pragma unroll 4
        for (int k = 0; k < cnt; ++k) {
            const vec4<T> s = sample4(b + k);
#pragma unroll
            for (int q = 0; q < Q; ++q) {
                const T dx = s.x - p[q].x, dy = s.y - p[q].y, dz = s.z - p[q].z;
                const T d2 = dx * dx + dy * dy + dz * dz;
                dmin[q] = d2 < dmin[q] ? d2 : dmin[q];
            }
        }
    };
    scan_sub((int64_t)tile0 * SDF_TILE + warp * 32);
#pragma unroll
    for (int q = 0; q < Q; ++q) sh[0][warp][lane + 32 * q] = dmin[q];
    __syncthreads();
#pragma unroll
    for (int q = 0; q < Q; ++q)
        for (int w = 0; w < TREE_NW; ++w) {
            const T o = sh[0][w][lane + 32 * q];
            dmin[q] = o < dmin[q] ? o : dmin[q];
        }
    // each query's nearest so far, with room for the rounding of the gaps, against a box
    auto beyond = [&](const float* box) {
        bool far = true;
#pragma unroll
        for (int q = 0; q < Q; ++q) far &= point_gap2<T>(box, p[q]) > (float)dmin[q] * 1.00001f + 1e-30f;
        return __all_sync(0xffffffffu, far);
    };
    float ub = 0.f;
#pragma unroll
    for (int q = 0; q < Q; ++q) ub = fmaxf(ub, (float)dmin[q] * 1.00001f + 1e-30f);
    for (int off = 16; off > 0; off >>= 1) ub = fmaxf(ub, __shfl_xor_sync(0xffffffffu, ub, off));
    for (int base = 0; base < n_tiles; base += 32) {
        const int t = base + lane;
        unsigned m = __ballot_sync(0xffffffffu, t < n_tiles && t != tile0 &&
                                                    !(box_gap2(tile_box + (int64_t)t * 6, lo, hi) > ub));
        while (m) {
            const int tt = base + __ffs(m) - 1;
            m &= m - 1;
            if (!beyond(sub_box + ((int64_t)tt * SUB + warp) * 6)) scan_sub((int64_t)tt * SDF_TILE + warp * 32);
        }
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < Q; ++q) sh[0][warp][lane + 32 * q] = dmin[q];

    // winding sum
    T wind[Q], err[Q], mag[Q];
    float2 wind2[Q];
#pragma unroll
    for (int q = 0; q < Q; ++q) {
        wind[q] = err[q] = mag[q] = T(0);
        wind2[q] = make_float2(0.f, 0.f);
    }
    if (!a.pmc_override) {
        const T* subs = nodes + (int64_t)n_tiles * NODE;
        auto all_far = [&](const T* nd) {
            const vec4<T> c = load4(nd);
            const T need = T(TREE_BETA) * c.w;
            bool far = true;
#pragma unroll
            for (int q = 0; q < Q; ++q) {
                const T dx = c.x - p[q].x, dy = c.y - p[q].y, dz = c.z - p[q].z;
                far &= dx * dx + dy * dy + dz * dz >= need * need * T(1.0001);
            }
            return __all_sync(0xffffffffu, far);
        };
        for (int base = 0; base < n_tiles; base += 32) {
            const int t = base + lane;
            const bool in = t < n_tiles;
            const bool far = in && node_far<T>(nodes + (int64_t)(in ? t : 0) * NODE, lo, hi);
            // far tiles: dealt to the warps
            unsigned mf = __ballot_sync(0xffffffffu, far) & (0x01010101u << warp);
            unsigned mn = __ballot_sync(0xffffffffu, in && !far);
            while (mf) {
                const int tt = base + __ffs(mf) - 1;
                mf &= mf - 1;
                node_eval<T, Q>(nodes + (int64_t)tt * NODE, p, wind, err, mag);
            }
            while (mn) {
                const int tt = base + __ffs(mn) - 1;
                mn &= mn - 1;
                if (all_far(nodes + (int64_t)tt * NODE)) {  // the same in every warp
                    if ((tt & (TREE_NW - 1)) == warp) node_eval<T, Q>(nodes + (int64_t)tt * NODE, p, wind, err, mag);
                    continue;
                }
                const T* nd = subs + ((int64_t)tt * SUB + warp) * NODE;
                const int64_t j0 = (int64_t)tt * SDF_TILE + warp * 32;
                const int cnt = (int)min((int64_t)32, a.n_b - j0);
                if (cnt <= 0) continue;
                if (all_far(nd)) {
                    node_eval<T, Q>(nd, p, wind, err, mag);
                    continue;
                }
                if constexpr (sizeof(T) == 4) {
                    const float* b = pairs + (j0 >> 1) * PAIR;
#pragma unroll 2
                    for (int k = 0; k < cnt; k += 2, b += PAIR) {
                        const float4 u = load4(b), v = load4(b + 4), w = load4(b + 8);
#pragma unroll
                        for (int q = 0; q < Q; ++q) {
                            const float2 dx = __fadd2_rn(make_float2(u.x, u.y), nx[q]),
                                         dy = __fadd2_rn(make_float2(u.z, u.w), ny[q]),
                                         dz = __fadd2_rn(make_float2(v.x, v.y), nz[q]);
                            const float2 d2 = __ffma2_rn(dz, dz, __ffma2_rn(dy, dy, __fmul2_rn(dx, dx)));
                            const float2 r = make_float2(rsqrt_(d2.x), rsqrt_(d2.y));
                            const float2 dot = __ffma2_rn(dz, make_float2(w.z, w.w),
                                                          __ffma2_rn(dy, make_float2(w.x, w.y),
                                                                     __fmul2_rn(dx, make_float2(v.z, v.w))));
                            wind2[q] = __ffma2_rn(dot, __fmul2_rn(__fmul2_rn(r, r), r), wind2[q]);
                        }
                    }
                    continue;
                }
#pragma unroll 4
                for (int k = 0; k < cnt; ++k) {
                    const vec4<T> s = sample4(a.bnd + j0 + k), nn = sample4(a.nrm + j0 + k);
#pragma unroll
                    for (int q = 0; q < Q; ++q) {
                        const T dx = s.x - p[q].x, dy = s.y - p[q].y, dz = s.z - p[q].z;
                        const T r = rsqrt_(dx * dx + dy * dy + dz * dz);
                        wind[q] += nn.w * (dx * nn.x + dy * nn.y + dz * nn.z) * r * r * r;
                    }
                }
            }
        }
    }
    constexpr float X = 1.f / TREE_BETA;
    constexpr float G = 4.f / (1.f - X) + X / ((1.f - X) * (1.f - X));
    constexpr double S = 4.0 * M_PI;
#pragma unroll
    for (int q = 0; q < Q; ++q) {
        sh[1][warp][lane + 32 * q] = wind[q] + T(wind2[q].x + wind2[q].y);
        sh[2][warp][lane + 32 * q] = err[q] * T(G * 1.001f) + mag[q] * T(1e-4);
    }
    __syncthreads();
    const int64_t i = (int64_t)blockIdx.x * (32 * Q) + threadIdx.x;
    if (threadIdx.x < 32 * Q && i < a.m) {
        T d = INFINITY, e = T(0.01 * S), over = T(0);
        for (int w = 0; w < TREE_NW; ++w) {
            const T o = sh[0][w][threadIdx.x];
            d = o < d ? o : d;
            over += sh[1][w][threadIdx.x];
            e += sh[2][w][threadIdx.x];
        }
        a.xi_abs[i] = sqrt(d);
        if (a.pmc_override) {
            a.pmc[i] = a.pmc_override[a.perm_q ? (int64_t)a.perm_q[i] : i] < 0 ? int8_t(-1) : int8_t(1);
        } else {
            over -= T(0.5 * S);
            a.pmc[i] = over > T(0) ? int8_t(-1) : int8_t(1);
            if (!(fabs(over) > e)) list[atomicAdd(list_n, 1)] = (int)i;  // undecided (or not a number)
        }
    }
}

// Membership of the listed queries from the sum over every sample.  Work items
// (256 queries, a share of the tiles) are dealt to a fixed grid, so that a few
// queries against many samples still fill it; a warp adds a query's shares.
constexpr int LIST_CTAS = GPU_SMS * 8;
__host__ __device__ __forceinline__ int list_splits(int chunks, int64_t n_tiles) {
    const int s = LIST_CTAS / (chunks > 0 ? chunks : 1);
    return s < 1 ? 1 : (s > n_tiles ? (int)n_tiles : s);
}

template <typename T>
__global__ void __launch_bounds__(SDF_TILE) k_sdf_wind_list(SdfArgs<T> a, const int* list, const int* list_n, T* part) {
    __shared__ vec4<T> sq[SDF_TILE], sn[SDF_TILE];
    const int n = *list_n, chunks = (n + SDF_TILE - 1) / SDF_TILE;
    const int splits = list_splits(chunks, a.n_tiles);
    const int64_t per = (a.n_tiles + splits - 1) / splits;
    for (int item = blockIdx.x; item < chunks * splits; item += gridDim.x) {
        const int e = (item / splits) * SDF_TILE + (int)threadIdx.x, split = item % splits;
        vec4<T> p;
        p.x = p.y = p.z = T(0);
        if (e < n) p = a.qry[a.perm_q ? (int64_t)a.perm_q[list[e]] : list[e]];
        T wind = T(0);
        const int64_t t_hi = min(a.n_b, (split + 1) * per * SDF_TILE);
        for (int64_t t0 = split * per * SDF_TILE; t0 < t_hi; t0 += SDF_TILE) {
            const int64_t j = t0 + threadIdx.x;
            __syncthreads();
            if (j < a.n_b) {
                sq[threadIdx.x] = a.bnd[j];
                sn[threadIdx.x] = a.nrm[j];
            }
            __syncthreads();
            const int cnt = (int)min((int64_t)SDF_TILE, a.n_b - t0);
            for (int k = 0; k < cnt; ++k) {
                const vec4<T> q = sq[k], nn = sn[k];
                const T dx = q.x - p.x, dy = q.y - p.y, dz = q.z - p.z;
                const T r = rsqrt(dx * dx + dy * dy + dz * dz);
                wind += nn.w * (dx * nn.x + dy * nn.y + dz * nn.z) * r * r * r;
            }
        }
        if (e < n) part[(int64_t)split * chunks * SDF_TILE + e] = wind;
    }
}

template <typename T>
__global__ void __launch_bounds__(SDF_TILE) k_sdf_wind_list_finish(SdfArgs<T> a, const int* list, const int* list_n,
                                                                   const T* part) {
    const int n = *list_n, chunks = (n + SDF_TILE - 1) / SDF_TILE;
    const int splits = list_splits(chunks, a.n_tiles);
    const int lane = threadIdx.x & 31;
    for (int e = (blockIdx.x * SDF_TILE + (int)threadIdx.x) / 32; e < n; e += (int)gridDim.x * SDF_TILE / 32) {  // a warp each
        T wind = T(0);
        for (int k = lane; k < splits; k += 32) wind += part[(int64_t)k * chunks * SDF_TILE + e];
        for (int off = 16; off > 0; off >>= 1) wind += __shfl_down_sync(0xffffffffu, wind, off);
        if (lane == 0) a.pmc[list[e]] = wind > T(2.0 * M_PI) ? int8_t(-1) : int8_t(1);
    }
}

// Kahan-compensated accumulation
template <typename T>
__device__ __forceinline__ void kahan_add(T& s, T& c, T v) {
    const T y = v - c;
    const T t = s + y;
    c = (t - s) - y;
    s = t;
}

template <typename T, int D, int PHI>
__global__ void __launch_bounds__(SDF_TILE) k_sdf_sum(SdfArgs<T> a, int tiles_per_split, cplx<T>* part) {
    __shared__ vec4<T> sq[SDF_TILE];
    __shared__ vec4<T> sn[SDF_TILE];
    __shared__ float wred[SDF_TILE / 32][7];
    __shared__ float box[7];  // lo[3], hi[3], reach
    float wbox[7] = {0, 0, 0, 0, 0, 0, 0};  // the warp's lo[3], hi[3], reach
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const bool live = i < a.m;
    const int64_t src = live ? (a.perm_q ? (int64_t)a.perm_q[i] : i) : 0;
    vec4<T> p;
    T xabs = T(1), xi = T(1);
    if (live) {
        p = a.qry[src];
        xabs = a.xi_abs[i];
        xi = a.pmc[i] < 0 ? -xabs : xabs;
    } else {
        p.x = p.y = p.z = p.w = T(0);
    }
    // CTA box and cutoff radius (1 + eps) max|xi| for the tile test
    const bool cull = PHI == SD_PHI_SDF && a.tile_box != nullptr && a.eps >= T(0);
    if (cull) {
        float v[7] = {FLT_MAX, FLT_MAX, FLT_MAX, -FLT_MAX, -FLT_MAX, -FLT_MAX, 0.f};
        if (live) {
            v[0] = v[3] = (float)p.x;
            v[1] = v[4] = (float)p.y;
            v[2] = v[5] = (D == 3) ? (float)p.z : 0.f;
            v[6] = (float)xabs;
        }
        for (int off = 16; off > 0; off >>= 1) {
            for (int d = 0; d < 3; ++d) v[d] = fminf(v[d], __shfl_down_sync(0xffffffffu, v[d], off));
            for (int d = 3; d < 7; ++d) v[d] = fmaxf(v[d], __shfl_down_sync(0xffffffffu, v[d], off));
        }
        if ((threadIdx.x & 31) == 0)
            for (int d = 0; d < 7; ++d) wred[threadIdx.x >> 5][d] = v[d];
        // this warp's own box and reach, for the sub-tile test
        for (int d = 0; d < 7; ++d) wbox[d] = __shfl_sync(0xffffffffu, v[d], 0);
        wbox[6] = wbox[6] * (1.f + (float)a.eps) * (1.f + 1e-4f) + 1e-6f;
        __syncthreads();
        if (threadIdx.x < 7) {
            float r = wred[0][threadIdx.x];
            for (int w = 1; w < SDF_TILE / 32; ++w)
                r = threadIdx.x < 3 ? fminf(r, wred[w][threadIdx.x]) : fmaxf(r, wred[w][threadIdx.x]);
            if (threadIdx.x == 6) r = r * (1.f + (float)a.eps) * (1.f + 1e-4f) + 1e-6f;
            box[threadIdx.x] = r;
        }
        __syncthreads();
    }
    const T lam = xi > T(0) ? a.lam1 : -a.lam2;
    // SDF: lambda/sqrt(2 pi) * 1/(sqrt(2 pi) sigma); proximal: lambda/sqrt(2 pi);
    // radial: 1/(sqrt(2 pi) sigma), times lambda1 (real) outside or lambda2 (imaginary) inside
    const T pref = PHI == SD_PHI_SDF      ? lam / (T(2.0 * M_PI) * a.sigma)
                   : PHI == SD_PHI_PROXIMAL ? lam / sqrt(T(2.0 * M_PI))
                                            : T(1) / (sqrt(T(2.0 * M_PI)) * a.sigma);
    const T inv_r = recip(a.radius);
    const T inv_xabs = recip(xabs);
    const T inv_2s2 = recip(T(2) * a.sigma * a.sigma);
    const T xi2 = xi * xi;
    T sr = 0, cr = 0, si = 0, ci = 0;
    const int64_t tile_lo = (int64_t)blockIdx.y * tiles_per_split;
    const int64_t t_hi = min(a.n_b, (tile_lo + tiles_per_split) * SDF_TILE);
    for (int64_t t0 = tile_lo * SDF_TILE, tile = tile_lo; t0 < t_hi; t0 += SDF_TILE, ++tile) {
        if (cull) {
            const float* tb = a.tile_box + tile * 6;
            const float g0 = fmaxf(0.f, fmaxf(tb[0] - box[3], box[0] - tb[3]));
            const float g1 = fmaxf(0.f, fmaxf(tb[1] - box[4], box[1] - tb[4]));
            const float g2 = (D == 3) ? fmaxf(0.f, fmaxf(tb[2] - box[5], box[2] - tb[5])) : 0.f;
            if (g0 * g0 + g1 * g1 + g2 * g2 > box[6] * box[6]) continue;  // same in every thread
        }
        const int64_t j = t0 + threadIdx.x;
        __syncthreads();
        if (j < a.n_b) {
            sq[threadIdx.x] = a.bnd[j];
            sn[threadIdx.x] = a.nrm[j];
        }
        __syncthreads();
        const int cnt = (int)min((int64_t)SDF_TILE, a.n_b - t0);
        for (int k = 0; k < cnt; ++k) {
            if (cull && a.sub_box && (k & 31) == 0) {
                // skip the 32-sample sub-tile when it lies beyond this warp's reach
                const float* sb = a.sub_box + (tile * (SDF_TILE / 32) + (k >> 5)) * 6;
                const float g0 = fmaxf(0.f, fmaxf(sb[0] - wbox[3], wbox[0] - sb[3]));
                const float g1 = fmaxf(0.f, fmaxf(sb[1] - wbox[4], wbox[1] - sb[4]));
                const float g2 = (D == 3) ? fmaxf(0.f, fmaxf(sb[2] - wbox[5], wbox[2] - sb[5])) : 0.f;
                if (g0 * g0 + g1 * g1 + g2 * g2 > wbox[6] * wbox[6]) {  // same in every lane of the warp
                    k += 31;
                    continue;
                }
            }
            const vec4<T> q = sq[k];
            const T dx = p.x - q.x, dy = p.y - q.y, dz = (D == 3) ? p.z - q.z : T(0);
            const T d2 = dx * dx + dy * dy + dz * dz;
            const T eta = sqrt(d2);
            const vec4<T> nn = sn[k];
            if constexpr (PHI == SD_PHI_RADIAL) {
                const T x = eta * inv_r - T(1);
                const T f = pref * exp(-x * x * inv_2s2) * (dx * nn.x + dy * nn.y + dz * nn.z) * recip(eta) * nn.w;
                if (xi > T(0)) kahan_add(sr, cr, a.lam1 * f);
                else kahan_add(si, ci, a.lam2 * f);
                continue;
            }
            const T rm1 = eta * inv_xabs - T(1);
            if (PHI == SD_PHI_SDF && a.eps >= T(0) && rm1 > a.eps) continue;
            const T E = PHI == SD_PHI_SDF ? exp(-rm1 * rm1 * inv_2s2) : T(1);
            const T cos_t = (dx * nn.x + dy * nn.y + dz * nn.z) * recip(eta);
            // zeta^-2 = (xi - i eta)^2 / (xi^2 + eta^2)^2
            const T den = xi2 + d2;
            const T inv_den2 = recip(den * den);
            const T zr = (xi2 - d2) * inv_den2;
            const T zi = T(-2) * xi * eta * inv_den2;
            T f = pref * E * cos_t * nn.w;
            if (D == 2) f *= T(2) * eta;  // planar angle measure
            kahan_add(sr, cr, f * zr);
            kahan_add(si, ci, f * zi);
        }
    }
    if (!live) return;
    part[(int64_t)blockIdx.y * a.m + i] = mk(sr, si);
}

// The same sum (3D, Eq. 15 with a truncation) over the tree: one CTA per 32
// queries as in k_sdf_tree, tiles tested 32 at a time against the warp's reach
// (1 + eps) max|xi|, each warp taking one of a tile's sub-tiles unless it lies beyond
// every lane's own reach: what is skipped holds no pair that passes Eq. 17t.  What a lane
// adds, and in which order, does not depend on what is skipped.  (One CTA per 256 queries, in lock-step over whole tiles: 14.0 ms for
// 5,000 spheres.)  Queries too few to fill the GPU have the tiles dealt to several CTAs
// (grid y, sum_splits; in turn, as a group's near tiles are neighbours), a partial sum
// each with its compensation, which k_sdf_sum_finish adds.
template <typename T>
__global__ void __launch_bounds__(32 * TREE_NW) k_sdf_sum_tree(SdfArgs<T> a, cplx<T>* part) {
    constexpr int SUB = SDF_TILE / 32;
    __shared__ T sh[4][TREE_NW][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t i = min((int64_t)blockIdx.x * 32 + lane, a.m - 1);
    const int64_t src = a.perm_q ? (int64_t)a.perm_q[i] : i;
    const vec4<T> p = a.qry[src];
    const T xabs = a.xi_abs[i];
    const T xi = a.pmc[i] < 0 ? -xabs : xabs;
    float lo[3], hi[3];
    const vec4<T> pp[1] = {p};
    warp_box<T, 1>(pp, lo, hi);
    float reach = (float)xabs;
    for (int off = 16; off > 0; off >>= 1) reach = fmaxf(reach, __shfl_xor_sync(0xffffffffu, reach, off));
    reach = reach * (1.f + (float)a.eps) * (1.f + 1e-4f) + 1e-6f;
    const float reach2 = reach * reach;
    const float own_reach = (float)xabs * (1.f + (float)a.eps) * (1.f + 1e-4f) + 1e-6f;
    const float own2 = own_reach * own_reach;
    const T lam = xi > T(0) ? a.lam1 : -a.lam2;
    const T pref = lam / (T(2.0 * M_PI) * a.sigma);
    const T inv_xabs = recip(xabs);
    const T inv_2s2 = recip(T(2) * a.sigma * a.sigma);
    const T xi2 = xi * xi;
    T sr = 0, cr = 0, si = 0, ci = 0;
    const int step = (int)gridDim.y, n_tiles = (int)a.n_tiles;
    for (int base = (int)blockIdx.y; base < n_tiles; base += 32 * step) {
        const int t = base + lane * step;
        // NaN reach (a query whose distance is none) keeps every tile
        const bool in = t < n_tiles && !(a.tile_box && box_gap2(a.tile_box + (int64_t)t * 6, lo, hi) > reach2);
        unsigned m = __ballot_sync(0xffffffffu, in);
        while (m) {
            const int tt = base + (__ffs(m) - 1) * step;
            m &= m - 1;
            const int64_t j0 = (int64_t)tt * SDF_TILE + warp * 32;
            const int cnt = (int)min((int64_t)32, a.n_b - j0);
            if (a.sub_box && __all_sync(0xffffffffu, point_gap2<T>(a.sub_box + ((int64_t)tt * SUB + warp) * 6, p) > own2))
                continue;
#pragma unroll 2
            for (int k = 0; k < cnt; ++k) {
                const vec4<T> q = sample4(a.bnd + j0 + k);
                const T dx = p.x - q.x, dy = p.y - q.y, dz = p.z - q.z;
                const T d2 = dx * dx + dy * dy + dz * dz;
                const T eta = sqrt(d2);
                const T rm1 = eta * inv_xabs - T(1);
                if (rm1 > a.eps) continue;
                const vec4<T> nn = sample4(a.nrm + j0 + k);
                const T E = exp(-rm1 * rm1 * inv_2s2);
                const T cos_t = (dx * nn.x + dy * nn.y + dz * nn.z) * recip(eta);
                // zeta^-2 = (xi - i eta)^2 / (xi^2 + eta^2)^2
                const T den = xi2 + d2;
                const T inv_den2 = recip(den * den);
                const T f = pref * E * cos_t * nn.w;
                kahan_add(sr, cr, f * ((xi2 - d2) * inv_den2));
                kahan_add(si, ci, f * (T(-2) * xi * eta * inv_den2));
            }
        }
    }
    sh[0][warp][lane] = sr;
    sh[1][warp][lane] = cr;
    sh[2][warp][lane] = si;
    sh[3][warp][lane] = ci;
    __syncthreads();
    if (warp != 0 || (int64_t)blockIdx.x * 32 + lane >= a.m) return;
    for (int w = 1; w < TREE_NW; ++w) {
        kahan_add(sr, cr, sh[0][w][lane]);
        kahan_add(sr, cr, -sh[1][w][lane]);
        kahan_add(si, ci, sh[2][w][lane]);
        kahan_add(si, ci, -sh[3][w][lane]);
    }
    if (part) {
        part[2 * ((int64_t)blockIdx.y * a.m + i)] = mk(sr, si);
        part[2 * ((int64_t)blockIdx.y * a.m + i) + 1] = mk(cr, ci);
        return;
    }
    const T v = a.vol[src];
    a.c_out[i] = mk(sr * v, si * v);
    if (a.rho_out) a.rho_out[src] = mk(sr, si);
    vec4<T> po = p;
    po.w = T(0);
    a.pos_out[i] = po;
}

// rho of each query: the partial sums added in split order (compensated; PAIRS: with the
// partials' own compensations), then the shape's sample c = rho v and position.
template <typename T, bool PAIRS>
__global__ void k_sdf_sum_finish(SdfArgs<T> a, int splits, const cplx<T>* part) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= a.m) return;
    T sr = 0, cr = 0, si = 0, ci = 0;
    for (int k = 0; k < splits; ++k) {
        const cplx<T>* p = part + ((int64_t)k * a.m + i) * (PAIRS ? 2 : 1);
        kahan_add(sr, cr, p[0].x);
        kahan_add(si, ci, p[0].y);
        if constexpr (PAIRS) {
            kahan_add(sr, cr, -p[1].x);
            kahan_add(si, ci, -p[1].y);
        }
    }
    const int64_t src = a.perm_q ? (int64_t)a.perm_q[i] : i;
    const T v = a.vol[src];
    a.c_out[i] = mk(sr * v, si * v);
    if (a.rho_out) a.rho_out[src] = mk(sr, si);
    vec4<T> po = a.qry[src];
    po.w = T(0);
    a.pos_out[i] = po;
}

template <typename T>
__global__ void k_boundary_order(const vec4<T>* bnd, const vec4<T>* nrm, const T* area, const int32_t* perm,
                                 int64_t n_b, int dim, vec4<T>* bnd_s, vec4<T>* nrm_s, float* tile_box,
                                 float* sub_box) {
    __shared__ float wred[SDF_TILE / 32][6];
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    float v[6] = {FLT_MAX, FLT_MAX, FLT_MAX, -FLT_MAX, -FLT_MAX, -FLT_MAX};
    if (i < n_b) {
        const int32_t j = perm[i];
        const vec4<T> q = bnd[j];
        vec4<T> nn = nrm[j];
        nn.w = area[j];
        bnd_s[i] = q;
        nrm_s[i] = nn;
        v[0] = v[3] = (float)q.x;
        v[1] = v[4] = (float)q.y;
        v[2] = v[5] = (dim == 3) ? (float)q.z : 0.f;
    }
    for (int off = 16; off > 0; off >>= 1) {
        for (int d = 0; d < 3; ++d) v[d] = fminf(v[d], __shfl_down_sync(0xffffffffu, v[d], off));
        for (int d = 3; d < 6; ++d) v[d] = fmaxf(v[d], __shfl_down_sync(0xffffffffu, v[d], off));
    }
    if ((threadIdx.x & 31) == 0) {
        for (int d = 0; d < 6; ++d) wred[threadIdx.x >> 5][d] = v[d];
        // the box of this warp's 32 samples (a sub-tile), widened like the tile's
        float* sb = sub_box + ((int64_t)blockIdx.x * (SDF_TILE / 32) + (threadIdx.x >> 5)) * 6;
        for (int d = 0; d < 6; ++d) {
            const float m = 1e-6f * (fabsf(v[d]) + 1.f);
            sb[d] = v[d] == FLT_MAX || v[d] == -FLT_MAX ? v[d] : (d < 3 ? v[d] - m : v[d] + m);
        }
    }
    __syncthreads();
    if (threadIdx.x < 6) {
        float r = wred[0][threadIdx.x];
        for (int w = 1; w < SDF_TILE / 32; ++w)
            r = threadIdx.x < 3 ? fminf(r, wred[w][threadIdx.x]) : fmaxf(r, wred[w][threadIdx.x]);
        // widen by a float ulp-scale margin so the tile test stays conservative
        const float m = 1e-6f * (fabsf(r) + 1.f);
        tile_box[blockIdx.x * 6 + threadIdx.x] = threadIdx.x < 3 ? r - m : r + m;
    }
}

template <typename T>
cudaError_t launch_boundary_order(const vec4<T>* bnd, const vec4<T>* nrm, const T* area, const int32_t* perm,
                                  int64_t n_b, int dim, vec4<T>* bnd_s, vec4<T>* nrm_s, float* tile_box,
                                  cudaStream_t st) {
    if (n_b == 0) return cudaSuccess;
    const int64_t n_tiles = (n_b + SDF_TILE - 1) / SDF_TILE;
    k_boundary_order<T><<<(unsigned)n_tiles, SDF_TILE, 0, st>>>(bnd, nrm, area, perm, n_b, dim, bnd_s, nrm_s, tile_box,
                                                                tile_box + n_tiles * 6);
    note_launch();
    return cudaGetLastError();
}

// Skin / core layers of the signed distance (no boundary sum):
// rho = lambda1 g(xi / R - 1) + i lambda2 g(xi / R + 1), g the normalised Gaussian
// of width sigma.
template <typename T>
__global__ void __launch_bounds__(SDF_TILE) k_sdf_skin(SdfArgs<T> a) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= a.m) return;
    const int64_t src = a.perm_q ? (int64_t)a.perm_q[i] : i;
    const vec4<T> p = a.qry[src];
    const T xi = a.pmc[i] < 0 ? -a.xi_abs[i] : a.xi_abs[i];
    const T inv_r = recip(a.radius);
    const T inv_2s2 = recip(T(2) * a.sigma * a.sigma);
    const T norm = T(1) / (sqrt(T(2.0 * M_PI)) * a.sigma);
    const T xo = xi * inv_r - T(1), xc = xi * inv_r + T(1);
    const T sr = a.lam1 * norm * exp(-xo * xo * inv_2s2);
    const T si = a.lam2 * norm * exp(-xc * xc * inv_2s2);
    const T v = a.vol[src];
    a.c_out[i] = mk(sr * v, si * v);
    if (a.rho_out) a.rho_out[src] = mk(sr, si);
    vec4<T> po = p;
    po.w = T(0);
    a.pos_out[i] = po;
}

// Boundary-tile splits per query block: enough CTAs for about four per SM.
static int sdf_splits(int64_t query_blocks, int64_t tiles, int most = 64) {
    static int sms = 0;
    if (!sms) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (sms <= 0) sms = 1;
    }
    int64_t s = (4 * (int64_t)sms + query_blocks - 1) / query_blocks;
    s = s < 1 ? 1 : (s > tiles ? tiles : s);
    return (int)(s > most ? most : s);
}

// Splits of the boundary's tiles for `groups` groups of 32 queries in the truncated sum:
// 16 CTAs a SM in all (8 and 32 within 15 % either way, 32 more for the finishing to
// add), a split with at least four tiles.  FP32, us a build without / with: 500 queries
// about 20,000 samples 1,107 / 290 (in a cube; 525 / 290 in a band at the boundary),
// 2,000 about 300,000 14,190 / 1,880 (3,600 / 1,230); FP64, 500 about 5,000 3,420 / 1,140.
static int sum_splits(int64_t groups, int64_t tiles) {
    const int64_t s = std::min((16 * GPU_SMS + groups - 1) / groups, std::min<int64_t>(tiles / 4, 256));
    return s < 1 ? 1 : (int)s;
}

// Whether the tree is faster than all pairs for nearest distances and memberships.  The
// tree's CTAs walk the whole boundary for 32 or 64 queries each (90 us for 5,000 samples,
// 1 ms for 300,000), so it takes queries enough to fill the GPU, and boundary enough to
// leave out; all pairs cost their number and split the boundary too.  The lines lie where
// builds of 1 to 50,000 queries (a cube and a band about a sphere of 100 to 300,000
// samples) change sides.  FP32, us a build by tree / pairs: 500 queries, 20,000 samples
// 346 / 220; 500, 300,000 1,109 / 450; 50,000, 1,000 267 / 242; 5,000, 20,000 366 / 329;
// 10,000, 20,000 391 / 415; 50,000, 5,000 365 / 452.  FP64 (the pair costs ten times as
// much, and so do the tree's nodes): 500, 5,000 1,335 / 540; 50,000, 300 1,334 / 960;
// 5,000, 5,000 1,329 / 1,280; 10,000, 5,000 1,731 / 2,830.
template <typename T>
static bool sdf_tree_pays(int64_t m, int64_t n_b) {
    return sizeof(T) == 4 ? (m - 3300) * n_b > 60000000 : (m - 500) * n_b > 25000000;
}

// Nearest distances and memberships: the tree in 3D (its nodes, and the list of
// queries left to the full sum), all pairs in 2D and in small builds.
template <typename T>
static cudaError_t launch_nearest(const SdfArgs<T>& a, int dim, cudaStream_t st) {
    const unsigned nb = (unsigned)((a.m + SDF_TILE - 1) / SDF_TILE);
    char* scratch = nullptr;
    cudaError_t e;
    if (dim == 2 || !sdf_tree_pays<T>(a.m, a.n_b)) {
        const int64_t tiles = (a.n_b + SDF_TILE - 1) / SDF_TILE;
        const int splits = sdf_splits(nb, tiles < 1 ? 1 : tiles, dim == 2 ? 64 : 256);
        const int tps = (int)((tiles + splits - 1) / splits);
        if ((e = pool_alloc((void**)&scratch, (size_t)2 * splits * a.m * sizeof(T), st)) != cudaSuccess) return e;
        T* d2 = reinterpret_cast<T*>(scratch);
        T* w = d2 + (size_t)splits * a.m;
        if (dim == 2) {
            k_sdf_nearest<T, 2><<<dim3(nb, splits), SDF_TILE, 0, st>>>(a, tps, d2, w);
            k_sdf_nearest_finish<T, 2><<<nb, SDF_TILE, 0, st>>>(a, splits, d2, w);
        } else {
            k_sdf_nearest<T, 3><<<dim3(nb, splits), SDF_TILE, 0, st>>>(a, tps, d2, w);
            k_sdf_nearest_finish<T, 3><<<nb, SDF_TILE, 0, st>>>(a, splits, d2, w);
        }
        note_launch(2);
    } else {
        const size_t nodes_bytes = (size_t)a.n_tiles * (1 + SDF_TILE / 32) * NODE * sizeof(T);
        const size_t parts = (size_t)SDF_TILE * (nb > LIST_CTAS ? nb : LIST_CTAS);
        const size_t list_bytes = ((size_t)a.m + 64) * sizeof(int) / 256 * 256 + 256;
        const size_t pairs_bytes = sizeof(T) == 4 ? (size_t)a.n_tiles * SDF_TILE / 2 * PAIR * sizeof(float) : 0;
        if ((e = pool_alloc((void**)&scratch, nodes_bytes + list_bytes + parts * sizeof(T) + pairs_bytes + 512, st)) !=
            cudaSuccess)
            return e;
        T* nodes = reinterpret_cast<T*>(scratch);
        int* list_n = reinterpret_cast<int*>(scratch + (nodes_bytes + 255) / 256 * 256);
        int* list = list_n + 1;
        T* part = reinterpret_cast<T*>(reinterpret_cast<char*>(list_n) + list_bytes);
        float* pairs = reinterpret_cast<float*>(reinterpret_cast<char*>(part) + (parts * sizeof(T) + 255) / 256 * 256);
        e = cudaMemsetAsync(list_n, 0, sizeof(int), st);
        if (e != cudaSuccess) {
            pool_free(scratch, st);
            return e;
        }
        const float* sub_box = a.tree_box + a.n_tiles * 6;
        k_sdf_nodes<T><<<(unsigned)a.n_tiles, SDF_TILE, 0, st>>>(a.bnd, a.nrm, a.n_b, a.tree_box, sub_box, nodes,
                                                                 a.n_tiles, pairs);
        note_launch();
        if (sizeof(T) == 4 && a.m >= TREE_PAIR_MIN)
            k_sdf_tree<T, 2><<<(unsigned)((a.m + 63) / 64), 32 * TREE_NW, 0, st>>>(a, nodes, a.tree_box, sub_box, pairs, list,
                                                                                         list_n);
        else
            k_sdf_tree<T, 1><<<(unsigned)((a.m + 31) / 32), 32 * TREE_NW, 0, st>>>(a, nodes, a.tree_box, sub_box, pairs, list,
                                                                                         list_n);
        note_launch();
        if (!a.pmc_override) {
            k_sdf_wind_list<T><<<LIST_CTAS, SDF_TILE, 0, st>>>(a, list, list_n, part);
            k_sdf_wind_list_finish<T><<<GPU_SMS, SDF_TILE, 0, st>>>(a, list, list_n, part);
            note_launch(2);
        }
    }
    pool_free(scratch, st);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_sdf(const SdfArgs<T>& a, int dim, cudaStream_t st) {
    if (a.m == 0) return cudaSuccess;
    if (a.phi != SD_PHI_SKIN && a.phi != SD_PHI_SDF && a.phi != SD_PHI_PROXIMAL && a.phi != SD_PHI_RADIAL)
        return cudaErrorInvalidValue;
    const unsigned nb = (unsigned)((a.m + SDF_TILE - 1) / SDF_TILE);
    cudaError_t e = launch_nearest<T>(a, dim, st);
    if (e != cudaSuccess) return e;
    if (a.phi == SD_PHI_SKIN) {  // the pointwise layers
        k_sdf_skin<T><<<nb, SDF_TILE, 0, st>>>(a);
        note_launch();
        return cudaGetLastError();
    }
    if (dim == 3 && a.phi == SD_PHI_SDF && a.eps >= T(0)) {
        const int64_t groups = (a.m + 31) / 32;
        const int splits = sum_splits(groups, a.n_tiles);
        cplx<T>* part = nullptr;
        if (splits > 1 && (e = pool_alloc((void**)&part, (size_t)splits * a.m * 2 * sizeof(cplx<T>), st)) != cudaSuccess) return e;
        k_sdf_sum_tree<T><<<dim3((unsigned)groups, splits), 32 * TREE_NW, 0, st>>>(a, part);
        note_launch();
        if (part) {
            k_sdf_sum_finish<T, true><<<nb, SDF_TILE, 0, st>>>(a, splits, part);
            note_launch();
            pool_free(part, st);
        }
        return cudaGetLastError();
    }
    // every pair (no truncation, or 2D): the boundary tiles of a query block split
    // over CTAs, one partial rho per split and query
    const int64_t tiles = (a.n_b + SDF_TILE - 1) / SDF_TILE;
    const int splits = sdf_splits(nb, tiles < 1 ? 1 : tiles);
    const int tps = (int)((tiles + splits - 1) / splits);
    cplx<T>* part = nullptr;
    if ((e = pool_alloc((void**)&part, (size_t)splits * a.m * sizeof(cplx<T>), st)) != cudaSuccess) return e;
    const dim3 grid(nb, splits);
#define SD_SUM(DD, PP) k_sdf_sum<T, DD, PP><<<grid, SDF_TILE, 0, st>>>(a, tps, part)
    switch (a.phi) {
        case SD_PHI_SDF:
            if (dim == 2) SD_SUM(2, SD_PHI_SDF);
            else SD_SUM(3, SD_PHI_SDF);
            break;
        case SD_PHI_PROXIMAL:
            if (dim == 2) SD_SUM(2, SD_PHI_PROXIMAL);
            else SD_SUM(3, SD_PHI_PROXIMAL);
            break;
        default:
            if (dim == 2) SD_SUM(2, SD_PHI_RADIAL);
            else SD_SUM(3, SD_PHI_RADIAL);
            break;
    }
#undef SD_SUM
    k_sdf_sum_finish<T, false><<<nb, SDF_TILE, 0, st>>>(a, splits, part);
    note_launch(2);
    pool_free(part, st);
    return cudaGetLastError();
}

template <typename T>
__global__ void k_radius(const vec4<T>* p, int64_t m, int dim, double* out) {
    double best = 0.0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < m; i += (int64_t)gridDim.x * blockDim.x) {
        const vec4<T> v = p[i];
        double r2 = (double)v.x * v.x + (double)v.y * v.y + (dim == 3 ? (double)v.z * v.z : 0.0);
        best = fmax(best, r2);
    }
    for (int off = 16; off > 0; off >>= 1) best = fmax(best, __shfl_down_sync(0xffffffffu, best, off));
    if ((threadIdx.x & 31) == 0) {
        // r2 >= 0: ordering of the IEEE bits matches the ordering of the values
        atomicMax(reinterpret_cast<unsigned long long*>(out), (unsigned long long)__double_as_longlong(best));
    }
}

template <typename T>
cudaError_t launch_radius(const vec4<T>* p, int64_t m, int dim, double* out, cudaStream_t st) {
    cudaError_t e = cudaMemsetAsync(out, 0, sizeof(double), st);
    if (e != cudaSuccess) return e;
    if (m == 0) return cudaSuccess;
    const int nb = (int)((m + 255) / 256 < 1024 ? (m + 255) / 256 : 1024);
    k_radius<T><<<nb, 256, 0, st>>>(p, m, dim, out);
    note_launch();
    return cudaGetLastError();
}

template cudaError_t launch_sdf<float>(const SdfArgs<float>&, int, cudaStream_t);
template cudaError_t launch_sdf<double>(const SdfArgs<double>&, int, cudaStream_t);
template cudaError_t launch_radius<float>(const vec4<float>*, int64_t, int, double*, cudaStream_t);
template cudaError_t launch_radius<double>(const vec4<double>*, int64_t, int, double*, cudaStream_t);
template cudaError_t launch_boundary_order<float>(const vec4<float>*, const vec4<float>*, const float*, const int32_t*,
                                                  int64_t, int, vec4<float>*, vec4<float>*, float*, cudaStream_t);
template cudaError_t launch_boundary_order<double>(const vec4<double>*, const vec4<double>*, const double*,
                                                   const int32_t*, int64_t, int, vec4<double>*, vec4<double>*, float*,
                                                   cudaStream_t);

}  // namespace sd
