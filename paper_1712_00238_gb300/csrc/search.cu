// Search over the per-rotation maxima (the argmax over T of Section 4) and the
// FP64 re-score of the best poses.
//
// top-k: one CTA finds the k-th candidate in the order (score descending, rotation
// ascending, translation index ascending, position) by radix selection, collects
// the k that do not come after it and sorts them in shared memory; up to three
// candidates take an arg-best pass each.
// re-score: f_c(R, t) = sum_ij c1_i c2_j G_{sigma_g sqrt 2}(R p2_j + t - p1_i) in
// FP64 (the continuous score of Eq. 8 for Gaussian-represented SDFs).  Pairs
// are screened in FP32 against a cutoff of 8 sigma_g sqrt 2 (with a margin), and
// CTA / tile bounding boxes skip whole blocks of far pairs.
#include <algorithm>
#include <float.h>
#include <limits.h>
#include <math.h>

#include "kernels.cuh"

namespace sd {

struct Cand {
    double score;
    int32_t rot;
    int32_t idx;
};

// A candidate's place in the order as one unsigned key, best first: the score's
// bits mapped so that larger scores come first (-0 counts as 0, NaN as -inf: last),
// then rotation and translation index, then position.
struct CandKey {
    unsigned long long a, b;
    unsigned c;
};
__device__ __forceinline__ CandKey cand_key(const Cand& v, int64_t pos) {
    const double s = v.score == v.score ? (v.score == 0.0 ? 0.0 : v.score) : -INFINITY;
    const unsigned long long u = (unsigned long long)__double_as_longlong(s);
    CandKey k;
    k.a = (u >> 63) ? u : ~(u | 0x8000000000000000ull);  // descending
    k.b = ((unsigned long long)((unsigned)v.rot ^ 0x80000000u) << 32) | ((unsigned)v.idx ^ 0x80000000u);
    k.c = (unsigned)pos;
    return k;
}
__device__ __forceinline__ bool key_less(const CandKey& x, const CandKey& y) {
    if (x.a != y.a) return x.a < y.a;
    if (x.b != y.b) return x.b < y.b;
    return x.c < y.c;
}
__device__ __forceinline__ Cand load_cand(const Cand* p) {
    const int2 v = *reinterpret_cast<const int2*>(&p->rot);  // records are 8-byte aligned
    Cand c;
    c.score = p->score;
    c.rot = v.x;
    c.idx = v.y;
    return c;
}

constexpr int TOPK_THREADS = 1024, TOPK_MAX = 4096;

// Up to three candidates take a pass each: the first in the order after the one before.
// The selection below reads the list at least three times and counts its bytes.  Passes
// against the selection, us a call: k = 1 of 54,000 candidates 74 against 205, of 2^20
// 641 against 2,760; k = 2 110 against 232 and 1,257 against 3,370; k = 3 (by the two
// above: 36 and 620 a pass) about 146 against 185 and 1,880 against 3,370; at k = 4 they
// are even.
constexpr int TOPK_PASSES = 3;

__global__ void __launch_bounds__(TOPK_THREADS) k_topk_passes(const Cand* cand, int64_t n, int k, Cand* out) {
    __shared__ CandKey won[TOPK_THREADS / 32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const CandKey none{~0ull, ~0ull, ~0u};  // after every candidate: no position is 2^32 - 1
    CandKey prev{0, 0, 0};
    for (int it = 0; it < k; ++it) {
        CandKey best = none;
#pragma unroll 4
        for (int64_t p = tid; p < n; p += TOPK_THREADS) {
            const CandKey q = cand_key(load_cand(cand + p), p);
            if (key_less(q, best) && (it == 0 || key_less(prev, q))) best = q;
        }
        for (int off = 16; off > 0; off >>= 1) {
            const CandKey o{__shfl_xor_sync(0xffffffffu, best.a, off), __shfl_xor_sync(0xffffffffu, best.b, off),
                            __shfl_xor_sync(0xffffffffu, best.c, off)};
            if (key_less(o, best)) best = o;
        }
        if (lane == 0) won[warp] = best;
        __syncthreads();
        for (int w = 0; w < TOPK_THREADS / 32; ++w)
            if (key_less(won[w], best)) best = won[w];
        __syncthreads();
        if (tid == 0) {
            Cand c;
            if (best.c != none.c) c = load_cand(cand + best.c);
            else { c.score = -INFINITY; c.rot = -1; c.idx = -1; }
            out[it] = c;
        }
        prev = best;
    }
}

// Radix selection a byte of the key at a time, most significant first, over the
// candidates that share the bytes fixed so far; bytes equal in all of them are
// skipped, and the selection ends when what is left of the k fills its bucket.  A
// few reads of the list by one SM, whatever k is (54,000 candidates, k = 100: 5.06 ms
// for k arg-best passes).  Shared memory: the k selected keys, then sorted.
__global__ void __launch_bounds__(TOPK_THREADS) k_topk(const Cand* cand, int64_t n, int k, Cand* out) {
    extern __shared__ __align__(16) unsigned char tk_raw[];
    __shared__ int hist[256];
    __shared__ unsigned long long diff_a, diff_b;
    __shared__ int bucket, left_s, in_bucket, taken;
    const int tid = threadIdx.x, lane = tid & 31;
    int p2 = 1;
    while (p2 < k) p2 <<= 1;
    unsigned long long* sa = reinterpret_cast<unsigned long long*>(tk_raw);
    unsigned long long* sb = sa + p2;
    unsigned* sc = reinterpret_cast<unsigned*>(sb + p2);
    const int64_t want = n < k ? n : k;
    // bits in which the keys differ at all
    if (tid == 0) {
        diff_a = diff_b = 0;
        taken = 0;
    }
    __syncthreads();
    {
        const CandKey first = cand_key(load_cand(cand), 0);
        unsigned long long da = 0, db = 0;
        for (int64_t p = tid; p < n; p += TOPK_THREADS) {
            const CandKey q = cand_key(load_cand(cand + p), p);
            da |= q.a ^ first.a;
            db |= q.b ^ first.b;
        }
        for (int off = 16; off > 0; off >>= 1) {
            da |= __shfl_xor_sync(0xffffffffu, da, off);
            db |= __shfl_xor_sync(0xffffffffu, db, off);
        }
        if (lane == 0) {
            atomicOr(&diff_a, da);
            atomicOr(&diff_b, db);
        }
    }
    __syncthreads();
    const CandKey first = cand_key(load_cand(cand), 0);
    CandKey pre{0, 0, 0}, mask{0, 0, 0};  // the bytes fixed so far
    int left = (int)want;                 // of the candidates that match them
    bool done = want == n;                // everything is taken
    for (int d = 0; d < 20 && !done; ++d) {  // bytes of a, b, c
        const int sh = 56 - 8 * (d & 7), shc = 24 - 8 * (d - 16);
        const unsigned long long byte = 0xffull << (sh & 63);
        if (d < 16 && !((d < 8 ? diff_a : diff_b) & byte)) {  // equal in every key
            if (d < 8) { pre.a |= first.a & byte; mask.a |= byte; }
            else { pre.b |= first.b & byte; mask.b |= byte; }
            continue;
        }
        for (int i = tid; i < 256; i += TOPK_THREADS) hist[i] = 0;
        __syncthreads();
        for (int64_t p0 = 0; p0 < n; p0 += TOPK_THREADS) {
            const int64_t p = p0 + tid;
            int dig = -1;
            if (p < n) {
                const CandKey q = cand_key(load_cand(cand + p), p);
                if ((q.a & mask.a) == pre.a && (q.b & mask.b) == pre.b && (q.c & mask.c) == pre.c)
                    dig = d < 8 ? (int)((q.a >> sh) & 255) : (d < 16 ? (int)((q.b >> sh) & 255) : (int)((q.c >> shc) & 255));
            }
            // keys share their leading bytes: one add per group of equal digits
            const unsigned same = __match_any_sync(0xffffffffu, dig);
            if (dig >= 0 && lane == __ffs(same) - 1) atomicAdd(&hist[dig], __popc(same));
        }
        __syncthreads();
        if (tid < 32) {  // the bucket of the `left`-th match
            int own[8], sum = 0;
            for (int i = 0; i < 8; ++i) sum += own[i] = hist[8 * lane + i];
            int incl = sum;
            for (int off = 1; off < 32; off <<= 1) {
                const int v = __shfl_up_sync(0xffffffffu, incl, off);
                if (lane >= off) incl += v;
            }
            int before = incl - sum;
            if (before < left && left <= incl) {
                int i = 0;
                while (before + own[i] < left) before += own[i++];
                bucket = 8 * lane + i;
                left_s = left - before;
                in_bucket = own[i];
            }
        }
        __syncthreads();
        const unsigned long long v = (unsigned long long)bucket;
        if (d < 8) { pre.a |= v << sh; mask.a |= byte; }
        else if (d < 16) { pre.b |= v << sh; mask.b |= byte; }
        else { pre.c |= (unsigned)(v << shc); mask.c |= 0xffu << shc; }
        left = left_s;
        done = left == in_bucket;
        __syncthreads();
    }
    // collect: everything not after the fixed bytes
    for (int64_t p = tid; p < n; p += TOPK_THREADS) {
        const CandKey q = cand_key(load_cand(cand + p), p);
        const CandKey m{q.a & mask.a, q.b & mask.b, q.c & mask.c};
        if (!key_less(pre, m)) {
            const int slot = atomicAdd(&taken, 1);
            if (slot < p2) { sa[slot] = q.a; sb[slot] = q.b; sc[slot] = q.c; }
        }
    }
    for (int i = tid; i < p2; i += TOPK_THREADS)
        if (i >= want) { sa[i] = ~0ull; sb[i] = ~0ull; sc[i] = ~0u; }
    __syncthreads();
    // bitonic sort, ascending
    for (int size = 2; size <= p2; size <<= 1)
        for (int stride = size >> 1; stride > 0; stride >>= 1) {
            for (int i = tid; i < p2 / 2; i += TOPK_THREADS) {
                const int lo = 2 * i - (i & (stride - 1)), hi = lo + stride;
                const CandKey x{sa[lo], sb[lo], sc[lo]}, y{sa[hi], sb[hi], sc[hi]};
                if (key_less(y, x) == ((lo & size) == 0)) {
                    sa[lo] = y.a; sb[lo] = y.b; sc[lo] = y.c;
                    sa[hi] = x.a; sb[hi] = x.b; sc[hi] = x.c;
                }
            }
            __syncthreads();
        }
    for (int i = tid; i < k; i += TOPK_THREADS) {
        Cand c;
        if (i < want) c = load_cand(cand + sc[i]);
        else { c.score = -INFINITY; c.rot = -1; c.idx = -1; }
        out[i] = c;
    }
}

cudaError_t launch_topk(const void* cand, int64_t n, int k, void* out, cudaStream_t st) {
    if (k <= TOPK_PASSES) {
        k_topk_passes<<<1, TOPK_THREADS, 0, st>>>(reinterpret_cast<const Cand*>(cand), n, k, reinterpret_cast<Cand*>(out));
        note_launch();
        return cudaGetLastError();
    }
    int p2 = 1;
    while (p2 < k) p2 <<= 1;
    constexpr size_t key = 2 * sizeof(unsigned long long) + sizeof(unsigned);
    const size_t smem = (size_t)p2 * key;
    if (smem > 32 * 1024) {
        // one value per kernel and device, always that of the largest k: a call on
        // another thread must not lower it between this one's setting and its launch
        const cudaError_t e = cudaFuncSetAttribute(k_topk, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(TOPK_MAX * key));
        if (e != cudaSuccess) return e;
    }
    k_topk<<<1, TOPK_THREADS, smem, st>>>(reinterpret_cast<const Cand*>(cand), n, k, reinterpret_cast<Cand*>(out));
    note_launch();
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------

constexpr int RS_TILE = 256;
constexpr int RS_WARPS = RS_TILE / 32;

// Block-wide bounding box of one point per thread (dead threads pass +inf/-inf);
// the result is valid in out_lo/out_hi (shared) after the call.
__device__ __forceinline__ void block_bbox(float lo[3], float hi[3], float (*wlo)[3], float (*whi)[3],
                                           float out_lo[3], float out_hi[3]) {
    for (int d = 0; d < 3; ++d)
        for (int off = 16; off > 0; off >>= 1) {
            lo[d] = fminf(lo[d], __shfl_down_sync(0xffffffffu, lo[d], off));
            hi[d] = fmaxf(hi[d], __shfl_down_sync(0xffffffffu, hi[d], off));
        }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (lane == 0)
        for (int d = 0; d < 3; ++d) { wlo[warp][d] = lo[d]; whi[warp][d] = hi[d]; }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int d = 0; d < 3; ++d) {
            float a = FLT_MAX, b = -FLT_MAX;
            for (int w = 0; w < RS_WARPS; ++w) { a = fminf(a, wlo[w][d]); b = fmaxf(b, whi[w][d]); }
            out_lo[d] = a;
            out_hi[d] = b;
        }
    }
    __syncthreads();
}

// Pose (R, t) of a candidate: rotation matrix (FP64) and translation of its grid index.
__device__ void pose_of(const Cand& cd, const double* quats, int N, double L, int dim, double Rm[9], double tv[3]) {
    const double h = L / N;
    int idx = cd.idx < 0 ? 0 : cd.idx;
    for (int d = 0; d < 3; ++d) {
        if (d < dim) {
            tv[d] = (double)(idx % N - N / 2) * h;
            idx /= N;
        } else {
            tv[d] = 0.0;
        }
    }
    const double* q = quats + 4 * (int64_t)cd.rot;
    const double w = q[0], x = q[1], y = q[2], z = q[3];
    const double n2 = w * w + x * x + y * y + z * z;
    const double s = n2 > 0 ? 2.0 / n2 : 0.0;
    Rm[0] = 1 - s * (y * y + z * z); Rm[1] = s * (x * y - w * z); Rm[2] = s * (x * z + w * y);
    Rm[3] = s * (x * y + w * z); Rm[4] = 1 - s * (x * x + z * z); Rm[5] = s * (y * z - w * x);
    Rm[6] = s * (x * z - w * y); Rm[7] = s * (y * z + w * x); Rm[8] = 1 - s * (x * x + y * y);
}

// Per pose: the moved samples y_j = R p2_j + t in FP64 and the float bounding box
// of every tile of RS_TILE consecutive samples.
template <typename T>
__global__ void __launch_bounds__(RS_TILE) k_rescore_move(RescoreArgs<T> a) {
    __shared__ double Rm[9], tv[3];
    __shared__ float wlo[RS_WARPS][3], whi[RS_WARPS][3];
    __shared__ float blo[3], bhi[3];
    const int pose = blockIdx.y;
    const Cand cd = reinterpret_cast<const Cand*>(a.top)[pose];
    const int ntiles = gridDim.x;
    float* tb = a.tile_box + ((int64_t)pose * ntiles + blockIdx.x) * 6;
    if (cd.rot < 0) {
        if (threadIdx.x < 3) { tb[threadIdx.x] = FLT_MAX; tb[3 + threadIdx.x] = -FLT_MAX; }
        return;
    }
    if (threadIdx.x == 0) pose_of(cd, a.quats, a.N, a.L, a.dim, Rm, tv);
    __syncthreads();
    const int64_t j = (int64_t)blockIdx.x * RS_TILE + threadIdx.x;
    float lo[3] = {FLT_MAX, FLT_MAX, FLT_MAX}, hi[3] = {-FLT_MAX, -FLT_MAX, -FLT_MAX};
    if (j < a.m2) {
        const vec4<T> p = a.p2[j];
        const double qx = p.x, qy = p.y, qz = (a.dim == 3) ? (double)p.z : 0.0;
        double4 y;
        y.x = Rm[0] * qx + Rm[1] * qy + Rm[2] * qz + tv[0];
        y.y = Rm[3] * qx + Rm[4] * qy + Rm[5] * qz + tv[1];
        y.z = (a.dim == 3) ? Rm[6] * qx + Rm[7] * qy + Rm[8] * qz + tv[2] : 0.0;
        y.w = 0.0;
        reinterpret_cast<double4*>(a.moved)[(int64_t)pose * a.m2 + j] = y;
        lo[0] = hi[0] = (float)y.x; lo[1] = hi[1] = (float)y.y; lo[2] = hi[2] = (float)y.z;
    }
    block_bbox(lo, hi, wlo, whi, blo, bhi);
    if (threadIdx.x < 3) { tb[threadIdx.x] = blo[threadIdx.x]; tb[3 + threadIdx.x] = bhi[threadIdx.x]; }
}

// Pairs that pass the FP32 screen are queued per warp and evaluated 32 at a
// time in FP64 with every lane busy: only the pose's total is needed, so any
// lane may take any pair.
// The FP64 pipe (1.06 TFLOP/s) bounds the kernel: 76 % busy over 21.6 ms at the
// docking pair's top 100.  The exponential is evaluated with as few FP64 operations
// as its accuracy allows, 8 instead of about 17: exp(-u) = 2^(-m / 256) e^(-f ln 2 / 256)
// with u 256 / ln 2 = m + f, m an integer (its fraction bits index a table of
// 2^(-i / 256) in shared memory, the rest goes into the exponent), |f| <= 1/2, and the
// last factor's Taylor series to the fourth order (the next term is below 4e-17).
constexpr int RS_QUEUE = 256;  // pair slots per warp
constexpr int RS_EXP = 256;    // entries of the table

// exp(-r2 / (2 s^2)) from r2 and k = 256 / (2 s^2 ln 2), r2 k >= 0.  The screen's FP32
// coordinates may lie a whole cutoff off where positions exceed s by their 24 bits, so
// any r2 can come: past 2^-1000 (m in the low word, the high word magic's own) the
// result is 0, by integer tests that take nothing from the FP64 pipe.
__device__ __forceinline__ double gauss_exp(double r2, double k, const double* tab) {
    const double magic = 6755399441055744.0;  // 1.5 * 2^52: the low word receives round(x)
    const double t = fma(r2, k, magic);
    const unsigned m = (unsigned)__double2loint(t);
    const double f = fma(r2, k, magic - t);
    static_assert(RS_EXP == 1 << 8, "");
    constexpr double c = -0.6931471805599453094 / RS_EXP;
    const double q = f * fma(f, fma(f, fma(f, c * c * c * c / 24.0, c * c * c / 6.0), c * c / 2.0), c);
    const double w = tab[m & (RS_EXP - 1)];
    const bool in = __double2hiint(t) == 0x43380000 && m < 1000u * RS_EXP;
    const double e = __hiloint2double(in ? __double2hiint(w) - (int)((m >> 8) << 20) : 0, in ? __double2loint(w) : 0);
    return fma(e, q, e);
}

template <typename T>
__global__ void __launch_bounds__(RS_TILE) k_rescore(RescoreArgs<T> a) {
    __shared__ double yx[RS_TILE], yy[RS_TILE], yz[RS_TILE], cr[RS_TILE], ci[RS_TILE];
    __shared__ double qx1[RS_TILE], qy1[RS_TILE], qz1[RS_TILE], ar1[RS_TILE], ai1[RS_TILE];
    __shared__ float4 fxyz[RS_TILE];  // FP32 copies of the moved samples for the screen (one load each)
    __shared__ unsigned short qpair[RS_WARPS][RS_QUEUE][2];  // (fixed slot, moving slot)
    __shared__ float wlo[RS_WARPS][3], whi[RS_WARPS][3];
    __shared__ float blo[3], bhi[3];
    __shared__ float slo[RS_WARPS][3], shi[RS_WARPS][3];  // boxes of the 32-sample slices of a moving tile
    __shared__ double tv[3];
    __shared__ double etab[RS_EXP];
    __shared__ int skip;
    const int pose = blockIdx.y;
    const Cand cd = reinterpret_cast<const Cand*>(a.top)[pose];
    if (cd.rot < 0) return;  // uniform over the block
    if (threadIdx.x == 0) {
        double Rm[9], t3[3];
        pose_of(cd, a.quats, a.N, a.L, a.dim, Rm, t3);
        tv[0] = t3[0]; tv[1] = t3[1]; tv[2] = t3[2];
    }
    const double sg2 = 2.0 * a.sigma_g * a.sigma_g;  // (sigma_g sqrt 2)^2
    const double kexp = RS_EXP / (2.0 * sg2 * 0.6931471805599453094);
    const double cut = 8.0 * sqrt(sg2);
    const float cut2f = (float)(cut * cut) * 1.001f;
    const double norm = (a.dim == 3) ? pow(2.0 * M_PI * sg2, -1.5) : 1.0 / (2.0 * M_PI * sg2);
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const bool live = i < a.m1;
    float lo[3] = {FLT_MAX, FLT_MAX, FLT_MAX}, hi[3] = {-FLT_MAX, -FLT_MAX, -FLT_MAX};
    float pxf = 0.f, pyf = 0.f, pzf = 0.f;
    {
        double px = 0, py = 0, pz = 0, ar = 0, ai = 0;
        if (live) {
            const vec4<T> p = a.p1[i];
            px = p.x; py = p.y; pz = (a.dim == 3) ? (double)p.z : 0.0;
            ar = a.c1[i].x; ai = a.c1[i].y;
            pxf = (float)px; pyf = (float)py; pzf = (float)pz;
            lo[0] = hi[0] = pxf; lo[1] = hi[1] = pyf; lo[2] = hi[2] = pzf;
        }
        qx1[threadIdx.x] = px; qy1[threadIdx.x] = py; qz1[threadIdx.x] = pz;
        ar1[threadIdx.x] = ar; ai1[threadIdx.x] = ai;
    }
    // this warp's box of fixed samples (every lane holds it)
    float flo[3], fhi[3];
    for (int d = 0; d < 3; ++d) {
        flo[d] = lo[d];
        fhi[d] = hi[d];
        for (int off = 16; off > 0; off >>= 1) {
            flo[d] = fminf(flo[d], __shfl_xor_sync(0xffffffffu, flo[d], off));
            fhi[d] = fmaxf(fhi[d], __shfl_xor_sync(0xffffffffu, fhi[d], off));
        }
    }
    block_bbox(lo, hi, wlo, whi, blo, bhi);
    // the moved samples lie in a ball of radius sqrt(r2max) around t
    if (threadIdx.x == 0) {
        double dd = 0.0;
        for (int d = 0; d < a.dim; ++d) {
            const double c = tv[d];
            const double e = c < blo[d] ? blo[d] - c : (c > bhi[d] ? c - bhi[d] : 0.0);
            dd += e * e;
        }
        const double reach = sqrt(a.r2max) * (1.0 + 1e-5) + cut * (1.0 + 1e-4) + 1e-6;
        skip = dd > reach * reach;
    }
    __syncthreads();
    if (skip) return;
    static_assert(RS_EXP == RS_TILE, "one table entry per thread");
    etab[threadIdx.x] = exp2(-(double)threadIdx.x / RS_EXP);  // visible after the first tile's barrier
    // tile test margin: float rounding of both boxes
    const double mag = fabs(tv[0]) + fabs(tv[1]) + fabs(tv[2]) + sqrt(a.r2max) + 1.0;
    const float cmarg = (float)(cut * (1.0 + 1e-4) + 1e-6 * mag);
    const float cm2 = cmarg * cmarg;
    const float blo0 = blo[0], blo1 = blo[1], blo2 = blo[2], bhi0 = bhi[0], bhi1 = bhi[1], bhi2 = bhi[2];
    const int ntiles = (int)((a.m2 + RS_TILE - 1) / RS_TILE);
    const float* tbase = a.tile_box + (int64_t)pose * ntiles * 6;
    const double4* moved = reinterpret_cast<const double4*>(a.moved) + (int64_t)pose * a.m2;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned short(*queue)[2] = qpair[warp];
    int qn = 0;  // entries in this warp's queue (same value in every lane)
    double sr = 0.0, si = 0.0;
    auto drain = [&](int upto) {  // evaluate queue entries [0, upto) in FP64
        for (int q0 = 0; q0 < upto; q0 += 32) {
            const int q = q0 + lane;
            if (q < upto) {
                const int fi = queue[q][0], mj = queue[q][1];
                const double dx = yx[mj] - qx1[fi], dy = yy[mj] - qy1[fi], dz = yz[mj] - qz1[fi];
                const double g = gauss_exp(dx * dx + dy * dy + dz * dz, kexp, etab);
                const double br = cr[mj] * g, bi = ci[mj] * g;
                sr += ar1[fi] * br - ai1[fi] * bi;
                si += ar1[fi] * bi + ai1[fi] * br;
            }
        }
    };
    // this CTA's share of the moving tiles (grid z splits them, so that the few
    // fixed blocks near the contact are spread over more CTAs)
    const int per = (ntiles + (int)gridDim.z - 1) / (int)gridDim.z;
    const int t_lo = (int)blockIdx.z * per, t_hi = min(ntiles, t_lo + per);
    for (int tile = t_lo; tile < t_hi; ++tile) {
        const float* tb = tbase + tile * 6;
        const float g0 = fmaxf(0.f, fmaxf(tb[0] - bhi0, blo0 - tb[3]));
        const float g1 = fmaxf(0.f, fmaxf(tb[1] - bhi1, blo1 - tb[4]));
        const float g2 = (a.dim == 3) ? fmaxf(0.f, fmaxf(tb[2] - bhi2, blo2 - tb[5])) : 0.f;
        if (g0 * g0 + g1 * g1 + g2 * g2 > cm2) continue;  // same decision in every thread
        const int64_t j = (int64_t)tile * RS_TILE + threadIdx.x;
        __syncthreads();
        {
            float mlo[3] = {FLT_MAX, FLT_MAX, FLT_MAX}, mhi[3] = {-FLT_MAX, -FLT_MAX, -FLT_MAX};
            if (j < a.m2) {
                const double4 y = moved[j];
                yx[threadIdx.x] = y.x; yy[threadIdx.x] = y.y; yz[threadIdx.x] = y.z;
                fxyz[threadIdx.x] = make_float4((float)y.x, (float)y.y, (float)y.z, 0.f);
                cr[threadIdx.x] = a.c2[j].x; ci[threadIdx.x] = a.c2[j].y;
                mlo[0] = mhi[0] = (float)y.x;
                mlo[1] = mhi[1] = (float)y.y;
                mlo[2] = mhi[2] = (float)y.z;
            }
            for (int d = 0; d < 3; ++d)
                for (int off = 16; off > 0; off >>= 1) {
                    mlo[d] = fminf(mlo[d], __shfl_down_sync(0xffffffffu, mlo[d], off));
                    mhi[d] = fmaxf(mhi[d], __shfl_down_sync(0xffffffffu, mhi[d], off));
                }
            if (lane == 0)
                for (int d = 0; d < 3; ++d) { slo[warp][d] = mlo[d]; shi[warp][d] = mhi[d]; }
        }
        __syncthreads();
        const int cnt = (int)min((int64_t)RS_TILE, a.m2 - (int64_t)tile * RS_TILE);
        for (int k = 0; k < cnt; ++k) {
            if ((k & 31) == 0) {  // skip a slice whose box is beyond the cutoff of this warp's box
                const int sl = k >> 5;
                const float h0 = fmaxf(0.f, fmaxf(slo[sl][0] - fhi[0], flo[0] - shi[sl][0]));
                const float h1 = fmaxf(0.f, fmaxf(slo[sl][1] - fhi[1], flo[1] - shi[sl][1]));
                const float h2 = (a.dim == 3) ? fmaxf(0.f, fmaxf(slo[sl][2] - fhi[2], flo[2] - shi[sl][2])) : 0.f;
                if (h0 * h0 + h1 * h1 + h2 * h2 > cm2) {  // same decision in every lane of the warp
                    k += 31;
                    continue;
                }
            }
            bool pass = false;
            if (live) {
                const float4 f = fxyz[k];
                const float dxf = f.x - pxf, dyf = f.y - pyf, dzf = f.z - pzf;
                pass = dxf * dxf + dyf * dyf + dzf * dzf <= cut2f;
            }
            const unsigned m = __ballot_sync(0xffffffffu, pass);
            if (m) {
                if (pass) {
                    const int slot = qn + __popc(m & ((1u << lane) - 1u));
                    queue[slot][0] = (unsigned short)threadIdx.x;
                    queue[slot][1] = (unsigned short)k;
                }
                qn += __popc(m);
                if (qn > RS_QUEUE - 32) {
                    __syncwarp();
                    drain(qn);
                    __syncwarp();
                    qn = 0;
                }
            }
        }
        __syncwarp();
        drain(qn);  // the tile's smem is overwritten by the next tile
        __syncwarp();
        qn = 0;
    }
    for (int off = 16; off > 0; off >>= 1) {
        sr += __shfl_down_sync(0xffffffffu, sr, off);
        si += __shfl_down_sync(0xffffffffu, si, off);
    }
    if (lane == 0) {
        atomicAdd(a.out + 2 * pose, norm * sr);
        atomicAdd(a.out + 2 * pose + 1, norm * si);
    }
}

template <typename T>
cudaError_t launch_rescore(const RescoreArgs<T>& a, cudaStream_t st) {
    cudaError_t e = cudaMemsetAsync(a.out, 0, sizeof(double) * 2 * (a.k > 0 ? a.k : 1), st);
    if (e != cudaSuccess || a.k == 0 || a.m1 == 0 || a.m2 == 0) return e;
    const unsigned ntiles = (unsigned)((a.m2 + RS_TILE - 1) / RS_TILE);
    k_rescore_move<T><<<dim3(ntiles, a.k), RS_TILE, 0, st>>>(a);
    note_launch();
    // split the moving tiles over grid z until there are about 64 CTAs per SM
    // (most CTAs find their fixed block beyond reach of the pose and return)
    static int sms = 0;
    if (sms == 0) {
        int dev = 0;
        if (cudaGetDevice(&dev) != cudaSuccess ||
            cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1)
            sms = 1;
    }
    const int64_t fixed_tiles = (a.m1 + RS_TILE - 1) / RS_TILE;
    const int64_t want = ((int64_t)64 * sms + fixed_tiles * a.k - 1) / (fixed_tiles * a.k);
    const unsigned groups = (unsigned)std::max<int64_t>(1, std::min<int64_t>({want, (int64_t)ntiles, 16}));
    const dim3 grid((unsigned)fixed_tiles, a.k, groups);
    k_rescore<T><<<grid, RS_TILE, 0, st>>>(a);
    note_launch();
    return cudaGetLastError();
}

template cudaError_t launch_rescore<float>(const RescoreArgs<float>&, cudaStream_t);
template cudaError_t launch_rescore<double>(const RescoreArgs<double>&, cudaStream_t);

int rescore_tiles(int64_t m2) { return (int)((m2 + RS_TILE - 1) / RS_TILE); }

}  // namespace sd
