// Half-spectrum inverse of the search passes.
//
// The search keeps Re f_N alone.  Re f_N is the inverse transform of the
// Hermitian part G(kappa) = (H(kappa) + conj H(-kappa)) / 2 of the product
// spectrum H = W F2, and G at kappa_x >= 0 determines it, so everything after the
// product works on half the columns:
//   fused last axis  column c = (ky, kx), kx < N/2, and its mirror c' = (-ky, -kx):
//                    conj F2(-kappa) along c' is the forward transform of the conjugated
//                    column, so both products land on the same mode kz of one line,
//                    G = W/2 FFT(x_c) + conj(W(-kappa))/2 FFT(conj x_c'), and one
//                    inverse transform serves the two;
//   inverse y        on N/2 columns (the ordinary pass);
//   inverse x        two real rows a, b as one complex line X = G_a + i G_b, extended by
//                    G(-kappa) = conj G(kappa): the line transform returns f_a + i f_b.
// A rotation's inverse work and the bytes it moves after the product are halved,
// and one inverse z transform in three goes.
#pragma once

#include "nufft_impl.cuh"

namespace sd {

// Whether a fused half pass reads its twiddles through L1 instead of shared
// memory: with them in shared memory a 384-point CTA (line buffer 49 KB, mode
// buffer 25 KB) would miss a third CTA per SM by 4 KB.  A warp's lanes walk
// columns, so each twiddle is one broadcast load.
template <typename T, int LENF>
__host__ __device__ constexpr bool half_tw_global() { return sizeof(T) == 4 && LENF == 384; }

template <typename T, int LENF, int TC>
__host__ __device__ constexpr size_t cols_half_smem() {
    return ((size_t)TC * (col_pitch(LENF) + col_pitch(LENF / 2)) +
            (half_tw_global<T, LENF>() ? 0 : tw_count(LENF) + tw_count(LENF / 2))) * sizeof(cplx<T>);
}

// TC half columns per CTA: forward transform of the columns, then of their
// conjugated mirrors, products summed in `acc`, inverse transform from there.
template <typename T, int LENF, int TC, bool PRUNED>
__device__ __forceinline__ void cols_half_body(const ColArgs<T>& a) {
    using C = cplx<T>;
    constexpr int LENI = LENF / 2, NH = LENI / 2;
    constexpr int NT = cta_threads_for<LENF>(TC);
    static_assert(NT % TC == 0, "a thread keeps one line through every stage");
    constexpr int LD = col_pitch(LENF), LDA = col_pitch(LENI);
    constexpr int NTWF = tw_count(LENF), NTWI = tw_count(LENI);
    constexpr int NB1 = LENF / plan_radix(LENF, 0);
    constexpr int PF = LENF / plan_last_radix(LENF), PI = LENI / plan_last_radix(LENI);
    constexpr bool TWG = half_tw_global<T, LENF>();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C* buf = reinterpret_cast<C*>(smem_raw);
    C* acc = buf + TC * LD;
    C* tws = acc + TC * LDA;
    const C* twF = TWG ? a.twF : tws;
    const C* twI = TWG ? a.twI : tws + NTWF;
    const bool rf = a.rot_fastest;
    const int b = rf ? (int)blockIdx.x : (int)blockIdx.z;
    // this thread's line: half column hc = ky NH + kx, its column and its mirror's
    const int ncols = a.ncols, hcols = ncols / 2;
    const int hc = (rf ? (int)blockIdx.y : (int)blockIdx.x) * TC + (int)threadIdx.x % TC;
    const bool ok = hc < hcols;
    const int ky = hc / NH, kx = hc - ky * NH;
    const int nky = ncols / LENI;  // 1 in 2D
    const C* in = a.in + (int64_t)b * a.in_rot_stride;
    const C* inA = in + ky * LENI + kx;
    const C* inB = in + (ky == 0 ? 0 : nky - ky) * LENI + (kx == 0 ? 0 : LENI - kx);
    const C* WA = a.W + hc;
    const C* WB = WA + LENI * hcols;
    C* out = a.out + (int64_t)b * a.out_rot_stride + hc;
    const int s = a.len_in;
    const C zero = mk(T(0), T(0));
    // input position of a line (pruned: cell a at position a; else the shifted sub-box)
    auto cell = [&](int i, int r) -> int {
        if constexpr (PRUNED) {
            return i + r * NB1;
        } else {
            const int e = i + r * NB1 + a.s_h;
            return e >= LENF ? e - LENF : e;
        }
    };
    // mode slot of output i + r PF, -1 where it is not kept
    auto slot = [&](int i, int r) -> int {
        if constexpr (PRUNED) {
            return kept_out<LENF>(r) ? i + kept_slot<LENF>(r) : -1;
        } else {
            const int o = i + r * PF;
            return o < LENI / 2 ? o : (o >= LENF - LENI / 2 ? o - LENI : -1);
        }
    };
    auto loadA = [&](int, int i, int r) -> C {
        const int e = cell(i, r);
        return (ok && e < s) ? inA[e * ncols] : zero;
    };
    auto emitA = [&](int line, int i, int r, C v) {
        const int kp = slot(i, r);
        if (kp >= 0 && ok) acc[line * LDA + kp] = cmul(v, WA[kp * hcols]);
    };
    auto loadB = [&](int, int i, int r) -> C {
        const int e = cell(i, r);
        return (ok && e < s) ? cconj(inB[e * ncols]) : zero;
    };
    auto emitB = [&](int line, int i, int r, C v) {  // the entries this thread wrote in emitA
        const int kp = slot(i, r);
        if (kp >= 0 && ok) {
            C* g = acc + line * LDA + kp;
            *g = cadd(*g, cmul(v, WB[kp * hcols]));
        }
    };
    auto emit_out = [&](int, int i, int r, C v) {
        if (ok) out[(i + r * PI) * hcols] = v;
    };
    if constexpr (!TWG) {
        for (int j = threadIdx.x; j < NTWF; j += NT) tws[j] = a.twF[j];
        for (int j = threadIdx.x; j < NTWI; j += NT) tws[NTWF + j] = a.twI[j];
        // visible after the barrier between the first two stages
    }
    fftp_lines<C, LENF, false, TC, NT, LAY_COL, false, false, PRUNED>(buf, LD, twF, loadA, emitA);
    // every thread has passed the barrier that follows the last stage's reads of
    // buf, so the second transform may overwrite it
    if constexpr (plan_radix(LENF, 1) == 0) __syncthreads();
    fftp_lines<C, LENF, false, TC, NT, LAY_COL, false, false, PRUNED>(buf, LD, twF, loadB, emitB);
    __syncthreads();
    fftp_lines<C, LENI, true, TC, NT, LAY_COL, false, true, false>(acc, LDA, twI, loadA, emit_out);
}

template <typename T, int LENF, int MB, int TC, bool PRUNED>
__global__ void __launch_bounds__(cta_threads_for<LENF>(TC), MB) k_cols_half(ColArgs<T> a) {
    cols_half_body<T, LENF, TC, PRUNED>(a);
}

// Inverse x of two real rows per line.  src: G_a (LEN/2 modes), then G_b.
// Input p of the complex line: G_a + i G_b below the Nyquist slot, conj G_a + i conj G_b
// of mode LEN - p above it; mode 0 is real, the Nyquist slot zero.
template <typename C, int LEN>
__device__ __forceinline__ C half_line_input(const C* src, int i, int r) {
    using T = decltype(C{}.x);
    constexpr int R1 = plan_radix(LEN, 0), NB1 = LEN / R1, H = LEN / 2;
    static_assert(R1 % 2 == 0, "first radix must be even");
    if (r < R1 / 2) {
        const int p = i + r * NB1;
        const C ga = src[p], gb = src[H + p];
        if (r == 0 && i == 0) return mk(ga.x, gb.x);
        return mk(ga.x - gb.y, ga.y + gb.x);
    }
    if (r == R1 / 2 && i == 0) return mk(T(0), T(0));
    const int q = LEN - (i + r * NB1);
    const C ga = src[q], gb = src[H + q];
    return mk(ga.x + gb.y, gb.x - ga.y);
}

constexpr int HALF_ROW_WAVE = 24;  // CTAs per SM a row pass leaves before its CTAs take more groups

// Row groups of TR lines (2 TR rows) handled by one CTA in turn: its K best are
// kept in registers across the groups and merged once.
template <typename T, int LEN, int K>
__device__ __forceinline__ void rows_half_body(const RowArgs<T>& a) {
    using C = cplx<T>;
    constexpr int TR = lines_per_cta<T, LEN>();
    constexpr int NT = cta_threads<T, LEN>();
    constexpr int LD = line_pitch(LEN);
    constexpr int NTW = tw_count(LEN);
    constexpr int PL = LEN / plan_last_radix(LEN);
    constexpr bool one_bfly = TR * (LEN / plan_last_radix(LEN)) <= NT;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C* buf = reinterpret_cast<C*>(smem_raw);
    C* tw = buf + TR * LD;
    for (int j = threadIdx.x; j < NTW; j += NT) tw[j] = a.tw[j];  // visible from the second stage on
    const C* in = a.in + (int64_t)blockIdx.y * a.in_rot_stride;
    const int nlines = a.nrows / 2, ngroups = (nlines + TR - 1) / TR;
    const C zero = mk(T(0), T(0));
    T bestA = -INFINITY, bestB = -INFINITY;
    int idxA = INT_MAX, idxB = INT_MAX;
    TopK<T, K> top;
    if constexpr (K > 1) top.init();
    for (int g = blockIdx.x; g < ngroups; g += gridDim.x) {
        const int line0 = g * TR;
        const int nl = nlines - line0;
        const C* src = in + (int64_t)line0 * LEN;
        auto load = [&](int line, int i, int r) -> C {
            return line < nl ? half_line_input<C, LEN>(src + line * LEN, i, r) : zero;
        };
        auto emit = [&](int line, int i, int r, C v) {
            if (line >= nl) return;
            const int o = 2 * (line0 + line) * LEN + i + r * PL;
            if constexpr (K > 1) {
                top.push(v.x, o);
                top.push(v.y, o + LEN);
            } else if constexpr (one_bfly) {
                // outputs (and groups) come in increasing index order: a strict
                // comparison keeps the lowest index of equal values
                if (v.x > bestA) { bestA = v.x; idxA = o; }
                if (v.y > bestB) { bestB = v.y; idxB = o + LEN; }
            } else {
                argmax_merge(bestA, idxA, v.x, o);
                argmax_merge(bestB, idxB, v.y, o + LEN);
            }
        };
        fftp_lines<C, LEN, true, TR, NT, LAY_ROW, true, false, false>(buf, LD, tw, load, emit);
        // the next group's first writes to buf come after the barrier that follows
        // this group's last reads
    }
    if constexpr (K > 1) {
        T* sv = reinterpret_cast<T*>(tw + NTW);
        int* si = reinterpret_cast<int*>(sv + NT * K);
        __shared__ T wv[32], bestv[K];
        __shared__ int wi[32], besti[K];
        block_topk_merge<T, K>(top, sv, si, wv, wi, bestv, besti);
        if (threadIdx.x < K) {
            const int64_t o = ((int64_t)blockIdx.y * gridDim.x + blockIdx.x) * K + threadIdx.x;
            a.part_score[o] = (double)bestv[threadIdx.x];
            a.part_idx[o] = besti[threadIdx.x];
        }
    } else {
        argmax_merge(bestA, idxA, bestB, idxB);
        block_argmax(bestA, idxA);
        if (threadIdx.x == 0) {
            const int64_t o = (int64_t)blockIdx.y * gridDim.x + blockIdx.x;
            a.part_score[o] = (double)bestA;
            a.part_idx[o] = idxA;
        }
    }
}

template <typename T, int LEN, int K>
__global__ void __launch_bounds__(cta_threads<T, LEN>(), K == 1 ? rows_inv_min_ctas<T, LEN>() : 0)
k_rows_half(RowArgs<T> a) {
    rows_half_body<T, LEN, K>(a);
}

// The two halves of the table: W(kappa) / 2 and conj W(-kappa) / 2 times the phase of
// an unshifted sub-box, exp(2 pi i s_h sum kappa / n) (the mirror's conjugated phase
// at -kappa is the same).  The Nyquist slots are zero in W.
template <typename T>
__global__ void k_whalf(const cplx<T>* W, int N, int dim, int n, int s_h, cplx<T>* out) {
    const int NH = N / 2;
    const int64_t tot = (dim == 2) ? (int64_t)N * NH : (int64_t)N * N * NH;
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= tot) return;
    const int kx = (int)(i % NH);
    int64_t r = i / NH;
    const int ky = (int)(r % N);
    const int kz = (dim == 3) ? (int)(r / N) : 0;
    auto sgn = [&](int k) { return k < NH ? k : k - N; };
    const int64_t ksum = kx + sgn(ky) + (dim == 3 ? sgn(kz) : 0);
    int64_t e = (ksum * s_h) % n;
    if (e < 0) e += n;
    double sn, cs;
    sincospi(2.0 * (double)e / (double)n, &sn, &cs);
    cs *= 0.5;
    sn *= 0.5;
    const int mx = kx ? N - kx : 0, my = ky ? N - ky : 0, mz = kz ? N - kz : 0;
    const cplx<T> wa = W[((int64_t)kz * N + ky) * N + kx], wb = W[((int64_t)mz * N + my) * N + mx];
    const double ar = wa.x, ai = wa.y, br = wb.x, bi = -(double)wb.y;
    out[i] = mk(T(ar * cs - ai * sn), T(ar * sn + ai * cs));
    out[tot + i] = mk(T(br * cs - bi * sn), T(br * sn + bi * cs));
}

// ---------------------------------------------------------------------------

template <typename T, int LENF, int TC, int MB, bool PRUNED>
static cudaError_t cols_half_launch(const ColArgs<T>& a, int batch, cudaStream_t st) {
    const int hcols = a.ncols / 2;
    const int nb = (hcols + TC - 1) / TC;
    if (nb == 0 || batch == 0) return cudaSuccess;
    if (a.nouter != 1 || a.N != LENF / 2 || a.ncols % a.N != 0) return cudaErrorInvalidValue;
    auto kern = k_cols_half<T, LENF, MB, TC, PRUNED>;
    constexpr size_t smem = cols_half_smem<T, LENF, TC>();
    cudaError_t e = set_smem(kern, smem);
    if (e != cudaSuccess) return e;
    const bool rf = a.rot_fastest;
    if (rf && nb > 65535) return cudaErrorInvalidValue;
    kern<<<rf ? dim3(batch, nb, 1) : dim3(nb, 1, batch), cta_threads_for<LENF>(TC), smem, st>>>(a);
    note_launch();
    return cudaGetLastError();
}

template <typename T, int LENF>
static cudaError_t cols_half_pruned(const ColArgs<T>& a, int batch, cudaStream_t st) {
    static_assert(prunable_len(LENF), "length not prunable");
    if constexpr (alt_cols_ok<T, LENF>()) {
        if (a.lines == LINES_NARROW)
            return cols_half_launch<T, LENF, alt_lines<T, LENF, 0>(), alt_min_ctas<T, LENF, 2, 0>(), true>(a, batch, st);
        if (a.lines == LINES_WIDE)
            return cols_half_launch<T, LENF, alt_lines<T, LENF, 1>(), alt_min_ctas<T, LENF, 2, 1>(), true>(a, batch, st);
    }
    if (a.lines != LINES_STD) return cudaErrorInvalidValue;
    return cols_half_launch<T, LENF, lines_per_cta<T, LENF>(), pruned_min_ctas<T, LENF, 2>(), true>(a, batch, st);
}

template <typename T>
cudaError_t launch_cols_half_t(bool pruned, const ColArgs<T>& a, int batch, cudaStream_t st) {
    if (pruned) {
        switch (a.n) {
#define SD_HALFP_CASE(L) \
    case L: return cols_half_pruned<T, L>(a, batch, st);
            SD_FOR_EACH_PLEN(SD_HALFP_CASE)
#undef SD_HALFP_CASE
        }
        return cudaErrorInvalidValue;
    }
    switch (a.n) {
#define SD_HALFF_CASE(L) \
    case L: return cols_half_launch<T, L, lines_per_cta<T, L>(), min_ctas_per_sm<T, L>(), false>(a, batch, st);
        SD_HALFF_CASE(16) SD_HALFF_CASE(32) SD_HALFF_CASE(48) SD_HALFF_CASE(64) SD_HALFF_CASE(96)
        SD_HALFF_CASE(128) SD_HALFF_CASE(192) SD_HALFF_CASE(256) SD_HALFF_CASE(384) SD_HALFF_CASE(512)
#undef SD_HALFF_CASE
    }
    return cudaErrorInvalidValue;
}

template <typename T, int LEN, int K>
static cudaError_t rows_half_launch(const RowArgs<T>& a, int batch, int* nparts, cudaStream_t st) {
    constexpr int TR = lines_per_cta<T, LEN>();
    constexpr int NT = cta_threads<T, LEN>();
    if (a.nrows % 2 != 0 || a.N != LEN) return cudaErrorInvalidValue;
    const int ngroups = (a.nrows / 2 + TR - 1) / TR;
    if (nparts) *nparts = 0;
    if (ngroups == 0 || batch == 0) return cudaSuccess;
    // groups per CTA: enough to amortise its merge, few enough to leave several
    // waves of CTAs (the K-best merge costs about as much as a group's transform)
    const int64_t total = (int64_t)ngroups * batch;
    int G = (int)(total / (HALF_ROW_WAVE * 152));
    G = G < 1 ? 1 : (G > 8 ? 8 : G);
    const int nb = (ngroups + G - 1) / G;
    if (nparts) *nparts = nb * K;
    const size_t smem = (size_t)(TR * line_pitch(LEN) + tw_count(LEN)) * sizeof(cplx<T>) +
                        (K > 1 ? (size_t)NT * K * (sizeof(T) + sizeof(int)) : 0);
    auto kern = k_rows_half<T, LEN, K>;
    cudaError_t e = set_smem(kern, smem);
    if (e != cudaSuccess) return e;
    kern<<<dim3(nb, batch), NT, smem, st>>>(a);
    note_launch();
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_rows_half_t(int keep, const RowArgs<T>& a, int batch, int* nparts, cudaStream_t st) {
    switch (a.N) {
#define SD_HALFR_CASE(L)                                                            \
    case L:                                                                         \
        switch (keep) {                                                             \
            case 1: return rows_half_launch<T, L, 1>(a, batch, nparts, st);         \
            case 2: return rows_half_launch<T, L, 2>(a, batch, nparts, st);         \
            case 4: return rows_half_launch<T, L, 4>(a, batch, nparts, st);         \
            case 8: return rows_half_launch<T, L, 8>(a, batch, nparts, st);         \
            case 16: return rows_half_launch<T, L, 16>(a, batch, nparts, st);       \
        }                                                                           \
        break;
        SD_HALFR_CASE(8) SD_HALFR_CASE(16) SD_HALFR_CASE(24) SD_HALFR_CASE(32) SD_HALFR_CASE(48) SD_HALFR_CASE(64)
        SD_HALFR_CASE(96) SD_HALFR_CASE(128) SD_HALFR_CASE(192) SD_HALFR_CASE(256)
#undef SD_HALFR_CASE
    }
    return cudaErrorInvalidValue;
}

template <typename T>
cudaError_t launch_whalf_t(const cplx<T>* W, int N, int dim, int n, int s_h, cplx<T>* out, cudaStream_t st) {
    const int64_t tot = (dim == 2) ? (int64_t)N * N / 2 : (int64_t)N * N * N / 2;
    k_whalf<T><<<(unsigned)((tot + 255) / 256), 256, 0, st>>>(W, N, dim, n, s_h, out);
    note_launch();
    return cudaGetLastError();
}

}  // namespace sd

#define SD_INSTANTIATE_HALF(T)                                                                                 \
    namespace sd {                                                                                             \
    template <> cudaError_t launch_cols_half<T>(bool pruned, const ColArgs<T>& a, int batch, cudaStream_t st) { \
        return launch_cols_half_t<T>(pruned, a, batch, st);                                                    \
    }                                                                                                          \
    template <> cudaError_t launch_rows_half<T>(int keep, const RowArgs<T>& a, int batch, int* np, cudaStream_t st) { \
        return launch_rows_half_t<T>(keep, a, batch, np, st);                                                  \
    }                                                                                                          \
    template <> cudaError_t launch_whalf<T>(const cplx<T>* W, int N, int dim, int n, int s_h, cplx<T>* out,     \
                                            cudaStream_t st) {                                                 \
        return launch_whalf_t<T>(W, N, dim, n, s_h, out, st);                                                  \
    }                                                                                                          \
    }
