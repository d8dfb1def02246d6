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
//   inverse y        on N/2 columns; its last stage holds outputs y and y + N/2 of a
//                    column in one thread and writes them as the modes kappa and -kappa
//                    of one complex line X = G_y + i G_(y + N/2), X(-kappa) = conj G_y + i conj G_(y + N/2)
//   inverse x        a plain line transform of X: f_y + i f_(y + N/2)
// A rotation's inverse work and the bytes it moves after the product are halved,
// and one inverse z transform in three goes.
#pragma once

#include "nufft_impl.cuh"

namespace sd {

// Twiddles in shared memory where that costs no resident CTA: a 384-point CTA (line
// buffer 49 KB, mode buffer 25 KB) would miss its third, and 512 points (99 KB)
// measured faster through L1 (12 rotations at N = 256: 894 against 1038 us; 256 points
// the other way, 68 rotations at N = 128: 562 against 524).
template <int LENF>
__host__ __device__ constexpr bool half_tw_smem() { return LENF <= 256; }
// Asynchronous copies of the table (W) and of the mirror column (B, see the body) hide
// a global latency each, but take registers and address arithmetic.  Fused pass, us, with
// neither / B only / W only / both: 192 points (64 rotations, N = 96) - / 256 / 271 / 255;
// 256 points (68, N = 128) 652 / - / 552 / 568; 384 points (60, N = 192) 1904 / 2003 /
// 1992 / 2081; 512 points (12, N = 256) - / 948 / - / 995.
template <int LENF>
__host__ __device__ constexpr bool half_prefetch_w() { return LENF <= 256; }
template <int LENF>
__host__ __device__ constexpr bool half_prefetch_b() { return LENF != 256 && LENF != 384; }

// Lines per CTA of the passes' form for few CTAs (2D jobs of few rotations), and whether it
// pays against `ctas` CTAs of `lines` lines each.  Half a spectrum is half the lines, and
// CTAs of 16 that leave SMs idle take as long as before or, with a transform more in the
// chain, longer.  An FP64 CTA keeps its SM's pipe busy by itself, so the count of waves
// decides, the smaller CTAs' at 1.15 (1.05 to 1.18 measured).
constexpr int FEW_LINES = 4;
inline bool few_pays(int64_t ctas, int lines) {
    auto waves = [](int64_t n) { return (double)((n + GPU_SMS - 1) / GPU_SMS); };
    const int split = lines / FEW_LINES;
    return 1.15 * waves(ctas * split) < split * waves(ctas);
}

template <typename T, int LENF, int TC>
__host__ __device__ constexpr size_t cols_half_smem() {
    return ((size_t)TC * (col_pitch(LENF) + col_pitch(LENF / 2)) +
            (half_tw_smem<LENF>() ? tw_count(LENF) + tw_count(LENF / 2) : 0)) * sizeof(cplx<T>);
}

// One complex element from global to shared memory without a register.
template <typename C>
__device__ __forceinline__ void copy_async(C* dst, const C* src) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(d), "l"(src), "n"((int)sizeof(C)) : "memory");
}
__device__ __forceinline__ void copy_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void copy_wait() { asm volatile("cp.async.wait_group 0;" ::: "memory"); }

// Last-stage emitter of an inverse column transform of LEN points that packs
// outputs o and o + LEN/2 (radix R even: both in one butterfly) into line o of
// packed rows: out = packed line 0, kx the column's mode.
template <typename C, int LEN>
struct PackEmit {
    static constexpr int R = plan_last_radix(LEN), PL = LEN / R;
    static_assert(R % 2 == 0, "a butterfly must hold outputs half a line apart");
    C* out;
    int kx;
    bool ok;
    C low[R / 2];
    __device__ __forceinline__ void operator()(int, int i, int r, C v) {
        using T = decltype(C{}.x);
        if (r < R / 2) {
            low[r] = v;
            return;
        }
        if (!ok) return;
        const C ga = low[r - R / 2];
        C* line = out + (int64_t)(i + (r - R / 2) * PL) * LEN;
        if (kx == 0) {  // a real mode, and the Nyquist slot
            line[0] = mk(ga.x, v.x);
            line[LEN / 2] = mk(T(0), T(0));
        } else {
            line[kx] = mk(ga.x - v.y, ga.y + v.x);
            line[LEN - kx] = mk(ga.x + v.y, v.x - ga.y);
        }
    }
};

// TC half columns per CTA: forward transform of the columns, then of their
// conjugated mirrors, products summed in `acc`, inverse transform from there.
template <typename T, int LENF, int TC, bool PRUNED, bool PACK>
__device__ __forceinline__ void cols_half_body(const ColArgs<T>& a) {
    using C = cplx<T>;
    constexpr int LENI = LENF / 2, NH = LENI / 2;
    constexpr int NT = cta_threads_for<LENF>(TC);
    static_assert(NT % TC == 0, "a thread keeps one line through every stage");
    constexpr int LD = col_pitch(LENF), LDA = col_pitch(LENI);
    constexpr int NB1 = LENF / plan_radix(LENF, 0);
    constexpr int PFL = LENF / plan_last_radix(LENF), PI = LENI / plan_last_radix(LENI);
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C* buf = reinterpret_cast<C*>(smem_raw);
    C* acc = buf + TC * LD;
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
    C* out = a.out + (int64_t)b * a.out_rot_stride;
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
    // mode slot of output i + r PFL, -1 where it is not kept
    auto slot = [&](int i, int r) -> int {
        if constexpr (PRUNED) {
            return kept_out<LENF>(r) ? i + kept_slot<LENF>(r) : -1;
        } else {
            const int o = i + r * PFL;
            return o < LENI / 2 ? o : (o >= LENF - LENI / 2 ? o - LENI : -1);
        }
    };
    constexpr bool PFW = half_prefetch_w<LENF>(), PFB = half_prefetch_b<LENF>();
    constexpr int R1 = plan_radix(LENF, 0), RL = plan_last_radix(LENF), RIN = PRUNED ? R1 / 2 : R1;
    const int line = (int)threadIdx.x % TC;
    const C *twF = a.twF, *twI = a.twI;
    if constexpr (half_tw_smem<LENF>()) {
        C* tws = acc + TC * LDA;
        for (int j = threadIdx.x; j < tw_count(LENF); j += NT) tws[j] = a.twF[j];
        for (int j = threadIdx.x; j < tw_count(LENI); j += NT) tws[tw_count(LENF) + j] = a.twI[j];
        twF = tws;
        twI = tws + tw_count(LENF);
    }
    // The mirror column's cells wait in buf (cell e of a line at e TC + line), the
    // first table half in the mode slots of acc it is multiplied into: both are
    // copied by the thread that reads them.
    auto loadA = [&](int, int i, int r) -> C {
        const int e = cell(i, r);
        return (ok && e < s) ? inA[e * ncols] : zero;
    };
    auto fetchW = [&] {
#pragma unroll
        for (int q = 0; q < (TC * PFL + NT - 1) / NT; ++q) {
            const int t = threadIdx.x + q * NT;
            if (ok && t < TC * PFL)
#pragma unroll
                for (int r = 0; r < RL; ++r) {
                    const int kp = slot(t / TC, r);
                    if (kp >= 0) copy_async(acc + line * LDA + kp, WA + kp * hcols);
                }
        }
        copy_commit();
    };
    auto fetchB = [&] {
#pragma unroll
        for (int q = 0; q < (TC * NB1 + NT - 1) / NT; ++q) {
            const int t = threadIdx.x + q * NT;
            if (ok && t < TC * NB1)
#pragma unroll
                for (int r = 0; r < RIN; ++r) {
                    const int e = cell(t / TC, r);
                    if (e < s) copy_async(buf + e * TC + line, inB + e * ncols);
                }
        }
        copy_commit();
    };
    auto emitA = [&](int, int i, int r, C v) {
        const int kp = slot(i, r);
        if (kp >= 0 && ok) {
            C* g = acc + line * LDA + kp;
            *g = cmul(v, PFW ? *g : WA[kp * hcols]);
        }
    };
    auto loadB = [&](int, int i, int r) -> C {
        const int e = cell(i, r);
        if (PFB) return (ok && e < s) ? cconj(buf[e * TC + line]) : zero;
        return (ok && e < s) ? cconj(inB[e * ncols]) : zero;
    };
    auto emitB = [&](int, int i, int r, C v) {  // the entries this thread wrote in emitA
        const int kp = slot(i, r);
        if (kp >= 0 && ok) {
            C* g = acc + line * LDA + kp;
            *g = cadd(*g, cmul(v, WB[kp * hcols]));
        }
    };
    fftp_lines<C, LENF, false, TC, NT, LAY_COL, false, false, PRUNED>(buf, LD, twF, loadA, emitA,
                                                                      Hooks(
                                                                          [&] {
                                                                              if constexpr (PFW) fetchW();
                                                                          },
                                                                          [&] {
                                                                              if constexpr (PFW) copy_wait();
                                                                              if constexpr (PFB) fetchB();
                                                                          }));
    if constexpr (PFB) copy_wait();
    // with copies, the barrier of loaded(): every thread has read its cells before buf is rewritten
    fftp_lines<C, LENF, false, TC, NT, LAY_COL, false, false, PRUNED>(buf, LD, twF, loadB, emitB, LoadedHook([] {
                                                                          if constexpr (PFB) __syncthreads();
                                                                      }));
    __syncthreads();
    if constexpr (PACK) {
        PackEmit<C, LENI> emit_out{out, kx, ok};
        fftp_lines<C, LENI, true, TC, NT, LAY_COL, false, true, false>(acc, LDA, twI, loadA, emit_out);
    } else {
        auto emit_out = [&](int, int i, int r, C v) {
            if (ok) out[(i + r * PI) * hcols + hc] = v;
        };
        fftp_lines<C, LENI, true, TC, NT, LAY_COL, false, true, false>(acc, LDA, twI, loadA, emit_out);
    }
}

template <typename T, int LENF, int MB, int TC, bool PRUNED, bool PACK>
__global__ void __launch_bounds__(cta_threads_for<LENF>(TC), MB) k_cols_half(ColArgs<T> a) {
    cols_half_body<T, LENF, TC, PRUNED, PACK>(a);
}

// The packing pass for launches of few CTAs (2D): FEW_LINES half columns per CTA, each
// column and its mirror transformed by threads of their own at the same time, so the
// chain is two transforms long where cols_half_body's is three.  us a launch by 16 (FP64
// from 384 points 8) columns a CTA / this: FP64 N = 128 20 CTAs 74 / 29 (the full
// spectrum's pass 45), 96 CTAs 74 / 61, 128 74 / 80, 192 (N = 96) 106 / 88; FP32, whose
// SMs hold several CTAs, N = 192 30 CTAs 11.7 / 7.6, 72 11.8 / 9.8, 108 even, N = 128 72
// CTAs 9.7 / 7.8, 128 9.6 / 10.1.
template <typename T, int LENF>
__host__ __device__ constexpr size_t cols_few_smem() {
    return (size_t)2 * FEW_LINES * (col_pitch(LENF) + col_pitch(LENF / 2)) * sizeof(cplx<T>);
}
template <typename T, int LENF, bool PRUNED>
__global__ void __launch_bounds__(cta_threads_for<LENF>(2 * FEW_LINES)) k_cols_few(ColArgs<T> a) {
    using C = cplx<T>;
    constexpr int LENI = LENF / 2, NH = LENI / 2, TC = FEW_LINES, NL = 2 * TC;
    constexpr int NT = cta_threads_for<LENF>(NL);
    static_assert(NT % NL == 0, "a thread keeps one line through the forward stages");
    constexpr int LD = col_pitch(LENF), LDA = col_pitch(LENI);
    constexpr int NB1 = LENF / plan_radix(LENF, 0);
    constexpr int RL = plan_last_radix(LENF), PFL = LENF / RL;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C* buf = reinterpret_cast<C*>(smem_raw);
    C* acc = buf + NL * LD;
    const int line = (int)threadIdx.x % NL;
    const bool mirror = line >= TC;
    const int kx = (int)blockIdx.x * TC + line % TC;
    const bool ok = kx < NH;
    const C* in = a.in + (int64_t)blockIdx.z * a.in_rot_stride + (mirror && kx ? LENI - kx : kx);
    const C* W = a.W + kx + (mirror ? LENI * NH : 0);
    C* out = a.out + (int64_t)blockIdx.z * a.out_rot_stride;
    const int s = a.len_in;
    const C zero = mk(T(0), T(0));
    // as in cols_half_body: the input position, and the mode slot of an output
    auto slot = [&](int i, int r) -> int {
        if constexpr (PRUNED) {
            return kept_out<LENF>(r) ? i + kept_slot<LENF>(r) : -1;
        } else {
            const int o = i + r * PFL;
            return o < NH ? o : (o >= LENF - NH ? o - LENI : -1);
        }
    };
    auto load = [&](int, int i, int r) -> C {
        int e = i + r * NB1;
        if constexpr (!PRUNED) {
            e += a.s_h;
            if (e >= LENF) e -= LENF;
        }
        const C v = (ok && e < s) ? in[e * LENI] : zero;
        return mirror ? cconj(v) : v;
    };
    // the table's entries wait in the slots they are multiplied into
    auto fetchW = [&] {
#pragma unroll
        for (int q = 0; q < (NL * PFL + NT - 1) / NT; ++q) {
            const int t = threadIdx.x + q * NT;
            if (t < NL * PFL)
#pragma unroll
                for (int r = 0; r < RL; ++r) {
                    const int kp = slot(t / NL, r);
                    if (kp < 0) continue;
                    if (ok) copy_async(acc + line * LDA + kp, W + kp * NH);
                    else acc[line * LDA + kp] = zero;
                }
        }
        copy_commit();
    };
    auto emit = [&](int, int i, int r, C v) {
        const int kp = slot(i, r);
        if (kp >= 0 && ok) {
            C* g = acc + line * LDA + kp;
            *g = cmul(v, *g);
        }
    };
    fftp_lines<C, LENF, false, NL, NT, LAY_COL, false, false, PRUNED>(buf, LD, a.twF, load, emit,
                                                                      Hooks([&] { fetchW(); }, [&] { copy_wait(); }));
    __syncthreads();
    constexpr int NBI = LENI / plan_radix(LENI, 0);
    auto sum = [&](int l, int i, int r) -> C {
        const int p = i + r * NBI;
        return cadd(acc[l * LDA + p], acc[(l + TC) * LDA + p]);
    };
    const int kxi = (int)blockIdx.x * TC + (int)threadIdx.x % TC;
    PackEmit<C, LENI> emit_out{out, kxi, kxi < NH};
    fftp_lines<C, LENI, true, TC, NT, LAY_COL, false, false, false>(buf, LDA, a.twI, sum, emit_out);
}

// Inverse y of half a spectrum (3D): columns (z, kx) of N points from the half
// volume to packed lines.
template <typename T, int LEN>
__global__ void __launch_bounds__(cta_threads<T, LEN>(), rows_inv_min_ctas<T, LEN>()) k_pack_y(ColArgs<T> a) {
    using C = cplx<T>;
    constexpr int TC = lines_per_cta<T, LEN>();
    constexpr int NT = cta_threads<T, LEN>();
    static_assert(NT % TC == 0, "a thread keeps one line through every stage");
    constexpr int LD = col_pitch(LEN), NH = LEN / 2;
    constexpr int NB1 = LEN / plan_radix(LEN, 0);
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C* buf = reinterpret_cast<C*>(smem_raw);
    const int kx = blockIdx.x * TC + (int)threadIdx.x % TC;
    const bool ok = kx < NH;
    const C* in = a.in + (int64_t)blockIdx.z * a.in_rot_stride + (int64_t)blockIdx.y * (LEN * NH) + kx;
    const C zero = mk(T(0), T(0));
    auto load = [&](int, int i, int r) -> C { return ok ? in[(i + r * NB1) * NH] : zero; };
    PackEmit<C, LEN> emit{a.out + (int64_t)blockIdx.z * a.out_rot_stride + (int64_t)blockIdx.y * (LEN * NH), kx, ok};
    fftp_lines<C, LEN, true, TC, NT, LAY_COL, false, false, false>(buf, LD, a.twI, load, emit);
}

// A row pass leaves this many CTAs per SM before its CTAs take more groups, up to a
// most each: the copies then run ahead, and a K-best merge (K block-wide rounds) is
// paid once.  (77 rotations at N = 96 keeping four: 133 us at 8 CTAs per SM and 32
// groups, 160 at 16 and 16.)
template <int K>
__host__ __device__ constexpr int half_row_wave() { return K == 1 ? 16 : 8; }
template <int K>
__host__ __device__ constexpr int half_row_most() { return K == 1 ? 16 : 32; }
// Resident CTAs a SM the row pass is compiled for (0: the compiler's choice): a bound
// only where it measured faster, us of the pass without a bound / as chosen.  FP32, one
// candidate: four, 64 registers (64 rotations at N = 128 148 / 144), but 192 points spill
// under it (60 rotations 516 at four / 457).  Two: none (60 at 192 858 at five / 605).
// Four: five at 96 points (64 rotations 131 / 106), four at 192 (60: 1,089 / 962).  More
// keep their lists in registers.  FP64 two, below 64 points three: the pipe bounds it, and
// the compiler's own 110 to 150 registers leave 192 points one CTA (15 rotations 3,166 /
// 2,999) and 48 points two (48 rotations 154 / 137); elsewhere they are even, where four
// and five spilled up to 3 KB (128 points keeping two 1,067 / 1,022).
template <typename T, int LEN, int K>
__host__ __device__ constexpr int rows_half_min_ctas() {
    if (K > 4) return 0;
    if (sizeof(T) == 8) return LEN < 64 ? 3 : 2;
    if (K == 1) return LEN == 192 ? 0 : 4;
    if (K == 4) return LEN == 96 ? 5 : (LEN == 192 ? 4 : 0);
    return 0;
}

// Inverse x of packed lines.  Row groups of TR lines (2 TR rows) are handled by one
// CTA in turn: its K best are kept in registers across the groups and merged once.
// Whether a row pass's groups are copied in ahead (two-stage FP32 lines; an FP64
// CTA's raw lines would cost it its shared memory).
template <typename T, int LEN>
__host__ __device__ constexpr bool rows_half_ahead() {
    return sizeof(T) == 4 && plan_radix(LEN, 1) != 0;
}
template <typename T, int LEN, int K, int TR>
__host__ __device__ constexpr size_t rows_half_smem() {
    constexpr int NT = cta_threads_for<LEN>(TR);
    return (size_t)(TR * ((rows_half_ahead<T, LEN>() ? LEN : 0) + line_pitch(LEN)) + tw_count(LEN)) * sizeof(cplx<T>) +
           (K > 1 ? (size_t)NT * K * (sizeof(T) + sizeof(int)) : 0);
}

// Sixteen bytes from global to shared memory without a register and past L1.
__device__ __forceinline__ void copy_async16(void* dst, const void* src) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(src) : "memory");
}

__device__ __forceinline__ float max_num(float a, float b) { return fmaxf(a, b); }
__device__ __forceinline__ double max_num(double a, double b) { return a > b || b != b ? a : b; }  // as fmax, but cheap

template <typename T, int LEN, int K, int TR>
__device__ __forceinline__ void rows_half_body(const RowArgs<T>& a) {
    using C = cplx<T>;
    constexpr int NT = cta_threads_for<LEN>(TR);
    constexpr int LD = line_pitch(LEN);
    constexpr int NTW = tw_count(LEN);
    constexpr int NB1 = LEN / plan_radix(LEN, 0);
    constexpr int RL = plan_last_radix(LEN), PL = LEN / RL;
    constexpr bool AHEAD = rows_half_ahead<T, LEN>();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C* raw = reinterpret_cast<C*>(smem_raw);
    C* buf = raw + (AHEAD ? TR * LEN : 0);
    C* tw = buf + TR * LD;
    constexpr int NH = LEN / 2;
    const C* in = a.in + (int64_t)blockIdx.y * a.in_rot_stride;
    const int nlines = a.nrows / 2, ngroups = (nlines + TR - 1) / TR;
    // a group's lines are contiguous (and a line is a multiple of 16 bytes): the CTA's
    // threads copy the next group in while this one is in its second stage
    auto fetch = [&](int g) {
        if (g < ngroups) {
            const int quads = min(TR, nlines - g * TR) * (int)(LEN * sizeof(C) / 16);
            const float4* src = reinterpret_cast<const float4*>(in + (int64_t)g * TR * LEN);
            for (int t = threadIdx.x; t < quads; t += NT) copy_async16(reinterpret_cast<float4*>(raw) + t, src + t);
        }
        copy_commit();
    };
    if constexpr (AHEAD) fetch(blockIdx.x);
    TwStage<C, NTW, NT> tws;
    tws.load(a.tw);
    const C zero = mk(T(0), T(0));
    T bestA = -INFINITY, bestB = -INFINITY;
    int idxA = INT_MAX, idxB = INT_MAX;
    TopK<T, K> top;
    if constexpr (K > 1) top.init();
    C keep[RL];
    for (int g = blockIdx.x; g < ngroups; g += gridDim.x) {
        const int line0 = g * TR;
        const int nl = nlines - line0;
        const C* src = in + (int64_t)line0 * LEN;
        if constexpr (AHEAD) {  // every thread's share has landed
            copy_wait();
            __syncthreads();
        }
        auto load = [&](int line, int i, int r) -> C {
            return line < nl ? (AHEAD ? raw : src)[line * LEN + i + r * NB1] : zero;
        };
        // a butterfly's outputs are kept until all are there: one maximum each, and the
        // comparisons with what the thread holds only where that maximum could enter it
        auto emit = [&](int line, int i, int r, C v) {
            keep[r] = v;
            if (r < RL - 1 || line >= nl) return;
            T mA = keep[0].x, mB = keep[0].y;
#pragma unroll
            for (int q = 1; q < RL; ++q) {
                mA = max_num(mA, keep[q].x);
                mB = max_num(mB, keep[q].y);
            }
            // line (z, y), y < N/2, holds rows (z, y) and (z, y + N/2)
            const int l = line0 + line, o = (l + l / NH * NH) * LEN + i;
            if constexpr (K > 1) {
                if (mA >= top.v[K - 1])
#pragma unroll
                    for (int q = 0; q < RL; ++q) top.push(keep[q].x, o + q * PL);
                if (mB >= top.v[K - 1])
#pragma unroll
                    for (int q = 0; q < RL; ++q) top.push(keep[q].y, o + NH * LEN + q * PL);
            } else {
                // a thread's outputs (and groups) come in increasing index order: strict
                // comparisons keep the lowest index of equal values
                if (mA > bestA) {
#pragma unroll
                    for (int q = 0; q < RL; ++q)
                        if (keep[q].x > bestA) { bestA = keep[q].x; idxA = o + q * PL; }
                }
                if (mB > bestB) {
#pragma unroll
                    for (int q = 0; q < RL; ++q)
                        if (keep[q].y > bestB) { bestB = keep[q].y; idxB = o + NH * LEN + q * PL; }
                }
            }
        };
        fftp_lines<C, LEN, true, TR, NT, LAY_ROW, true, false, false>(
            buf, LD, tw, load, emit,
            StagedHooks(
                [&] {
                    if (g == (int)blockIdx.x) tws.store(tw);
                },
                [&] {
                    if constexpr (AHEAD) fetch(g + gridDim.x);
                }));
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

template <typename T, int LEN, int K, int TR>
__global__ void __launch_bounds__(cta_threads_for<LEN>(TR), TR == FEW_LINES ? 0 : rows_half_min_ctas<T, LEN, K>())
k_rows_half(RowArgs<T> a) {
    rows_half_body<T, LEN, K, TR>(a);
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

template <typename T, int LENF, int TC, int MB, bool PRUNED, bool PACK = false>
static cudaError_t cols_half_launch(const ColArgs<T>& a, int batch, cudaStream_t st) {
    const int hcols = a.ncols / 2;
    const int nb = (hcols + TC - 1) / TC;
    if (nb == 0 || batch == 0) return cudaSuccess;
    if (a.nouter != 1 || a.N != LENF / 2 || a.ncols != (PACK ? a.N : a.N * a.N)) return cudaErrorInvalidValue;
    auto kern = k_cols_half<T, LENF, MB, TC, PRUNED, PACK>;
    constexpr size_t smem = cols_half_smem<T, LENF, TC>();
    cudaError_t e = set_smem(kern, smem);
    if (e != cudaSuccess) return e;
    const bool rf = a.rot_fastest;
    if (rf && nb > 65535) return cudaErrorInvalidValue;
    kern<<<rf ? dim3(batch, nb, 1) : dim3(nb, 1, batch), cta_threads_for<LENF>(TC), smem, st>>>(a);
    note_launch();
    return cudaGetLastError();
}

// 2D: N/2 columns a rotation.
template <typename T, int LENF, int MB, bool PRUNED>
static cudaError_t cols_half_2d(const ColArgs<T>& a, int batch, cudaStream_t st) {
    constexpr int TC = lines_per_cta<T, LENF>();
    const int64_t ctas = (int64_t)((a.ncols / 2 + TC - 1) / TC) * batch;
    if (ctas > 0 && (sizeof(T) == 8 ? few_pays(ctas, TC) : ctas <= 96)) {
        if (a.nouter != 1 || a.N != LENF / 2 || a.rot_fastest) return cudaErrorInvalidValue;
        constexpr size_t smem = cols_few_smem<T, LENF>();
        auto kern = k_cols_few<T, LENF, PRUNED>;
        cudaError_t e = set_smem(kern, smem);
        if (e != cudaSuccess) return e;
        kern<<<dim3((a.ncols / 2 + FEW_LINES - 1) / FEW_LINES, 1, batch), cta_threads_for<LENF>(2 * FEW_LINES), smem, st>>>(a);
        note_launch();
        return cudaGetLastError();
    }
    return cols_half_launch<T, LENF, TC, MB, PRUNED, true>(a, batch, st);
}

template <typename T, int LENF>
static cudaError_t cols_half_pruned(const ColArgs<T>& a, int batch, cudaStream_t st) {
    static_assert(prunable_len(LENF), "length not prunable");
    if (a.ncols == a.N) return cols_half_2d<T, LENF, pruned_min_ctas<T, LENF, 2>(), true>(a, batch, st);
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
#define SD_HALFF_CASE(L)                                                                                          \
    case L:                                                                                                       \
        return a.ncols == a.N                                                                                     \
                   ? cols_half_2d<T, L, min_ctas_per_sm<T, L>(), false>(a, batch, st) \
                   : cols_half_launch<T, L, lines_per_cta<T, L>(), min_ctas_per_sm<T, L>(), false>(a, batch, st);
        SD_HALFF_CASE(16) SD_HALFF_CASE(32) SD_HALFF_CASE(48) SD_HALFF_CASE(64) SD_HALFF_CASE(96)
        SD_HALFF_CASE(128) SD_HALFF_CASE(192) SD_HALFF_CASE(256) SD_HALFF_CASE(384) SD_HALFF_CASE(512)
#undef SD_HALFF_CASE
    }
    return cudaErrorInvalidValue;
}

template <typename T, int LEN>
static cudaError_t pack_y_launch(const ColArgs<T>& a, int batch, cudaStream_t st) {
    constexpr int TC = lines_per_cta<T, LEN>();
    if (batch == 0) return cudaSuccess;
    if (a.nouter != LEN || a.ncols != LEN / 2 || a.in == a.out) return cudaErrorInvalidValue;
    const size_t smem = (size_t)TC * col_pitch(LEN) * sizeof(cplx<T>);
    auto kern = k_pack_y<T, LEN>;
    cudaError_t e = set_smem(kern, smem);
    if (e != cudaSuccess) return e;
    kern<<<dim3((LEN / 2 + TC - 1) / TC, LEN, batch), cta_threads<T, LEN>(), smem, st>>>(a);
    note_launch();
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_pack_y_t(const ColArgs<T>& a, int batch, cudaStream_t st) {
    switch (a.N) {
#define SD_PACK_CASE(L) \
    case L: return pack_y_launch<T, L>(a, batch, st);
        SD_PACK_CASE(8) SD_PACK_CASE(16) SD_PACK_CASE(24) SD_PACK_CASE(32) SD_PACK_CASE(48) SD_PACK_CASE(64)
        SD_PACK_CASE(96) SD_PACK_CASE(128) SD_PACK_CASE(192) SD_PACK_CASE(256)
#undef SD_PACK_CASE
    }
    return cudaErrorInvalidValue;
}

template <typename T, int LEN, int K, int TR>
static cudaError_t rows_half_launch_tr(const RowArgs<T>& a, int batch, int* nparts, cudaStream_t st) {
    constexpr int NT = cta_threads_for<LEN>(TR);
    if (a.nrows % 2 != 0 || a.N != LEN) return cudaErrorInvalidValue;
    const int ngroups = (a.nrows / 2 + TR - 1) / TR;
    if (nparts) *nparts = 0;
    if (ngroups == 0 || batch == 0) return cudaSuccess;
    const int64_t total = (int64_t)ngroups * batch;
    int G = (int)(total / (half_row_wave<K>() * GPU_SMS));
    G = G < 1 ? 1 : (G > half_row_most<K>() ? half_row_most<K>() : G);
    const int nb = (ngroups + G - 1) / G;
    if (nparts) *nparts = nb * K;
    constexpr size_t smem = rows_half_smem<T, LEN, K, TR>();
    auto kern = k_rows_half<T, LEN, K, TR>;
    cudaError_t e = set_smem(kern, smem);
    if (e != cudaSuccess) return e;
    kern<<<dim3(nb, batch), NT, smem, st>>>(a);
    note_launch();
    return cudaGetLastError();
}

// Fewer lines per CTA where few_pays (FP64, and FP32's short lists, whose insertions two
// rows of a thread's outputs double): FP64 15 rotations at N = 128 22 -> 16 us, keeping four
// 37 -> 26, 192 points 33 -> 20; FP32 keeping four 256 points, 320 CTAs 22 -> 16.  Long lists
// pay for more partials to reduce: below half a wave only (72 CTAs at 96 points keeping 16
// 74 -> 70, 192 CTAs 117 -> 143).
template <typename T, int LEN, int K>
static cudaError_t rows_half_launch(const RowArgs<T>& a, int batch, int* nparts, cudaStream_t st) {
    constexpr int TR = lines_per_cta<T, LEN>();
    if constexpr (sizeof(T) == 8 || K == 2 || K == 4) {
        const int64_t ctas = (int64_t)((a.nrows / 2 + TR - 1) / TR) * batch;
        if (few_pays(ctas, TR) && (K <= 4 || 2 * ctas <= GPU_SMS))
            return rows_half_launch_tr<T, LEN, K, FEW_LINES>(a, batch, nparts, st);
    }
    return rows_half_launch_tr<T, LEN, K, TR>(a, batch, nparts, st);
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
    template <> cudaError_t launch_pack_y<T>(const ColArgs<T>& a, int batch, cudaStream_t st) {                \
        return launch_pack_y_t<T>(a, batch, st);                                                               \
    }                                                                                                          \
    template <> cudaError_t launch_rows_half<T>(int keep, const RowArgs<T>& a, int batch, int* np, cudaStream_t st) { \
        return launch_rows_half_t<T>(keep, a, batch, np, st);                                                  \
    }                                                                                                          \
    template <> cudaError_t launch_whalf<T>(const cplx<T>* W, int N, int dim, int n, int s_h, cplx<T>* out,     \
                                            cudaStream_t st) {                                                 \
        return launch_whalf_t<T>(W, N, dim, n, s_h, out, st);                                                  \
    }                                                                                                          \
    }
