// Score and gradient at arbitrary poses by a type-2 gather (the adjoint of the
// spreading step), for the gradient-driven pose search of Section 6.
//
// The fixed shape's band-limited field Phi(x) = sum_i c1_i K_N(x - p1_i) and its
// gradient are tabulated once on the oversampled periodic grid (inverse FFT of
// the deconvolved spectrum).  For pose (R, t): f = sum_j c2_j Phi(R p2_j + t),
// interpolated with the same exponential-of-semicircle kernel as the spreading.
// With g_j = Re(c2_j grad Phi(y_j)):  d Re f / dt = sum_j g_j, the torque
// tau = sum_j (R p2_j) x g_j is d Re f / d omega for a left perturbation
// R <- exp([omega]x) R, and d Re f / d q = 2 ((0, tau) (x) q/|q|) / |q| through
// R(q/|q|) (a vector orthogonal to q).
#pragma once
#include <math.h>

#include "kernels.cuh"

namespace sd {

constexpr int GA_THREADS = 256;

__device__ __forceinline__ int wrap_n(int a, int n) {
    a %= n;
    return a < 0 ? a + n : a;
}

// The fields of cell i side by side, (Phi, dPhi/dx, dPhi/dy, dPhi/dz): 32 bytes in FP32,
// one load (FP64: two).  A tap box's row of six cells is 192 bytes and touches 2.25
// cache lines on average; as two planes of 16-byte cells its two rows touched 3.25.
__device__ __forceinline__ void load_cell(const cplx<float>* G, int64_t i, cplx<float> f[4]) {
    const cplx<float>* p = G + 4 * i;
    asm("ld.global.nc.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
        : "=f"(f[0].x), "=f"(f[0].y), "=f"(f[1].x), "=f"(f[1].y), "=f"(f[2].x), "=f"(f[2].y), "=f"(f[3].x), "=f"(f[3].y)
        : "l"(p));
}
__device__ __forceinline__ void load_cell(const cplx<double>* G, int64_t i, cplx<double> f[4]) {
    const cplx<double>* p = G + 4 * i;
    asm("ld.global.nc.v4.f64 {%0, %1, %2, %3}, [%4];"
        : "=d"(f[0].x), "=d"(f[0].y), "=d"(f[1].x), "=d"(f[1].y) : "l"(p));
    asm("ld.global.nc.v4.f64 {%0, %1, %2, %3}, [%4];"
        : "=d"(f[2].x), "=d"(f[2].y), "=d"(f[3].x), "=d"(f[3].y) : "l"(p + 2));
}

// Score, d / dq and d / dt of a pose from the gather's sums.
template <typename T>
__device__ __forceinline__ void grad_finish(const double a[7], int64_t p, int dim, const T* quats, T* score, T* dq,
                                            T* dt) {
    score[p] = (T)a[0];
    dt[3 * p + 0] = (T)a[1];
    dt[3 * p + 1] = (T)a[2];
    dt[3 * p + 2] = (T)(dim == 3 ? a[3] : 0.0);
    const double tx = a[4], ty = a[5], tz = a[6];
    const T* q = quats + 4 * p;
    const double w = q[0], x = q[1], y = q[2], z = q[3];
    const double nq = sqrt(w * w + x * x + y * y + z * z);
    const double inv = nq > 0 ? 1.0 / nq : 0.0;
    const double u0 = w * inv, ux = x * inv, uy = y * inv, uz = z * inv;
    // (0, tau) (x) u = (-tau.u, u0 tau + tau x u)
    const double s0 = -(tx * ux + ty * uy + tz * uz);
    const double sx = u0 * tx + (ty * uz - tz * uy);
    const double sy = u0 * ty + (tz * ux - tx * uz);
    const double sz = u0 * tz + (tx * uy - ty * ux);
    dq[4 * p + 0] = (T)(2.0 * s0 * inv);
    dq[4 * p + 1] = (T)(2.0 * sx * inv);
    dq[4 * p + 2] = (T)(2.0 * sy * inv);
    dq[4 * p + 3] = (T)(2.0 * sz * inv);
}

// q <- exp(theta) (x) q / |.| for a rotation vector theta (left multiplication).
__device__ __forceinline__ void rotate_left(double q[4], const double th[3]) {
    const double a = sqrt(th[0] * th[0] + th[1] * th[1] + th[2] * th[2]);
    double o[4] = {q[0], q[1], q[2], q[3]};
    if (a > 0.0) {
        const double c = cos(0.5 * a), s = sin(0.5 * a) / a;
        const double ew = c, ex = s * th[0], ey = s * th[1], ez = s * th[2];
        o[0] = ew * q[0] - ex * q[1] - ey * q[2] - ez * q[3];
        o[1] = ew * q[1] + ex * q[0] + ey * q[3] - ez * q[2];
        o[2] = ew * q[2] - ex * q[3] + ey * q[0] + ez * q[1];
        o[3] = ew * q[3] + ex * q[2] - ey * q[1] + ez * q[0];
    }
    const double n = sqrt(o[0] * o[0] + o[1] * o[1] + o[2] * o[2] + o[3] * o[3]);
    for (int k = 0; k < 4; ++k) q[k] = n > 0.0 ? o[k] / n : o[k];
}

// One update of a pose from the gather's sums a (score, force
// F = d Re f / dt, torque T = sum (R p2) x g): the score goes to hist (if
// given); unless `last` the pose moves by
//   ascent:    t += lr_t F / max|F|, q += lr_q dq / max|dq| (dq = d Re f / dq), q normalised;
//   CG:        Polak-Ribiere directions (beta clipped at 0) kept per block, t moved
//              lr_t along the translation direction, R rotated lr_q radians about
//              the rotation direction;
//   dynamics:  v <- (1 - gamma) v + h F / m, w <- (1 - gamma) w + h T / I,
//              t += h v, q <- exp(h w) q.
// state (P x 12 doubles): CG (gF, gT, dF, dT) of the previous step; dynamics (v, w).
// WARP: one warp a pose; the ascent's divisions go to its lanes (serial FP64 division is
// most of the update's time), the other rules run on lane 0.  Else one thread a pose.
template <typename T, bool WARP>
__device__ __forceinline__ void refine_update(const double a[7], int64_t p, int dim, const RefineParams& rp, T* quats,
                                              T* trans, double* state, int first) {
    T* qo = quats + 4 * p;
    T* to = trans + 3 * p;
    double q[4] = {qo[0], qo[1], qo[2], qo[3]};
    double t[3] = {to[0], to[1], dim == 3 ? (double)to[2] : 0.0};
    const double F[3] = {a[1], a[2], dim == 3 ? a[3] : 0.0};
    const double Tq[3] = {a[4], a[5], a[6]};
    double* st = state ? state + 12 * p : nullptr;
    if (rp.method == SD_REFINE_ASCENT) {
        const double nq = sqrt(q[0] * q[0] + q[1] * q[1] + q[2] * q[2] + q[3] * q[3]);
        const double inv = nq > 0 ? 1.0 / nq : 0.0;
        const double u0 = q[0] * inv, ux = q[1] * inv, uy = q[2] * inv, uz = q[3] * inv;
        const double tx = Tq[0], ty = Tq[1], tz = Tq[2];
        const double dq[4] = {2.0 * inv * -(tx * ux + ty * uy + tz * uz), 2.0 * inv * (u0 * tx + (ty * uz - tz * uy)),
                              2.0 * inv * (u0 * ty + (tz * ux - tx * uz)), 2.0 * inv * (u0 * tz + (tx * uy - ty * ux))};
        double sf = 1e-30, sq = 1e-30;
        for (int k = 0; k < 3; ++k) sf = fmax(sf, fabs(F[k]));
        for (int k = 0; k < 4; ++k) sq = fmax(sq, fabs(dq[k]));
        if constexpr (!WARP) {
            double qn[4];
            for (int k = 0; k < 4; ++k) qn[k] = q[k] + rp.lr_q * dq[k] / sq;
            const double nn = sqrt(qn[0] * qn[0] + qn[1] * qn[1] + qn[2] * qn[2] + qn[3] * qn[3]);
            for (int k = 0; k < 4; ++k) qo[k] = (T)(nn > 0 ? qn[k] / nn : qn[k]);
            for (int k = 0; k < dim; ++k) to[k] = (T)(t[k] + rp.lr_t * F[k] / sf);
            return;
        }
        // lanes 0-3: a quaternion entry each, lanes 4-6: a translation entry
        const int lane = threadIdx.x & 31, k = lane & 3;
        const bool is_t = (lane & 4) != 0;
        const double cur = is_t ? (k == 0 ? t[0] : (k == 1 ? t[1] : t[2]))
                                : (k == 0 ? q[0] : (k == 1 ? q[1] : (k == 2 ? q[2] : q[3])));
        const double dir = is_t ? (k == 0 ? F[0] : (k == 1 ? F[1] : F[2]))
                                : (k == 0 ? dq[0] : (k == 1 ? dq[1] : (k == 2 ? dq[2] : dq[3])));
        const double moved = cur + (is_t ? rp.lr_t : rp.lr_q) * dir / (is_t ? sf : sq);
        double qn[4];
        for (int j = 0; j < 4; ++j) qn[j] = __shfl_sync(0xffffffffu, moved, j);
        const double nn = sqrt(qn[0] * qn[0] + qn[1] * qn[1] + qn[2] * qn[2] + qn[3] * qn[3]);
        if (lane < 4) qo[k] = (T)(nn > 0 ? moved / nn : moved);
        else if (lane < 4 + dim) to[k] = (T)moved;
        return;
    }
    if (WARP && (threadIdx.x & 31) != 0) return;
    if (rp.method == SD_REFINE_CG) {
        const double* g[2] = {F, Tq};
        double d[2][3];
        for (int b = 0; b < 2; ++b) {
            double beta = 0.0;
            if (!first) {
                const double* gp = st + 3 * b;
                double num = 0.0, den = 0.0;
                for (int k = 0; k < 3; ++k) {
                    num += g[b][k] * (g[b][k] - gp[k]);
                    den += gp[k] * gp[k];
                }
                beta = den > 0.0 ? fmax(0.0, num / den) : 0.0;
            }
            for (int k = 0; k < 3; ++k) d[b][k] = g[b][k] + (first ? 0.0 : beta * st[6 + 3 * b + k]);
        }
        for (int b = 0; b < 2; ++b)
            for (int k = 0; k < 3; ++k) {
                st[3 * b + k] = g[b][k];
                st[6 + 3 * b + k] = d[b][k];
            }
        const double nt = sqrt(d[0][0] * d[0][0] + d[0][1] * d[0][1] + d[0][2] * d[0][2]);
        const double nr = sqrt(d[1][0] * d[1][0] + d[1][1] * d[1][1] + d[1][2] * d[1][2]);
        if (nt > 0.0)
            for (int k = 0; k < 3; ++k) t[k] += rp.lr_t * d[0][k] / nt;
        if (nr > 0.0) {
            const double th[3] = {rp.lr_q * d[1][0] / nr, rp.lr_q * d[1][1] / nr, rp.lr_q * d[1][2] / nr};
            rotate_left(q, th);
        }
    } else {  // SD_REFINE_DYNAMICS
        double v[3], w[3];
        for (int k = 0; k < 3; ++k) {
            v[k] = (first ? 0.0 : (1.0 - rp.damping) * st[k]) + rp.h * F[k] / rp.mass;
            w[k] = (first ? 0.0 : (1.0 - rp.damping) * st[3 + k]) + rp.h * Tq[k] / rp.inertia;
            st[k] = v[k];
            st[3 + k] = w[k];
            t[k] += rp.h * v[k];
        }
        const double th[3] = {rp.h * w[0], rp.h * w[1], rp.h * w[2]};
        rotate_left(q, th);
    }
    for (int k = 0; k < 4; ++k) qo[k] = (T)q[k];
    to[0] = (T)t[0];
    to[1] = (T)t[1];
    if (dim == 3) to[2] = (T)t[2];
}

// The last CTA's warp 0: reads a pose's sums, clears them, and writes the gradient
// or moves the pose.  Out of line, so that its FP64 takes no registers of the gather.
template <typename T, int D>
__device__ __noinline__ void finish_pose(const GatherArgs<T>& a, int pose) {
    const int lane = threadIdx.x & 31;
    double* sums = a.acc + 8 * (int64_t)pose;
    double f[7];
#pragma unroll
    for (int k = 0; k < 7; ++k) f[k] = __ldcg(sums + k);
    __syncwarp();
    if (lane < 8) __stcg(sums + lane, 0.0);
    if (a.step) {
        if (a.hist && lane == 0) a.hist[pose] = (T)f[0];
        if (!a.last) refine_update<T, true>(f, pose, D, a.rp, a.quats_io, a.trans_io, a.state, a.first);
    } else if (lane == 0) {
        grad_finish<T>(f, pose, D, a.quats, a.score, a.dq, a.dt);
    }
}

// The same by one thread a pose, in a launch of its own, after gathers of many CTAs
// (launch_gather): there the update's FP64 chain in every pose's last CTA, and the 64
// registers that its call holds in all of them, cost more than a launch.
template <typename T>
__global__ void __launch_bounds__(32) k_finish_poses(GatherArgs<T> a, int dim) {
    const int64_t pose = (int64_t)blockIdx.x * 32 + threadIdx.x;
    if (pose >= a.P) return;
    double f[7];
#pragma unroll
    for (int k = 0; k < 7; ++k) {
        f[k] = a.acc[8 * pose + k];
        a.acc[8 * pose + k] = 0.0;
    }
    if (a.step) {
        if (a.hist) a.hist[pose] = (T)f[0];
        if (!a.last) refine_update<T, false>(f, pose, dim, a.rp, a.quats_io, a.trans_io, a.state, a.first);
    } else {
        grad_finish<T>(f, pose, dim, a.quats, a.score, a.dq, a.dt);
    }
}

// One CTA per (pose, chunk of CHUNK samples).  Each thread stages one sample
// (kernel weights, weight value, rotated position, tap-box origin); the warps
// then take the staged samples round-robin and gather each with their lanes on
// consecutive taps, so a load instruction reads a few rows of adjacent cells
// instead of one cell per sample.  A lane keeps, per sample, the weighted sums
// of the four fields over its taps, applies c and the torque arm R p2 to them,
// and accumulates score, force and torque over its samples; lanes and warps are
// summed in FP64 and added to the pose's accumulators.  The CTA that adds the last
// share of a pose finishes it (gradient outputs, or the pose's update) and clears the
// accumulators for the next launch, so a refinement step of few poses is one launch: 57 us with a
// clearing and an update launch of its own and 256 samples per CTA, at 10 poses x
// 2,280 samples, 26 now.  Few poses take fewer samples per CTA (a.chunk), so many that
// one wave of four CTAs per SM holds them all: eight CTAs per SM took 34 us a step,
// two 28 (each CTA's FP64 sums and last-CTA count are paid again).
// 256 poses x 20,000 samples are bound by the L1 data pipe (73 %; 2,452 us with the
// fields in two planes, 2,292 with 32-byte cells).
// Samples per CTA: as many as fit a 40 KiB stage, at most one per thread.
template <typename T, int D, int W>
__host__ __device__ constexpr int gather_chunk() {
    constexpr int rec = D * W + 7;
    constexpr int fit = (40 * 1024) / (rec * (int)sizeof(T)) / 32 * 32;
    return fit < GA_THREADS ? fit : GA_THREADS;
}

// Rotation (row-major) and translation of a pose (q, t may lie in shared memory).
template <typename T, int D>
__device__ __forceinline__ void pose_matrix(const T* q, const T* t, T Rm[9], T tv[3]) {
    const T w = q[0], x = q[1], y = q[2], z = q[3];
    const T n2 = w * w + x * x + y * y + z * z;
    const T s = n2 > T(0) ? T(2) / n2 : T(0);
    Rm[0] = T(1) - s * (y * y + z * z); Rm[1] = s * (x * y - w * z); Rm[2] = s * (x * z + w * y);
    Rm[3] = s * (x * y + w * z); Rm[4] = T(1) - s * (x * x + z * z); Rm[5] = s * (y * z - w * x);
    Rm[6] = s * (x * z - w * y); Rm[7] = s * (y * z + w * x); Rm[8] = T(1) - s * (x * x + y * y);
    tv[0] = t[0];
    tv[1] = t[1];
    tv[2] = (D == 3) ? t[2] : T(0);
}

// A staged sample: weights, c (2), R p2 (3), origin cell (wrapped into [0, n)), spare.
template <int D, int W>
__host__ __device__ constexpr int gather_rec() { return D * W + 7; }

// Stages samples [j0, j0 + nj) of a CTA of NT threads: one per thread, or (few) four
// threads each, one axis a thread (the fourth: the weight).
template <typename T, int D, int W, int NT>
__device__ __forceinline__ void gather_stage(const GatherArgs<T>& a, const T Rm[9], const T tv[3], int64_t j0, int nj,
                                             bool few, T* stage) {
    using C = cplx<T>;
    constexpr int REC = gather_rec<D, W>();
    const int n = a.n, pn = a.pn;
    const T half = T(W) * T(0.5), inv_half = T(2) / T(W);
    if (!few) {
        if ((int)threadIdx.x < nj) {
            const int64_t j = j0 + threadIdx.x;
            const vec4<T> p = a.p2[j];
            const C c = a.c2[j];
            const T pz = (D == 3) ? p.z : T(0);
            T rp[3];
            rp[0] = Rm[0] * p.x + Rm[1] * p.y + Rm[2] * pz;
            rp[1] = Rm[3] * p.x + Rm[4] * p.y + Rm[5] * pz;
            rp[2] = (D == 3) ? Rm[6] * p.x + Rm[7] * p.y + Rm[8] * pz : T(0);
            T* r = stage + threadIdx.x * REC;
            int base = 0, mul = 1;
#pragma unroll
            for (int d = 0; d < D; ++d) {
                const T g = (rp[d] + tv[d]) * a.inv_h;
                const int u0 = (int)ceil(g - half);
#pragma unroll
                for (int k = 0; k < W; ++k) {
                    const T zz = (T(u0 + k) - g) * inv_half;
                    const T z2 = zz * zz;
                    r[d * W + k] = (z2 <= T(1)) ? exp(a.beta * (sqrt(T(1) - z2) - T(1))) : T(0);
                }
                base += wrap_n(u0, n) * mul;  // taps reach index n - 1 + W - 1 < pn: no wrapping per tap
                mul *= pn;
            }
            r[D * W] = c.x;
            r[D * W + 1] = c.y;
            r[D * W + 2] = rp[0];
            r[D * W + 3] = rp[1];
            r[D * W + 4] = rp[2];
            // cell indices below 2^31 (pn <= 528 in 3D) travel as the bits of a T
            reinterpret_cast<int*>(r + D * W + 5)[0] = base;
        }
        return;
    }
    for (int s0 = 0; s0 < nj; s0 += NT / 4) {
        const int js = s0 + ((int)threadIdx.x >> 2), part = (int)threadIdx.x & 3;
        const bool act = js < nj;
        T* r = stage + js * REC;
        int base = 0;
        if (act && part == 3) {
            const C c = a.c2[j0 + js];
            r[D * W] = c.x;
            r[D * W + 1] = c.y;
            if (D == 2) r[D * W + 4] = T(0);
        } else if (act && part < D) {
            const vec4<T> p = a.p2[j0 + js];
            const T pz = (D == 3) ? p.z : T(0);
            const T r0 = part == 0 ? Rm[0] : (part == 1 ? Rm[3] : Rm[6]), r1 = part == 0 ? Rm[1] : (part == 1 ? Rm[4] : Rm[7]),
                    r2 = part == 0 ? Rm[2] : (part == 1 ? Rm[5] : Rm[8]);
            const T rp = r0 * p.x + r1 * p.y + r2 * pz;
            const T g = (rp + (part == 0 ? tv[0] : (part == 1 ? tv[1] : tv[2]))) * a.inv_h;
            const int u0 = (int)ceil(g - half);
#pragma unroll
            for (int k = 0; k < W; ++k) {
                const T zz = (T(u0 + k) - g) * inv_half;
                const T z2 = zz * zz;
                r[part * W + k] = (z2 <= T(1)) ? exp(a.beta * (sqrt(T(1) - z2) - T(1))) : T(0);
            }
            r[D * W + 2 + part] = rp;
            base = wrap_n(u0, n) * (part == 0 ? 1 : (part == 1 ? pn : pn * pn));
        }
        base += __shfl_xor_sync(0xffffffffu, base, 1);
        base += __shfl_xor_sync(0xffffffffu, base, 2);
        if (act && part == 0) reinterpret_cast<int*>(r + D * W + 5)[0] = base;
    }
}

// The staged samples' shares of the pose's seven sums, added to the lane's.
template <typename T, int D, int W>
struct Gatherer {
    static constexpr int TAPS = (D == 3) ? W * W * W : W * W;
    static constexpr int ROUNDS = (TAPS + 31) / 32;
    static constexpr bool TABLE = ROUNDS <= 8;  // per-lane tap table in registers (else derived per round)
    static constexpr int NT = TABLE ? ROUNDS : 1;
    int toff[NT];  // grid offsets of taps: below pn^3 < 2^28
    int tk[NT];    // (kx, ky, kz)
    int pn;
    __device__ __forceinline__ static void tap_of(int q, int& kx, int& ky, int& kz) {
        const int tap = min(q * 32 + (int)(threadIdx.x & 31), TAPS - 1);
        kx = tap % W;
        ky = (tap / W) % W;
        kz = (D == 3) ? tap / (W * W) : 0;
    }
    __device__ __forceinline__ explicit Gatherer(int pitch) : pn(pitch) {
        if constexpr (TABLE) {
#pragma unroll
            for (int q = 0; q < ROUNDS; ++q) {
                int kx, ky, kz;
                tap_of(q, kx, ky, kz);
                toff[q] = kx + pn * (ky + pn * kz);
                tk[q] = kx | (ky << 8) | (kz << 16);
            }
        }
    }
    // samples first, first + step, ... below nj, a warp each
    __device__ __forceinline__ void add(const cplx<T>* G, const T* stage, int nj, int first, int step, T acc[7]) const {
        using C = cplx<T>;
        constexpr int REC = gather_rec<D, W>();
        const int lane = threadIdx.x & 31;
        for (int jj = first; jj < nj; jj += step) {
            const T* r = stage + jj * REC;
            const int base = reinterpret_cast<const int*>(r + D * W + 5)[0];
            C f0 = mk(T(0), T(0)), f1 = f0, f2 = f0, f3 = f0;
#pragma unroll(TABLE ? ROUNDS : 1)
            for (int q = 0; q < ROUNDS; ++q) {
                if (TAPS % 32 == 0 || q * 32 + lane < TAPS) {
                    int kx, ky, kz, off;
                    if constexpr (TABLE) {
                        kx = tk[q] & 255;
                        ky = (tk[q] >> 8) & 255;
                        kz = tk[q] >> 16;
                        off = toff[q];
                    } else {
                        tap_of(q, kx, ky, kz);
                        off = kx + pn * (ky + pn * kz);
                    }
                    T wgt = r[kx] * r[W + ky];
                    if (D == 3) wgt *= r[2 * W + kz];
                    C f[4];
                    load_cell(G, base + off, f);
                    f0 = cadd(f0, cscale(f[0], wgt));
                    f1 = cadd(f1, cscale(f[1], wgt));
                    f2 = cadd(f2, cscale(f[2], wgt));
                    if (D == 3) f3 = cadd(f3, cscale(f[3], wgt));
                }
            }
            const T cx = r[D * W], cy = r[D * W + 1];
            const T rx = r[D * W + 2], ry = r[D * W + 3], rz = r[D * W + 4];
            const T gx = cx * f1.x - cy * f1.y;
            const T gy = cx * f2.x - cy * f2.y;
            const T gz = (D == 3) ? cx * f3.x - cy * f3.y : T(0);
            acc[0] += cx * f0.x - cy * f0.y;
            acc[1] += gx;
            acc[2] += gy;
            acc[3] += gz;
            acc[4] += ry * gz - rz * gy;
            acc[5] += rz * gx - rx * gz;
            acc[6] += rx * gy - ry * gx;
        }
    }
};

// Warp sums of the seven values in FP64, halving the values a lane holds with the
// lanes they are summed over (9 additions instead of 35: the FP64 pipe was 47 % busy
// with them when CTAs take few samples); lane 4 k ends with value k, written to out.
template <typename T>
__device__ __forceinline__ void warp_sums(const T acc[7], double* out) {
    const int lane = threadIdx.x & 31;
    double v[8];
#pragma unroll
    for (int k = 0; k < 7; ++k) v[k] = (double)acc[k];
    v[7] = 0.0;
#pragma unroll
    for (int half = 4; half > 0; half >>= 1) {
        const int mask = 4 * half;
        const bool up = (lane & mask) != 0;
#pragma unroll
        for (int k = 0; k < half; ++k) {
            const double keep = up ? v[k + half] : v[k], send = up ? v[k] : v[k + half];
            v[k] = keep + __shfl_xor_sync(0xffffffffu, send, mask);
        }
    }
    v[0] += __shfl_xor_sync(0xffffffffu, v[0], 2);
    v[0] += __shfl_xor_sync(0xffffffffu, v[0], 1);
    if ((lane & 3) == 0 && (lane >> 2) < 7) out[lane >> 2] = v[0];
}

// APART: k_finish_poses finishes the poses.  (With finish_pose 64 registers: four CTAs per
// SM; without, 37 to 48 in most forms, and five to six.)
template <typename T, int D, int W, bool APART>
__global__ void __launch_bounds__(GA_THREADS, sizeof(T) == 4 && W <= 6 && !APART ? 4 : 0) k_gather(GatherArgs<T> a) {
    constexpr int NWARP = GA_THREADS / 32;
    __shared__ T stage[gather_chunk<T, D, W>() * gather_rec<D, W>()];
    __shared__ double red[NWARP][7];
    const int pose = blockIdx.y;
    const Gatherer<T, D, W> gather(a.pn);
    // a refinement's launches overlap: the next one's CTAs may start as these leave, and
    // wait here for the poses this one moves
    asm volatile("griddepcontrol.launch_dependents;");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    T Rm[9], tv[3];
    if constexpr (sizeof(T) == 4) {
        pose_matrix<T, D>(a.quats + 4 * (int64_t)pose, a.trans + 3 * (int64_t)pose, Rm, tv);
    } else {  // FP64 by one warp: eight would queue for the pipe
        __shared__ T pm[12];
        if (threadIdx.x < 32) {
            pose_matrix<T, D>(a.quats + 4 * (int64_t)pose, a.trans + 3 * (int64_t)pose, Rm, tv);
            if (threadIdx.x == 0) {
                for (int k = 0; k < 9; ++k) pm[k] = Rm[k];
                for (int k = 0; k < 3; ++k) pm[9 + k] = tv[k];
            }
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < 9; ++k) Rm[k] = pm[k];
#pragma unroll
        for (int k = 0; k < 3; ++k) tv[k] = pm[9 + k];
    }
    const int64_t j0 = (int64_t)blockIdx.x * a.chunk;
    const int nj = (int)((a.m2 - j0) < (int64_t)a.chunk ? (a.m2 - j0) : (int64_t)a.chunk);
    gather_stage<T, D, W, GA_THREADS>(a, Rm, tv, j0, nj, a.few, stage);
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    T acc[7] = {T(0), T(0), T(0), T(0), T(0), T(0), T(0)};
    gather.add(a.G, stage, nj, warp, NWARP, acc);
    warp_sums<T>(acc, red[warp]);
    __syncthreads();
    if (threadIdx.x < 7) {
        double s = 0.0;
        for (int w = 0; w < NWARP; ++w) s += red[w][threadIdx.x];
        atomicAdd(a.acc + 8 * (int64_t)pose + threadIdx.x, s);
        if (!APART) __threadfence();  // before the count below
    }
    if constexpr (APART) return;
    __syncthreads();
    if (warp != 0) return;
    double* sums = a.acc + 8 * (int64_t)pose;
    unsigned* count = reinterpret_cast<unsigned*>(sums + 7);
    unsigned before = 0;
    if (lane == 0) before = atomicAdd(count, 1u);
    if (__shfl_sync(0xffffffffu, before, 0) != gridDim.x - 1) return;
    __threadfence();  // every share is in
    finish_pose<T, D>(a, pose);
}

template <typename T>
cudaError_t launch_gather(const GatherArgs<T>& args, int dim, cudaStream_t st) {
    if (args.P == 0 || args.m2 == 0) return cudaSuccess;
    GatherArgs<T> a = args;
    constexpr int64_t CTAS = 4 * GPU_SMS;  // one wave
    bool apart = false;
    // Samples per CTA: at most what its stage holds, at least one per warp, the wave's CTAs
    // shared out evenly among the poses (512 poses x 50 samples in chunks of 48 took a second
    // CTA each for two samples: FP64 in 2D 191 us a gradient, 105 now).
    // Four threads a sample shorten the stage's latency but spend a lane in four (in 2D two)
    // on no weight: not where the FP64 pipe is what bounds it (400 samples x 64 poses in 2D
    // 116 us with, 100 without; in 3D 20 samples x 200 poses 62 with, 88 without).
    // Poses are finished apart beyond two waves of CTAs (FP64: one), us a refinement of 20
    // steps with finishing inside / apart: 2,000 poses x 130 samples in 2D by CG 2,118 / 1,100
    // (a step kernel always: 1,533), x 2,000 in 2D 9,160 / 7,920; 512 x 400 in 3D at w = 8
    // (1,024 CTAs) 5,340 / 5,740, FP64 in 2D 14,520 / 13,700.
    auto grid = [&](int most) {
        const int64_t per_pose = a.P < CTAS ? CTAS / a.P : 1;
        const int64_t want = ((a.m2 + per_pose - 1) / per_pose + 7) / 8 * 8;
        a.chunk = (int)(want < 8 ? 8 : (want > most ? most : want));
        const unsigned ctas = (unsigned)((a.m2 + a.chunk - 1) / a.chunk);
        a.few = a.chunk <= GA_THREADS / 4 && (sizeof(T) == 4 || dim == 3 || ctas * a.P <= GPU_SMS);
        apart = ctas * a.P > (sizeof(T) == 4 ? 2 : 1) * CTAS;
        return dim3(ctas, (unsigned)a.P);
    };
    // the second and later steps of a refinement may be set up while the previous runs
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    auto launch = [&](void (*kern)(GatherArgs<T>), dim3 g) {
        cudaLaunchConfig_t cfg{};
        cfg.gridDim = g;
        cfg.blockDim = dim3(GA_THREADS);
        cfg.stream = st;
        cfg.attrs = attr;
        cfg.numAttrs = a.step && !a.first ? 1 : 0;
        return cudaLaunchKernelEx(&cfg, kern, a);
    };
    cudaError_t e = cudaSuccess;
#define SD_GATHER_CASE(WW)                                                                          \
    case WW:                                                                                        \
        if (dim == 2) {                                                                             \
            const dim3 g = grid(gather_chunk<T, 2, WW>());                                          \
            e = launch(apart ? k_gather<T, 2, WW, true> : k_gather<T, 2, WW, false>, g);            \
        } else {                                                                                    \
            const dim3 g = grid(gather_chunk<T, 3, WW>());                                          \
            e = launch(apart ? k_gather<T, 3, WW, true> : k_gather<T, 3, WW, false>, g);            \
        }                                                                                           \
        note_launch();                                                                              \
        if (e == cudaSuccess) e = cudaGetLastError();                                               \
        if (e != cudaSuccess || !apart) return e;                                                   \
        k_finish_poses<T><<<(unsigned)((a.P + 31) / 32), 32, 0, st>>>(a, dim);                      \
        note_launch();                                                                              \
        return cudaGetLastError();
    switch (a.w) {
        SD_GATHER_CASE(4) SD_GATHER_CASE(5) SD_GATHER_CASE(6) SD_GATHER_CASE(7) SD_GATHER_CASE(8)
        SD_GATHER_CASE(10) SD_GATHER_CASE(12) SD_GATHER_CASE(16)
    }
#undef SD_GATHER_CASE
    return cudaErrorInvalidValue;
}

}  // namespace sd
