// Spectral-bound estimates for the expansion (Sec. II-C: the polynomial
// expansions need estimates eps_1, eps_N of the spectral bounds, and the
// number of products grows with the width they span).
//
// Gershgorin discs always contain the spectrum but, for a dense rotated Hp,
// span ~20-50x its true width, which costs SP2 about 2 log2 of that ratio in
// extra products (and the finite-temperature recursion extra doublings).
// Here kLanczosSteps steps of the Lanczos recurrence (FP32 vectors and
// products, FP64 sums), from a fixed
// pseudo-random unit vector, give Ritz values theta_min, theta_max inside the
// spectrum; the estimate is
//     [theta_min - |beta_k s_min|, theta_max + |beta_k s_max|],
// widened by the residuals of the extreme Ritz pairs (s the unit eigenvector
// of the tridiagonal T) and clipped to the Gershgorin interval.
//
// An estimate is not a bound, so it is certified before use (k_check_bounds):
// with X0 = (hi I - Hp)/(hi - lo), kCheckSteps logistic steps
// X <- 4 X (I - X) give X_3 = (I - T_8(A))/2, T_8 the Chebyshev polynomial and
// A = (2 Hp - (hi + lo) I)/(hi - lo).  |T_8| <= 1 on [-1, 1] and
// T_8(a) = cosh(8 arccosh |a|) outside, so every eigenvalue a of A satisfies
// (cosh(8 arccosh |a|) - 1)/2 <= ||X_3||_F, i.e.
//     |a| <= cosh(arccosh(1 + 2 ||X_3||_F) / 8),
// and the interval widened by that factor contains the spectrum.  Eigenvalues
// inside the estimate keep X_3 in [0, 1] (||X_3||_F <= sqrt(n): at most a
// ~25% widening); one that the estimate missed grows X_3 and widens the
// bound just enough to take it in.
//
// No reorthogonalisation: loss of orthogonality only repeats converged Ritz
// values, which cannot move the extreme ones outward.
#include <cfloat>

#include "fe_dev.cuh"
#include "fe_kernels.cuh"

namespace fe {

namespace {

// SplitMix64 finaliser: a fixed, well-mixed 64-bit value per index
__device__ __forceinline__ uint64_t mix64(uint64_t z) {
    z += 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

// Sum over the block's threads, of which those from `cnt` on hold zero, as a
// binary tree (t + t + 256, t + t + 128, ...; the zero levels left out); thread 0
// hands it to `done`, and what that writes to shared memory is visible to all
// when the call returns.  The scalar arithmetic belongs in `done`: run by every
// thread, an FP64 square root and a division took the 16 warps of a block 4 us.
template <class F>
__device__ __forceinline__ void block_sum(double v, double *sh, int cnt, F done) {
    const int t = threadIdx.x;
    if (cnt > 32) {
        int o = kLzThreads / 2;
        while (o >= cnt) o >>= 1;
        sh[t] = v;
        __syncthreads();
        for (; o >= 32; o >>= 1) {
            if (t < o) {
                v += sh[t + o];
                sh[t] = v;
            }
            __syncthreads();
        }
    } else {
        __syncthreads();
    }
    if (t < 32) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (t == 0) done(v);
    }
    __syncthreads();
}

// scalars of a step, from thread 0 to its block
struct LzScalars {
    float alpha, beta, inv;
    int stop;
    double bn;
};

// number of eigenvalues of the tridiagonal (a, b) below x (Sturm sequence),
// in FP32 with the squared couplings b2[i] = b[i]^2 (GB300 runs FP64 at 1/64
// of the FP32 rate; the estimate needs no more than FP32 precision, since the
// certificate that follows decides the bounds)
__device__ int sturm_count_f(const float *a, const float *b2, int k, float x) {
    int c = 0;
    float q = a[0] - x;
    if (q < 0.0f) ++c;
    for (int i = 1; i < k; ++i) {
        if (q == 0.0f) q = 1e-30f;
        q = a[i] - x - b2[i] / q;
        if (q < 0.0f) ++c;
    }
    return c;
}

// eigenvalue number `idx` (0-based, ascending) of T in [lo, hi] by 32-point
// multisection over the warp (every lane calls it): each round lane l counts
// the eigenvalues below lo + (hi - lo)(l + 1)/33, and the interval shrinks to
// the two neighbouring points that bracket eigenvalue idx (33x per round),
// down to FP32 resolution.
__device__ double tri_eig(const float *a, const float *b2, int k, int idx, double lo, double hi) {
    const int lane = threadIdx.x & 31;
    for (int r = 0; r < 8; ++r) {
        const double w = hi - lo;
        if (!(w > 3e-7 * fmax(fabs(lo), fabs(hi)))) break;
        const double x = lo + w * static_cast<double>(lane + 1) / 33.0;
        const unsigned above = __ballot_sync(0xffffffffu, sturm_count_f(a, b2, k, static_cast<float>(x)) > idx);
        const int f = above ? __ffs(above) - 1 : 32;  // first point above the eigenvalue
        // the points either side of it, from the lanes that hold them
        const double below = __shfl_sync(0xffffffffu, x, (f + 31) & 31), over = __shfl_sync(0xffffffffu, x, f & 31);
        if (f > 0) lo = below;
        if (f < 32) hi = over;
    }
    return 0.5 * (lo + hi);
}

// |last component| of the unit eigenvector of T for eigenvalue th (forward
// three-term recurrence, rescaled to stay finite)
__device__ double tri_last_comp(const double *a, const double *b, int k, double th) {
    double s_prev = 0.0, s = 1.0, norm2 = 1.0;
    for (int i = 0; i + 1 < k; ++i) {
        // (a_i - th) s_i + b_i s_{i-1} + b_{i+1} s_{i+1} = 0
        const double bn = b[i + 1];
        const double s_next = (bn != 0.0) ? -((a[i] - th) * s + b[i] * s_prev) / bn : 0.0;
        s_prev = s;
        s = s_next;
        norm2 += s * s;
        if (norm2 > 1e200) {
            const double r = 1e-100;
            s *= r;
            s_prev *= r;
            norm2 *= r * r;
        }
    }
    return fabs(s) / sqrt(norm2);
}

}  // namespace

// The recurrence runs in FP32 (vectors, H entries, products) with FP64 sums:
// the estimate needs no more (the certificate decides the bounds), and GB300
// runs FP64 arithmetic at 1/64 of the FP32 rate.

namespace {

// Grid barrier number k of a cooperative launch: complete once all nb blocks
// arrived, i.e. the arrival counter (zeroed before the launch) reaches
// (k + 1) nb.  The wait is bounded: when it runs out the block records
// kErrTimeoutGrid and every caller returns false (the blocks still running
// give up at their own next barrier).
__device__ bool grid_barrier(unsigned *cnt, unsigned k, unsigned nb, DevCtl *ctl, int *flag) {
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        atomicAdd(cnt, 1u);
        const unsigned target = (k + 1u) * nb;
        bool ok = true;
        if (ld_acquire_u32(cnt) < target) {
            // the timer is slow to read: every 64 polls
            const uint64_t lim = ctl->wait_ns, t0 = globaltimer();
            for (unsigned it = 1; ld_acquire_u32(cnt) < target; ++it) {
                if ((it & 63u) == 0 && globaltimer() - t0 > lim) {
                    ok = false;
                    break;
                }
            }
        }
        if (!ok) atomicCAS(&ctl->err, 0, kErrTimeoutGrid);
        __threadfence();
        *flag = ok ? 1 : 0;
    }
    __syncthreads();
    return *flag != 0;
}

// entry i of the fixed start vector, uniform in [-1, 1)
__device__ __forceinline__ float lz_entry(int i) {
    return static_cast<float>(static_cast<double>(mix64(0xF00Dull + static_cast<uint64_t>(i)) >> 11) *
                              (2.0 / 9007199254740992.0) - 1.0);
}

// v = the start vector at unit length, vp = 0 (the whole block; either array may
// be shared or global memory)
__device__ void lz_unit(float *vp, float *v, int n, double *sh, LzScalars *sc) {
    double ss = 0.0;
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        const float x = lz_entry(i);
        v[i] = x;
        vp[i] = 0.0f;
        ss += static_cast<double>(x) * x;
    }
    block_sum(ss, sh, n, [&](double sum) {
        const double nrm = sqrt(sum);
        sc->inv = nrm > 0.0 ? static_cast<float>(1.0 / nrm) : 0.0f;
    });
    const float inv = sc->inv;
    for (int i = threadIdx.x; i < n; i += blockDim.x) v[i] *= inv;
}

__device__ void lz_start(const MmaProb &pr, double *sh, LzScalars *sc) {
    SolveState *st = pr.st;
    if (!st->lz_on) return;
    lz_unit(pr.lzv, pr.lzv + pr.n, pr.n, sh, sc);
    if (threadIdx.x == 0) {
        st->lz_k = 0;
        st->lz_b[0] = 0.0;
    }
}

// sum_j H_row,j v_j by a warp: H from its FP32 copy in the problem's FP32 master
// (written by k_bounds_rows; rows 16-byte aligned, ld a multiple of 4) as 16-byte
// quadruples, four per lane in flight
template <class V4, class V1>
__device__ __forceinline__ double lz_row(const float *h, int n, int lane, V4 v4, V1 v1) {
    const int m = n >> 2;
    const float4 *h4 = reinterpret_cast<const float4 *>(h);
    float s0 = 0.0f, s1 = 0.0f, s2 = 0.0f, s3 = 0.0f;
    int k = lane;
    auto dot4 = [&](const float4 a, int q, float acc) {
        const float4 x = v4(q);
        return fmaf(a.x, x.x, fmaf(a.y, x.y, fmaf(a.z, x.z, fmaf(a.w, x.w, acc))));
    };
    for (; k + 96 < m; k += 128) {
        const float4 a0 = h4[k], a1 = h4[k + 32], a2 = h4[k + 64], a3 = h4[k + 96];
        s0 = dot4(a0, k, s0);
        s1 = dot4(a1, k + 32, s1);
        s2 = dot4(a2, k + 64, s2);
        s3 = dot4(a3, k + 96, s3);
    }
    for (; k < m; k += 32) s0 = dot4(h4[k], k, s0);
    for (int jj = 4 * m + lane; jj < n; jj += 32) s1 = fmaf(h[jj], v1(jj), s1);
    return warp_sum(static_cast<double>((s0 + s1) + (s2 + s3)));
}

// This block's share of w = H v: rows blockIdx.x * kLzWarps + warp, stepping
// by the grid's warps, one warp per row.  v comes from shared memory when `vs`
// holds it, else from L2 (ld.cg: another block wrote it since this launch
// began, so L1 may hold a stale copy).  The block's partial of w . v goes to its
// partial slot.
template <bool kStaged>
__device__ void lz_matvec(const MmaProb &pr, const float *vs, double *red) {
    constexpr int kWarps = kLzWarps;
    const int n = pr.n;
    const float *v = kStaged ? vs : pr.lzv + n;
    float *w = pr.lzv + 2 * static_cast<size_t>(n);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    auto v1 = [&](int i) { return kStaged ? v[i] : __ldcg(v + i); };
    auto v4 = [&](int q) {
        if (kStaged) return reinterpret_cast<const float4 *>(v)[q];
        return make_float4(v1(4 * q), v1(4 * q + 1), v1(4 * q + 2), v1(4 * q + 3));  // v at an odd offset
    };
    double part = 0.0;
    for (int row = blockIdx.x * kWarps + wid; row < n; row += gridDim.x * kWarps) {
        const double s = lz_row(pr.Y + static_cast<size_t>(row) * pr.ldy, n, lane, v4, v1);
        if (lane == 0) {
            w[row] = static_cast<float>(s);
            part += s * static_cast<double>(v1(row));
        }
    }
    if (lane == 0) red[wid] = part;
    __syncthreads();
    if (threadIdx.x == 0) {
        double a = 0.0;
        for (int q = 0; q < kWarps; ++q) a += red[q];
        pr.part[static_cast<size_t>(blockIdx.x) * kPartStride] = a;
    }
    __syncthreads();
}

// beta_{j+1} = ||w'|| from its square, whether the subspace is invariant (to
// FP32 accuracy), and 1 / beta_{j+1}
__device__ __forceinline__ void lz_norm(double sum, double alpha, LzScalars *sc) {
    sc->bn = sqrt(sum);
    sc->stop = !(sc->bn > 1e-6 * fmax(fabs(alpha), 1e-300));
    sc->inv = sc->stop ? 0.0f : static_cast<float>(1.0 / sc->bn);
}

// alpha_j = w . v (the blocks' partials, in block order); w' = w - alpha_j v
// - beta_j v_prev; beta_{j+1} = ||w'||; v_prev <- v, v <- w' / beta_{j+1}
// (the whole block; everything another block wrote is read through L2)
__device__ void lz_update(const MmaProb &pr, int j, double *sh, LzScalars *sc) {
    SolveState *st = pr.st;
    const int n = pr.n;
    float *vp = pr.lzv, *v = pr.lzv + n, *w = pr.lzv + 2 * static_cast<size_t>(n);
    double a = 0.0, alpha = 0.0;
    for (int b = threadIdx.x; b < static_cast<int>(gridDim.x); b += blockDim.x)
        a += __ldcg(pr.part + static_cast<size_t>(b) * kPartStride);
    block_sum(a, sh, static_cast<int>(gridDim.x), [&](double sum) {
        alpha = sum;
        sc->alpha = static_cast<float>(sum);
        sc->beta = static_cast<float>(st->lz_b[j]);
    });
    const float af = sc->alpha, bf = sc->beta;
    float ssf = 0.0f;
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        const float x = fmaf(-af, v[i], fmaf(-bf, vp[i], __ldcg(w + i)));
        w[i] = x;
        ssf = fmaf(x, x, ssf);
    }
    block_sum(static_cast<double>(ssf), sh, n, [&](double sum) { lz_norm(sum, alpha, sc); });
    const float inv = sc->inv;
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        vp[i] = v[i];
        v[i] = w[i] * inv;
    }
    if (threadIdx.x == 0) {
        st->lz_a[j] = alpha;
        st->lz_b[j + 1] = sc->stop ? 0.0 : sc->bn;
        st->lz_k = sc->stop ? -(j + 1) : j + 1;  // negative: stopped after |lz_k| steps
    }
}

// bounds from the tridiagonal, then the X0 preparation (the whole block; warp 0
// takes the lowest Ritz pair, warp 1 the highest)
__device__ void lz_finish(const MmaProb &pr, double narrow) {
    SolveState *st = pr.st;
    const int t = threadIdx.x;
    const int k = st->lz_k < 0 ? -st->lz_k : st->lz_k;
    const double glo = st->gersh_lo, ghi = st->gersh_hi;
    __shared__ double a[kLanczosSteps], b[kLanczosSteps + 1];  // b[i] couples i-1 and i, b[k] the residual
    __shared__ float af[kLanczosSteps], b2f[kLanczosSteps + 1];
    __shared__ double end[2];
    if (t < kLanczosSteps) {
        a[t] = st->lz_a[t];
        af[t] = static_cast<float>(a[t]);
    }
    if (t <= kLanczosSteps) {
        b[t] = st->lz_b[t];
        b2f[t] = static_cast<float>(b[t] * b[t]);
    }
    __syncthreads();
    if (k >= 2 && t < 64) {
        const bool top = t >= 32;
        const double th = tri_eig(af, b2f, k, top ? k - 1 : 0, glo, ghi);
        const double r = b[k] * tri_last_comp(a, b, k, th);
        if ((t & 31) == 0) end[top] = top ? fmin(ghi, th + r) : fmax(glo, th - r);
    }
    __syncthreads();
    if (t != 0) return;
    double lo = glo, hi = ghi;
    if (k >= 2) {
        lo = end[0];
        hi = end[1];
        if (!(hi > lo)) {
            lo = glo;
            hi = ghi;
        }
    }
    if (narrow < 1.0) {
        const double mid = 0.5 * (lo + hi), half = 0.5 * (hi - lo) * narrow;
        lo = mid - half;
        hi = mid + half;
    }
    // X0 on the estimate, for the certificate steps (k_control issues them)
    st->lz_lo = lo;
    st->lz_hi = hi;
    st->chk_left = kCheckSteps;
    setup_from_bounds(pr, st, lo, hi);
}

}  // namespace

// The whole estimate in one cooperative launch (see fe_kernels.cuh).  Block b
// starts, updates and finishes the problems b, b + grid, ...; every block
// takes part in every product.  Each product and each update ends at a grid
// barrier; a problem whose recurrence stopped (lz_k < 0, written by its
// updating block before the barrier) is skipped from then on.
__global__ void __launch_bounds__(kLzThreads, 2)
    k_lanczos_run(const MmaProb *probs, int k0, int m, int vcap, double narrow, DevCtl *ctl, unsigned *bar) {
    extern __shared__ __align__(16) float vs[];  // v of the problem in hand, when n <= vcap
    __shared__ double sh[kLzThreads];
    __shared__ int flag;
    __shared__ LzScalars sc;
    const unsigned nb = gridDim.x;
    unsigned nbar = 0;
    for (int q = blockIdx.x; q < m; q += nb) lz_start(probs[k0 + q], sh, &sc);
    if (!grid_barrier(bar, nbar++, nb, ctl, &flag)) return;
    for (int j = 0; j < kLanczosSteps; ++j) {
        for (int q = 0; q < m; ++q) {
            const MmaProb &pr = probs[k0 + q];
            const SolveState *st = pr.st;
            if (!st->lz_on || *reinterpret_cast<const volatile int *>(&st->lz_k) < 0) continue;
            const int n = pr.n;
            if (n <= vcap) {
                for (int i = threadIdx.x; i < n; i += blockDim.x) vs[i] = __ldcg(pr.lzv + n + i);
                __syncthreads();
                lz_matvec<true>(pr, vs, sh);
            } else {
                lz_matvec<false>(pr, vs, sh);
            }
        }
        if (!grid_barrier(bar, nbar++, nb, ctl, &flag)) return;
        for (int q = blockIdx.x; q < m; q += nb) {
            const MmaProb &pr = probs[k0 + q];
            if (pr.st->lz_on && pr.st->lz_k >= 0) lz_update(pr, j, sh, &sc);
            __syncthreads();
        }
        if (!grid_barrier(bar, nbar++, nb, ctl, &flag)) return;
    }
    for (int q = blockIdx.x; q < m; q += nb) {
        if (probs[k0 + q].st->lz_on) lz_finish(probs[k0 + q], narrow);
        __syncthreads();
    }
}

// The estimate of one problem with at most kLzWarps `parts` rows, every block
// keeping v and v_prev in shared memory and making the update itself (the same
// arithmetic in each): a step has one grid barrier, and no block waits for
// another's update.  Row r is a warp of block r % grid; w and the rows'
// products w_r v_r go through L2, in two copies that alternate, so that a step
// may write while a slower block still reads the step before.  The products
// are added as k_lanczos_run adds them (16 rows in order, then a tree over
// those groups), so both kernels give the same bounds.
// All 12 steps and the end: n = 384 in 261 us with two barriers a step and the
// scalar arithmetic in every thread, 102 us here; n = 4096 in 376 and 212 us.  A
// step is bound by the latencies of the barrier and of the two sums, at n = 4096
// also by the 67 MB of H from L2.
__global__ void __launch_bounds__(kLzThreads, 1)
    k_lanczos_one(const MmaProb *probs, int k, double narrow, DevCtl *ctl, unsigned *bar) {
    extern __shared__ float4 dyn[];
    __shared__ double sh[kLzThreads];
    __shared__ int flag;
    __shared__ LzScalars sc;
    const MmaProb &pr = probs[k];
    SolveState *st = pr.st;
    const int n = pr.n, t = threadIdx.x, lane = t & 31, wid = t >> 5;
    const unsigned nb = gridDim.x;
    float *v = reinterpret_cast<float *>(dyn), *vp = v + ((n + 3) & ~3);
    const bool first = blockIdx.x == 0 && t == 0;
    double alpha = 0.0, beta = 0.0;  // thread 0
    lz_unit(vp, v, n, sh, &sc);
    if (first) {
        st->lz_k = 0;
        st->lz_b[0] = 0.0;
    }
    __syncthreads();
    const int groups = (n + kLzWarps - 1) / kLzWarps;
    for (int j = 0; j < kLanczosSteps; ++j) {
        float *w = pr.lzv + static_cast<size_t>(j & 1) * n;
        double *rp = reinterpret_cast<double *>(pr.lzv + 2 * static_cast<size_t>(n)) + static_cast<size_t>(j & 1) * n;
        for (int row = wid * static_cast<int>(nb) + static_cast<int>(blockIdx.x); row < n; row += kLzWarps * static_cast<int>(nb)) {
            const double s = lz_row(pr.Y + static_cast<size_t>(row) * pr.ldy, n, lane,
                                    [&](int q) { return reinterpret_cast<const float4 *>(v)[q]; },
                                    [&](int i) { return v[i]; });
            if (lane == 0) {
                w[row] = static_cast<float>(s);
                rp[row] = s * static_cast<double>(v[row]);
            }
        }
        if (!grid_barrier(bar, static_cast<unsigned>(j), nb, ctl, &flag)) return;
        double a = 0.0;
        if (t < groups) {
            double p[kLzWarps];
#pragma unroll
            for (int q = 0; q < kLzWarps; ++q) {
                const int r = t * kLzWarps + q;
                p[q] = r < n ? __ldcg(rp + r) : 0.0;
            }
#pragma unroll
            for (int q = 0; q < kLzWarps; ++q) a += p[q];
        }
        block_sum(a, sh, groups, [&](double sum) {
            alpha = sum;
            sc.alpha = static_cast<float>(sum);
            sc.beta = static_cast<float>(beta);
        });
        const float af = sc.alpha, bf = sc.beta;
        float ssf = 0.0f;
        for (int i = t; i < n; i += kLzThreads) {
            const float x = fmaf(-af, v[i], fmaf(-bf, vp[i], __ldcg(w + i)));
            vp[i] = v[i];
            v[i] = x;
            ssf = fmaf(x, x, ssf);
        }
        block_sum(static_cast<double>(ssf), sh, n, [&](double sum) {
            lz_norm(sum, alpha, &sc);
            beta = sc.stop ? 0.0 : sc.bn;
        });
        const float inv = sc.inv;
        const bool stop = sc.stop;
        for (int i = t; i < n; i += kLzThreads) v[i] *= inv;
        if (first) {
            st->lz_a[j] = alpha;
            st->lz_b[j + 1] = beta;
            st->lz_k = stop ? -(j + 1) : j + 1;  // negative: stopped after |lz_k| steps
        }
        __syncthreads();
        if (stop) break;
    }
    if (blockIdx.x == 0) lz_finish(pr, narrow);
}

// Certified bounds from the check steps, then the X0 preparation (one thread
// per problem, blockIdx.x)
__global__ void k_check_bounds(const MmaProb *probs, int k0) {
    const MmaProb &pr = probs[k0 + blockIdx.x];
    SolveState *st = pr.st;
    if (threadIdx.x != 0 || !st->lz_on) return;
    const double mid = 0.5 * (st->lz_lo + st->lz_hi), half = 0.5 * (st->lz_hi - st->lz_lo);
    const double a = st->chk_amax;
    double lo = st->gersh_lo, hi = st->gersh_hi;
    if (a < 1e300 && half > 0.0) {  // NaN and overflow keep the Gershgorin interval
        lo = fmax(lo, mid - half * a);
        hi = fmin(hi, mid + half * a);
    }
    st->chk = 0;
    st->chk_left = 0;
    st->kind = kNone;
    setup_from_bounds(pr, st, lo, hi);
}

}  // namespace fe
