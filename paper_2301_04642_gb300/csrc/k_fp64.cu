// FP64 SP2 step (Sec. II-B1 Eq. (1)) on the upper-triangle 16x16 tiles of X^2,
// for every product of the plain FP64 schedule.  (X^2)_ij = sum_k X_ik X_jk
// since X is symmetric.  The epilogue writes X' = X^2 or 2X - X^2 to the other
// FP64 buffer (and its mirror) and per-tile partials: tr X', ||X'||_F^2 and
// ||X^2 - X||_F^2.
//
// Bound: GB300's FP64 units, 2 fused multiply-adds per clock and SM, so one
// warp per sub-partition keeps them busy and all that matters is that every SM
// has an equal share.  A 16x16 tile (one element per thread) is 65536 FMAs at
// n = 256, 16 us of one SM, and n = 256 has 136 of them for 152 SMs; the 64x64
// tiles used before gave 10 SMs 260 us of work each.  Measured on a solve at
// n = 256 (25 products and 3 certificate products): 9.37 ms with 64x64 tiles,
// 1.64 ms with these.  Operand loads (32 doubles per 256 FMAs) stay far below
// the L2 rate at every n.  The sum over k runs in ascending order in one FMA
// chain per element, whatever the tile.
#include "fe_dev.cuh"
#include "fe_kernels.cuh"

namespace fe {

namespace {
constexpr int kBK = 32;        // K per shared-memory stage
constexpr int kLd = kBK + 2;   // row stride: 16-byte reads of 8 rows hit all banks
}  // namespace

__global__ void __launch_bounds__(256) k_fp64_step(const MmaProb *probs, const TileF64 *tiles, int ntiles,
                                                   const DevCtl *ctl) {
    __shared__ __align__(16) double sA[2][kTileF64][kLd];
    __shared__ __align__(16) double sB[2][kTileF64][kLd];
    __shared__ double sT[kTileF64][kTileF64 + 1];
    __shared__ double red[3][8];
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    if (ctl->hold) return;

    for (int t = blockIdx.x; t < ntiles; t += gridDim.x) {
        const TileF64 te = tiles[t];
        const MmaProb &pr = probs[te.prob];
        const SolveState *st = pr.st;
        if (*reinterpret_cast<const volatile int *>(&st->kind) != kFp64) continue;
        const int n = pr.n;
        const double *X = pr.Xd[st->xcur];
        const long long ldx = pr.ldx;
        const int i0 = te.I * kTileF64, j0 = te.J * kTileF64;
        // thread (ty, tx) stages row ty of both panels, columns tx and tx + 16
        const double *ra = (i0 + ty < n) ? X + (i0 + ty) * ldx : nullptr;
        const double *rb = (j0 + ty < n) ? X + (j0 + ty) * ldx : nullptr;
        double a0, a1, b0, b1;
        auto fetch = [&](int k0) {
            const int ka = k0 + tx, kb = ka + 16;
            a0 = (ra && ka < n) ? ra[ka] : 0.0;
            a1 = (ra && kb < n) ? ra[kb] : 0.0;
            b0 = (rb && ka < n) ? rb[ka] : 0.0;
            b1 = (rb && kb < n) ? rb[kb] : 0.0;
        };
        fetch(0);
        double P = 0.0;
        int buf = 0;
        for (int k0 = 0; k0 < n; k0 += kBK, buf ^= 1) {
            sA[buf][ty][tx] = a0;
            sA[buf][ty][tx + 16] = a1;
            sB[buf][ty][tx] = b0;
            sB[buf][ty][tx + 16] = b1;
            __syncthreads();  // the other buffer was last read before this barrier
            if (k0 + kBK < n) fetch(k0 + kBK);
#pragma unroll
            for (int kk = 0; kk < kBK; kk += 2) {
                const double2 a = *reinterpret_cast<const double2 *>(&sA[buf][ty][kk]);
                const double2 b = *reinterpret_cast<const double2 *>(&sB[buf][tx][kk]);
                P = fma(a.x, b.x, P);
                P = fma(a.y, b.y, P);
            }
        }

        // epilogue: the SP2 branch plus the trace correction gamma (X - X^2),
        // which commutes with Hp and moves each eigenvalue by gamma x (1 - x)
        double *Xo = pr.Xd[st->xcur ^ 1];  // the control kernel flips xcur afterwards
        const int sq = st->sq;
        const int chk = st->chk;  // bound-certificate step: X' = 4 X (I - X)
        const double gamma = st->gamma;
        const int i = i0 + ty, j = j0 + tx;
        double tr = 0.0, s2 = 0.0, id = 0.0, xn = 0.0;
        if (i < n && j < n && j >= i) {
            const double xo = X[i * ldx + j];
            xn = chk ? 4.0 * (xo - P) : (sq ? P : 2.0 * xo - P) + gamma * (xo - P);
            Xo[i * ldx + j] = xn;
            const double dd = P - xo;
            const double w = (j != i) ? 2.0 : 1.0;
            if (j == i) tr = xn;
            s2 = w * xn * xn;
            id = w * dd * dd;
        }
        sT[tx][ty] = xn;
        if (te.I == te.J) tr = warp_sum(tr);  // zero elsewhere
        s2 = warp_sum(s2);
        id = warp_sum(id);
        const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
        if (lane == 0) { red[0][wid] = tr; red[1][wid] = s2; red[2][wid] = id; }
        __syncthreads();
        // mirror: thread (ty, tx) writes row j0 + ty, column i0 + tx
        if (j0 + ty < n && i0 + tx < j0 + ty) Xo[(j0 + ty) * ldx + i0 + tx] = sT[ty][tx];
        // one sum per lane: an FP64 addition takes the pipe as long for one lane as for
        // three (with the packed sums of the control step, n = 256: 39.2 -> 37.7 us a step)
        if (threadIdx.x < 3) {
            double a = 0;
            for (int w = 0; w < 8; ++w) a += red[threadIdx.x][w];
            double *slot = pr.part + static_cast<size_t>(te.slot) * kPartStride;
            slot[threadIdx.x == 2 ? 3 : threadIdx.x] = a;
            if (threadIdx.x == 0) slot[2] = 0.0;
        }
        __syncthreads();
    }
}

}  // namespace fe
