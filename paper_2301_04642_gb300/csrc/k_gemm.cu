// The products on either side of the density-matrix step in Chebyshev-
// filtered subspace iteration (Sec. I and Sec. III-A): the Rayleigh-Ritz
// projection Hp = Psi^T (H Psi) that forms the input of the expansion, and
// the rotation Psi D that uses its output (density or subspace update).
// Psi is the m x n block of filtered vectors (m grid points, m >> n).
//
// Both are contractions C = A B^T over a K dimension, A and B given as K-major
// FP16 slices (hi + lo of s X, 22-bit operands, s a power of two from max|X|),
// computed on the 5th-generation tensor cores with FP32 accumulation:
//   projection: A = Psi^T, B = (H Psi)^T (both n x m, K = m), C symmetric n x n
//               (upper tiles, mirrored); the long K is cut into nsplit parts
//               whose FP32 partial tiles are summed in FP64, in a fixed order,
//               by k_gemm_reduce (split-K: more work units to balance over the
//               SMs, and shorter FP32 sums);
//   rotation:   A = Psi (m x n, K = n), B = D (n x n, symmetric), C = Psi D
//               written in FP64 by the epilogue.
// As in the expansion's kernel, an accumulator in tensor memory lives for one
// 64-wide K chunk (cross terms hi*lo, lo*hi first, hi*hi last) and the chunks
// are summed in registers with round-to-nearest.
//
// Tiles are 256 rows x bn columns (bn = 256, 128, 64 or 32), computed by a
// cluster of two CTAs (cta_group::2): each CTA holds 128 rows of A, bn/2 rows of
// B and the accumulators of its 128 rows, so that a chunk costs a CTA 64 KiB from L2
// for twice the products of a 128 x 192 tile (80 KiB).  A projection of 131072 x
// 4096 takes 4.0 ms here (5.5 ms with 128 x 192 tiles of one CTA), the rotation
// 9.2 ms (12.5 ms); narrow tiles fill the chip for small n (n = 517 from m = 9001:
// 27 us of 143).  Bound: the tensor cores at large n (6.6 and 13.2 TFLOP in those,
// 3.5 and 6.9 ms at 1.9 PFLOP/s) and, in the rotation, the 4.3 GB of FP64 output.
// The width is the one of the least modelled time (gemm_width).
// Warp roles (384 threads; warpgroup 0 hands registers to warpgroups 1-2):
//   warp 0      TMA producer: per K chunk one box per slice for this CTA's rows
//               of A (128) and of B (bn/2), three stages of 64 KiB;
//   warp 1      TMEM owner; in the leader CTA the MMA issuer: per chunk 4 x 3
//               MMAs M256 Nbn K16 into one of two chunk buffers;
//   warps 2-3   idle;
//   warps 4-11  drain + epilogue: warp w reads TMEM lanes 32 (w % 4) .. +31
//               and columns bn/2 ((w - 4) / 4) .. +bn/2-1 of the chunk.
// Every wait is bounded; on a timeout the kernel records an error code,
// waits (bounded) for its own copies and products in flight, frees TMEM and
// returns.
#include <cfloat>

#include "fe_dev.cuh"
#include "fe_kernels.cuh"

namespace fe {

namespace {

constexpr int kGemmStages = 3;
constexpr int kOutLd = 34;  // column stride of the output staging (no bank conflicts either way)
constexpr int kGemmHalf = kTileM * kTileK * 2;  // 16 KiB: 128 rows of one slice

struct alignas(1024) GemmStage {
    uint8_t a[kMaxSlices][kGemmHalf];
    uint8_t b[kMaxSlices][kGemmHalf];
};

struct GemmTail {
    uint64_t full[kGemmStages];   // leader: both CTAs' operand bytes have landed
    uint64_t empty[kGemmStages];  // both: the stage's MMAs are done
    uint64_t cfull[2];            // both: a chunk is in TMEM
    uint64_t cempty[2];           // leader: all drain warps of the pair have read it
    uint32_t tmem_base;
    int pad;
    float stage[kEpiWarps][16 * kOutLd];  // per-warp staging of 16 columns x 32 rows
};

constexpr size_t kGemmSmemBytes = 1024 + sizeof(GemmStage) * kGemmStages + sizeof(GemmTail);

__device__ __forceinline__ void record_error(DevCtl *ctl, int code) { atomicCAS(&ctl->err, 0, code); }

// e with m < 2^e <= 2 m for the largest magnitude m (bit pattern of an FP64 value;
// e = 0 for Inf, 1 for NaN and 0); slices are scaled by 2^(14 - e), so that they
// stay finite in FP16
__device__ __forceinline__ int max_exp(unsigned long long bits) {
    double m = __longlong_as_double(static_cast<long long>(bits));
    if (!(m > 0.0)) m = 1.0;
    int e;
    frexp(m, &e);  // m < 2^e
    return e;
}

// 16 columns of a warp's sums (lane = row) to its buffer
__device__ __forceinline__ void group_out(const float (&acc)[128], int gr, float *buf, int lane) {
#define FE_GROUP(G)                                                                        \
    case G: {                                                                              \
        _Pragma("unroll") for (int c = 0; c < 16; ++c) buf[c * kOutLd + lane] = acc[16 * G + c]; \
    } break;
    switch (gr) {
        FE_GROUP(0)
        FE_GROUP(1)
        FE_GROUP(2)
        FE_GROUP(3)
        FE_GROUP(4)
        FE_GROUP(5)
        FE_GROUP(6)
        FE_GROUP(7)
    }
#undef FE_GROUP
}

// x 2^e in FP64, rounded to nearest, by integer operations alone: a branch to FP64
// arithmetic for the rare encodings (which the compiler turned into selects) cost the
// rotation of 131072 x 4096 2.2 of 11.4 ms, of 20000 x 300 43 of 110 us
__device__ __forceinline__ double f32_to_f64_scaled(float x, int e) {
    const unsigned b = __float_as_uint(x);
    unsigned m = b & 0x7FFFFFu;
    int f = static_cast<int>((b >> 23) & 0xFFu);
    if (f == 0) {  // zero, or m 2^-149: leading bit to position 23
        const int z = __clz(static_cast<int>(m)) - 8;
        f = m ? 1 - z : -100000;
        m = (m << (z & 31)) & 0x7FFFFFu;
    }
    int r = f + 896 + e;
    unsigned long long v = (static_cast<unsigned long long>(m) << 29);
    if (f == 255) {
        r = 2047;  // Inf, NaN
    } else if (r >= 2047) {
        r = 2047;
        v = 0;
    } else if (r <= 0) {  // subnormal: the 53 bits shifted down, ties to even
        const int sh = min(1 - r, 60);
        const unsigned long long w = v | (1ull << 52), half = 1ull << (sh - 1);
        v = (w + (half - 1) + ((w >> sh) & 1)) >> sh;
        r = 0;  // a carry to 2^52 is the least normal number
    }
    v += (static_cast<unsigned long long>(r) << 52) | (static_cast<unsigned long long>(b >> 31) << 63);
    return __longlong_as_double(static_cast<long long>(v));
}

// Work unit u: part u / ntiles of tile u % ntiles.  The parts go outermost, so
// the work units that run at the same time (consecutive u over the pairs) read
// the same K range of their panels: one part of every panel fits L2 and is read
// from DRAM about once per wave.  Tiles: all of them row by row (nsplit = 0), or
// those of the upper triangle column by column.
struct Unit {
    int I, J, k0, k1;
};

__device__ __forceinline__ void tile_at(const GemmArgs &g, int t, int &I, int &J) {
    if (g.nsplit == 0) {
        I = t / g.ntj;
        J = t - I * g.ntj;
        return;
    }
    // q columns of width bn per 256 rows: column J has J / q + 1 tiles, the first
    // q b of them hold q b (b + 1) / 2
    const int q = 256 / g.bn;
    int b = static_cast<int>(sqrtf(2.0f * static_cast<float>(t) / static_cast<float>(q) + 0.25f) - 0.5f);
    while (b > 0 && static_cast<long long>(q) * b * (b + 1) / 2 > t) --b;
    while (static_cast<long long>(q) * (b + 1) * (b + 2) / 2 <= t) ++b;
    const int r = t - static_cast<int>(static_cast<long long>(q) * b * (b + 1) / 2);
    J = q * b + r / (b + 1);
    I = r % (b + 1);
}

__device__ __forceinline__ Unit unit_of(const GemmArgs &g, int u) {
    const int S = g.nsplit > 0 ? g.nsplit : 1;
    const int nk = (g.kdim + kTileK - 1) / kTileK;
    const int cs = (nk + S - 1) / S;
    Unit r;
    tile_at(g, u % g.ntiles, r.I, r.J);
    r.k0 = (u / g.ntiles) * cs;
    r.k1 = min(nk, r.k0 + cs);
    return r;
}

}  // namespace

__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kSymThreads, 1)
    k_gemm_split(const __grid_constant__ GemmArgs g, DevCtl *ctl) {
    extern __shared__ uint8_t smem_raw[];
    const uint32_t base_u32 = smem_u32(smem_raw);
    uint8_t *smem = smem_raw + ((1024u - (base_u32 & 1023u)) & 1023u);
    GemmStage *stages = reinterpret_cast<GemmStage *>(smem);
    GemmTail *tail = reinterpret_cast<GemmTail *>(smem + sizeof(GemmStage) * kGemmStages);
    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    const uint32_t rank = cluster_ctarank();
    const uint64_t wait_ns = ctl->wait_ns;
    const int nunits = g.ntiles * (g.nsplit > 0 ? g.nsplit : 1);
    const int u0 = blockIdx.x >> 1, du = gridDim.x >> 1;
    const int bn = g.bn;

    if (threadIdx.x == 0) {
        for (int s = 0; s < kGemmStages; ++s) {
            mbar_init(&tail->full[s], 1);
            mbar_init(&tail->empty[s], 1);
        }
        for (int a = 0; a < 2; ++a) {
            mbar_init(&tail->cfull[a], 1);
            mbar_init(&tail->cempty[a], 2 * kEpiWarps);
        }
        fence_barrier_init();
    }
    if (warp == 1) tmem_alloc_pair(&tail->tmem_base, 512);
    tc_fence_before();
    __syncthreads();
    cluster_sync();  // the peer's barriers are ready before anything signals them
    tc_fence_after();
    const uint32_t tmem_base = tail->tmem_base;

    if (warp < kSymEpiWarp0) setmaxnreg_dec<kSymRegsLow>();
    if (warp == 0) {
        // ------------------------------------------------------------ producer
        uint32_t stage = 0, phase = 0;
        bool ok = true;
        uint32_t last_phase[kGemmStages];
        bool issued[kGemmStages];
        for (int s = 0; s < kGemmStages; ++s) { issued[s] = false; last_phase[s] = 0; }
        // both CTAs' operands: 128 rows of A and bn/2 of B each
        const uint32_t bytes = static_cast<uint32_t>(2 * kMaxSlices * (kGemmHalf + bn * kTileK));
        for (int u = u0; u < nunits && ok; u += du) {
            const Unit un = unit_of(g, u);
            const int ya = (2 * un.I + static_cast<int>(rank)) * kTileM;
            const int yb = un.J * bn + static_cast<int>(rank) * (bn >> 1);
            for (int kc = un.k0; kc < un.k1; ++kc) {
                bool got = true;
                if (lane == 0) got = mbar_wait_bounded(&tail->empty[stage], phase ^ 1u, wait_ns);
                got = __shfl_sync(0xffffffffu, got, 0);
                if (!got) {
                    if (lane == 0) record_error(ctl, kErrTimeoutEmpty);
                    ok = false;
                    break;
                }
                if (lane == 0) {
                    if (rank == 0) mbar_expect_tx(&tail->full[stage], bytes);
                    const uint32_t bar = mapa_u32(&tail->full[stage], 0);
                    for (int s = 0; s < kMaxSlices; ++s) {
                        tma_load_2d_pair(stages[stage].a[s], &g.tA[s], bar, kc * kTileK, ya);
                        tma_load_2d_pair(stages[stage].b[s], &g.tB[s], bar, kc * kTileK, yb);
                    }
                }
                __syncwarp();
                issued[stage] = true;
                last_phase[stage] = phase;
                if (++stage == kGemmStages) { stage = 0; phase ^= 1u; }
            }
        }
        if (!ok && lane == 0) {
            // no TMA write may still be in flight when the CTA exits: the
            // leader's barriers count both CTAs' bytes, and the pair leaves
            // together; the peer gives its loads (microseconds) a millisecond
            if (rank == 0) {
                for (int s = 0; s < kGemmStages; ++s)
                    if (issued[s]) (void)mbar_wait_bounded(&tail->full[s], last_phase[s], wait_ns);
            } else {
                const uint64_t t0 = globaltimer();
                while (globaltimer() - t0 < 1000000ull) __nanosleep(1000);
            }
        }
        __syncwarp();
    } else if (warp == 1) {
        // ------------------------------------------------------------ MMA issuer
        uint32_t stage = 0, phase = 0, chunk = 0;
        bool ok = true, any_commit = false;
        const uint32_t idesc = idesc_f16(2 * kTileM, 0, 0) | (static_cast<uint32_t>(bn >> 3) << 17);
        for (int u = u0; rank == 0 && u < nunits && ok; u += du) {
            const Unit un = unit_of(g, u);
            for (int kc = un.k0; kc < un.k1; ++kc) {
                const uint32_t buf = chunk & 1u;
                const uint32_t cph = (chunk >> 1) & 1u;
                bool got = true;
                if (lane == 0) got = mbar_wait_bounded(&tail->cempty[buf], cph ^ 1u, wait_ns);
                got = __shfl_sync(0xffffffffu, got, 0);
                if (got) {
                    if (lane == 0) got = mbar_wait_bounded(&tail->full[stage], phase, wait_ns);
                    got = __shfl_sync(0xffffffffu, got, 0);
                    if (!got && lane == 0) record_error(ctl, kErrTimeoutFull);
                } else if (lane == 0) {
                    record_error(ctl, kErrTimeoutTmem);
                }
                if (!got) {
                    ok = false;
                    break;
                }
                tc_fence_after();
                if (lane == 0) {
                    const uint32_t tmem_d = tmem_base + buf * kTileN;
                    const uint64_t a0 = smem_desc_sw128(stages[stage].a[0]);
                    const uint64_t a1 = smem_desc_sw128(stages[stage].a[1]);
                    const uint64_t b0 = smem_desc_sw128(stages[stage].b[0]);
                    const uint64_t b1 = smem_desc_sw128(stages[stage].b[1]);
                    uint32_t accum = 0;
                    // small cross terms first: hi * lo, lo * hi
#pragma unroll
                    for (int kk = 0; kk < kTileK / 16; ++kk) {
                        const uint64_t off = static_cast<uint64_t>(kk * 2);  // 32 B along K
                        tc_mma_f16_pair(tmem_d, a0 + off, b1 + off, idesc, accum);
                        accum = 1;
                        tc_mma_f16_pair(tmem_d, a1 + off, b0 + off, idesc, accum);
                    }
                    // the full-magnitude hi * hi terms last
#pragma unroll
                    for (int kk = 0; kk < kTileK / 16; ++kk) {
                        const uint64_t off = static_cast<uint64_t>(kk * 2);
                        tc_mma_f16_pair(tmem_d, a0 + off, b0 + off, idesc, 1u);
                    }
                    tc_commit_pair(&tail->empty[stage]);  // smem stage may be refilled
                    tc_commit_pair(&tail->cfull[buf]);    // chunk ready for the drain
                    any_commit = true;
                }
                __syncwarp();
                if (++stage == kGemmStages) { stage = 0; phase ^= 1u; }
                ++chunk;
            }
        }
        if (!ok) {
            // every issued MMA must finish before TMEM is released
            if (lane == 0 && any_commit) {
                uint64_t *drain = &tail->cfull[chunk & 1u];
                tc_commit_pair(drain);
                (void)mbar_wait_bounded(drain, (chunk >> 1) & 1u, wait_ns);
            }
            __syncwarp();
        }
    } else if (warp >= kSymEpiWarp0) {
        // ------------------------------------------------------------ drain + epilogue
        setmaxnreg_inc<kSymRegsHigh>();
        const int ew = warp - kSymEpiWarp0;  // 0..7
        const int q = warp & 3;              // TMEM lane quadrant (hardware rule: warp % 4)
        const int h = ew >> 2;               // column half of the tile
        const int ncol = bn >> 1;
        const uint32_t cempty0[2] = {mapa_u32(&tail->cempty[0], 0), mapa_u32(&tail->cempty[1], 0)};
        uint32_t chunk = 0;
        bool ok = true;
        const int inv_e = max_exp(g.amax[0]) + max_exp(g.amax[1]) - 28;  // C = accumulator * 2^inv_e
        float *stg = tail->stage[ew];
        for (int u = u0; u < nunits && ok; u += du) {
            const Unit un = unit_of(g, u);
            const int i0 = (2 * un.I + static_cast<int>(rank)) * kTileM + q * 32;
            const int cb = un.J * bn + h * ncol;
            float acc[128];
#pragma unroll
            for (int c = 0; c < 128; ++c) acc[c] = 0.0f;
            for (int kc = un.k0; kc < un.k1; ++kc) {
                const uint32_t buf = chunk & 1u;
                const uint32_t cph = (chunk >> 1) & 1u;
                bool got = mbar_wait_bounded(&tail->cfull[buf], cph, wait_ns);
                got = __all_sync(0xffffffffu, got);
                if (!got) {
                    if (lane == 0) record_error(ctl, kErrTimeoutTmem);
                    ok = false;
                    break;
                }
                tc_fence_after();
                const uint32_t tbase = tmem_base + (static_cast<uint32_t>(q * 32) << 16) + buf * kTileN +
                                       static_cast<uint32_t>(h * ncol);
                if (ncol >= 32) {
#pragma unroll
                    for (int c4 = 0; c4 < 4; ++c4) {
                        if (c4 * 32 < ncol) {
                            float v[32];
                            tmem_ld32(tbase + c4 * 32, v);
#pragma unroll
                            for (int x = 0; x < 32; ++x) acc[c4 * 32 + x] += v[x];
                        }
                    }
                } else {
                    float v[16];
                    tmem_ld16(tbase, v);
#pragma unroll
                    for (int x = 0; x < 16; ++x) acc[x] += v[x];
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive_cluster(cempty0[buf]);
                ++chunk;
            }
            if (!ok) break;
            if (i0 >= g.rows_a || cb >= g.rows_b) continue;
            if (g.nsplit > 0) {
                // FP32 partial tile of this unit, [CTA][column][row]: a column's 32
                // rows of this warp are 128 consecutive bytes
                float *w = g.ws + (static_cast<size_t>(u) * 2 + rank) * static_cast<size_t>(kTileM * bn) +
                           static_cast<size_t>(h * ncol) * kTileM + q * 32 + lane;
#pragma unroll
                for (int c = 0; c < 128; ++c)
                    if (c < ncol) w[static_cast<size_t>(c) * kTileM] = acc[c];
                continue;
            }
            // direct FP64 output C[i][j], i < rows_a, j < rows_b.  Groups of 16 columns
            // go through the warp's buffer as FP32 (column-major, stride 34), then eight
            // lanes write the 128 bytes of a row and a store covers four rows.  The
            // scale is a power of two, added to the exponent by integer operations: as
            // an FP64 product with its conversion it took GB300's FP64 pipe (2 lanes a
            // clock and SM) 32 clocks per element and lane.  The loop over the groups
            // stays rolled (only the copy out of acc is unrolled): unrolled sixteen
            // times with an FP64 buffer the rotation of 131072 x 4096 took 20 ms, 9.2 with
            // this.
            const bool pair = (g.ldc & 1) == 0 && (reinterpret_cast<uintptr_t>(g.C) & 15u) == 0;
            const int c2 = 2 * (lane & 7), rr = lane >> 3;
#pragma unroll 1
            for (int gr = 0; gr < (ncol >> 4); ++gr) {
                const int j0 = cb + 16 * gr;
                if (j0 >= g.rows_b) break;
                group_out(acc, gr, stg, lane);
                __syncwarp();
                const int j = j0 + c2;
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    const int ii = i0 + 4 * k + rr;
                    const double v0 = f32_to_f64_scaled(stg[c2 * kOutLd + 4 * k + rr], inv_e);
                    const double v1 = f32_to_f64_scaled(stg[(c2 + 1) * kOutLd + 4 * k + rr], inv_e);
                    double *p = g.C + static_cast<long long>(ii) * g.ldc + j;
                    if (ii < g.rows_a) {
                        if (pair && j + 1 < g.rows_b) {
                            *reinterpret_cast<double2 *>(p) = make_double2(v0, v1);
                        } else {
                            if (j < g.rows_b) p[0] = v0;
                            if (j + 1 < g.rows_b) p[1] = v1;
                        }
                    }
                }
                __syncwarp();
            }
        }
    }

    tc_fence_before();
    __syncthreads();
    cluster_sync();  // nothing signals a CTA that has left
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc_pair(tmem_base, 512);
    }
}

// Sum of the nsplit FP32 partial tiles of every tile in a fixed order (FP64),
// scaled back by 1 / (s_A s_B), written to the upper part of the symmetric C
// and mirrored.  One block per 16 columns of a CTA's half of a tile (the partial
// tiles are [column][row]), so that few tiles still fill the chip: n = 517 from m =
// 9001 has 9 of 256 x 128, 144 blocks, 27 us; one block per tile took 234 us.  Bound
// at large n by the FP64 additions (2 per clock and SM); the FP32 terms are widened by
// integer operations to keep the conversions off that pipe (n = 4096 from m = 131072,
// 16 parts: 0.56 ms with a branch to the conversion for the rare encodings, 0.31 ms
// without one).  The upper rows go out through shared memory, 128 bytes at a time; the
// mirrored ones are written as they are read.
__global__ void __launch_bounds__(256) k_gemm_reduce(const __grid_constant__ GemmArgs g) {
    constexpr int kCols = 16;
    __shared__ double t[kTileM][kCols + 1];
    const int tile = blockIdx.x >> 1, rank = blockIdx.x & 1, c0 = blockIdx.y * kCols;
    int I, J;
    tile_at(g, tile, I, J);
    const int n = g.rows_a;
    const int i0 = (2 * I + rank) * kTileM, j0 = J * g.bn + c0;
    if (i0 >= n || j0 >= n || j0 + kCols - 1 < i0) return;
    const int S = g.nsplit;
    const double inv = ldexp(1.0, max_exp(g.amax[0]) + max_exp(g.amax[1]) - 28);
    const size_t half = static_cast<size_t>(kTileM) * g.bn;
    // part s at unit s * ntiles + tile
    const float *base = g.ws + static_cast<size_t>(2 * tile + rank) * half + static_cast<size_t>(c0) * kTileM;
    const size_t pstride = 2 * static_cast<size_t>(g.ntiles) * half;
    // thread: one row, columns cc, cc + 2, ...
    const int r = threadIdx.x % kTileM, cc = threadIdx.x / kTileM;
    const int i = i0 + r;
    double sum[kCols / 2];
#pragma unroll
    for (int q = 0; q < kCols / 2; ++q) sum[q] = 0.0;
    const float *b = base + static_cast<size_t>(cc) * kTileM + r;
    for (int s = 0; s < S; ++s, b += pstride) {
        float v[kCols / 2];
#pragma unroll
        for (int q = 0; q < kCols / 2; ++q) v[q] = b[2 * q * kTileM];
#pragma unroll
        for (int q = 0; q < kCols / 2; ++q) sum[q] += f32_to_f64_scaled(v[q], 0);
    }
#pragma unroll
    for (int q = 0; q < kCols / 2; ++q) {
        const int j = j0 + cc + 2 * q;
        const double v = sum[q] * inv;
        t[r][cc + 2 * q] = v;
        if (i < n && j < n && j > i) g.C[static_cast<long long>(j) * g.ldc + i] = v;
    }
    __syncthreads();
    for (int idx = threadIdx.x; idx < kTileM * kCols; idx += blockDim.x) {
        const int rr = idx / kCols, c = idx % kCols;
        const int ii = i0 + rr, jj = j0 + c;
        if (ii < n && jj < n && jj >= ii) g.C[static_cast<long long>(ii) * g.ldc + jj] = t[rr][c];
    }
}

namespace {

// hi = fp16(s x), lo = fp16(s x - hi) with s x formed in FP32 (s a power of
// two): hi + lo equals x to 2^-24 relative besides the FP32 rounding of x
__device__ __forceinline__ void split_pair(float x0, float x1, float s, __half2 &h, __half2 &l) {
    const float y0 = x0 * s, y1 = x1 * s;
    h = __floats2half2_rn(y0, y1);
    const float2 back = __half22float2(h);
    l = __floats2half2_rn(y0 - back.x, y1 - back.y);
}

}  // namespace

// max |X_ij| of both operands (blockIdx.y: which) as the bit pattern of a
// non-negative FP64 value (ordered like the value), atomically into *amax.
// Block b takes rows b, b + grid, ...; 16-byte loads where the rows are aligned,
// four in flight per thread.
__global__ void __launch_bounds__(256) k_absmax(const __grid_constant__ SplitArgs sa) {
    constexpr unsigned long long kAbs = 0x7FFFFFFFFFFFFFFFull;
    const SplitArgs::Op &op = sa.op[blockIdx.y];
    const long long rows = op.rows, cols = op.cols, ld = op.ld;
    const int t = threadIdx.x, nt = blockDim.x;
    unsigned long long m = 0;
    auto mag = [](double x) { return static_cast<unsigned long long>(__double_as_longlong(x)) & kAbs; };
    const bool pair = (ld & 1) == 0 && (reinterpret_cast<uintptr_t>(op.X) & 15u) == 0;
    for (long long r = blockIdx.x; r < rows; r += gridDim.x) {
        const double *row = op.X + r * ld;
        long long c = 0;
        if (pair) {
            const double2 *row2 = reinterpret_cast<const double2 *>(row);
            const long long half = cols >> 1;
            long long k = t;
            for (; k + 3 * nt < half; k += 4 * nt) {
                const double2 a = row2[k], b = row2[k + nt], d = row2[k + 2 * nt], e = row2[k + 3 * nt];
                m = max(max(max(m, max(mag(a.x), mag(a.y))), max(mag(b.x), mag(b.y))),
                        max(max(mag(d.x), mag(d.y)), max(mag(e.x), mag(e.y))));
            }
            for (; k < half; k += nt) {
                const double2 a = row2[k];
                m = max(m, max(mag(a.x), mag(a.y)));
            }
            c = 2 * half;
        }
        for (c += t; c < cols; c += nt) m = max(m, mag(row[c]));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((t & 31) == 0 && m != 0) atomicMax(op.amax, m);
}

// FP16 slices of both operands (blockIdx.y: which): hi = fp16(s x), lo =
// fp16(s x - hi), s from *amax.  A block of 256 threads takes 64 x 64 tiles, 16
// entries per thread in registers (rows ty + 8 k, columns 2 tx and 2 tx + 1):
// transpose = 0: out[r][c], one 128-byte row segment per warp and slice;
// transpose = 1: out[c][r], turned through shared memory.
// Bound by HBM: 8 bytes read and 4 written per element, after k_absmax has read
// the 8 bytes once.  Both operands of a 131072 x 4096 projection: 4.69 ms with the
// separate launches and a branching FP64-to-FP32 conversion, 3.38 with these.
__global__ void __launch_bounds__(256) k_split(const __grid_constant__ SplitArgs sa) {
    __shared__ float t[64][65];
    const SplitArgs::Op &op = sa.op[blockIdx.y];
    const double *__restrict__ X = op.X;
    const long long rows = op.rows, cols = op.cols, ld = op.ld, lds = op.lds;
    const int tid = threadIdx.x, tx = tid & 31, ty = tid >> 5;
    const long long tiles_c = (cols + 63) / 64, tiles_r = (rows + 63) / 64;
    const long long ntiles = tiles_r * tiles_c;
    const bool pair = (ld & 1) == 0 && (reinterpret_cast<uintptr_t>(X) & 15u) == 0;  // 16-byte loads
    const float s = ldexpf(1.0f, 14 - max_exp(*op.amax));
    for (long long tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        const long long br = tile / tiles_c, bc = tile - br * tiles_c;
        const long long r0 = br * 64 + ty, c = bc * 64 + 2 * tx;
        double x0[8], x1[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const long long r = r0 + 8 * k;
            x0[k] = x1[k] = 0.0;
            if (r < rows) {
                const double *p = X + r * ld + c;
                if (pair && c + 1 < cols) {
                    const double2 d = *reinterpret_cast<const double2 *>(p);
                    x0[k] = d.x;
                    x1[k] = d.y;
                } else {
                    if (c < cols) x0[k] = p[0];
                    if (c + 1 < cols) x1[k] = p[1];
                }
            }
        }
        if (!sa.transpose) {
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const long long r = r0 + 8 * k;
                if (r < rows && c < cols) {
                    __half2 h, l;
                    split_pair(f64_to_f32_rn(x0[k]), f64_to_f32_rn(x1[k]), s, h, l);
                    *reinterpret_cast<__half2 *>(op.hi + r * lds + c) = h;  // lds even
                    *reinterpret_cast<__half2 *>(op.lo + r * lds + c) = l;
                }
            }
            continue;
        }
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            t[2 * tx][ty + 8 * k] = f64_to_f32_rn(x0[k]);
            t[2 * tx + 1][ty + 8 * k] = f64_to_f32_rn(x1[k]);
        }
        __syncthreads();
        // output rows c, columns r: two columns per lane
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const int cc = ty + 8 * k;
            const long long oc = bc * 64 + cc, r = br * 64 + 2 * tx;
            if (oc < cols && r < rows) {
                __half2 h, l;
                split_pair(t[cc][2 * tx], t[cc][2 * tx + 1], s, h, l);
                *reinterpret_cast<__half2 *>(op.hi + oc * lds + r) = h;  // lds even, r even
                *reinterpret_cast<__half2 *>(op.lo + oc * lds + r) = l;
            }
        }
        __syncthreads();
    }
}

size_t gemm_smem_bytes() { return kGemmSmemBytes; }

}  // namespace fe
