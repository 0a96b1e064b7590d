// Symmetric products on the 5th-generation tensor cores with the update of
// the expansion fused into the epilogue (Sec. II-B1 Eq. (1), Sec. II-B3;
// Sec. III-B: the matrix product dominates the cost).
//
// Every step multiplies two symmetric, mutually commuting matrices given by
// their small parts A~, B~ (the identity parts are FP64 scalars in the solve
// state), so the product is symmetric and only upper-triangle 128x128 blocks
// are computed.  (A~ B~)_ij = sum_k A~_ik B~_jk: both operands are row panels
// of K-major FP16 slice arrays, loaded by TMA with 128-byte swizzling.  The
// epilogue evaluates up to three outputs  a v + b1 E1 + b2 E2 + c [i == j]
// (v the product, E1/E2 FP32 masters), writes them as FP32 masters, FP16
// slices for the next step and/or FP64 matrices, mirrors every value to the
// lower triangle, and leaves per-tile FP64 partials (trace and squared
// Frobenius norm of one output, trace of another, and an auxiliary sum of
// squares used as the idempotency measure ||X^2 - X||_F^2).  The step to run
// is described by the ProdOp the control step wrote into the solve state.
//
// Tiles and what bounds them.  A tile is 256 rows x bn columns (bn = 256, 128,
// 64 or 32), computed by a cluster of two CTAs (cta_group::2, M = 256): each
// CTA keeps 128 rows of A and bn/2 rows of B in its shared memory and the
// accumulators of its 128 rows in its tensor memory.  A split-FP16 chunk of
// K = 64 is twelve MMAs, 1536 clocks at bn = 256; a CTA of its own would have
// to take in 96 KiB for them (128 rows of A, 256 of B, two slices each), which
// an SM's 64 bytes a clock just cover and a loaded L2 does not; a pair takes in
// 64 KiB per CTA, and the third stage that then fits hides the load latency.
// A chunk takes 0.98 us at n = 8192 (0.65 in the single-FP16 form), against 1.21
// us for a CTA of its own; 0.80 (0.50) of it remains with every load and drain taken
// out, the hand-over of two tensor-memory buffers between the CTAs.  Launches at
// n = 16384: 11.6 -> 8.8 ms split, 8.4 -> 6.4 ms single.
// The narrow tiles are for problems with few tiles: a step's time is then one
// tile's K loop plus its store phase, both shorter the narrower it is
// (n = 384: 53 us a launch with tiles of 128 x 256, 27 with 256 x 32; n = 517,
// finite temperature: 133 and 40).  The host picks bn (choose_widths in fe_api.cu).
//
// Accuracy: the tensor core adds every MMA into its FP32 accumulator with a
// one-sided rounding, so an accumulator that lives for the whole K loop
// collects an error that grows with K.  Here an accumulator lives for one
// 64-wide K chunk only: per chunk the small cross terms hi*lo and lo*hi are
// issued first and the four hi*hi MMAs last, so the truncating additions at
// full magnitude are four per chunk.  The drain warps read each chunk from
// TMEM and sum the chunks in registers (round-to-nearest FP32) while the MMA
// thread fills the other chunk buffer.  A tile's chunks are summed in at most
// two runs, each in K order, whose cut run_cut() computes from the launch's
// work alone: an element's rounding depends neither on bn nor on which CTA
// computes it.
//
// Steps per launch.  With max_steps > 1 (a cooperative launch) the kernel runs
// the control step of every problem between two products, with a meeting of
// all CTAs before and after it, until a problem needs another kernel family,
// none is left, or max_steps products ran (see StepFlags).  As a pass of a graph
// loop (switch, product, control) a step cost about 25 us besides its product; the
// two meetings take 1.6 us each and the control step 4 to 9: n = 384 went from
// 77 us a step to 31, n = 517 at finite temperature from 146 to 35.
//
// Warp roles (384 threads; warpgroup 0 hands registers to warpgroups 1-2):
//   warp 0      TMA producer: per K chunk one box per slice for this CTA's
//               rows of A (128) and of B (bn/2), signalling the leader's barrier.
//   warp 1      TMEM owner; in the leader CTA the MMA issuer: per chunk
//               4 x (1 or 3) MMAs M256 Nbn K16 into one of two chunk buffers
//               (2 x 256 columns).
//   warps 2-3   idle (give their registers away)
//   warps 4-11  drain + epilogue: warp w reads TMEM lanes 32 (w % 4) .. +31
//               and the columns bn/2 ((w - 4) / 4) .. +bn/2-1; between steps
//               the control step and the next schedule table.
// Every wait is bounded; on a timeout the kernel records an error code,
// drains its own copies and MMAs, frees TMEM and returns.
#include "k_control.cuh"

namespace fe {

namespace {

constexpr int kSymStages = 3;
constexpr int kSymHalfBytes = kTileM * kTileK * 2;  // 16 KiB: 128 rows of one slice

struct alignas(1024) StageSmem {
    uint8_t a[kMaxSlices][kSymHalfBytes];
    uint8_t b[kMaxSlices][kSymHalfBytes];
};

// The step's schedule (built before every step by the drain warps).  Problems
// appear in two orders: by position in the launch's table (the reference
// tiling that run_cut() works on) and by descending dimension (the order
// in which tiles are handed out, so that the last ones are the small ones).
struct SchedHead {
    long long units;  // reference work units of the step
    int tiles;        // tiles of the step (pairs of CTAs)
    int rtiles;       // reference tiles
    int bnmin, wmin, wmax;
    int cont;         // 1: run this step, 0: leave
};
struct SchedRow {
    long long units;   // reference units of problems 0..q (inclusive)
    int rtiles;        // reference tiles of problems 0..q (inclusive)
    int w;             // reference units per tile of problem q (0: no work)
    int tiles;         // s-th largest problem and those before it: tiles (inclusive)
    int prob;          // the s-th largest problem
};

// One output of a step as the store phase reads it (shared memory, one copy
// per drain warp: read from the op descriptor in global memory the fields would
// be re-loaded after every store, which could alias them).
struct OutCache {
    float a, b1, b2, s, g1r, g1c, g2r, g2c;
    int flags, pad;
    float *master;
    __half *sl0, *sl1;
    double c, q, l1, l2;        // diagonal entry: c + a v_ii + q dx_i dy_i + l1 dx_i + l2 dy_i
    const double *dx, *dy;      // diagonal form: d vectors (null: 0)
    double *dgm;                // ... of the target, and their FP32 copy
    float *dgfm;
    double *X;                  // FP64 outputs: target, and addend (null: none)
    const double *Xa;
};
struct OpCache {
    float inv, ra, rb, rc;
    int nout, pout;
    const float *E1, *E2, *F1, *F2;  // E masters; FP32 diagonals that scale them (diagonal form)
    float *rsum;                     // reference-tile sums: squared sums of 8 columns (null: tile partials)
    long long ldr;
    OutCache out[3];
};

// Copies what the store phase needs of the step's operands; whole warp.
__device__ __forceinline__ void load_op(OpCache &oc, const MmaProb &pr, const ProdOp &op, int lane) {
    if (lane < 3) {
        const OutSpec &o = op.out[lane];
        OutCache &c = oc.out[lane];
        if (lane < op.nout) {
            const int fl = o.flags, mat = o.mat, dx = o.dx, dy = o.dy;
            c.a = o.a;
            c.b1 = o.b1;
            c.b2 = o.b2;
            c.s = o.s;
            c.g1r = o.g1r;
            c.g1c = o.g1c;
            c.g2r = o.g2r;
            c.g2c = o.g2c;
            c.flags = fl;
            c.master = pr.mats[mat].master;
            c.sl0 = pr.mats[mat].sl[0];
            c.sl1 = pr.mats[mat].sl[1];
            c.c = o.c;
            c.q = o.q;
            c.l1 = o.l1;
            c.l2 = o.l2;
            const bool dform = (fl & kOutDiag) != 0;
            c.dx = (dform && dx >= 0) ? pr.dg[dx] : nullptr;
            c.dy = (dform && dy >= 0) ? pr.dg[dy] : nullptr;
            c.dgm = dform ? pr.dg[mat] : nullptr;
            c.dgfm = dform ? pr.dgf[mat] : nullptr;
            c.X = pr.Xd[(fl & kOutF64b) ? 1 : 0];
            c.Xa = (fl & kOutF64Add) ? pr.Xd[(fl & kOutF64b) ? 0 : 1] : nullptr;
        }
    } else if (lane == 3) {
        oc.inv = op.inv;
        oc.ra = op.ra;
        oc.rb = op.rb;
        oc.rc = op.rc;
        oc.nout = op.nout;
        oc.pout = op.part_out;
        oc.E1 = (op.E1 >= 0) ? pr.mats[op.E1].master : nullptr;
        oc.E2 = (op.E2 >= 0) ? pr.mats[op.E2].master : nullptr;
        // the outputs of one step share their E1 / E2 coefficient vectors (the
        // control step sets them so)
        const float *f1 = nullptr, *f2 = nullptr;
        for (int o = 0; o < op.nout; ++o) {
            if (!(op.out[o].flags & kOutDiag)) continue;
            if (op.out[o].v1 >= 0) f1 = pr.dgf[op.out[o].v1];
            if (op.out[o].v2 >= 0) f2 = pr.dgf[op.out[o].v2];
        }
        oc.F1 = f1;
        oc.F2 = f2;
        oc.rsum = op.ref_sums ? pr.rsum : nullptr;
        oc.ldr = pr.ldr;
    }
    // every lane reads the copy, and an epilogue-only step has no chunk loop whose
    // barriers would stand between
    __syncwarp();
}

// FP64 partials of a tile, one thread's share.
struct TilePart {
    double tr = 0.0, sq = 0.0, tr1 = 0.0, rr = 0.0;
};

// Eight consecutive columns of one row: a lane's share of a 16-column group.
struct Eight {
    float x[8];
    __device__ __forceinline__ void zero() {
#pragma unroll
        for (int u = 0; u < 8; ++u) x[u] = 0.0f;
    }
    __device__ __forceinline__ void load(const float *p) {  // 16-byte aligned
        const float4 a = *reinterpret_cast<const float4 *>(p), b = *reinterpret_cast<const float4 *>(p + 4);
        x[0] = a.x; x[1] = a.y; x[2] = a.z; x[3] = a.w;
        x[4] = b.x; x[5] = b.y; x[6] = b.z; x[7] = b.w;
    }
};

// ---- Store phase of one warp's strip: rows i0 .. i0 + 31, columns cb .. cb +
// ncol - 1, from the register sums (lane = row, acc[c] = column cb + c).
//
// Groups of 16 columns go through a small per-warp buffer (column-major, stride
// 34: no bank conflicts either way) that turns lane = row into two lanes per
// row, eight columns each.  From there everything is in registers: E1/E2 come
// in as one full 32-byte sector per lane, E1 two half groups (of 16 rows) ahead,
// the FP16 slices are formed once for both places they go to, a row's 16
// columns leave as full sectors (lane pairs swap halves of the FP32 master), and
// the mirrored copies as 64-byte (master) and 32-byte (slices) runs over 16
// rows.  The loop over the groups is not unrolled: only the copy out of acc is,
// eight times 16 stores.  A 128 x 256 tile's phase takes 36 us at n = 4096 and 39 at
// n = 16384 (finite temperature, one output), all SMs storing at once at 2.6 TB/s
// over the chip; a 128 x 32 tile on the diagonal (three outputs), whose entries had
// loaded their operands one by one, went from 33 to 10 us.
//
// A group off the matrix edge and above the diagonal takes vector accesses;
// the others guarded 4-byte and 2-byte ones.
constexpr int kBufLd = 34;

__device__ __forceinline__ void group_to_buf(const float (&acc)[128], int g, float inv, float *buf, int lane) {
#define FE_GROUP(G)                                                                              \
    case G: {                                                                                    \
        _Pragma("unroll") for (int c = 0; c < 16; ++c) buf[c * kBufLd + lane] = acc[16 * G + c] * inv; \
    } break;
    switch (g) {
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

// packed FP16 pairs (columns 2p, 2p + 1) of s x: hi and lo slices
__device__ __forceinline__ void split_eight(const float *x, float s, uint32_t *hi, uint32_t *lo) {
#pragma unroll
    for (int p = 0; p < 4; ++p) {
        const float y0 = x[2 * p] * s, y1 = x[2 * p + 1] * s;
        const __half2 h = __floats2half2_rn(y0, y1);
        const float2 back = __half22float2(h);
        const __half2 l = __floats2half2_rn(y0 - back.x, y1 - back.y);
        hi[p] = *reinterpret_cast<const uint32_t *>(&h);
        lo[p] = *reinterpret_cast<const uint32_t *>(&l);
    }
}

// Mirrored slices of a lane's eight columns: lanes on neighbouring rows trade
// halves, so that each stores pairs (rows i, i + 1) of four columns.
__device__ __forceinline__ void put_mirror(__half *sl, const uint32_t *w, size_t at, int lds, bool odd) {
    __half *p0 = sl + at + (odd ? lds - 1 : 0);
    const size_t step = 2 * static_cast<size_t>(lds);
#pragma unroll
    for (int p = 0; p < 4; ++p) {
        // even row: column 2p of both rows; odd row: column 2p + 1
        const uint32_t nb = __shfl_xor_sync(0xffffffffu, w[p], 2);
        *reinterpret_cast<uint32_t *>(p0 + p * step) =
            odd ? __byte_perm(nb, w[p], 0x7632) : __byte_perm(w[p], nb, 0x5410);
    }
}

// Coefficient of an E term, q + g f.  Sums of a whole group of eight columns
// contract it, element-wise ones (the edge, the diagonal, FP64 outputs) round
// the product; results are bit for bit the same only while each place keeps its form.
__device__ __forceinline__ float e_coef(float g, float f, float q, bool whole) {
    return whole ? fmaf(g, f, q) : __fadd_rn(q, __fmul_rn(g, f));
}

template <bool kLean>
struct Strip {
    const OpCache &oc;
    const int n, ldy, lds, ldx, i0, cb, lane, half, r2;
    const float *const buf;
    TilePart &pt;

    // One half group on the vector path: rows i0 + r2 + 16 T, eight columns of this
    // lane from jb on.
    template <int T>
    __device__ __forceinline__ void vec(int jg, const Eight &e1, const float *E2, const float *F1, const float *F2,
                                        float d1, float d2) {
        const int jb = jg + 8 * half, i = i0 + r2 + 16 * T;
        const bool odd = (r2 & 1) != 0;
        Eight e2;
        e2.zero();
        if (!kLean && E2) e2.load(E2 + static_cast<size_t>(i) * ldy + jb);
        Eight f1, f2;
        if (!kLean) {
            f1.zero();
            f2.zero();
            if (F1) f1.load(F1 + jb);  // jb % 8 == 0, 64-byte aligned vectors
            if (F2) f2.load(F2 + jb);
        }
        float v[8];
        float crr = 0.0f;
        const float ra = oc.ra, rb = oc.rb;
#pragma unroll
        for (int u = 0; u < 8; ++u) v[u] = buf[(8 * half + u) * kBufLd + r2 + 16 * T];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const float r = fmaf(ra, v[u], rb * e1.x[u]);
            crr = fmaf(r, r, crr);
        }
        pt.rr = fma(2.0, f32_to_f64(crr), pt.rr);
        const size_t so = static_cast<size_t>(i) * lds + jb;
        const size_t ms = static_cast<size_t>(jb) * lds + i;
        const size_t mo = static_cast<size_t>(jb) * ldy + i;
        const int nout = kLean ? 1 : oc.nout, pout = kLean ? 0 : oc.pout;
#pragma unroll 1
        for (int o = 0; o < nout; ++o) {
            const OutCache &os = oc.out[o];
            const int fl = kLean ? (kOutMaster | kOutSlices) : os.flags;
            const bool dform = !kLean && (fl & kOutDiag);
            float val[8];
            float csq = 0.0f;
            const float oa = os.a, ob = os.b1;
            if (kLean) {
#pragma unroll
                for (int u = 0; u < 8; ++u) val[u] = fmaf(oa, v[u], ob * e1.x[u]);
            } else if (dform) {
                // per-row / per-column coefficients of E1 and E2
                const float q1 = fmaf(os.g1r, d1, ob), q2 = fmaf(os.g2r, d2, os.b2), g1 = os.g1c, g2 = os.g2c;
                const bool whole = !(fl & (kOutF64a | kOutF64b));
#pragma unroll
                for (int u = 0; u < 8; ++u)
                    val[u] = fmaf(oa, v[u], fmaf(e_coef(g1, f1.x[u], q1, whole), e1.x[u],
                                                 e_coef(g2, f2.x[u], q2, whole) * e2.x[u]));
            } else {
                const float b2 = os.b2;
#pragma unroll
                for (int u = 0; u < 8; ++u) val[u] = fmaf(oa, v[u], fmaf(ob, e1.x[u], b2 * e2.x[u]));
            }
            if (!kLean && (fl & (kOutF64a | kOutF64b))) {
                f64_out<true>(os, o == pout, o == 1, val, v, i, jb);
                continue;
            }
#pragma unroll
            for (int u = 0; u < 8; ++u) csq = fmaf(val[u], val[u], csq);
            if (!kLean && oc.rsum) oc.rsum[(jb >> 3) * oc.ldr + i] = 2.0f * csq;
            else if (o == pout) pt.sq = fma(2.0, f32_to_f64(csq), pt.sq);
            if (fl & kOutSlices) {
                uint32_t hi[4], lo[4];
                split_eight(val, os.s, hi, lo);
                *reinterpret_cast<uint4 *>(os.sl0 + so) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
                *reinterpret_cast<uint4 *>(os.sl1 + so) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
                put_mirror(os.sl0, hi, ms, lds, odd);
                put_mirror(os.sl1, lo, ms, lds, odd);
            }
            if (fl & kOutMaster) {
                if (!dform) {  // diagonal form: upper master only
                    float *m = os.master + mo;
#pragma unroll
                    for (int u = 0; u < 8; ++u, m += ldy) *m = val[u];
                }
                // the even lane keeps columns 0..3 of its eight and takes the odd
                // lane's 0..3, so that a lane pair fills a 32-byte sector per store
                float x[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) x[k] = __shfl_xor_sync(0xffffffffu, half ? val[k] : val[4 + k], 1);
                float *m = os.master + static_cast<size_t>(i) * ldy + jg + 4 * half;
                *reinterpret_cast<float4 *>(m) =
                    half ? make_float4(x[0], x[1], x[2], x[3]) : make_float4(val[0], val[1], val[2], val[3]);
                *reinterpret_cast<float4 *>(m + 8) =
                    half ? make_float4(val[4], val[5], val[6], val[7]) : make_float4(x[0], x[1], x[2], x[3]);
            }
        }
    }

    // FP64 output of eight columns.  FP32 terms are summed in FP32 and converted
    // exactly by integer operations: GB300's FP64 pipe (1/64 of the FP32 rate) keeps
    // only the FP64 diagonal, the FP64 addend and the squared norm.
    template <bool kVec>
    __device__ __forceinline__ void f64_out(const OutCache &os, bool part, bool part1, const float *val, const float *v,
                                            int i, int jb) {
        const size_t xo = static_cast<size_t>(i) * ldx + jb;
        auto ok = [&](int u) { return kVec || (i < n && jb + u < n && jb + u >= i); };
        double d[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) d[u] = (os.Xa && ok(u)) ? os.Xa[xo + u] : 0.0;
        const int ud = kVec ? -1 : i - jb;  // this lane's diagonal entry, if 0 <= ud < 8 and i < n
        double dv = 0.0;
        if (!kVec && ud >= 0 && ud < 8 && i < n) {
            float vd = 0.0f, wd = 0.0f;
#pragma unroll
            for (int u = 0; u < 8; ++u)
                if (u == ud) {
                    vd = v[u];
                    wd = val[u];
                }
            dv = (os.flags & kOutDiag) ? diag_entry(os, vd, i) : f32_to_f64(wd) + os.c;
        }
        double *X = os.X;
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            if (!ok(u)) continue;
            const bool dg = !kVec && u == ud;
            const double x = dg ? dv : f32_to_f64(val[u]);
            d[u] = os.Xa ? x + d[u] : x;
            X[xo + u] = d[u];
            if (!dg) X[static_cast<size_t>(jb + u) * ldx + i] = d[u];
            if (part) {
                if (dg) pt.tr += d[u];
                pt.sq = fma(dg ? d[u] : 2.0 * d[u], d[u], pt.sq);
            }
            if (part1 && dg) pt.tr1 += d[u];
        }
    }

    // diagonal entry of an output in the diagonal form, FP64
    __device__ __forceinline__ double diag_entry(const OutCache &os, float vd, int i) {
        const double dx = os.dx ? os.dx[i] : 0.0, dy = os.dy ? os.dy[i] : 0.0;
        const double r = os.c + static_cast<double>(os.a) * static_cast<double>(vd);
        return r + os.q * dx * dy + os.l1 * dx + os.l2 * dy;
    }

    // A half group with entries on or below the diagonal or beyond the edge.
    __device__ __forceinline__ void slow(int jg, int t, const float *E1, const float *E2, const float *F1,
                                         const float *F2, float d1, float d2) {
        const int jb = jg + 8 * half, i = i0 + r2 + 16 * t;
        unsigned okm = 0;  // entries of this lane that exist and lie on or above the diagonal
#pragma unroll
        for (int u = 0; u < 8; ++u)
            if (i < n && jb + u < n && jb + u >= i) okm |= 1u << u;
        const int ud = i - jb;
        const bool has_diag = ud >= 0 && ud < 8 && (okm >> ud & 1u);
        // a whole group of eight above the diagonal counts twice; elsewhere each
        // element is weighted by itself
        const bool full8 = i0 + 32 <= n && jb + 8 <= n && jb >= i0 + 32;
        const size_t ro = static_cast<size_t>(i) * ldy + jb;
        Eight e1, e2, f1, f2;
        e1.zero();
        e2.zero();
        f1.zero();
        f2.zero();
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const bool k = okm >> u & 1u;
            if (E1 && k) e1.x[u] = E1[ro + u];
            if (!kLean && E2 && k) e2.x[u] = E2[ro + u];
            if (!kLean && F1 && k) f1.x[u] = F1[jb + u];
            if (!kLean && F2 && k) f2.x[u] = F2[jb + u];
        }
        float v[8], vd = 0.0f;
        float crr = 0.0f;
        const float ra = oc.ra, rb = oc.rb, rc = oc.rc;
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            v[u] = buf[(8 * half + u) * kBufLd + r2 + 16 * t];
            const bool dg = u == ud;
            if (dg) vd = v[u];
            const float r = fmaf(ra, v[u], rb * e1.x[u]) + (dg ? rc : 0.0f);
            if (okm >> u & 1u) crr = fmaf(dg || full8 ? r : 2.0f * r, r, crr);
        }
        pt.rr = fma(full8 ? 2.0 : 1.0, f32_to_f64(crr), pt.rr);
        const int nout = kLean ? 1 : oc.nout, pout = kLean ? 0 : oc.pout;
#pragma unroll 1
        for (int o = 0; o < nout; ++o) {
            const OutCache &os = oc.out[o];
            const int fl = kLean ? (kOutMaster | kOutSlices) : os.flags;
            const bool dform = !kLean && (fl & kOutDiag);
            float val[8];
            const float q1 = dform ? fmaf(os.g1r, d1, os.b1) : os.b1, q2 = dform ? fmaf(os.g2r, d2, os.b2) : os.b2;
            const float g1 = dform ? os.g1c : 0.0f, g2 = dform ? os.g2c : 0.0f;
            const bool whole = full8 && !(fl & (kOutF64a | kOutF64b));
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                if (kLean) val[u] = fmaf(os.a, v[u], os.b1 * e1.x[u]);
                else val[u] = fmaf(os.a, v[u], fmaf(e_coef(g1, f1.x[u], q1, whole), e1.x[u],
                                                    e_coef(g2, f2.x[u], q2, whole) * e2.x[u]));
            }
            if (!kLean && (fl & (kOutF64a | kOutF64b))) {
                f64_out<false>(os, o == pout, o == 1, val, v, i, jb);
                continue;
            }
            if (has_diag) {
                float nd;  // the stored small part's diagonal entry
                if (dform) {
                    // the diagonal goes to the FP64 vector; the small part keeps 0
                    const double dv = diag_entry(os, vd, i);
                    os.dgm[i] = dv;
                    os.dgfm[i] = static_cast<float>(dv);
                    if (o == pout) {
                        pt.tr += dv;
                        pt.sq += dv * dv;
                    }
                    if (o == 1) pt.tr1 += dv;
                    nd = 0.0f;
                } else {
                    nd = 0.0f;
#pragma unroll
                    for (int u = 0; u < 8; ++u)
                        if (u == ud) nd = val[u] + static_cast<float>(os.c);
                    if (o == pout) pt.tr += static_cast<double>(nd);
                    if (o == 1) pt.tr1 += static_cast<double>(nd);
                }
#pragma unroll
                for (int u = 0; u < 8; ++u)
                    if (u == ud) val[u] = nd;
            }
            float csq = 0.0f;
            const float sc = os.s;
            uint32_t hi[4], lo[4];
            split_eight(val, sc, hi, lo);
            float *md = os.master + ro, *mm = os.master + static_cast<size_t>(jb) * ldy + i;
            __half *s0 = os.sl0, *s1 = os.sl1;
            const size_t so = static_cast<size_t>(i) * lds + jb, ms = static_cast<size_t>(jb) * lds + i;
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const bool k = okm >> u & 1u, dg = u == ud;
                if (k) csq = fmaf(dg || full8 ? val[u] : 2.0f * val[u], val[u], csq);
                if (k && (fl & kOutMaster)) {
                    md[u] = val[u];
                    if (!dg && !dform) mm[static_cast<size_t>(u) * ldy] = val[u];
                }
                if (k && (fl & kOutSlices)) {
                    const uint16_t h = static_cast<uint16_t>((u & 1) ? hi[u >> 1] >> 16 : hi[u >> 1] & 0xFFFFu);
                    const uint16_t l = static_cast<uint16_t>((u & 1) ? lo[u >> 1] >> 16 : lo[u >> 1] & 0xFFFFu);
                    reinterpret_cast<uint16_t *>(s0)[so + u] = h;
                    reinterpret_cast<uint16_t *>(s1)[so + u] = l;
                    if (!dg) {
                        reinterpret_cast<uint16_t *>(s0)[ms + static_cast<size_t>(u) * lds] = h;
                        reinterpret_cast<uint16_t *>(s1)[ms + static_cast<size_t>(u) * lds] = l;
                    }
                }
            }
            if (!kLean && oc.rsum) {
                if (i < n) oc.rsum[(jb >> 3) * oc.ldr + i] = full8 ? 2.0f * csq : csq;
            } else if (o == pout) {
                pt.sq = fma(full8 ? 2.0 : 1.0, f32_to_f64(csq), pt.sq);
            }
        }
    }

    __device__ __forceinline__ void run(const float (&acc)[128], float *wbuf, int ncol) {
        const float inv = oc.inv;
        const float *const E1 = oc.E1, *const E2 = kLean ? nullptr : oc.E2;
        const float *const F1 = kLean ? nullptr : oc.F1, *const F2 = kLean ? nullptr : oc.F2;
        // the rows' entries of the coefficient vectors, rows r2 and r2 + 16
        const int ia = i0 + r2, ib = ia + 16;
        float d1a = 0.0f, d1b = 0.0f, d2a = 0.0f, d2b = 0.0f;
        if (!kLean) {
            if (F1 && ia < n) d1a = F1[ia];
            if (F1 && ib < n) d1b = F1[ib];
            if (F2 && ia < n) d2a = F2[ia];
            if (F2 && ib < n) d2b = F2[ib];
        }
        const int ng = ncol >> 4;
        auto full16 = [&](int g) {
            const int jg = cb + 16 * g;
            return g < ng && i0 + 32 <= n && jg + 16 <= n && jg >= i0 + 32;
        };
        Eight pa, pb;  // E1 of rows r2 and r2 + 16, one group ahead
        pa.zero();
        pb.zero();
        const float *ea = E1 ? E1 + static_cast<size_t>(ia) * ldy + cb + 8 * half : nullptr;
        const size_t rows16 = 16 * static_cast<size_t>(ldy);
        if (E1 && full16(0)) {
            pa.load(ea);
            pb.load(ea + rows16);
        }
#pragma unroll 1
        for (int g = 0; g < ng; ++g) {
            const int jg = cb + 16 * g;
            if (jg >= n) break;
            const bool next = E1 && full16(g + 1);
            const float *en = ea + 16 * (g + 1);
            if (jg + 15 < i0) {  // wholly below the diagonal
                if (next) {
                    pa.load(en);
                    pb.load(en + rows16);
                }
                continue;
            }
            group_to_buf(acc, g, inv, wbuf, lane);
            __syncwarp();
            if (full16(g)) {
                Eight e = pa;
                if (next) pa.load(en);
                vec<0>(jg, e, E2, F1, F2, d1a, d2a);
                e = pb;
                if (next) pb.load(en + rows16);
                vec<1>(jg, e, E2, F1, F2, d1b, d2b);
            } else {
                slow(jg, 0, E1, E2, F1, F2, d1a, d2a);
                slow(jg, 1, E1, E2, F1, F2, d1b, d2b);
                if (next) {
                    pa.load(en);
                    pb.load(en + rows16);
                }
            }
            __syncwarp();  // the buffer is free for the next group
        }
    }
};

template <bool kLean>
__device__ __forceinline__ void store_strip(const float (&acc)[128], const OpCache &oc, const MmaProb &pr, float *buf,
                                            int i0, int cb, int ncol, int lane, TilePart &pt) {
    Strip<kLean> st{oc, pr.n, pr.ldy, pr.lds, pr.ldx, i0, cb, lane, lane & 1, lane >> 1, buf, pt};
    st.run(acc, buf, ncol);
}

struct MmaSmemTail {
    uint64_t full[kSymStages];   // leader: both CTAs' operand bytes have landed
    uint64_t empty[kSymStages];  // both: the stage's MMAs are done
    uint64_t cfull[2];           // both: a chunk is in TMEM
    uint64_t cempty[2];          // leader: all drain warps of the pair have read it
    uint32_t tmem_base;
    int step_ok;
    double red[kEpiWarps][4];
    int vote[kEpiWarps];
    union {
        float buf[kEpiWarps][16 * kBufLd];  // per-warp transposition buffer of the store phase
        ControlSmem ctl;                    // between steps
    };
    OpCache oc[kEpiWarps];
    SchedHead head;
    SchedRow row[kSchedTabProbs];
};

constexpr size_t kMmaSmemBytes = 1024 + sizeof(StageSmem) * kSymStages + sizeof(MmaSmemTail);
static_assert(kMmaSmemBytes <= 227 * 1024, "shared memory of one CTA");

__device__ __forceinline__ int step_kind(const SolveState *st) {
    return *reinterpret_cast<const volatile int *>(&st->kind);
}

__device__ __forceinline__ bool tc_kind(int kind) {
    return kind == kTcSingle || kind == kTcSplit || kind == kTcElem || kind == kTcDelta;
}

// FP16 slices per operand: two for the split products
__device__ __forceinline__ int step_slices(const SolveState *st) {
    const int kind = step_kind(st);
    return (kind == kTcSplit || kind == kTcDelta) ? 2 : 1;
}

// K chunks of this step (0 for an epilogue-only step)
__device__ __forceinline__ int step_chunks(const SolveState *st, int n) {
    return step_kind(st) == kTcElem ? 0 : (n + kTileK - 1) / kTileK;
}

__device__ __forceinline__ void record_error(DevCtl *ctl, int code) { atomicCAS(&ctl->err, 0, code); }

// named barriers: the 8 drain/epilogue warps; all 12 warps of the CTA
__device__ __forceinline__ void epi_bar() { asm volatile("bar.sync 1, 256;" ::: "memory"); }
__device__ __forceinline__ void step_bar() { asm volatile("bar.sync 2, 384;" ::: "memory"); }

// ---- Where a tile's chunk sum is cut.  The reference schedule, on which the
// rounding of a step is defined, runs over the reference tiles of the active
// problems in table order (128 rows x ref_bn columns, ref_bn = 256 or 128), each
// worth `units` = its chunks (1 for an epilogue-only step) times its width over
// the narrowest one.  When every tile is worth the same and there are at least
// two waves of `ref_ctas` tiles, whole waves are left whole; the remaining one
// to two waves (all tiles otherwise) are cut into G <= ref_ctas equal contiguous
// ranges of units, G at most the number of largest tiles, so a tile holds at
// most one range end.  A chunk belongs to the range that holds its first unit.

// Position of reference tile (I, J) in its problem's list: bands of
// kRefBand (kRefBandN for 128-wide tiles) row panels, column by column.
__device__ __forceinline__ int ref_index(int n, int ref_bn, int I, int J) {
    const int T = (n + kTileM - 1) / kTileM;
    if (ref_bn == kTileM) {
        const int b0 = I / kRefBandN * kRefBandN, R = min(kRefBandN, T - b0);
        const int base = b0 * T - b0 * (b0 - 1) / 2;  // tiles of the bands before
        const int d = J - b0, m = min(d, R);            // columns before J; those not yet full
        return base + m * (m + 1) / 2 + (d - m) * R + (I - b0);
    }
    const int TP = (T + 1) / 2;
    const int b0 = I / kRefBand * kRefBand, R = min(kRefBand, T - b0);
    const int base = b0 * TP - (b0 > 0 ? (b0 - 1) * (b0 - 1) / 4 : 0);
    const int d = J - b0 / 2, m = min(d, R / 2);
    return base + m * (m + 1) + (d - m) * R + (I - b0);
}

// First chunk of the second run of block (I, column block J128) of problem q
// (0: one run).  nk: the step's chunks.
__device__ int run_cut(const SchedHead &sh, const SchedRow *row, const MmaProb &pr, int q, int ref_ctas, int nk, int I,
                       int J128) {
    if (nk < 2) return 0;
    const long long r = ref_index(pr.n, pr.ref_bn, I, pr.ref_bn == kTileM ? J128 : J128 / 2);
    long long whole = 0;  // tiles in whole waves
    if (sh.wmin == sh.wmax && sh.rtiles >= 2 * ref_ctas)
        whole = (sh.rtiles % ref_ctas == 0) ? sh.rtiles : static_cast<long long>(sh.rtiles / ref_ctas - 1) * ref_ctas;
    if ((q ? row[q - 1].rtiles : 0) + r < whole) return 0;
    const int w = row[q].w, f = pr.ref_bn / sh.bnmin;
    const long long u0 = whole * sh.wmax;
    const long long W = sh.units - u0;
    long long G = W / sh.wmax;
    G = G > ref_ctas ? ref_ctas : G;
    if (G < 2) return 0;
    const long long x = (q ? row[q - 1].units : 0) + r * w - u0;  // the tile's first unit
    // the first range end beyond x; ends lie at floor(W b / G)
    long long b = x * G / W + 1;
    while (b < G && W * b / G <= x) ++b;
    if (b >= G) return 0;
    const long long ku = W * b / G - x;
    if (ku >= w) return 0;
    const int k = static_cast<int>((ku + f - 1) / f);
    return k < nk ? k : 0;
}

// The sums that a finite-temperature step hands to the control of mu (tr z and
// ||z||_F^2; D follows mu continuously, and a last bit of a sum can flip FP32
// roundings all over the next stages) are defined on the reference tiles, so that
// they depend neither on bn nor on which CTA stored what: per row of a tile's
// 32 x (ref_bn / 2) strips, FP64 sums over the 8-column FP32 sums the store phase
// left in rsum, in column order, with the diagonal's square before its group; a
// tree over the strip's rows; the strips in order.  256 threads, one tile per call.
template <class Bar>
__device__ void ref_tile_sums(const MmaProb &pr, int tile, double (*red)[4], int t, Bar bar) {
    const int n = pr.n, T = (n + kTileM - 1) / kTileM;
    const int w = t >> 5, lane = t & 31, q = w & 3, h = w >> 2;
    const bool wide = pr.ref_bn == kTileN;
    const int TP = wide ? (T + 1) / 2 : T;
    // row-major tile number -> (I, J), J >= I / 2 (or I)
    auto row0 = [&](int I) {
        return wide ? I * TP - (I > 0 ? (I - 1) * (I - 1) / 4 : 0) : I * TP - I * (I - 1) / 2;
    };
    int lo = 0, hi = T - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (row0(mid) <= tile) lo = mid;
        else hi = mid - 1;
    }
    const int I = lo, J = tile - row0(I) + (wide ? I / 2 : I);
    const int i0 = I * kTileM + q * 32, i = i0 + lane;
    const int ncol = pr.ref_bn >> 1, cb = J * pr.ref_bn + h * ncol;
    double tr = 0.0, sq = 0.0;
    if (cb / kTileM >= I && i0 < n) {
        const SolveState *st = pr.st;
        const double *dg = pr.dg[st->op.out[0].mat];
        for (int g = 0; g < ncol / 8; ++g) {
            const int j0 = cb + 8 * g;
            if (j0 >= n) break;
            if (j0 + 7 < i0) continue;
            if (i >= j0 && i < j0 + 8 && i < n) {
                const double dv = __ldcg(dg + i);
                tr += dv;
                sq += dv * dv;
            }
            if (i < n) sq += static_cast<double>(__ldcg(pr.rsum + static_cast<size_t>(j0 >> 3) * pr.ldr + i));
        }
    }
    tr = warp_sum(tr);
    sq = warp_sum(sq);
    if (lane == 0) {
        red[w][0] = tr;
        red[w][1] = sq;
    }
    bar();
    if (t < 2) {
        double a = 0.0;
        for (int x = 0; x < kEpiWarps; ++x) a += red[x][t];
        pr.part[static_cast<size_t>(tile) * kPartStride + t] = a;
    }
    bar();
}

// The schedule table of the next step, by the 256 drain threads.  Returns
// bit 0: some problem has tensor-core work, bit 1: some problem waits for
// another kernel family, bit 2: some step of bit 0 has reference-tile sums.
// A table beyond kSchedTabProbs has its rows in global memory (one copy per CTA) and
// keeps the table's order.
__device__ int sched_build(SchedHead *sh, SchedRow *row, const MmaProb *probs, int np, int t, int *mask) {
    // per problem: w = units per reference tile before the width factor,
    // rtiles, tiles, and in units the reference width
    if (t == 0) *mask = 0;
    epi_bar();
    int m = 0;
    for (int q = t; q < np; q += kCtlThreads) {
        const MmaProb &pr = probs[q];
        const int kind = step_kind(pr.st);
        const bool act = pr.tc_ntiles > 0 && tc_kind(kind);
        if (act) m |= 1;
        if (act && *reinterpret_cast<const volatile int *>(&pr.st->op.ref_sums)) m |= 4;
        if (kind == kDigit || kind == kFp64) m |= 2;
        const int nk = act ? step_chunks(pr.st, pr.n) : 0;
        row[q].w = act ? (nk > 0 ? nk : 1) : 0;
        row[q].rtiles = act ? pr.ref_ntiles : 0;
        row[q].units = act ? pr.ref_bn : 0;
        row[q].tiles = act ? pr.tc_ntiles : 0;
        row[q].prob = q;
    }
    if (m) atomicOr(mask, m);
    epi_bar();
    if (np > 1 && np <= kSchedTabProbs) {
        // order by descending dimension (ties: table order)
        int rank = 0, tl = 0;
        if (t < np) {
            const int n = probs[t].n;
            for (int r = 0; r < np; ++r) {
                const int nr = probs[r].n;
                rank += (nr > n || (nr == n && r < t)) ? 1 : 0;
            }
            tl = row[t].tiles;
        }
        epi_bar();
        if (t < np) {
            row[rank].tiles = tl;
            row[rank].prob = t;
        }
        epi_bar();
    }
    if (t < 32) {
        int bm = kTileN;
        for (int q = t; q < np; q += 32)
            if (row[q].w > 0) bm = min(bm, static_cast<int>(row[q].units));
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) bm = min(bm, __shfl_xor_sync(0xffffffffu, bm, o));
        const int per = (np + 31) / 32;
        const int q0 = t * per, q1 = min(q0 + per, np);
        long long su = 0;
        int sr = 0, sl = 0, wmin = 0x7fffffff, wmax = 1;
        for (int q = q0; q < q1; ++q) {
            const int c = row[q].w;
            const int w = c > 0 ? c * (static_cast<int>(row[q].units) / bm) : 0;
            if (c > 0) {
                wmin = min(wmin, w);
                wmax = max(wmax, w);
            }
            su += static_cast<long long>(row[q].rtiles) * w;
            sr += row[q].rtiles;
            sl += row[q].tiles;
            row[q].w = w;
            row[q].units = su;
            row[q].rtiles = sr;
            row[q].tiles = sl;
        }
        long long eu = su;
        int er = sr, el = sl;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const long long yu = __shfl_up_sync(0xffffffffu, eu, o);
            const int yr = __shfl_up_sync(0xffffffffu, er, o);
            const int yl = __shfl_up_sync(0xffffffffu, el, o);
            if (t >= o) {
                eu += yu;
                er += yr;
                el += yl;
            }
        }
        if (t == 31) {
            sh->units = eu;
            sh->rtiles = er;
            sh->tiles = el;
        }
        eu -= su;
        er -= sr;
        el -= sl;
        for (int q = q0; q < q1; ++q) {
            row[q].units += eu;
            row[q].rtiles += er;
            row[q].tiles += el;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            wmin = min(wmin, __shfl_xor_sync(0xffffffffu, wmin, o));
            wmax = max(wmax, __shfl_xor_sync(0xffffffffu, wmax, o));
        }
        if (t == 0) {
            sh->bnmin = bm;
            sh->wmin = wmin;
            sh->wmax = wmax;
        }
    }
    const int due = *mask;
    epi_bar();
    return due;
}

// The tiles of one step that this cluster computes: rounds of one tile per
// cluster, every other round in reverse, so that over two rounds of a list
// ordered by size every cluster gets about the same work.
struct TileIter {
    const SchedHead *sh;
    const SchedRow *row;
    int np, cluster, nclusters, round;

    __device__ TileIter(const SchedHead *h, const SchedRow *r, int n)
        : sh(h), row(r), np(n), cluster(blockIdx.x >> 1), nclusters(gridDim.x >> 1), round(0) {}

    // problem and index in its tile list
    __device__ bool next(int &prob, int &idx) {
        const long long g = static_cast<long long>(round) * nclusters +
                            ((round & 1) ? nclusters - 1 - cluster : cluster);
        ++round;
        if (g >= sh->tiles) return false;  // (only in the last round)
        int lo = 0, hi = np - 1;
        while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if (row[mid].tiles > g) hi = mid;
            else lo = mid + 1;
        }
        prob = row[lo].prob;
        idx = static_cast<int>(g) - (lo ? row[lo - 1].tiles : 0);
        return true;
    }
};

// All blocks of the launch meet (a cooperative launch: all are resident).
// The counter grows by the number of blocks per meeting.  CTAs without a tile
// wait here for the whole step, so the limit is eight of the bounded waits.
// With fail_partner set the wait watches a word nothing writes.
__device__ bool grid_meet(unsigned *cnt, unsigned nb, DevCtl *ctl, uint64_t wait_ns) {
    __threadfence();
    const unsigned old = atomicAdd(cnt, 1u);
    const unsigned target = old - old % nb + nb;
    const unsigned *watch = ctl->fail_partner ? reinterpret_cast<const unsigned *>(&ctl->never) : cnt;
    const unsigned want = ctl->fail_partner ? 1u : target;
    bool ok = true;
    if (static_cast<int>(ld_acquire_u32(watch) - want) < 0) {
        const uint64_t t0 = globaltimer();
        while (static_cast<int>(ld_acquire_u32(watch) - want) < 0) {
            if (globaltimer() - t0 > 8 * wait_ns) {
                ok = false;
                break;
            }
            __nanosleep(20);
        }
    }
    if (!ok) record_error(ctl, kErrTimeoutGrid);
    __threadfence();
    return ok;
}

}  // namespace

__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kSymThreads, 1)
    k_sym_mma(const MmaProb *__restrict__ probs, int nprobs, const TileEnt *__restrict__ tiles, DevCtl *ctl,
              float *ws, char *gsched, StepFlags *flags, int ref_ctas, int max_steps) {
    extern __shared__ uint8_t smem_raw[];
    const uint32_t base_u32 = smem_u32(smem_raw);
    uint8_t *smem = smem_raw + ((1024u - (base_u32 & 1023u)) & 1023u);
    StageSmem *stages = reinterpret_cast<StageSmem *>(smem);
    MmaSmemTail *tail = reinterpret_cast<MmaSmemTail *>(smem + sizeof(StageSmem) * kSymStages);
    SchedRow *row = nprobs <= kSchedTabProbs
                        ? tail->row
                        : reinterpret_cast<SchedRow *>(gsched) + static_cast<size_t>(blockIdx.x) * nprobs;

    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    const uint32_t rank = cluster_ctarank();
    const uint64_t wait_ns = ctl->wait_ns;

    if (threadIdx.x == 0) {
        for (int s = 0; s < kSymStages; ++s) {
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
        uint32_t last_phase[kSymStages];
        bool issued[kSymStages];
        for (int s = 0; s < kSymStages; ++s) { issued[s] = false; last_phase[s] = 0; }
        for (;;) {
            step_bar();
            if (!tail->head.cont) break;
            fence_proxy_async_global();  // slices written by other SMs since the last step
            TileIter it(&tail->head, row, nprobs);
            int prob, idx;
            while (ok && it.next(prob, idx)) {
                const MmaProb &pr = probs[prob];
                const TileEnt te = tiles[pr.tc_tile0 + idx];
                const SolveState *st = pr.st;
                const int S = step_slices(st);
                const int bn = te.bn, nk = step_chunks(st, pr.n);
                const CUtensorMap *tma = pr.mats[st->op.A].tm128;
                const MatSlot &mb = pr.mats[st->op.B];
                const CUtensorMap *tmb = bn == 256 ? mb.tm128 : bn == 128 ? mb.tm64 : bn == 64 ? mb.tm32 : mb.tm16;
                const int ya = (2 * te.I + static_cast<int>(rank)) * kTileM;
                const int yb = te.Jp * bn + static_cast<int>(rank) * (bn >> 1);
                // both CTAs' operands: 128 rows of A and bn/2 of B each
                const uint32_t bytes = static_cast<uint32_t>(2 * S * (kSymHalfBytes + bn * kTileK));
                for (int kc = 0; kc < nk; ++kc) {
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
                        for (int s = 0; s < S; ++s) {
                            tma_load_2d_pair(stages[stage].a[s], &tma[s], bar, kc * kTileK, ya);
                            tma_load_2d_pair(stages[stage].b[s], &tmb[s], bar, kc * kTileK, yb);
                        }
                    }
                    __syncwarp();
                    issued[stage] = true;
                    last_phase[stage] = phase;
                    if (++stage == kSymStages) { stage = 0; phase ^= 1u; }
                }
            }
            step_bar();
        }
        if (!ok) {
            // no TMA write may still be in flight when the CTA exits: the
            // leader's barriers count both CTAs' bytes, and the pair leaves
            // together; the peer gives its loads (microseconds) a millisecond
            if (lane == 0) {
                if (rank == 0) {
                    for (int s = 0; s < kSymStages; ++s)
                        if (issued[s]) (void)mbar_wait_bounded(&tail->full[s], last_phase[s], wait_ns);
                } else {
                    const uint64_t t0 = globaltimer();
                    while (globaltimer() - t0 < 1000000ull) __nanosleep(1000);
                }
            }
            __syncwarp();
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------ MMA issuer
        uint32_t stage = 0, phase = 0;
        uint32_t chunk = 0;  // chunk counter of this pair: buffer = chunk & 1
        bool ok = true;
        bool any_commit = false;
        for (;;) {
            step_bar();
            if (!tail->head.cont) break;
            TileIter it(&tail->head, row, nprobs);
            int prob, idx;
            while (rank == 0 && ok && it.next(prob, idx)) {
                const MmaProb &pr = probs[prob];
                const SolveState *st = pr.st;
                const int S = step_slices(st), nk = step_chunks(st, pr.n);
                const uint32_t idesc = idesc_f16(2 * kTileM, 0, 0) | (static_cast<uint32_t>(tiles[pr.tc_tile0 + idx].bn >> 3) << 17);
                for (int kc = 0; kc < nk; ++kc) {
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
                        const uint64_t b0 = smem_desc_sw128(stages[stage].b[0]);
                        uint32_t accum = 0;
                        if (S == 2) {
                            const uint64_t a1 = smem_desc_sw128(stages[stage].a[1]);
                            const uint64_t b1 = smem_desc_sw128(stages[stage].b[1]);
                            // small cross terms first: hi * lo, lo * hi
#pragma unroll
                            for (int kk = 0; kk < kTileK / 16; ++kk) {
                                const uint64_t off = static_cast<uint64_t>(kk * 2);  // 32 B along K
                                tc_mma_f16_pair(tmem_d, a0 + off, b1 + off, idesc, accum);
                                accum = 1;
                                tc_mma_f16_pair(tmem_d, a1 + off, b0 + off, idesc, accum);
                            }
                        }
                        // the full-magnitude hi * hi terms last
#pragma unroll
                        for (int kk = 0; kk < kTileK / 16; ++kk) {
                            const uint64_t off = static_cast<uint64_t>(kk * 2);
                            tc_mma_f16_pair(tmem_d, a0 + off, b0 + off, idesc, accum);
                            accum = 1;
                        }
                        tc_commit_pair(&tail->empty[stage]);  // smem stage may be refilled
                        tc_commit_pair(&tail->cfull[buf]);    // chunk ready for the drain
                        any_commit = true;
                    }
                    __syncwarp();
                    if (++stage == kSymStages) { stage = 0; phase ^= 1u; }
                    ++chunk;
                }
            }
            step_bar();
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
    } else if (warp < kSymEpiWarp0) {
        for (;;) {
            step_bar();
            if (!tail->head.cont) break;
            step_bar();
        }
    } else {
        // ------------------------------------------------------------ drain + epilogue
        setmaxnreg_inc<kSymRegsHigh>();
        const int ew = warp - kSymEpiWarp0;    // 0..7
        const int et = threadIdx.x - 32 * kSymEpiWarp0;
        const int q = warp & 3;                // TMEM lane quadrant (hardware rule: warp % 4)
        const int h = ew >> 2;                 // column half of the tile
        const uint32_t cempty0[2] = {mapa_u32(&tail->cempty[0], 0), mapa_u32(&tail->cempty[1], 0)};
        float *const wrow = ws + static_cast<size_t>(blockIdx.x) * kRunSlotFloats +
                            (static_cast<size_t>(ew) * 32 + lane) * 128;  // the first run's sums
        uint32_t chunk = 0;
        bool ok = true;
        int steps = 0;
        bool controlled = false;  // the control step of the last product ran here
        int last_due = 0;
        for (;;) {
            // ---- the next step's schedule.  While another family's step is
            // due the loop pauses: from the start one product is run (its
            // control step follows that family's kernels), after a control
            // step the kernel leaves.
            const int due = sched_build(&tail->head, row, probs, nprobs, et, &tail->step_ok);
            const bool single = max_steps <= 1 || (due & 2);
            const bool cont = ok && (due & 1) && steps < max_steps && (steps == 0 || (controlled && !(due & 2)));
            if (et == 0) tail->head.cont = cont ? 1 : 0;
            last_due = due;
            step_bar();
            if (!cont) break;
            ++steps;
            controlled = false;
            TileIter it(&tail->head, row, nprobs);
            int prob, idx;
            while (ok && it.next(prob, idx)) {
                const MmaProb &pr = probs[prob];
                const TileEnt te = tiles[pr.tc_tile0 + idx];
                const SolveState *st = pr.st;
                const int n = pr.n;
                const int ncol = te.bn >> 1;  // columns of this warp's strip
                const int I = 2 * te.I + static_cast<int>(rank);
                const int cb = te.Jp * te.bn + h * ncol;  // first column of the strip
                const int nk = step_chunks(st, n);
                // a strip wholly outside the upper triangle is drained, not kept
                const bool live = cb / kTileM >= I && cb < n && I * kTileM < n;
                __syncwarp();
                load_op(tail->oc[ew], pr, st->op, lane);
                const int cut = live ? run_cut(tail->head, row, pr, prob, ref_ctas, nk, I, cb / kTileM) : 0;
                float acc[128];
#pragma unroll
                for (int c = 0; c < 128; ++c) acc[c] = 0.0f;
                for (int kc = 0; kc < nk; ++kc) {
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
                    if (kc == cut && kc > 0) {
                        // the second run starts: the first one's sums wait in L2
#pragma unroll
                        for (int c = 0; c < 32; ++c)
                            if (4 * c < ncol) {
                                __stcg(reinterpret_cast<float4 *>(wrow) + c,
                                       make_float4(acc[4 * c], acc[4 * c + 1], acc[4 * c + 2], acc[4 * c + 3]));
                                acc[4 * c] = acc[4 * c + 1] = acc[4 * c + 2] = acc[4 * c + 3] = 0.0f;
                            }
                    }
                    const uint32_t tbase = tmem_base + (static_cast<uint32_t>(q * 32) << 16) +
                                           buf * kTileN + static_cast<uint32_t>(h * ncol);
                    if (!live) {
                        // nothing to keep
                    } else if (ncol >= 64) {
#pragma unroll
                        for (int c2 = 0; c2 < 2; ++c2) {
                            if (c2 * 64 < ncol) {
                                float v[64];
                                tmem_ld64(tbase + c2 * 64, v);
#pragma unroll
                                for (int u = 0; u < 64; ++u) acc[c2 * 64 + u] += v[u];
                            }
                        }
                    } else if (ncol == 32) {
                        float v[32];
                        tmem_ld32(tbase, v);
#pragma unroll
                        for (int u = 0; u < 32; ++u) acc[u] += v[u];
                    } else {
                        float v[16];
                        tmem_ld16(tbase, v);
#pragma unroll
                        for (int u = 0; u < 16; ++u) acc[u] += v[u];
                    }
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive_cluster(cempty0[buf]);
                    ++chunk;
                }
                if (cut > 0) {
#pragma unroll
                    for (int c = 0; c < 32; ++c) {
                        if (4 * c >= ncol) break;
                        const float4 p4 = __ldcg(reinterpret_cast<const float4 *>(wrow) + c);
                        acc[4 * c] += p4.x;
                        acc[4 * c + 1] += p4.y;
                        acc[4 * c + 2] += p4.z;
                        acc[4 * c + 3] += p4.w;
                    }
                }

                TilePart pt;
                const int i0 = I * kTileM + q * 32;
                if (live && ok && i0 < n) {
                    const OpCache &oc = tail->oc[ew];
                    const bool lean = oc.nout == 1 && oc.pout == 0 && !oc.E2 &&
                                      oc.out[0].flags == (kOutMaster | kOutSlices);
                    if (lean) store_strip<true>(acc, oc, pr, tail->buf[ew], i0, cb, ncol, lane, pt);
                    else store_strip<false>(acc, oc, pr, tail->buf[ew], i0, cb, ncol, lane, pt);
                }
                // per-tile partials in a fixed order: warp tree, then the 8 warps.  Only
                // tiles on the diagonal have traces.
                const bool on_diag = cb < I * kTileM + kTileM;
                pt.sq = warp_sum(pt.sq);
                pt.rr = warp_sum(pt.rr);
                if (on_diag) {
                    pt.tr = warp_sum(pt.tr);
                    pt.tr1 = warp_sum(pt.tr1);
                }
                if (lane == 0) {
                    tail->vote[ew] = ok ? 1 : 0;
                    tail->red[ew][0] = pt.tr;
                    tail->red[ew][1] = pt.sq;
                    tail->red[ew][2] = pt.tr1;
                    tail->red[ew][3] = pt.rr;
                }
                epi_bar();
                if (et < 4) {
                    double a = 0.0;
                    for (int w = 0; w < kEpiWarps; ++w) a += tail->red[w][et];
                    pr.part[static_cast<size_t>(2 * te.slot + static_cast<int>(rank)) * kPartStride + et] = a;
                }
                // a warp whose chunk loop ended early (only on a timeout) stored
                // nothing; all of them leave together
                for (int w = 0; w < kEpiWarps; ++w) ok = ok && tail->vote[w] != 0;
                epi_bar();
            }
            step_bar();  // every warp is done with this step's table
            if (max_steps <= 1 || (single && !(due & 4))) continue;
            // ---- control step between two products: everything this step
            // wrote is visible before it, its decisions before the next product
            __threadfence();
            fence_proxy_async_global();
            epi_bar();
            // (a CTA that failed meets the others all the same: the control step
            // sees its error and ends every problem)
            auto meet = [&]() {
                if (et == 0) tail->step_ok = grid_meet(&ctl->sym_bar, gridDim.x, ctl, wait_ns) ? 1 : 0;
                epi_bar();
                const bool met = tail->step_ok != 0;
                epi_bar();
                return met;
            };
            bool met = meet();
            if (met && (due & 4)) {
                for (int p = 0; p < nprobs; ++p) {
                    const MmaProb &pr = probs[p];
                    if (row[p].w == 0 || !pr.st->op.ref_sums) continue;
                    for (int k = blockIdx.x; k < pr.ref_ntiles; k += gridDim.x)
                        ref_tile_sums(pr, k, tail->red, et, [] { epi_bar(); });
                }
                __threadfence();
                epi_bar();
                met = meet();
            }
            if (single) {
                ok = ok && met;
                continue;
            }
            if (met)
                for (int p = blockIdx.x; p < nprobs; p += gridDim.x) {
                    (void)control_one(probs[p], ctl, &tail->ctl, et, [] { epi_bar(); });
                    epi_bar();
                }
            ok = met && meet() && ok;
            controlled = true;
        }
        if (et == 0 && blockIdx.x == 0 && flags && steps > 0) {
            flags->n_steps += static_cast<unsigned>(controlled ? steps : steps - 1);
            flags->controlled = (controlled && ok) ? 1u : 0u;
            // products of this kernel and of another family that are due in the same
            // step run in the same pass, the next one
            ctl->hold = (controlled && ok && (last_due & 1) && (last_due & 2)) ? 1 : 0;
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

__global__ void __launch_bounds__(kCtlThreads) k_ref_sums(const MmaProb *__restrict__ probs, int nprobs) {
    __shared__ double red[kEpiWarps][4];
    for (int p = 0; p < nprobs; ++p) {
        const MmaProb &pr = probs[p];
        if (pr.tc_ntiles == 0 || !tc_kind(step_kind(pr.st)) || !pr.st->op.ref_sums) continue;
        for (int k = blockIdx.x; k < pr.ref_ntiles; k += gridDim.x)
            ref_tile_sums(pr, k, red, threadIdx.x, [] { __syncthreads(); });
    }
}

size_t mma_smem_bytes() { return kMmaSmemBytes; }
size_t sched_row_bytes() { return sizeof(SchedRow); }

}  // namespace fe
