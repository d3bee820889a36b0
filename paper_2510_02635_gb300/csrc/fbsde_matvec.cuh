// fbsde_matvec.cuh -- the matrix-free product of the regression operator (the dominant
// work of a solve), fed by bulk copies (TMA) through an mbarrier-synchronised
// shared-memory ring.  Included after fbsde_kernels.cuh.
#pragma once
#include "fbsde_kernels.cuh"

namespace fbsde {
namespace dev {

// ---------------------------------------------------------------------------
// mbarrier + bulk-copy (TMA) helpers.  Every wait is bounded: after kWaitNs of
// %globaltimer without completion it returns false and the caller records
// FBSDE_ERR_TIMEOUT instead of spinning forever.
// ---------------------------------------------------------------------------
constexpr unsigned long long kWaitNs = 5ull * 1000 * 1000 * 1000;

__device__ __forceinline__ uint32_t smem_u32(const void *ptr)
{
    return (uint32_t)__cvta_generic_to_shared(ptr);
}
__device__ __forceinline__ unsigned long long globaltimer_ns()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}
__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count)
                 : "memory");
}
__device__ __forceinline__ void fence_mbar_init()
{
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t *bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)),
                 "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t *bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t *bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n"
        "  .reg .pred q;\n"
        "  mbarrier.try_wait.parity.shared::cta.b64 q, [%1], %2;\n"
        "  selp.u32 %0, 1, 0, q;\n"
        "}\n"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}
// Waits for the completion of the barrier phase with the given parity; false on timeout.
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, uint32_t parity,
                                          unsigned long long limit_ns = kWaitNs)
{
    if (mbar_try_wait(bar, parity)) return true;
    const unsigned long long t0 = globaltimer_ns();
    for (;;) {
        if (mbar_try_wait(bar, parity)) return true;
        if (globaltimer_ns() - t0 > limit_ns) return false;
    }
}
// Bounded wait whose failure is sticky: after the first timeout of this thread, later
// waits only poll once, so a broken pipeline costs one kWaitNs per thread, not one per
// stage.
__device__ __forceinline__ void mbar_wait_or_flag(uint64_t *bar, uint32_t parity, bool &timed_out,
                                                  unsigned long long limit_ns = kWaitNs)
{
    if (timed_out) {
        (void)mbar_try_wait(bar, parity);
        return;
    }
    if (!mbar_wait(bar, parity, limit_ns)) timed_out = true;
}

// Bulk copy global -> shared memory; completion is signalled on bar as transaction bytes.
__device__ __forceinline__ void bulk_g2s(void *dst, const void *src, uint32_t bytes, uint64_t *bar)
{
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::
            "r"(smem_u32(dst)),
        "l"(src), "r"(bytes), "r"(smem_u32(bar))
        : "memory");
}

// ---------------------------------------------------------------------------
// Matrix-free product of the regression (Sec. 2.4, Steps 1 and 2) on the centred operator:
// for one chunk g of a query's rows, partial_g = sum_j w_j (D_j . r) D_j and the share
// sum_j w_j (D_j . r)^2 of r^T A r, r = vR(s, 0).  The rows reach shared memory by bulk
// copies; nteams teams of tw warps take one row at a time: dot product, team sum (warp
// butterfly + one named barrier), then the weighted row sum into register accumulators.
// The team of a row is its index in the chunk modulo nteams, so the sums do not depend on
// how the rows are staged; k_matvec (one launch per product) and k_cg_loop (the whole CG
// in one launch) run these functions on the same chunks and give the same bits.
// ---------------------------------------------------------------------------
struct MvTeam {
    int tw, nteams, tthreads, team, tl, wt, lane, nch;
    __device__ __forceinline__ MvTeam(int tw_, int nteams_, int nch_)   // consumers: warps 1..
        : tw(tw_), nteams(nteams_), tthreads(32 * tw_), lane(threadIdx.x & 31), nch(nch_)
    {
        const int ct = (int)threadIdx.x - 32;
        team = ct / tthreads;
        tl = ct - team * tthreads;
        wt = tl >> 5;
    }
};

// Dot product and weighted sum of 16-byte chunks; FP32 as pairs (one packed instruction for
// two fused multiply-adds).
template <typename Real> struct DotAcc;
template <> struct DotAcc<double> {
    double s;
    __device__ __forceinline__ void init() { s = 0.0; }
    __device__ __forceinline__ void add(const Chunk<double> &a, const Chunk<double> &b)
    {
        s = fma(a.v[0], b.v[0], s);
        s = fma(a.v[1], b.v[1], s);
    }
    __device__ __forceinline__ double sum() const { return s; }
};
template <> struct DotAcc<float> {
    float2 s;
    __device__ __forceinline__ void init() { s = make_float2(0.f, 0.f); }
    __device__ __forceinline__ void add(const Chunk<float> &a, const Chunk<float> &b)
    {
        s = __ffma2_rn(make_float2(a.v[0], a.v[1]), make_float2(b.v[0], b.v[1]), s);
        s = __ffma2_rn(make_float2(a.v[2], a.v[3]), make_float2(b.v[2], b.v[3]), s);
    }
    __device__ __forceinline__ float sum() const { return s.x + s.y; }
};
__device__ __forceinline__ void chunk_axpy(Chunk<double> &y, double a, const Chunk<double> &x)
{
    y.v[0] = fma(a, x.v[0], y.v[0]);
    y.v[1] = fma(a, x.v[1], y.v[1]);
}
__device__ __forceinline__ void chunk_axpy(Chunk<float> &y, float a, const Chunk<float> &x)
{
    const float2 aa = make_float2(a, a);
    const float2 l = __ffma2_rn(aa, make_float2(x.v[0], x.v[1]), make_float2(y.v[0], y.v[1]));
    const float2 h = __ffma2_rn(aa, make_float2(x.v[2], x.v[3]), make_float2(y.v[2], y.v[3]));
    y.v[0] = l.x;
    y.v[1] = l.y;
    y.v[2] = h.x;
    y.v[3] = h.y;
}

// Sum of w t^2 over a team's rows, in the team's first thread.  FP32 rows: compensated FP32 sums
// (64-bit operations in the row loop cost it 4 to 30%), of t scaled by a power of two near
// 1 / |r|: t^2 itself leaves the FP32 range where t does not (sigma = 1e-5: t ~ 1e-20 after a few
// passes).  The rounding of the two products does not show: with their rounding errors added
// back the slopes are as far from 64 bits (d = 1000 reverse sweep, eight seeds, 5.62e-6 both
// ways; d = 64, 1.42e-6 and 1.45e-6).  FP64 rows: one multiply-add a row.
template <typename Real> struct DeltaAcc;
template <> struct DeltaAcc<float> {
    RedAcc<float> a;
    float scale;   // 2^-e
    // rr: r . r, now or a pass before; only its exponent counts (integer arithmetic:
    // FP64 comparisons in every warp held the SM's FP64 pipe for 0.3 us a pass at d = 64)
    __device__ __forceinline__ void init(double rr)
    {
        a.init();
        const int f = (__double2hiint(rr) >> 20) & 0xFFF;   // sign and exponent
        const int e = f > 0 && f < 0x7FF ? max(-126, min(126, (f - 1023) / 2)) : 0;
        scale = __uint_as_float((uint32_t)(127 - e) << 23);
    }
    __device__ __forceinline__ void add(float w, float t)
    {
        const float ts = __fmul_rn(t, scale);
        a.add(__fmul_rn(__fmul_rn(w, ts), ts));
    }
    __device__ __forceinline__ double value() const { return a.value(); }   // scaled by 4^-e
    // A sum of such values times 4^e, by its exponent (0, infinities and NaN stay)
    __device__ __forceinline__ double back(double d) const
    {
        const int e = 127 - (int)(__float_as_uint(scale) >> 23);
        const int hi = __double2hiint(d), f = (hi >> 20) & 0x7FF;
        return f == 0 || f == 0x7FF ? d : __hiloint2double(hi + ((2 * e) << 20), __double2loint(d));
    }
};
template <> struct DeltaAcc<double> {
    double d;
    __device__ __forceinline__ void init(double) { d = 0.0; }
    __device__ __forceinline__ void add(double w, double t) { d += w * t * t; }
    __device__ __forceinline__ double value() const { return d; }
    __device__ __forceinline__ double back(double v) const { return v; }
};

// NR rows at a time (1 or 2): t = row . r, acc += w t row in row order; the team's first
// thread adds w t^2 to dacc.  rel0, rel1: "empty" barriers of the stages whose last rows
// these are (or null); with the rows held in registers they are released before the
// butterfly, which leaves the ring more bytes in flight.  Two rows share the latency of the loads, the butterfly and the
// team's barrier: the butterfly's first step leaves one row's sums in each half of the warp,
// so its other steps add both at once.  Each row's sum has the same bits either way.
// kReread: the thread's chunks of the row are read from shared memory again for the weighted
// sum (teams of more than 10 warps, or 16 chunks per thread, whose registers are short); with
// 16 the operand too is read from memory for every row.
template <typename Real, int VPT, bool kReread, int NR>
__device__ __forceinline__ void mv_rows(const Real *const (&row)[NR], const Real (&w)[NR],
                                        const Real *opmem, const Chunk<Real> (&pc)[VPT],
                                        Chunk<Real> (&acc)[VPT], DeltaAcc<Real> &dacc, const MvTeam &m,
                                        Real *slots, int &phase, uint64_t *rel0, uint64_t *rel1)
{
    constexpr int E = Chunk<Real>::E;
    constexpr bool kOpMem = VPT > 8;
    auto release = [&]() {
        __syncwarp();
        if (m.lane == 0) {
            if (rel0) mbar_arrive(rel0);
            if (rel1) mbar_arrive(rel1);
        }
    };
    constexpr int kHeld = kReread ? 1 : VPT;
    Chunk<Real> dl[NR][kHeld];
    DotAcc<Real> ta[NR];
#pragma unroll
    for (int n = 0; n < NR; ++n) ta[n].init();
#pragma unroll
    for (int v = 0; v < VPT; ++v) {
        // past the row's end: its last chunk, with a zero operand (and sums never stored)
        const int c = m.tl + m.tthreads * v, cc = min(c, m.nch - 1);
        Chunk<Real> o;
        if (!kOpMem) {
            o = pc[v];
        } else {
            if (c < m.nch) o = ldg_chunk(opmem + c * E);
            else zero(o);
        }
#pragma unroll
        for (int n = 0; n < NR; ++n) {
            Chunk<Real> &x = dl[n][kReread ? 0 : v];
            x = ld_chunk(row[n] + cc * E);
            ta[n].add(x, o);
        }
    }
    Real t[NR];
#pragma unroll
    for (int n = 0; n < NR; ++n) t[n] = ta[n].sum();
    if (!kReread) release();   // the rows are in registers
    if constexpr (NR == 2) {
        const bool hi = m.lane & 16;
        Real keep = hi ? t[1] : t[0];
        const Real give = hi ? t[0] : t[1];
        keep += __shfl_xor_sync(0xffffffffu, give, 16);
#pragma unroll
        for (int o = 8; o; o >>= 1) keep += __shfl_xor_sync(0xffffffffu, keep, o);
        if (m.tw == 1) {
            const Real other = __shfl_xor_sync(0xffffffffu, keep, 16);
            t[0] = hi ? other : keep;
            t[1] = hi ? keep : other;
        } else {
            Real *sl = slots + (size_t)(m.team * 2 + phase) * 32;
            if ((m.lane & 15) == 0) sl[2 * m.wt + (hi ? 1 : 0)] = keep;
        }
    } else {
#pragma unroll
        for (int o = 16; o; o >>= 1) t[0] += __shfl_xor_sync(0xffffffffu, t[0], o);
        if (m.tw > 1) {
            Real *sl = slots + (size_t)(m.team * 2 + phase) * 32;
            if (m.lane == 0) sl[2 * m.wt] = t[0];
        }
    }
    if (m.tw > 1) {
        const Real *sl = slots + (size_t)(m.team * 2 + phase) * 32;
        bar_named(1 + m.team, m.tthreads);
        if constexpr (sizeof(Real) == 8) {
            // a lane per warp's sum, a half-warp per row: log2(tw) adds for both rows in place of
            // 2 tw.  A warp's FP64 add holds the SM's FP64 pipe for 16 cycles, and the pipe bounds
            // the product (d = 1203, M = 2048: 23.4 us a pass, 25.5 us with tw adds a row).
            const int i = m.lane & 15, n = NR == 2 ? m.lane >> 4 : 0;
            Real x = i < m.tw ? sl[2 * i + n] : Real(0);
            for (int o = 1; o < m.tw; o <<= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
#pragma unroll
            for (int k = 0; k < NR; ++k) t[k] = __shfl_sync(0xffffffffu, x, 16 * k);
        } else {
#pragma unroll
            for (int n = 0; n < NR; ++n) t[n] = Real(0);
            for (int w2 = 0; w2 < m.tw; ++w2) {
#pragma unroll
                for (int n = 0; n < NR; ++n) t[n] += sl[2 * w2 + n];
            }
        }
        phase ^= 1;
    }
#pragma unroll
    for (int n = 0; n < NR; ++n) {
        const Real coef = w[n] * t[n];
        if (m.tl == 0) dacc.add(w[n], t[n]);
#pragma unroll
        for (int v = 0; v < VPT; ++v) {
            if (kReread) dl[n][0] = ld_chunk(row[n] + min(m.tl + m.tthreads * v, m.nch - 1) * E);
            chunk_axpy(acc[v], coef, dl[n][kReread ? 0 : v]);
        }
    }
    if (kReread) release();
}

// How a team of 8 chunks per thread walks its rows (4 and fewer: always held, in pairs):
//   kMvHold  several teams share the rows: one row at a time, held in registers, its stage
//            released before the butterfly (d = 1000, M = 4096, 64 queries: 169 us a product,
//            184 us in pairs, whose two stages leave the ring fewer bytes in flight);
//   kMvPair  one team for all rows: two at a time, read again for the weighted sum, so that
//            one butterfly and one barrier serve both (d = 10^4, M = 16384, 16 queries:
//            1375 us a product, 1540 us one at a time: the chain of a row's steps bounds it);
//   kMvWide  as kMvPair with teams of 11 to 16 warps.
enum MvMode { kMvHold = 0, kMvPair = 1, kMvWide = 2 };

// Rows of a chunk that a thread adds up in FP32 before the sum goes on elsewhere: an FP32 run of n
// rows loses about sqrt(n) roundings.  d = 5003, M = 16000, one query: slopes 7.2e-6 from the
// FP64 path with runs of 105 rows, 5.8e-6 with 32.
constexpr int kMvRun = 32;

// Position of a consumer in the ring of row stages.
struct MvRing {
    int slot, par, S, R;
    __device__ __forceinline__ void next()
    {
        if (++slot == S) {
            slot = 0;
            par ^= 1;
        }
    }
};

// The thread's chunks of `sum` (shared memory) added to its accumulators.
template <typename Real, int VPT>
__device__ __forceinline__ void mv_add_runs(const Real *sum, const MvTeam &m, Chunk<Real> (&acc)[VPT])
{
    constexpr int E = Chunk<Real>::E;
#pragma unroll
    for (int v = 0; v < VPT; ++v) {
        const int c = m.tl + m.tthreads * v;
        if (c < m.nch) {
            const Chunk<Real> o = ld_chunk(sum + c * E);
#pragma unroll
            for (int e = 0; e < E; ++e) acc[v].v[e] += o.v[e];
        }
    }
}

// The consumers' part of one chunk, rows [r0, r1): its stages of R rows (a multiple of the
// teams) from the ring, released after use unless they stay (release = false).  wv: the
// weights from row r0 on.  kPair: two rows of a team at a time (of two stages where a stage
// holds one row per team).  FP32 rows of one team that reads them again, or of one chunk per thread:
// every kMvRun rows of a team its accumulators go into its row of `sum` ([nteams][ld] in shared
// memory, each thread its own chunks); returns whether they did.
template <typename Real, int VPT, bool kReread, bool kPair>
__device__ __forceinline__ bool mv_chunk(long long r0, long long r1, Real *sum, const Real *wv,
                                         const Real *opmem, const Chunk<Real> (&pc)[VPT],
                                         Chunk<Real> (&acc)[VPT], DeltaAcc<Real> &dacc, const MvTeam &m,
                                         const Real *ring, uint64_t *full, uint64_t *empty,
                                         MvRing &rg, bool release, Real *slots, int &phase,
                                         bool &timed_out)
{
    const size_t ld = (size_t)m.nch * Chunk<Real>::E;
    const int nrows = (int)(r1 - r0), nt = m.nteams;
    const bool across = kPair && rg.R == nt;
    auto one = [&](const Real *p0, Real w0, uint64_t *rel) {
        const Real *const row[1] = {p0};
        const Real w[1] = {w0};
        mv_rows<Real, VPT, kReread, 1>(row, w, opmem, pc, acc, dacc, m, slots, phase, rel, nullptr);
    };
    auto none = [&](uint64_t *rel0, uint64_t *rel1) {   // stages without a row for this team
        if (m.lane == 0) {
            if (rel0) mbar_arrive(rel0);
            if (rel1) mbar_arrive(rel1);
        }
    };
    // the weights of the team's next two rows, requested one step ahead of their use
    auto weight = [&](int j) { return j < nrows ? wv[j] : Real(0); };
    Real n0 = weight(m.team), n1 = weight(m.team + nt);
    // Runs end at the team's row 32, 64, ..: a pair never straddles two, so that they do not
    // depend on the stages.  (Rows of one team that are read again come one a stage, where run
    // stays even, or a few of them stay resident.)
    constexpr bool kRuns = sizeof(Real) == 4 && kReread, kRunsIn = sizeof(Real) == 4 && VPT == 1;
    const bool more = kRunsIn && nrows > kMvRun * nt;   // a team has more than one run
    Real *const mine = sum + (size_t)m.team * ld;
    bool flushed = false;
    int run = 0;
    auto next_run = [&]() {   // before a row of the team
        if (run < kMvRun) return;
        if (flushed) mv_add_runs<Real, VPT>(mine, m, acc);
#pragma unroll
        for (int v = 0; v < VPT; ++v) {
            const int c = m.tl + m.tthreads * v;
            if (c < m.nch) st_chunk(mine + c * Chunk<Real>::E, acc[v]);
            zero(acc[v]);
        }
        flushed = true;
        run = 0;
    };
    for (int base = 0; base < nrows;) {
        if (kRuns || (more && across && base + m.team < nrows)) next_run();
        const int a = rg.slot, rows = min(rg.R, nrows - base);
        const Real *buf = ring + (size_t)a * rg.R * ld;
        uint64_t *ea = release ? &empty[a] : nullptr;
        if (across) {
            const int j = base + m.team, j2 = j + nt;
            const bool two = base + nt < nrows;   // this stage and the next
            const Real w0 = n0, w1 = n1;
            n0 = weight(j + 2 * nt);
            n1 = weight(j + 3 * nt);
            mbar_wait_or_flag(&full[a], (uint32_t)rg.par, timed_out);
            rg.next();
            const int b = rg.slot;
            if (two) {
                mbar_wait_or_flag(&full[b], (uint32_t)rg.par, timed_out);
                rg.next();
            }
            uint64_t *eb = release && two ? &empty[b] : nullptr;
            const Real *p0 = buf + (size_t)m.team * ld;
            const Real *p1 = ring + ((size_t)b * rg.R + m.team) * ld;
            if constexpr (kPair) {
                if (j2 < nrows) {
                    const Real *const row[2] = {p0, p1};
                    const Real w[2] = {w0, w1};
                    mv_rows<Real, VPT, kReread, 2>(row, w, opmem, pc, acc, dacc, m, slots, phase, ea,
                                                   eb);
                } else if (j < nrows) {
                    none(eb, nullptr);
                    one(p0, w0, ea);
                } else {
                    none(ea, eb);
                }
            }
            base += two ? 2 * rg.R : rg.R;
            run += 2;
            continue;
        }
        int rr = m.team;
        mbar_wait_or_flag(&full[a], (uint32_t)rg.par, timed_out);
        rg.next();
        if (rr >= rows) none(ea, nullptr);
        do {
            int end = rows;   // rows of this stage and run
            if (more) {
                if (rr < rows) next_run();
                end = min(rows, rr + (kMvRun - run) * nt);
            }
            if constexpr (kPair) {
                for (; rr + nt < end; rr += 2 * nt) {
                    const Real w[2] = {n0, n1};
                    const Real *const row[2] = {buf + (size_t)rr * ld, buf + (size_t)(rr + nt) * ld};
                    n0 = weight(base + rr + 2 * nt);
                    n1 = weight(base + rr + 3 * nt);
                    mv_rows<Real, VPT, kReread, 2>(row, w, opmem, pc, acc, dacc, m, slots, phase,
                                                   rr + 2 * nt < rows ? nullptr : ea, nullptr);
                    if (kRunsIn) run += 2;
                }
            }
            for (; rr < end; rr += nt) {
                const Real w = n0;
                n0 = n1;
                n1 = weight(base + rr + 2 * nt);
                one(buf + (size_t)rr * ld, w, rr + nt < rows ? nullptr : ea);
                if (kRunsIn) ++run;
            }
        } while (more && rr < rows);
        base += rg.R;
    }
    return flushed;
}

// The chunk's results: the teams' accumulators added in team order (through red,
// [nteams][ld], free for the consumers' use) into partial g, and the teams' shares of
// r^T A r into dpart.  flushed: the team's earlier runs are in red.  Called by every consumer
// thread.
template <typename Real, int VPT>
__device__ __forceinline__ void mv_finish(const Params &p, int s, int g, const MvTeam &m,
                                          Chunk<Real> (&acc)[VPT], bool flushed, const DeltaAcc<Real> &dacc, Real *red,
                                          double *dsl)
{
    constexpr int E = Chunk<Real>::E;
    const WS<Real> ws(p);
    Real *dst = ws.part(s, g, 0);
    double *dp = p.dpart + ((size_t)s * p.G + g) * kDpart;
    if (flushed) mv_add_runs<Real, VPT>(red + (size_t)m.team * m.nch * E, m, acc);
    if (m.nteams == 1) {
#pragma unroll
        for (int v = 0; v < VPT; ++v) {
            const int c = m.tl + m.tthreads * v;
            if (c < m.nch) st_chunk(dst + c * E, acc[v]);
        }
        if (m.tl == 0) *dp = dacc.back(dacc.value());
        return;
    }
    const int nthreads = m.tthreads * m.nteams;
    const int ct = (int)threadIdx.x - 32;
    const size_t ld = (size_t)m.nch * E;
#pragma unroll
    for (int v = 0; v < VPT; ++v) {
        const int c = m.tl + m.tthreads * v;
        if (c < m.nch) st_chunk(red + (size_t)m.team * ld + c * E, acc[v]);
    }
    if (m.tl == 0) dsl[m.team] = dacc.value();
    bar_named(15, nthreads);
    // the last warp (it has no more chunks of the sum to add than any other) adds the shares
    if (ct >= nthreads - 32) {
        double d = m.lane < m.nteams ? dsl[m.lane] : 0.0;
#pragma unroll
        for (int o = 8; o; o >>= 1) d += __shfl_xor_sync(0xffffffffu, d, o);
        if (m.lane == 0) *dp = dacc.back(d);
    }
    for (int c = ct; c < m.nch; c += nthreads) {
        Chunk<Real> sum = ld_chunk(red + c * E);
        for (int t2 = 1; t2 < m.nteams; ++t2) {
            const Chunk<Real> o = ld_chunk(red + (size_t)t2 * ld + c * E);
#pragma unroll
            for (int e = 0; e < E; ++e) sum.v[e] += o.v[e];
        }
        st_chunk(dst + c * E, sum);
    }
}

// The product as its own launch (grid (G, Q)).  Warp 0 is the producer: one lane streams
// the chunk's rows, mv_rows consecutive rows (one contiguous block) per stage, into a ring
// of mv_stages shared-memory stages with cp.async.bulk, completion counted on the stage's
// "full" mbarrier.  Each consumer warp arrives on the stage's "empty" mbarrier when done,
// which lets the producer refill it.
// MODE (MvMode): how a team walks its rows; set with the geometry.
template <typename Real, int VPT, int MODE>
__global__ void __launch_bounds__(MODE == kMvWide ? 544 : (VPT >= 8 ? 352 : 512),
                                  VPT == 1 && sizeof(Real) == 4 ? 2 : 1)
    k_matvec(Params p)
{
    constexpr int E = Chunk<Real>::E;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    __shared__ double dsl[16];
    const int g = blockIdx.x, s = blockIdx.y;
    if (p.st[s].done) return;
    const WS<Real> ws(p);
    const int nch = p.ld / E;
    const int S = p.mv_stages, R = p.mv_rows;
    const int tw = p.team_warps;
    const int nteams = (blockDim.x / 32 - 1) / tw;
    const size_t row_elems = (size_t)p.ld;
    const uint32_t row_bytes = (uint32_t)(row_elems * sizeof(Real));
    Real *ring = reinterpret_cast<Real *>(smem_raw);                     // [S][R][ld]
    uint64_t *full = reinterpret_cast<uint64_t *>(ring + (size_t)S * R * row_elems);
    uint64_t *empty = full + S;
    Real *slots = reinterpret_cast<Real *>(empty + S);                   // [nteams][2][32]
    Real *runs = slots + (size_t)nteams * 64;                            // [nteams][ld]
    long long r0, r1;
    row_range(p.M, p.G, g, r0, r1);
    const long long nst = (r1 - r0 + R - 1) / R;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int st = 0; st < S; ++st) {
            mbar_init(&full[st], 1);
            mbar_init(&empty[st], nteams * tw);
        }
        fence_mbar_init();
    }
    __syncthreads();
    bool timed_out = false;

    if (warp == 0) {
        if (lane == 0) {
            for (long long i = 0; i < nst; ++i) {
                const int st = (int)(i % S);
                const uint32_t par = (uint32_t)((i / S) & 1);
                if (i >= S) mbar_wait_or_flag(&empty[st], par ^ 1u, timed_out);
                const long long row0 = r0 + i * R;
                const uint32_t rows = (uint32_t)min((long long)R, r1 - row0);
                mbar_arrive_expect_tx(&full[st], rows * row_bytes);
                bulk_g2s(ring + (size_t)st * R * row_elems, ws.row(s, row0), rows * row_bytes,
                         &full[st]);
            }
            // drain: the last copy into every stage has landed before the CTA can exit
            for (long long i = max(0ll, nst - S); i < nst; ++i)
                mbar_wait_or_flag(&full[i % S], (uint32_t)((i / S) & 1), timed_out);
        }
    } else {
        const MvTeam m(tw, nteams, nch);
        const Real *pv = ws.vR(s, 0);
        Chunk<Real> acc[VPT], pc[VPT];
#pragma unroll
        for (int v = 0; v < VPT; ++v) {
            const int c = m.tl + m.tthreads * v;
            zero(acc[v]);
            if (VPT <= 8 && c < nch) pc[v] = ldg_chunk(pv + c * E);
            else zero(pc[v]);
        }
        int phase = 0;
        DeltaAcc<Real> dacc;
        dacc.init(p.st[s].rr);
        MvRing rg{0, 0, S, R};
        const bool flushed =
            mv_chunk<Real, VPT, (MODE != kMvHold), (VPT <= 8 && (VPT <= 4 || MODE != kMvHold))>(
                r0, r1, runs, ws.w(s) + r0, pv, pc, acc, dacc, m, ring, full, empty, rg,
                true, slots, phase, timed_out);
        if (nteams > 1) bar_named(15, m.tthreads * nteams);   // past the last ring read
        // the same for every team, and as the host counts (mv_runs_bytes)
        const bool own = sizeof(Real) == 4 && (nteams == 1 || VPT == 1) &&
                         r1 - r0 > (long long)kMvRun * nteams;
        mv_finish<Real, VPT>(p, s, g, m, acc, flushed, dacc, own ? runs : ring, dsl);
    }
    if (timed_out) atomicCAS(&p.st[s].status, 0, (int)FBSDE_ERR_TIMEOUT);
}

}  // namespace dev
}  // namespace fbsde
