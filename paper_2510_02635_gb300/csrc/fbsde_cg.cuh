// fbsde_cg.cuh -- the conjugate-gradient solve of one regression (all queries of a call).
// Included after fbsde_matvec.cuh.
//
// The iteration is that of Chronopoulos and Gear (1989), conjugate gradients with one
// reduction per pass.  With A = Gamma_c + lambda I, gamma = r . r and
//   delta = r . A r = (1/W) sum_j w_j (D_j . r)^2 - (S . r)^2 + lambda gamma,
// whose sum over the particles comes with the product's own dot products,
//   t = 0: beta = 0, a = gamma / delta;
//   t > 0: beta = gamma / gamma_prev, a = gamma / (delta - beta gamma / a_prev),
//   p = r + beta p,  s = A r + beta s (= A p),  x += a p,  r -= a s.
// A pass is two phases with one exchange between the CTAs after each:
//   A  chunks of a query's rows: partial product and share of delta (fbsde_matvec.cuh);
//   B  tiles of a query's coordinates: the partial vectors added in a fixed order
//      (compensated), a and beta, the four vector updates, shares of gamma and S . r.
// Two forms run the same device functions on the same chunks and tiles, so they give the
// same bits:
//   k_cg_loop             every pass in one cooperative launch, a grid barrier per phase;
//   k_matvec, k_cg_tile   one launch per phase (product timing, plans with several
//                         branches, rows too wide for the loop's block).
#pragma once
#include "fbsde_matvec.cuh"

namespace fbsde {
namespace dev {

// Threads of k_cg_tile (at most) and k_level_moments: a warp for the scalars beside those that read the
// partials; FP32 blocks of 56 registers, three an SM (two of 512 threads and 64 registers before:
// 65 queries, d = 700: 18.9 -> 14.1 us a launch).
constexpr int kCgThreads = 384;
constexpr int kCgWarps = 10;      // warps 1..10 read a tile's partials (warp 0 waits at the
                                  // grid barrier, and its first loads after that are slow)
constexpr int kCgQueries = 64;    // most queries of k_cg_loop (every CTA keeps their scalars)

// Scalars of one query's pass.
struct CgScal {
    double gam, sp, gprev, aprev;   // r . r, S . r; r . r and step of the pass before
    double beta, bg;                // beta, beta gamma / a_prev (0 in the first pass)
    double a, invW, lambda, rhs2;
    int t, done, ok;
};

__device__ __forceinline__ double warp_add(double v)
{
#pragma unroll
    for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Shares of S . r and r . r of a query's tiles, one 32-byte sector each: tiles of different
// CTAs never write the same sector (slot 5 of the FP64 vectors, four doubles per tile of at
// least four coordinates: the product itself never leaves phase B).
template <typename Real> __device__ __forceinline__ double *cg_shares(const WS<Real> &ws, int s)
{
    return ws.v64(s, 5);
}

// beta and beta gamma / a_prev of the pass that starts with these scalars.
__device__ __forceinline__ void cg_prepare(CgScal &c)
{
    c.beta = 0.0;
    c.bg = 0.0;
    if (c.t > 0) {
        c.beta = c.gam / c.gprev;
        c.bg = c.beta * c.gam / c.aprev;
    }
}

// One warp: delta from the chunks' shares, then the pass's step a.  Lanes return the same
// values.
template <typename Real>
__device__ __forceinline__ void cg_step_scalar(const Params &p, int s, const CgScal &c, double &a,
                                               int &ok)
{
    const double *dp = p.dpart + (size_t)s * p.G * kDpart;
    const int lane = threadIdx.x & 31;
    double d = 0.0;
    for (int g0 = lane; g0 < p.G; g0 += 32 * 8) {
        double v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) v[u] = g0 + 32 * u < p.G ? __ldcg(dp + (size_t)kDpart * (g0 + 32 * u)) : 0.0;
        d += ((v[0] + v[1]) + (v[2] + v[3])) + ((v[4] + v[5]) + (v[6] + v[7]));
    }
    d = warp_add(d);
    const double den = fma(d, c.invW, fma(-c.sp, c.sp, c.lambda * c.gam)) - c.bg;
    a = c.gam / den;
    ok = (den > 0.0 && isfinite(a)) ? 1 : 0;
}

// gamma and S . r after the pass from the tiles' shares: one thread adds up to kCgSerial tiles
// (many queries, few tiles each: a thread per query), a whole warp more than that.  Every
// caller of a shape uses the same form, so the sums have the same bits.
constexpr int kCgSerial = 16;
template <typename Real>
__device__ __forceinline__ void cg_add_shares(const Params &p, const WS<Real> &ws, int s, double &sr,
                                              double &rr)
{
    const double2 *sh = reinterpret_cast<const double2 *>(cg_shares(ws, s));
    sr = 0.0;
    rr = 0.0;
    if (p.nblk <= kCgSerial) {
        for (int b0 = 0; b0 < p.nblk; b0 += 4) {
            double2 v[4];
#pragma unroll
            for (int u = 0; u < 4; ++u)
                v[u] = b0 + u < p.nblk ? __ldcg(sh + 2 * (b0 + u)) : make_double2(0.0, 0.0);
            sr += (v[0].x + v[1].x) + (v[2].x + v[3].x);
            rr += (v[0].y + v[1].y) + (v[2].y + v[3].y);
        }
        return;
    }
    const int lane = threadIdx.x & 31;
    for (int b0 = lane; b0 < p.nblk; b0 += 32 * 4) {
        double2 v[4];
#pragma unroll
        for (int u = 0; u < 4; ++u)
            v[u] = b0 + 32 * u < p.nblk ? __ldcg(sh + 2 * (b0 + 32 * u)) : make_double2(0.0, 0.0);
        sr += (v[0].x + v[1].x) + (v[2].x + v[3].x);
        rr += (v[0].y + v[1].y) + (v[2].y + v[3].y);
    }
#pragma unroll
    for (int o = 16; o; o >>= 1) {
        sr += __shfl_xor_sync(0xffffffffu, sr, o);
        rr += __shfl_xor_sync(0xffffffffu, rr, o);
    }
}

// The scalars after a pass: convergence, exhaustion, and breakdown (a share of r . r below 0
// marks it: the step was not positive and finite, and the iterate of the pass before stays).
// Returns a status to record (0: none).
__device__ __forceinline__ int cg_commit(const Params &p, CgScal &c, double sr, double rr,
                                         int &exhausted)
{
    exhausted = 0;
    if (rr < 0.0) {
        c.done = 1;
        return c.gam <= p.cg_tol2 * c.rhs2 ? 0 : (int)FBSDE_ERR_CG;
    }
    c.gprev = c.gam;
    c.aprev = c.a;
    c.gam = rr;
    c.sp = sr;
    c.t += 1;
    if (rr <= p.cg_tol2 * c.rhs2) {
        c.done = 1;
    } else if (c.t >= p.cg_max_iter) {
        c.done = 1;
        exhausted = 1;
        return (int)FBSDE_ERR_CG;
    }
    return 0;
}

__device__ __forceinline__ CgScal cg_load(const SolveState &st)
{
    CgScal c;
    c.gam = __ldcg(&st.rr);
    c.sp = __ldcg(&st.sp);
    c.gprev = __ldcg(&st.rr_prev);
    c.aprev = __ldcg(&st.cg_alpha);
    c.invW = __ldcg(&st.invW);
    c.lambda = __ldcg(&st.lambda);
    c.rhs2 = __ldcg(&st.rhs2);
    c.t = __ldcg(&st.iters);
    c.done = __ldcg(&st.done);
    c.a = 1.0;   // of a query whose step this CTA does not need
    c.ok = 1;
    return c;
}

__device__ __forceinline__ void cg_store(SolveState &st, const CgScal &c, int status, int exhausted,
                                         int passes)
{
    st.rr_prev = c.gprev;
    st.cg_alpha = c.aprev;
    st.rr = c.gam;
    st.sp = c.sp;
    st.iters = c.t;
    st.cg_total += passes;
    if (exhausted) st.cg_exhausted += 1;
    if (status) atomicCAS(&st.status, 0, status);   // the first status met stays
    __threadfence();
    *reinterpret_cast<volatile int *>(&st.done) = c.done;
}

// Compensated sum of two (sum, error) pairs of the FP32 reduction; FP64 plain.
template <typename Real> struct CgPart;
template <> struct CgPart<float> {
    using Acc = RedAcc<float>;
    static __device__ __forceinline__ void join(Acc &a, float hi, float lo) { a.merge(hi, lo); }
    // a + the lane o away's v
    static __device__ __forceinline__ void across(Acc &a, const Acc &v, int o)
    {
        const float hi = __shfl_xor_sync(0xffffffffu, v.s, o);
        const float lo = __shfl_xor_sync(0xffffffffu, v.c, o);
        a.merge(hi, lo);
    }
};
template <> struct CgPart<double> {
    using Acc = RedAcc<double>;
    static __device__ __forceinline__ void join(Acc &a, double hi, double lo) { a.merge(hi, lo); }
    static __device__ __forceinline__ void across(Acc &a, const Acc &v, int o)
    {
        a.s += __shfl_xor_sync(0xffffffffu, v.s, o);
    }
};

// Shared memory of one phase-B tile: the warps' sums of its coordinates (hi, lo) and the
// shares of the warps that own coordinates.
template <typename Real> struct CgTileSm {
    Real hi[kCgWarps][kRedTile];
    Real lo[kCgWarps][kRedTile];
    double sh[4][2];
};

// Warps that read the partial vectors of a tile.
__device__ __forceinline__ int cg_part_warps(const Params &p)
{
    const int per = 32 / p.cg_lpr;
    return min(kCgWarps, (p.G + per - 1) / per);
}

// The sums of partial vector `vec` of a tile over the groups of each of the warps 1 ..
// kCgWarps, into sm.hi and sm.lo (cg_join adds the warps after a barrier).  A lane reads four
// coordinates of every (kCgWarps 32 / lpr)-th partial.
template <typename Real>
__device__ __forceinline__ void cg_partials(const Params &p, int s, int tile, int vec,
                                            CgTileSm<Real> &sm)
{
    using Part = CgPart<Real>;
    using Acc = typename Part::Acc;
    constexpr int kB = 4;   // loads in flight per lane
    const WS<Real> ws(p);
    const int lpr = p.cg_lpr, width = 4 * lpr;
    const int lane = threadIdx.x & 31, warp = (int)(threadIdx.x >> 5) - 1;
    const int per = 32 / lpr, groups = kCgWarps * per;
    const int warps = cg_part_warps(p);
    if (warp >= 0 && warp < warps) {
        // the partial vectors g = group, group + groups, .. of this lane's four coordinates
        const int grp = warp * per + lane / lpr;
        const int e0 = tile * width + 4 * (lane & (lpr - 1));
        Acc acc[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) acc[e].init();
        if (e0 < p.ld) {   // ld is a multiple of 4
            const Real *src = ws.part(s, grp, vec) + e0;
            const size_t stride = (size_t)p.part_vecs * p.ld * groups;
            for (int g0 = grp; g0 < p.G; g0 += kB * groups, src += kB * stride) {
                Quad<Real> q[kB];
#pragma unroll
                for (int u = 0; u < kB; ++u)
                    if (g0 + u * groups < p.G) q[u] = ldcg_quad(src + u * stride);
#pragma unroll
                for (int u = 0; u < kB; ++u)
                    if (g0 + u * groups < p.G) {
#pragma unroll
                        for (int e = 0; e < 4; ++e) acc[e].add(q[u].v[e]);
                    }
            }
        }
        // sums over the warp's groups, scattered: the first two exchanges halve the
        // coordinates a lane carries (4 -> 2 -> 1), the others add the one left
        int e = 0, o = 16;
        if (o >= lpr) {
            const bool up = lane & o;
            Acc k0 = up ? acc[2] : acc[0], k1 = up ? acc[3] : acc[1];
            Part::across(k0, up ? acc[0] : acc[2], o);
            Part::across(k1, up ? acc[1] : acc[3], o);
            acc[0] = k0;
            acc[1] = k1;
            e = up ? 2 : 0;
            o = 8;
            if (o >= lpr) {
                const bool up2 = lane & o;
                Acc k = up2 ? acc[1] : acc[0];
                Part::across(k, up2 ? acc[0] : acc[1], o);
                acc[0] = k;
                e += up2 ? 1 : 0;
                for (o = 4; o >= lpr; o >>= 1) Part::across(acc[0], acc[0], o);
                if (!(lane & (7 & ~(lpr - 1)))) {   // one of the lanes with the same sum
                    sm.hi[warp][4 * (lane & (lpr - 1)) + e] = acc[0].hi();
                    sm.lo[warp][4 * (lane & (lpr - 1)) + e] = (Real)acc[0].lo();
                }
            } else {   // lpr = 16: two coordinates a lane
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    sm.hi[warp][4 * (lane & 15) + e + u] = acc[u].hi();
                    sm.lo[warp][4 * (lane & 15) + e + u] = (Real)acc[u].lo();
                }
            }
        } else {
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                sm.hi[warp][4 * lane + u] = acc[u].hi();
                sm.lo[warp][4 * lane + u] = (Real)acc[u].lo();
            }
        }
    }
}

// Coordinate t's sum over the warps: four interleaved runs (independent additions in flight).
template <typename Real>
__device__ __forceinline__ double cg_join(const Params &p, const CgTileSm<Real> &sm, int t)
{
    using Part = CgPart<Real>;
    using Acc = typename Part::Acc;
    const int warps = cg_part_warps(p);
    Acc a[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) a[u].init();
    for (int w = 0; w < warps; w += 4)
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (w + u < warps) Part::join(a[u], sm.hi[w + u][t], sm.lo[w + u][t]);
    Part::join(a[0], a[1].hi(), a[1].lo());
    Part::join(a[2], a[3].hi(), a[3].lo());
    Part::join(a[0], a[2].hi(), a[2].lo());
    return a[0].value();
}

// Phase B of one tile of 4 lpr coordinates (lpr = 1, 2, .. 32 lanes a row of partials, so
// 32 / lpr partials are read by a warp at a time): all NT threads of the block.  c's scalars
// and the step (c.a, c.ok) are read after the first barrier.  Thread 32 + t, t < 4 lpr, owns
// coordinate t of the tile: its vector loads are issued first.  The partials are read by
// warps 1 .. kCgWarps at most, so the order of the sums does not depend on NT.
template <typename Real, int NT>
__device__ __forceinline__ void cg_tile(const Params &p, int s, int tile, const CgScal &c,
                                        CgTileSm<Real> &sm)
{
    static_assert(NT >= 32 * (kCgWarps + 1), "warps of the partial sums");
    const WS<Real> ws(p);
    const int lpr = p.cg_lpr, width = 4 * lpr;
    const int t = (int)threadIdx.x - 32, lane = threadIdx.x & 31, warp = t >> 5;   // warp 0: -1
    const int i = tile * width + t;
    const bool own = t >= 0 && t < width && i < p.ld;
    const bool first = c.t == 0;
    double rv = 0.0, pv = 0.0, sv = 0.0, xv = 0.0, Sv = 0.0;
    if (own) {
        rv = ws.v64(s, 1)[i];
        xv = ws.v64(s, 0)[i];
        Sv = ws.v64(s, 3)[i];
        if (!first) {
            pv = ws.v64(s, 2)[i];
            sv = ws.v64(s, 7)[i];
        }
    }
    cg_partials<Real>(p, s, tile, 0, sm);
    __syncthreads();
    if (t < 0 || t >= max(width, 32)) return;   // whole warps
    double sr = 0.0, rr = 0.0;
    if (!c.ok) {
        rr = -1.0;
    } else if (own) {
        const double wi = fma(cg_join<Real>(p, sm, t), c.invW, fma(-Sv, c.sp, c.lambda * rv));
        const double pi = first ? rv : fma(c.beta, pv, rv);
        const double si = first ? wi : fma(c.beta, sv, wi);
        const double rn = fma(-c.a, si, rv);   // the one operation behind the step
        ws.vR(s, 0)[i] = (Real)rn;
        ws.v64(s, 1)[i] = rn;
        ws.v64(s, 2)[i] = pi;
        ws.v64(s, 7)[i] = si;
        ws.v64(s, 0)[i] = fma(c.a, pi, xv);
        sr = Sv * rn;
        rr = rn * rn;
    }
    for (int o = min(width, 32) / 2; o; o >>= 1) {
        sr += __shfl_xor_sync(0xffffffffu, sr, o);
        rr += __shfl_xor_sync(0xffffffffu, rr, o);
    }
    double2 *out = reinterpret_cast<double2 *>(cg_shares(ws, s)) + 2 * tile;
    if (width <= 32) {
        if (t == 0) *out = make_double2(sr, rr);
        return;
    }
    if (lane == 0) {
        sm.sh[warp][0] = sr;
        sm.sh[warp][1] = rr;
    }
    bar_named(14, width);
    if (t == 0) {
        sr = sm.sh[0][0];
        rr = sm.sh[0][1];
        for (int w = 1; w < width / 32; ++w) {
            sr += sm.sh[w][0];
            rr += sm.sh[w][1];
        }
        *out = make_double2(sr, rr);
    }
}

// The last tile of query s to finish (arrival counter) adds the shares and commits the
// pass: true in thread 0 of that block.  Called by every thread of the block after cg_tile;
// the owners' stores precede thread 0's through the barrier.
template <typename Real>
__device__ __forceinline__ bool cg_arrive(const Params &p, int s, const CgScal &c, int *flag)
{
    SolveState &st = p.st[s];
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        *flag = atomicAdd(&st.arrive_q, 1) == p.nblk - 1;
    }
    __syncthreads();
    if (!*flag || threadIdx.x >= 32) return false;
    __threadfence();
    const WS<Real> ws(p);
    double sr, rr;
    cg_add_shares(p, ws, s, sr, rr);
    if (threadIdx.x != 0) return false;
    CgScal n = c;
    int ex;
    const int before = n.t;
    const int status = cg_commit(p, n, sr, rr, ex);
    st.arrive_q = 0;
    cg_store(st, n, status, ex, n.t - before);
    return true;
}

// Phase B as its own launch, grid (nblk, Q).  In a CUDA graph (use_h = 1) the last query to
// finish sets the while-loop condition: 1 while some query has not converged and fewer than
// cg_max_iter passes ran (with one query, its last tile does so without a second arrival).
template <typename Real>
__global__ void __launch_bounds__(kCgThreads, sizeof(Real) == 4 ? 3 : 2) k_cg_tile(Params p, cudaGraphConditionalHandle h,
                                                        int use_h)
{
    __shared__ CgTileSm<Real> sm;
    __shared__ CgScal sc;
    __shared__ int flag;
    const int s = blockIdx.y;
    SolveState &st = p.st[s];
    bool answer = false;
    if (st.done) {
        answer = blockIdx.x == 0 && threadIdx.x == 0;   // one block answers for a finished query
    } else {
        if (threadIdx.x >= blockDim.x - 32) {   // a warp that reads no partials
            CgScal c = cg_load(st);
            cg_prepare(c);
            cg_step_scalar<Real>(p, s, c, c.a, c.ok);
            if (threadIdx.x == blockDim.x - 32) sc = c;
        }
        __syncthreads();
        cg_tile<Real, kCgThreads>(p, s, blockIdx.x, sc, sm);
        answer = cg_arrive<Real>(p, s, sc, &flag);
    }
    if (use_h && answer) {
        bool last_q = true;
        if (p.Q > 1) {
            __threadfence();
            last_q = atomicAdd(&p.st[0].arrive, 1) == p.Q - 1;
        }
        if (last_q) {
            if (p.Q > 1) __threadfence();
            p.st[0].arrive = 0;
            const int count = ++p.st[0].loop_iter;
            bool active = false;
            for (int q2 = 0; q2 < p.Q && !active; ++q2)
                active = *reinterpret_cast<volatile int *>(&p.st[q2].done) == 0;
            if (count >= p.cg_max_iter) active = false;
            cudaGraphSetConditional(h, active ? 1u : 0u);
        }
    }
}

// Barrier of all CTAs of a cooperative launch.  The word's low 31 bits count the arrivals
// and return to 0 with the last one, which flips the top bit (the first CTA adds
// 2^31 - (n - 1), the others 1).  Bounded wait: false if the other CTAs did not arrive
// within limit_ns; the word may then keep a partial count, so the kernel before every loop
// sets it to 0 (k_level_rhs, k_adj_setup, k_moments_finalize).
__device__ __forceinline__ bool grid_barrier(unsigned int *word, int *flag,
                                             unsigned long long limit_ns = kWaitNs)
{
    __syncthreads();
    if (threadIdx.x == 0) {
        const unsigned int add = blockIdx.x == 0 ? 0x80000000u - (gridDim.x - 1u) : 1u;
        unsigned int old, cur;
        asm volatile("atom.add.acq_rel.gpu.global.u32 %0, [%1], %2;"
                     : "=r"(old) : "l"(word), "r"(add) : "memory");
        int ok = 1;
        unsigned long long t0 = 0;
        for (unsigned int n = 1;; ++n) {
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(cur) : "l"(word) : "memory");
            if ((cur ^ old) & 0x80000000u) break;
            if ((n & 255u) == 0) {
                const unsigned long long now = globaltimer_ns();
                if (!t0) t0 = now;
                else if (now - t0 > limit_ns) {
                    ok = 0;
                    break;
                }
            }
        }
        *flag = ok;
    }
    __syncthreads();
    return *flag != 0;
}

// Position of the loop's producer: its chunk pw, that chunk's next row and the rows left of
// it, ring slot and the parity of its use, whether every slot has been used, stages requested
// beyond the finished passes' (lead) and in the CTA's whole list.
struct CgProducer {
    const void *src;
    int pw, left, slot, par, full, lead, list;
};

// Every pass of the CG in one cooperative launch (one CTA per SM).  CTA b works on the
// chunks b, b + gridDim.x, .. of the Q G chunks (phase A) and the tiles b, b + gridDim.x, ..
// of the Q nblk tiles (phase B).  Warp 0 streams the rows as in k_matvec, but through a ring
// that lives as long as the loop:
//   - cg_res = 1: every CTA has one chunk at most and the ring holds it; it is copied once
//     and every pass reads it from shared memory;
//   - one query otherwise: the next pass's first stages are requested as this pass frees
//     the ring, so the copies run on through both barriers.
// What bounds a pass of a small cloud is its chain of latencies: two barriers of about 1.2 us,
// the reads of r, of the partials and of the shares (0.5 to 1 us each through L2), and two
// chains of dependent FP64 operations (64 cycles each).  Measured with one query: d = 1000,
// M = 4096, 8.6 us a pass in place of 20.5 us in three launches; d = 2503, M = 8192, 21 us
// (82 MB of rows, phase A 12 us) in place of 43 us; FP64, d = 1203, M = 2048, 23 us in place
// of 63 us (the product had 64 CTAs).  Warp 0 polls the barrier; the first loads a warp makes
// after its polls take 4 us longer (measured on 80 of the 152 SMs), so it takes no part in
// phase B and the scalars fall to the last warp.
// Every CTA keeps the scalars of all queries (the shares are added in the same order
// everywhere), and the step of those whose tiles it owns.  After a wait that gave up in an
// earlier launch of the solve the loop ends at once.
template <typename Real, int VPT, int NT, bool HOLD>
__global__ void __launch_bounds__(NT, 1) k_cg_loop(Params p)
{
    constexpr int E = Chunk<Real>::E;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    __shared__ double dsl[16];
    __shared__ int flag;
    __shared__ CgProducer pr;
    const int before = __ldcg(&p.st[0].status);   // of the solve so far; checked below
    const WS<Real> ws(p);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int nch = p.ld / E, S = p.cg_stages, R = p.cg_rows;
    const int tw = p.team_warps, nteams = p.cg_teams, nct = 32 * tw * nteams;
    const size_t row_elems = (size_t)p.ld;
    const uint32_t row_bytes = (uint32_t)(row_elems * sizeof(Real));
    Real *ring = reinterpret_cast<Real *>(smem_raw);                       // cg_ring rows
    Real *op = ring + (size_t)p.cg_ring * row_elems;                       // [ld] operand r
    // the teams' sums (phase A) and the warps' sums (phase B) share the next region
    unsigned char *both = reinterpret_cast<unsigned char *>(op + (p.cg_op ? row_elems : 0));
    Real *red = reinterpret_cast<Real *>(both);
    CgTileSm<Real> &tsm = *reinterpret_cast<CgTileSm<Real> *>(both);
    CgScal *sc = reinterpret_cast<CgScal *>(both + p.cg_both);             // [Q]
    uint64_t *full = reinterpret_cast<uint64_t *>(sc + p.Q);
    uint64_t *empty = full + S;
    Real *slots = reinterpret_cast<Real *>(empty + S);                     // [nteams][2][32]
    Real *wsm = slots + (size_t)nteams * 64;                               // [cg_ring], cg_res only
    const bool resident = p.cg_res != 0;
    const bool spec = resident && p.Q == 1;   // phase A runs ahead of the convergence test
    const int nwork = p.Q * p.G, ntile = p.Q * p.nblk;
    const bool consumer = warp >= 1 && (int)threadIdx.x - 32 < nct;
    if (threadIdx.x == 0) {
        for (int st = 0; st < S; ++st) {
            mbar_init(&full[st], 1);
            mbar_init(&empty[st], nteams * tw);
        }
        fence_mbar_init();
    }
    if (threadIdx.x < (unsigned)p.Q) {
        CgScal c = cg_load(p.st[threadIdx.x]);
        cg_prepare(c);
        sc[threadIdx.x] = c;
    }
    if (resident && (int)blockIdx.x < nwork) {
        const int s = blockIdx.x / p.G;
        long long r0, r1;
        row_range(p.M, p.G, (int)blockIdx.x - s * p.G, r0, r1);
        for (int j = threadIdx.x; j < (int)(r1 - r0); j += NT) wsm[j] = ws.w(s)[r0 + j];
    }
    __syncthreads();
    if (before == FBSDE_ERR_TIMEOUT) return;
    bool timed_out = false;
    // producer (thread 0): its state lives in shared memory, out of the consumers' registers
    if (threadIdx.x == 0) {
        pr.pw = (int)blockIdx.x - (int)gridDim.x;
        pr.left = pr.slot = pr.par = pr.full = pr.lead = pr.list = 0;
        for (int w = blockIdx.x; w < nwork; w += gridDim.x) {   // stages of the whole list
            long long r0, r1;
            row_range(p.M, p.G, w % p.G, r0, r1);
            pr.list += (int)((r1 - r0 + R - 1) / R);
        }
    }
    // Requests up to `most` stages: to the end of the list, where the position returns to its
    // start, or (wrap) on from its start.
    auto request = [&](int most, bool wrap) {
        CgProducer c = pr;
        while (most > 0) {
            if (c.left == 0) {   // the next chunk of a query that iterates
                int w = c.pw + gridDim.x;
                while (w < nwork && sc[w / p.G].done) w += gridDim.x;
                if (w >= nwork) {
                    c.pw = (int)blockIdx.x - (int)gridDim.x;
                    if (!wrap) break;
                    continue;
                }
                const int s = w / p.G;
                long long r0, r1;
                row_range(p.M, p.G, w - s * p.G, r0, r1);
                c.pw = w;
                c.left = (int)(r1 - r0);
                c.src = ws.row(s, r0);
            }
            const int rows = min(R, c.left);
            const uint32_t bytes = (uint32_t)rows * row_bytes;
            if (c.full) mbar_wait_or_flag(&empty[c.slot], (uint32_t)c.par ^ 1u, timed_out);
            mbar_arrive_expect_tx(&full[c.slot], bytes);
            bulk_g2s(ring + (size_t)c.slot * R * row_elems, c.src, bytes, &full[c.slot]);
            c.src = static_cast<const char *>(c.src) + bytes;
            c.left -= rows;
            ++c.lead;
            --most;
            if (++c.slot == S) {
                c.slot = 0;
                c.par ^= 1;
                c.full = 1;   // every slot has been used once
            }
        }
        pr = c;
    };
    // scalars after a pass: threads or warps first, first + step, .. take a query each
    auto commit_query = [&](int q, bool writer) {
        if (sc[q].done) return;
        CgScal c = sc[q];
        double sr, rr;
        cg_add_shares(p, ws, q, sr, rr);
        const int t0 = c.t;
        int ex;
        const int status = cg_commit(p, c, sr, rr, ex);
        if (!c.done) cg_prepare(c);
        if (p.nblk > kCgSerial) __syncwarp();
        if (writer) {
            sc[q] = c;
            if (blockIdx.x == 0) cg_store(p.st[q], c, status, ex, c.t - t0);
        }
    };
    auto commit = [&](int first_warp, int warps) {
        if (p.nblk <= kCgSerial) {
            for (int q = 32 * first_warp + lane; q < p.Q; q += 32 * warps) commit_query(q, true);
            __syncwarp();
        } else {
            for (int q = first_warp; q < p.Q; q += warps) commit_query(q, lane == 0);
        }
    };
    const MvTeam m(tw, nteams, nch);
    int phase = 0;
    MvRing rg{0, 0, S, R};   // consumers' position
    double rr_spec = sc[0].gam;   // of the pass before where phase A runs ahead
    for (int pass = 0;; ++pass) {
        // ---------------- is any query still iterating?
        if (pass == 0 || !spec) {
            if (pass > 0) {
                if (warp > 0) commit(warp - 1, NT / 32 - 1);
                __syncthreads();
            }
            int any = 0;
            for (int q = lane; q < p.Q; q += 32) any |= !sc[q].done;
            if (!__any_sync(0xffffffffu, any)) break;
        }
        // ---------------- phase A
        if (spec && pass > 0 && warp == NT / 32 - 1)
            commit(0, 1);   // while the consumers work on the next product
        if (warp == 0) {
            if (lane == 0) {
                if (resident) {
                    if (pass == 0) request(S, false);
                } else if (p.Q == 1) {   // to S stages into the next pass
                    if (pr.list) {
                        request(pr.list + S - pr.lead, true);
                        pr.lead -= pr.list;
                    }
                } else {
                    request(0x7fffffff, false);
                }
            }
            __syncwarp();   // the other lanes wait for the producer here, not at the barrier
        } else if (consumer) {
            for (int w = blockIdx.x; w < nwork; w += gridDim.x) {
                const int s = w / p.G, g = w - s * p.G;
                if (!spec && sc[s].done) continue;
                long long r0, r1;
                row_range(p.M, p.G, g, r0, r1);
                const Real *pv = ws.vR(s, 0);
                Chunk<Real> acc[VPT], pc[VPT];
                if (p.cg_op) {   // several teams: the operand through shared memory
                    for (int c = threadIdx.x - 32; c < nch; c += nct)
                        st_chunk(op + c * E, ldcg_chunk(pv + c * E));
                    bar_named(15, nct);
                }
#pragma unroll
                for (int v = 0; v < VPT; ++v) {
                    const int c = m.tl + m.tthreads * v;
                    zero(acc[v]);
                    if (c < nch) pc[v] = p.cg_op ? ld_chunk(op + c * E) : ldcg_chunk(pv + c * E);
                    else zero(pc[v]);
                }
                DeltaAcc<Real> dacc;
                dacc.init(spec ? rr_spec : sc[s].gam);
                if (resident) rg.slot = rg.par = 0;   // every pass reads the same copy
                const bool flushed = mv_chunk<Real, VPT, (VPT >= 8 && !HOLD), (VPT <= 4 || !HOLD)>(
                    r0, r1, red, resident ? wsm : ws.w(s) + r0, pv, pc, acc, dacc, m, ring,
                    full, empty, rg, !resident, slots, phase, timed_out);
                mv_finish<Real, VPT>(p, s, g, m, acc, flushed, dacc, red, dsl);
                // op and red are written again only past the barriers of the next chunk
            }
        }
        if (spec && pass > 0) {
            __syncthreads();
            if (sc[0].done) break;
        }
        if (!grid_barrier(p.bar, &flag)) {
            timed_out = true;
            break;
        }
        // ---------------- phase B
        rr_spec = sc[0].gam;
        for (int q = NT / 32 - 1 - warp; warp > 0 && q < p.Q; q += NT / 32 - 1) {
            // a tile of query q is this CTA's: the first w >= q nblk with w = blockIdx.x mod
            // gridDim.x lies below (q + 1) nblk
            const int lo = q * p.nblk, n = gridDim.x, b = blockIdx.x;
            const int w = lo <= b ? b : b + (lo - b + n - 1) / n * n;
            if (w >= lo + p.nblk || sc[q].done) continue;
            double a;
            int ok;
            cg_step_scalar<Real>(p, q, sc[q], a, ok);
            __syncwarp();
            if (lane == 0) {
                sc[q].a = a;
                sc[q].ok = ok;
            }
        }
        for (int w = blockIdx.x; w < ntile; w += gridDim.x) {
            const int s = w / p.nblk;
            if (!sc[s].done) cg_tile<Real, NT>(p, s, w - s * p.nblk, sc[s], tsm);
            __syncthreads();
        }
        if (!grid_barrier(p.bar, &flag)) {
            timed_out = true;
            break;
        }
    }
    // every copy requested has landed before the CTA exits: the last use of each slot
    if (threadIdx.x == 0)
        for (int st = 0; st < S; ++st) {
            const int use = st < pr.slot ? pr.par : pr.par ^ 1;
            if (st < pr.slot || pr.full) mbar_wait_or_flag(&full[st], (uint32_t)use, timed_out);
        }
    if (timed_out) atomicCAS(&p.st[0].status, 0, (int)FBSDE_ERR_TIMEOUT);
}

}  // namespace dev
}  // namespace fbsde
