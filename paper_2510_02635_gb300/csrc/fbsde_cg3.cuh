// fbsde_cg3.cuh -- the CG pass in three launches (FP32): product, reduction of its partial
// vectors, vector updates.  Included after fbsde_cg.cuh.  It keeps the wide tiling of the
// product (608 CTAs over the queries, one partial each) and forms delta = w . r from the
// reduced product, so a pass has two exchanges instead of one.  It serves the shapes whose
// passes are long enough not to feel that, wherever the loop is not taken and a row has one team
// (rows above 16 KB): several queries whose rows stream from HBM, rows too wide for the loop's
// block (d > 10240), more than 64 queries (also of small clouds); and the forward SDE, whose
// slopes are a small remainder of a large mean shift (their rounding shows in the fifth digit, so
// its sums keep this order).  Measured: d = 10^4, M = 16384, 16 queries, 338.0 ms for five levels here and
// 338.2 ms in two launches (product 1390 and 1375 us).
#pragma once
#include "fbsde_cg.cuh"

namespace fbsde {
namespace dev {

// Partial product of the CTA's rows: as k_matvec, one row per team at a time, without the
// shares of r . A r.
template <typename Real, int VPT, bool WIDE>
__global__ void __launch_bounds__(WIDE ? 544 : (VPT >= 8 ? 352 : 288), 1) k_product(Params p)
{
    constexpr int E = Chunk<Real>::E;
    extern __shared__ __align__(128) unsigned char smem_raw[];
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
        const int ct = threadIdx.x - 32;
        const int tthreads = 32 * tw;
        const int team = ct / tthreads, tl = ct - team * tthreads, wt = tl >> 5;
        const Real *pv = ws.vR(s, 0);
        const Real *wv = ws.w(s);
        Chunk<Real> acc[VPT], pc[VPT];   // pc: the operand r
#pragma unroll
        for (int v = 0; v < VPT; ++v) {
            zero(acc[v]);
            const int c = tl + tthreads * v;
            if (c < nch) pc[v] = ldg_chunk(pv + c * E);
            else zero(pc[v]);
        }
        int phase = 0;
        for (long long i = 0; i < nst; ++i) {
            const int st = (int)(i % S);
            mbar_wait_or_flag(&full[st], (uint32_t)((i / S) & 1), timed_out);
            const long long row0 = r0 + i * R;
            const int rows = (int)min((long long)R, r1 - row0);
            const Real *buf = ring + (size_t)st * R * row_elems;
            for (int rr = team; rr < rows; rr += nteams) {
                const Real *row = buf + (size_t)rr * row_elems;
                // the row's weight, loaded before the dot product so that its latency is
                // hidden behind the product and the team sum instead of following them
                const Real wrow = wv[row0 + rr];
                // narrow teams keep their chunks of the row in registers between the dot
                // product and the weighted sum (one shared-memory read of the row instead
                // of two); the 11- to 16-warp teams of the widest rows have no registers to
                // spare
                constexpr bool kReread = WIDE;
                constexpr int kHeld = kReread ? 1 : VPT;
                Chunk<Real> dl[kHeld];
                Real t = Real(0);
#pragma unroll
                for (int v = 0; v < VPT; ++v) {
                    const int c = tl + tthreads * v;
                    Chunk<Real> &x = dl[kReread ? 0 : v];
                    if (c < nch) x = ld_chunk(row + c * E);
                    else zero(x);
#pragma unroll
                    for (int e = 0; e < E; ++e) t += x.v[e] * pc[v].v[e];
                }
#pragma unroll
                for (int o = 16; o; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
                if (tw > 1) {
                    Real *sl = slots + (size_t)(team * 2 + phase) * 32;
                    if (lane == 0) sl[wt] = t;
                    bar_named(1 + team, tthreads);
                    t = Real(0);
                    for (int w2 = 0; w2 < tw; ++w2) t += sl[w2];
                    phase ^= 1;
                }
                const Real coef = wrow * t;
#pragma unroll
                for (int v = 0; v < VPT; ++v) {
                    const int c = tl + tthreads * v;
                    if (c < nch) {
                        if (kReread) dl[0] = ld_chunk(row + c * E);
                        const Chunk<Real> &x = dl[kReread ? 0 : v];
#pragma unroll
                        for (int e = 0; e < E; ++e) acc[v].v[e] += coef * x.v[e];
                    }
                }
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&empty[st]);
        }
        // team accumulators -> CTA partial (teams summed in team order via the ring)
        Real *dst = ws.part(s, g, 0);
        if (nteams == 1) {
#pragma unroll
            for (int v = 0; v < VPT; ++v) {
                const int c = tl + tthreads * v;
                if (c < nch) st_chunk(dst + c * E, acc[v]);
            }
        } else {
            bar_named(15, 32 * nteams * tw);   // every consumer is past its last ring read
#pragma unroll
            for (int v = 0; v < VPT; ++v) {
                const int c = tl + tthreads * v;
                if (c < nch) st_chunk(ring + (size_t)team * row_elems + c * E, acc[v]);
            }
            bar_named(15, 32 * nteams * tw);
            for (int c = ct; c < nch; c += 32 * nteams * tw) {
                Chunk<Real> sum = ld_chunk(ring + c * E);
                for (int t2 = 1; t2 < nteams; ++t2) {
                    const Chunk<Real> o = ld_chunk(ring + (size_t)t2 * row_elems + c * E);
#pragma unroll
                    for (int e = 0; e < E; ++e) sum.v[e] += o.v[e];
                }
                st_chunk(dst + c * E, sum);
            }
        }
    }
    if (timed_out) atomicCAS(&p.st[s].status, 0, (int)FBSDE_ERR_TIMEOUT);
}

// Sum of the G partial products in the order of k_reduce_partials, then
//   w = sum / W - S (S . r) + lambda r   (Gamma_c r + lambda r, Eq. 3.19's operator)
// into slot 5 and this block's share of w . r into bpart.  Grid (ceil(ld / kRedTile), Q).
template <typename Real>
__global__ void __launch_bounds__(512) k_product_reduce(Params p)
{
    using Acc = RedAcc<Real>;
    using Lo = decltype(Acc{}.lo());
    constexpr int kB = 8;  // loads in flight per lane
    __shared__ Real sh_s[16][kRedTile];
    __shared__ Lo sh_c[16][kRedTile];
    __shared__ double sh_w[4];
    const int s = blockIdx.y;
    SolveState &st = p.st[s];
    if (st.done) return;
    const int lane = threadIdx.x & 31, gg = threadIdx.x >> 5, GR = blockDim.x >> 5;
    const int e0 = blockIdx.x * kRedTile + 4 * lane;  // first element of this lane
    const bool in = e0 < p.ld;                        // ld is a multiple of 4
    const WS<Real> ws(p);
    const size_t stride = (size_t)kPartVecs * p.ld * GR;   // between this group's partials
    {
        Acc acc[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) acc[e].init();
        if (in) {
            const Real *src = ws.part(s, gg, 0) + e0;
            for (int g0 = gg; g0 < p.G; g0 += kB * GR, src += kB * stride) {
                Quad<Real> t[kB];
#pragma unroll
                for (int u = 0; u < kB; ++u)
                    if (g0 + u * GR < p.G) t[u] = ld_quad(src + u * stride);
#pragma unroll
                for (int u = 0; u < kB; ++u) {
                    if (g0 + u * GR < p.G) {
#pragma unroll
                        for (int e = 0; e < 4; ++e) acc[e].add(t[u].v[e]);
                    }
                }
            }
        }
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            sh_s[gg][4 * lane + e] = acc[e].hi();
            sh_c[gg][4 * lane + e] = acc[e].lo();
        }
        __syncthreads();
        if (threadIdx.x < kRedTile) {
            const int t = threadIdx.x, i = blockIdx.x * kRedTile + t;
            Acc tot;
            tot.init();
            for (int k = 0; k < GR; ++k) tot.merge(sh_s[k][t], sh_c[k][t]);
            const double sum = tot.value();
            double wr = 0.0;
            if (i < p.ld) {
                const double ri = ws.v64(s, 1)[i];
                const double wi = sum * st.invW - ws.v64(s, 3)[i] * st.sp + st.lambda * ri;
                ws.v64(s, 5)[i] = wi;
                wr = wi * ri;
            }
#pragma unroll
            for (int o = 16; o; o >>= 1) wr += __shfl_xor_sync(0xffffffffu, wr, o);
            if (lane == 0) sh_w[t >> 5] = wr;
        }
        __syncthreads();
    }
    if (threadIdx.x == 0)   // the next kernel boundary makes the shares visible
        p.bpart[((size_t)s * p.nblk3 + blockIdx.x) * kBpart] = ((sh_w[0] + sh_w[1]) + sh_w[2]) + sh_w[3];
}

// Four consecutive values at a 16-byte aligned address (two 16-byte accesses for doubles,
// one for floats).
__device__ __forceinline__ void ld4(double (&v)[4], const double *q)
{
    const double2 a = *reinterpret_cast<const double2 *>(q);
    const double2 b = *reinterpret_cast<const double2 *>(q + 2);
    v[0] = a.x; v[1] = a.y; v[2] = b.x; v[3] = b.y;
}
__device__ __forceinline__ void st4(double *q, const double (&v)[4])
{
    *reinterpret_cast<double2 *>(q) = make_double2(v[0], v[1]);
    *reinterpret_cast<double2 *>(q + 2) = make_double2(v[2], v[3]);
}
__device__ __forceinline__ void st4(float *q, const float (&v)[4])
{
    *reinterpret_cast<float4 *>(q) = make_float4(v[0], v[1], v[2], v[3]);
}

// The pass's scalars (every block adds the shares of w . r in the same order) and vector
// updates, one warp per tile of kRedTile elements, four consecutive ones per lane.  The
// query's last block (arrival counter) adds the shares of S . r and r . r, stores the new
// state and tests convergence; in a CUDA graph (use_h = 1) the last query to finish sets the
// while-loop condition.  Grid (ceil(ld / kRedTile), Q).
template <typename Real>
__global__ void __launch_bounds__(32) k_cg_update(Params p, cudaGraphConditionalHandle h, int use_h)
{
    const int s = blockIdx.y, lane = threadIdx.x;
    SolveState &st = p.st[s];
    bool global_arrive = false;
    if (st.done) {
        global_arrive = blockIdx.x == 0;   // one block answers for a finished query
    } else {
        const WS<Real> ws(p);
        double *x = ws.v64(s, 0), *r = ws.v64(s, 1), *pp = ws.v64(s, 2), *S = ws.v64(s, 3),
               *w = ws.v64(s, 5), *sv = ws.v64(s, 7);
        Real *rR = ws.vR(s, 0);
        double *bp = p.bpart + (size_t)s * p.nblk3 * kBpart;
        const int t = st.iters;
        const double gam = st.rr;
        const int i0 = blockIdx.x * kRedTile + 4 * lane;
        const bool in = i0 < p.ld;   // ld is a multiple of 4
        // every value of the lane's four elements is loaded first, before the pass's scalars
        // are derived and before the first store (the vectors may alias as far as the
        // compiler can tell, so it would not move a later element's loads above a store)
        double rv[4], wv[4], pv[4], svv[4], xv[4], Sv[4];
        if (in) {
            ld4(rv, r + i0);
            ld4(wv, w + i0);
            ld4(xv, x + i0);
            ld4(Sv, S + i0);
            if (t > 0) {
                ld4(pv, pp + i0);
                ld4(svv, sv + i0);
            }
        }
        double dl = 0.0;   // delta = w . r: the shares in a fixed order, the same in every block
        for (int b = lane; b < p.nblk3; b += 32) dl += __ldcg(bp + (size_t)b * kBpart);
#pragma unroll
        for (int o = 16; o; o >>= 1) dl += __shfl_xor_sync(0xffffffffu, dl, o);
        double beta = 0.0, den = dl;
        if (t > 0) {
            beta = gam / st.rr_prev;
            den = dl - beta * gam / st.cg_alpha;
        }
        const double a = gam / den;
        const int ok = (den > 0.0 && isfinite(a)) ? 1 : 0;
        double sr = 0.0, rr = 0.0;
        if (ok && in) {
            Real rn4[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const double pi = t > 0 ? rv[e] + beta * pv[e] : rv[e];
                const double si = t > 0 ? wv[e] + beta * svv[e] : wv[e];
                pv[e] = pi;
                svv[e] = si;
                xv[e] += a * pi;
                const double rn = rv[e] - a * si;
                rv[e] = rn;
                rn4[e] = (Real)rn;
                sr += Sv[e] * rn;
                rr += rn * rn;
            }
            st4(pp + i0, pv);
            st4(sv + i0, svv);
            st4(x + i0, xv);
            st4(r + i0, rv);
            st4(rR + i0, rn4);
        }
#pragma unroll
        for (int o = 16; o; o >>= 1) {
            sr += __shfl_xor_sync(0xffffffffu, sr, o);
            rr += __shfl_xor_sync(0xffffffffu, rr, o);
        }
        int last = 0;
        if (lane == 0) {
            bp[(size_t)blockIdx.x * kBpart + 1] = sr;
            bp[(size_t)blockIdx.x * kBpart + 2] = rr;
            __threadfence();
            last = atomicAdd(&st.arrive_q, 1) == p.nblk3 - 1;
        }
        last = __shfl_sync(0xffffffffu, last, 0);
        if (last) {
            __threadfence();
            double c0 = 0.0, c1 = 0.0;
            for (int b = lane; b < p.nblk3; b += 32) {
                c0 += __ldcg(bp + (size_t)b * kBpart + 1);
                c1 += __ldcg(bp + (size_t)b * kBpart + 2);
            }
#pragma unroll
            for (int o = 16; o; o >>= 1) {
                c0 += __shfl_xor_sync(0xffffffffu, c0, o);
                c1 += __shfl_xor_sync(0xffffffffu, c1, o);
            }
            if (lane == 0) {
                st.arrive_q = 0;
                if (!ok) {  // breakdown: keep the current iterate
                    st.done = 1;
                    if (!(gam <= p.cg_tol2 * st.rhs2) && st.status == 0) st.status = FBSDE_ERR_CG;
                } else {
                    st.rr_prev = gam;
                    st.cg_alpha = a;
                    st.rr = c1;
                    st.sp = c0;
                    st.iters = t + 1;
                    st.cg_total += 1;
                    if (c1 <= p.cg_tol2 * st.rhs2) {
                        st.done = 1;
                    } else if (t + 1 >= p.cg_max_iter) {
                        st.done = 1;
                        st.cg_exhausted += 1;
                        if (st.status == 0) st.status = FBSDE_ERR_CG;
                    }
                }
                global_arrive = true;
            }
        }
    }
    if (use_h && global_arrive && lane == 0) {
        bool last_q = true;   // one query: its last block is the last arrival
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

}  // namespace dev
}  // namespace fbsde
