// fbsde_level.cuh -- the d-vector work of a level around its CG, over tiles of coordinates
// (the CG's own tiles, fbsde_cg.cuh): the set-up of the regression from its moments, and the
// intercept and next starting guess from its solution.  Included after fbsde_cg.cuh.
//   k_level_moments   the partial moments added, S, b', Gx = sum w (D . x) D / W;
//   k_level_rhs       lambda, right-hand side, residual; the query's last tile sets the
//                     scalars the CG starts from;
//   k_level_end       next starting guess, alpha_x of the level; the query's last tile sets
//                     alpha and what the next level (or u(0, x0)) takes from it.
// Each replaces a kernel of one CTA per query (k_reduce_partials with k_moments_finalize, and
// k_cg_post), whose FP64 chains ran over all coordinates: one query, d = 1000: 33 + 7 us of
// set-up and 20 us after the CG before, 8 + 7.5 and 6.5 us here (an arrival counter, the shares
// and 64-cycle FP64 chains).  The forward SDE and the
// three-launch CG keep those (their sums stay in that order).
#pragma once
#include "fbsde_cg.cuh"

namespace fbsde {
namespace dev {

constexpr int kTileThreads = 128;   // threads of the kernels without partial vectors

// Sums of NV shares [tile][4] over the tiles of a query, by one warp (all lanes the same).
template <int NV>
__device__ __forceinline__ void tile_shares(const double *sh, int n, double (&v)[NV])
{
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int i = 0; i < NV; ++i) v[i] = 0.0;
    for (int b0 = lane; b0 < n; b0 += 32 * 4) {
        double q[4][NV];
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
            for (int i = 0; i < NV; ++i)
                q[u][i] = b0 + 32 * u < n ? __ldcg(sh + 4 * (b0 + 32 * u) + i) : 0.0;
#pragma unroll
        for (int i = 0; i < NV; ++i) v[i] += (q[0][i] + q[1][i]) + (q[2][i] + q[3][i]);
    }
    warp_sum(v);
}

// A tile's shares: sums of the owners' values (thread t < kTileThreads in the four warps) into
// out[0 .. NV).  sm: [4][NV].  Every owner thread calls it; bar_id: a named barrier of theirs.
template <int NV>
__device__ __forceinline__ void tile_put(double (&v)[NV], double (*sm)[NV], int t, double *out)
{
    warp_sum(v);
    if ((t & 31) == 0)
#pragma unroll
        for (int i = 0; i < NV; ++i) sm[t >> 5][i] = v[i];
    bar_named(14, kTileThreads);
    if (t == 0)
#pragma unroll
        for (int i = 0; i < NV; ++i) out[i] = (sm[0][i] + sm[1][i]) + (sm[2][i] + sm[3][i]);
}

// True in every thread of the query's last tile to arrive, whose later reads then see the
// other tiles' writes.  Called by all threads of the block.
__device__ __forceinline__ bool tile_last(const Params &p, int s, int *flag)
{
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        const bool last = atomicAdd(&p.st[s].arrive_q, 1) == p.nblk - 1;
        if (last) {
            p.st[s].arrive_q = 0;
            __threadfence();
        }
        *flag = last;
    }
    __syncthreads();
    return *flag != 0;
}

// Level k = p.level - 1's moments: the partial vectors (p.G of them, part_vecs = 3) of the
// tile added as in the CG, the scalar partials by one more warp of every block.  warm = 0: no
// starting guess.  Shares (|S|^2, S . x) into slot 7, free until the CG.
template <typename Real>
__global__ void __launch_bounds__(kCgThreads) k_level_moments(Params p, int warm)
{
    extern __shared__ __align__(128) unsigned char smem_raw[];
    CgTileSm<Real> *sm = reinterpret_cast<CgTileSm<Real> *>(smem_raw);   // [3]
    __shared__ double sc[3], tsm[4][2];
    const int s = blockIdx.y, tile = blockIdx.x;
    const WS<Real> ws(p);
    SolveState &st = p.st[s];
    const int width = 4 * p.cg_lpr;
    const int t = (int)threadIdx.x - 32, i = tile * width + t;
    const bool own = t >= 0 && t < width && i < p.ld;
    double xv = 0.0;
    if (own) {
        if (warm) xv = ws.v64(s, 0)[i];
        else ws.v64(s, 0)[i] = 0.0;
    }
    if (threadIdx.x >= kCgThreads - 32) {   // W, sum w (Y - yref), sum w |D|^2
        double v[3];
        tile_shares(ws.spart(s, 0), p.nsp, v);
        if (threadIdx.x == kCgThreads - 32) {
            const double invW = 1.0 / v[0], cp = v[1] * invW;
            sc[0] = invW;
            if (tile == 0) {
                st.invW = invW;
                st.c = cp + st.yref;
                st.sumz_l = cp;               // for k_level_rhs
                st.zz_l = v[2] * invW;
            }
        }
    }
#pragma unroll
    for (int v = 0; v < 3; ++v) cg_partials<Real>(p, s, tile, v, sm[v]);
    __syncthreads();
    if (t < 0 || t >= kTileThreads) return;
    double a[2] = {0.0, 0.0};
    if (own) {
        const double invW = sc[0];
        const double S = cg_join<Real>(p, sm[0], t) * invW;
        ws.v64(s, 3)[i] = S;
        ws.v64(s, 4)[i] = cg_join<Real>(p, sm[1], t) * invW;
        ws.v64(s, 5)[i] = cg_join<Real>(p, sm[2], t) * invW;
        a[0] = S * S;
        a[1] = S * xv;
    }
    tile_put(a, tsm, t, ws.v64(s, 7) + 4 * tile);
}

// lambda = ridge_rel (sum w |D|^2 / W - |S|^2) / d (Remark 2.2), rhs = b' - c' S (Eq. 3.19),
// r = rhs - (Gx - S (S . x)) - lambda x.  Shares (|rhs|^2, |r|^2, S . r) into slot 2.
template <typename Real>
__global__ void __launch_bounds__(kTileThreads) k_level_rhs(Params p)
{
    __shared__ double sc[2], tsm[4][3];
    __shared__ int flag;
    const int s = blockIdx.y, tile = blockIdx.x, t = threadIdx.x;
    const WS<Real> ws(p);
    SolveState &st = p.st[s];
    const int width = 4 * p.cg_lpr, i = tile * width + t;
    const bool own = t < width && i < p.ld;
    double S = 0.0, B = 0.0, Gx = 0.0, x = 0.0;
    if (own) {
        S = ws.v64(s, 3)[i];
        B = ws.v64(s, 4)[i];
        Gx = ws.v64(s, 5)[i];
        x = ws.v64(s, 0)[i];
    }
    const double cp = st.sumz_l;
    if (s == 0 && tile == 0 && t == 0) *p.bar = 0u;   // the CG loop's grid barrier
    if (t < 32) {
        double v[2];
        tile_shares(ws.v64(s, 7), p.nblk, v);
        if (t == 0) {
            sc[0] = p.ridge_rel * (st.zz_l - v[0]) / p.d;
            sc[1] = v[1];
        }
    }
    __syncthreads();
    const double lambda = sc[0], sx = sc[1];
    double a[3] = {0.0, 0.0, 0.0};
    if (own) {
        const double rhs = fma(-cp, S, B);
        const double r = (rhs - fma(-S, sx, Gx)) - lambda * x;
        ws.v64(s, 4)[i] = rhs;
        ws.v64(s, 1)[i] = r;
        ws.vR(s, 0)[i] = (Real)r;
        if (p.tape_v) p.tape_v[(((size_t)s * p.N + (p.level - 1)) * 2 + 0) * p.ld + i] = S;
        a[0] = rhs * rhs;
        a[1] = r * r;
        a[2] = S * r;
    }
    tile_put(a, tsm, t, ws.v64(s, 2) + 4 * tile);
    if (!tile_last(p, s, &flag) || t >= 32) return;
    double v[3];
    tile_shares(ws.v64(s, 2), p.nblk, v);
    if (t == 0) {
        if (p.newton_level >= 0 && p.tr_newton)
            p.tr_newton[(size_t)s * p.N + p.newton_level] = st.newton_max;
        st.lambda = lambda;
        if (p.tape_s) {
            double *ts = p.tape_s + ((size_t)s * p.N + (p.level - 1)) * 4;
            ts[0] = lambda;
            ts[1] = st.invW;
        }
        st.rhs2 = v[0];
        st.rr = v[1];
        st.sp = v[2];
        st.iters = 0;
        st.done = (v[1] <= p.cg_tol2 * v[0]) ? 1 : 0;
    }
}

// After the CG of level k (driftless; as k_cg_post): alpha = c - S . alpha_x (Eq. 3.20),
// Z_k = sigma alpha_x, the next level's starting guess g = 2 alpha_x^k - alpha_x^{k+1}
// (alpha_x^k at the top level), traces; at k = 0 the Newton step at x0 gives u(0, x0).  Shares
// (S . alpha_x, sum alpha_x, |alpha_x|^2) into slot 7, free after the CG.
template <typename Real>
__global__ void __launch_bounds__(kTileThreads) k_level_end(Params p)
{
    __shared__ double tsm[4][3];
    __shared__ int flag;
    const int s = blockIdx.y, tile = blockIdx.x, t = threadIdx.x, k = p.level;
    const WS<Real> ws(p);
    SolveState &st = p.st[s];
    const int width = 4 * p.cg_lpr, i = tile * width + t;
    double a[3] = {0.0, 0.0, 0.0};
    if (t < width && i < p.ld) {
        const double xi = ws.v64(s, 0)[i], S = ws.v64(s, 3)[i];
        const double g = k + 1 < p.N ? 2.0 * xi - ws.v64(s, 8)[i] : xi;
        ws.v64(s, 8)[i] = xi;
        ws.v64(s, 0)[i] = g;
        ws.vR(s, 3)[i] = (Real)g;
        ws.vR(s, 1)[i] = (Real)xi;
        if (i < p.d) {
            if (p.tr_alpha_x) p.tr_alpha_x[((size_t)s * p.N + k) * p.d + i] = xi;
            if (k == 0 && p.grad) p.grad[(size_t)s * p.d + i] = xi;
        }
        if (p.tape_v) p.tape_v[(((size_t)s * p.N + k) * 2 + 1) * p.ld + i] = xi;
        a[0] = S * xi;
        a[1] = xi;
        a[2] = xi * xi;
    }
    tile_put(a, tsm, t, ws.v64(s, 7) + 4 * tile);
    if (!tile_last(p, s, &flag) || t >= 32) return;
    double v[3];
    tile_shares(ws.v64(s, 7), p.nblk, v);
    if (t != 0) return;
    const double alpha = st.c - v[0];
    st.alpha = alpha;
    st.yref = alpha;
    st.sumz = p.sigma * v[1];
    st.zz = p.sigma * p.sigma * v[2];
    st.sum_ax = v[1];
    st.newton_max = 0;
    if (p.tr_alpha) p.tr_alpha[(size_t)s * p.N + k] = alpha;
    if (p.tape_s) p.tape_s[((size_t)s * p.N + k) * 4 + 2] = alpha;
    if (p.tr_cg) p.tr_cg[(size_t)s * p.N + k] = st.iters;
    if (k == 0) {   // every particle of level 0 sits at x0: one Newton solve
        const double feat = f_feature(p, 0.0, st.phi0, st.sumz, st.zz, st.psi0);
        int it;
        const double u = newton(p, alpha, feat, it);
        if (it < 0 && st.status == 0) st.status = FBSDE_ERR_NEWTON;
        const int used = it < 0 ? p.newton_max_iter : it;
        st.newton_max_all = max(st.newton_max_all, used);
        if (p.tr_newton) p.tr_newton[(size_t)s * p.N] = used;
        if (!isfinite(u) && st.status == 0) st.status = FBSDE_ERR_NONFINITE;
        p.u0[s] = u;
    }
}

}  // namespace dev
}  // namespace fbsde
