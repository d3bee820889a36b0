// Checks of the solve's kernels below the C ABI, linked against the library's own objects:
//   barrier   the CG loop's grid barrier gives up after its limit when a CTA does not arrive
//             (and the launch ends), a partial count left in its word does not reach the next
//             loop, and a loop after a recorded timeout ends at once.
//   delta     the product's shares of r^T A r, sum_j w_j (D_j . r)^2, against the same sum in
//             long double, on rows and operands whose dot products are exact in FP32.
//   runs      the product's FP32 sums over long chunks, on rows of which one is 2^25 times the
//             others: only the rest of its run is lost beside it.
// Prints one line per check and exits 1 when one fails.
#include "fbsde_api.cu"

#include <cstdio>
#include <string>

namespace check {

using fbsde::Layout;
using fbsde::Params;
using fbsde::SolveState;
using LR = fbsde::Launch<float>;

int failures = 0;
void report(const char *what, bool ok)
{
    std::printf("%s: %s\n", what, ok ? "ok" : "FAILED");
    if (!ok) ++failures;
}
#define CUDA_OK(x)                                                                \
    do {                                                                          \
        const cudaError_t e_ = (x);                                               \
        if (e_ != cudaSuccess) {                                                  \
            std::printf("%s: %s\n", #x, cudaGetErrorString(e_));                  \
            std::exit(2);                                                         \
        }                                                                         \
    } while (0)

// CTAs 1 .. arrive - 1 and CTA 0 meet at the barrier, the others return at once.
__global__ void k_meet(unsigned int *word, int arrive, unsigned long long limit_ns, int *out,
                       unsigned long long *ns)
{
    __shared__ int flag;
    if ((int)blockIdx.x >= arrive) return;
    const unsigned long long t0 = fbsde::dev::globaltimer_ns();
    const bool ok = fbsde::dev::grid_barrier(word, &flag, limit_ns);
    if (threadIdx.x == 0) {
        out[blockIdx.x] = ok ? 1 : 0;
        ns[blockIdx.x] = fbsde::dev::globaltimer_ns() - t0;
    }
}

// A driftless FP32 solve up to the first CG loop, on a workspace of its own.
struct FirstLoop {
    Layout L;
    Params p, ps;
    char *ws = nullptr;
    double *x0 = nullptr, *u0 = nullptr;
    explicit FirstLoop(int d, int M)
    {
        fbsde_problem P{};
        P.kind = FBSDE_AC_MANUFACTURED;
        P.d = d;
        P.N = 3;
        P.M = M;
        P.sigma = 1.0;
        P.T = 0.5;
        P.ridge_rel = 1e-3;
        P.cg_tol = 1e-7;
        P.precision = FBSDE_FP32;
        if (fbsde::make_layout(&P, 1, L) != FBSDE_OK) std::exit(2);
        CUDA_OK(cudaMalloc(&ws, L.total));
        CUDA_OK(cudaMemset(ws, 0, L.total));
        CUDA_OK(cudaMalloc(&x0, d * sizeof(double)));
        CUDA_OK(cudaMemset(x0, 0, d * sizeof(double)));
        CUDA_OK(cudaMalloc(&u0, sizeof(double)));
        p = fbsde::make_params(&P, L, ws, 5, 0, u0, nullptr, nullptr);
        p.level = P.N;
        p.newton_level = -1;
        ps = p;
        ps.G = L.Gs;
        CUDA_OK(LR::setup(p, x0, nullptr, 0));
        CUDA_OK(LR::step(ps, L, 0));
        CUDA_OK(LR::level_moments(ps, L, 0, 0));
    }
    ~FirstLoop()
    {
        cudaFree(ws);
        cudaFree(x0);
        cudaFree(u0);
    }
    Params loop() const
    {
        Params q = p;
        q.level = p.N - 1;
        return fbsde::product_params(q, L);
    }
    std::vector<double> solution() const
    {
        std::vector<double> x(L.ld);
        CUDA_OK(cudaMemcpy(x.data(), p.vec64, L.ld * sizeof(double), cudaMemcpyDeviceToHost));
        return x;
    }
    SolveState state() const
    {
        SolveState st;
        CUDA_OK(cudaMemcpy(&st, p.st, sizeof st, cudaMemcpyDeviceToHost));
        return st;
    }
};

void check_barrier()
{
    unsigned int *word;
    int *out;
    unsigned long long *ns;
    CUDA_OK(cudaMalloc(&word, 4));
    CUDA_OK(cudaMalloc(&out, 4 * sizeof(int)));
    CUDA_OK(cudaMalloc(&ns, 4 * sizeof(unsigned long long)));
    for (int arrive : {4, 3}) {
        CUDA_OK(cudaMemset(word, 0, 4));
        CUDA_OK(cudaMemset(out, 0, 4 * sizeof(int)));
        CUDA_OK(cudaMemset(ns, 0, 4 * sizeof(unsigned long long)));
        unsigned long long limit = 20'000'000ull;
        void *args[] = {&word, &arrive, &limit, &out, &ns};
        CUDA_OK(cudaLaunchCooperativeKernel(reinterpret_cast<void *>(k_meet), dim3(4), dim3(64),
                                            args, 0, 0));
        CUDA_OK(cudaDeviceSynchronize());
        int h[4];
        unsigned long long t[4];
        CUDA_OK(cudaMemcpy(h, out, sizeof h, cudaMemcpyDeviceToHost));
        CUDA_OK(cudaMemcpy(t, ns, sizeof t, cudaMemcpyDeviceToHost));
        bool ok = true;
        for (int b = 0; b < arrive; ++b)
            ok = ok && (arrive == 4 ? h[b] == 1 : h[b] == 0 && t[b] >= limit && t[b] < 10 * limit);
        report(arrive == 4 ? "barrier of all CTAs" : "barrier with a CTA missing", ok);
    }
    CUDA_OK(cudaFree(word));
    CUDA_OK(cudaFree(out));
    CUDA_OK(cudaFree(ns));

    std::vector<double> ref;
    for (unsigned int left : {0u, 1u, 0x80000007u}) {   // the word as a given-up wait leaves it
        FirstLoop f(300, 900);
        CUDA_OK(cudaMemcpy(f.p.bar, &left, 4, cudaMemcpyHostToDevice));
        CUDA_OK(LR::level_rhs(f.ps, f.L, 0));
        unsigned int word_now = 1;
        CUDA_OK(cudaMemcpy(&word_now, f.p.bar, 4, cudaMemcpyDeviceToHost));
        const bool reset = word_now == 0;
        report("barrier word reset before the loop", reset);
        if (!reset) return;   // the loop must not run on it
        CUDA_OK(LR::cg_loop(f.loop(), f.L, 0));
        CUDA_OK(cudaDeviceSynchronize());
        const std::vector<double> x = f.solution();
        const SolveState st = f.state();
        if (ref.empty()) ref = x;
        report("loop after a partial count", st.status == 0 && st.done == 1 && st.iters > 1 && x == ref);
    }
    {
        FirstLoop f(300, 900);
        CUDA_OK(LR::level_rhs(f.ps, f.L, 0));
        SolveState st = f.state();
        st.status = FBSDE_ERR_TIMEOUT;
        CUDA_OK(cudaMemcpy(f.p.st, &st, sizeof st, cudaMemcpyHostToDevice));
        CUDA_OK(LR::cg_loop(f.loop(), f.L, 0));
        CUDA_OK(cudaDeviceSynchronize());
        const SolveState now = f.state();
        report("loop after a recorded timeout",
               now.status == FBSDE_ERR_TIMEOUT && now.iters == 0 && now.done == 0);
    }
}

// Rows and r of small integers (r scaled by a power of two): every dot product t is exact in
// FP32, in any order.  Each term w t^2 has two FP32 roundings, 2 2^-24 of it at most; the sums
// are compensated, n rows a team leave (n 2^-24)^2 of them (Neumaier's bound).
void check_delta(int d, int M)
{
    for (float scale : {1.0f, 0x1p-70f, 0x1p50f}) {
        FirstLoop f(d, M);
        const Layout &L = f.L;
        std::vector<float> rows((size_t)M * L.ld), r(L.ld), w(M);
        uint32_t seed = 12345;
        auto next = [&] { return (seed = seed * 1664525u + 1013904223u) >> 8; };
        for (int i = 0; i < L.ld; ++i) r[i] = i < d ? scale * (float)((int)(next() % 7) - 3) : 0.0f;
        long double want = 0.0L;
        for (int j = 0; j < M; ++j) {
            w[j] = (float)next() * 0x1p-24f;
            long double t = 0.0L;
            for (int i = 0; i < L.ld; ++i) {
                const float x = i < d ? (float)((int)(next() % 7) - 3) : 0.0f;
                rows[(size_t)j * L.ld + i] = x;
                t += (long double)x * r[i];
            }
            want += (long double)w[j] * t * t;
        }
        CUDA_OK(cudaMemcpy(f.p.delta, rows.data(), rows.size() * 4, cudaMemcpyHostToDevice));
        CUDA_OK(cudaMemcpy(f.p.vecR, r.data(), r.size() * 4, cudaMemcpyHostToDevice));
        CUDA_OK(cudaMemcpy(f.p.w, w.data(), w.size() * 4, cudaMemcpyHostToDevice));
        SolveState st = f.state();
        st.rr = 0.0;
        for (float v : r) st.rr += (double)v * v;
        CUDA_OK(cudaMemcpy(f.p.st, &st, sizeof st, cudaMemcpyHostToDevice));
        const Params q = f.loop();
        CUDA_OK(LR::matvec(q, L, 0));
        CUDA_OK(cudaDeviceSynchronize());
        std::vector<double> share((size_t)L.Gc * fbsde::kDpart);
        CUDA_OK(cudaMemcpy(share.data(), q.dpart, share.size() * 8, cudaMemcpyDeviceToHost));
        double got = 0.0;
        for (int g = 0; g < L.Gc; ++g) got += share[(size_t)g * fbsde::kDpart];
        const double err = std::fabs((double)(((long double)got - want) / want));
        std::printf("d %d M %d scale %.1e: error %.1e (%d chunks, %d teams)\n", d, M, scale, err, L.Gc,
                    L.teams);
        const double n = (M + L.Gc * L.teams - 1) / (L.Gc * L.teams) + 1.0;
        report("delta", err <= 0x1.00001p-23 + n * n * 0x1p-48);
    }
}

// Every row has D_0 = 1 and r = e_0, so t = w = 1 and coordinate 1 of a chunk's partial vector is
// the sum of the rows' D_1: 1 in the chunk's first row and 2^-25 in the others.  In FP32 the 1
// swallows what is added to it one by one: the other kMvRun - 1 rows of its run (one unit of
// 2^-25 each); after that every addition to it rounds by two units at most, one for each further
// run of the team and for each other team.
void check_runs(int d, int M)
{
    FirstLoop f(d, M);
    const Layout &L = f.L;
    std::vector<float> rows((size_t)M * L.ld, 0.0f), r(L.ld, 0.0f), w(M, 1.0f);
    r[0] = 1.0f;
    std::vector<int> count(L.Gc);
    for (int g = 0; g < L.Gc; ++g) {
        const long long r0 = (long long)M * g / L.Gc, r1 = (long long)M * (g + 1) / L.Gc;
        count[g] = (int)(r1 - r0);
        for (long long j = r0; j < r1; ++j) {
            rows[(size_t)j * L.ld] = 1.0f;
            rows[(size_t)j * L.ld + 1] = j == r0 ? 1.0f : 0x1p-25f;
        }
    }
    CUDA_OK(cudaMemcpy(f.p.delta, rows.data(), rows.size() * 4, cudaMemcpyHostToDevice));
    CUDA_OK(cudaMemcpy(f.p.vecR, r.data(), r.size() * 4, cudaMemcpyHostToDevice));
    CUDA_OK(cudaMemcpy(f.p.w, w.data(), w.size() * 4, cudaMemcpyHostToDevice));
    const Params q = f.loop();
    CUDA_OK(LR::matvec(q, L, 0));
    CUDA_OK(cudaDeviceSynchronize());
    std::vector<float> part((size_t)L.Gc * L.ld);
    CUDA_OK(cudaMemcpy(part.data(), q.part, part.size() * 4, cudaMemcpyDeviceToHost));
    double worst = 0.0;
    bool ok = true;
    const int run = fbsde::dev::kMvRun;
    for (int g = 0; g < L.Gc; ++g) {
        const double exact = 1.0 + (count[g] - 1) * 0x1p-25;
        const double lost = std::fabs(part[(size_t)g * L.ld + 1] - exact) * 0x1p25;   // units
        const int team = (count[g] + L.teams - 1) / L.teams;
        ok = ok && lost <= run - 1 + 2 * ((team - 1) / run) + 2 * (L.teams - 1);
        worst = std::max(worst, lost);
    }
    std::printf("d %d M %d: %d chunks of %d rows, %d teams, resident %d: %.0f units lost\n", d, M, L.Gc,
                count[0], L.teams, L.cg_res, worst);
    report("runs", ok && (L.teams > 1 || count[0] > 4 * run));
}

}  // namespace check

int main(int argc, char **argv)
{
    const std::string what = argc > 1 ? argv[1] : "";
    if (what == "barrier") check::check_barrier();
    else if (what == "delta")   // several teams; chunks of more than 32 rows a team; one team a row
        for (auto [d, M] : {std::pair{301, 900}, {33, 90001}, {5003, 4001}}) check::check_delta(d, M);
    else if (what == "runs")   // one team a row; several, streaming and in shared memory
        for (auto [d, M] : {std::pair{5003, 20011}, {33, 456007}, {4, 900001}}) check::check_runs(d, M);
    else return 2;
    return check::failures ? 1 : 0;
}
