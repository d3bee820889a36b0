// Checks of the per-anchor kernels below the C ABI (compiled with fbsde_anchored.cu itself):
//   weights   the column sums of the weights, formed in the distance product's epilogue, where a
//             sum over 64 rows and more rounds in FP32.
// Prints one line per check and exits 1 when one fails.
#include "fbsde_anchored.cu"

#include <cstdio>
#include <cstdlib>
#include <string>

namespace fbsde {
namespace anchored {
namespace check {

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
template <typename T> T *upload(const std::vector<T> &v)
{
    T *p = nullptr;
    CUDA_OK(cudaMalloc(&p, v.size() * sizeof(T)));
    CUDA_OK(cudaMemcpy(p, v.data(), v.size() * sizeof(T), cudaMemcpyHostToDevice));
    return p;
}
template <typename T> std::vector<T> download(const T *p, size_t n)
{
    std::vector<T> v(n);
    CUDA_OK(cudaMemcpy(v.data(), p, n * sizeof(T), cudaMemcpyDeviceToHost));
    return v;
}

// Uniform weights (scale 0: w = 1) and Y that is 2^24 - 1 in the first row of every 128-row
// tile, 1 in its rows 32, 64 and 96 and 0 elsewhere: the tile's sum 2^24 + 2 is exact in 32-row
// FP32 sums that are widened before they are added, and 2^24 in FP32 throughout.  The batch
// window covers every row (K = M).
void check_weights()
{
    const int M = 256, ld = 16;
    std::vector<float> rows((size_t)M * ld, 0.0f);
    std::vector<double> norms(M, 0.0), Y(M, 0.0);
    for (int j = 0; j < M; j += 128) {
        Y[j] = 16777215.0;
        Y[j + 32] = Y[j + 64] = Y[j + 96] = 1.0;
    }
    float *P = upload(rows), *A = upload(rows), *W = upload(std::vector<float>((size_t)M * M));
    double *n = upload(norms), *y = upload(Y), *part = upload(std::vector<double>(2 * M * 3));
    int *status = upload(std::vector<int>(1, 0));
    CUDA_OK(gemm_tc<false>(M, M, ld, ld, P, ld, A, ld,
                           TcWeightsEpi{n, n, y, W, part, M, M, 1.0f, 0.0f}, status, 0,
                           dev::Band{M, M}));
    CUDA_OK(cudaDeviceSynchronize());
    const std::vector<double> got = download(part, 2 * M * 3);
    bool ok = download(status, 1)[0] == 0;
    for (int i = 0; i < 2 * M; ++i)
        ok = ok && got[3 * i] == 128.0 && got[3 * i + 1] == 16777218.0 && got[3 * i + 2] == 0.0;
    report("column sums of the weights", ok);
}

}  // namespace check
}  // namespace anchored
}  // namespace fbsde

int main(int argc, char **argv)
{
    const std::string what = argc > 1 ? argv[1] : "";
    if (what == "weights") fbsde::anchored::check::check_weights();
    else return 2;
    return fbsde::anchored::check::failures ? 1 : 0;
}
