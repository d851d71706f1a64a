// The LU panel kernel with its rows in global memory against the form with the rows in
// shared memory: the first is chosen only when a CTA's rows do not fit (n above about
// 117000), so it is launched here at a small size.  Both must write the same bits.
#include <cstdio>
#include <cstring>
#include <vector>

#include "k_lu.cu"

namespace lsi {
cudaError_t set_smem_limit(const void *func, size_t smem) {
    return cudaFuncSetAttribute(func, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
}
}  // namespace lsi

using namespace lsi;

static bool ok(cudaError_t e, const char *what) {
    if (e != cudaSuccess) std::printf("%s: %s\n", what, cudaGetErrorString(e));
    return e == cudaSuccess;
}

int main() {
    const LuKernels K = lu_kernels();
    const int NB = K.nb, CTAS = 152;
    int bad = 0, runs = 0;
    const int sizes[] = {33, 64, 333, 1000};
    for (int n : sizes) {
        const long long ld = (n + 2) / 2 * 2;
        std::vector<double> W((size_t)n * ld);
        unsigned long long x = 88172645463325252ull;
        for (size_t e = 0; e < W.size(); e++) {
            x ^= x << 13;
            x ^= x >> 7;
            x ^= x << 17;
            W[e] = (double)(long long)x * 0x1p-63 * (1.0 + (double)(e / ld) / n);   // the last rows win
        }
        const size_t nw = (size_t)2 * CTAS + (size_t)2 * (CTAS + 1) * NB;
        const int starts[] = {0, n / 2 / NB * NB, (n - 1) / NB * NB};
        for (int k0 : starts)
            for (int R : {64, 100}) {
                std::vector<double> out[2];
                std::vector<int> piv[2];
                for (int form = 0; form < 2; form++) {
                    double *dW, *rowbuf;
                    int *ipiv;
                    LuWord *words;
                    State *st;
                    if (!ok(cudaMalloc(&dW, W.size() * 8), "malloc") || !ok(cudaMalloc(&rowbuf, (size_t)(n + R) * NB * 8), "malloc") ||
                        !ok(cudaMalloc(&ipiv, n * 4), "malloc") || !ok(cudaMalloc(&words, nw * sizeof(LuWord)), "malloc") ||
                        !ok(cudaMalloc(&st, sizeof(State)), "malloc"))
                        return 2;
                    cudaMemcpy(dW, W.data(), W.size() * 8, cudaMemcpyHostToDevice);
                    cudaMemset(ipiv, 0, n * 4);
                    cudaMemset(words, 0, nw * sizeof(LuWord));
                    cudaMemset(st, 0, sizeof(State));
                    LuArgs a{};
                    a.n = n;
                    a.W = dW;
                    a.ld = ld;
                    a.ipiv = ipiv;
                    a.slots = words;
                    a.xrows = words + 2 * CTAS;
                    a.rowbuf = rowbuf;
                    a.st = st;
                    int kk0 = k0, kk1 = k0 + NB < n ? k0 + NB : n, RR = R;
                    void *args[] = {&a, &kk0, &kk1, &RR};
                    if (!ok(cudaLaunchCooperativeKernel(form ? K.factor_global : K.factor, dim3((n - k0 + R - 1) / R),
                                                        dim3(K.factor_block), args, lu_factor_smem(R, form == 0), 0),
                            "launch") ||
                        !ok(cudaDeviceSynchronize(), "run"))
                        return 2;
                    State hs;
                    out[form].resize(W.size());
                    piv[form].resize(n);
                    cudaMemcpy(&hs, st, sizeof(State), cudaMemcpyDeviceToHost);
                    cudaMemcpy(out[form].data(), dW, W.size() * 8, cudaMemcpyDeviceToHost);
                    cudaMemcpy(piv[form].data(), ipiv, n * 4, cudaMemcpyDeviceToHost);
                    if (hs.err || hs.status) bad++;
                    cudaFree(dW);
                    cudaFree(rowbuf);
                    cudaFree(ipiv);
                    cudaFree(words);
                    cudaFree(st);
                }
                runs++;
                if (std::memcmp(out[0].data(), out[1].data(), W.size() * 8) || piv[0] != piv[1] ||
                    (n - k0 > 1 && !std::memcmp(out[0].data(), W.data(), W.size() * 8))) {
                    std::printf("n %d, panel at %d, %d rows a CTA: different\n", n, k0, R);
                    bad++;
                }
            }
    }
    std::printf("runs %d mismatches %d\n", runs, bad);
    return bad != 0;
}
