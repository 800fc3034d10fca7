// FP64 BP3.5 kernels (Algorithm 4): the operator and its variant fused with
// the PCG direction update p <- z + beta p and the p . Ap reduction.  See
// bp35_fx.cuh for the arithmetic.
#define FEM_FX_TABLES
#include "bp35_fx.cuh"

namespace fem {
namespace {

// Threads a block aims for, and resident blocks per SM that the register
// allocation must allow, from sweeps of 64 to 320 threads and 2 to 16 blocks
// on GB300 (32^3 elements up to N = 7, the same number of nodes above).  The
// kernel alternates between phases that wait for shared or global memory and
// phases bound by the integer multiply-adds, so many small blocks out of step
// beat few large ones (N = 7: 321 us with 8 blocks of 128 threads, 428 with 2
// of 256), down to where the registers would spill (N = 13: 559 us with 3
// blocks of 224, 634 with 5).  256 threads where 128 would leave a warp
// half-empty (n^2 = 36, 49, 81, 100; N = 5 on 40^3 elements: 315 us against 326,
// and 1.17 times more for elements that stay in FP64).
__host__ __device__ constexpr int fx35_threads(int N) { return (N == 5 || N == 6 || N == 8 || N == 9) ? 256 : 128; }
__host__ __device__ constexpr int fx35_min_blocks(int N) {
    constexpr int t[16] = {1, 8, 8, 8, 8, 4, 4, 8, 3, 4, 5, 4, 3, 4, 3, 3};
    return t[N];
}

template <int N>
struct Fx35Cfg : Fx35Layout<N, pick_epb(N + 1, 3 * Box<N + 1, N + 1, N + 1>::size * 8, fx35_threads(N))> {};

template <int N, bool PCG>
__global__ void __launch_bounds__(Fx35Cfg<N>::threads, fx35_min_blocks(N))
bp35_fx_kernel(int64_t E, const double *__restrict__ G, double lambda, const double *__restrict__ q,
               double *__restrict__ Aq, const double *__restrict__ z, double *p, const double *__restrict__ beta,
               double *__restrict__ partials) {
    using C = Fx35Cfg<N>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int64_t e0 = (int64_t)blockIdx.x * C::EPB;
    const int nel = (int)((E - e0) < C::EPB ? (E - e0) : C::EPB);
    bp35_fx_block<N, C::EPB, PCG>(smem_raw, e0, nel, G, lambda, q, Aq, z, p, beta,
                                  PCG ? partials + blockIdx.x : nullptr);
}

template <int N>
struct Fx35Launch {
    static cudaError_t run(int64_t E, const double *G, double lambda, const double *q, double *Aq, const double *z,
                           double *p, const double *beta, double *partials, cudaStream_t s) {
        using C = Fx35Cfg<N>;
        const unsigned blocks = (unsigned)((E + C::EPB - 1) / C::EPB);
        if (p)
            bp35_fx_kernel<N, true><<<blocks, C::threads, C::smem, s>>>(E, G, lambda, nullptr, Aq, z, p, beta, partials);
        else
            bp35_fx_kernel<N, false><<<blocks, C::threads, C::smem, s>>>(E, G, lambda, q, Aq, nullptr, nullptr,
                                                                          nullptr, nullptr);
        return cudaGetLastError();
    }
};

template <int N>
struct Fx35Blocks {
    static cudaError_t run(int64_t E, int64_t *out) {
        *out = (E + Fx35Cfg<N>::EPB - 1) / Fx35Cfg<N>::EPB;
        return cudaSuccess;
    }
};

template <int N>
struct Fx35Prepare {
    static cudaError_t run() {
        cudaError_t e = cudaFuncSetAttribute(bp35_fx_kernel<N, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             Fx35Cfg<N>::smem);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(bp35_fx_kernel<N, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     Fx35Cfg<N>::smem);
        return e;
    }
};

FEM_DEFINE_FX_UPLOAD(upload_fx_bp35_tu)

}  // namespace

cudaError_t launch_bp35(const fem_basis *b, int64_t E, const double *G, double lambda, const double *q, double *Aq,
                        cudaStream_t s) {
    return dispatch_degree<Fx35Launch>(b->host.N, E, G, lambda, q, Aq, (const double *)nullptr, (double *)nullptr,
                                       (const double *)nullptr, (double *)nullptr, s);
}

cudaError_t launch_bp35_pcg(const fem_basis *b, int64_t E, const double *G, double lambda, const double *z, double *p,
                            const double *beta, double *Ap, double *partials, cudaStream_t s) {
    return dispatch_degree<Fx35Launch>(b->host.N, E, G, lambda, (const double *)nullptr, Ap, z, p, beta, partials, s);
}

int64_t bp35_fx_blocks(int N, int64_t E) {
    int64_t out = 0;
    dispatch_degree<Fx35Blocks>(N, E, &out);
    return out;
}

cudaError_t prepare_bp35_fx(int N, const double *fold_table) {
    cudaError_t e = upload_fx_bp35_tu(fold_table);
    if (e != cudaSuccess) return e;
    return dispatch_degree<Fx35Prepare>(N);
}

}  // namespace fem
