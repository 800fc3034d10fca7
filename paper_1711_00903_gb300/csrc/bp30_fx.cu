// FP64 BP3.0 kernels (Algorithm 5): the operator, its variant fused with the
// PCG direction update p <- z + beta p and the p . Ap reduction, and BP1.0 and
// BP3.0 of one field in one pass.  See bp30_fx.cuh for the arithmetic.
//
// Measured at N = 7 on 32^3 elements: BP3.0 879 us against 3820 us of the FP64
// lines, which ran at the FP64 pipe's rate; both operators in one pass 1074
// against 4609 us.  HBM is at 28 %: what bounds the kernel is the latency of
// its fourteen phases between barriers together with the integer
// multiply-adds (12 contractions, 27 products at a point).
#define FEM_FX_TABLES
#include "bp30_fx.cuh"

namespace fem {
namespace {

// Threads a block aims for, and resident blocks per SM that the register
// allocation must allow, from sweeps of 128 and 256 threads and 1 to 8 blocks
// on GB300 (32^3 elements up to N = 7, the same number of nodes above): many
// warps up to where the registers spill, as in bp35_fx.cu (N = 7: 849 us with
// 3 blocks of 256 threads, 949 with 2, 1128 with 4 of 128; N = 15: 1391 with
// 1 block of 320, 1741 with 3).  128 threads where 256 would not fill whole
// warps or 128 do (m^2 = 16, 25, 64, 121).
__host__ __device__ constexpr int fx30_threads(int N) { return (N == 2 || N == 3 || N == 6 || N == 9) ? 128 : 256; }
__host__ __device__ constexpr int fx30_min_blocks(int N) {
    constexpr int t[16] = {1, 3, 6, 8, 3, 3, 4, 3, 3, 4, 3, 2, 2, 2, 1, 1};
    return t[N];
}

template <int N>
struct Fx30Cfg : Fx30Layout<N, pick_epb(N + 2, 4 * Box<N + 2, N + 2, N + 2>::size * 8, fx30_threads(N))> {};

template <int N, bool PCG, bool MASS>
__global__ void __launch_bounds__(Fx30Cfg<N>::threads, fx30_min_blocks(N))
bp30_fx_kernel(int64_t E, const double *__restrict__ G, double lambda, const double *__restrict__ q,
               double *__restrict__ Aq, double *__restrict__ Mq, const double *__restrict__ z, double *p,
               const double *__restrict__ beta, double *__restrict__ partials) {
    using C = Fx30Cfg<N>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int64_t e0 = (int64_t)blockIdx.x * C::EPB;
    const int nel = (int)((E - e0) < C::EPB ? (E - e0) : C::EPB);
    bp30_fx_block<N, C::EPB, PCG, MASS>(smem_raw, e0, nel, G, lambda, q, Aq, Mq, z, p, beta,
                                        PCG ? partials + blockIdx.x : nullptr);
}

template <int N>
struct Fx30Launch {
    static cudaError_t run(int64_t E, const double *G, double lambda, const double *q, double *Aq, double *Mq,
                           const double *z, double *p, const double *beta, double *partials, cudaStream_t s) {
        using C = Fx30Cfg<N>;
        const unsigned blocks = (unsigned)((E + C::EPB - 1) / C::EPB);
        if (p)
            bp30_fx_kernel<N, true, false><<<blocks, C::threads, C::smem, s>>>(E, G, lambda, nullptr, Aq, nullptr, z, p,
                                                                               beta, partials);
        else if (Mq)
            bp30_fx_kernel<N, false, true><<<blocks, C::threads, C::smem, s>>>(E, G, lambda, q, Aq, Mq, nullptr, nullptr,
                                                                               nullptr, nullptr);
        else
            bp30_fx_kernel<N, false, false><<<blocks, C::threads, C::smem, s>>>(E, G, lambda, q, Aq, nullptr, nullptr,
                                                                                nullptr, nullptr, nullptr);
        return cudaGetLastError();
    }
};

template <int N>
struct Fx30Blocks {
    static cudaError_t run(int64_t E, int64_t *out) {
        *out = (E + Fx30Cfg<N>::EPB - 1) / Fx30Cfg<N>::EPB;
        return cudaSuccess;
    }
};

template <int N>
struct Fx30Prepare {
    template <bool PCG, bool MASS>
    static cudaError_t one() {
        return cudaFuncSetAttribute(bp30_fx_kernel<N, PCG, MASS>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    Fx30Cfg<N>::smem);
    }
    static cudaError_t run() {
        cudaError_t e = one<false, false>();
        if (e == cudaSuccess) e = one<true, false>();
        if (e == cudaSuccess) e = one<false, true>();
        return e;
    }
};

FEM_DEFINE_FX_UPLOAD(upload_fx_bp30_tu)

// Layout check of degree N: each point of the four boxes on a distinct word of
// its share, the element's line words, statistics and the flags past the boxes.
template <int N>
int fx30_layout_violations_of() {
    using C = Fx30Cfg<N>;
    constexpr int n = N + 1, m = N + 2;
    static_assert(C::off_e >= C::EPB * 4 * C::S * 8 && C::off_s >= C::off_e + C::EPB * 3 * C::mm * 4 &&
                      C::off_b >= C::off_s + C::EPB * kFx30Stats * 4 && C::smem >= C::off_b + 8,
                  "regions of the block overlap");
    return box_layout_violations<typename C::B0, n, n, n>(C::S) + box_layout_violations<typename C::B1, m, n, n>(C::S) +
           box_layout_violations<typename C::B2, m, m, n>(C::S) + box_layout_violations<typename C::B3, m, m, m>(C::S);
}
template <int... Ns>
int fx30_layout_violations_all(std::integer_sequence<int, Ns...>) {
    return (0 + ... + fx30_layout_violations_of<Ns + 1>());
}

}  // namespace

cudaError_t launch_bp30(const fem_basis *b, int64_t E, const double *G, double lambda, const double *q, double *Aq,
                        cudaStream_t s) {
    return dispatch_degree<Fx30Launch>(b->host.N, E, G, lambda, q, Aq, (double *)nullptr, (const double *)nullptr,
                                       (double *)nullptr, (const double *)nullptr, (double *)nullptr, s);
}

cudaError_t launch_bp1_bp30(const fem_basis *b, int64_t E, const double *G, double lambda, const double *q, double *Mq,
                            double *Aq, cudaStream_t s) {
    return dispatch_degree<Fx30Launch>(b->host.N, E, G, lambda, q, Aq, Mq, (const double *)nullptr, (double *)nullptr,
                                       (const double *)nullptr, (double *)nullptr, s);
}

cudaError_t launch_bp30_pcg(const fem_basis *b, int64_t E, const double *G, double lambda, const double *z, double *p,
                            const double *beta, double *Ap, double *partials, cudaStream_t s) {
    return dispatch_degree<Fx30Launch>(b->host.N, E, G, lambda, (const double *)nullptr, Ap, (double *)nullptr, z, p, beta,
                                       partials, s);
}

int64_t bp30_fx_blocks(int N, int64_t E) {
    int64_t out = 0;
    dispatch_degree<Fx30Blocks>(N, E, &out);
    return out;
}

int layout_violations_fx30() { return fx30_layout_violations_all(std::make_integer_sequence<int, kMaxN>{}); }

cudaError_t prepare_bp30_fx(int N, const double *fold_table) {
    cudaError_t e = upload_fx_bp30_tu(fold_table);
    if (e != cudaSuccess) return e;
    return dispatch_degree<Fx30Prepare>(N);
}

}  // namespace fem
