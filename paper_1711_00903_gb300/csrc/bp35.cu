// FP32 BP3.5 kernels (Algorithm 4), the inner operator of the mixed-precision
// solver:
//   Aq = D_r^T Rr + D_s^T Rs + D_t^T Rt + lambda wJ q,
//   [Rr Rs Rt] = G [q_r q_s q_t],  q_r = (D x I x I) q, ...
// and the variant fused with the PCG direction update p <- z + beta p and the
// p . Ap reduction.  The FP64 operator is in bp35_fx.cu.
//
// GB300 design (bp35_body.cuh), bound by HBM:
//   * every one-dimensional contraction is one thread applying the even-odd
//     folded D or D^T to a whole line (eo.cuh), operator entries as
//     constant-bank operands;
//   * q^e and the r and s partial results of the element live in shared
//     memory (padded boxes), the t-direction work of a thread's (i, j)
//     column stays in registers, four barriers per element;
//   * several elements per block (n^2 threads each), coalesced loads of q
//     and of each geometric-factor plane, coalesced stores;
//   * where it measured faster, a persistent TMA stream (bp35_stream.cuh).
#include "bp35_stream.cuh"

namespace fem {
namespace {

template <typename T, int N, bool PCG>
__device__ __forceinline__ void bp35_entry(int64_t E, const T *__restrict__ G, double lambda, const T *__restrict__ q,
                                           T *__restrict__ Aq, const T *__restrict__ z, T *__restrict__ p,
                                           const double *__restrict__ beta, double *__restrict__ partials) {
    using C = Bp35Cfg<T, N>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int64_t e0 = (int64_t)blockIdx.x * C::EPB;
    const int nel = (int)((E - e0) < C::EPB ? (E - e0) : C::EPB);
    bp35_block<T, N, C::EPB, PCG>(smem_raw, e0, nel, G, lambda, q, Aq, z, p, beta,
                                  PCG ? partials + blockIdx.x : nullptr);
}

template <typename T, int N, bool PCG>
__global__ void __launch_bounds__(Bp35Cfg<T, N>::threads)
bp35_kernel(int64_t E, const T *__restrict__ G, double lambda, const T *__restrict__ q, T *__restrict__ Aq,
            const T *__restrict__ z, T *__restrict__ p, const double *__restrict__ beta,
            double *__restrict__ partials) {
    bp35_entry<T, N, PCG>(E, G, lambda, q, Aq, z, p, beta, partials);
}

template <typename T, int N, bool PCG>
__global__ void __launch_bounds__(Bp35Cfg<T, N>::threads, bp35_min_blocks<T, N>())
bp35_kernel_capped(int64_t E, const T *__restrict__ G, double lambda, const T *__restrict__ q, T *__restrict__ Aq,
                   const T *__restrict__ z, T *__restrict__ p, const double *__restrict__ beta,
                   double *__restrict__ partials) {
    bp35_entry<T, N, PCG>(E, G, lambda, q, Aq, z, p, beta, partials);
}

template <typename T, int N, bool PCG>
constexpr auto bp35_fn() {
    if constexpr (bp35_min_blocks<T, N>() > 0)
        return &bp35_kernel_capped<T, N, PCG>;
    else
        return &bp35_kernel<T, N, PCG>;
}

template <int N>
struct Bp35F32Launch {
    static cudaError_t run(int64_t E, const float *G, double lambda, const float *q, float *Aq,
                           cudaStream_t s) {
        if constexpr (bp35_streamed<N, false, float>()) {
            return launch_stream35<N, false>(E, G, lambda, q, Aq, nullptr, nullptr, nullptr, nullptr, s);
        } else if constexpr (bp35_streamed1<N, false, float>()) {
            return launch_stream35_1<N, false>(E, G, lambda, q, Aq, nullptr, nullptr, nullptr, nullptr, s);
        } else {
            using C = Bp35Cfg<float, N>;
            const int64_t blocks = (E + C::EPB - 1) / C::EPB;
            bp35_fn<float, N, false>()<<<(unsigned)blocks, C::threads, C::smem, s>>>(
                E, G, lambda, q, Aq, nullptr, nullptr, nullptr, nullptr);
            return cudaGetLastError();
        }
    }
};

template <int N>
struct Bp35PcgF32Launch {
    static cudaError_t run(int64_t E, const float *G, double lambda, const float *z, float *p, const double *beta,
                           float *Ap, double *partials, cudaStream_t s, double *status) {
        if constexpr (bp35_streamed<N, true, float>()) {
            return launch_stream35<N, true>(E, G, lambda, nullptr, Ap, z, p, beta, partials, s, nullptr, status);
        } else if constexpr (bp35_streamed1<N, true, float>()) {
            return launch_stream35_1<N, true>(E, G, lambda, nullptr, Ap, z, p, beta, partials, s, nullptr, status);
        } else {
            using C = Bp35Cfg<float, N>;
            const int64_t blocks = (E + C::EPB - 1) / C::EPB;
            bp35_fn<float, N, true>()<<<(unsigned)blocks, C::threads, C::smem, s>>>(E, G, lambda, nullptr, Ap, z, p,
                                                                                   beta, partials);
            return cudaGetLastError();
        }
    }
};

template <int N>
struct Bp35Blocks {
    static cudaError_t run(int64_t E, int64_t *out) {
        using F = Bp35Cfg<float, N>;
        int64_t b = (E + F::EPB - 1) / F::EPB;
        if constexpr (bp35_streamed<N, true, float>()) {
            using S = Bp35Stream<N, true>;
            b = stream_grid35((E + S::EPS - 1) / S::EPS, S::blocks_per_sm);
        } else if constexpr (bp35_streamed1<N, true, float>()) {
            b = stream_grid35(E, Bp35Stream1<N, true, float>::blocks_per_sm);
        }
        *out = b;
        return cudaSuccess;
    }
};

template <int N>
struct Bp35Prepare {
    template <typename T, bool PCG>
    static cudaError_t one() {
        return cudaFuncSetAttribute(bp35_fn<T, N, PCG>(), cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    Bp35Cfg<T, N>::smem);
    }
    static cudaError_t run() {
        cudaError_t e = one<float, false>();
        if (e == cudaSuccess) e = one<float, true>();
        // the stream kernels keep all operands in shared memory: they ask
        // for the largest carveout
        if constexpr (bp35_two_stage_fits(N))
            if (e == cudaSuccess) e = prepare_stream35<N, float>();
        if (e == cudaSuccess) e = prepare_stream35_1<N, float>();
        return e;
    }
};

FEM_DEFINE_FOLD_UPLOAD(upload_fold_bp35_tu)

}  // namespace

FEM_DEFINE_WAIT_COUNTER(wait_timeouts_bp35)

cudaError_t launch_bp35_f32(const fem_basis *b, int64_t E, const float *G, double lambda, const float *q,
                            float *Aq, cudaStream_t s) {
    return dispatch_degree<Bp35F32Launch>(b->host.N, E, G, lambda, q, Aq, s);
}

cudaError_t launch_bp35_pcg_f32(const fem_basis *b, int64_t E, const float *G, double lambda, const float *z,
                                float *p, const double *beta, float *Ap, double *partials, cudaStream_t s,
                                double *status) {
    return dispatch_degree<Bp35PcgF32Launch>(b->host.N, E, G, lambda, z, p, beta, Ap, partials, s, status);
}

int64_t bp35_blocks(int N, int64_t E, bool f32) {
    if (!f32) return bp35_fx_blocks(N, E);
    int64_t out = 0;
    dispatch_degree<Bp35Blocks>(N, E, &out);
    return out;
}

cudaError_t prepare_bp35(int N, const double *fold_table) {
    cudaError_t e = upload_fold_bp35_tu(fold_table);
    if (e != cudaSuccess) return e;
    e = dispatch_degree<Bp35Prepare>(N);
    return e == cudaSuccess ? prepare_bp35_fx(N, fold_table) : e;
}

namespace {
// Layout check of degree N: the n^3 box of the FP32 stream kernels and that of
// the FP64 (Fx35Layout) and block kernels, each point mapped to a distinct word inside
// the box's share of the per-element buffer; the swizzled boxes (N = 7,
// 15) also serve every direction's warp line accesses without a bank
// conflict.
template <int N>
int bp35_layout_violations_of() {
    constexpr int n = N + 1;
    using T = typename Bp35Layout<float, N, 1, true>::B;
    using P = typename Bp35Layout<double, N, 1>::B;
    int bad = box_layout_violations<T, n, n, n>(T::size) + box_layout_violations<P, n, n, n>(P::size);
    if constexpr (N == 7 || N == 15) bad += box_line_conflicts<T, n>();
    return bad;
}
template <int... Ns>
int bp35_layout_violations_all(std::integer_sequence<int, Ns...>) {
    return (0 + ... + bp35_layout_violations_of<Ns + 1>());
}
}  // namespace

int layout_violations_bp35() { return bp35_layout_violations_all(std::make_integer_sequence<int, kMaxN>{}); }

}  // namespace fem
