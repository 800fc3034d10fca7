// FP64 BP1.0 mass matvec (Algorithm 3):
//   Mq = (I^T x I^T x I^T) wJ (I x I x I) q   per element,
// interpolation GLL -> Gauss (Algorithm 1) and projection back (Algorithm 2)
// as three one-dimensional contractions each.  See bp30_fx.cuh for the
// arithmetic.  Measured at N = 7 on 32^3 elements: 330 us against 1505 us of
// the FP64 lines; N = 12 on 17^3: 307 against 1404.
#define FEM_FX_TABLES
#include "bp30_fx.cuh"

namespace fem {
namespace {

// Threads a block aims for, and resident blocks per SM that the register
// allocation must allow, from sweeps of 128 and 256 threads and 1 to 8 blocks
// on GB300 (N = 7: 320 us with 4 blocks of 256 threads, 395 with 2, 591 with
// 1; N = 12: 420 with 3, 608 with 1).
__host__ __device__ constexpr int fx1_threads(int N) { return (N == 5 || N == 7 || N >= 11) ? 256 : 128; }
__host__ __device__ constexpr int fx1_min_blocks(int N) {
    constexpr int t[16] = {1, 8, 8, 8, 8, 4, 8, 4, 6, 6, 4, 3, 3, 3, 2, 2};
    return t[N];
}

// TARGET: the block's thread target (32 for meshes too small to give every
// SM two blocks, where one element per block spreads the work)
template <int N, int TARGET>
struct Fx1Cfg : Fx1Layout<N, pick_epb(N + 2, Fx1Layout<N, 1>::per * 8, TARGET)> {};

template <int N, int TARGET>
__global__ void __launch_bounds__(Fx1Cfg<N, TARGET>::threads, fx1_min_blocks(N))
bp1_fx_kernel(int64_t E, const double *__restrict__ wJ, const double *__restrict__ q, double *__restrict__ Mq) {
    using C = Fx1Cfg<N, TARGET>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int64_t e0 = (int64_t)blockIdx.x * C::EPB;
    const int nel = (int)((E - e0) < C::EPB ? (E - e0) : C::EPB);
    bp1_fx_block<N, C::EPB>(smem_raw, e0, nel, wJ, q, Mq);
}

template <int N>
struct Fx1Launch {
    static cudaError_t run(int64_t E, const double *wJ, const double *q, double *Mq, cudaStream_t s) {
        using C = Fx1Cfg<N, fx1_threads(N)>;
        using Cs = Fx1Cfg<N, 32>;
        const int64_t blocks = (E + C::EPB - 1) / C::EPB;
        if (blocks < 2 * 152)  // small mesh: one element (or a few) per block
            bp1_fx_kernel<N, 32><<<(unsigned)((E + Cs::EPB - 1) / Cs::EPB), Cs::threads, Cs::smem, s>>>(E, wJ, q, Mq);
        else
            bp1_fx_kernel<N, fx1_threads(N)><<<(unsigned)blocks, C::threads, C::smem, s>>>(E, wJ, q, Mq);
        return cudaGetLastError();
    }
};

template <int N>
struct Fx1Prepare {
    static cudaError_t run() {
        cudaError_t e = cudaFuncSetAttribute(bp1_fx_kernel<N, fx1_threads(N)>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             Fx1Cfg<N, fx1_threads(N)>::smem);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(bp1_fx_kernel<N, 32>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     Fx1Cfg<N, 32>::smem);
        return e;
    }
};

FEM_DEFINE_FX_UPLOAD(upload_fx_bp1_tu)

// Layout check of degree N: the boxes of q and of the twice interpolated field
// in one buffer (one at a time), that of the once interpolated field behind it.
template <int N>
int fx1_layout_violations_of() {
    using C = Fx1Cfg<N, fx1_threads(N)>;
    constexpr int n = N + 1, m = N + 2;
    static_assert(C::off_stats >= C::EPB * C::per * 8 && C::off_b >= C::off_stats + C::EPB * kFx30Stats * 4 &&
                      C::smem >= C::off_b + 8,
                  "regions of the block overlap");
    return box_layout_violations<typename C::B0, n, n, n>(C::SA) + box_layout_violations<typename C::B2, m, m, n>(C::SA) +
           box_layout_violations<typename C::B1, m, n, n>(C::per - C::SA);
}
template <int... Ns>
int fx1_layout_violations_all(std::integer_sequence<int, Ns...>) {
    return (0 + ... + fx1_layout_violations_of<Ns + 1>());
}

}  // namespace

cudaError_t launch_bp1(const fem_basis *b, int64_t E, const double *wJ, const double *q, double *Mq, cudaStream_t s) {
    return dispatch_degree<Fx1Launch>(b->host.N, E, wJ, q, Mq, s);
}

int layout_violations_fx1() { return fx1_layout_violations_all(std::make_integer_sequence<int, kMaxN>{}); }

cudaError_t prepare_bp1(int N, const double *fold_table) {
    cudaError_t e = upload_fx_bp1_tu(fold_table);
    if (e != cudaSuccess) return e;
    return dispatch_degree<Fx1Prepare>(N);
}

}  // namespace fem
