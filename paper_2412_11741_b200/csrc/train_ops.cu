// One training step of the offline dictionary ("NeuralDict", Algorithm 1, procedure
// TrainNeurDict; the MSE loss, the diversity loss L_div = ||I - W^T W||_F^2 / N^2, the complete
// loss L = L_MSE + beta * L_div and ReNorm).  The sparse codes of the batch are computed by
// the matching-pursuit encoder before these kernels run and are held fixed while the loss
// is differentiated (the alternating scheme of dictionary learning), so with
// e_x = x - W r(x):
//
//   dL_MSE / d d_n = -2 * sum over (x, g) with i_g(x) = n of  c_g(x) * e_x
//   dL_div / d d_n = (4 / N^2) * sum_j (G[n][j] - delta_nj) * d_j,      G = D D^T
//
//   mse_grad_kernel   one warp per row: restores x^ from the codes, forms e = x - x^, adds
//                     ||e||^2 to the loss (fp64 atomic) and scatters -2 c_g e into the
//                     gradient rows of the s selected atoms (fp32 atomic adds).
//   diversity term    the N x N product is not formed: (D D^T - I_N) D = D (D^T D - I_d) and
//                     ||D D^T - I_N||^2 = ||C||^2 - 2 tr C + N with C = D^T D, a d x d matrix.
//                     gram_kernel sums C in fp64 (the products of fp32 values are exact there, and the
//                     differences that the loss and near-orthonormal atoms leave keep 1e-16 of what they
//                     came from), 2 N d^2 operations instead of 2 N^2 d.  The two N x N products on the tensor
//                     cores (split bf16 operands, 2^-16 relative) instead: 2267 us for a step of 65536 rows at N = 8192,
//                     s = 8; so 2095.
//   update_kernel     d_n <- ReNorm(d_n - lr * (g_mse + beta * g_div)), g_div = (4 / N^2) d_n (C - I) on
//                     the way, and L_div.
#include "common.cuh"

namespace csr {
namespace {

__device__ __forceinline__ float load_x(const void* X, int x_dtype, int64_t off) { return load_elem(X, x_dtype, off); }

// A lane's channels of a row, PER = D_ / 32 next to one another.
template <int PER>
struct Lane;
template <>
struct Lane<4> {
    using V = float4;
    static __device__ __forceinline__ void get(const V& v, float (&a)[4]) { a[0] = v.x, a[1] = v.y, a[2] = v.z, a[3] = v.w; }
    static __device__ __forceinline__ V make(const float (&a)[4], float c) { return make_float4(c * a[0], c * a[1], c * a[2], c * a[3]); }
};
template <>
struct Lane<2> {
    using V = float2;
    static __device__ __forceinline__ void get(const V& v, float (&a)[2]) { a[0] = v.x, a[1] = v.y; }
    static __device__ __forceinline__ V make(const float (&a)[2], float c) { return make_float2(c * a[0], c * a[1]); }
};

// Bound by the L2's atomic adds: s * D_ * 4 bytes of them per row.  A lane's channels go in one vector
// add (the same values as scalar adds, in fewer requests); the row's codes are read once, one per
// lane, and the gathers of four atoms are in flight together.  A whole step of 65536 rows, N = 8192,
// s = 8, d = 128 in the exact mode: 3060 us with scalar adds, 2993 us so.
template <int D_>
__global__ void __launch_bounds__(256)
mse_grad_kernel(const float* __restrict__ D, int N, const void* __restrict__ X, int x_dtype, int64_t M, int s,
                const uint16_t* __restrict__ idx, const float* __restrict__ coef, float* __restrict__ grad,
                double* __restrict__ losses) {
    constexpr int PER = D_ / 32;
    using V = typename Lane<PER>::V;
    const int lane = threadIdx.x & 31;
    const int64_t warp0 = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const int64_t nwarps = (int64_t)gridDim.x * (blockDim.x >> 5);
    double local = 0.0;
    for (int64_t m = warp0; m < M; m += nwarps) {
        float e[PER];
#pragma unroll
        for (int k = 0; k < PER; ++k) e[k] = load_x(X, x_dtype, m * D_ + lane * PER + k);
        // up to 64 entries, two per lane
        int my_i[2];
        float my_c[2];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int g = u * 32 + lane;
            my_i[u] = g < s ? min(static_cast<int>(idx[m * s + g]), N - 1) : 0;
            my_c[u] = g < s ? coef[m * s + g] : 0.f;
        }
#pragma unroll 4
        for (int g = 0; g < s; ++g) {                     // e = x - sum_g c_g d_{i_g}, stored order
            const int i = __shfl_sync(0xffffffffu, g < 32 ? my_i[0] : my_i[1], g & 31);
            const float c = __shfl_sync(0xffffffffu, g < 32 ? my_c[0] : my_c[1], g & 31);
            float d[PER];
            Lane<PER>::get(__ldg(reinterpret_cast<const V*>(D + (int64_t)i * D_) + lane), d);
#pragma unroll
            for (int k = 0; k < PER; ++k) e[k] = fmaf(-c, d[k], e[k]);
        }
        float ss = 0.f;
#pragma unroll
        for (int k = 0; k < PER; ++k) ss = fmaf(e[k], e[k], ss);
        for (int o = 16; o; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
        local += (double)ss;
#pragma unroll 4
        for (int g = 0; g < s; ++g) {
            const int i = __shfl_sync(0xffffffffu, g < 32 ? my_i[0] : my_i[1], g & 31);
            const float c2 = -2.f * __shfl_sync(0xffffffffu, g < 32 ? my_c[0] : my_c[1], g & 31);
            atomicAdd(reinterpret_cast<V*>(grad + (int64_t)i * D_) + lane, Lane<PER>::make(e, c2));
        }
    }
    if (lane == 0 && local != 0.0) atomicAdd(&losses[0], local);
}

// C += D^T D over this CTA's atoms, all of C in registers: a thread has D_ / 16 x D_ / 16 of its elements (channels
// 2 (16 k + ty) and the next of the rows, the same with tx of the columns: a warp reads shared memory without
// conflicts).  Bound by fp64 FMA issue, half a warp a cycle and scheduler; the atoms are widened once, on their way into
// shared memory (a conversion takes as long as four of the FMAs).
constexpr int GRAM_ATOMS = 32;                            // staged at a time
template <int D_>
__global__ void __launch_bounds__(256)
gram_kernel(const float* __restrict__ D, int N, double* __restrict__ C) {
    constexpr int P = D_ / 32;                            // pairs of rows (columns) per thread
    __shared__ alignas(16) double A[GRAM_ATOMS][D_];
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    const int n0 = static_cast<int>(static_cast<int64_t>(N) * blockIdx.x / gridDim.x);
    const int n1 = static_cast<int>(static_cast<int64_t>(N) * (blockIdx.x + 1) / gridDim.x);
    double c[2 * P][2 * P];
#pragma unroll
    for (int i = 0; i < 2 * P; ++i)
#pragma unroll
        for (int j = 0; j < 2 * P; ++j) c[i][j] = 0.0;
    for (int b = n0; b < n1; b += GRAM_ATOMS) {
        const int rows = min(GRAM_ATOMS, n1 - b);
        __syncthreads();
        for (int f = threadIdx.x; f < rows * (D_ / 4); f += 256) {
            const float4 v = __ldg(reinterpret_cast<const float4*>(D + static_cast<int64_t>(b) * D_) + f);
            double2* dst = reinterpret_cast<double2*>(&A[0][0]) + 2 * f;
            dst[0] = make_double2(v.x, v.y);
            dst[1] = make_double2(v.z, v.w);
        }
        __syncthreads();
#pragma unroll 1
        for (int r = 0; r < rows; ++r) {
            double x[2 * P], y[2 * P];
#pragma unroll
            for (int k = 0; k < P; ++k) {
                const double2 u = *reinterpret_cast<const double2*>(&A[r][2 * (16 * k + ty)]);
                const double2 v = *reinterpret_cast<const double2*>(&A[r][2 * (16 * k + tx)]);
                x[2 * k] = u.x, x[2 * k + 1] = u.y;
                y[2 * k] = v.x, y[2 * k + 1] = v.y;
            }
#pragma unroll
            for (int i = 0; i < 2 * P; ++i)
#pragma unroll
                for (int j = 0; j < 2 * P; ++j) c[i][j] = fma(x[i], y[j], c[i][j]);
        }
    }
#pragma unroll
    for (int i = 0; i < 2 * P; ++i)
#pragma unroll
        for (int j = 0; j < 2 * P; ++j)
            atomicAdd(C + (2 * (16 * (i / 2) + ty) + i % 2) * D_ + 2 * (16 * (j / 2) + tx) + j % 2, c[i][j]);
}

// 32 atoms per CTA, a warp has four of them whole (lane: D_ / 32 channels).  C - I in fp32 (rounded from fp64) and the
// atoms in shared memory.  The first CTA takes the loss from C.
constexpr int UPD_ATOMS = 32;
template <int D_>
constexpr size_t update_smem() {
    return (static_cast<size_t>(D_) * D_ + UPD_ATOMS * D_) * sizeof(float);
}
template <int D_>
__global__ void __launch_bounds__(256)
update_kernel(float* __restrict__ D, int N, const float* __restrict__ grad_mse, const double* __restrict__ C, double* __restrict__ losses,
              float lr, float beta) {
    constexpr int PER = D_ / 32;
    using V = typename Lane<PER>::V;
    extern __shared__ __align__(16) float upd_smem[];
    float* E = upd_smem;                                  // [D_][D_]: C - I
    float* W = upd_smem + D_ * D_;                        // [UPD_ATOMS][D_]
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int n0 = blockIdx.x * UPD_ATOMS;
#pragma unroll 4
    for (int f = threadIdx.x; f < D_ * D_ / 2; f += 256) {
        const double2 v = __ldg(reinterpret_cast<const double2*>(C) + f);
        const int i = 2 * f / D_, j = 2 * f % D_;
        reinterpret_cast<float2*>(E)[f] =
            make_float2(static_cast<float>(v.x - (i == j ? 1.0 : 0.0)), static_cast<float>(v.y - (i == j + 1 ? 1.0 : 0.0)));
    }
    for (int f = threadIdx.x; f < UPD_ATOMS * D_ / 4; f += 256) {
        const int n = n0 + f / (D_ / 4);
        const float4 v = n < N ? *(reinterpret_cast<const float4*>(D + static_cast<int64_t>(n0) * D_) + f) : make_float4(0.f, 0.f, 0.f, 0.f);
        reinterpret_cast<float4*>(W)[f] = v;
    }
    if (blockIdx.x == 0) {                                // L_div = (||C||^2 - 2 tr C + N) / N^2
        double sum = 0.0;
        for (int f = threadIdx.x; f < D_ * D_; f += 256) {
            const double v = __ldg(C + f);
            sum += v * v - (f / D_ == f % D_ ? 2.0 * v : 0.0);
        }
        for (int o = 16; o; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
        __shared__ double part[8];
        if (lane == 0) part[warp] = sum;
        __syncthreads();
        if (threadIdx.x == 0) {
            sum = 0.0;
            for (int w = 0; w < 8; ++w) sum += part[w];
            sum += static_cast<double>(N);
            losses[1] = (sum < 0.0 ? 0.0 : sum) / (static_cast<double>(N) * static_cast<double>(N));
        }
    }
    __syncthreads();
    float g[4][PER];
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int k = 0; k < PER; ++k) g[a][k] = 0.f;
#pragma unroll 2
    for (int i = 0; i < D_; i += 4) {
        float w[4][4], e[4][PER];
#pragma unroll
        for (int a = 0; a < 4; ++a) {
            const float4 v = *reinterpret_cast<const float4*>(W + (4 * warp + a) * D_ + i);
            w[a][0] = v.x, w[a][1] = v.y, w[a][2] = v.z, w[a][3] = v.w;
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) Lane<PER>::get(*(reinterpret_cast<const V*>(E + (i + q) * D_) + lane), e[q]);
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int q = 0; q < 4; ++q)
#pragma unroll
                for (int k = 0; k < PER; ++k) g[a][k] = fmaf(w[a][q], e[q][k], g[a][k]);
    }
    const float scale = 4.0f / (static_cast<float>(N) * static_cast<float>(N));
#pragma unroll
    for (int a = 0; a < 4; ++a) {
        const int n = n0 + 4 * warp + a;
        if (n >= N) continue;                             // (the whole warp)
        float w[PER], gm[PER];
        Lane<PER>::get(*(reinterpret_cast<const V*>(W + (4 * warp + a) * D_) + lane), w);
        Lane<PER>::get(__ldg(reinterpret_cast<const V*>(grad_mse + static_cast<int64_t>(n) * D_) + lane), gm);
        float ss = 0.f;
#pragma unroll
        for (int k = 0; k < PER; ++k) {
            w[k] -= lr * fmaf(beta, scale * g[a][k], gm[k]);
            ss = fmaf(w[k], w[k], ss);
        }
        for (int o = 16; o; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
        const float inv = ss > 0.f ? 1.0f / sqrtf(ss) : 0.f;
        *(reinterpret_cast<V*>(D + static_cast<int64_t>(n) * D_) + lane) = Lane<PER>::make(w, inv);
    }
}

size_t grad_bytes(int N, int d) { return ((size_t)N * d * sizeof(float) + 255) / 256 * 256; }

template <int D_>
int run(const TrainArgs& a) {
    // (the gradient and C lie next to one another: one clear)
    cudaError_t e = cudaMemsetAsync(a.grad_mse, 0, dict_train_scratch_bytes(a.N, D_), a.stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(a.losses, 0, 2 * sizeof(double), a.stream);
    if (e != cudaSuccess) return fail(CSR_ERR_CUDA, "cudaMemsetAsync: %s", cudaGetErrorString(e));
    double* C = reinterpret_cast<double*>(reinterpret_cast<char*>(a.grad_mse) + grad_bytes(a.N, D_));
    if (a.M > 0) {
        int64_t blocks = (a.M + 7) / 8;
        const int64_t cap = (int64_t)sm_count() * 8;
        if (blocks > cap) blocks = cap;
        mse_grad_kernel<D_><<<(int)blocks, 256, 0, a.stream>>>(a.D, a.N, a.X, a.x_dtype, a.M, a.s, a.idx, a.coef,
                                                              a.grad_mse, a.losses);
    }
    const int most = (a.N + 15) / 16;                     // (fewer than 16 atoms are not worth adding up a C for)
    gram_kernel<D_><<<most < sm_count() ? most : sm_count(), 256, 0, a.stream>>>(a.D, a.N, C);
    constexpr size_t smem = update_smem<D_>();
    e = cudaFuncSetAttribute(update_kernel<D_>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return fail(CSR_ERR_CUDA, "cudaFuncSetAttribute: %s", cudaGetErrorString(e));
    update_kernel<D_><<<(a.N + UPD_ATOMS - 1) / UPD_ATOMS, 256, smem, a.stream>>>(a.D, a.N, a.grad_mse, C, a.losses, a.lr, a.beta);
    e = cudaGetLastError();
    if (e != cudaSuccess) return fail(CSR_ERR_CUDA, "dict_train launch: %s", cudaGetErrorString(e));
    return CSR_OK;
}

}  // namespace

size_t dict_train_scratch_bytes(int N, int d) { return grad_bytes(N, d) + (size_t)d * d * sizeof(double); }

int launch_dict_train(const TrainArgs& a) {
    if (a.d == 128) return run<128>(a);
    return run<64>(a);
}

}  // namespace csr
