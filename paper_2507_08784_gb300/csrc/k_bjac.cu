// The paper-exact refresh (Eq. SVD-P1 with the full m' x m' basis) above m' = 1024: the
// eigen-decomposition H = Mbar Mbar^T = U diag(lambda) U^T by parallel block-cyclic two-sided
// Jacobi.
//
// H (n x n, n a multiple of 128) is cut into m = n / 64 blocks of 64 indices.  A round pairs the
// blocks by the circle method of a round-robin tournament (block 0 fixed, the others rotating one
// slot per round, so that every two blocks meet once in m - 1 rounds, one sweep), and the pairs
// of a round are stored next to each other: pair k holds rows and columns 128 k .. 128 k + 127.
// A round
//   1. takes each pair's 128 x 128 diagonal block S_k and forms J_k, one sweep of parallel scalar
//      Jacobi over the pair's two blocks started from the identity (bjac_pair_kernel, k_pair.cuh; in
//      a sweep's first round over the indices inside each block too), so that J_k stays close to
//      the identity and no reordering inside the pair is needed;
//   2. applies the block-diagonal J = diag(J_k) on the tensor cores (tc_kernel<BjacMul>, k_tc.cu,
//      split TF32: A B + A_lo B + A B_lo): T^T = (H J)^T, then H <- T^T J = J^T H J and V <- V J, the
//      last two writing every 64-block straight to its place in the next round's storage order.
//      H is symmetric: after the first round only its 128 x 128 blocks on and below the diagonal
//      hold values;
// and a sweep ends with the off-diagonal norm, checked on the host against tol^2 of the total.
// V starts as the identity, so its columns follow H's storage order; at the end V is orthogonalised
// once more in fp32, and diag(H) and V are sorted by descending eigenvalue with the sign rule of the
// small solvers (sort_group).
//
// Every product keeps its output's TF32 low part beside it (H_lo, T^T_lo, V_lo; J_lo from the
// pair sweep), so each operand enters the MMAs as hi + lo.
#include "k_pair.cuh"

namespace glr {

namespace {

// Per matrix, per CTA: the squared diagonal and off-diagonal sums of H (part[2 (mat G + cta)]), from its
// 128 x 128 blocks on and below the diagonal.
__global__ void __launch_bounds__(256) bjac_norms_kernel(const __grid_constant__ BjacGroup g, float* part) {
    chain_begin();
    const BjacMat& M = g.mat[blockIdx.y];
    const int n = M.n;
    float d = 0.f, o = 0.f;
    for (int r = blockIdx.x; r < n; r += gridDim.x) {
        const float* row = M.H + (int64_t)r * n;
        const int c0 = r & ~127;
        for (int c = threadIdx.x; c < c0 + 128; c += 256) {
            const float v = row[c];
            if (c == r) d += v * v;
            else o += (c < c0 ? 2.f : 1.f) * (v * v);
        }
    }
    __shared__ float red[2][8];
#pragma unroll
    for (int s = 16; s > 0; s >>= 1) {
        d += __shfl_xor_sync(0xffffffffu, d, s);
        o += __shfl_xor_sync(0xffffffffu, o, s);
    }
    if ((threadIdx.x & 31) == 0) { red[0][threadIdx.x >> 5] = d; red[1][threadIdx.x >> 5] = o; }
    __syncthreads();
    if (threadIdx.x == 0) {
        float sd = 0.f, so = 0.f;
        for (int w = 0; w < 8; ++w) { sd += red[0][w]; so += red[1][w]; }
        float* out = part + 2 * ((int64_t)blockIdx.y * gridDim.x + blockIdx.x);
        out[0] = sd; out[1] = so;
    }
}

// J_k of the 128 x 128 diagonal pair block S_k of H, from W = I (k_pair.cuh): the 64 cross rounds
// of the pair's two blocks, or with `full` (a sweep's first round, so that every two indices of a
// block meet once a sweep too) all 127 rounds.  J_k^T is written row-major with its TF32 low part.
// On the 2048 x 2048 problem the cross-only rounds take as many sweeps as 127 rounds in each pairing
// do or one or two more, at half the work of a round.
// Where the pairs leave most SMs idle (n = 2048: 16 pairs), four CTAs share one, each with a quarter
// of W's rows (WR = 2): the same bits.
template <int WR>
__global__ void __launch_bounds__(pair::PTHREADS, 1) bjac_pair_kernel(const __grid_constant__ BjacGroup g, int full) {
    chain_begin();
    using namespace pair;
    constexpr int PARTS = 8 / WR, ROWS = 16 * WR;
    extern __shared__ __align__(16) float psm[];
    const int tile = blockIdx.x / PARTS, w0 = blockIdx.x % PARTS * ROWS;
    int mi = 0;
    while (mi + 1 < g.nmat && g.mat[mi + 1].tile0p <= tile) ++mi;
    const BjacMat& M = g.mat[mi];
    const int n = M.n, k = tile - M.tile0p;
    const float* W = sweep<WR>(M.H + (int64_t)(PN * k) * (n + 1), n, w0, full, psm,
                               [](const float* p) { return *reinterpret_cast<const float2*>(p); });
    // J_k^T (row c = column c of W) and its TF32 low part: the rotations' MMA operands
    float* Jt = M.J + (int64_t)k * PN * PN + w0;
    float* Jl = M.Jlo + (int64_t)k * PN * PN + w0;
    for (int e = threadIdx.x; e < PN * ROWS; e += PTHREADS) {
        const int c = e / ROWS, r = e % ROWS;
        const float v = W[r * PLD + c];
        Jt[c * PN + r] = v;
        Jl[c * PN + r] = v - __uint_as_float(__float_as_uint(v) & 0xffffe000u);
    }
}

// Before the first round, per problem: H's TF32 low part, V = I and V's low part 0.
__global__ void bjac_prep_kernel(const __grid_constant__ BjacPrepGroup g) {
    const BjacPrep& P = g.mat[blockIdx.y];
    const int n = P.n;
    for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < (int64_t)n * n; q += (int64_t)gridDim.x * blockDim.x) {
        const int r = (int)(q / n), c = (int)(q % n);
        const float h = P.H[q];
        P.Hlo[q] = h - __uint_as_float(__float_as_uint(h) & 0xffffe000u);
        P.V[q] = r == c ? 1.f : 0.f;
        P.Vlo[q] = 0.f;
    }
}

__global__ void count_flag_kernel(int* flag, int v) { atomicAdd(flag, v); }

__global__ void bjac_diag_kernel(const float* H, int n, float* evals) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) evals[i] = H[(int64_t)i * n + i];
}
__global__ void add_diagonal_kernel(float* A, int n, float v) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) A[(int64_t)i * n + i] += v;
}

}  // namespace

cudaError_t bjac_pairs(BjacGroup& g, int full, cudaStream_t st) {
    if (g.nmat <= 0) return cudaSuccess;
    int tiles = 0;
    for (int i = 0; i < g.nmat; ++i) {
        BjacMat& M = g.mat[i];
        if (M.n < 256 || M.n % 128 || M.n > kBjacMaxN) return cudaErrorInvalidValue;
        M.tile0p = tiles;
        tiles += M.n / 128;
    }
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    const bool parts = 4 * tiles <= sms;
    // per device: set on every call (cheap next to the launch)
    e = parts ? cudaFuncSetAttribute(bjac_pair_kernel<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)pair::kSmem)
              : cudaFuncSetAttribute(bjac_pair_kernel<8>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)pair::kSmem);
    if (e != cudaSuccess) return e;
    if (parts) launch_chain(bjac_pair_kernel<2>, 4 * tiles, pair::PTHREADS, pair::kSmem, st, g, full);
    else launch_chain(bjac_pair_kernel<8>, tiles, pair::PTHREADS, pair::kSmem, st, g, full);
    return cudaGetLastError();
}

cudaError_t bjac_norms(const BjacGroup& g, float* part, cudaStream_t st) {
    if (g.nmat <= 0) return cudaSuccess;
    launch_chain(bjac_norms_kernel, dim3(kBjacNormCtas, g.nmat), 256, 0, st, g, part);
    return cudaGetLastError();
}

cudaError_t bjac_prep(const BjacPrepGroup& g, cudaStream_t st) {
    if (g.nmat <= 0) return cudaSuccess;
    bjac_prep_kernel<<<dim3(64, g.nmat), 256, 0, st>>>(g);
    return cudaGetLastError();
}

cudaError_t count_flag(int* flag, int v, cudaStream_t st) {
    count_flag_kernel<<<1, 1, 0, st>>>(flag, v);
    return cudaGetLastError();
}

cudaError_t add_diagonal(float* A, int n, float v, cudaStream_t st) {
    add_diagonal_kernel<<<(n + 255) / 256, 256, 0, st>>>(A, n, v);
    return cudaGetLastError();
}

cudaError_t bjac_diag(const float* H, int n, float* evals, cudaStream_t st) {
    bjac_diag_kernel<<<(n + 255) / 256, 256, 0, st>>>(H, n, evals);
    return cudaGetLastError();
}

}  // namespace glr
