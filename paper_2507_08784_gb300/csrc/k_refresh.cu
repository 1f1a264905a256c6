// Refresh kernels (the Semi-Lazy SVD step of Eq. SVD-P1): the order and sign rule of the
// eigenpairs, the CholeskyQR factors, and the Householder reconstruction of a truncated basis's
// complement (the eigenproblems are in k_eig.cu and k_bjac.cu).
#include "glr_internal.cuh"

namespace glr {

namespace {

// ------------------------------------------------------------------------------------------
// Parallel cyclic two-sided Jacobi (one CTA).  Each round applies n/2 disjoint plane
// rotations chosen by the circle (round-robin) ordering: every rotation angle is computed
// from its own 2 x 2 diagonal block, then H <- J^T H J is applied block-wise (each 2 x 2
// block of H depends only on the rotations of its row pair and column pair, so the update
// is in place) and V <- V J.  Rotation formula: Golub & Van Loan, sym.schur2.
// ------------------------------------------------------------------------------------------
__device__ __forceinline__ int circle(int x, int nm1) { return 1 + ((x % nm1) + nm1) % nm1; }

__global__ void __launch_bounds__(1024) jacobi_kernel(float* Hg, int n, float* Vg, float* evals,
                                                      int* sweeps_out, int* failed, int use_smem, int max_sweeps,
                                                      float tol) {
    extern __shared__ float sm[];
    const int npad = n + (n & 1), half = npad / 2, nm1 = npad - 1;
    const int tid = threadIdx.x, nth = blockDim.x;
    float* H = use_smem ? sm : Hg;
    float* V = use_smem ? sm + (size_t)n * n : Vg;
    float* cs = use_smem ? sm + 2 * (size_t)n * n : sm;
    float* sn = cs + half;
    int* pp = reinterpret_cast<int*>(sn + half);
    int* qq = pp + half;
    __shared__ float red_off[32], red_tot[32];
    __shared__ int done;
    if (use_smem)
        for (int e = tid; e < n * n; e += nth) H[e] = Hg[e];
    for (int e = tid; e < n * n; e += nth) V[e] = (e / n == e % n) ? 1.f : 0.f;
    __syncthreads();
    int sweep = 0;
    for (;; ++sweep) {
        float off = 0.f, tot = 0.f;
        for (int e = tid; e < n * n; e += nth) {
            const float h = H[e];
            tot += h * h;
            if (e / n != e % n) off += h * h;
        }
        for (int o = 16; o > 0; o >>= 1) {
            off += __shfl_xor_sync(0xffffffffu, off, o);
            tot += __shfl_xor_sync(0xffffffffu, tot, o);
        }
        if ((tid & 31) == 0) { red_off[tid >> 5] = off; red_tot[tid >> 5] = tot; }
        __syncthreads();
        if (tid == 0) {
            float o2 = 0.f, t2 = 0.f;
            for (int w = 0; w < (nth + 31) / 32; ++w) { o2 += red_off[w]; t2 += red_tot[w]; }
            done = o2 <= tol * tol * t2 ? 1 : sweep < max_sweeps ? 0 : o2 > tol * tol * t2 ? 2 : 1;
        }
        __syncthreads();
        if (done) break;
        for (int rd = 0; rd < nm1; ++rd) {
            for (int i = tid; i < half; i += nth) {
                int p = (i == 0) ? 0 : circle(rd + i, nm1);
                int q = (i == 0) ? circle(rd, nm1) : circle(rd - i, nm1);
                if (p > q) { const int tmp = p; p = q; q = tmp; }
                float c = 1.f, s = 0.f;
                if (q < n) {
                    const float hpq = H[(size_t)p * n + q];
                    const float hpp = H[(size_t)p * n + p], hqq = H[(size_t)q * n + q];
                    if (fabsf(hpq) > 1e-30f && fabsf(hpq) > 1e-9f * sqrtf(fabsf(hpp * hqq))) {
                        const float theta = (hqq - hpp) / (2.f * hpq);
                        float t;
                        if (fabsf(theta) > 1e15f) t = 0.5f / theta;
                        else t = copysignf(1.f, theta) / (fabsf(theta) + sqrtf(theta * theta + 1.f));
                        c = 1.f / sqrtf(t * t + 1.f);   // correctly rounded: keeps c^2 + s^2 = 1 tight
                        s = t * c;
                    }
                }
                cs[i] = c; sn[i] = s; pp[i] = p; qq[i] = q;
            }
            __syncthreads();
            for (int e = tid; e < half * half; e += nth) {
                const int bi = e / half, bj = e % half;
                const int pi = pp[bi], qi = qq[bi], pj = pp[bj], qj = qq[bj];
                const float ci = cs[bi], si = sn[bi], cj = cs[bj], sj = sn[bj];
                if (si == 0.f && sj == 0.f) continue;
                const bool vqi = qi < n, vqj = qj < n;
                float h00 = H[(size_t)pi * n + pj];
                float h01 = vqj ? H[(size_t)pi * n + qj] : 0.f;
                float h10 = vqi ? H[(size_t)qi * n + pj] : 0.f;
                float h11 = (vqi && vqj) ? H[(size_t)qi * n + qj] : 0.f;
                // rows: J_i^T
                const float a00 = ci * h00 - si * h10, a01 = ci * h01 - si * h11;
                const float a10 = si * h00 + ci * h10, a11 = si * h01 + ci * h11;
                // columns: J_j
                float n00 = cj * a00 - sj * a01, n01 = sj * a00 + cj * a01;
                float n10 = cj * a10 - sj * a11, n11 = sj * a10 + cj * a11;
                if (bi == bj && si != 0.f) { n01 = 0.f; n10 = 0.f; }
                H[(size_t)pi * n + pj] = n00;
                if (vqj) H[(size_t)pi * n + qj] = n01;
                if (vqi) H[(size_t)qi * n + pj] = n10;
                if (vqi && vqj) H[(size_t)qi * n + qj] = n11;
            }
            for (int e = tid; e < n * half; e += nth) {
                const int a = e / half, bj = e % half;
                const float sj = sn[bj];
                if (sj == 0.f) continue;
                const int pj = pp[bj], qj = qq[bj];
                const float cj = cs[bj];
                const float vp = V[(size_t)a * n + pj], vq = V[(size_t)a * n + qj];
                V[(size_t)a * n + pj] = cj * vp - sj * vq;
                V[(size_t)a * n + qj] = sj * vp + cj * vq;
            }
            __syncthreads();
        }
    }
    for (int i = tid; i < n; i += nth) evals[i] = H[(size_t)i * n + i];
    if (use_smem)
        for (int e = tid; e < n * n; e += nth) Vg[e] = V[e];
    if (tid == 0 && sweeps_out) *sweeps_out = sweep;
    if (tid == 0 && done == 2 && failed) atomicAdd(failed, 1);
}

__device__ __forceinline__ uint32_t float_order(float f) {
    const uint32_t u = __float_as_uint(f);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

// Column statistics of 32 columns from col0 of A (rows x cols, leading dimension ld) by a CTA of 32 x
// 32 threads, lanes along the columns: the sign of the largest-magnitude entry (first row on
// ties) and the sum of squares, both valid in row ty = 0.
__device__ __forceinline__ void column_stats(const float* A, int rows, int64_t ld, int col, bool in, float& sign, float& ss) {
    __shared__ float sbest[32][33], sval[32][33], ssum[32][33];
    __shared__ int sidx[32][33];
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    float best = -1.f, val = 0.f, sum = 0.f;
    int idx = 0x7fffffff;
    if (in)
        for (int a0 = ty; a0 < rows; a0 += 32 * 8) {       // eight rows' reads in flight
            float v[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) v[i] = a0 + 32 * i < rows ? A[(a0 + 32 * i) * ld + col] : 0.f;
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const float m = fabsf(v[i]);
                if (a0 + 32 * i >= rows) break;
                sum = fmaf(v[i], v[i], sum);
                if (m > best) { best = m; val = v[i]; idx = a0 + 32 * i; }
            }
        }
    __syncthreads();
    sbest[ty][tx] = best; sval[ty][tx] = val; ssum[ty][tx] = sum; sidx[ty][tx] = idx;
    __syncthreads();
    if (ty == 0) {
        for (int o = 16; o > 0; o >>= 1)                   // pairwise: what a warp's xor reduction gives
            for (int q = 0; q < o; ++q) ssum[q][tx] += ssum[q + o][tx];
        sum = ssum[0][tx];
        for (int q = 0; q < 32; ++q) {
            if (sbest[q][tx] > best || (sbest[q][tx] == best && sidx[q][tx] < idx)) {
                best = sbest[q][tx]; val = sval[q][tx]; idx = sidx[q][tx];
            }
        }
        sign = val < 0.f ? -1.f : 1.f;
        ss = sum;
    }
}

// Eigenpairs by descending value (ties by index; NaN ordered as its bits), in two launches: a CTA per
// 32 columns counts each one's rank and writes the column's number and its scale (sign rule, unit
// norm: thousands of plane rotations let the norms drift by a few ulp each) there, then a CTA per
// row gathers the row.  One CTA sorting and moving everything took 10.3 ms for n = 2048.
__global__ void __launch_bounds__(1024) sort_rank_kernel(const __grid_constant__ SortGroup g) {
    chain_begin();
    const SortMat& M = g.mat[blockIdx.y];
    const int n = M.n, tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    if ((int)blockIdx.x * 32 >= n) return;
    const int col = blockIdx.x * 32 + tx;
    __shared__ int cnt[32][33];
    int c = 0;
    if (col < n) {
        const uint32_t mine = float_order(M.evals[col]);
        for (int j = ty; j < n; j += 32) {
            const uint32_t other = float_order(M.evals[j]);
            c += (other > mine || (other == mine && j < col)) ? 1 : 0;
        }
    }
    cnt[ty][tx] = c;
    float sign = 1.f, ss = 1.f;
    column_stats(M.V, n, n, col, col < n, sign, ss);       // its barriers cover cnt
    if (ty == 0 && col < n) {
        int rank = 0;
        for (int q = 0; q < 32; ++q) rank += cnt[q][tx];
        M.order[rank] = col;
        M.scale[rank] = sign / sqrtf(ss);
        if (M.evals_sorted) M.evals_sorted[rank] = M.evals[col];
    }
    if (n > 32) return;
    __syncthreads();                                       // one CTA holds it all: no second launch
    if (col < n && ty < n) M.Out[(size_t)ty * n + col] = M.scale[col] * M.V[(size_t)ty * n + M.order[col]];
}
__global__ void __launch_bounds__(256) sort_gather_kernel(const __grid_constant__ SortGroup g) {
    chain_begin();
    extern __shared__ float srow[];
    const SortMat& M = g.mat[blockIdx.y];
    const int n = M.n;
    if (n <= 32) return;
    for (int r = blockIdx.x; r < n; r += gridDim.x) {
        __syncthreads();
        for (int c = threadIdx.x; c < n; c += 256) srow[c] = M.V[(size_t)r * n + c];
        __syncthreads();
        for (int c = threadIdx.x; c < n; c += 256) M.Out[(size_t)r * n + c] = M.scale[c] * srow[M.order[c]];
    }
}

// The largest-magnitude entry of each column of Q (m' x k) positive; a CTA per 32 columns.
__global__ void __launch_bounds__(1024) fix_signs_group_kernel(const __grid_constant__ FinishGroup g) {
    chain_begin();
    const FinishMat& M = g.mat[blockIdx.y];
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5, col = blockIdx.x * 32 + tx;
    if ((int)blockIdx.x * 32 >= M.k) return;
    __shared__ float sg[32];
    float sign = 1.f, ss;
    column_stats(M.Q, M.mp, M.k, col, col < M.k, sign, ss);
    if (ty == 0) sg[tx] = sign;
    __syncthreads();
    if (col < M.k && sg[tx] < 0.f)
        for (int a0 = ty; a0 < M.mp; a0 += 32 * 8) {       // eight rows' reads in flight
            float v[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) v[i] = a0 + 32 * i < M.mp ? M.Q[(size_t)(a0 + 32 * i) * M.k + col] : 0.f;
#pragma unroll
            for (int i = 0; i < 8; ++i)
                if (a0 + 32 * i < M.mp) M.Q[(size_t)(a0 + 32 * i) * M.k + col] = -v[i];
        }
}

// Right-looking Cholesky (one CTA) with a diagonal shift retry on breakdown.
__global__ void __launch_bounds__(1024) cholesky_kernel(float* A, int n, float* orig, int* flag) {
    const int tid = threadIdx.x, nth = blockDim.x;
    __shared__ int fail;
    __shared__ float shift, trace;
    for (int e = tid; e < n * n; e += nth) orig[e] = A[e];
    if (tid == 0) {
        float tr = 0.f;
        for (int i = 0; i < n; ++i) tr += orig[(size_t)i * n + i];
        trace = tr;
        shift = 0.f;
    }
    __syncthreads();
    int attempt = 0;
    for (; attempt < 6; ++attempt) {
        if (attempt > 0) {
            for (int e = tid; e < n * n; e += nth) A[e] = orig[e] + ((e / n == e % n) ? shift : 0.f);
        }
        if (tid == 0) fail = 0;
        __syncthreads();
        const float thresh = 1e-12f * fmaxf(trace / n, 1e-30f);
        for (int j = 0; j < n; ++j) {
            const float d = A[(size_t)j * n + j];
            if (!(d > thresh)) { fail = 1; break; }      // uniform: every thread reads the same d
            const float ljj = sqrtf(d);
            __syncthreads();
            if (tid == 0) A[(size_t)j * n + j] = ljj;
            for (int i = j + 1 + tid; i < n; i += nth) A[(size_t)i * n + j] /= ljj;
            __syncthreads();
            const int rem = n - j - 1;
            for (int e = tid; e < rem * rem; e += nth) {
                const int i = j + 1 + e / rem, l = j + 1 + e % rem;
                if (l <= i) A[(size_t)i * n + l] -= A[(size_t)i * n + j] * A[(size_t)l * n + j];
            }
            __syncthreads();
        }
        __syncthreads();
        if (!fail) break;
        if (tid == 0) shift = chol_shift(attempt, fmaxf(trace / n, 1e-30f));
        __syncthreads();
    }
    for (int e = tid; e < n * n; e += nth)
        if (e % n > e / n) A[e] = 0.f;
    if (tid == 0 && flag) {
        *flag = attempt;
        // no factorisation after every shift, or a Gram matrix with no positive trace (a zero or
        // non-finite block): the refresh cannot orthonormalise it (flag + 6 counts these)
        if (attempt == 6 || !(trace > 0.f) || !isfinite(trace)) atomicAdd(flag + 6, 1);
    }
}

// Q <- Q L^{-T}: one warp per row, y_j = (x_j - sum_{l<j} y_l L_jl) / L_jj.
__global__ void trsm_kernel(float* Q, int rows, int n, const float* L) {
    const int warp = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    if (warp >= rows) return;
    float* y = Q + (size_t)warp * n;
    for (int j = 0; j < n; ++j) {
        float acc = 0.f;
        for (int l = lane; l < j; l += 32) acc = fmaf(y[l], L[(size_t)j * n + l], acc);
        for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
        const float val = (y[j] - acc) / L[(size_t)j * n + j];
        __syncwarp();
        if (lane == 0) y[j] = val;
        __syncwarp();
    }
}

__global__ void random_block_kernel(float* Q, int rows, int cols, uint64_t seed, uint32_t t) {
    const int nq = (cols + 3) / 4;
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= (int64_t)rows * nq) return;
    const int i = static_cast<int>(e / nq), q = static_cast<int>(e % nq);
    const float4 g = gauss4(seed, t, static_cast<uint32_t>(i), static_cast<uint32_t>(q), kTagPowerInit);
    const float gv[4] = {g.x, g.y, g.z, g.w};
    for (int v = 0; v < 4; ++v)
        if (q * 4 + v < cols) Q[(size_t)i * cols + q * 4 + v] = gv[v];
}

// Householder reconstruction, top block: modified LU of S - Q[:k, :k] with s_j = -sign of the
// current Schur-complement entry of Q (so every pivot has magnitude >= 1); then
// T Y1^T = Utilde S by forward substitution.  W (k x k scratch) ends holding L1\Utilde.
__device__ __forceinline__ void hh_top_body(const float* Q, int k, float* W, float* Y, float* T, float* s) {
    const int tid = threadIdx.x, nth = blockDim.x;
    for (int e = tid; e < k * k; e += nth) W[e] = -Q[e];   // rows 0..k-1 of Q (ld = k)
    __syncthreads();
    for (int j = 0; j < k; ++j) {
        const float qjj = -W[(size_t)j * k + j];
        const float sj = qjj >= 0.f ? -1.f : 1.f;
        __syncthreads();
        if (tid == 0) { W[(size_t)j * k + j] += sj; s[j] = sj; }
        __syncthreads();
        const float piv = W[(size_t)j * k + j];
        for (int i = j + 1 + tid; i < k; i += nth) W[(size_t)i * k + j] /= piv;
        __syncthreads();
        const int rem = k - j - 1;
        for (int e = tid; e < rem * rem; e += nth) {
            const int i = j + 1 + e / rem, l = j + 1 + e % rem;
            W[(size_t)i * k + l] -= W[(size_t)i * k + j] * W[(size_t)j * k + l];
        }
        __syncthreads();
    }
    for (int e = tid; e < k * k; e += nth) {
        const int i = e / k, l = e % k;
        Y[(size_t)i * k + l] = i > l ? W[e] : (i == l ? 1.f : 0.f);
    }
    // T row i: T[i][l] = Ut[i][l] s_l - sum_{c<l} T[i][c] Y1[l][c]  (T upper triangular)
    for (int i = tid; i < k; i += nth) {
        float* Ti = T + (size_t)i * k;
        for (int l = 0; l < k; ++l) {
            if (l < i) { Ti[l] = 0.f; continue; }
            float x = W[(size_t)i * k + l] * s[l];
            for (int c = i; c < l; ++c) x -= Ti[c] * W[(size_t)l * k + c];
            Ti[l] = x;
        }
    }
}

__global__ void __launch_bounds__(1024) hh_top_kernel(const float* Q, int k, float* W, float* Y, float* T,
                                                      float* s) {
    hh_top_body(Q, k, W, Y, T, s);
}
// Rows a >= k: Y[a, :] Utilde = -Q[a, :], one warp per row (forward substitution).
__device__ __forceinline__ void hh_rows_body(const float* Q, int mp, int k, const float* W, float* Y, int warp) {
    const int lane = threadIdx.x & 31;
    const int a = k + warp;
    if (a >= mp) return;
    float* y = Y + (size_t)a * k;
    const float* qa = Q + (size_t)a * k;
    for (int l = 0; l < k; ++l) {
        float acc = 0.f;
        for (int c = lane; c < l; c += 32) acc = fmaf(y[c], W[(size_t)c * k + l], acc);
        for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
        const float val = (-qa[l] - acc) / W[(size_t)l * k + l];
        __syncwarp();
        if (lane == 0) y[l] = val;
        __syncwarp();
    }
}
__global__ void hh_rows_kernel(const float* Q, int mp, int k, const float* W, float* Y) {
    hh_rows_body(Q, mp, k, W, Y, blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5));
}
__global__ void wy_basis_kernel(int mp, int k, const float* Y, const float* Yt, const float* dsign, float* U) {
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= (int64_t)mp * mp) return;
    const int a = static_cast<int>(e / mp), j = static_cast<int>(e % mp);
    float v = (a == j) ? 1.f : 0.f;
    for (int c = 0; c < k; ++c) v = fmaf(-Y[(size_t)a * k + c], Yt[(size_t)j * k + c], v);
    if (j < k) v *= dsign[j];
    U[e] = v;
}

}  // namespace

cudaError_t jacobi_eig(float* H, int n, float* V, float* evals, int* sweeps, int* failed, cudaStream_t st) {
    const int npad = n + (n & 1), half = npad / 2;
    const size_t pair_bytes = (size_t)half * 16;
    const size_t full = 2 * sizeof(float) * (size_t)n * n + pair_bytes;
    const int use_smem = full <= 200 * 1024 ? 1 : 0;
    const size_t smem = use_smem ? full : pair_bytes;
    {   // per device: set on every call (cheap next to the launch)
        const cudaError_t ea = cudaFuncSetAttribute(jacobi_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 210 * 1024);
        if (ea != cudaSuccess) return ea;
    }
    const float tol = 4.f * 5.96e-8f * sqrtf(static_cast<float>(n)) + 1e-7f;
    // one thread per 2 x 2 block update of a round, rounded to whole warps (at most 1024)
    const int work = n * half > half * half ? n * half : half * half;
    const int nth = work >= 1024 ? 1024 : ((work + 31) / 32) * 32;
    jacobi_kernel<<<1, nth, smem, st>>>(H, n, V, evals, sweeps, failed, use_smem, kJacobiSweeps, tol);
    return cudaGetLastError();
}

cudaError_t sort_group(const SortGroup& g, cudaStream_t st) {
    if (g.nmat <= 0) return cudaSuccess;
    int n = 0;
    for (int i = 0; i < g.nmat; ++i) n = g.mat[i].n > n ? g.mat[i].n : n;
    launch_chain(sort_rank_kernel, dim3((n + 31) / 32, g.nmat), 1024, 0, st, g);
    if (n <= 32) return cudaGetLastError();
    ++more_launches;
    launch_chain(sort_gather_kernel, dim3(n < 1024 ? n : 1024, g.nmat), 256, sizeof(float) * n, st, g);
    return cudaGetLastError();
}

namespace {
// Packed lower triangle: element (i, l), l <= i, at i (i + 1) / 2 + l.
__device__ __forceinline__ int tri(int i, int l) { return i * (i + 1) / 2 + l; }

// S = L^{-T} with L L^T = G (n x n symmetric positive definite, n <= 256): one CTA, the packed lower
// triangle in shared memory.  Right-looking Cholesky (a warp per row of the trailing update, lanes
// along the row); if a pivot is not positive a diagonal shift (1e-7, then x100, times the mean
// diagonal) is added and the factorisation restarts, at most six attempts, the attempts counted
// in *flag.  Then L^{-1} in place, column by column from the last: for j = n-1..0 the entries
// below the diagonal of column j are -(L^{-1}[i, j+1..i] . L[j+1..i, j]) / L_jj.  Each step first
// copies the column it reads into a contiguous array (a column of the packed triangle is strided
// by the row lengths, which would make the lanes' reads collide in the banks).  S (row-major
// n x n) is the transpose of L^{-1}.
__global__ void __launch_bounds__(1024) chol_inverse_kernel(const float* G, int n, float* S, int* flag) {
    extern __shared__ float L[];                       // n (n + 1) / 2 packed, then n + n temporaries
    float* col = L + n * (n + 1) / 2;
    float* tmp = col + n;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = blockDim.x >> 5;
    __shared__ int fail;
    __shared__ float shift, trace;
    if (warp == 0) {                                   // trace: a warp sum in a fixed order
        float tr = 0.f;
        for (int i = lane; i < n; i += 32) tr += G[(size_t)i * n + i];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) tr += __shfl_xor_sync(0xffffffffu, tr, o);
        if (lane == 0) { trace = tr; shift = 0.f; }
    }
    __syncthreads();
    int attempt = 0;
    for (; attempt < 6; ++attempt) {
        for (int i = warp; i < n; i += nw)
            for (int l = lane; l <= i; l += 32) L[tri(i, l)] = G[(size_t)i * n + l] + (l == i ? shift : 0.f);
        if (tid == 0) fail = 0;
        __syncthreads();
        const float thresh = 1e-12f * fmaxf(trace / n, 1e-30f);
        for (int j = 0; j < n; ++j) {
            const float d = L[tri(j, j)];
            if (!(d > thresh)) { fail = 1; break; }      // uniform: every thread reads the same d
            const float ljj = sqrtf(d);
            __syncthreads();
            if (tid == 0) L[tri(j, j)] = ljj;
            for (int i = j + 1 + tid; i < n; i += blockDim.x) {
                const float v = L[tri(i, j)] / ljj;
                L[tri(i, j)] = v;
                col[i] = v;
            }
            __syncthreads();
            for (int i = j + 1 + warp; i < n; i += nw) {
                const float lij = col[i];
                for (int l = j + 1 + lane; l <= i; l += 32) L[tri(i, l)] -= lij * col[l];
            }
            __syncthreads();
        }
        __syncthreads();
        if (!fail) break;
        if (tid == 0) shift = chol_shift(attempt, fmaxf(trace / n, 1e-30f));
        __syncthreads();
    }
    if (tid == 0 && flag) {
        *flag = attempt;
        // no factorisation after every shift, or a Gram matrix with no positive trace (a zero or
        // non-finite block): the refresh cannot orthonormalise it (flag + 6 counts these)
        if (attempt == 6 || !(trace > 0.f) || !isfinite(trace)) atomicAdd(flag + 6, 1);
    }
    for (int j = n - 1; j >= 0; --j) {
        for (int l = j + 1 + tid; l < n; l += blockDim.x) col[l] = L[tri(l, j)];
        __syncthreads();
        for (int i = j + 1 + warp; i < n; i += nw) {
            float t = 0.f;
            for (int l = j + 1 + lane; l <= i; l += 32) t += L[tri(i, l)] * col[l];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
            if (lane == 0) tmp[i] = t;
        }
        __syncthreads();
        const float ajj = 1.0f / L[tri(j, j)];
        for (int i = j + 1 + tid; i < n; i += blockDim.x) L[tri(i, j)] = -tmp[i] * ajj;
        if (tid == 0) L[tri(j, j)] = ajj;
        __syncthreads();
    }
    for (int e = tid; e < n * n; e += blockDim.x) {
        const int r = e / n, c = e % n;
        S[e] = c >= r ? L[tri(c, r)] : 0.f;
    }
}

// ---- blocked factor and inverse of the grouped refreshes, n <= 256 --------------------------------
// One CTA of 16 warps a matrix, the lower triangle as 32 x 32 blocks in shared memory (block (i, j) at
// i (i + 1) / 2 + j, pitch 36: rows 16-byte aligned, the products' reads free of bank conflicts),
// padded to whole blocks with a multiple of the identity.  A panel: one warp factors the diagonal block with a row
// a lane and hands each column on; in the same steps a warp inverts that block and a warp per block
// below solves against it by substitution; then the trailing blocks are 32 x 32 x 32 products, a
// warp each.  The inverse goes block column by block column from the last, in place:
// T_i = sum_{j < k <= i} X_ik L_kj, X_ij = -T_i X_jj.  Bound by the diagonal blocks' chain of square
// roots, quotients and shuffles (n = 256: 0.20 ms, n = 128: 66 us; factoring and inverting column by
// column, four barriers each, took 0.80 and 0.22 ms).
constexpr int CB = 32, CP = 36, CBLK = CB * CP, CWARPS = 16;
constexpr int kCholMaxBlocks = 8;
// a block more than the triangle and T: the eliminations' dead reads
constexpr size_t kCholSmem = sizeof(float) * CBLK * (kCholMaxBlocks * (kCholMaxBlocks + 1) / 2 + kCholMaxBlocks);

__device__ __forceinline__ float* cblk(float* L, int i, int j) { return L + (size_t)(i * (i + 1) / 2 + j) * CBLK; }

// acc += A B or A B^T over a 32 x 32 block: rows r0 + lane / 4 + 8 i, columns as cmm_col.
template <int ROWS, bool TB>
__device__ __forceinline__ void cmm(const float* A, const float* B, int r0, int lane, float (&acc)[ROWS][8]) {
    const float* a = A + (r0 + (lane >> 2)) * CP;
    const float* b = TB ? B + (lane & 3) * CP : B + 8 * (lane & 3);
#pragma unroll 4
    for (int k = 0; k < CB; ++k) {
        float av[ROWS], bv[8];
#pragma unroll
        for (int i = 0; i < ROWS; ++i) av[i] = a[8 * i * CP + k];
        if (TB) {
#pragma unroll
            for (int c = 0; c < 8; ++c) bv[c] = b[4 * c * CP + k];
        } else {
            const float4 x = *reinterpret_cast<const float4*>(b + k * CP), y = *reinterpret_cast<const float4*>(b + k * CP + 4);
            bv[0] = x.x; bv[1] = x.y; bv[2] = x.z; bv[3] = x.w; bv[4] = y.x; bv[5] = y.y; bv[6] = y.z; bv[7] = y.w;
        }
#pragma unroll
        for (int i = 0; i < ROWS; ++i)
#pragma unroll
            for (int c = 0; c < 8; ++c) acc[i][c] = fmaf(av[i], bv[c], acc[i][c]);
    }
}
template <bool TB> __device__ __forceinline__ int cmm_col(int lane, int c) { return TB ? (lane & 3) + 4 * c : 8 * (lane & 3) + c; }

// The 32-step eliminations below keep a lane's 32 values in registers and shift them down by one a step, so
// that the step's code is the same every time: unrolled over the steps they are ten thousand
// instructions run once, and the instruction fetches took ten times the arithmetic (k = 256 top
// block 1.93 ms).  Reads past the block (dead values) stay inside the padded shared memory.

__device__ __forceinline__ void load_row(float (&a)[CB], const float* row) {
#pragma unroll
    for (int c = 0; c < CB; c += 4) {
        const float4 x = *reinterpret_cast<const float4*>(row + c);
        a[c] = x.x; a[c + 1] = x.y; a[c + 2] = x.z; a[c + 3] = x.w;
    }
}

// Substitution against the triangular block D: x_c = a_c (/ D_cc), a_q -= x_c D(c, q) for q > c, the
// coefficients dq apart from the diagonal on; x_c to out[c * os].  One warp, a system a lane.
template <bool DIV>
__device__ __forceinline__ void eliminate(float (&a)[CB], const float* D, int dq, float* out, int os) {
#pragma unroll 1
    for (int c = 0; c < CB; ++c) {
        const float* d = D + c * (CP + 1);
        const float x = DIV ? a[0] / d[0] : a[0];
#pragma unroll
        for (int q = 1; q < CB; ++q) a[q - 1] = fmaf(-x, d[q * dq], a[q]);
        a[CB - 1] = 0.f;
        __syncwarp();                                  // out may be D's row c, read by now
        out[c * os] = x;
    }
}

__global__ void __launch_bounds__(CWARPS * 32) chol_group_kernel(const __grid_constant__ CholGroup g) {
    chain_begin();
    extern __shared__ __align__(16) float csm[];
    const CholMat& M = g.mat[blockIdx.x];
    const int n = M.n, nb = (n + CB - 1) / CB, t = threadIdx.x, warp = t >> 5, lane = t & 31;
    float* L = csm;
    float* T = L + (size_t)(nb * (nb + 1) / 2) * CBLK;
    __shared__ int fail;
    __shared__ float shift, trace;
    __shared__ float colb[2][2 * CB];                  // column c of L_pp; past it zeros, read for dead values
    if (t < 2 * CB) colb[t / CB][CB + t % CB] = 0.f;
    auto entry = [&](int i, int l) {
        if (M.tri_only == kTriUpper) return M.part[(size_t)l * M.n + i];           // L = U^T
        if (M.tri_only == kTriUnitLower) return i == l ? 1.f : M.part[(size_t)i * M.n + l];
        return M.part[(size_t)i * M.ld + l];
    };
    if (warp == 0) {                                   // trace: a warp sum in a fixed order
        float tr = 0.f;
        if (!M.tri_only)
            for (int i = lane; i < n; i += 32) tr += entry(i, i);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) tr += __shfl_xor_sync(0xffffffffu, tr, o);
        if (lane == 0) { trace = tr; shift = 0.f; }
    }
    int attempt = 0;
    for (; attempt < 6; ++attempt) {
        __syncthreads();
        const float pad = M.tri_only ? 1.f : fmaxf(trace / n, 1e-30f);   // its pivots pass like the matrix's own
#pragma unroll 4
        for (int q = warp; q < nb * (nb + 1) / 2 * CB; q += CWARPS) {    // a block row a warp
            int i = 0, j = q / CB;                                       // j = i (i + 1) / 2 + block column
            while (j > i) { j -= i + 1; ++i; }
            const int r = i * CB + q % CB, c = j * CB + lane;
            float v = r == c ? pad : 0.f;
            if (r < n && c < n) {
                v = c <= r ? entry(r, c) : 0.f;
                if (r == c && !M.tri_only) v += shift;
            }
            cblk(L, i, j)[(q % CB) * CP + lane] = v;
        }
        if (t == 0) fail = 0;
        __syncthreads();
        if (M.tri_only) break;
        const float thresh = 1e-12f * fmaxf(trace / n, 1e-30f);
        for (int p = 0; p < nb; ++p) {
            // L_pp by warp 0 (lane = row), a column a step; the others take each column as it comes: warp 1
            // to X_pp = L_pp^{-1} (lane = column, over L_pp, which nothing else reads), a warp per block
            // below to L_ip = A_ip L_pp^{-T} (lane = row)
            const int i = p + warp - 1;
            const bool on = warp < 2 || i < nb;
            float* A = warp < 2 ? cblk(L, p, p) + (warp ? lane : lane * CP) : on ? cblk(L, i, p) + lane * CP : nullptr;
            const int os = warp == 1 ? CP : 1;
            float a[CB];
            if (warp != 1 && on) load_row(a, A);
            else
#pragma unroll
                for (int q = 0; q < CB; ++q) a[q] = lane == q ? 1.f : 0.f;
            bool ok = true;
#pragma unroll 1
            for (int c = 0; c < CB; ++c) {
                float* cb = colb[c & 1];
                float v = 0.f;
                if (warp == 0) {
                    const float d = __shfl_sync(0xffffffffu, a[0], c);
                    ok = ok && d > thresh;
                    const float l = sqrtf(d);
                    v = lane == c ? l : lane > c ? a[0] / l : 0.f;
                    cb[lane] = v;
                }
                __syncthreads();
                if (warp == 0) {
#pragma unroll
                    for (int q = 1; q < CB; ++q) a[q - 1] = fmaf(-v, __shfl_sync(0xffffffffu, v, (c + q) & 31), a[q]);
                    a[CB - 1] = 0.f;
                } else if (on) {
                    const float x = a[0] / cb[c];
#pragma unroll
                    for (int q = 1; q < CB; ++q) a[q - 1] = fmaf(-x, cb[c + q], a[q]);
                    a[CB - 1] = 0.f;
                    A[c * os] = x;
                }
            }
            if (warp == 0 && lane == 0 && !ok) fail = 1;
            __syncthreads();
            if (fail) break;                           // uniform: read after the barrier, written before it
            const int m = nb - p - 1;
            for (int q = warp; q < m * (m + 1) / 2; q += CWARPS) {       // A_ij -= L_ip L_jp^T
                int i = 0, j = q;
                while (j > i) { j -= i + 1; ++i; }
                i += p + 1; j += p + 1;
                float acc[4][8] = {};
                cmm<4, true>(cblk(L, i, p), cblk(L, j, p), 0, lane, acc);
                float* C = cblk(L, i, j);
#pragma unroll
                for (int r = 0; r < 4; ++r)
#pragma unroll
                    for (int c = 0; c < 8; ++c) C[((lane >> 2) + 8 * r) * CP + cmm_col<true>(lane, c)] -= acc[r][c];
            }
            __syncthreads();
        }
        if (!fail) break;
        __syncthreads();
        if (t == 0) shift = chol_shift(attempt, fmaxf(trace / n, 1e-30f));
    }
    __syncthreads();
    if (t == 0 && !M.tri_only && M.flag) {
        *M.flag = attempt;
        // no factorisation after every shift, or a Gram matrix with no positive trace (a zero or
        // non-finite block): the refresh cannot orthonormalise it (flag + 6 counts these)
        if (attempt == 6 || !(trace > 0.f) || !isfinite(trace)) atomicAdd(M.flag + 6, 1);
    }
    for (int j = warp; j < nb && M.tri_only; j += CWARPS) {              // X_jj in place, lane = column
        float a[CB];
#pragma unroll
        for (int i = 0; i < CB; ++i) a[i] = lane == i ? 1.f : 0.f;
        eliminate<true>(a, cblk(L, j, j), CP, cblk(L, j, j) + lane, CP);
    }
    __syncthreads();
    for (int j = nb - 2; j >= 0; --j) {
        const int m = nb - 1 - j;                      // half a block (16 rows) a task
        for (int q = warp; q < 2 * m; q += CWARPS) {
            const int i = nb - 1 - (q >> 1), r0 = 16 * (q & 1);          // the longest sums first
            float acc[2][8] = {};
            for (int k = j + 1; k <= i; ++k) cmm<2, false>(cblk(L, i, k), cblk(L, k, j), r0, lane, acc);
            float* C = T + (size_t)(i - j - 1) * CBLK;
#pragma unroll
            for (int r = 0; r < 2; ++r)
#pragma unroll
                for (int c = 0; c < 8; ++c) C[(r0 + (lane >> 2) + 8 * r) * CP + cmm_col<false>(lane, c)] = -acc[r][c];
        }
        __syncthreads();
        for (int q = warp; q < 2 * m; q += CWARPS) {
            const int i = j + 1 + (q >> 1), r0 = 16 * (q & 1);
            float acc[2][8] = {};
            cmm<2, false>(T + (size_t)(i - j - 1) * CBLK, cblk(L, j, j), r0, lane, acc);
            float* C = cblk(L, i, j);
#pragma unroll
            for (int r = 0; r < 2; ++r)
#pragma unroll
                for (int c = 0; c < 8; ++c) C[(r0 + (lane >> 2) + 8 * r) * CP + cmm_col<false>(lane, c)] = acc[r][c];
        }
        __syncthreads();
    }
    for (int e = t; e < M.ld * M.ld; e += CWARPS * 32) {
        const int r = e / M.ld, c = e % M.ld;
        M.out[e] = (c <= r && r < n) ? cblk(L, r / CB, c / CB)[(r % CB) * CP + c % CB] : 0.f;
    }
}
// Householder reconstruction, top blocks of the grouped refreshes: the modified LU of hh_top_kernel
// (pivots W_jj + s_j, s_j = -sign of the current Schur complement of Q) in 32-column panels: the
// panel's column and row blocks in shared memory, the diagonal block by one warp with a row a lane,
// the others by substitution, a warp each, the trailing blocks as 32 x 32 x 32 products on the matrix
// in L2.  W ends holding L1 \ U, Y's top the unit lower L1, and Us = U diag(s) (zero below), from
// which T = Us L1^{-T}.  Column by column, with T by a thread per row: 2.1 ms for k = 256.
constexpr size_t kHhSmem = sizeof(float) * CBLK * (2 * kCholMaxBlocks);

__global__ void __launch_bounds__(CWARPS * 32) hh_lu_group_kernel(const __grid_constant__ FinishGroup g) {
    chain_begin();
    extern __shared__ __align__(16) float hsm[];
    const FinishMat& M = g.mat[blockIdx.x];
    const int k = M.k, nb = (k + CB - 1) / CB, t = threadIdx.x, warp = t >> 5, lane = t & 31;
    float* const W = M.Wtop;
    for (int e = t; e < k * k; e += CWARPS * 32) W[e] = -M.Q[e];         // rows 0..k-1 of Q (ld = k)
    __syncthreads();
    for (int p = 0; p < nb; ++p) {
        const int m = nb - p;                          // column blocks p .., then row blocks p + 1 ..
        for (int q = warp; q < (2 * m - 1) * CB; q += CWARPS) {
            const int blk = q / CB, r = (blk < m ? p + blk : p) * CB + q % CB, c = (blk < m ? p : p + 1 + blk - m) * CB + lane;
            hsm[(size_t)blk * CBLK + (q % CB) * CP + lane] = r < k && c < k ? W[(size_t)r * k + c] : r == c ? 1.f : 0.f;
        }
        __syncthreads();
        float* D = hsm;
        if (warp == 0) {
            float a[CB];
            load_row(a, D + lane * CP);
#pragma unroll 1
            for (int c = 0; c < CB; ++c) {
                const float d = __shfl_sync(0xffffffffu, a[0], c), sj = d <= 0.f ? -1.f : 1.f, piv = d + sj;
                if (lane == c && p * CB + c < k) M.s[p * CB + c] = sj;
                const float v = lane > c ? a[0] / piv : 0.f;
                D[lane * CP + c] = lane > c ? v : lane == c ? piv : a[0];
#pragma unroll
                for (int q = 1; q < CB; ++q) a[q - 1] = fmaf(-v, __shfl_sync(0xffffffffu, a[q], c), a[q]);
                a[CB - 1] = 0.f;
            }
        }
        __syncthreads();
        for (int blk = 1 + warp; blk < 2 * m - 1; blk += CWARPS) {
            float* A = hsm + (size_t)blk * CBLK;
            float a[CB];
            if (blk < m) {                             // L = A U^{-1}, lane = row
                load_row(a, A + lane * CP);
                eliminate<true>(a, D, 1, A + lane * CP, 1);
            } else {                                   // U = L1^{-1} A, lane = column
#pragma unroll
                for (int c = 0; c < CB; ++c) a[c] = A[c * CP + lane];
                eliminate<false>(a, D, CP, A + lane, CP);
            }
        }
        __syncthreads();
        for (int q = warp; q < (2 * m - 1) * CB; q += CWARPS) {
            const int blk = q / CB, r = (blk < m ? p + blk : p) * CB + q % CB, c = (blk < m ? p : p + 1 + blk - m) * CB + lane;
            if (r < k && c < k) W[(size_t)r * k + c] = hsm[(size_t)blk * CBLK + (q % CB) * CP + lane];
        }
        for (int q = warp; q < (m - 1) * (m - 1); q += CWARPS) {
            const int i = q / (m - 1), j = q % (m - 1);
            float acc[4][8] = {};
            cmm<4, false>(hsm + (size_t)(1 + i) * CBLK, hsm + (size_t)(m + j) * CBLK, 0, lane, acc);
            const int c0 = (p + 1 + j) * CB + 8 * (lane & 3);
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const int row = (p + 1 + i) * CB + (lane >> 2) + 8 * r;
#pragma unroll
                for (int h = 0; h < 2; ++h) {          // k is a multiple of 4
                    if (row >= k || c0 + 4 * h >= k) continue;
                    float4* C = reinterpret_cast<float4*>(W + (size_t)row * k + c0 + 4 * h);
                    float4 x = *C;
                    x.x -= acc[r][4 * h]; x.y -= acc[r][4 * h + 1]; x.z -= acc[r][4 * h + 2]; x.w -= acc[r][4 * h + 3];
                    *C = x;
                }
            }
        }
        __syncthreads();
    }
    for (int e = t; e < k * k; e += CWARPS * 32) {
        const int i = e / k, l = e % k;
        const float w = W[e];
        M.Y[e] = i > l ? w : i == l ? 1.f : 0.f;
        M.Us[e] = i <= l ? w * M.s[l] : 0.f;
    }
}

// ---- the end of the k <= 32 refreshes (the fp32 conv layers), all matrices of a step in each launch ----
// Bound by chains of quotients, roots and barriers at these sizes, so a matrix's small work sits in
// one CTA or warp, and the four launches replace twelve a matrix on as many streams.  The operations
// and their order are those of jacobi_kernel, hh_top_kernel, hh_rows_kernel and the products.

// jacobi_kernel and sort_rank_kernel for n <= 32: a thread keeps one 2 x 2 block of H and one pair of V's
// entries for all rounds, so their indices are formed once, and the round's pairs advance along the
// circle by increments (eight matrices, k = 16: 43 us; 68 + 9 us for the two kernels).
__host__ __device__ __forceinline__ int tail_threads(int n) { return (n * ((n + 1) / 2) + 31) / 32 * 32; }

__global__ void __launch_bounds__(512) tail_ritz_kernel(const __grid_constant__ TailGroup g) {
    chain_begin();
    constexpr int P = 33;
    __shared__ float H[32 * P], V[32 * P];
    __shared__ float4 rot[16];                             // c, s, then p and q as row offsets
    __shared__ float red_off[16], red_tot[16], ev[32];
    __shared__ int done;
    const TailMat& M = g.mat[blockIdx.x];
    const int n = M.k, half = (n + 1) / 2, nm1 = 2 * half - 1, nth = tail_threads(n);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const float tol = 4.f * 5.96e-8f * sqrtf(static_cast<float>(n)) + 1e-7f;
    // this thread's entries of the norms (n^2 <= 2 nth), its block of H and its entries of V
    int he[2];
    bool hd[2];
    for (int i = 0; i < 2; ++i) {
        const int e = tid + i * nth, r = e / n, c = e % n;
        he[i] = tid < nth && e < n * n ? r * P + c : -1;
        hd[i] = r == c;
        if (he[i] >= 0) {
            H[he[i]] = M.H[e];
            V[he[i]] = hd[i] ? 1.f : 0.f;
        }
    }
    const int bi = tid / half, bj = tid % half;
    int xp = tid % nm1, xq = (nm1 - tid % nm1) % nm1;      // the circle's places of pair tid < half
    const int xp0 = xp, xq0 = xq;
    __syncthreads();
    int sweep = 0;
    for (;; ++sweep) {
        float off = 0.f, tot = 0.f;
#pragma unroll
        for (int i = 0; i < 2; ++i)
            if (he[i] >= 0) {
                const float h = H[he[i]];
                tot += h * h;
                if (!hd[i]) off += h * h;
            }
        for (int o = 16; o > 0; o >>= 1) {
            off += __shfl_xor_sync(0xffffffffu, off, o);
            tot += __shfl_xor_sync(0xffffffffu, tot, o);
        }
        if (lane == 0) { red_off[warp] = off; red_tot[warp] = tot; }
        __syncthreads();
        if (tid == 0) {
            float o2 = 0.f, t2 = 0.f;
            for (int w = 0; w < nth / 32; ++w) { o2 += red_off[w]; t2 += red_tot[w]; }
            done = o2 <= tol * tol * t2 ? 1 : sweep < kJacobiSweeps ? 0 : 2;
        }
        __syncthreads();
        if (done) break;
        xp = xp0; xq = xq0;
        for (int rd = 0; rd < nm1; ++rd) {
            if (tid < half) {
                int p = (tid == 0) ? 0 : 1 + xp;
                int q = 1 + xq;
                if (p > q) { const int tmp = p; p = q; q = tmp; }
                float c = 1.f, s = 0.f;
                if (q < n) {
                    const float hpq = H[p * P + q];
                    const float hpp = H[p * P + p], hqq = H[q * P + q];
                    if (fabsf(hpq) > 1e-30f && fabsf(hpq) > 1e-9f * sqrtf(fabsf(hpp * hqq))) {
                        const float theta = (hqq - hpp) / (2.f * hpq);
                        float t;
                        if (fabsf(theta) > 1e15f) t = 0.5f / theta;
                        else t = copysignf(1.f, theta) / (fabsf(theta) + sqrtf(theta * theta + 1.f));
                        c = 1.f / sqrtf(t * t + 1.f);
                        s = t * c;
                    }
                }
                rot[tid] = make_float4(c, s, __int_as_float(p), __int_as_float(q));
                xp = xp + 1 == nm1 ? 0 : xp + 1;
                xq = xq + 1 == nm1 ? 0 : xq + 1;
            }
            __syncthreads();
            if (tid < n * half) {
                const float4 rj = rot[bj];
                const float cj = rj.x, sj = rj.y;
                const int pj = __float_as_int(rj.z), qj = __float_as_int(rj.w);
                if (tid < half * half) {
                    const float4 ri = rot[bi];
                    const float ci = ri.x, si = ri.y;
                    const int pi = __float_as_int(ri.z), qi = __float_as_int(ri.w);
                    if (si != 0.f || sj != 0.f) {
                        const bool vqi = qi < n, vqj = qj < n;
                        float h00 = H[pi * P + pj];
                        float h01 = vqj ? H[pi * P + qj] : 0.f;
                        float h10 = vqi ? H[qi * P + pj] : 0.f;
                        float h11 = (vqi && vqj) ? H[qi * P + qj] : 0.f;
                        const float a00 = ci * h00 - si * h10, a01 = ci * h01 - si * h11;
                        const float a10 = si * h00 + ci * h10, a11 = si * h01 + ci * h11;
                        float n00 = cj * a00 - sj * a01, n01 = sj * a00 + cj * a01;
                        float n10 = cj * a10 - sj * a11, n11 = sj * a10 + cj * a11;
                        if (bi == bj && si != 0.f) { n01 = 0.f; n10 = 0.f; }
                        H[pi * P + pj] = n00;
                        if (vqj) H[pi * P + qj] = n01;
                        if (vqi) H[qi * P + pj] = n10;
                        if (vqi && vqj) H[qi * P + qj] = n11;
                    }
                }
                if (sj != 0.f) {                           // row bi of V
                    const float vp = V[bi * P + pj], vq = V[bi * P + qj];
                    V[bi * P + pj] = cj * vp - sj * vq;
                    V[bi * P + qj] = sj * vp + cj * vq;
                }
            }
            __syncthreads();
        }
    }
    if (tid < n) {
        ev[tid] = H[tid * P + tid];
        M.evals[tid] = ev[tid];
    }
    if (tid == 0 && M.sweeps) *M.sweeps = sweep;
    if (tid == 0 && done == 2 && M.failed) atomicAdd(M.failed, 1);
    __syncthreads();
    // sorted by descending value (ties by index), unit columns, largest entry positive: a warp a column
    for (int col = warp; col < n; col += blockDim.x >> 5) {
        const uint32_t mine = float_order(ev[col]), other = lane < n ? float_order(ev[lane]) : 0u;
        const int rank = __popc(__ballot_sync(0xffffffffu, lane < n && (other > mine || (other == mine && lane < col))));
        const float v = lane < n ? V[lane * P + col] : 0.f;
        float ss = v * v, best = lane < n && fabsf(v) >= 0.f ? fabsf(v) : -1.f, val = best < 0.f ? 0.f : v;
        int idx = best < 0.f ? 0x7fffffff : lane;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            ss += __shfl_xor_sync(0xffffffffu, ss, o);
            const float ob = __shfl_xor_sync(0xffffffffu, best, o), ov = __shfl_xor_sync(0xffffffffu, val, o);
            const int oi = __shfl_xor_sync(0xffffffffu, idx, o);
            if (ob > best || (ob == best && oi < idx)) { best = ob; val = ov; idx = oi; }
        }
        const float scale = (val < 0.f ? -1.f : 1.f) / sqrtf(ss);
        if (lane < n) M.R[lane * n + rank] = scale * v;
        if (lane == 0 && M.evals_sorted) M.evals_sorted[rank] = ev[col];
    }
}

// The sign of each column of Q (its largest-|entry| positive, the first row on ties) by the whole CTA, then
// the top block of the Householder reconstruction by one warp, a row a lane in registers that move
// down by one a column: the modified LU of hh_top_kernel and T by substitution along its columns
// (m' = 512, k = 16: 11 us; fix_signs and hh_top_kernel 13 + 17 us).
template <int KM>
__global__ void __launch_bounds__(1024) tail_top_kernel(const __grid_constant__ TailGroup g) {
    chain_begin();
    constexpr int RG = 1024 / KM;
    __shared__ float sbest[RG][KM + 1], sval[RG][KM + 1];
    __shared__ int sidx[RG][KM + 1];
    __shared__ float sg[32], Ss[32];
    __shared__ float Ws[2 * KM][KM + 1];                   // rows past k: read for values nobody uses
    const TailMat& M = g.mat[blockIdx.x];
    const int k = M.k, mp = M.mp, tid = threadIdx.x, lane = tid & 31;
    {
        const int col = tid % KM, rg = tid / KM;
        float best = -1.f, val = 0.f;
        int idx = 0x7fffffff;
        if (col < k)
#pragma unroll 8
            for (int a = rg; a < mp; a += RG) {
                const float v = M.Q[(size_t)a * k + col], m = fabsf(v);
                if (m > best) { best = m; val = v; idx = a; }
            }
        sbest[rg][col] = best; sval[rg][col] = val; sidx[rg][col] = idx;
    }
    for (int e = tid; e < 2 * KM * (KM + 1); e += 1024) (&Ws[0][0])[e] = 0.f;
    __syncthreads();
    for (int col = tid >> 5; col < k; col += 32) {         // a warp a column
        float best = -1.f, val = 0.f;
        int idx = 0x7fffffff;
#pragma unroll
        for (int q = lane; q < RG; q += 32)
            if (sbest[q][col] > best || (sbest[q][col] == best && sidx[q][col] < idx)) {
                best = sbest[q][col]; val = sval[q][col]; idx = sidx[q][col];
            }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const float ob = __shfl_xor_sync(0xffffffffu, best, o), ov = __shfl_xor_sync(0xffffffffu, val, o);
            const int oi = __shfl_xor_sync(0xffffffffu, idx, o);
            if (ob > best || (ob == best && oi < idx)) { best = ob; val = ov; idx = oi; }
        }
        if (lane == 0) { sg[col] = val < 0.f ? -1.f : 1.f; M.sign[col] = sg[col]; }
    }
    __syncthreads();
    if (tid >= 32) return;
    float a[KM];
#pragma unroll
    for (int c = 0; c < KM; ++c) {
        const float q = lane < k && c < k ? M.Q[(size_t)lane * k + c] : 0.f;
        a[c] = c < k && sg[c] < 0.f ? q : -q;              // -Q with the signs
    }
#pragma unroll 1
    for (int j = 0; j < k; ++j) {
        const float wjj = __shfl_sync(0xffffffffu, a[0], j), sj = -wjj >= 0.f ? -1.f : 1.f, piv = wjj + sj;
        const float v = lane > j ? a[0] / piv : lane == j ? piv : a[0];
#pragma unroll
        for (int q = 1; q < KM; ++q) {
            const float u = __shfl_sync(0xffffffffu, a[q], j);
            a[q - 1] = lane > j ? fmaf(-v, u, a[q]) : a[q];
        }
        a[KM - 1] = 0.f;
        if (lane < KM) Ws[lane][j] = v;
        if (lane == 0) Ss[j] = sj;
    }
    __syncwarp();
#pragma unroll
    for (int l = 0; l < KM; ++l) a[l] = lane < KM && l < k ? Ws[lane][l] * Ss[l] : 0.f;
    float* Ti = M.T + (size_t)lane * k;
#pragma unroll 1
    for (int c = 0; c < k; ++c) {                          // T[i][l] -= T[i][c] Y1[l][c] for l > c
        const bool in = c >= lane;
        const float x = in ? a[0] : 0.f;
#pragma unroll
        for (int q = 1; q < KM; ++q) a[q - 1] = in ? fmaf(-x, Ws[c + q][c], a[q]) : a[q];
        if (lane < k) Ti[c] = x;
    }
    for (int e = lane; e < k * k; e += 32) M.W[e] = Ws[e / k][e % k];
    if (lane < k) M.s[lane] = Ss[lane];
}

// A CTA per 32 rows, a warp four rows side by side, lane = column: the signs, Y (rows >= k by
// substitution against Utilde, the others from L1), Yt = Y T^T, and the copies of both (17 us for eight
// matrices up to m' = 512; six kernels a matrix, 29 us together).
__global__ void __launch_bounds__(256) tail_rows_kernel(const __grid_constant__ TailGroup g) {
    chain_begin();
    __shared__ float Ws[32][33], Ts[32][33], ys[2][32][33];
    const TailMat& M = g.mat[blockIdx.y];
    const int k = M.k, mp = M.mp, tp = M.tp, a0 = blockIdx.x * 32;
    if (a0 >= tp) return;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    for (int e = tid; e < k * k; e += 256) {
        Ws[e / k][e % k] = M.W[e];
        Ts[e / k][e % k] = M.T[e];
    }
    const float sg = lane < k ? M.sign[lane] : 1.f;
    float q[4], y[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int a = a0 + 4 * warp + i;
        q[i] = 0.f; y[i] = 0.f;
        if (a < mp && lane < k) {
            q[i] = M.Q[(size_t)a * k + lane];
            if (sg < 0.f) M.Q[(size_t)a * k + lane] = q[i] = -q[i];
        }
    }
    __syncthreads();
#pragma unroll 1
    for (int l = 0; l < k; ++l) {
        const float w = lane < l ? Ws[lane][l] : 0.f, d = Ws[l][l];
        float acc[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) acc[i] = lane < l ? fmaf(y[i], w, 0.f) : 0.f;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
#pragma unroll
            for (int i = 0; i < 4; ++i) acc[i] += __shfl_xor_sync(0xffffffffu, acc[i], o);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float val = (-__shfl_sync(0xffffffffu, q[i], l) - acc[i]) / d;
            if (lane == l) y[i] = val;
        }
    }
    float yt[4] = {};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int a = a0 + 4 * warp + i;
        if (a < k) y[i] = lane < a ? Ws[a][lane] : lane == a ? 1.f : 0.f;
        if (a >= mp || lane >= k) y[i] = 0.f;
    }
#pragma unroll 4
    for (int c = 0; c < k; ++c) {
        const float t = lane < k ? Ts[lane][c] : 0.f;
#pragma unroll
        for (int i = 0; i < 4; ++i) yt[i] = fmaf(__shfl_sync(0xffffffffu, y[i], c), t, yt[i]);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        ys[0][4 * warp + i][lane] = y[i];
        ys[1][4 * warp + i][lane] = lane < k ? yt[i] : 0.f;
    }
    __syncthreads();
    const int rows = mp - a0 < 32 ? mp - a0 : 32;          // may be <= 0: padding only
    for (int e = tid; e < rows * k; e += 256) {
        M.Y[(size_t)a0 * k + e] = ys[0][e / k][e % k];
        M.Yt[(size_t)a0 * k + e] = ys[1][e / k][e % k];
    }
    for (int c = warp; c < k; c += 8)
        if (a0 + lane < tp) {
            M.YT[(size_t)c * tp + a0 + lane] = ys[0][lane][c];
            M.YtT[(size_t)c * tp + a0 + lane] = ys[1][lane][c];
        }
    if (!M.YF) return;
    const int KT = (k + 7) / 8, up = (mp + 7) & ~7, frows = up - a0 < 32 ? up - a0 : 32;
    for (int e = tid; e < frows * KT * 8; e += 256) {
        int r, c;
        frag_coord(e, KT, 0, r, c);
        M.YF[(size_t)a0 * KT * 8 + e] = ys[0][r][c];
        frag_coord(e, KT, 1, r, c);
        M.YtF[(size_t)a0 * KT * 8 + e] = ys[1][r][c];
    }
}
}  // namespace

cudaError_t finish_group(const FinishGroup& g, int stage, cudaStream_t st) {
    if (g.nmat <= 0) return cudaSuccess;
    int kmax = 0;
    for (int i = 0; i < g.nmat; ++i) {
        kmax = g.mat[i].k > kmax ? g.mat[i].k : kmax;
        if (stage == 2 && (g.mat[i].k > CB * kCholMaxBlocks || g.mat[i].k % 4)) return cudaErrorInvalidValue;
    }
    if (stage == 1) {                                   // column signs of Q
        launch_chain(fix_signs_group_kernel, dim3((kmax + 31) / 32, g.nmat), 1024, 0, st, g);
    } else {                                            // Householder top block
        const cudaError_t ea = cudaFuncSetAttribute(hh_lu_group_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kHhSmem);
        if (ea != cudaSuccess) return ea;
        launch_chain(hh_lu_group_kernel, g.nmat, CWARPS * 32, kHhSmem, st, g);
    }
    return cudaGetLastError();
}

cudaError_t tail_group(const TailGroup& g, int stage, cudaStream_t st) {
    if (g.nmat <= 0) return cudaSuccess;
    int kmax = 0, tp = 0;
    for (int i = 0; i < g.nmat; ++i) {
        if (g.mat[i].k < 1 || g.mat[i].k > 32) return cudaErrorInvalidValue;
        kmax = g.mat[i].k > kmax ? g.mat[i].k : kmax;
        tp = g.mat[i].tp > tp ? g.mat[i].tp : tp;
    }
    if (stage == 0) launch_chain(tail_ritz_kernel, g.nmat, tail_threads(kmax), 0, st, g);
    else if (stage == 2) launch_chain(tail_rows_kernel, dim3((tp + 31) / 32, g.nmat), 256, 0, st, g);
    else if (kmax <= 16) launch_chain(tail_top_kernel<16>, g.nmat, 1024, 0, st, g);
    else launch_chain(tail_top_kernel<32>, g.nmat, 1024, 0, st, g);
    return cudaGetLastError();
}

cudaError_t chol_group(const CholGroup& g, cudaStream_t st) {
    if (g.nmat <= 0) return cudaSuccess;
    int nmax = 0;
    for (int i = 0; i < g.nmat; ++i) {
        if (g.mat[i].n < 1 || g.mat[i].n > 256 || g.mat[i].ld < g.mat[i].n) return cudaErrorInvalidValue;
        nmax = g.mat[i].n > nmax ? g.mat[i].n : nmax;
    }
    const int nb = (nmax + CB - 1) / CB;
    const size_t smem = sizeof(float) * CBLK * (nb * (nb + 1) / 2 + nb);
    {   // per device: set on every call (cheap next to the launch)
        const cudaError_t ea = cudaFuncSetAttribute(chol_group_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                   (int)kCholSmem);
        if (ea != cudaSuccess) return ea;
    }
    launch_chain(chol_group_kernel, g.nmat, CWARPS * 32, smem, st, g);
    return cudaGetLastError();
}

cudaError_t chol_inverse(const float* G, int n, float* S, int* flag, cudaStream_t st) {
    if (n < 1 || n > 256) return cudaErrorInvalidValue;
    const size_t smem = sizeof(float) * ((size_t)n * (n + 1) / 2 + 2 * n);
    // the largest factor (n = 256) and its temporaries, below the per-CTA limit with the
    // kernel's few static bytes
    {   // per device: set on every call (cheap next to the launch)
        const cudaError_t ea = cudaFuncSetAttribute(chol_inverse_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                   (int)(sizeof(float) * (256 * 257 / 2 + 2 * 256)));
        if (ea != cudaSuccess) return ea;
    }
    chol_inverse_kernel<<<1, 1024, smem, st>>>(G, n, S, flag);
    return cudaGetLastError();
}

cudaError_t cholesky(float* A, int n, float* scratch, int* flag, cudaStream_t st) {
    cholesky_kernel<<<1, 1024, 0, st>>>(A, n, scratch, flag);
    return cudaGetLastError();
}

cudaError_t trsm_right_lt(float* Q, int rows, int n, const float* L, cudaStream_t st) {
    trsm_kernel<<<(rows + 7) / 8, 256, 0, st>>>(Q, rows, n, L);
    return cudaGetLastError();
}

cudaError_t random_block(float* Q, int rows, int cols, uint64_t seed, uint32_t t, cudaStream_t st) {
    const int64_t total = (int64_t)rows * ((cols + 3) / 4);
    random_block_kernel<<<(unsigned)((total + 255) / 256), 256, 0, st>>>(Q, rows, cols, seed, t);
    return cudaGetLastError();
}

cudaError_t householder_reconstruct(const float* Q, int mp, int k, float* Y, float* T, float* s,
                                    float* scratch, cudaStream_t st) {
    hh_top_kernel<<<1, 1024, 0, st>>>(Q, k, scratch, Y, T, s);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    if (mp <= k) return e;
    ++more_launches;
    hh_rows_kernel<<<(mp - k + 7) / 8, 256, 0, st>>>(Q, mp, k, scratch, Y);
    return cudaGetLastError();
}

cudaError_t materialize_wy_basis(int mp, int k, const float* Y, const float* Yt, const float* dsign,
                                 float* U, cudaStream_t st) {
    const int64_t total = (int64_t)mp * mp;
    wy_basis_kernel<<<(unsigned)((total + 255) / 256), 256, 0, st>>>(mp, k, Y, Yt, dsign, U);
    return cudaGetLastError();
}

}  // namespace glr
