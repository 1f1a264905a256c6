// Streaming kernels of the GreedyLore step: the error-feedback compose pass (K1), the
// decompress + optimizer pass (K3), the deferred error materialisation, and a generic
// strided fp32 GEMM used by the small projections and the refresh.
#include "glr_internal.cuh"

namespace glr {

// ------------------------------------------------------------------------------------------
// Generic strided batched SGEMM: 64 x 64 output tile, K chunks of 16, 256 threads, 4 x 4
// outputs per thread.  Operand tiles are staged through shared memory with the load order
// chosen from the unit stride so global reads coalesce.
// ------------------------------------------------------------------------------------------
namespace {
constexpr int GB_M = 64, GB_N = 64, GB_K = 16;

// 64 x 64 tile (i0, j0) of A B over [kbeg, kend): the next two slabs' elements are on their way to
// registers while the current one is multiplied (one barrier a slab); every output is one fma chain
// over k ascending.  Without prefetch a slab of 16 waited out the whole load latency (3.4 us), with one
// slab ahead still half of it where a product has fewer tiles than SMs, and the warps past a thin
// product's rows took their share of the shared-memory reads (four 333 x 777 layers, r = 5: a step
// 141 -> 111 us with two slabs ahead and those warps idle).
struct GemmTile {
    const float* A; int64_t sAi, sAp;
    const float* B; int64_t sBp, sBj;
    int M, N;
};
using f32x2 = unsigned long long;
__device__ __forceinline__ f32x2 pack2(float lo, float hi) {
    f32x2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void gemm_tile(const GemmTile& g, int i0, int j0, int kbeg, int kend, float (&acc)[4][4]) {
    __shared__ __align__(16) float As[2][GB_K][GB_M + 4], Bs[2][GB_K][GB_N + 4];
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    const bool ai = g.sAi == 1, bj = g.sBj == 1;            // consecutive threads along the contiguous index
    const int aii = ai ? tid & 63 : tid / GB_K, app = ai ? tid >> 6 : tid % GB_K;
    const int bjj = bj ? tid & 63 : tid / GB_K, bpp = bj ? tid >> 6 : tid % GB_K;
    constexpr int NL = GB_K / 4, IS = 256 / GB_K;           // elements a thread; index step along i or j
    float ra[2][NL], rb[2][NL];                             // two slabs on their way
    f32x2 c[4][2] = {};
    const bool rows = i0 + (tid >> 5) * 8 < g.M;            // a warp whose eight rows are past M only stages
    auto load = [&](int p0, float (&ra)[NL], float (&rb)[NL]) {
#pragma unroll
        for (int u = 0; u < NL; ++u) {
            const int ii = ai ? aii : aii + IS * u, pa = p0 + (ai ? app + 4 * u : app);
            ra[u] = i0 + ii < g.M && pa < kend ? g.A[(int64_t)(i0 + ii) * g.sAi + (int64_t)pa * g.sAp] : 0.f;
            const int jj = bj ? bjj : bjj + IS * u, pb = p0 + (bj ? bpp + 4 * u : bpp);
            rb[u] = j0 + jj < g.N && pb < kend ? g.B[(int64_t)pb * g.sBp + (int64_t)(j0 + jj) * g.sBj] : 0.f;
        }
    };
    if (kbeg < kend) load(kbeg, ra[0], rb[0]);
    if (kbeg + GB_K < kend) load(kbeg + GB_K, ra[1], rb[1]);
    for (int p0 = kbeg; p0 < kend; p0 += 2 * GB_K) {
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            const int ps = p0 + s * GB_K;
            if (ps >= kend) break;
#pragma unroll
            for (int u = 0; u < NL; ++u) {
                As[s][ai ? app + 4 * u : app][ai ? aii : aii + IS * u] = ra[s][u];
                Bs[s][bj ? bpp + 4 * u : bpp][bj ? bjj : bjj + IS * u] = rb[s][u];
            }
            __syncthreads();                                // the other buffer is read up to here
            if (ps + 2 * GB_K < kend) load(ps + 2 * GB_K, ra[s], rb[s]);
            if (!rows) continue;
#pragma unroll
            for (int p = 0; p < GB_K; ++p) {
                const float4 a = *reinterpret_cast<const float4*>(&As[s][p][ty * 4]);
                const ulonglong2 b = *reinterpret_cast<const ulonglong2*>(&Bs[s][p][tx * 4]);
                const float av[4] = {a.x, a.y, a.z, a.w};
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const f32x2 aa = pack2(av[u], av[u]);
                    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(c[u][0]) : "l"(aa), "l"(b.x));
                    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(c[u][1]) : "l"(aa), "l"(b.y));
                }
            }
        }
    }
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int v = 0; v < 2; ++v) asm("mov.b64 {%0, %1}, %2;" : "=f"(acc[u][2 * v]), "=f"(acc[u][2 * v + 1]) : "l"(c[u][v]));
}

__global__ void __launch_bounds__(256) gemm_f32_kernel(GemmDesc d, int kchunk) {
    chain_begin();
    const bool split = kchunk > 0;                  // blockIdx.z = K slice (batch == 1)
    const int z = split ? 0 : blockIdx.z;
    float* C = d.C + z * d.sCz;
    const int i0 = blockIdx.y * GB_M, j0 = blockIdx.x * GB_N;
    const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
    const int kbeg = split ? blockIdx.z * kchunk : 0;
    const int kend = split ? min(d.K, kbeg + kchunk) : d.K;
    const GemmTile g{d.A + z * d.sAz, d.sAi, d.sAp, d.B + z * d.sBz, d.sBp, d.sBj, d.M, d.N};
    float acc[4][4];
    gemm_tile(g, i0, j0, kbeg, kend, acc);
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const int gi = i0 + ty * 4 + u;
        if (gi >= d.M) continue;
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            const int gj = j0 + tx * 4 + v;
            if (gj >= d.N) continue;
            if (split) {
                d.ws[((int64_t)blockIdx.z * d.M + gi) * d.N + gj] = acc[u][v];
                continue;
            }
            float* c = C + gi * d.sCi + gj * d.sCj;
            const float val = d.alpha * acc[u][v];
            *c = d.beta == 0.f ? val : fmaf(d.beta, *c, val);
        }
    }
}

// C = alpha * sum_z ws[z] + beta * C, slices added in order.
__global__ void gemm_splitk_reduce(GemmDesc d, int splits) {
    chain_begin();
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= (int64_t)d.M * d.N) return;
    const int i = static_cast<int>(e / d.N), j = static_cast<int>(e % d.N);
    float acc = 0.f;
    for (int zz = 0; zz < splits; ++zz) acc += d.ws[(int64_t)zz * d.M * d.N + e];
    float* c = d.C + i * d.sCi + j * d.sCj;
    const float val = d.alpha * acc;
    *c = d.beta == 0.f ? val : fmaf(d.beta, *c, val);
}
}  // namespace

cudaError_t gemm_f32(const GemmDesc& d, cudaStream_t st) {
    if (d.M <= 0 || d.N <= 0 || d.batch <= 0) { --more_launches; return cudaSuccess; }
    const int tiles = ((d.N + GB_N - 1) / GB_N) * ((d.M + GB_M - 1) / GB_M);
    int splits = 1;
    if (d.batch == 1 && d.ws && tiles < 148 && d.K >= 512) {
        splits = d.K / 256;
        splits = splits < 296 / tiles ? splits : 296 / tiles;
        const int64_t fit = d.ws_floats / ((int64_t)d.M * d.N);
        splits = (int64_t)splits < fit ? splits : (int)fit;
    }
    if (splits > 1) {
        const int kchunk = ((d.K + splits - 1) / splits + GB_K - 1) / GB_K * GB_K;
        splits = (d.K + kchunk - 1) / kchunk;
        dim3 grid((d.N + GB_N - 1) / GB_N, (d.M + GB_M - 1) / GB_M, splits);
        gemm_f32_kernel<<<grid, 256, 0, st>>>(d, kchunk);
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
        const int64_t total = (int64_t)d.M * d.N;
        ++more_launches;
        launch_chain(gemm_splitk_reduce, (unsigned)((total + 255) / 256), 256, 0, st, d, splits);
        return cudaGetLastError();
    }
    dim3 grid((d.N + GB_N - 1) / GB_N, (d.M + GB_M - 1) / GB_M, d.batch);
    gemm_f32_kernel<<<grid, 256, 0, st>>>(d, 0);
    return cudaGetLastError();
}

// ------------------------------------------------------------------------------------------
// K1 compose.  A 32 x 32 tile of the oriented m' x n' layout per CTA (32 x 8 threads, four
// rows per thread).  The tile's rows of Pprev (32 x r) stay in shared memory for all nodes;
// node i's columns of Rw_i (r x 32) and its G tile (transposed through shared memory when
// m > n) are staged per node.  The node sum is kept in registers.
// ------------------------------------------------------------------------------------------
namespace {
constexpr int CT = 32;

__global__ void __launch_bounds__(256) compose_kernel(const __grid_constant__ ComposeGroup g) {
    chain_begin();
    int mi = 0;
    while (mi + 1 < g.nmat && g.tile0[mi + 1] <= (int)blockIdx.x) ++mi;
    const ComposeArgs& a = g.mat[mi];
    const int tiles_b = (a.np + CT - 1) / CT, lt = (int)blockIdx.x - g.tile0[mi];
    extern __shared__ float sm[];
    float* Ps = sm;                       // CT x r
    float* Rs = Ps + CT * a.r;            // r x CT
    float* Gs = Rs + a.r * CT;            // CT x (CT + 1)
    const int a0 = lt / tiles_b * CT, b0 = lt % tiles_b * CT;
    const int tx = threadIdx.x, ty = threadIdx.y, tid = ty * CT + tx;
    const bool corr = !a.e_zero;
    if (corr) {
        for (int e = tid; e < CT * a.r; e += 256) {
            const int aa = e / a.r, q = e % a.r;
            Ps[e] = (a0 + aa < a.mp) ? a.Pprev[(int64_t)(a0 + aa) * a.r + q] : 0.f;
        }
    }
    float sum[4] = {0.f, 0.f, 0.f, 0.f};
    for (int i = 0; i < a.N; ++i) {
        const void* G = a.G[i];
        float* Bi = a.B + (int64_t)i * a.mp * a.np;
        float old[4] = {0.f, 0.f, 0.f, 0.f};     // in flight together with the tiles below
        if (corr) {
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int aa = a0 + ty + 8 * u, b = b0 + tx;
                if (aa < a.mp && b < a.np) old[u] = Bi[(int64_t)aa * a.np + b];
            }
        }
        if (a.transposed) {       // G_i(a, b) = G_i[b * m' + a]: read along a
            for (int rr = ty; rr < CT; rr += 8) {
                const int b = b0 + rr, aa = a0 + tx;
                Gs[tx * (CT + 1) + rr] = (b < a.np && aa < a.mp) ? load_grad(G, (int64_t)b * a.mp + aa, a.grad_dtype) : 0.f;
            }
        } else {
            for (int rr = ty; rr < CT; rr += 8) {
                const int aa = a0 + rr, b = b0 + tx;
                Gs[rr * (CT + 1) + tx] = (aa < a.mp && b < a.np) ? load_grad(G, (int64_t)aa * a.np + b, a.grad_dtype) : 0.f;
            }
        }
        if (corr) {
            const float* Rw = a.Rw + (int64_t)i * a.r * a.np;
            for (int e = tid; e < a.r * CT; e += 256) {
                const int q = e / CT, bb = e % CT;
                Rs[e] = (b0 + bb < a.np) ? Rw[(int64_t)q * a.np + b0 + bb] : 0.f;
            }
        }
        __syncthreads();
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int rr = ty + 8 * u, aa = a0 + rr, b = b0 + tx;
            if (aa >= a.mp || b >= a.np) continue;
            float mval = Gs[rr * (CT + 1) + tx];
            const int64_t idx = (int64_t)aa * a.np + b;
            if (corr) {
                float c = 0.f;
                for (int q = 0; q < a.r; ++q) c = fmaf(Ps[rr * a.r + q], Rs[q * CT + tx], c);
                mval += old[u] - c;
            }
            if (a.write_B) Bi[idx] = mval;
            sum[u] += mval;
        }
        __syncthreads();
    }
    const float invN = 1.0f / static_cast<float>(a.N);
    bool bad = false;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const int aa = a0 + ty + 8 * u, b = b0 + tx;
        if (aa < a.mp && b < a.np) {
            a.Mbar[(int64_t)aa * a.np + b] = sum[u] * invN;
            bad |= !isfinite(sum[u]);
        }
    }
    flag_nonfinite(bad, a.nonfinite);
}
}  // namespace

cudaError_t compose(ComposeGroup& g, cudaStream_t st) {
    if (g.nmat <= 0) return cudaSuccess;
    int tiles = 0, r = 0;
    for (int i = 0; i < g.nmat; ++i) {
        const auto& a = g.mat[i];
        g.tile0[i] = tiles;
        tiles += ((a.np + CT - 1) / CT) * ((a.mp + CT - 1) / CT);
        r = a.r > r ? a.r : r;
    }
    const size_t smem = sizeof(float) * (2 * CT * r + CT * (CT + 1));
    {   // per device: set on every call (cheap next to the launch)
        const cudaError_t ea = cudaFuncSetAttribute(compose_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 160 * 1024);
        if (ea != cudaSuccess) return ea;
    }
    compose_kernel<<<tiles, dim3(CT, 8), smem, st>>>(g);
    return cudaGetLastError();
}

// ------------------------------------------------------------------------------------------
// K3 decompress + optimizer.  Ghat for a 32 x 32 oriented tile is formed with coalesced reads
// into shared memory, then X / M / V are updated in X's own layout (transposed when m > n).
// ------------------------------------------------------------------------------------------
namespace {
__global__ void __launch_bounds__(256) update_kernel(const __grid_constant__ UpdateTileGroup grp) {
    chain_begin();
    int mi = 0;
    while (mi + 1 < grp.nmat && grp.tile0[mi + 1] <= (int)blockIdx.x) ++mi;
    const UpdateArgs& a = grp.mat[mi];
    const int tiles_b = (a.np + CT - 1) / CT, lt = (int)blockIdx.x - grp.tile0[mi];
    extern __shared__ float sm[];
    float* Ps = sm;                       // CT x r
    float* Rs = Ps + CT * a.r;            // r x CT
    float* Gt = Rs + a.r * CT;            // CT x (CT + 1)
    const int a0 = lt / tiles_b * CT, b0 = lt % tiles_b * CT;
    const int tx = threadIdx.x, ty = threadIdx.y, tid = ty * CT + tx;
    if (a.compressed) {
        for (int e = tid; e < CT * a.r; e += 256) {
            const int aa = e / a.r, q = e % a.r;
            Ps[e] = (a0 + aa < a.mp) ? a.P[(int64_t)(a0 + aa) * a.r + q] : 0.f;
        }
        for (int e = tid; e < a.r * CT; e += 256) {
            const int q = e / CT, bb = e % CT;
            Rs[e] = (b0 + bb < a.np) ? a.Rbar[(int64_t)q * a.np + b0 + bb] : 0.f;
        }
        __syncthreads();
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const int rr = ty + 8 * u, aa = a0 + rr, b = b0 + tx;
        float g = 0.f;
        if (aa < a.mp && b < a.np) {
            if (a.compressed) {
                for (int q = 0; q < a.r; ++q) g = fmaf(Ps[rr * a.r + q], Rs[q * CT + tx], g);
            } else {
                g = a.Mbar[(int64_t)aa * a.np + b];
            }
        }
        Gt[rr * (CT + 1) + tx] = g;
    }
    __syncthreads();
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const int rr = ty + 8 * u;
        int64_t xi;
        float g;
        if (a.transposed) {   // X is n' x m' (m > n): X[b][a], contiguous along a
            const int b = b0 + rr, aa = a0 + tx;
            if (b >= a.np || aa >= a.mp) continue;
            xi = (int64_t)b * a.mp + aa;
            g = Gt[tx * (CT + 1) + rr];
        } else {
            const int aa = a0 + rr, b = b0 + tx;
            if (aa >= a.mp || b >= a.np) continue;
            xi = (int64_t)aa * a.np + b;
            g = Gt[rr * (CT + 1) + tx];
        }
        const float m1 = fmaf(a.beta1, a.Mo[xi], (1.0f - a.beta1) * g);
        a.Mo[xi] = m1;
        if (a.optimizer == GLR_ADAM) {
            const float v1 = fmaf(a.beta2, a.Vo[xi], (1.0f - a.beta2) * g * g);
            a.Vo[xi] = v1;
            a.X[xi] -= a.lr * m1 / (sqrtf(v1) + a.eps);
        } else {
            a.X[xi] -= a.lr * m1;
        }
    }
}

__global__ void __launch_bounds__(256) error_kernel(int mp, int np, int r, int e_zero, const float* B,
                                                    const float* Pprev, const float* Rw, float* E) {
    const int64_t idx = (int64_t)blockIdx.x * 256 + threadIdx.x;
    if (idx >= (int64_t)mp * np) return;
    if (e_zero) { E[idx] = 0.f; return; }
    const int aa = static_cast<int>(idx / np), b = static_cast<int>(idx % np);
    float c = 0.f;
    for (int q = 0; q < r; ++q) c = fmaf(Pprev[(int64_t)aa * r + q], Rw[(int64_t)q * np + b], c);
    E[idx] = B[idx] - c;
}
}  // namespace

cudaError_t update(UpdateTileGroup& g, cudaStream_t st) {
    if (g.nmat <= 0) return cudaSuccess;
    int tiles = 0, r = 0;
    for (int i = 0; i < g.nmat; ++i) {
        const auto& a = g.mat[i];
        g.tile0[i] = tiles;
        tiles += ((a.np + CT - 1) / CT) * ((a.mp + CT - 1) / CT);
        r = a.r > r ? a.r : r;
    }
    const size_t smem = sizeof(float) * (2 * CT * r + CT * (CT + 1));
    {   // per device: set on every call (cheap next to the launch)
        const cudaError_t ea = cudaFuncSetAttribute(update_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 160 * 1024);
        if (ea != cudaSuccess) return ea;
    }
    update_kernel<<<tiles, dim3(CT, 8), smem, st>>>(g);
    return cudaGetLastError();
}

cudaError_t materialize_error(int mp, int np, int r, int e_zero, const float* B, const float* Pprev,
                              const float* Rw, float* E, cudaStream_t st) {
    const int64_t total = (int64_t)mp * np;
    error_kernel<<<(unsigned)((total + 255) / 256), 256, 0, st>>>(mp, np, r, e_zero, B, Pprev, Rw, E);
    return cudaGetLastError();
}

}  // namespace glr

// ------------------------------------------------------------------------------------------
// Grouped fp32 products (the refresh's k-wide fp32 steps: Gram matrices, CholeskyQR's X L^{-T},
// the Rayleigh-Ritz rotation Q W, Yt = Y T^T): a 64 x 64 output tile per CTA of 256 threads, each
// thread a 4 x 4 block, K staged through shared memory 16 at a time; sums in a fixed order.
// ------------------------------------------------------------------------------------------
namespace glr {
namespace {

// K elements of a slice: whole slabs.
__host__ __device__ __forceinline__ int gemm_chunk(const GemmMat& M) {
    return ((M.K + M.splits - 1) / M.splits + GB_K - 1) / GB_K * GB_K;
}

__global__ void __launch_bounds__(256) gemm_group_kernel(const __grid_constant__ GemmGroup g) {
    chain_begin();
    const int tile = blockIdx.x;
    int lo = 0, hi = g.nmat - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (g.mat[mid].tile0 <= tile) lo = mid; else hi = mid - 1;
    }
    const GemmMat& M = g.mat[lo];
    const int tn = (M.N + 63) / 64, tiles = tn * ((M.M + 63) / 64);
    const int lt = (tile - M.tile0) % tiles, z = (tile - M.tile0) / tiles;
    const int i0 = (lt / tn) * 64, j0 = (lt % tn) * 64;
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    const int chunk = gemm_chunk(M), kend = min(M.K, (z + 1) * chunk);
    const GemmTile t{M.A, M.sAi, M.sAp, M.B, M.sBp, M.sBj, M.M, M.N};
    float acc[4][4];
    gemm_tile(t, i0, j0, z * chunk, kend, acc);
    const float alpha = M.alpha != 0.f ? M.alpha : 1.f;
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            const int i = i0 + ty * 4 + u, j = j0 + tx * 4 + v;
            if (i >= M.M || j >= M.N) continue;
            if (M.splits > 1) M.ws[((int64_t)z * M.M + i) * M.N + j] = acc[u][v];
            else M.C[(int64_t)i * M.sCi + (int64_t)j * M.sCj] = alpha * acc[u][v];
        }
}

// C = alpha times the sum of the K slices, added in order.
__global__ void __launch_bounds__(256) gemm_group_reduce(const __grid_constant__ GemmGroup g) {
    chain_begin();
    const GemmMat& M = g.mat[blockIdx.y];
    if (M.splits <= 1) return;
    const float alpha = M.alpha != 0.f ? M.alpha : 1.f;
    const int64_t mn = (int64_t)M.M * M.N;
    for (int64_t e = (int64_t)blockIdx.x * 256 + threadIdx.x; e < mn; e += (int64_t)gridDim.x * 256) {
        float acc = 0.f;
        for (int z = 0; z < M.splits; ++z) acc += M.ws[z * mn + e];
        M.C[(e / M.N) * M.sCi + (e % M.N) * M.sCj] = alpha * acc;
    }
}

}  // namespace

cudaError_t gemm_group_f32(GemmGroup& g, cudaStream_t st) {
    g.total_tiles = 0;
    bool reduce = false;
    for (int i = 0; i < g.nmat; ++i) {
        GemmMat& M = g.mat[i];
        const int tiles = ((M.M + 63) / 64) * ((M.N + 63) / 64);
        // long products with few tiles (a Gram matrix: 16 tiles, K = 4096) in K slices of at least 256, by
        // the product's own sizes so that its sums do not depend on the group: 677 -> about 60 us there
        M.splits = 1;
        if (M.ws && tiles <= 16 && M.K >= 512) {
            M.splits = M.K / 256 < 16 ? M.K / 256 : 16;
            while ((int64_t)M.splits * M.M * M.N > kGemmWsFloats) --M.splits;
            if (M.splits < 1) M.splits = 1;
        }
        if (M.splits > 1) M.splits = (M.K + gemm_chunk(M) - 1) / gemm_chunk(M);
        reduce = reduce || M.splits > 1;
        M.tile0 = g.total_tiles;
        g.total_tiles += tiles * M.splits;
    }
    if (g.total_tiles <= 0) { --more_launches; return cudaSuccess; }
    gemm_group_kernel<<<g.total_tiles, 256, 0, st>>>(g);
    if (reduce) {
        ++more_launches;
        launch_chain(gemm_group_reduce, dim3(64, g.nmat), 256, 0, st, g);
    }
    return cudaGetLastError();
}

}  // namespace glr
