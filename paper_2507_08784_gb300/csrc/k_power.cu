// Grouped block power iteration for the truncated-basis refresh (the Semi-Lazy SVD of Eq.
// SVD-P1 restricted to the top-k subspace): every refreshing matrix of a step advances together,
// one launch per stage.  One half-iteration is one pass over Mbar:
//   Z = (Mbar^T Q) S        (pow_t_kernel, column tiles of Mbar)        then S <- chol(Z^T Z)^-1
//   Q = (Mbar Z) S          (pow_n_kernel split-K partials, pow_r_kernel) then S <- chol(Q^T Q)^-1
// where S (k x k) is the inverse Cholesky factor that orthonormalises the previous iterate
// (CholeskyQR, Yamamoto et al. 2015), applied to the small output instead of the tall input:
// Mbar^T (Q S) = (Mbar^T Q) S.  The Gram matrices are summed from per-tile partials in a fixed
// order in fp64 and factored by one CTA per matrix (pow_chol_kernel).  The final CholeskyQR2
// uses pow_apply_kernel; the Rayleigh-Ritz Gram H = Z^T Z comes out of pow_t_kernel the same way.
#include <cooperative_groups.h>

#include "glr_internal.cuh"

namespace glr {

namespace {

constexpr int TP = 256;                // threads per CTA (pow_r_kernel, pow_apply_kernel)
constexpr int TM = 128;                // threads per CTA of the products
constexpr int PC = 64;                 // columns of Mbar per tile / split-K chunk, rows per row tile
constexpr int PR = 32;                 // rows of Mbar per staged block (pow_t_kernel)
constexpr int PS = 6;                  // staged blocks in flight (pow_t_kernel)
constexpr int NCH = 512;               // columns per split-K chunk (pow_n_kernel)
constexpr int NR = 32;                 // rows per CTA (pow_n_kernel)
constexpr int NS = 4;                  // its staged 32 x 64 blocks in flight
constexpr int NP = PC + 4;             // their row pitch: 16-byte rows, no bank conflicts down a column of float4

// 16 or 4 bytes into shared memory asynchronously, zeros where !in (src is not read then).
__device__ __forceinline__ void cp16(void* dst, const float* src, bool in) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(
                     static_cast<uint32_t>(__cvta_generic_to_shared(dst))), "l"(src), "r"(in ? 16 : 0) : "memory");
}
__device__ __forceinline__ void cp4(void* dst, const float* src, bool in) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(
                     static_cast<uint32_t>(__cvta_generic_to_shared(dst))), "l"(src), "r"(in ? 4 : 0) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// Gram partial of the 64 x KM block Zs (rows < nrows valid) into gout (KM x KM, row-major), a 2 x 2 block of
// entries at a time.
template <int KM, int NT>
__device__ __forceinline__ void gram_partial(const float* Zs, int nrows, float* gout) {
    constexpr int KH = KM / 2;
    for (int o = threadIdx.x; o < KH * KH; o += NT) {
        const int a = 2 * (o / KH), b = 2 * (o % KH);
        float s00 = 0.f, s01 = 0.f, s10 = 0.f, s11 = 0.f;
#pragma unroll 8
        for (int c = 0; c < nrows; ++c) {
            const float2 x = *reinterpret_cast<const float2*>(Zs + c * KM + a);
            const float2 y = *reinterpret_cast<const float2*>(Zs + c * KM + b);
            s00 = fmaf(x.x, y.x, s00); s01 = fmaf(x.x, y.y, s01);
            s10 = fmaf(x.y, y.x, s10); s11 = fmaf(x.y, y.y, s11);
        }
        *reinterpret_cast<float2*>(gout + a * KM + b) = make_float2(s00, s01);
        *reinterpret_cast<float2*>(gout + (a + 1) * KM + b) = make_float2(s10, s11);
    }
}

// out (64 x KM block in smem, rows < nrows) <- in S (KM x KM in smem), into out (may alias
// nothing).  A thread computes KM / 4 entries of a row.
template <int KM, int NT>
__device__ __forceinline__ void apply_S(const float* in, const float* S, float* out) {
    constexpr int KPT = KM / 4;
    const int row = threadIdx.x & 63;
    for (int kq = threadIdx.x >> 6; kq < 4; kq += NT / 64) {
        float acc[KPT];
#pragma unroll
        for (int e = 0; e < KPT; ++e) acc[e] = 0.f;
#pragma unroll 8
        for (int l = 0; l < KM; ++l) {
            const float v = in[row * KM + l];
#pragma unroll
            for (int e = 0; e < KPT; ++e) acc[e] = fmaf(v, S[l * KM + kq * KPT + e], acc[e]);
        }
#pragma unroll
        for (int e = 0; e < KPT; ++e) out[row * KM + kq * KPT + e] = acc[e];
    }
}

template <int KM> constexpr size_t kPowTSmem = sizeof(float) * PS * (PR * PC + PR * KM);
template <int KM> constexpr size_t kPowNSmem = sizeof(float) * NS * (NR * NP + PC * KM);

// Z[c][:] = (sum_a Mbar[a][c] Q[a][:]) (S if apply_s), for a tile of 64 columns; Gram partial of
// the tile's rows of Z into G[tile].  Bound by what shared memory can return to registers (6 floats a
// thread for 8 products) and its latency: six blocks of 32 rows in flight by cp.async, a thread two
// columns by KM / 4, a few rows' reads issued together (conv stack, k = 16: 23.4 -> 18.5 us a pass;
// four columns a thread on half the warps 20.5).
template <int KM>
__global__ void __launch_bounds__(TM) pow_t_kernel(const __grid_constant__ PowGroup g, int apply_s) {
    chain_begin();
    constexpr int KPT = KM / 4, RB = KM == 16 ? 8 : 4;
    extern __shared__ __align__(16) float stage[];             // PS blocks of PR x PC of Mbar, then of PR x KM of Q
    __shared__ __align__(16) float Zs[PC * KM];
    __shared__ __align__(16) float Z2[PC * KM];
    __shared__ __align__(16) float Ss[KM * KM];
    int mi = 0;
    while (mi + 1 < g.nmat && blockIdx.x >= static_cast<unsigned>(g.mat[mi + 1].t0)) ++mi;
    const PowMat& M = g.mat[mi];
    if (!M.active) return;
    const int tile = blockIdx.x - M.t0, c0 = tile * PC;
    const int mp = M.mp, np = M.np, k = M.k;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int cl = 2 * ((lane & 15) + 16 * (warp & 1)), kq = (lane >> 4) + 2 * (warp >> 1);
    float* As = stage;
    float* Xs = stage + PS * PR * PC;
    // this thread's copies of a block: rows tid / 16 + 8 l of Mbar, four columns each; Q's rows are one
    // contiguous piece when k = KM
    const int fr = tid >> 4, fc = 4 * (tid & 15);
    const bool fin = c0 + fc < np;                             // n' % 4 == 0
    const float* fsrc = fin ? M.Mbar + (int64_t)fr * np + c0 + fc : M.Mbar;
    auto fetch = [&](int blk) {                                // block blk of 32 rows
        const int a0 = blk * PR, b = blk % PS;
        if (a0 < mp) {
            const float* src = fin ? fsrc + (int64_t)a0 * np : fsrc;
            float* dst = As + b * PR * PC + fr * PC + fc;
#pragma unroll
            for (int l = 0; l < PR / 8; ++l) {
                const bool in = fin && a0 + fr + 8 * l < mp;
                cp16(dst + 8 * l * PC, in ? src + (int64_t)8 * l * np : M.Mbar, in);
            }
            float* xd = Xs + b * PR * KM;
            if (k == KM) {
#pragma unroll
                for (int l = 0; l < PR * KM / 4 / TM; ++l) {
                    const int o = 4 * (tid + l * TM);
                    const bool in = a0 + o / KM < mp;
                    cp16(xd + o, in ? M.Q + (int64_t)a0 * KM + o : M.Q, in);
                }
            } else {
#pragma unroll
                for (int l = 0; l < PR * KM / TM; ++l) {
                    const int o = tid + l * TM, rr = o / KM, q = o % KM, a = a0 + rr;
                    const bool in = a < mp && q < k;
                    cp4(xd + o, in ? M.Q + (int64_t)a * k + q : M.Q, in);
                }
            }
        }
        cp_commit();
    };
    float acc[2][KPT] = {};
    const int nblk = (mp + PR - 1) / PR;
    for (int i = 0; i < PS - 1; ++i) fetch(i);
    if (apply_s)
        for (int o = tid; o < KM * KM; o += TM) {
            const int a = o / KM, b = o % KM;
            Ss[o] = a < k && b < k ? M.S[a * k + b] : (a == b ? 1.f : 0.f);
        }
    for (int blk = 0; blk < nblk; ++blk) {
        cp_wait<PS - 2>();                                     // this thread's copies of the block, then everyone's
        __syncthreads();
        fetch(blk + PS - 1);                                   // over the block read before the barrier
        const float* A = As + (blk % PS) * PR * PC + cl;
        const float* X = Xs + (blk % PS) * PR * KM + kq * KPT;
#pragma unroll 2
        for (int r0 = 0; r0 < PR; r0 += RB) {                  // RB rows' reads issued together
            float2 m[RB];
            float4 x[RB][KPT / 4];
#pragma unroll
            for (int r = 0; r < RB; ++r) {
                m[r] = *reinterpret_cast<const float2*>(A + (r0 + r) * PC);
#pragma unroll
                for (int e = 0; e < KPT; e += 4) x[r][e / 4] = *reinterpret_cast<const float4*>(X + (r0 + r) * KM + e);
            }
#pragma unroll
            for (int r = 0; r < RB; ++r)
#pragma unroll
                for (int e = 0; e < KPT; e += 4) {
                    const float xv[4] = {x[r][e / 4].x, x[r][e / 4].y, x[r][e / 4].z, x[r][e / 4].w};
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        acc[0][e + j] = fmaf(m[r].x, xv[j], acc[0][e + j]);
                        acc[1][e + j] = fmaf(m[r].y, xv[j], acc[1][e + j]);
                    }
                }
        }
    }
#pragma unroll
    for (int j = 0; j < 2; ++j)
#pragma unroll
        for (int e = 0; e < KPT; ++e) Zs[(cl + j) * KM + kq * KPT + e] = acc[j][e];
    __syncthreads();
    const float* Zo = Zs;
    if (apply_s) {
        apply_S<KM, TM>(Zs, Ss, Z2);
        Zo = Z2;
        __syncthreads();
    }
    const int nrows = np - c0 < PC ? np - c0 : PC;
    for (int o = tid; o < nrows * KM; o += TM) {
        const int c = o / KM, q = o % KM;
        if (q < k) M.Z[(int64_t)(c0 + c) * k + q] = Zo[o];
    }
    gram_partial<KM, TM>(Zo, nrows, M.G + (int64_t)tile * KM * KM);
}

// part[chunk][q][a] = sum over the chunk's NCH columns c of Mbar[a][c] Z[c][q], for one tile of
// 32 rows a: CTA (row tile, chunk), the chunk walked in 64-column blocks, four in flight; a thread holds
// one row by KM / 4 (conv stack: 20.4 -> 16.4 us; 64-row tiles, four rows a thread 20.5).
template <int KM>
__global__ void __launch_bounds__(TM) pow_n_kernel(const __grid_constant__ PowGroup g) {
    chain_begin();
    constexpr int KPT = KM / 4;
    extern __shared__ __align__(16) float stage[];             // NS blocks of NR x NP of Mbar, then of PC x KM of Z
    int mi = 0;
    const int bid = blockIdx.x / (PC / NR);                    // the group counts tiles of 64 rows
    while (mi + 1 < g.nmat && bid >= g.mat[mi + 1].n0) ++mi;
    const PowMat& M = g.mat[mi];
    const int nrt = (M.mp + PC - 1) / PC;
    const int chunk = (bid - M.n0) / nrt, rt = (bid - M.n0) % nrt;
    const int a0 = rt * PC + NR * (blockIdx.x % (PC / NR)), cbeg = chunk * NCH;
    const int mp = M.mp, np = M.np, k = M.k;
    if (!M.active || a0 >= mp) return;
    const int cend = cbeg + NCH < np ? cbeg + NCH : np;
    const int tid = threadIdx.x, lane = tid & 31, kq = tid >> 5;
    float* As = stage;
    float* Ys = stage + NS * NR * NP;
    const int fr = tid >> 4, fc = 4 * (tid & 15);
    const float* fsrc = M.Mbar + (int64_t)(a0 + fr) * np + cbeg + fc;
    auto fetch = [&](int blk) {
        const int c0 = cbeg + blk * PC, b = blk % NS;
        if (c0 < cend) {
            const bool fin = c0 + fc < cend;
            float* dst = As + b * NR * NP + fr * NP + fc;
#pragma unroll
            for (int l = 0; l < NR / 8; ++l) {
                const bool in = fin && a0 + fr + 8 * l < mp;
                cp16(dst + 8 * l * NP, in ? fsrc + (int64_t)8 * l * np + blk * PC : M.Mbar, in);
            }
            float* yd = Ys + b * PC * KM;
            if (k == KM) {
#pragma unroll
                for (int l = 0; l < PC * KM / 4 / TM; ++l) {
                    const int o = 4 * (tid + l * TM);
                    const bool in = c0 + o / KM < cend;
                    cp16(yd + o, in ? M.Z + (int64_t)c0 * KM + o : M.Z, in);
                }
            } else {
#pragma unroll
                for (int l = 0; l < PC * KM / TM; ++l) {
                    const int o = tid + l * TM, cc = o / KM, q = o % KM, c = c0 + cc;
                    const bool in = c < cend && q < k;
                    cp4(yd + o, in ? M.Z + (int64_t)c * k + q : M.Z, in);
                }
            }
        }
        cp_commit();
    };
    float acc[KPT] = {};
    const int nblk = (cend - cbeg + PC - 1) / PC;
    for (int i = 0; i < NS - 1; ++i) fetch(i);
    for (int blk = 0; blk < nblk; ++blk) {
        cp_wait<NS - 2>();
        __syncthreads();
        fetch(blk + NS - 1);
        const float* A = As + (blk % NS) * NR * NP + lane * NP;
        const float* Y = Ys + (blk % NS) * PC * KM + kq * KPT;
#pragma unroll 2
        for (int cc = 0; cc < PC; cc += 8) {                   // eight columns' reads issued together
            const float4 p = *reinterpret_cast<const float4*>(A + cc), q = *reinterpret_cast<const float4*>(A + cc + 4);
            const float m[8] = {p.x, p.y, p.z, p.w, q.x, q.y, q.z, q.w};
            float4 y[8][KPT / 4];
#pragma unroll
            for (int j = 0; j < 8; ++j)
#pragma unroll
                for (int e = 0; e < KPT; e += 4) y[j][e / 4] = *reinterpret_cast<const float4*>(Y + (cc + j) * KM + e);
#pragma unroll
            for (int j = 0; j < 8; ++j)
#pragma unroll
                for (int e = 0; e < KPT; e += 4) {
                    const float4 v = y[j][e / 4];
                    acc[e] = fmaf(m[j], v.x, acc[e]); acc[e + 1] = fmaf(m[j], v.y, acc[e + 1]);
                    acc[e + 2] = fmaf(m[j], v.z, acc[e + 2]); acc[e + 3] = fmaf(m[j], v.w, acc[e + 3]);
                }
        }
    }
    const int a = a0 + lane;
    float* part = M.part + (int64_t)chunk * KM * mp;
    if (a < mp)
#pragma unroll
        for (int e = 0; e < KPT; ++e) part[(int64_t)(kq * KPT + e) * mp + a] = acc[e];
}

// Q[a][:] = (sum over chunks of part[chunk][:][a]) S for a tile of 64 rows; Gram partial into G.
template <int KM>
__global__ void __launch_bounds__(TP) pow_r_kernel(const __grid_constant__ PowGroup g) {
    chain_begin();
    constexpr int KPT = KM / 4;
    __shared__ __align__(16) float Qs[PC * KM];
    __shared__ __align__(16) float Q2[PC * KM];
    __shared__ __align__(16) float Ss[KM * KM];
    int mi = 0;
    while (mi + 1 < g.nmat && blockIdx.x >= static_cast<unsigned>(g.mat[mi + 1].r0)) ++mi;
    const PowMat& M = g.mat[mi];
    if (!M.active) return;
    const int tile = blockIdx.x - M.r0, a0 = tile * PC;
    const int mp = M.mp, k = M.k, nch = M.nn;
    const int tid = threadIdx.x, al = tid & 63, kq = tid >> 6;
    const int a = a0 + al;
    float acc[KPT];
#pragma unroll
    for (int e = 0; e < KPT; ++e) acc[e] = 0.f;
    if (a < mp)
#pragma unroll 8
        for (int ch = 0; ch < nch; ++ch) {                      // fixed order over the chunks
            const float* p = M.part + (int64_t)ch * KM * mp + a;
#pragma unroll
            for (int e = 0; e < KPT; ++e) acc[e] += p[(int64_t)(kq * KPT + e) * mp];
        }
#pragma unroll
    for (int e = 0; e < KPT; ++e) Qs[al * KM + kq * KPT + e] = acc[e];
    for (int o = tid; o < KM * KM; o += TP) {
        const int r = o / KM, c = o % KM;
        Ss[o] = r < k && c < k ? M.S[r * k + c] : (r == c ? 1.f : 0.f);
    }
    __syncthreads();
    apply_S<KM, TP>(Qs, Ss, Q2);
    __syncthreads();
    const int nrows = mp - a0 < PC ? mp - a0 : PC;
    for (int o = tid; o < nrows * KM; o += TP) {
        const int r = o / KM, q = o % KM;
        if (q < k) M.Q[(int64_t)(a0 + r) * k + q] = Q2[o];
    }
    gram_partial<KM, TP>(Q2, nrows, M.G + (int64_t)tile * KM * KM);
}

// Q[a][:] <- Q[a][:] S for a tile of 64 rows (rows are independent: in place); Gram partial
// into G when gram.
template <int KM>
__global__ void __launch_bounds__(TP) pow_apply_kernel(const __grid_constant__ PowGroup g, int gram) {
    chain_begin();
    __shared__ __align__(16) float Qs[PC * KM];
    __shared__ __align__(16) float Q2[PC * KM];
    __shared__ __align__(16) float Ss[KM * KM];
    int mi = 0;
    while (mi + 1 < g.nmat && blockIdx.x >= static_cast<unsigned>(g.mat[mi + 1].r0)) ++mi;
    const PowMat& M = g.mat[mi];
    if (!M.active) return;
    const int tile = blockIdx.x - M.r0, a0 = tile * PC;
    const int mp = M.mp, k = M.k, tid = threadIdx.x;
    const int nrows = mp - a0 < PC ? mp - a0 : PC;
    for (int o = tid; o < PC * KM; o += TP) {
        const int r = o / KM, q = o % KM;
        Qs[o] = r < nrows && q < k ? M.Q[(int64_t)(a0 + r) * k + q] : 0.f;
    }
    for (int o = tid; o < KM * KM; o += TP) {
        const int r = o / KM, c = o % KM;
        Ss[o] = r < k && c < k ? M.S[r * k + c] : (r == c ? 1.f : 0.f);
    }
    __syncthreads();
    apply_S<KM, TP>(Qs, Ss, Q2);
    __syncthreads();
    for (int o = tid; o < nrows * KM; o += TP) {
        const int r = o / KM, q = o % KM;
        if (q < k) M.Q[(int64_t)(a0 + r) * k + q] = Q2[o];
    }
    if (gram) gram_partial<KM, TP>(Q2, nrows, M.G + (int64_t)tile * KM * KM);
}

// Gm = sum over the ntile partials (fp64 accumulation, tile order), then by one CTA
// mode 0: Gm = L L^T (fp32 Cholesky, retried with a growing diagonal shift on breakdown) and
// S = L^{-T}, so X S has orthonormal columns when Gm = X^T X; mode 1: the sum itself into H (the
// Rayleigh-Ritz Gram).  The fp64 additions and conversions of 72 partials took one SM most of 17 us, so a
// cluster of eight CTAs shares a matrix's lower triangle; the first one factors, a column bound by its
// root, quotient and barrier (17 -> 10 us).
constexpr int TCH = 256, CCH = 8;      // threads and CTAs per matrix of pow_chol_kernel

// num / den; a zero numerator (most of the identity's) does not take the division's slow path.
__device__ __forceinline__ float quotient(float num, float den) {
    const float q = (num == 0.f ? 1.f : num) / den;
    return num == 0.f ? num : q;
}

template <int KM>
__global__ void __cluster_dims__(CCH, 1, 1) __launch_bounds__(TCH)
    pow_chol_kernel(const __grid_constant__ PowGroup g, int use_t_tiles, int mode) {
    chain_begin();
    __shared__ float Gs[KM][KM + 1];
    __shared__ float colj[2][KM], rowj[2][KM];
    const PowMat& M = g.mat[blockIdx.x / CCH];
    if (!M.active) return;
    namespace cg = cooperative_groups;
    cg::cluster_group cl = cg::this_cluster();
    const int k = M.k, tid = threadIdx.x, lane = tid & 31, rank = blockIdx.x % CCH;
    const int nt = use_t_tiles ? M.nt : M.nr;
    cl.sync();                                                 // the first CTA's shared memory is there
    float* G0 = cl.map_shared_rank(&Gs[0][0], 0);
    // entry o = a (a + 1) / 2 + b of the sum over the nt partials (the other triangle is the same bits): four
    // threads take the tiles t = j (mod 4), each with two accumulators, and the four slices are
    // added in order
    const int tri = k * (k + 1) / 2;
    for (int w0 = 0; w0 < 4 * tri; w0 += CCH * TCH) {          // a warp's eight entries to each CTA in turn
        const int w = w0 + ((tid >> 5) * CCH + rank) * 32 + (tid & 31), o = w >> 2, j = w & 3;
        int a = 0;
        while ((a + 1) * (a + 2) / 2 <= o) ++a;
        const int b = o - a * (a + 1) / 2;
        double s0 = 0.0, s1 = 0.0;
        if (o < tri) {
            const float* p = M.G + a * KM + b;
            int t = j;
#pragma unroll 4
            for (; t + 4 < nt; t += 8) {
                s0 += static_cast<double>(p[(int64_t)t * KM * KM]);
                s1 += static_cast<double>(p[(int64_t)(t + 4) * KM * KM]);
            }
            if (t < nt) s0 += static_cast<double>(p[(int64_t)t * KM * KM]);
        }
        double s = s0 + s1;
        s += __shfl_xor_sync(0xffffffffu, s, 1);
        s += __shfl_xor_sync(0xffffffffu, s, 2);
        if (o < tri && j == 0) {
            const float v = static_cast<float>(s);
            G0[a * (KM + 1) + b] = v;
            G0[b * (KM + 1) + a] = v;
        }
    }
    cl.sync();
    if (rank != 0) return;
    if (mode == 1) {
        for (int o = tid; o < k * k; o += TCH) M.H[o] = Gs[o / k][o % k];
        return;
    }
    float tr = 0.f;
    for (int i = 0; i < k; ++i) tr += Gs[i][i];
    if (tid == 0 && M.flag && (!(tr > 0.f) || !isfinite(tr))) atomicAdd(M.flag + 6, 1);   // degenerate block
    // right-looking factor and, in the same steps, the substitution for L^{-1} along L's columns: a thread
    // holds entries (i, c) of both; a step needs column j of the one and row j of the other
    constexpr int E = KM * KM / TCH;
    const int c = tid % KM, i0 = tid / KM;
    float shift = 0.f;
    for (int attempt = 0; attempt < 6; ++attempt) {
        float a[E], r[E], x[E];
#pragma unroll
        for (int m = 0; m < E; ++m) {
            const int i = i0 + m * (TCH / KM);
            a[m] = i < k && c < k ? Gs[i][c] + (i == c ? shift : 0.f) : 0.f;
            r[m] = i == c ? 1.f : 0.f;
            x[m] = 0.f;
            if (c == 0) colj[0][i] = a[m];
            if (i == 0) rowj[0][c] = r[m];
        }
        __syncthreads();
        bool ok = true;
        for (int j = 0; j < k; ++j) {
            const float* cj = colj[j & 1];
            const float d = cj[j];
            ok = d > 0.f;                                      // the same value in every thread
            if (!ok) break;
            // every warp forms L's column and the inverse's row: a quotient a lane (two for KM = 32)
            const float ljj = sqrtf(d), *rj = rowj[j & 1];
            const float q0 = quotient(KM == 32 || lane < KM ? cj[lane] : rj[lane % KM], ljj);
            const float q1 = KM == 32 ? quotient(rj[lane], ljj) : q0;
            const float qc = __shfl_sync(0xffffffffu, q0, c), xj = __shfl_sync(0xffffffffu, q1, KM == 32 ? c : KM + c);
            const float vc = c > j ? qc : 0.f;
#pragma unroll
            for (int m = 0; m < E; ++m) {
                const int i = i0 + m * (TCH / KM);
                const float vi = __shfl_sync(0xffffffffu, q0, i);
                if (i == j) x[m] = xj;
                if (i > j) {
                    a[m] = fmaf(-vi, vc, a[m]);
                    r[m] = fmaf(-xj, vi, r[m]);
                }
                if (c == j + 1) colj[(j + 1) & 1][i] = a[m];
                if (i == j + 1) rowj[(j + 1) & 1][c] = r[m];
            }
            __syncthreads();
        }
        if (ok) {
#pragma unroll
            for (int m = 0; m < E; ++m) {
                const int i = i0 + m * (TCH / KM);
                if (i < k && c < k) M.S[c * k + i] = x[m];     // S = L^{-T}
            }
            if (attempt > 0 && tid == 0 && M.flag) atomicAdd(M.flag, 1);
            return;
        }
        shift = chol_shift(attempt, tr > 0.f ? tr / k : 1.f);
        __syncthreads();
    }
    // no factorisation: leave S as identity and count it
    for (int o = tid; o < k * k; o += TCH) M.S[o] = o / k == o % k ? 1.f : 0.f;
    if (tid == 0 && M.flag) { atomicAdd(M.flag, 1000); atomicAdd(M.flag + 6, 1); }
}

template <int KM>
cudaError_t pow_launch(const PowGroup& g, int stage, int arg, cudaStream_t st) {
    switch (stage) {
        case 0: {
            const cudaError_t e = cudaFuncSetAttribute(pow_t_kernel<KM>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kPowTSmem<KM>);
            if (e != cudaSuccess) return e;
            launch_chain(pow_t_kernel<KM>, g.tot_t, TM, kPowTSmem<KM>, st, g, arg);
            break;
        }
        case 1: {
            const cudaError_t e = cudaFuncSetAttribute(pow_n_kernel<KM>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kPowNSmem<KM>);
            if (e != cudaSuccess) return e;
            launch_chain(pow_n_kernel<KM>, g.tot_n * (PC / NR), TM, kPowNSmem<KM>, st, g);
            break;
        }
        case 2: launch_chain(pow_r_kernel<KM>, g.tot_r, TP, 0, st, g); break;
        case 3: launch_chain(pow_apply_kernel<KM>, g.tot_r, TP, 0, st, g, arg); break;
        case 4: launch_chain(pow_chol_kernel<KM>, g.nmat * CCH, TCH, 0, st, g, arg, 0); break;
        case 5: launch_chain(pow_chol_kernel<KM>, g.nmat * CCH, TCH, 0, st, g, arg, 1); break;
        default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

}  // namespace

int pow_tile() { return PC; }
int pow_chunk() { return NCH; }

cudaError_t pow_stage(const PowGroup& g, int stage, int arg, cudaStream_t st) {
    if (g.nmat <= 0) return cudaSuccess;
    int kmax = 0;
    for (int i = 0; i < g.nmat; ++i) kmax = g.mat[i].k > kmax ? g.mat[i].k : kmax;
    if (kmax <= 16) return pow_launch<16>(g, stage, arg, st);
    if (kmax <= 32) return pow_launch<32>(g, stage, arg, st);
    return cudaErrorInvalidValue;
}

}  // namespace glr
