// The k x k Rayleigh-Ritz problems of truncated refreshes, several at once (any symmetric n x n
// eigenproblem up to n = 1024).  Two-sided Jacobi in fp32; a problem stops at the start of the first sweep whose
// off-diagonal norm is within tol of the total; one that is not (or not a number) after max_sweeps ends there
// and is counted in *failed.
//
// n <= 128: one CTA a problem (eig_small_kernel), every sweep on the registers of k_pair.cuh: 127
// rounds for n > 64, 63, 31 or 15 for the smaller problems (with a quarter of the warps each).
//
// n > 128: the blocked Jacobi of k_bjac.cu (blocks of 64 indices paired by a round-robin
// tournament, n padded to a multiple of 128 with zeros, whose rotations are the identity) in one
// cooperative launch for all problems (eig_group_kernel).  A round is two grid steps: the pair
// sweeps J_k, one CTA a pair, then H <- J^T H J and V <- V J in 64-row jobs spread over the grid,
// fp32 products through shared memory (a job of H: T = J_k[:, rows]^T H_kl, then T J_l, written to
// the next round's place and, mirrored, to the other side of the diagonal).  After a sweep's m - 1
// rounds the blocks are back in their own order.  A problem's sequence does not depend on what it is
// grouped with: its norm check adds fixed chunks in a fixed order, and steps only wait for one
// another.
//
// Polish.  Hundreds of rotations a column leave V off by several fp32 roundings, in orthogonality
// and in the eigenvectors.  At the end one step of the refinement of Ogita and Aishima (2018) takes
// that back: R = I - V^T V, S = V^T H V from the H the solve began with, V <- V + V E with E_ij = R_ij / 2
// + (S_ij + R_ij (l_i + l_j) / 2) / (l_j - l_i), l_i = S_ii; the second part only where it is below 2^-15 (its
// second-order error is then below fp32's): for closer eigenvalues orthogonality alone.  Leading
// eigenvectors against 64 bits, 512 x 4608 conv gradients: 3.4e-6 without it, 4e-7 with.
//
// What bounds it: the pair sweeps, a serial chain of 64 rounds on one SM a pair (about 30 us of the
// 45 us of a round, two steps and two barriers).
//
// The grid barrier is an arrival counter and a generation word in global memory; a waiting CTA
// polls with short sleeps and gives up after about a second, counts the event in *err and returns.
// The cooperative launch keeps every CTA resident, which is what makes the barrier safe to wait on.
// Data written by one CTA and read by another is read through L2 (ld.cg, cp.async.cg).
#include "k_pair.cuh"

namespace glr {

namespace {

using namespace pair;

constexpr int kNormChunks = 64;

__device__ __forceinline__ float h_entry(const EigMat& M, int r, int c) {
    return r < M.n && c < M.n ? M.H[(size_t)r * M.ld + c] : 0.f;
}

// E_ij of the polish from (V^T V)_ij and S_ij, i < j, for both sides of the diagonal: half of R_ij and
// a part that is antisymmetric to the bit, so that E_ij + E_ji = R_ij whatever the rounding of S.
__device__ __forceinline__ float polish(float s, float g, float li, float lj, bool diag) {
    const float r = (diag ? 1.f : 0.f) - g, num = fmaf(0.5f * (li + lj), r, s), gap = lj - li;
    return 0.5f * r + (!diag && gap != 0.f && fabsf(num) <= 0x1p-15f * fabsf(gap) ? num / gap : 0.f);
}

// Rows r0 .. + 7, columns c0 .. + 3 of A B, or with TRANS of A^T B (R x R, pitch PLD).
template <int R, bool TRANS>
__device__ __forceinline__ void small_product(const float* A, const float* B, int r0, int c0, bool on, u64 (&acc)[8][2]) {
#pragma unroll
    for (int r = 0; r < 8; ++r) { acc[r][0] = 0; acc[r][1] = 0; }
    if (!on) return;
#pragma unroll 2
    for (int k = 0; k < R; ++k) {
        const u64 b0 = *reinterpret_cast<const u64*>(B + k * PLD + c0), b1 = *reinterpret_cast<const u64*>(B + k * PLD + c0 + 2);
#pragma unroll
        for (int r = 0; r < 8; ++r) {
            const float a = TRANS ? A[k * PLD + r0 + r] : A[(r0 + r) * PLD + k];
            const u64 aa = pk(a, a);
            acc[r][0] = fma2(aa, b0, acc[r][0]);
            acc[r][1] = fma2(aa, b1, acc[r][1]);
        }
    }
}

template <int LIM>
__global__ void __launch_bounds__(8 * LIM, 1) eig_small_kernel(const __grid_constant__ EigGroup g) {
    chain_begin();
    constexpr int R = 2 * LIM, NT = 8 * LIM;
    extern __shared__ __align__(16) float esm[];
    float* S = esm;
    float* W = S + R * PLD;
    float* xch = W + R * PLD;
    float* apq = xch + 2 * 16 * 128;
    __shared__ float red[2][16];
    __shared__ int stop;
    const EigMat& M = g.mat[blockIdx.x];
    const int n = M.n, t = threadIdx.x, warp = t >> 5, lane = t & 31;
    for (int e = t; e < R * PLD; e += NT) {
        const int r = e / PLD, c = e - r * PLD;
        S[e] = h_entry(M, r, c);
        W[e] = r == c ? 1.f : 0.f;
    }
    __syncthreads();
    Block<8> b;
    int sweep = 0;
    for (;; ++sweep) {
        float off = 0.f, tot = 0.f;
        for (int r = warp; r < n; r += NT / 32)
            for (int c = lane; c < n; c += 32) {
                const float v = S[r * PLD + c];
                tot += v * v;
                if (r != c) off += v * v;
            }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            off += __shfl_xor_sync(0xffffffffu, off, o);
            tot += __shfl_xor_sync(0xffffffffu, tot, o);
        }
        if (lane == 0) { red[0][warp] = off; red[1][warp] = tot; }
        __syncthreads();
        if (t == 0) {
            float o2 = 0.f, t2 = 0.f;
            for (int w = 0; w < NT / 32; ++w) { o2 += red[0][w]; t2 += red[1][w]; }
            stop = (o2 <= M.tol * M.tol * t2 || sweep >= g.max_sweeps) ? 1 : 0;
            red[0][0] = o2; red[1][0] = t2;                // for the count at the end (kept out of the sweeps' code)
        }
        __syncthreads();
        if (stop) break;
        for (int lv = LIM; lv >= 1; lv >>= 1) {
            b.load(S, W, lv, warp, lane);
            b.level(S, lv, xch, apq, warp, lane, LIM);
            __syncthreads();
            b.store(S, W, lv, warp, lane);
            __syncthreads();
        }
    }
    // the polish: S <- H, T = H W, then S_ = W^T T and W^T W in registers, E over S, V = W + W E
    float* T = apq + 2 * 64;
    float* lam = xch;
    for (int e = t; e < R * PLD; e += NT) {
        const int r = e / PLD, c = e - r * PLD;
        S[e] = h_entry(M, r, c);
    }
    __syncthreads();
    u64 x[8][2], y[8][2];
    const int r0 = 8 * warp, c0 = 4 * lane;
    const bool cols = c0 < R;
    small_product<R, false>(S, W, r0, c0, cols, x);
    if (cols)
#pragma unroll
        for (int r = 0; r < 8; ++r)
#pragma unroll
            for (int q = 0; q < 2; ++q) *reinterpret_cast<u64*>(T + (r0 + r) * PLD + c0 + 2 * q) = x[r][q];
    __syncthreads();
    small_product<R, true>(W, T, r0, c0, cols, x);
    small_product<R, true>(W, W, r0, c0, cols, y);
#pragma unroll
    for (int r = 0; r < 8; ++r)
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            float u[2];
            unpk(x[r][q >> 1], u[0], u[1]);
            if (r0 + r == c0 + q) lam[r0 + r] = u[q & 1];
        }
    __syncthreads();                                       // T is read: S_ takes its place
    if (cols)
#pragma unroll
        for (int r = 0; r < 8; ++r)
#pragma unroll
            for (int q = 0; q < 2; ++q) *reinterpret_cast<u64*>(T + (r0 + r) * PLD + c0 + 2 * q) = x[r][q];
    __syncthreads();
    if (cols)
#pragma unroll
        for (int r = 0; r < 8; ++r)
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                float g0, g1;
                unpk(y[r][q], g0, g1);
                const int i = r0 + r, j = c0 + 2 * q;
                const float s0 = i < j ? T[i * PLD + j] : T[j * PLD + i];
                const float s1 = i < j + 1 ? T[i * PLD + j + 1] : T[(j + 1) * PLD + i];
                *reinterpret_cast<u64*>(S + i * PLD + j) =
                    pk(polish(s0, g0, lam[i], lam[j], i == j), polish(s1, g1, lam[i], lam[j + 1], i == j + 1));
            }
    __syncthreads();
    small_product<R, false>(W, S, r0, c0, cols, x);
#pragma unroll
    for (int r = 0; r < 8; ++r)
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            float u[2];
            unpk(x[r][q >> 1], u[0], u[1]);
            const int i = r0 + r, j = c0 + q;
            if (i < n && j < n) M.V[(size_t)i * n + j] = W[i * PLD + j] + u[q & 1];
        }
    for (int i = t; i < n; i += NT) M.evals[i] = lam[i];
    if (t == 0 && M.sweeps) *M.sweeps = sweep;
    if (t == 0 && sweep >= g.max_sweeps && M.failed && !(red[0][0] <= M.tol * M.tol * red[1][0])) atomicAdd(M.failed, 1);
}
template <int LIM> constexpr size_t small_smem() {
    return sizeof(float) * (3 * (2 * LIM) * PLD + 2 * 16 * 128 + 2 * 64);
}

// ---- n > 128 -------------------------------------------------------------------------------
__host__ __device__ __forceinline__ int pad128(int n) { return (n + 127) & ~127; }

// All CTAs arrive; false when the wait timed out.  *count returns to 0 after every barrier.
__device__ bool grid_barrier(int* count, int* genp, int& gen) {
    __shared__ int s_ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        int ok = 1;
        const int target = gen + 1;
        __threadfence();
        if (atomicAdd(count, 1) == static_cast<int>(gridDim.x) - 1) {
            atomicExch(count, 0);
            __threadfence();
            atomicExch(genp, target);
        } else {
            for (int spin = 0; *reinterpret_cast<volatile int*>(genp) != target; ++spin) {
                if (spin > 20000000) { ok = 0; break; }          // about a second of 32-64 ns sleeps
                __nanosleep(32);
            }
        }
        __threadfence();
        s_ok = ok;
    }
    __syncthreads();
    gen += 1;
    return s_ok != 0;
}

__device__ __forceinline__ void cp16(float* dst, const float* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;"
                 ::"r"(static_cast<uint32_t>(__cvta_generic_to_shared(dst))), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// rows x 128 floats from global (leading dimension ld) to shared memory (pitch 128).
__device__ __forceinline__ void fetch(float* dst, const float* src, int64_t ld, int rows) {
    for (int e = threadIdx.x; e < rows * 32; e += PTHREADS) {
        const int r = e >> 5, c = 4 * (e & 31);
        cp16(dst + r * 128 + c, src + r * ld + c);
    }
}

// C (64 x 128) = A (64 x 128) B (128 x 128), all in shared memory: warp w rows 4 w .. + 3, lane l
// columns 4 l .. + 3.
__device__ __forceinline__ void product(const float* A, const float* B, int warp, int lane, u64 (&acc)[4][2]) {
#pragma unroll
    for (int r = 0; r < 4; ++r) { acc[r][0] = 0; acc[r][1] = 0; }
    const float* a = A + 4 * warp * 128;
    const float* bp = B + 4 * lane;
#pragma unroll 4
    for (int k = 0; k < 128; k += 4) {
        float4 av[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) av[r] = *reinterpret_cast<const float4*>(a + r * 128 + k);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const ulonglong2 bv = *reinterpret_cast<const ulonglong2*>(bp + (k + q) * 128);
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const float x = q == 0 ? av[r].x : q == 1 ? av[r].y : q == 2 ? av[r].z : av[r].w;
                const u64 xx = pk(x, x);
                acc[r][0] = fma2(xx, bv.x, acc[r][0]);
                acc[r][1] = fma2(xx, bv.y, acc[r][1]);
            }
        }
    }
}

// kCopy .. kFinal: the polish (H again; T = H V and V^T V; S = V^T T; V + V E)
enum : int { kCheck = 0, kPending = 1, kPair = 2, kApply = 3, kCopy = 4, kProducts = 5, kProject = 6, kFinal = 7, kDone = 8 };

struct Work {                       // the parts of a problem's workspace
    int np, P, m;
    float *H0, *H1, *V0, *V1, *J, *Jt;
    __device__ __forceinline__ explicit Work(const EigMat& M) {
        np = pad128(M.n); P = np / 128; m = np / 64;
        const size_t nn = (size_t)np * np, jj = (size_t)np * 128;
        H0 = M.ws; H1 = H0 + nn; V0 = H1 + nn; V1 = V0 + nn; J = V1 + nn; Jt = J + jj;
    }
};

// J_k of pair k, row-major in J and transposed in Jt: all of it, or with WR = 2 the quarter `part` of
// its rows.
template <int WR>
__device__ void pair_job(const Work& w, const float* H, int k, int part, int full, float* sm) {
    constexpr int ROWS = 16 * WR;
    const int w0 = part * ROWS;
    const float* W = pair::sweep<WR>(H + (int64_t)(PN * k) * (w.np + 1), w.np, w0, full, sm,
                                     [](const float* p) { return __ldcg(reinterpret_cast<const float2*>(p)); });
    float* J = w.J + (int64_t)k * PN * PN;
    float* Jt = w.Jt + (int64_t)k * PN * PN;
    for (int e = threadIdx.x; e < PN * ROWS; e += PTHREADS) {
        J[(w0 + e / PN) * PN + e % PN] = W[e / PN * PLD + e % PN];
        Jt[e / ROWS * PN + w0 + e % ROWS] = W[e % ROWS * PLD + e / ROWS];
    }
    __syncthreads();
}

// Next round's place of row or column x (in this round's storage order).
__device__ __forceinline__ int dest(int x, int m, int rd) { return 64 * bjac_dest_of(x >> 6, m, rd) + (x & 63); }

__device__ void h_job(const Work& w, const float* H, float* Hn, int k, int l, int strip, int rd, float* sm) {
    float *As = sm, *Bs = As + 64 * 128, *Js = Bs + 128 * 128, *Ts = Js + 128 * 128;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    fetch(As, w.Jt + (int64_t)k * PN * PN + strip * 64 * 128, 128, 64);
    fetch(Bs, H + (int64_t)(128 * k) * w.np + 128 * l, w.np, 128);
    cp_commit();
    fetch(Js, w.J + (int64_t)l * PN * PN, 128, 128);
    cp_commit();
    cp_wait<1>();
    __syncthreads();
    u64 acc[4][2];
    product(As, Bs, warp, lane, acc);
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        u64* to = reinterpret_cast<u64*>(Ts + (4 * warp + r) * 128 + 4 * lane);
        to[0] = acc[r][0]; to[1] = acc[r][1];
    }
    cp_wait<0>();
    __syncthreads();
    product(Ts, Js, warp, lane, acc);
    const int c0 = 128 * k + 64 * strip + 4 * warp, z0 = 128 * l + 4 * lane;
    const int rc = dest(c0, w.m, rd), rz = dest(z0, w.m, rd);
    float o[4][4];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        unpk(acc[r][0], o[r][0], o[r][1]);
        unpk(acc[r][1], o[r][2], o[r][3]);
        *reinterpret_cast<float4*>(Hn + (int64_t)(rc + r) * w.np + rz) = make_float4(o[r][0], o[r][1], o[r][2], o[r][3]);
    }
    if (k != l) {
#pragma unroll
        for (int c = 0; c < 4; ++c)
            *reinterpret_cast<float4*>(Hn + (int64_t)(rz + c) * w.np + rc) = make_float4(o[0][c], o[1][c], o[2][c], o[3][c]);
    }
    __syncthreads();
}

__device__ void v_job(const Work& w, const float* V, float* Vn, int strip, int l, int rd, float* sm) {
    float *As = sm, *Js = As + 64 * 128;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    fetch(As, V + (int64_t)(64 * strip) * w.np + 128 * l, w.np, 64);
    fetch(Js, w.J + (int64_t)l * PN * PN, 128, 128);
    cp_commit();
    cp_wait<0>();
    __syncthreads();
    u64 acc[4][2];
    product(As, Js, warp, lane, acc);
    const int rz = dest(128 * l + 4 * lane, w.m, rd);
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        float a, b, c, d;
        unpk(acc[r][0], a, b);
        unpk(acc[r][1], c, d);
        *reinterpret_cast<float4*>(Vn + (int64_t)(64 * strip + 4 * warp + r) * w.np + rz) = make_float4(a, b, c, d);
    }
    __syncthreads();
}

// 64 x 128 tile (i0, j0) of A^T B (np x np each, read by their rows), to C.
__device__ void tn_job(const Work& w, const float* A, const float* B, float* C, int i0, int j0, float* sm) {
    float *As = sm, *Bs = As + 64 * 128;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    u64 acc[4][2] = {};
    for (int k0 = 0; k0 < w.np; k0 += 128) {
        for (int e = threadIdx.x; e < 128 * 16; e += PTHREADS)
            cp16(As + (e >> 4) * 64 + 4 * (e & 15), A + (int64_t)(k0 + (e >> 4)) * w.np + i0 + 4 * (e & 15));
        fetch(Bs, B + (int64_t)k0 * w.np + j0, w.np, 128);
        cp_commit();
        cp_wait<0>();
        __syncthreads();
#pragma unroll 8
        for (int k = 0; k < 128; ++k) {
            const float4 a = *reinterpret_cast<const float4*>(As + k * 64 + 4 * warp);
            const ulonglong2 bv = *reinterpret_cast<const ulonglong2*>(Bs + k * 128 + 4 * lane);
            const float av[4] = {a.x, a.y, a.z, a.w};
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const u64 xx = pk(av[r], av[r]);
                acc[r][0] = fma2(xx, bv.x, acc[r][0]);
                acc[r][1] = fma2(xx, bv.y, acc[r][1]);
            }
        }
        __syncthreads();
    }
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        u64* to = reinterpret_cast<u64*>(C + (int64_t)(i0 + 4 * warp + r) * w.np + j0 + 4 * lane);
        to[0] = acc[r][0]; to[1] = acc[r][1];
    }
}

// 64 x 128 tile (i0, j0) of V + V E to M.V (n x n); E from S and Gm = V^T V.
__device__ void final_job(const EigMat& M, const Work& w, const float* V, const float* S, const float* Gm, int i0, int j0,
                          float* sm) {
    float *As = sm, *Es = As + 64 * 128;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    u64 sum[4][2] = {};
    for (int k0 = 0; k0 < w.np; k0 += 128) {
        fetch(As, V + (int64_t)i0 * w.np + k0, w.np, 64);
        cp_commit();
        for (int e = threadIdx.x; e < 128 * 128; e += PTHREADS) {
            const int i = k0 + (e >> 7), j = j0 + (e & 127);
            const int64_t at = (int64_t)i * w.np + j;
            Es[e] = polish(__ldcg(S + (i < j ? at : (int64_t)j * w.np + i)), __ldcg(Gm + at), __ldcg(S + (int64_t)i * (w.np + 1)),
                           __ldcg(S + (int64_t)j * (w.np + 1)), i == j);
        }
        cp_wait<0>();
        __syncthreads();
        u64 acc[4][2];
        product(As, Es, warp, lane, acc);
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            sum[r][0] = fma2(pk(1.f, 1.f), acc[r][0], sum[r][0]);
            sum[r][1] = fma2(pk(1.f, 1.f), acc[r][1], sum[r][1]);
        }
        __syncthreads();
    }
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        const int i = i0 + 4 * warp + r;
        float u[4];
        unpk(sum[r][0], u[0], u[1]);
        unpk(sum[r][1], u[2], u[3]);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int j = j0 + 4 * lane + q;
            if (i < M.n && j < M.n) M.V[(size_t)i * M.n + j] = __ldcg(V + (int64_t)i * w.np + j) + u[q];
        }
    }
}

__global__ void __launch_bounds__(PTHREADS, 1) eig_group_kernel(const __grid_constant__ EigGroup g) {
    extern __shared__ __align__(16) float gsm[];
    const int G = gridDim.x, b = blockIdx.x, t = threadIdx.x, warp = t >> 5, lane = t & 31;
    const int64_t gtid = (int64_t)b * PTHREADS + t, gsz = (int64_t)G * PTHREADS;
    __shared__ int sstate[kEigGroupMax], sround[kEigGroupMax], ssweep[kEigGroupMax], sflip[kEigGroupMax];
    __shared__ float red[2][16];
    int gen = 0;
    for (int mi = 0; mi < g.nmat; ++mi) {                 // H padded with zeros, V = I
        const EigMat& M = g.mat[mi];
        const Work w(M);
        for (int64_t e = gtid; e < (int64_t)w.np * w.np; e += gsz) {
            const int r = (int)(e / w.np), c = (int)(e % w.np);
            w.H0[e] = h_entry(M, r, c);
            w.V0[e] = r == c ? 1.f : 0.f;
        }
    }
    if (t < g.nmat) { sstate[t] = kCheck; sround[t] = 0; ssweep[t] = 0; sflip[t] = 0; }
    bool ok = grid_barrier(g.bar, g.bar + 1, gen);
    while (ok) {
        for (int mi = warp; mi < g.nmat; mi += PTHREADS / 32) {          // decide on the last step's partials
            if (sstate[mi] != kPending) continue;
            const EigMat& M = g.mat[mi];
            float o2 = 0.f, t2 = 0.f;
            for (int c = lane; c < kNormChunks; c += 32) {
                o2 += __ldcg(g.part + (2 * mi) * kNormChunks + c);
                t2 += __ldcg(g.part + (2 * mi + 1) * kNormChunks + c);
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                o2 += __shfl_xor_sync(0xffffffffu, o2, o);
                t2 += __shfl_xor_sync(0xffffffffu, t2, o);
            }
            __syncwarp();
            if (lane == 0) {
                const bool converged = o2 <= M.tol * M.tol * t2;
                if (converged || ssweep[mi] >= g.max_sweeps) {
                    sstate[mi] = kCopy;
                    if (b == 0 && M.sweeps) *M.sweeps = ssweep[mi];
                    if (b == 0 && !converged && M.failed) atomicAdd(M.failed, 1);
                } else {
                    sstate[mi] = kPair;
                    sround[mi] = 0;
                }
            }
        }
        __syncthreads();
        bool any = false;
        for (int mi = 0; mi < g.nmat; ++mi) any = any || sstate[mi] != kDone;
        if (!any) break;
        int item = 0;                                     // the step's jobs, dealt out in turn
        for (int mi = 0; mi < g.nmat; ++mi) {
            const EigMat& M = g.mat[mi];
            const Work w(M);
            const float* Hc = sflip[mi] ? w.H1 : w.H0;
            const float* Vc = sflip[mi] ? w.V1 : w.V0;
            const int state = sstate[mi], rd = sround[mi];
            if (state == kCheck) {
                for (int c = (b - item % G + G) % G; c < kNormChunks; c += G) {
                    float off = 0.f, tot = 0.f;
                    for (int r = c; r < M.n; r += kNormChunks)
                        for (int q = t; q < M.n; q += PTHREADS) {
                            const float h = __ldcg(Hc + (int64_t)r * w.np + q);
                            tot += h * h;
                            if (r != q) off += h * h;
                        }
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) {
                        off += __shfl_xor_sync(0xffffffffu, off, o);
                        tot += __shfl_xor_sync(0xffffffffu, tot, o);
                    }
                    if (lane == 0) { red[0][warp] = off; red[1][warp] = tot; }
                    __syncthreads();
                    if (t == 0) {
                        float o2 = 0.f, t2 = 0.f;
                        for (int q = 0; q < 16; ++q) { o2 += red[0][q]; t2 += red[1][q]; }
                        g.part[(2 * mi) * kNormChunks + c] = o2;
                        g.part[(2 * mi + 1) * kNormChunks + c] = t2;
                    }
                    __syncthreads();
                }
                item += kNormChunks;
            } else if (state == kPair) {
                for (int k = (b - item % G + G) % G; k < w.P * g.parts; k += G) {
                    if (g.parts == 4) pair_job<2>(w, Hc, k >> 2, k & 3, rd == 0, gsm);
                    else pair_job<8>(w, Hc, k, 0, rd == 0, gsm);
                }
                item += w.P * g.parts;
            } else if (state == kApply) {
                const int nh = w.P * (w.P + 1), nv = w.m * w.P;
                float* Hn = sflip[mi] ? w.H0 : w.H1;
                float* Vn = sflip[mi] ? w.V0 : w.V1;
                for (int j = (b - item % G + G) % G; j < nh + nv; j += G) {
                    if (j < nh) {
                        int l = 0, q = j >> 1;            // q = l (l + 1) / 2 + k, k <= l
                        while (q > l) { q -= l + 1; ++l; }
                        h_job(w, Hc, Hn, q, l, j & 1, rd, gsm);
                    } else {
                        v_job(w, Vc, Vn, (j - nh) / w.P, (j - nh) % w.P, rd, gsm);
                    }
                }
                item += nh + nv;
            } else if (state >= kCopy && state <= kFinal) {
                float *Ha = sflip[mi] ? w.H1 : w.H0, *Hb = sflip[mi] ? w.H0 : w.H1, *Vb = sflip[mi] ? w.V0 : w.V1;
                const int tiles = w.m * w.P, jobs = state == kCopy ? w.m : state == kProducts ? 2 * tiles : tiles;
                for (int j = (b - item % G + G) % G; j < jobs; j += G) {
                    const int i0 = 64 * ((j % tiles) / w.P), j0 = 128 * (j % w.P);
                    if (state == kCopy) {
                        for (int e = t; e < 64 * w.np; e += PTHREADS) {
                            const int r = 64 * j + e / w.np, c = e % w.np;
                            Ha[(int64_t)r * w.np + c] = h_entry(M, r, c);
                        }
                    } else if (state == kProducts) {
                        if (j < tiles) tn_job(w, Ha, Vc, Hb, i0, j0, gsm);
                        else tn_job(w, Vc, Vc, Vb, i0, j0, gsm);
                    } else if (state == kProject) {
                        tn_job(w, Vc, Hb, Ha, i0, j0, gsm);
                    } else {
                        final_job(M, w, Vc, Ha, Vb, i0, j0, gsm);
                        if (j0 == 0 && t < 64 && i0 + t < M.n) M.evals[i0 + t] = __ldcg(Ha + (int64_t)(i0 + t) * (w.np + 1));
                    }
                }
                item += jobs;
            }
        }
        __syncthreads();
        if (t < g.nmat) {                                 // every CTA advances the same stages
            const int m = pad128(g.mat[t].n) / 64;
            if (sstate[t] == kCheck) sstate[t] = kPending;   // decided on at the start of the next step
            else if (sstate[t] == kPair) sstate[t] = kApply;
            else if (sstate[t] == kApply) {
                sflip[t] ^= 1;
                if (++sround[t] == m - 1) { sstate[t] = kCheck; ++ssweep[t]; }
                else sstate[t] = kPair;
            } else if (sstate[t] != kDone) {
                ++sstate[t];                              // kPending is left only above
            }
        }
        ok = grid_barrier(g.bar, g.bar + 1, gen);
    }
    if (!ok && t == 0 && g.err) atomicAdd(g.err, 1);
}

constexpr size_t kGroupSmem = sizeof(float) * (2 * 64 * 128 + 2 * 128 * 128);
static_assert(kGroupSmem >= kSmem, "the pair sweeps share the jobs' shared memory");

template <int LIM>
cudaError_t launch_small(const EigGroup& g, cudaStream_t st) {
    const cudaError_t e = cudaFuncSetAttribute(eig_small_kernel<LIM>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                               (int)small_smem<LIM>());
    if (e != cudaSuccess) return e;
    launch_chain(eig_small_kernel<LIM>, g.nmat, 8 * LIM, small_smem<LIM>(), st, g);
    return cudaGetLastError();
}

}  // namespace

size_t eig_ws_floats(int n) {
    if (n <= kEigSmall) return 0;
    const size_t np = pad128(n);
    return 4 * np * np + 2 * np * 128;
}

// By size class (16, 32, 64, 128), so that a problem's rounds do not depend on the group.
cudaError_t eig_small_group(const EigGroup& g, cudaStream_t st) {
    --more_launches;
    for (int lim = 8; lim <= 64; lim *= 2) {
        EigGroup c = g;
        c.nmat = 0;
        for (int i = 0; i < g.nmat; ++i) {
            const int n = g.mat[i].n;
            if (n < 1 || n > kEigSmall) return cudaErrorInvalidValue;
            if (n <= 2 * lim && (lim == 8 || n > lim)) c.mat[c.nmat++] = g.mat[i];
        }
        if (c.nmat == 0) continue;
        ++more_launches;
        const cudaError_t e = lim == 8 ? launch_small<8>(c, st) : lim == 16 ? launch_small<16>(c, st)
                              : lim == 32 ? launch_small<32>(c, st) : launch_small<64>(c, st);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

cudaError_t eig_group(EigGroup& g, cudaStream_t st) {
    if (g.nmat <= 0) return cudaSuccess;
    int pairs = 0;
    for (int i = 0; i < g.nmat; ++i) {
        if (g.mat[i].n <= kEigSmall || g.mat[i].n > 1024 || !g.mat[i].ws) return cudaErrorInvalidValue;
        pairs += pad128(g.mat[i].n) / 128;
    }
    int dev = 0, sms = 0, coop = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev);
    if (e == cudaSuccess)      // per device: set on every call (cheap next to the launch)
        e = cudaFuncSetAttribute(eig_group_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kGroupSmem);
    if (e == cudaSuccess) e = cudaMemsetAsync(g.bar, 0, 2 * sizeof(int), st);    // arrivals and generation
    if (e != cudaSuccess) return e;
    g.parts = 4 * pairs <= sms ? 4 : 1;      // four CTAs a pair where they are to spare (the same bits)
    if (!coop) {               // one CTA: the barriers wait for nobody
        eig_group_kernel<<<1, PTHREADS, kGroupSmem, st>>>(g);
        return cudaGetLastError();
    }
    void* args[] = {&g};
    return cudaLaunchCooperativeKernel(reinterpret_cast<const void*>(eig_group_kernel), dim3(sms), dim3(PTHREADS), args,
                                       kGroupSmem, st);
}

}  // namespace glr
