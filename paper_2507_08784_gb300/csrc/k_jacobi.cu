// Full-basis refresh (Eq. SVD-P1, the paper-exact basis): the eigen-decomposition of the m' x m'
// Gram matrices H = Mbar Mbar^T of every refreshing matrix by parallel cyclic two-sided Jacobi,
// above m' = 512 all matrices in one cooperative launch.  A round applies n/2 disjoint plane rotations chosen by
// the circle (round-robin) ordering — each angle from its own 2 x 2 diagonal block (Golub & Van
// Loan, sym.schur2) — then H <- J^T H J block-wise (each 2 x 2 block of H depends only on the
// rotations of its row and column pairs) and V <- V J.  The updates of a round are spread over
// every CTA of the grid, rounds separated by grid-wide barriers; a matrix stops at the start of
// the first sweep whose off-diagonal norm is within tol of the total.  One that is not after max_sweeps ends
// there and is counted in *failed (a matrix with NaNs, which no sweep can help, is not: the compose
// pass has counted those).
//
// The grid barrier is an arrival counter and a generation word in global memory; a waiting CTA
// polls with short sleeps and gives up after about a second, counts the event in *err and
// returns, so a stuck barrier ends the kernel instead of hanging it.  The cooperative launch
// keeps every CTA resident, which is what makes the barrier safe to wait on.  Data written by one
// CTA and read by another (H, V, the norm partials) is read through L2 (__ldcg), so no stale L1
// line survives a barrier.
//
// For n <= 512 a matrix is solved in the shared memory of one thread-block cluster
// (jacobi_cluster_kernel): the row pairs of H are spread over up to 16 CTAs, one a warp (16 x 16 pairs:
// hence 512; 76 KB a CTA there, 227 KB would hold n = 896), a round's rotations go
// to all of them over distributed shared memory; two hardware cluster barriers a round.  The
// rotations, their order and every product and sum are those of the grid-wide kernel, so the results
// are the same bits.  A round takes 3.2 us at n = 512 (bound by instruction issue) and 2 us below
// n = 128 (the rotation's chain of quotients and roots, two cluster barriers); the grid-wide kernel
// pays 6 us at n = 512 alone and 14 us for the eight matrices of a conv stack, its barrier in global
// memory and the L2 round trips.  Above 512 a warp would take several pairs: tried on one matrix, 5.7 us
// a round at n = 768 (39 ms; grid-wide 9.1 us, 63 ms) and 7.0 us at 896 (10.6), the same bits; not built in.
#include <cooperative_groups.h>

#include "glr_internal.cuh"

namespace glr {

namespace {

constexpr int JT = 256;                 // threads per CTA

__device__ __forceinline__ int circle(int x, int nm1) { return 1 + ((x % nm1) + nm1) % nm1; }

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
        gen = target;
        s_ok = ok;
    }
    __syncthreads();
    return s_ok != 0;
}

// Each matrix runs its own sequence — a norm check, then its own n' - 1 rounds (n' = n rounded up
// to even), then the next check, ... — one stage per grid step, so what a matrix computes does not
// depend on the matrices it is grouped with.  In a round every CTA forms all of the round's
// rotations itself (from the current H, in shared memory) and applies its share of the 2 x 2
// block updates from the current H into the other H buffer (every block is written, rotated or
// not), so no CTA can see a diagonal block another CTA has already updated; V is updated in place
// (each entry by one thread).  A check's partial norms are written in one step and decided on at
// the start of the next, identically by every CTA.  One grid barrier per step.
enum : int { kCheck = 0, kRound = 1, kPending = 2, kDone = 3 };

__global__ void __launch_bounds__(JT) jacobi_group_kernel(const __grid_constant__ JacobiGroup g) {
    const int G = gridDim.x, b = blockIdx.x, t = threadIdx.x;
    const int64_t gtid = (int64_t)b * JT + t, gsz = (int64_t)G * JT;
    __shared__ int sstate[kGroupMax], sround[kGroupMax], ssweep[kGroupMax], sflip[kGroupMax];
    __shared__ float red[2][JT / 32];
    extern __shared__ float srot[];                     // per matrix at M.soff: cs, sn, pp, qq (half each)
    int gen = 0;
    bool ok = true;
    for (int mi = 0; mi < g.nmat; ++mi) {
        const JacobiMat& M = g.mat[mi];
        const int64_t nn = (int64_t)M.n * M.n;
        for (int64_t e = gtid; e < nn; e += gsz) M.V[e] = (e / M.n == e % M.n) ? 1.f : 0.f;
    }
    if (t < g.nmat) { sstate[t] = kCheck; sround[t] = 0; ssweep[t] = 0; sflip[t] = 0; }
    ok = grid_barrier(g.bar, g.bar + 1, gen);
    while (ok) {
        if (t < g.nmat && sstate[t] == kPending) {      // decide on last step's partials
            const JacobiMat& M = g.mat[t];
            float o2 = 0.f, t2 = 0.f;
            for (int c = 0; c < G; ++c) { o2 += __ldcg(g.part + (2 * t) * G + c); t2 += __ldcg(g.part + (2 * t + 1) * G + c); }
            if (o2 <= M.tol * M.tol * t2 || ssweep[t] >= g.max_sweeps) {
                sstate[t] = kDone;
                if (b == 0 && M.sweeps) *M.sweeps = ssweep[t];
                if (b == 0 && o2 > M.tol * M.tol * t2 && M.failed) atomicAdd(M.failed, 1);
            } else {
                sstate[t] = kRound;
                sround[t] = 0;
            }
        }
        __syncthreads();
        bool any = false;
        for (int mi = 0; mi < g.nmat; ++mi) any = any || sstate[mi] != kDone;
        if (!any) break;
        // norm checks, and every round's rotations (each matrix in its own shared slice)
        for (int mi = 0; mi < g.nmat; ++mi) {
            const JacobiMat& M = g.mat[mi];
            const int n = M.n;
            const float* Hc = sflip[mi] ? M.H2 : M.H;
            if (sstate[mi] == kCheck) {                 // off-diagonal and total squared norms, per CTA
                const int64_t nn = (int64_t)n * n;
                float off = 0.f, tot = 0.f;
                for (int64_t e = gtid; e < nn; e += gsz) {
                    const float h = __ldcg(Hc + e);
                    tot += h * h;
                    if (e / n != e % n) off += h * h;
                }
                for (int o = 16; o > 0; o >>= 1) {
                    off += __shfl_xor_sync(0xffffffffu, off, o);
                    tot += __shfl_xor_sync(0xffffffffu, tot, o);
                }
                if ((t & 31) == 0) { red[0][t >> 5] = off; red[1][t >> 5] = tot; }
                __syncthreads();
                if (t == 0) {
                    float o2 = 0.f, t2 = 0.f;
                    for (int w = 0; w < JT / 32; ++w) { o2 += red[0][w]; t2 += red[1][w]; }
                    g.part[(2 * mi) * G + b] = o2;
                    g.part[(2 * mi + 1) * G + b] = t2;
                }
                __syncthreads();
                continue;
            }
            if (sstate[mi] != kRound) continue;
            const int npad = n + (n & 1), half = npad / 2, nm1 = npad - 1, r = sround[mi];
            float* scs = srot + M.soff;
            float* ssn = scs + half;
            int* spp = reinterpret_cast<int*>(ssn + half);
            int* sqq = spp + half;
            for (int i = t; i < half; i += JT) {        // all of the round's rotations, in this CTA
                int p = (i == 0) ? 0 : circle(r + i, nm1);
                int q = (i == 0) ? circle(r, nm1) : circle(r - i, nm1);
                if (p > q) { const int tmp = p; p = q; q = tmp; }
                float c = 1.f, s = 0.f;
                if (q < n) {
                    const float hpq = __ldcg(Hc + (size_t)p * n + q);
                    const float hpp = __ldcg(Hc + (size_t)p * n + p), hqq = __ldcg(Hc + (size_t)q * n + q);
                    if (fabsf(hpq) > 1e-30f && fabsf(hpq) > 1e-9f * sqrtf(fabsf(hpp * hqq))) {
                        const float theta = (hqq - hpp) / (2.f * hpq);
                        float tt;
                        if (fabsf(theta) > 1e15f) tt = 0.5f / theta;
                        else tt = copysignf(1.f, theta) / (fabsf(theta) + sqrtf(theta * theta + 1.f));
                        c = 1.f / sqrtf(tt * tt + 1.f);
                        s = tt * c;
                    }
                }
                scs[i] = c; ssn[i] = s; spp[i] = p; sqq[i] = q;
            }
        }
        __syncthreads();
        // every round's updates
        for (int mi = 0; mi < g.nmat; ++mi) {
            if (sstate[mi] != kRound) continue;
            const JacobiMat& M = g.mat[mi];
            const int n = M.n, half = (n + (n & 1)) / 2;
            const float* Hc = sflip[mi] ? M.H2 : M.H;
            float* Hn = sflip[mi] ? M.H : M.H2;
            const float* scs = srot + M.soff;
            const float* ssn = scs + half;
            const int* spp = reinterpret_cast<const int*>(ssn + half);
            const int* sqq = spp + half;
            const int64_t hh = (int64_t)half * half;
            for (int64_t e = gtid; e < hh; e += gsz) {   // Hn = J^T Hc J, 2 x 2 block by block
                const int bi = static_cast<int>(e / half), bj = static_cast<int>(e % half);
                const float si = ssn[bi], sj = ssn[bj], ci = scs[bi], cj = scs[bj];
                const int pi = spp[bi], qi = sqq[bi], pj = spp[bj], qj = sqq[bj];
                const bool vqi = qi < n, vqj = qj < n;
                const float h00 = __ldcg(Hc + (size_t)pi * n + pj);
                const float h01 = vqj ? __ldcg(Hc + (size_t)pi * n + qj) : 0.f;
                const float h10 = vqi ? __ldcg(Hc + (size_t)qi * n + pj) : 0.f;
                const float h11 = (vqi && vqj) ? __ldcg(Hc + (size_t)qi * n + qj) : 0.f;
                float n00 = h00, n01 = h01, n10 = h10, n11 = h11;
                if (si != 0.f || sj != 0.f) {
                    const float a00 = ci * h00 - si * h10, a01 = ci * h01 - si * h11;
                    const float a10 = si * h00 + ci * h10, a11 = si * h01 + ci * h11;
                    n00 = cj * a00 - sj * a01; n01 = sj * a00 + cj * a01;
                    n10 = cj * a10 - sj * a11; n11 = sj * a10 + cj * a11;
                    if (bi == bj && si != 0.f) { n01 = 0.f; n10 = 0.f; }
                }
                Hn[(size_t)pi * n + pj] = n00;
                if (vqj) Hn[(size_t)pi * n + qj] = n01;
                if (vqi) Hn[(size_t)qi * n + pj] = n10;
                if (vqi && vqj) Hn[(size_t)qi * n + qj] = n11;
            }
            const int64_t nv = (int64_t)n * half;
            for (int64_t e = gtid; e < nv; e += gsz) {   // V <- V J, in place
                const int a = static_cast<int>(e / half), bj = static_cast<int>(e % half);
                const float sj = ssn[bj];
                if (sj == 0.f) continue;
                const int pj = spp[bj], qj = sqq[bj];
                const float cj = scs[bj];
                const float vp = __ldcg(M.V + (size_t)a * n + pj), vq = __ldcg(M.V + (size_t)a * n + qj);
                M.V[(size_t)a * n + pj] = cj * vp - sj * vq;
                M.V[(size_t)a * n + qj] = sj * vp + cj * vq;
            }
        }
        __syncthreads();                                 // the shared rotations are rewritten next step
        if (t < g.nmat) {                               // every CTA advances the same stages
            if (sstate[t] == kCheck) {
                sstate[t] = kPending;
            } else if (sstate[t] == kRound) {
                sflip[t] ^= 1;
                const int nm1 = g.mat[t].n + (g.mat[t].n & 1) - 1;
                if (++sround[t] == nm1) { sstate[t] = kCheck; ++ssweep[t]; }
            }
        }
        ok = grid_barrier(g.bar, g.bar + 1, gen);
    }
    if (!ok) {
        if (t == 0 && g.err) atomicAdd(g.err, 1);
        return;
    }
    for (int mi = 0; mi < g.nmat; ++mi) {
        const JacobiMat& M = g.mat[mi];
        const float* Hc = sflip[mi] ? M.H2 : M.H;
        for (int64_t i = gtid; i < M.n; i += gsz) M.evals[i] = __ldcg(Hc + (size_t)i * M.n + i);
    }
}

// ---- n <= 512: one cluster a matrix ------------------------------------------------------------
constexpr int CT = 512;

__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_sync() { cluster_arrive(); cluster_wait(); }
template <class T> __device__ __forceinline__ T* peer(T* p, int cta) {       // p in another CTA of the cluster
    return cooperative_groups::this_cluster().map_shared_rank(p, cta);
}
// c x - s y and s x + c y, rounded as the grid-wide kernel's expressions are (checked bit for bit)
__device__ __forceinline__ float rot_dif(float c, float x, float s, float y) { return __fmaf_rn(c, x, -__fmul_rn(s, y)); }
__device__ __forceinline__ float rot_sum(float s, float x, float c, float y) { return __fmaf_rn(s, x, __fmul_rn(c, y)); }
// Rotations of a round in the log: whole 16-byte units.
__host__ __device__ __forceinline__ int log_stride(int half) { return (half + 1) & ~1; }
// Slots (row pairs) a CTA and CTAs a matrix.
__host__ __device__ __forceinline__ int cluster_slots(int half) { return half > 128 ? (half + 15) / 16 : 8; }
__host__ __device__ __forceinline__ int cluster_ctas(int n) {
    const int half = (n + 1) / 2, S = cluster_slots(half);
    return (half + S - 1) / S;
}
size_t cluster_smem(int n) {
    const size_t half = (n + 1) / 2, S = cluster_slots((int)half), C = cluster_ctas(n);
    const size_t rows = (2 * S + 3) + (n > 256 ? 0 : (n + C - 1) / C);
    return sizeof(float) * (4 * (size_t)log_stride((int)half) + rows * n);
}

// The round's pairs sit in npad / 2 slots (T, B); slot 0's T is index 0, the others move by one slot a
// round: T to the left, B to the right, T of slot 1 to B of slot 0, B of the last slot to its T.  A
// CTA holds the H rows of S consecutive slots, in two rings of row buffers with a spare each, so
// that only one T and one B row a round go to a neighbour's spare, written there in place of the
// row itself.  A row pair's 2 x 2 blocks are then one thread's and are updated in place.
// JU: the rotations a lane looks at (n <= 64 JU), whose indices it carries from round to round; ODD: n odd
// (index n of the padded problem has no column).  V <- V J: up to n = 256 by the same CTAs, each its share
// of the rows, while the round's second barrier completes; above (LOG) from the log afterwards (n = 512:
// 3.5 -> 3.2 us a round; n = 128: 1.8 us a round here, 2.1 with the log).
template <int JU, bool ODD>
__global__ void __launch_bounds__(CT, 1) jacobi_cluster_kernel(const __grid_constant__ JacobiMat M, int max_sweeps) {
    constexpr bool LOG = JU > 4;
    extern __shared__ __align__(16) float csm[];
    __shared__ float red[2][CT / 32], part[2];
    __shared__ int stop;
    const int n = M.n, C = gridDim.x, b = blockIdx.x, t = threadIdx.x, warp = t >> 5, lane = t & 31;
    const int npad = n + (n & 1), half = npad / 2, nm1 = npad - 1, Smax = cluster_slots(half);
    const int s0 = b * Smax, S = half - s0 < Smax ? half - s0 : Smax;          // own slots s0 .. s0 + S - 1
    const int slast = half - (C - 1) * Smax;                                // the last CTA's slots
    const int ST = b == 0 ? S - 1 : S, LT = ST + 1, LB = S + 1;             // rings (slot 0's T is apart)
    const int lstride = log_stride(half);
    float2* const scs = reinterpret_cast<float2*>(csm);                     // 2 x lstride: cos, sin
    float* const F = csm + 4 * lstride;                                        // index 0's row
    float* const Tr = F + n;
    float* const Br = Tr + (size_t)(Smax + 1) * n;
    const int R = (n + C - 1) / C, v0 = b * R, vrows = LOG ? 0 : n - v0 < R ? (n - v0 > 0 ? n - v0 : 0) : R;
    float* const V = Br + (size_t)(Smax + 1) * n;                           // own rows of V (unless LOG)
    for (int e = t; e < vrows * n; e += CT) V[e] = v0 + e / n == e % n ? 1.f : 0.f;
    float2* log = reinterpret_cast<float2*>(M.log);                         // this round's rotations
    // the buffer of the first ring T and of the first B: own, of the left and of the right neighbour
    const int LTl = b == 1 ? Smax : Smax + 1, LBr = (b + 1 == C - 1 ? slast : Smax) + 1;
    int tb = 0, bb = 0, tbl = 0, bbr = 0, par = 0;
    auto wrap = [](int x, int L) { return x >= L ? x - L : x; };
    auto trow = [&](int i) -> float* {                                      // T, B of own slot s0 + i
        return b == 0 ? (i == 0 ? F : Tr + (size_t)wrap(tb + i - 1, LT) * n) : Tr + (size_t)wrap(tb + i, LT) * n;
    };
    auto brow = [&](int i) -> float* { return Br + (size_t)wrap(bb + i, LB) * n; };
    auto tidx = [&](int slot, int rd) { return slot == 0 ? 0 : 1 + (rd + slot < nm1 ? rd + slot : rd + slot - nm1); };
    auto bidx = [&](int slot, int rd) { return 1 + (rd - slot < 0 ? rd - slot + nm1 : rd - slot); };
    for (int e = t; e < 2 * S * n; e += CT) {
        const int i = (e / n) >> 1, c = e % n, low = (e / n) & 1;
        const int r = low ? bidx(s0 + i, 0) : tidx(s0 + i, 0);
        (low ? brow(i) : trow(i))[c] = r < n ? M.H[(size_t)r * n + c] : 0.f;
    }
    cluster_sync();
    // the columns' rotations in this thread's share of the work: warps share a slot when there are few
    const int G = S > 8 ? 1 : S > 4 ? 2 : S > 2 ? 4 : S > 1 ? 8 : 16;
    int jx[JU], jy[JU];                                                     // T, B of slot lane + 32 u in this round
#pragma unroll
    for (int u = 0; u < JU; ++u) {
        const int j = lane + 32 * u < half ? lane + 32 * u : 0;
        jx[u] = tidx(j, 0);
        jy[u] = bidx(j, 0);
    }
    int sweep = 0;
    for (;; ++sweep) {
        float off = 0.f, tot = 0.f;
        for (int e = t; e < 2 * S * n; e += CT) {
            const int i = (e / n) >> 1, c = e % n, low = (e / n) & 1;
            const float h = (low ? brow(i) : trow(i))[c];
            tot += h * h;
            if ((low ? bidx(s0 + i, 0) : tidx(s0 + i, 0)) != c) off += h * h;
        }
        for (int o = 16; o > 0; o >>= 1) {
            off += __shfl_xor_sync(0xffffffffu, off, o);
            tot += __shfl_xor_sync(0xffffffffu, tot, o);
        }
        if (lane == 0) { red[0][warp] = off; red[1][warp] = tot; }
        __syncthreads();
        if (t == 0) {
            float o2 = 0.f, t2 = 0.f;
            for (int w = 0; w < CT / 32; ++w) { o2 += red[0][w]; t2 += red[1][w]; }
            part[0] = o2; part[1] = t2;
        }
        cluster_sync();
        if (t == 0) {                                   // the same sums, the same decision in every CTA
            float o2 = 0.f, t2 = 0.f;
            for (int c = 0; c < C; ++c) { o2 += peer(part, c)[0]; t2 += peer(part, c)[1]; }
            stop = o2 <= M.tol * M.tol * t2 ? 1 : sweep < max_sweeps ? 0 : o2 > M.tol * M.tol * t2 ? 2 : 1;
        }
        cluster_sync();                                 // part is read before anyone writes it again
        if (stop) break;
        for (int rd = 0; rd < nm1; ++rd) {
            float2* cs = scs + par * lstride;
            for (int e = t; e < S * C; e += CT) {       // own slots' rotations, to every CTA
                const int i = e % S, to = e / S, x = tidx(s0 + i, rd), y = bidx(s0 + i, rd);
                const int p = x < y ? x : y, q = x < y ? y : x;
                float c = 1.f, s = 0.f;
                if (!ODD || q < n) {
                    const float* rp = x < y ? trow(i) : brow(i);
                    const float* rq = x < y ? brow(i) : trow(i);
                    const float hpq = rp[q], hpp = rp[p], hqq = rq[q];
                    if (fabsf(hpq) > 1e-30f && fabsf(hpq) > 1e-9f * sqrtf(fabsf(hpp * hqq))) {
                        const float theta = (hqq - hpp) / (2.f * hpq);
                        float tt;
                        if (fabsf(theta) > 1e15f) tt = 0.5f / theta;
                        else tt = copysignf(1.f, theta) / (fabsf(theta) + sqrtf(theta * theta + 1.f));
                        c = 1.f / sqrtf(tt * tt + 1.f);
                        s = tt * c;
                    }
                }
                peer(cs, to)[s0 + i] = make_float2(c, s);
            }
            cluster_sync();
            if (LOG && b == 0 && t == 0) {
                // the round's rotations to the log, as an asynchronous copy: the cluster barrier's release
                // would wait for plain stores to global memory (0.4 us a round).  The copy before this one
                // has read its buffer by the time its rows of shared memory are written again.
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;"
                             ::"l"(log), "r"(static_cast<uint32_t>(__cvta_generic_to_shared(cs))), "r"(lstride * 8) : "memory");
                asm volatile("cp.async.bulk.commit_group;" ::: "memory");
                asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");
            }
            int pj[JU], qj[JU];
            float2 rj[JU];
#pragma unroll
            for (int u = 0; u < JU; ++u) {
                pj[u] = jx[u] < jy[u] ? jx[u] : jy[u];
                qj[u] = jx[u] < jy[u] ? jy[u] : jx[u];
                rj[u] = cs[lane + 32 * u < half ? lane + 32 * u : 0];
                jx[u] = jx[u] == 0 ? 0 : jx[u] == nm1 ? 1 : jx[u] + 1;
                jy[u] = jy[u] == nm1 ? 1 : jy[u] + 1;
            }
            if (warp / G < S) {                                             // a row pair (S <= 16): its rows, and where each goes
                const int i = warp / G, slot = s0 + i;
                float *tr = trow(i), *br = brow(i), *to = tr, *bo = br;
                if (slot > 0 && i == (b == 0 ? 1 : 0)) {                    // the first ring T leaves
                    if (b == 0) to = Br + (size_t)wrap(bb + S, LB) * n;
                    else to = peer(Tr, b - 1) + (size_t)wrap(tbl + LTl - 1, LTl) * n;
                }
                if (i == S - 1 && half > 1) {                               // the last B leaves
                    if (b == C - 1) bo = Tr + (size_t)wrap(tb + ST, LT) * n;
                    else bo = peer(Br, b + 1) + (size_t)wrap(bbr + LBr - 1, LBr) * n;
                }
                const bool up = tidx(slot, rd) < bidx(slot, rd);
                const float *hp = up ? tr : br, *hq = up ? br : tr;
                float *op = up ? to : bo, *oq = up ? bo : to;
                const float2 ri = cs[slot];
#pragma unroll
                for (int u = 0; u < JU; ++u) {
                    if ((G > 1 && (u % G) != warp % G) || lane + 32 * u >= half) continue;
                    const bool vq = !ODD || qj[u] < n;
                    const float h00 = hp[pj[u]], h10 = hq[pj[u]], h01 = vq ? hp[qj[u]] : 0.f, h11 = vq ? hq[qj[u]] : 0.f;
                    const float a00 = rot_dif(ri.x, h00, ri.y, h10), a01 = rot_dif(ri.x, h01, ri.y, h11);
                    const float a10 = rot_sum(ri.y, h00, ri.x, h10), a11 = rot_sum(ri.y, h01, ri.x, h11);
                    const bool diag = lane + 32 * u == slot && ri.y != 0.f;
                    op[pj[u]] = rot_dif(rj[u].x, a00, rj[u].y, a01);
                    oq[pj[u]] = diag ? 0.f : rot_dif(rj[u].x, a10, rj[u].y, a11);
                    if (vq) {
                        op[qj[u]] = diag ? 0.f : rot_sum(rj[u].y, a00, rj[u].x, a01);
                        oq[qj[u]] = rot_sum(rj[u].y, a10, rj[u].x, a11);
                    }
                }
            }
            cluster_arrive();
            for (int r = warp; r < vrows; r += CT / 32) {
                float* w = V + (size_t)r * n;
                float v[JU][2];
#pragma unroll
                for (int u = 0; u < JU; ++u) {
                    v[u][0] = w[pj[u]];
                    v[u][1] = !ODD || qj[u] < n ? w[qj[u]] : 0.f;
                }
#pragma unroll
                for (int u = 0; u < JU; ++u) {
                    if (lane + 32 * u >= half) continue;
                    w[pj[u]] = rot_dif(rj[u].x, v[u][0], rj[u].y, v[u][1]);
                    if (!ODD || qj[u] < n) w[qj[u]] = rot_sum(rj[u].y, v[u][0], rj[u].x, v[u][1]);
                }
            }
            cluster_wait();
            log += lstride;
            par ^= 1;
            if (half > 1) {
                tb = wrap(tb + 1, LT); tbl = wrap(tbl + 1, LTl);
                bb = bb == 0 ? LB - 1 : bb - 1; bbr = bbr == 0 ? LBr - 1 : bbr - 1;
            }
        }
    }
    for (int e = t; e < 2 * S; e += CT) {
        const int i = e >> 1, r = (e & 1) ? bidx(s0 + i, 0) : tidx(s0 + i, 0);
        if (r < n) M.evals[r] = ((e & 1) ? brow(i) : trow(i))[r];
    }
    for (int e = t; e < vrows * n; e += CT) M.V[(size_t)v0 * n + e] = V[e];
    if (b == 0 && t == 0) {
        *M.sweeps = sweep;
        if (stop == 2 && M.failed) atomicAdd(M.failed, 1);
        if (LOG) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");   // the log is complete before the CTA ends
    }
}

// V, the product of the logged rotations in their order, a warp a row: its rows depend on nothing else, so
// they are spread over the whole GPU afterwards (n = 512: 0.5 ms, against 1.1 us of the 3.5 us of every
// round in the cluster).
template <int JU, bool ODD>
__global__ void __launch_bounds__(128) jacobi_rows_kernel(const __grid_constant__ JacobiMat M) {
    extern __shared__ __align__(16) float vsm[];
    const int n = M.n, warp = threadIdx.x >> 5, lane = threadIdx.x & 31, r = blockIdx.x * 4 + warp;
    const int npad = n + (n & 1), half = npad / 2, nm1 = npad - 1;
    if (r >= n) return;
    float* w = vsm + (size_t)warp * n;
    for (int c = lane; c < n; c += 32) w[c] = r == c ? 1.f : 0.f;
    int jx[JU], jy[JU];
    float2 next[JU];
    const float2* log = reinterpret_cast<const float2*>(M.log);
    const int rounds = *M.sweeps * nm1;
#pragma unroll
    for (int u = 0; u < JU; ++u) {
        const int j = lane + 32 * u;
        jx[u] = j == 0 ? 0 : 1 + j % nm1;                   // circle(0 + j), circle(0 - j)
        jy[u] = j == 0 || j >= half ? 1 : 1 + nm1 - j;
        next[u] = j < half && rounds > 0 ? log[j] : make_float2(1.f, 0.f);
    }
    __syncwarp();
    for (int rd = 0; rd < rounds; ++rd) {
        log += log_stride(half);
        float2 cs[JU];
        float v[JU][2];
        int p[JU], q[JU];
#pragma unroll
        for (int u = 0; u < JU; ++u) {
            cs[u] = next[u];
            if (lane + 32 * u < half && rd + 1 < rounds) next[u] = log[lane + 32 * u];
            p[u] = jx[u] < jy[u] ? jx[u] : jy[u];
            q[u] = jx[u] < jy[u] ? jy[u] : jx[u];
            jx[u] = jx[u] == 0 ? 0 : jx[u] == nm1 ? 1 : jx[u] + 1;
            jy[u] = jy[u] == nm1 ? 1 : jy[u] + 1;
            if (lane + 32 * u >= half) continue;
            v[u][0] = w[p[u]];
            v[u][1] = !ODD || q[u] < n ? w[q[u]] : 0.f;
        }
#pragma unroll
        for (int u = 0; u < JU; ++u) {
            if (lane + 32 * u >= half) continue;
            w[p[u]] = rot_dif(cs[u].x, v[u][0], cs[u].y, v[u][1]);
            if (!ODD || q[u] < n) w[q[u]] = rot_sum(cs[u].y, v[u][0], cs[u].x, v[u][1]);
        }
        __syncwarp();
    }
    for (int c = lane; c < n; c += 32) M.V[(size_t)r * n + c] = w[c];
}

using ClusterKernel = void (*)(const JacobiMat, int);

template <bool ODD> ClusterKernel cluster_kernel_of(int n) {
    return n <= 64 ? jacobi_cluster_kernel<1, ODD> : n <= 128 ? jacobi_cluster_kernel<2, ODD>
           : n <= 256 ? jacobi_cluster_kernel<4, ODD> : jacobi_cluster_kernel<8, ODD>;
}
ClusterKernel cluster_kernel(int n) { return n & 1 ? cluster_kernel_of<true>(n) : cluster_kernel_of<false>(n); }

cudaLaunchConfig_t cluster_config(int n, cudaLaunchAttribute* attr, cudaStream_t st) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(cluster_ctas(n));
    cfg.blockDim = dim3(CT);
    cfg.dynamicSmemBytes = cluster_smem(n);
    cfg.stream = st;
    attr->id = cudaLaunchAttributeClusterDimension;
    attr->val.clusterDim.x = cluster_ctas(n); attr->val.clusterDim.y = 1; attr->val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cfg;
}

// per device: set on every call (cheap next to the launch)
cudaError_t cluster_attributes(int n) {
    const void* k = reinterpret_cast<const void*>(cluster_kernel(n));
    const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)cluster_smem(512));
    return e != cudaSuccess ? e : cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
}

}  // namespace

bool jacobi_cluster_ok(int n) {
    if (n < 1 || n > 512) return false;
    cudaLaunchAttribute attr{};
    const cudaLaunchConfig_t cfg = cluster_config(n, &attr, nullptr);
    int clusters = 0;
    if (cluster_attributes(n) != cudaSuccess ||
        cudaOccupancyMaxActiveClusters(&clusters, reinterpret_cast<const void*>(cluster_kernel(n)), &cfg) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return clusters > 0;
}

cudaError_t jacobi_cluster(const JacobiMat& M, int max_sweeps, cudaStream_t st) {
    if (M.n < 1 || M.n > 512 || (M.n > 256 && !M.log) || !M.sweeps) return cudaErrorInvalidValue;
    const cudaError_t e = cluster_attributes(M.n);
    if (e != cudaSuccess) return e;
    cudaLaunchAttribute attr{};
    const cudaLaunchConfig_t cfg = cluster_config(M.n, &attr, st);
    const cudaError_t le = cudaLaunchKernelEx(&cfg, cluster_kernel(M.n), M, max_sweeps);
    if (le != cudaSuccess || M.n <= 256) return le;
    ++more_launches;
    if (M.n & 1) jacobi_rows_kernel<8, true><<<(M.n + 3) / 4, 128, sizeof(float) * 4 * M.n, st>>>(M);
    else jacobi_rows_kernel<8, false><<<(M.n + 3) / 4, 128, sizeof(float) * 4 * M.n, st>>>(M);
    return cudaGetLastError();
}

size_t jacobi_log_floats(int n, int max_sweeps) {
    if (n <= 256 || n > 512) return 0;
    const size_t npad = n + (n & 1);
    return (size_t)max_sweeps * (npad - 1) * 2 * log_stride((int)npad / 2);
}

int jacobi_group_grid() {
    static int grid = 0;
    if (!grid) {
        int dev = 0, sms = 0, per = 0, coop = 0;
        if (cudaGetDevice(&dev) != cudaSuccess ||
            cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
            cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) != cudaSuccess || !coop ||
            cudaFuncSetAttribute(jacobi_group_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kJacobiMaxSmem) != cudaSuccess ||
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, jacobi_group_kernel, JT, kJacobiMaxSmem) != cudaSuccess || per < 1)
            return 0;
        grid = sms * (per < 2 ? per : 2);
    }
    return grid;
}

size_t jacobi_rot_floats(int n) { return 4 * (size_t)((n + (n & 1)) / 2); }

cudaError_t jacobi_group(const JacobiGroup& g, int grid, cudaStream_t st) {
    if (g.nmat <= 0) return cudaSuccess;
    if (grid <= 0 || grid > kJacobiMaxGrid) return cudaErrorInvalidValue;
    size_t smem = 0;
    for (int i = 0; i < g.nmat; ++i) {
        if (g.mat[i].soff != (int)smem) return cudaErrorInvalidValue;
        smem += jacobi_rot_floats(g.mat[i].n);
    }
    smem *= sizeof(float);
    if (smem > kJacobiMaxSmem) return cudaErrorInvalidValue;
    {   // per device: set on every call (cheap next to the launch)
        const cudaError_t ea = cudaFuncSetAttribute(jacobi_group_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kJacobiMaxSmem);
        if (ea != cudaSuccess) return ea;
    }
    cudaError_t e = cudaMemsetAsync(g.bar, 0, 2 * sizeof(int), st);    // arrivals and generation
    if (e != cudaSuccess) return e;
    void* args[] = {const_cast<JacobiGroup*>(&g)};
    return cudaLaunchCooperativeKernel(reinterpret_cast<const void*>(jacobi_group_kernel), dim3(grid), dim3(JT), args, smem, st);
}

}  // namespace glr
