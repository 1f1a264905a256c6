// One sweep of parallel two-sided Jacobi on a 128 x 128 symmetric block, held in the registers of
// one 512-thread CTA: the inner solver of the blocked Jacobis (k_bjac.cu, k_eig.cu), and for 128
// indices or fewer, repeated, the whole solver.
//
// The 128 indices are split into groups of 2 g consecutive ones, each group into a half A and a
// half B of g.  A level of g rounds rotates every A index once against every B index of its group
// (round s pairs A_j with B_(j + s) mod g).  Level g = 64 is the cross sweep of two 64-index blocks;
// the levels 64, 32, .., 1 together visit every pair of the 128 indices once (127 rounds).
//
// B is kept in its rotated order, so a round always pairs position j of A with position j of B and
// the 2 x 2 block of rotations i, j is (AA, AB, BA, BB)[i][j]: four values of one thread.  Warp w
// holds rows 4 w .. + 3 of the four 64 x 64 quadrants and lane l columns 2 l and 2 l + 1 as packed
// fp32 pairs (fma.rn.f32x2), and the eigenvector block W the same way (8 rows a warp, or 2).  After a
// round B moves on by one position: columns by one shuffle per value pair, rows inside the warp's
// registers with the last one from the next warp through shared memory (double-buffered, one
// barrier a round).  Every warp forms all 64 rotations itself, two a lane, from the diagonal, which
// it carries along (app - t apq, aqq + t apq), and the 64 off-diagonal entries of the next round's
// pairs, which their owners publish with the boundary rows.  W trails the rotations by a round, so
// that its updates fill the latency of the next rotations.
//
// Bound by instruction issue (16 warps, 340 instructions each a round, 0.58 of the issue slots; 96
// packed fmas at two cycles): 1.15 us a round.  A sweep that keeps S and W in shared memory and
// updates them through indices takes 2.4 us a round.
#pragma once

#include "glr_internal.cuh"

namespace glr {
namespace pair {

constexpr int PN = 128, PTHREADS = 512;
constexpr int PLD = 130;                                   // pitch of S and W in shared memory
constexpr size_t kSmem = sizeof(float) * (2 * PN * PLD + 2 * 16 * 128 + 2 * 64);

using u64 = unsigned long long;
__device__ __forceinline__ u64 pk(float lo, float hi) {
    u64 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void unpk(u64 v, float& lo, float& hi) { asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v)); }
__device__ __forceinline__ u64 mul2(u64 a, u64 b) {
    u64 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ u64 fma2(u64 a, u64 b, u64 c) {
    u64 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}

// The plane rotation that zeroes apq (Golub & Van Loan, sym.schur2), t = tan; the identity when apq
// is negligible.  t only sets the angle, so its division and roots are the hardware's approximations;
// c is refined by a Newton step, so that c^2 + s^2 = c^2 (1 + t^2) is 1 to rounding.
__device__ __forceinline__ void rotation(float app, float aqq, float apq, float& c, float& s, float& t) {
    float root;
    asm("sqrt.approx.f32 %0, %1;" : "=f"(root) : "f"(fabsf(app * aqq)));
    const bool on = fabsf(apq) > 1e-30f && fabsf(apq) > 1e-9f * root;
    const float theta = __fdividef(aqq - app, 2.f * apq);
    asm("sqrt.approx.f32 %0, %1;" : "=f"(root) : "f"(fmaf(theta, theta, 1.f)));
    t = on ? copysignf(__fdividef(1.f, fabsf(theta) + root), theta) : 0.f;
    const float h = fmaf(t, t, 1.f);
    float r;
    asm("rsqrt.approx.f32 %0, %1;" : "=f"(r) : "f"(h));
    c = r * fmaf(-0.5f * h * r, r, 1.5f);
    c = on ? c : 1.f;
    s = t * c;
}

// WR: rows of W a warp (8: all 128 in this CTA; 2: a quarter of them, where four CTAs share a pair, each
// with all of S: the rotations are the same in every one).
template <int WR>
struct Block {
    u64 AA[4], AB[4], BA[4], BB[4], WA[WR], WB[WR];

    // Position j of half A / B at level g -> index in the block.
    static __device__ __forceinline__ int posA(int j, int g) { return 2 * (j & ~(g - 1)) + (j & (g - 1)); }
    static __device__ __forceinline__ int posB(int j, int g) { return posA(j, g) + g; }

    static __device__ __forceinline__ u64 row2(const float* row, int p0, int p1, bool v2) {
        if (v2) return *reinterpret_cast<const u64*>(row + p0);
        return pk(row[p0], row[p1]);
    }
    static __device__ __forceinline__ void put2(float* row, int p0, int p1, bool v2, u64 v) {
        if (v2) { *reinterpret_cast<u64*>(row + p0) = v; return; }
        unpk(v, row[p0], row[p1]);
    }

    // The S quadrants (and W) of level g from / to shared memory.
    __device__ __forceinline__ void load(const float* S, const float* W, int g, int warp, int lane) {
        const bool v2 = g > 1;
        const int a0 = posA(2 * lane, g), a1 = posA(2 * lane + 1, g);
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const float* ra = S + posA(4 * warp + r, g) * PLD;
            const float* rb = S + posB(4 * warp + r, g) * PLD;
            AA[r] = row2(ra, a0, a1, v2); AB[r] = row2(ra, a0 + g, a1 + g, v2);
            BA[r] = row2(rb, a0, a1, v2); BB[r] = row2(rb, a0 + g, a1 + g, v2);
        }
#pragma unroll
        for (int r = 0; r < WR; ++r) {
            const float* rw = W + (WR * warp + r) * PLD;
            WA[r] = row2(rw, a0, a1, v2); WB[r] = row2(rw, a0 + g, a1 + g, v2);
        }
    }
    __device__ __forceinline__ void store(float* S, float* W, int g, int warp, int lane) const {
        const bool v2 = g > 1;
        const int a0 = posA(2 * lane, g), a1 = posA(2 * lane + 1, g);
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            float* ra = S + posA(4 * warp + r, g) * PLD;
            float* rb = S + posB(4 * warp + r, g) * PLD;
            put2(ra, a0, a1, v2, AA[r]); put2(ra, a0 + g, a1 + g, v2, AB[r]);
            put2(rb, a0, a1, v2, BA[r]); put2(rb, a0 + g, a1 + g, v2, BB[r]);
        }
        storeW(W, g, warp, lane);
    }
    __device__ __forceinline__ void storeW(float* W, int g, int warp, int lane) const {
        const bool v2 = g > 1;
        const int a0 = posA(2 * lane, g), a1 = posA(2 * lane + 1, g);
#pragma unroll
        for (int r = 0; r < WR; ++r) {
            float* rw = W + (WR * warp + r) * PLD;
            put2(rw, a0, a1, v2, WA[r]); put2(rw, a0 + g, a1 + g, v2, WB[r]);
        }
    }

    // The g rounds of level g.  S and W hold the block in shared memory and the registers its
    // level-g arrangement; on return only the registers are current (B back in its own order).
    // xch: 2 x 16 x 128 floats, apq: 2 x 64 floats of shared memory.  A block of 2 lim < 128 indices
    // takes lim / 4 warps and levels up to lim; the columns past it hold zeros.
    __device__ __forceinline__ void level(const float* S, int g, float* xch, float* apq, int warp, int lane, int lim = 64) {
        const int j0 = 2 * lane, j1 = 2 * lane + 1;
        float app0 = 0.f, app1 = 0.f, aqq0 = 0.f, aqq1 = 0.f, apq0 = 0.f, apq1 = 0.f;
        if (j0 < lim) {
            app0 = S[posA(j0, g) * (PLD + 1)]; app1 = S[posA(j1, g) * (PLD + 1)];
            aqq0 = S[posB(j0, g) * (PLD + 1)]; aqq1 = S[posB(j1, g) * (PLD + 1)];
            apq0 = S[posA(j0, g) * PLD + posB(j0, g)]; apq1 = S[posA(j1, g) * PLD + posB(j1, g)];
        }
        const int hg = g > 1 ? g / 2 : 1;
        const int src = (lane & ~(hg - 1)) | ((lane + 1) & (hg - 1));
        const int row = 4 * warp;                              // next warp's first row in the group
        const int nw = g >= 8 ? (((row + 4) & (g - 1)) ? warp + 1 : (row + 4 - g) >> 2) : warp;
        u64 pc = pk(1.f, 1.f), ps = 0;                         // the previous round's rotations, for W
        for (int s = 0; s < g; ++s) {
            float c0, s0, t0, c1, s1, t1;
            rotation(app0, aqq0, apq0, c0, s0, t0);
            rotation(app1, aqq1, apq1, c1, s1, t1);
            if (s > 0) turnW(pc, ps, g, src);
            app0 = fmaf(-t0, apq0, app0); aqq0 = fmaf(t0, apq0, aqq0);
            app1 = fmaf(-t1, apq1, app1); aqq1 = fmaf(t1, apq1, aqq1);
            const u64 cj = pk(c0, c1), sj = pk(s0, s1), nj = pk(-s0, -s1);
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const float cr = __shfl_sync(0xffffffffu, (r & 1) ? c1 : c0, 2 * warp + (r >> 1));
                const float sr = __shfl_sync(0xffffffffu, (r & 1) ? s1 : s0, 2 * warp + (r >> 1));
                const u64 ci = pk(cr, cr), si = pk(sr, sr), ni = pk(-sr, -sr);
                const u64 a00 = fma2(ci, AA[r], mul2(ni, BA[r])), a10 = fma2(si, AA[r], mul2(ci, BA[r]));
                const u64 a01 = fma2(ci, AB[r], mul2(ni, BB[r])), a11 = fma2(si, AB[r], mul2(ci, BB[r]));
                AA[r] = fma2(cj, a00, mul2(nj, a01)); AB[r] = fma2(sj, a00, mul2(cj, a01));
                BA[r] = fma2(cj, a10, mul2(nj, a11)); BB[r] = fma2(sj, a10, mul2(cj, a11));
            }
            pc = cj; ps = sj;
            if (g == 1) break;                                 // one pair a group: nothing moves
            // B moves on by one: the columns of AB and BB (and the diagonal) ...
#pragma unroll
            for (int r = 0; r < 4; ++r) { AB[r] = turn(AB[r], src); BB[r] = turn(BB[r], src); }
            const float q = __shfl_sync(0xffffffffu, aqq0, src);
            aqq0 = aqq1; aqq1 = q;
            // ... and the rows of BA and BB; the next round's off-diagonal entries go out
            float* xb = xch + (s & 1) * (16 * 128);
            float* ab = apq + (s & 1) * 64;
            *reinterpret_cast<u64*>(xb + warp * 128 + 2 * lane) = BA[0];
            *reinterpret_cast<u64*>(xb + warp * 128 + 64 + 2 * lane) = BB[0];
            if ((lane >> 1) == warp) {
                float x, y, z;
                unpk((lane & 1) ? AB[2] : AB[0], x, z);
                unpk((lane & 1) ? AB[3] : AB[1], z, y);
                *reinterpret_cast<float2*>(ab + 2 * lane) = make_float2(x, y);
            }
            __syncthreads();
            if (j0 < lim) {
                const float2 nx = *reinterpret_cast<const float2*>(ab + 2 * lane);
                apq0 = nx.x; apq1 = nx.y;
            }
            if (g > 2) {
                BA[0] = BA[1]; BA[1] = BA[2]; BA[2] = BA[3];
                BB[0] = BB[1]; BB[1] = BB[2]; BB[2] = BB[3];
                BA[3] = *reinterpret_cast<const u64*>(xb + nw * 128 + 2 * lane);
                BB[3] = *reinterpret_cast<const u64*>(xb + nw * 128 + 64 + 2 * lane);
            } else {
                u64 x = BA[0]; BA[0] = BA[1]; BA[1] = x;
                x = BA[2]; BA[2] = BA[3]; BA[3] = x;
                x = BB[0]; BB[0] = BB[1]; BB[1] = x;
                x = BB[2]; BB[2] = BB[3]; BB[3] = x;
            }
        }
        turnW(pc, ps, g, src);
    }

private:
    static __device__ __forceinline__ u64 turn(u64 v, int src) {
        float lo, hi;
        unpk(v, lo, hi);
        return pk(hi, __shfl_sync(0xffffffffu, lo, src));
    }
    __device__ __forceinline__ void turnW(u64 c, u64 s, int g, int src) {
        float s0, s1;
        unpk(s, s0, s1);
        const u64 n = pk(-s0, -s1);
#pragma unroll
        for (int r = 0; r < WR; ++r) {
            const u64 x = fma2(c, WA[r], mul2(n, WB[r])), y = fma2(s, WA[r], mul2(c, WB[r]));
            WA[r] = x;
            WB[r] = g > 1 ? turn(y, src) : y;
        }
    }
};

// The sweep of one pair block: S from S0 (row pitch ld), the CTA's rows w0 .. w0 + 16 WR - 1 of W from
// the identity; the 64 cross rounds, or with `full` all 127.  On return W holds those rows (pitch PLD).
// sm: kSmem bytes.
template <int WR, class Load>
__device__ __forceinline__ float* sweep(const float* S0, int64_t ld, int w0, int full, float* sm, Load load2) {
    float* S = sm;
    float* W = S + PN * PLD;
    float* xch = W + PN * PLD;
    float* apq = xch + 2 * 16 * 128;
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
    for (int e = t; e < PN * PN / 2; e += PTHREADS) {
        const int r = e >> 6, c = 2 * (e & 63);
        *reinterpret_cast<float2*>(S + r * PLD + c) = load2(S0 + (int64_t)r * ld + c);
        if (r < 16 * WR)
            *reinterpret_cast<float2*>(W + r * PLD + c) = make_float2(w0 + r == c ? 1.f : 0.f, w0 + r == c + 1 ? 1.f : 0.f);
    }
    __syncthreads();
    Block<WR> b;
    const int last = full ? 1 : 64;
    for (int lv = 64;; lv >>= 1) {
        b.load(S, W, lv, warp, lane);
        b.level(S, lv, xch, apq, warp, lane);
        __syncthreads();
        if (lv == last) { b.storeW(W, lv, warp, lane); break; }
        b.store(S, W, lv, warp, lane);
        __syncthreads();
    }
    __syncthreads();
    return W;
}

}  // namespace pair
}  // namespace glr
