// The refresh's eigen-solvers at their sweep limit, called as the host code calls them (linked with
// libglr.so): a random symmetric matrix is counted in *failed after one sweep and not within the
// ordinary limit; with a NaN in it the solvers of the truncated refresh count it, those of the full
// basis do not.  Prints "ok" or the first violation.
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <vector>

#include "glr_internal.cuh"

using namespace glr;

#define CK(x)                                                                                     \
    do {                                                                                          \
        const cudaError_t e_ = (x);                                                               \
        if (e_ != cudaSuccess) { std::printf("%s: %s\n", #x, cudaGetErrorString(e_)); return -1; } \
    } while (0)

enum Solver { kSmall, kGroup, kCluster, kGrid, kOneCta, kTail };

// The failures counted for an n x n problem with this sweep limit; -1 on a CUDA error.
static int failures(Solver solver, int n, int max_sweeps, bool nan) {
    std::vector<float> H((size_t)n * n);
    std::srand(n);
    for (int i = 0; i < n; ++i)
        for (int j = 0; j <= i; ++j) H[(size_t)i * n + j] = H[(size_t)j * n + i] = std::rand() / (float)RAND_MAX - 0.5f;
    if (nan) H[0] = NAN;
    float *dH, *H2, *V, *evals, *ws, *part, *log, *R;
    int* flags;                                            // sweeps, failed, two of a barrier, the barrier's errors
    const size_t nn = (size_t)n * n * sizeof(float);
    CK(cudaMalloc(&dH, nn)); CK(cudaMalloc(&H2, nn)); CK(cudaMalloc(&V, nn)); CK(cudaMalloc(&R, nn));
    CK(cudaMalloc(&evals, 2 * n * sizeof(float)));
    CK(cudaMalloc(&ws, (eig_ws_floats(n) + 1) * sizeof(float)));
    CK(cudaMalloc(&part, (size_t)2 * kGroupMax * kJacobiMaxGrid * sizeof(float)));
    CK(cudaMalloc(&log, (jacobi_log_floats(n, max_sweeps) + 1) * sizeof(float)));
    CK(cudaMalloc(&flags, 8 * sizeof(int)));
    CK(cudaMemset(flags, 0, 8 * sizeof(int)));
    CK(cudaMemcpy(dH, H.data(), nn, cudaMemcpyHostToDevice));
    const float tol = 4.f * 5.96e-8f * std::sqrt((float)n) + 1e-7f;
    if (solver == kSmall || solver == kGroup) {
        EigGroup g{};
        g.nmat = 1; g.max_sweeps = max_sweeps; g.bar = flags + 2; g.err = flags + 4; g.part = part;
        EigMat& M = g.mat[0];
        M.n = n; M.tol = tol; M.H = dH; M.ld = n; M.V = V; M.evals = evals; M.sweeps = flags; M.ws = ws; M.failed = flags + 1;
        if (solver == kSmall) CK(eig_small_group(g, nullptr));
        else CK(eig_group(g, nullptr));
    } else if (solver == kTail) {
        TailGroup g{};
        g.nmat = 1;
        TailMat& M = g.mat[0];
        M.mp = n; M.k = n; M.H = dH; M.evals = evals; M.evals_sorted = evals + n; M.sweeps = flags; M.failed = flags + 1; M.R = R;
        CK(tail_group(g, 0, nullptr));
    } else {
        JacobiMat M{};
        M.n = n; M.tol = tol; M.H = dH; M.H2 = H2; M.V = V; M.evals = evals; M.sweeps = flags; M.failed = flags + 1; M.log = log;
        if (solver == kCluster) {
            if (!jacobi_cluster_ok(n)) { std::printf("no room for a cluster\n"); return -1; }
            CK(jacobi_cluster(M, max_sweeps, nullptr));
        } else if (solver == kGrid) {
            JacobiGroup g{};
            g.nmat = 1; g.max_sweeps = max_sweeps; g.bar = flags + 2; g.err = flags + 4; g.part = part; g.mat[0] = M;
            CK(jacobi_group(g, jacobi_group_grid(), nullptr));
        } else {
            CK(jacobi_eig(dH, n, V, evals, flags, flags + 1, nullptr));
        }
    }
    CK(cudaDeviceSynchronize());
    int got[8];
    CK(cudaMemcpy(got, flags, sizeof(got), cudaMemcpyDeviceToHost));
    for (void* p : {(void*)dH, (void*)H2, (void*)V, (void*)R, (void*)evals, (void*)ws, (void*)part, (void*)log, (void*)flags}) CK(cudaFree(p));
    if (got[4]) { std::printf("a barrier gave up\n"); return -1; }
    return got[1];
}

int main() {
    const struct { Solver solver; const char* name; int n; bool limited, counts_nan; } cases[] = {
        {kSmall, "eig_small_group", 12, true, true},   {kSmall, "eig_small_group", 100, true, true},
        {kGroup, "eig_group", 132, true, true},        {kGroup, "eig_group", 256, true, true},
        {kCluster, "jacobi_cluster", 100, true, false}, {kCluster, "jacobi_cluster", 301, true, false},
        {kGrid, "jacobi_group", 520, true, false},     {kOneCta, "jacobi_eig", 40, false, false},
        {kTail, "tail_group", 16, false, true},        {kTail, "tail_group", 31, false, true},
    };
    for (const auto& c : cases) {
        const int one = c.limited ? failures(c.solver, c.n, 1, false) : 1;
        const int usual = failures(c.solver, c.n, kJacobiSweeps, false), nan = failures(c.solver, c.n, kJacobiSweeps, true);
        if (one != 1 || usual != 0 || nan != (c.counts_nan ? 1 : 0)) {
            std::printf("%s n %d: %d failures after one sweep, %d within the limit, %d with a NaN\n", c.name, c.n, one, usual, nan);
            return 1;
        }
    }
    std::printf("ok\n");
    return 0;
}
