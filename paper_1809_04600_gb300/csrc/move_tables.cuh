// Tabulated single moves of the strings of V.
#pragma once
#include <algorithm>

#include "context.cuh"
#include "enumerate.cuh"

namespace shci {

// Single moves p -> r of a determinant (A, B): the element is
//   [h_pr + sum_{k in A} ((pr|kk) - (pk|kr))] + sum_{k in B} (pr|kk)
// (k = p contributes an exact zero to the first sum), a term of the moving
// string and one of the other.  Both are tabulated for every string of V and
// every orbital pair, M[u][0][pr] and M[u][1][pr], so that a move costs one
// FP64 addition instead of one per electron: those additions held the FP64
// pipe (74 % busy in the count pass).
template <int W>
static __global__ void k_move_tables(const uint64_t *__restrict__ str, int64_t U, DevInts I, double *__restrict__ M) {
    const int n = I.n, np = n * (n + 1) / 2;
    const int64_t total = U * np;
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < total; t += (int64_t)gridDim.x * blockDim.x) {
        const int64_t u = t / np;
        const int pr = (int)(t - u * np);
        int p = (int)((sqrtf(8.0f * (float)pr + 1.0f) - 1.0f) * 0.5f);
        while (p * (p + 1) / 2 > pr) p--;
        while ((p + 1) * (p + 2) / 2 <= pr) p++;
        const int r = pr - p * (p + 1) / 2;
        const double *jk = I.jk1 + (int64_t)(p * n + r) * n, *j1 = I.j1 + (int64_t)(p * n + r) * n;
        double same = __ldg(&I.h[p * n + r]), opp = 0.0;
        for_bits_above<W>(load_str<W>(str, u), -1, [&](int k) {
            same += __ldg(&jk[k]);
            opp += __ldg(&j1[k]);
        });
        M[2 * u * np + pr] = same;
        M[(2 * u + 1) * np + pr] = opp;
    }
}

// the tables of V's strings: [U][2][n (n + 1) / 2] per spin
template <int W>
static void make_move_tables(shci_ctx *c, const DevInts &I, DevBuf<double> &ma, DevBuf<double> &mb) {
    const int64_t np = (int64_t)c->n_orb * (c->n_orb + 1) / 2;
    ma.alloc((size_t)(2 * c->Ua * np));
    mb.alloc((size_t)(2 * c->Ub * np));
    auto grid = [&](int64_t m) { return (unsigned)std::min<int64_t>(ceil_div(m, 256), (int64_t)c->n_sm * 32); };
    k_move_tables<W><<<grid(c->Ua * np), 256, 0, c->st>>>(c->astr.p, c->Ua, I, ma.p);
    k_move_tables<W><<<grid(c->Ub * np), 256, 0, c->st>>>(c->bstr.p, c->Ub, I, mb.p);
    KERNEL_CHECK();
    g_kernel_launches += 2;
}

}  // namespace shci
