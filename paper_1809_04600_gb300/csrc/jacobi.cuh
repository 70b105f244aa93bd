// Subspace eigen-solver of the Davidson iteration (one CTA per matrix).
#pragma once
#include "common.cuh"

namespace shci {

// Cholesky-QR coefficients for kb (<= SHCI_MAX_K) vectors with Gram matrix S
// (kb x kb, row-major).  Column l is dropped when its component outside the
// span of the accepted earlier columns has squared norm below rel * ref[l]
// (ref: S's diagonal when null).  Writes M (kb x kb) such that the accepted
// columns q_l' = sum_j M[j * kb + l'] t_j are orthonormal (columns l' >=
// count are zero) and returns the number accepted.  Single thread.
__device__ __forceinline__ int cholqr_coef(const double *S, int kb, const double *ref, double rel, double *M) {
    double R[SHCI_MAX_K][SHCI_MAX_K];
    double Mi[SHCI_MAX_K][SHCI_MAX_K];   // Mi[j][l]: coefficient of t_j in q_l
    int acc[SHCI_MAX_K];
    int na = 0;
    for (int l = 0; l < kb; l++)
        for (int j = 0; j < kb; j++) { R[j][l] = 0.0; Mi[j][l] = 0.0; }
    for (int l = 0; l < kb; l++) {
        // R[j][l] for accepted j < l
        for (int x = 0; x < na; x++) {
            int j = acc[x];
            double s = S[j * kb + l];
            for (int y = 0; y < x; y++) s -= R[acc[y]][j] * R[acc[y]][l];
            R[j][l] = s / R[j][j];
        }
        double d = S[l * kb + l];
        for (int x = 0; x < na; x++) d -= R[acc[x]][l] * R[acc[x]][l];
        double r0 = ref ? ref[l] : S[l * kb + l];
        if (!(d > rel * r0) || !(d > 1e-300)) continue;      // numerically dependent: drop
        R[l][l] = sqrt(d);
        // q_l = (t_l - sum_{j acc} R[j][l] q_j) / R[l][l]
        for (int j = 0; j < kb; j++) {
            double v = (j == l) ? 1.0 : 0.0;
            for (int x = 0; x < na; x++) v -= R[acc[x]][l] * Mi[j][acc[x]];
            Mi[j][l] = v / R[l][l];
        }
        acc[na++] = l;
    }
    for (int j = 0; j < kb; j++)
        for (int x = 0; x < kb; x++) M[j * kb + x] = x < na ? Mi[j][acc[x]] : 0.0;
    return na;
}

// Eigen-decomposition of the symmetric m x m matrix G (row-major, leading
// dimension ld) by cyclic Jacobi with Brent-Luk parallel ordering (m/2
// disjoint rotations per round).
//
// Warm start: when m_prev > 0, evec holds the eigenvectors of G's leading
// m_prev x m_prev block from the previous call (G only grew since), so in
// the basis blockdiag(evec, I) the leading block is diag(eval) and only the
// new border has to be transformed.  Rotations whose off-diagonal element is
// below 1e-14 (|a_pp| + |a_qq|) become the identity, a round with none active
// is skipped, and sweeps stop when one applies no rotation.  A round applies
// its active rotations in one pass over the 2 x 2 blocks they touch (two
// barriers per round).  One SM issues few FP64 instructions (a warp-wide FP64
// instruction occupies its FP64 pipe for many cycles), so no FP64 work is
// spent on identity blocks and the work is packed into few warps.  Output:
// eigenvalues (the converged diagonal) ascending and eigenvectors as columns,
// evec[l * ld + a] = component a of vector l.
//
// The working matrix A lives in shared memory (jsm).  The accumulated
// rotation Q lives there too (QSHARED, JACOBI_SMEM bytes in all), or in the
// global scratch qg of JACOBI_Q_DOUBLES doubles owned by the calling CTA
// (JACOBI_SMEM_A bytes of shared memory), accessed through L2.
template <bool QSHARED = true>
__device__ __forceinline__ void jacobi_solve(const double *G, int ld, int m, int m_prev,
                                             double *__restrict__ eval, double *__restrict__ evec, double *jsm,
                                             double *qg = nullptr) {
    constexpr int QL = SHCI_MAX_SUB + 1;
    double (*A)[QL] = reinterpret_cast<double (*)[QL]>(jsm);
    double *Qp = QSHARED ? jsm + SHCI_MAX_SUB * QL : qg;
    auto qget = [&](int r, int c) { return QSHARED ? Qp[r * QL + c] : __ldcg(&Qp[r * QL + c]); };
    auto qset = [&](int r, int c, double v) {
        if (QSHARED) Qp[r * QL + c] = v;
        else __stcg(&Qp[r * QL + c], v);
    };
    __shared__ double cs[SHCI_MAX_SUB / 2], sn[SHCI_MAX_SUB / 2];
    __shared__ int pp[SHCI_MAX_SUB / 2], qq[SHCI_MAX_SUB / 2];
    __shared__ double lam[SHCI_MAX_SUB];
    const int mm = (m + 1) & ~1;
    const int tid = threadIdx.x, nt = blockDim.x;
    const int mp = (m_prev > 0 && m_prev <= m) ? m_prev : 0;
    // G is read symmetrised, (G + G^T) / 2, from L2 (ld.global.cg: the caller may
    // have written it earlier in the same kernel)
    auto gs = [&](int r, int c) { return 0.5 * (__ldcg(&G[r * ld + c]) + __ldcg(&G[c * ld + r])); };
    // Q = blockdiag(previous eigenvectors, I)
    for (int e = tid; e < mm * mm; e += nt) {
        int r = e / mm, c = e % mm;
        double q = (r == c) ? 1.0 : 0.0;
        if (r < mp && c < mp) q = __ldcg(&evec[c * ld + r]);
        qset(r, c, q);
    }
    __syncthreads();
    // A = Q^T G Q: leading block diag(previous eigenvalues), border transformed, trailing block copied
    for (int e = tid; e < mm * mm; e += nt) {
        int r = e / mm, c = e % mm;
        double v = 0.0;
        if (r < m && c < m) {
            if (r < mp && c < mp) {
                v = (r == c) ? __ldcg(&eval[r]) : 0.0;
            } else if (r < mp) {          // (Q^T G)[r][c] for border column c
                for (int s = 0; s < mp; s++) v = fma(qget(s, r), gs(s, c), v);
            } else if (c < mp) {
                for (int s = 0; s < mp; s++) v = fma(qget(s, c), gs(r, s), v);
            } else {
                v = gs(r, c);
            }
        }
        A[r][c] = v;
    }
    __syncthreads();
    if (mm != m && tid == 0) {
        // padding index: decoupled, with a diagonal value above every Gershgorin bound
        double bound = 0.0;
        for (int r = 0; r < m; r++) {
            double s = 0.0;
            for (int c = 0; c < m; c++) s += fabs(A[r][c]);
            bound = fmax(bound, s);
        }
        A[m][m] = 2.0 * bound + 1.0;
    }
    __syncthreads();
    const int half = mm / 2;                 // <= 32: the rotations of a round fit one warp
    __shared__ int act_idx[SHCI_MAX_SUB / 2];
    __shared__ int act_pos[SHCI_MAX_SUB / 2];
    __shared__ int n_act[2];
    for (int sweep = 0; sweep < 30; sweep++) {
        int swept = 0;
        for (int round = 0; round < mm - 1; round++) {
            // warp 0: the round's mm/2 disjoint pairs, their rotations and the list of
            // active ones (an inactive pair is the identity)
            if (tid < 32) {
                int active = 0;
                if (tid < half) {
                    int x = tid, y = mm - 1 - tid;
                    int p = x == 0 ? 0 : ((x - 1 + round) % (mm - 1)) + 1;
                    int q = y == 0 ? 0 : ((y - 1 + round) % (mm - 1)) + 1;
                    if (p > q) { int t = p; p = q; q = t; }
                    const double apq = A[p][q];
                    double c = 1.0, s = 0.0;
                    if (fabs(apq) > 1e-14 * (fabs(A[p][p]) + fabs(A[q][q])) + 1e-300) {
                        active = 1;
                        const double diff = A[q][q] - A[p][p];
                        const float tauf = (float)diff / (2.0f * (float)apq);
                        if (fabs(apq) > 1e-30 && isfinite(tauf)) {
                            // rotation angle in FP32 (an FP64 divide or square root is a long
                            // chain of FP64 instructions, and one SM issues few of those),
                            // then (c, s) renormalised in FP64 so that c^2 + s^2 = 1 to FP64
                            // precision: the rotation stays exactly orthogonal and zeroes
                            // a_pq to ~1e-7 relative, which the next sweep finishes
                            const float tf = copysignf(1.0f, tauf) / (fabsf(tauf) + sqrtf(1.0f + tauf * tauf));
                            const float cf = rsqrtf(1.0f + tf * tf);
                            c = (double)cf;
                            s = (double)(tf * cf);
                            double f = 1.5 - 0.5 * (c * c + s * s);
                            c *= f;
                            s *= f;
                            f = 1.5 - 0.5 * (c * c + s * s);
                            c *= f;
                            s *= f;
                        } else {
                            const double tau = diff / (2.0 * apq);
                            const double t = (tau >= 0.0 ? 1.0 : -1.0) / (fabs(tau) + sqrt(1.0 + tau * tau));
                            c = 1.0 / sqrt(1.0 + t * t);
                            s = t * c;
                        }
                    }
                    cs[tid] = c;
                    sn[tid] = s;
                    pp[tid] = p;
                    qq[tid] = q;
                }
                const unsigned mask = __ballot_sync(0xffffffffu, active);
                const int pos = __popc(mask & ((1u << tid) - 1u));
                if (active) act_idx[pos] = tid;
                if (tid < half) act_pos[tid] = active ? pos : -1;
                if (tid == 0) n_act[round & 1] = __popc(mask);
            }
            __syncthreads();
            const int na = n_act[round & 1];       // double-buffered: warp 0 may run ahead
            if (na == 0) continue;                 // uniform
            swept = 1;
            // A <- J^T A J in one pass over 2 x 2 blocks (rows of pair t, columns of
            // pair u): a block depends only on itself and on rotations t and u.  Only
            // blocks touched by an active rotation are computed, enumerated densely
            // (active t, any u; the block of two active pairs once) so that the FP64
            // work sits in as few warps as possible; the block u, t is written as
            // the transpose, which keeps A exactly symmetric.
            for (int e = tid; e < na * half; e += nt) {
                const int x = e / half, u = e - x * half;
                const int t = act_idx[x];
                const int pu = act_pos[u];
                if (pu >= 0 && pu < x) continue;
                const int p = pp[t], q = qq[t], r = pp[u], v = qq[u];
                const double ct = cs[t], st = sn[t], cu = cs[u], su = sn[u];
                const double apr = A[p][r], apv = A[p][v], aqr = A[q][r], aqv = A[q][v];
                const double bpr = ct * apr - st * aqr, bpv = ct * apv - st * aqv;   // rows
                const double bqr = st * apr + ct * aqr, bqv = st * apv + ct * aqv;
                const double npr = cu * bpr - su * bpv, npv = su * bpr + cu * bpv;  // columns
                const double nqr = cu * bqr - su * bqv, nqv = su * bqr + cu * bqv;
                if (t == u) {                      // r = p, v = q
                    A[p][p] = npr;
                    A[q][q] = nqv;
                    A[p][q] = npv;
                    A[q][p] = npv;
                } else {
                    A[p][r] = npr;
                    A[p][v] = npv;
                    A[q][r] = nqr;
                    A[q][v] = nqv;
                    A[r][p] = npr;
                    A[v][p] = npv;
                    A[r][q] = nqr;
                    A[v][q] = nqv;
                }
            }
            // Q <- Q J over the active rotations
            for (int e = tid; e < mm * na; e += nt) {
                const int i = e / na, t = act_idx[e - i * na];
                const int p = pp[t], q = qq[t];
                const double c = cs[t], s = sn[t];
                const double qp = qget(i, p), qv = qget(i, q);
                qset(i, p, c * qp - s * qv);
                qset(i, q, s * qp + c * qv);
            }
            __syncthreads();
        }
        if (!swept) break;               // uniform
    }
    for (int a = tid; a < mm; a += nt) lam[a] = A[a][a];
    __syncthreads();
    // sort ascending (rank by value, ties by index) and write out the first m
    for (int a = tid; a < mm; a += nt) {
        double va = lam[a];
        int rank = 0;
        for (int b = 0; b < mm; b++) {
            double vb = lam[b];
            rank += (vb < va) || (vb == va && b < a);
        }
        if (rank < m) {
            eval[rank] = va;
            for (int r = 0; r < m; r++) evec[rank * ld + r] = qget(r, a);
        }
    }
}

// 1 / t and 1 / sqrt(t) to about an ulp for |t| within FP32's normal range: an
// FP32 value and two Newton steps, straight-line code that several can be in
// flight of.  Outside that range the result is not finite or zero.
__device__ __forceinline__ double fast_rcp(double t) {
    double r = (double)__frcp_rn((float)t);
    r = fma(r, fma(-t, r, 1.0), r);
    return fma(r, fma(-t, r, 1.0), r);
}

__device__ __forceinline__ double fast_rsqrt(double t) {
    double r = (double)__frsqrt_rn((float)t);
    r = fma(0.5 * r, fma(-t * r, r, 1.0), r);
    return fma(0.5 * r, fma(-t * r, r, 1.0), r);
}

// The eigen-decomposition after one more basis vector: eval / evec hold the
// eigenpairs of G's leading n x n block, and row / column n joins.  In their
// basis the matrix is an arrowhead [D z; z^T alpha], whose eigenvalues are the
// roots of f(x) = alpha - x - sum z_i^2 / (d_i - x), one in each interval
// between the poles d_i.  Each root is solved for as its distance mu to the
// nearer pole (a quadratic in mu with that pole kept and the rest linearised:
// in FP32 to ~1e-5, then two steps in FP64), so that every x_j - d_i keeps its
// relative accuracy; the border z is then recomputed from the roots (Gu and
// Eisenstat 1994), which makes the eigenvectors z_i / (x_j - d_i) orthogonal
// to FP64 precision.  A z_i below 1e-15 of the matrix leaves its pair as it is.
// Returns false (uniformly; eval and evec as they were) when two poles with a
// border element lie closer than 1e-12 of the matrix, or a value leaves the
// range of the above: the caller then uses Jacobi.
//
// A warp's FP64 instruction occupies its quarter of the SM for ~76 cycles, so
// sums over poles are split four ways over warps of different quarters (warp
// w: terms w mod 4, roots 32 (w / 4) on).  Needs 256 threads and
// JACOBI_SMEM_A bytes at jsm.
__device__ __forceinline__ bool append_eig(const double *G, int ld, int n, double *__restrict__ eval,
                                           double *__restrict__ evec, double *jsm) {
    constexpr int QL = SHCI_MAX_SUB + 1;
    constexpr int MS = SHCI_MAX_SUB;
    // V is written last; until then its place holds the partial sums.  Little
    // static shared memory: the batched solver runs five CTAs per SM.
    double (*V)[QL] = reinterpret_cast<double (*)[QL]>(jsm);
    double (*part)[4][MS] = reinterpret_cast<double (*)[4][MS]>(jsm);
    __shared__ double dd[MS], zz[MS];                     // all pairs
    __shared__ double d[MS], z[MS];                       // those with a border element
    __shared__ float df[MS], zf[MS];                      // d - alpha and z in units of the scale
    __shared__ double mu[MS], val[MS];
    __shared__ double scale_sh;
    __shared__ uint8_t idx[MS], slot[MS], pole[MS], rank[MS];
    __shared__ int bad, n_on;
    const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, warp = tid >> 5, nw = nt >> 5;
    const int quarter = warp & 3, mine = lane + 32 * (warp >> 2);     // this thread's share of the split sums
    auto gs = [&](int r, int c) { return 0.5 * (__ldcg(&G[r * ld + c]) + __ldcg(&G[c * ld + r])); };
    __syncthreads();
    // z = Q^T g, one warp per pair
    for (int i = warp; i < n; i += nw) {
        double v = 0.0;
        for (int s = lane; s < n; s += 32) v = fma(__ldcg(&evec[i * ld + s]), gs(s, n), v);
#pragma unroll
        for (int o = 16; o >= 1; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (lane == 0) {
            zz[i] = v;
            dd[i] = __ldcg(&eval[i]);
        }
    }
    const double alpha = gs(n, n);
    __syncthreads();
    // scale, the pairs with a border element, their gaps: one warp
    if (warp == 0) {
        double sc = fabs(alpha);
        for (int i = lane; i < n; i += 32) sc = fmax(sc, fmax(fabs(dd[i]), fabs(zz[i])));
        bool wrong = false;
        for (int i = lane; i < n; i += 32) wrong = wrong || !isfinite(dd[i]) || !isfinite(zz[i]);
#pragma unroll
        for (int o = 16; o >= 1; o >>= 1) sc = fmax(sc, __shfl_xor_sync(0xffffffffu, sc, o));
        wrong = wrong || !isfinite(sc) || !isfinite(alpha);
        const double cut = 1e-15 * sc;
        int np = 0;
        for (int i0 = 0; i0 < n; i0 += 32) {
            const int i = i0 + lane;
            const bool on = i < n && fabs(zz[i]) > cut;
            const unsigned m = __ballot_sync(0xffffffffu, on);
            const int at = np + __popc(m & ((1u << lane) - 1u));
            if (on) {
                idx[at] = (uint8_t)i;
                d[at] = dd[i];
                z[at] = zz[i];
            }
            if (i < n) slot[i] = (uint8_t)(on ? 255 : i - at);        // rank among the untouched pairs
            np += __popc(m);
        }
        __syncwarp();
        const float inv = 1.0f / (float)sc;
        for (int i = lane; i < np; i += 32) {
            if (i > 0) wrong = wrong || !(d[i] - d[i - 1] > 1e-12 * sc);
            df[i] = (float)(d[i] - alpha) * inv;
            zf[i] = (float)z[i] * inv;
        }
        wrong = __any_sync(0xffffffffu, wrong);
        if (lane == 0) {
            bad = wrong;
            n_on = np;
            scale_sh = sc;
        }
    }
    __syncthreads();
    if (bad) return false;
    const int p = n_on, total = n + 1;
    const double scale = scale_sh;
    // roots 0 .. p, root r between the poles r - 1 and r; a thread each (warps 0 and 1).
    // z_K^2 / mu + a + b mu = 0 with a + b mu the tangent of the rest of f at the last
    // mu, b < 0: one root of each sign.
    double m = 0.0, lo = 0.0, hi = 0.0, base = 0.0, q = 0.0;
    bool neg = false;
    if (tid <= p && p > 0) {
        const int r = tid;
        int K = r == p ? p - 1 : 0;
        if (r > 0 && r < p) {
            // the nearer pole by the sign of f at the middle (close to zero either pole serves)
            const float at = 0.5f * (df[r - 1] + df[r]);
            float f = -at;
#pragma unroll 4
            for (int i = 0; i < p; i++) f -= zf[i] * __fdividef(zf[i], df[i] - at);
            K = f > 0.0f ? r : r - 1;                     // f descends: positive here, the root is right of it
        }
        const float inv = 1.0f / (float)scale;
        float zn = 0.0f;
        for (int i = 0; i < p; i++) zn = fmaf(zf[i], zf[i], zn);
        neg = K == r;                                     // the root lies left of its pole
        const double out = 1.001 * scale * (double)sqrtf(zn);
        // |mu| is at most the distance to the next pole, or the Gershgorin bound outside them
        const double reach = r == 0 ? fmax(0.0, d[K] - alpha) + out
                                    : (r == p ? fmax(0.0, alpha - d[K]) + out : d[r] - d[r - 1]);
        lo = neg ? -reach : 0.0;
        hi = neg ? 0.0 : reach;
        q = z[K] * z[K];
        base = alpha - d[K];
        const float dfK = df[K], bf = -dfK, qf = zf[K] * zf[K], lof = (float)lo * inv, hif = (float)hi * inv;
        float mf = 0.0f;
        for (int it = 0; it < 10; it++) {
            float s = 0.0f, s1 = 1.0f;
#pragma unroll 4
            for (int i = 0; i < p; i++) {
                const float w = i == K ? 0.0f : __fdividef(zf[i], (df[i] - dfK) - mf);
                s = fmaf(w, zf[i], s);
                s1 = fmaf(w, w, s1);
            }
            const float b = -s1, aa = (bf - mf - s) - b * mf;
            const float e = -aa - copysignf(sqrtf(fmaf(aa, aa, -4.0f * b * qf)), aa);
            const float x = (neg == (aa > 0.0f)) ? __fdividef(2.0f * qf, e) : __fdividef(e, 2.0f * b);
            if (!isfinite(x)) break;
            const float y = fminf(fmaxf(x, lof), hif);
            const bool done = fabsf(y - mf) <= 1e-5f * fabsf(y);
            mf = y;
            if (done) break;
        }
        m = (double)mf * scale;
        if (m == 0.0) m = (neg ? lo : hi) * 0x1p-40;
        pole[r] = (uint8_t)K;
        mu[r] = m;
    }
    __syncthreads();
    if (p > 0) {
        bool done = false;
        for (int it = 0; it < 20; it++) {
            if (mine <= p) {
                const int K = pole[mine];
                const double dK = d[K], mm = mu[mine];
                double s = 0.0, w2 = 0.0;
                for (int i0 = quarter; i0 < p; i0 += 16) {           // four reciprocals in flight
                    double w[4], zi[4];
#pragma unroll
                    for (int u = 0; u < 4; u++) {
                        const int i = min(i0 + 4 * u, p - 1);
                        zi[u] = i0 + 4 * u < p && i != K ? z[i] : 0.0;
                        w[u] = zi[u] * fast_rcp((d[i] - dK) - mm);
                    }
#pragma unroll
                    for (int u = 0; u < 4; u++) {
                        s = fma(w[u], zi[u], s);
                        w2 = fma(w[u], w[u], w2);
                    }
                }
                part[0][quarter][mine] = s;
                part[1][quarter][mine] = w2;
            }
            __syncthreads();
            if (tid <= p && !done) {
                const double s = (part[0][0][tid] + part[0][1][tid]) + (part[0][2][tid] + part[0][3][tid]);
                const double b = -(1.0 + ((part[1][0][tid] + part[1][1][tid]) + (part[1][2][tid] + part[1][3][tid])));
                const double a = (base - m - s) - b * m, y = fma(a, a, -4.0 * b * q);
                const double e = -a - copysign(y * fast_rsqrt(y), a);
                double x = (neg == (a > 0.0)) ? 2.0 * q * fast_rcp(e) : e * fast_rcp(2.0 * b);
                if (!(x >= lo && x <= hi)) x = 0.5 * (m + (x < lo ? lo : hi));
                done = fabs(x - m) <= 1e-8 * fabs(x);     // the error squares from step to step
                m = x;
                mu[tid] = x;
            }
            if (!__syncthreads_or(tid <= p && !done)) break;
        }
        if (tid <= p && (!done || m == 0.0 || !isfinite(m))) bad = 1;     // a root on its pole
    } else if (tid == 0) {
        pole[0] = 0;
    }
    if (tid <= p) val[tid] = p > 0 ? d[pole[tid]] + m : alpha;
    __syncthreads();
    if (bad) return false;
    auto diff = [&](int j, int i) { return (d[pole[j]] - d[i]) + mu[j]; };      // x_j - d_i
    // z_i^2 = -prod_j (x_j - d_i) / prod_j (d_j - d_i): root j or j + 1 over pole j
    if (mine < p) {
        double up = 1.0, dn = 1.0;
        for (int j = quarter; j < p; j += 4) {
            if (j == mine) continue;
            up *= diff(j < mine ? j : j + 1, mine);
            dn *= d[j] - d[mine];
        }
        part[0][quarter][mine] = up / dn;
    }
    // places: the roots are elements 0 .. p, the untouched pairs follow in order
    if (tid > p && tid < total) {
        int i = 0;
        while (slot[i] != tid - p - 1) i++;
        pole[tid] = (uint8_t)i;
        val[tid] = dd[i];
    }
    __syncthreads();
    if (tid < p) {
        const double w = (part[0][0][tid] * part[0][1][tid]) * (part[0][2][tid] * part[0][3][tid]) *
                         (-diff(tid, tid) * diff(tid + 1, tid));
        if (!(w > 0.0) || !isfinite(w)) bad = 1;
        z[tid] = copysign(w * fast_rsqrt(w), z[tid]);
    }
    if (tid >= 64 && tid < 64 + total) {
        const int e = tid - 64;
        int rk = 0;
        for (int j = 0; j < total; j++) rk += val[j] < val[e] || (val[j] == val[e] && j < e);
        rank[e] = (uint8_t)rk;
    }
    __syncthreads();
    if (bad) return false;
    for (int e = tid; e < total * total; e += nt) V[e / total][e % total] = 0.0;
    __syncthreads();
    // eigenvectors in the old basis, unnormalised: z_i / (x_j - d_i), and 1 for the new vector
    for (int e = tid; e < p * (p + 1); e += nt) {
        const int i = e / (p + 1), j = e - i * (p + 1);
        V[idx[i]][rank[j]] = z[i] * fast_rcp(diff(j, i));
    }
    if (tid <= p) V[n][rank[tid]] = 1.0;
    else if (tid < total) V[pole[tid]][rank[tid]] = 1.0;
    __syncthreads();
    // norms (in place of d, z, mu and zz, which are done with), and the sign that
    // makes the largest component positive
    if (mine < total) {
        double nn = 0.0;
#pragma unroll 4
        for (int i = quarter; i < total; i += 4) {
            const double u = V[i][mine];
            nn = fma(u, u, nn);
        }
        (quarter < 2 ? (quarter == 0 ? d : z) : (quarter == 2 ? mu : zz))[mine] = nn;
    }
    __syncthreads();
    if (tid < total) {
        int big = 0, sign = 0;
#pragma unroll 4
        for (int i = 0; i < total; i++) {
            const int h = __double2hiint(V[i][tid]);
            if ((h & 0x7FFFFFFF) > big) {
                big = h & 0x7FFFFFFF;
                sign = h < 0;
            }
        }
        const double f = flip_sign(fast_rsqrt((d[tid] + z[tid]) + (mu[tid] + zz[tid])), sign);
        if (!isfinite(f)) bad = 1;
        zz[tid] = f;
    }
    __syncthreads();
    if (bad) return false;
    // Q <- [Q 0; 0 1] V, a warp per component (its row of Q in the lanes' registers)
    for (int r = warp; r <= n; r += nw) {
        double q0 = 0.0, q1 = 0.0;
        if (r < n) {
            if (lane < n) q0 = __ldcg(&evec[lane * ld + r]);
            if (lane + 32 < n) q1 = __ldcg(&evec[(lane + 32) * ld + r]);
        }
        const int l0 = min(lane, total - 1), l1 = min(lane + 32, total - 1);
        double v0 = 0.0, v1 = 0.0;
        if (r == n) {
            v0 = V[n][l0];
            v1 = V[n][l1];
        } else if (total <= 32) {
#pragma unroll 4
            for (int i = 0; i < n; i++) v0 = fma(__shfl_sync(0xffffffffu, q0, i), V[i][l0], v0);
        } else {
#pragma unroll 4
            for (int i = 0; i < n; i++) {
                const double q = __shfl_sync(0xffffffffu, i < 32 ? q0 : q1, i & 31);
                v0 = fma(q, V[i][l0], v0);
                v1 = fma(q, V[i][l1], v1);
            }
        }
        if (lane < total) evec[lane * ld + r] = v0 * zz[lane];
        if (lane + 32 < total) evec[(lane + 32) * ld + r] = v1 * zz[lane + 32];
    }
    if (tid < total) eval[rank[tid]] = val[tid];
    __syncthreads();
    return true;
}

// Signs of the eigenvectors.  An eigenvector's sign is free, but a caller that
// follows a root from call to call relies on it not changing with the method,
// and the Jacobi iteration's is the outcome of all its rotations.  So those are
// carried out, on the bordered matrix in the old eigenvectors' basis, in FP32
// and without the rotations too small to matter for a sign (angles below
// 1e-4): X holds the eigenvectors they lead to, ~1e-5 accurate, by columns.
// That decides the sign where FP32 tells the eigenvalues apart, which append_eig
// needs of the poles too (closer ones it refuses), and where no rotation's two
// diagonal elements are closer than that (it may turn by +45 degrees here and by
// -45 in FP64).
// FP32 runs at 75 times the FP64 rate, so this takes a third of the FP64
// iteration's time.  A, Qf: 64 x 65 floats each in shared memory; X overwrites A.
__device__ __forceinline__ void jacobi_signs(const double *G, int ld, int m, int mp, const double *eval,
                                             const double *evec, float (*A)[SHCI_MAX_SUB + 1],
                                             float (*Qf)[SHCI_MAX_SUB + 1]) {
    __shared__ float cs[SHCI_MAX_SUB / 2], sn[SHCI_MAX_SUB / 2];
    __shared__ uint8_t pp[SHCI_MAX_SUB / 2], qq[SHCI_MAX_SUB / 2], act[SHCI_MAX_SUB / 2];
    __shared__ int8_t pos[SHCI_MAX_SUB / 2];
    __shared__ int n_act[2];
    const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, warp = tid >> 5, nw = nt >> 5;
    const int mm = (m + 1) & ~1, half = mm / 2;
    auto gs = [&](int r, int c) { return 0.5 * (__ldcg(&G[r * ld + c]) + __ldcg(&G[c * ld + r])); };
    const double shift = __ldcg(&eval[0]);
    __syncthreads();
    for (int e = tid; e < mm * mm; e += nt) {
        const int r = e / mm, c = e % mm;
        float v = 0.0f;
        if (r == c) v = r < mp ? (float)(__ldcg(&eval[r]) - shift) : (r < m ? (float)(gs(r, r) - shift) : 3.0e18f);
        else if (r >= mp && c >= mp && r < m && c < m) v = (float)gs(r, c);
        A[r][c] = v;
        Qf[r][c] = r == c ? 1.0f : 0.0f;
    }
    __syncthreads();
    // the border in the old basis, a warp per entry
    for (int e = warp; e < mp * (m - mp); e += nw) {
        const int i = e % mp, c = mp + e / mp;
        double v = 0.0;
        for (int s = lane; s < mp; s += 32) v = fma(__ldcg(&evec[i * ld + s]), gs(s, c), v);
#pragma unroll
        for (int o = 16; o >= 1; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (lane == 0) {
            A[i][c] = (float)v;
            A[c][i] = (float)v;
        }
    }
    __syncthreads();
    for (int sweep = 0; sweep < 10; sweep++) {
        bool some = false;                                // a sweep without rotations is not made
        for (int e = tid; e < mm * mm; e += nt) {
            const int p = e / mm, q = e - p * mm;
            const float apq = fabsf(A[p][q]);
            some = some || (p < q && apq > 1e-4f * fabsf(A[q][q] - A[p][p]) && apq > 1e-30f);
        }
        if (!__syncthreads_or(some)) break;               // uniform
        int xr = tid, yr = mm - 1 - tid;                  // the pairs and order of jacobi_solve
        for (int round = 0; round < mm - 1; round++) {
            if (tid < 32) {
                int active = 0;
                if (tid < half) {
                    int p = xr, q = yr;
                    if (p > q) { const int t = p; p = q; q = t; }
                    if (tid > 0 && ++xr == mm) xr = 1;
                    if (++yr == mm) yr = 1;
                    const float apq = A[p][q], diff = A[q][q] - A[p][p];
                    float c = 1.0f, s = 0.0f;
                    if (fabsf(apq) > 1e-4f * fabsf(diff)) {
                        active = fabsf(apq) > 1e-30f;
                        const float tau = diff / (2.0f * apq);
                        const float t = copysignf(1.0f, tau) / (fabsf(tau) + sqrtf(1.0f + tau * tau));
                        c = rsqrtf(1.0f + t * t);
                        s = t * c;
                    }
                    cs[tid] = c;
                    sn[tid] = s;
                    pp[tid] = (uint8_t)p;
                    qq[tid] = (uint8_t)q;
                }
                const unsigned mask = __ballot_sync(0xffffffffu, active);
                const int at = __popc(mask & ((1u << tid) - 1u));
                if (active) act[at] = (uint8_t)tid;
                if (tid < half) pos[tid] = (int8_t)(active ? at : -1);
                if (tid == 0) n_act[round & 1] = __popc(mask);
            }
            __syncthreads();
            const int na = n_act[round & 1];
            if (na == 0) continue;                        // uniform
            for (int e = tid; e < na * half; e += nt) {
                const int x = e / half, u = e - x * half, t = act[x], pu = pos[u];
                if (pu >= 0 && pu < x) continue;
                const int p = pp[t], q = qq[t], r = pp[u], v = qq[u];
                const float ct = cs[t], st = sn[t];
                const float cu = pu >= 0 ? cs[u] : 1.0f, su = pu >= 0 ? sn[u] : 0.0f;
                const float apr = A[p][r], apv = A[p][v], aqr = A[q][r], aqv = A[q][v];
                const float bpr = ct * apr - st * aqr, bpv = ct * apv - st * aqv;
                const float bqr = st * apr + ct * aqr, bqv = st * apv + ct * aqv;
                const float npr = cu * bpr - su * bpv, npv = su * bpr + cu * bpv;
                const float nqr = cu * bqr - su * bqv, nqv = su * bqr + cu * bqv;
                if (t == u) {
                    A[p][p] = npr;
                    A[q][q] = nqv;
                    A[p][q] = npv;
                    A[q][p] = npv;
                } else {
                    A[p][r] = npr;
                    A[p][v] = npv;
                    A[q][r] = nqr;
                    A[q][v] = nqv;
                    A[r][p] = npr;
                    A[v][p] = npv;
                    A[r][q] = nqr;
                    A[v][q] = nqv;
                }
            }
            for (int e = tid; e < mm * na; e += nt) {
                const int i = e / na, t = act[e - i * na], p = pp[t], q = qq[t];
                const float c = cs[t], s = sn[t], qp = Qf[i][p], qv = Qf[i][q];
                Qf[i][p] = c * qp - s * qv;
                Qf[i][q] = s * qp + c * qv;
            }
            __syncthreads();
        }
    }
    __syncthreads();
    // X = [evec 0; 0 1] Qf
    for (int e = tid; e < m * m; e += nt) {
        const int r = e / m, c = e % m;
        float v = 0.0f;
        if (r >= mp) {
            v = Qf[r][c];
        } else {
            for (int i = 0; i < mp; i++) v = fmaf((float)__ldcg(&evec[i * ld + r]), Qf[i][c], v);
        }
        A[r][c] = v;
    }
    __syncthreads();
}

// the sign of each new eigenvector is that of the column of X it is nearest to
__device__ __forceinline__ void apply_signs(int ld, int m, double *__restrict__ evec,
                                            const float (*X)[SHCI_MAX_SUB + 1]) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    __syncthreads();
    for (int l = warp; l < m; l += nw) {
        const float e0 = lane < m ? (float)__ldcg(&evec[l * ld + lane]) : 0.0f;
        const float e1 = lane + 32 < m ? (float)__ldcg(&evec[l * ld + lane + 32]) : 0.0f;
        float d0 = 0.0f, d1 = 0.0f;                       // against columns lane and lane + 32
        const int c0 = min(lane, m - 1), c1 = min(lane + 32, m - 1);
        for (int r = 0; r < m; r++) {
            const float e = __shfl_sync(0xffffffffu, r < 32 ? e0 : e1, r & 31);
            d0 = fmaf(e, X[r][c0], d0);
            d1 = fmaf(e, X[r][c1], d1);
        }
        float best = fabsf(d0) >= fabsf(d1) ? d0 : d1;
#pragma unroll
        for (int o = 16; o >= 1; o >>= 1) {
            const float y = __shfl_xor_sync(0xffffffffu, best, o);
            if (fabsf(y) > fabsf(best)) best = y;
        }
        if (best < 0.0f) {
            if (lane < m) evec[l * ld + lane] = -__ldcg(&evec[l * ld + lane]);
            if (lane + 32 < m) evec[l * ld + lane + 32] = -__ldcg(&evec[l * ld + lane + 32]);
        }
    }
    __syncthreads();
}

// Eigen-decomposition of the m x m matrix G whose leading m_prev x m_prev
// block's is in eval / evec (m_prev = 0: nothing is known): vector by vector
// when the block only grew, by Jacobi otherwise (the first solve after a
// restart).  SIGNS: with the signs of the Jacobi iteration (jsm: JACOBI_SMEM_SIGNS
// bytes); where an append is refused, that iteration from the old eigenvectors
// itself, which are kept until then when several vectors are appended (a first one
// refused leaves them as they were).  A batch returns energies only and does
// without.  Per Davidson step of a whole solve: 176 us with Jacobi alone and 88
// with this, 52 of it for the signs, for one root (up to 24 vectors), 1.2 ms and
// 0.30 for the slowest of eight batched systems of four roots (up to 48 vectors,
// no signs).
template <bool QSHARED, bool SIGNS>
__device__ __forceinline__ void subspace_eig(const double *G, int ld, int m, int m_prev, double *__restrict__ eval,
                                             double *__restrict__ evec, double *jsm, double *qg = nullptr) {
    const int old = m_prev > 0 && m_prev <= m ? m_prev : 0;
    int have = old;
    if (have == 0 || have == m) {
        jacobi_solve<QSHARED>(G, ld, m, have, eval, evec, jsm, qg);
        return;
    }
    typedef float (*Rows)[SHCI_MAX_SUB + 1];
    Rows X = reinterpret_cast<Rows>(jsm + SHCI_MAX_SUB * (SHCI_MAX_SUB + 1));     // behind append_eig's matrix
    const bool keep = SIGNS && m - old > 1;
    double *kept = jsm + 2 * SHCI_MAX_SUB * (SHCI_MAX_SUB + 1);       // behind jacobi_solve's two matrices
    if (keep) {
        for (int e = threadIdx.x; e < old * (old + 1); e += blockDim.x) {
            const int l = e / (old + 1), r = e - l * (old + 1);
            kept[e] = r < old ? __ldcg(&evec[l * ld + r]) : __ldcg(&eval[l]);
        }
    }
    if (SIGNS) jacobi_signs(G, ld, m, old, eval, evec, X, reinterpret_cast<Rows>(jsm));
    while (have < m && append_eig(G, ld, have, eval, evec, jsm)) have++;
    if (have == m) {
        if (SIGNS) apply_signs(ld, m, evec, X);
        return;
    }
    if (keep && have > old) {
        for (int e = threadIdx.x; e < old * (old + 1); e += blockDim.x) {
            const int l = e / (old + 1), r = e - l * (old + 1);
            if (r < old) evec[l * ld + r] = kept[e];
            else eval[l] = kept[e];
        }
        have = old;
        __syncthreads();
    }
    jacobi_solve<QSHARED>(G, ld, m, have, eval, evec, jsm, qg);
}

constexpr size_t JACOBI_SMEM_A = sizeof(double) * SHCI_MAX_SUB * (SHCI_MAX_SUB + 1);
constexpr size_t JACOBI_SMEM = 2 * JACOBI_SMEM_A;
constexpr size_t JACOBI_SMEM_SIGNS = JACOBI_SMEM + sizeof(double) * SHCI_MAX_SUB * (SHCI_MAX_SUB + 1);
constexpr int JACOBI_Q_DOUBLES = SHCI_MAX_SUB * (SHCI_MAX_SUB + 1);

}  // namespace shci
