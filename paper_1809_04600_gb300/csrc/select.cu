// Heat-bath selection of new determinants (Sec. II.A, Eq. 2): D_a outside V is
// selected when some D_i in V has |H_ai c_i| >= eps1.
//
// Double excitations are found the way the paper describes: for every pair
// of occupied orbitals, the magnitudes of the matrix elements of all double
// excitations from that pair depend only on the four orbitals, so they are
// computed once per set of integrals and stored sorted in decreasing order;
// a determinant walks the list of each of its occupied pairs and stops at
// the first element below eps1 / |c_i|.  Single excitations depend on the
// whole determinant and are evaluated exactly (Slater-Condon) for every
// occupied -> virtual move.  Candidates are written per determinant (count
// pass, scan, fill pass) as sort keys, sorted, made unique and removed when
// already in V.
#include <algorithm>
#include <cfloat>
#include <cmath>

#include "context.cuh"
#include "enumerate.cuh"

namespace shci {

constexpr int SEL_THREADS = 256;

// ---------------------------------------------------------------- sorted double-excitation lists

// Tuple t = ((p n + q) n + r) n + s.  List 0 (same spin): p < q, r < s,
// {r, s} disjoint from {p, q}, magnitude |(pr|qs) - (ps|qr)|.  List 1
// (opposite spin, p and r alpha, q and s beta): r != p, s != q, magnitude
// |(pr|qs)|.  Entries with magnitude 0 never meet eps1 > 0 and are dropped.
__device__ __forceinline__ bool hb_entry(const DevInts &I, int same, int64_t t, int &slot, int &r, int &s,
                                         double &v) {
    // v is signed: the element without the excitation's phase
    const int n = I.n;
    s = (int)(t % n);
    r = (int)((t / n) % n);
    const int q = (int)((t / ((int64_t)n * n)) % n);
    const int p = (int)(t / ((int64_t)n * n * n));
    slot = p * n + q;
    if (same) {
        if (!(p < q && r < s) || r == p || r == q || s == p || s == q) return false;
        v = eri_get(I, p, r, q, s) - eri_get(I, p, s, q, r);
    } else {
        if (r == p || s == q) return false;
        v = eri_get(I, p, r, q, s);
    }
    return fabs(v) > 0.0;
}

// key: slot in the high word, then the magnitude rounded toward zero to FP32
// with its bits inverted (ascending keys = decreasing magnitude); excluded
// tuples get the largest key and sort last
__global__ void k_hb_gen(const DevInts I, int same, int64_t total, uint64_t *__restrict__ keys,
                         uint32_t *__restrict__ vals, unsigned long long *__restrict__ cnt) {
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < total; t += (int64_t)gridDim.x * blockDim.x) {
        int slot, r, s;
        double v;
        vals[t] = (uint32_t)t;
        if (!hb_entry(I, same, t, slot, r, s, v)) {
            keys[t] = ~0ull;
            continue;
        }
        const uint32_t fb = __float_as_uint(__double2float_rz(fabs(v)));
        keys[t] = ((uint64_t)slot << 32) | (uint64_t)(~fb);
        atomicAdd(&cnt[slot], 1ull);
    }
}

__global__ void k_hb_final(const DevInts I, int same, int64_t n_valid, const uint32_t *__restrict__ vals,
                           uint32_t *__restrict__ rs, double *__restrict__ val, float *__restrict__ kf) {
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n_valid;
         e += (int64_t)gridDim.x * blockDim.x) {
        int slot, r, s;
        double v = 0.0;
        hb_entry(I, same, (int64_t)vals[e], slot, r, s, v);
        rs[e] = (uint32_t)r | ((uint32_t)s << 16);
        val[e] = v;
        kf[e] = __double2float_rz(fabs(v));
    }
}

static void build_hb_list(shci_ctx *c, int same, HBList &L) {
    cudaStream_t st = c->st;
    const int n = c->n_orb;
    const int64_t total = (int64_t)n * n * n * n;
    const DevInts I = dev_ints(c);
    DevBuf<uint64_t> keys;
    DevBuf<uint32_t> vals;
    DevBuf<unsigned long long> cnt;
    keys.alloc((size_t)total);
    vals.alloc((size_t)total);
    cnt.alloc((size_t)n * n + 1);
    CUDA_TRY(cudaMemsetAsync(cnt.p, 0, sizeof(unsigned long long) * (n * n + 1), st));
    const int blocks = (int)std::min<int64_t>(ceil_div(total, SEL_THREADS), (int64_t)c->n_sm * 16);
    k_hb_gen<<<blocks, SEL_THREADS, 0, st>>>(I, same, total, keys.p, vals.p, cnt.p);
    KERNEL_CHECK();
    g_kernel_launches += 1;
    radix_sort<1>(keys.p, vals.p, total, c->sw, st);
    L.off.alloc((size_t)n * n + 1);
    DevBuf<int64_t> tmp;
    tmp.alloc((size_t)scan_tmp_len(n * n + 1));
    exclusive_scan<int64_t>(reinterpret_cast<const int64_t *>(cnt.p), L.off.p, (int64_t)n * n, tmp.p, st);
    int64_t n_valid = 0;
    CUDA_TRY(cudaMemcpyAsync(&n_valid, L.off.p + (int64_t)n * n, sizeof(int64_t), cudaMemcpyDeviceToHost, st));
    CUDA_TRY(cudaStreamSynchronize(st));
    L.rs.alloc((size_t)std::max<int64_t>(n_valid, 1));
    L.val.alloc((size_t)std::max<int64_t>(n_valid, 1));
    L.kf.alloc((size_t)std::max<int64_t>(n_valid, 1));
    if (n_valid > 0) {
        k_hb_final<<<(int)std::min<int64_t>(ceil_div(n_valid, SEL_THREADS), (int64_t)c->n_sm * 16), SEL_THREADS, 0,
                     st>>>(I, same, n_valid, vals.p, L.rs.p, L.val.p, L.kf.p);
        KERNEL_CHECK();
        g_kernel_launches += 1;
    }
    L.entries = n_valid;
    CUDA_TRY(cudaStreamSynchronize(st));
}

// ---------------------------------------------------------------- sort keys

// The key a determinant is sorted by: both strings in one word when 2 n_orb <=
// 64 (KW = 1: the alpha string in the low n_orb bits), else the 2W words
// themselves (alpha first, word 0 least significant).  Both order by (beta,
// alpha).  One word instead of two takes a third off the bytes that every pass
// of the sort moves (12 instead of 20 per element with its index).
template <int KW>
struct Key {
    uint64_t w[KW];
    __device__ __forceinline__ bool operator==(const Key &o) const {
        bool eq = true;
#pragma unroll
        for (int k = 0; k < KW; k++) eq &= w[k] == o.w[k];
        return eq;
    }
};

template <int W, int KW>
__device__ __forceinline__ Key<KW> make_key(const Str<W> &a, const Str<W> &b, int n_orb) {
    Key<KW> k;
    if constexpr (KW == 1) {
        k.w[0] = a.w[0] | (b.w[0] << n_orb);
    } else {
#pragma unroll
        for (int x = 0; x < W; x++) {
            k.w[x] = a.w[x];
            k.w[W + x] = b.w[x];
        }
    }
    return k;
}

template <int W, int KW>
__device__ __forceinline__ void split_key(const Key<KW> &k, int n_orb, Str<W> &a, Str<W> &b) {
    if constexpr (KW == 1) {
        a.w[0] = k.w[0] & ((1ull << n_orb) - 1);         // n_orb <= 32 here
        b.w[0] = k.w[0] >> n_orb;
    } else {
#pragma unroll
        for (int x = 0; x < W; x++) {
            a.w[x] = k.w[x];
            b.w[x] = k.w[W + x];
        }
    }
}

template <int KW>
__device__ __forceinline__ Key<KW> load_key(const uint64_t *p, int64_t i) {
    Key<KW> k;
    if constexpr (KW == 1) {
        k.w[0] = p[i];
    } else {                                             // buffers of whole keys from cudaMalloc: 16-byte aligned
#pragma unroll
        for (int x = 0; x < KW; x += 2) {
            const ulonglong2 v = *reinterpret_cast<const ulonglong2 *>(p + i * KW + x);
            k.w[x] = v.x;
            k.w[x + 1] = v.y;
        }
    }
    return k;
}

template <int KW>
__device__ __forceinline__ void store_key(uint64_t *p, int64_t i, const Key<KW> &k) {
#pragma unroll
    for (int x = 0; x < KW; x++) p[i * KW + x] = k.w[x];
}

template <int KW>
__device__ __forceinline__ Key<KW> shfl_key(const Key<KW> &k, int lane) {
    Key<KW> o;
#pragma unroll
    for (int x = 0; x < KW; x++) o.w[x] = __shfl_sync(0xffffffffu, k.w[x], lane);
    return o;
}

// is the key in the sorted list vs[nv]?
template <int KW>
__device__ __forceinline__ bool in_sorted(const uint64_t *__restrict__ vs, int64_t nv, const Key<KW> &x) {
    int64_t lo = 0, hi = nv;
    while (lo < hi) {
        const int64_t mid = (lo + hi) >> 1;
        bool less = false;
#pragma unroll
        for (int w = 0; w < KW; w++) {                   // the last word that differs decides
            const uint64_t v = __ldg(&vs[mid * KW + w]);
            if (v != x.w[w]) less = v < x.w[w];
        }
        if (less) lo = mid + 1;
        else hi = mid;
    }
    if (lo >= nv) return false;
    bool eq = true;
#pragma unroll
    for (int w = 0; w < KW; w++) eq &= __ldg(&vs[lo * KW + w]) == x.w[w];
    return eq;
}

template <int W, int KW>
__global__ void k_det_keys(const uint64_t *__restrict__ dets, int64_t n, int n_orb, uint64_t *__restrict__ keys) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        store_key<KW>(keys, i, make_key<W, KW>(load_str<W>(dets, 2 * i), load_str<W>(dets, 2 * i + 1), n_orb));
}

// the key bits that n_orb orbitals can set
template <int W, int KW>
struct KeyMask {
    uint64_t w[KW];
    explicit KeyMask(int n_orb) {
        auto low = [](int bits) { return bits >= 64 ? ~0ull : (bits <= 0 ? 0ull : (1ull << bits) - 1); };
        for (int k = 0; k < KW; k++) w[k] = KW == 1 ? low(2 * n_orb) : low(n_orb - 64 * (k % W));
    }
};

// V's determinants as sorted keys
template <int W, int KW>
static void sorted_space(shci_ctx *c, DevBuf<uint64_t> &vs) {
    const int64_t n = c->n_det;
    vs.alloc((size_t)n * KW);
    const int blocks = (int)std::min<int64_t>(ceil_div(n, SEL_THREADS), (int64_t)c->n_sm * 16);
    k_det_keys<W, KW><<<blocks, SEL_THREADS, 0, c->st>>>(c->dets.p, n, c->n_orb, vs.p);
    KERNEL_CHECK();
    g_kernel_launches += 1;
    radix_sort<KW>(vs.p, nullptr, n, c->sw, c->st, KeyMask<W, KW>(c->n_orb).w, RS_KEYS);
}

// ---------------------------------------------------------------- selection kernels

struct SelArgs {
    int64_t n_det;
    const uint64_t *dets;                   // [n][2W]
    int k;
    const double *c;                        // [k][n]
    double eps1;
    int n, na, nb;
    const int64_t *ss_off, *os_off;
    const uint32_t *ss_rs, *os_rs;
    const double *ss_v, *os_v;
    const float *ss_kf, *os_kf;
    unsigned long long *cnt;                // count pass: candidates per determinant
    const int64_t *off;                     // fill pass: first slot of each determinant
    uint64_t *out;                          // fill pass: [total] sort keys
    // second-order energy: the terms H_ai c_i of determinants a in hash batch `batch` of `nbatch`
    int nbatch, batch;
    double *terms;                          // fill pass: [total]
    // stochastic estimator (Eq. 9): per sampled determinant w/p and
    // w (n_d - 1) / p - w^2 / p^2; second term and |H_ai c_i| per candidate
    const double *f1, *f2;
    double *terms2, *mags;
};

static SelArgs sel_args(const shci_ctx *c, double eps) {
    SelArgs S{};
    S.n_det = c->n_det;
    S.dets = c->dets.p;
    S.k = 1;
    S.eps1 = eps;
    S.n = c->n_orb;
    S.na = c->n_alpha;
    S.nb = c->n_beta;
    S.ss_off = c->hb_same.off.p;
    S.ss_rs = c->hb_same.rs.p;
    S.ss_v = c->hb_same.val.p;
    S.ss_kf = c->hb_same.kf.p;
    S.os_off = c->hb_opp.off.p;
    S.os_rs = c->hb_opp.rs.p;
    S.os_v = c->hb_opp.val.p;
    S.os_kf = c->hb_opp.kf.p;
    S.nbatch = 1;
    return S;
}

// batch of a determinant (a SplitMix64-style mix of its words)
template <int W>
__device__ __forceinline__ int det_batch(const Str<W> &a, const Str<W> &b, int nbatch) {
    uint64_t z = 0x9E3779B97F4A7C15ull;
#pragma unroll
    for (int k = 0; k < 2 * W; k++) {
        z ^= k < W ? a.w[k] : b.w[k - W];
        z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
        z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
        z ^= z >> 31;
    }
    return (int)(z % (uint64_t)nbatch);
}

template <int W>
__device__ __forceinline__ bool has_bit(const Str<W> &s, int b) {
    return (s.w[b >> 6] >> (b & 63)) & 1ull;
}

// Above this bound no later entry of a list can meet the threshold: a key is
// the magnitude rounded toward zero to FP32, so the magnitude is below
// key (1 + 2^-23) for normal keys and below FLT_MIN otherwise.
__device__ __forceinline__ double key_bound(float kf) {
    return kf < FLT_MIN ? (double)FLT_MIN : (double)kf * (1.0 + 0x1p-22);
}

// Occupied and empty orbitals of both strings, ascending, listed by a warp.
struct OrbLists {
    uint8_t occ[2][SHCI_MAX_ORB], vir[2][SHCI_MAX_ORB];
};

template <int W>
__device__ __forceinline__ void list_orbitals(OrbLists &L, int spin, const Str<W> &s, int n) {
    const int lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u;
    int no = 0, nv = 0;
    for (int o0 = 0; o0 < n; o0 += 32) {
        const int o = o0 + lane;
        const bool in = o < n, set = in && has_bit(s, o);
        const unsigned mo = __ballot_sync(0xffffffffu, set), mv = __ballot_sync(0xffffffffu, in && !set);
        if (set) L.occ[spin][no + __popc(mo & lt)] = (uint8_t)o;
        else if (in) L.vir[spin][nv + __popc(mv & lt)] = (uint8_t)o;
        no += __popc(mo);
        nv += __popc(mv);
    }
}

// One warp per determinant.  First every single move (alpha then beta), a lane
// per move.  Then the double excitations: for 32 occupied pairs at a time a
// lane finds by bisection how many leading entries of its pair's sorted list
// can meet the threshold, and the warp takes those entries of all 32 lists as
// one sequence, 32 at a time (a lane finds its list in the prefix sums), so
// that no lane waits for another's longer list and candidates leave as one
// contiguous, ordered run.  Walking one list per lane and reserving slots one
// by one took 17.7 ms (count) and 24.2 ms (fill) for the 1.8e8 terms of 200,003
// determinants of 24 orbitals (eps 1e-5); this form 5.5 and 7.8.
template <int W, int KW, bool FILL, bool PT>
__global__ void __launch_bounds__(SEL_THREADS) k_select(SelArgs S, DevInts I) {
    __shared__ OrbLists lists[SEL_THREADS / 32];
    const int lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u;
    OrbLists &L = lists[threadIdx.x >> 5];
    const int n = S.n, na = S.na, nb = S.nb;
    const int u_sa = na * (n - na), u_sb = nb * (n - nb);
    const int u_paa = na * (na - 1) / 2, u_pbb = nb * (nb - 1) / 2, u_pab = na * nb;
    const int pairs = u_paa + u_pbb + u_pab;
    const int64_t warps = (int64_t)gridDim.x * (SEL_THREADS / 32);
    for (int64_t i = ((int64_t)blockIdx.x * SEL_THREADS + threadIdx.x) >> 5; i < S.n_det; i += warps) {
        double cmax = 0.0, ci = 0.0, f1 = 0.0, f2 = 0.0;
        if (PT) {
            ci = __ldg(&S.c[i]);
            cmax = fabs(ci);
            if (FILL && S.f1) {
                f1 = __ldg(&S.f1[i]);
                f2 = __ldg(&S.f2[i]);
            }
        } else {
            for (int l = 0; l < S.k; l++) cmax = fmax(cmax, fabs(__ldg(&S.c[(int64_t)l * S.n_det + i])));
        }
        int64_t pos = FILL ? __ldg(&S.off[i]) : 0;        // next slot, or candidates so far
        if (cmax > 0.0) {
            const Str<W> A = load_str<W>(S.dets, 2 * i), B = load_str<W>(S.dets, 2 * i + 1);
            // Record this round's candidates (a, b) with the elements hv.  Second-order
            // mode (PT): only determinants of the current hash batch, with their terms.
            auto emit = [&](bool keep, const Str<W> &a, const Str<W> &b, double hv) {
                if (PT && S.nbatch > 1) keep = keep && det_batch<W>(a, b, S.nbatch) == S.batch;
                const unsigned mask = __ballot_sync(0xffffffffu, keep);
                if (FILL && keep) {
                    const int64_t slot = pos + __popc(mask & lt);
                    store_key<KW>(S.out, slot, make_key<W, KW>(a, b, n));
                    if (PT) {
                        if (S.f1) {
                            S.terms[slot] = f1 * ci * hv;
                            S.terms2[slot] = f2 * ci * ci * hv * hv;
                            S.mags[slot] = fabs(hv) * cmax;
                        } else {
                            S.terms[slot] = hv * ci;
                            if (S.mags) S.mags[slot] = fabs(hv) * cmax;
                        }
                    }
                }
                pos += __popc(mask);
            };
            __syncwarp();
            list_orbitals(L, 0, A, n);
            list_orbitals(L, 1, B, n);
            __syncwarp();
            for (int spin = 0; spin < 2; spin++) {
                const int units = spin ? u_sb : u_sa, nv = n - (spin ? nb : na);
                const Str<W> &si = spin ? B : A;
                for (int u0 = 0; u0 < units; u0 += 32) {
                    const int u = u0 + lane;
                    bool keep = false;
                    Str<W> sj = si;
                    double hv = 0.0;
                    if (u < units) {
                        flip_bit(sj, L.occ[spin][u / nv]);
                        flip_bit(sj, L.vir[spin][u % nv]);
                        hv = single_exc<W>(I, si, sj, spin ? A : B);
                        keep = fabs(hv) * cmax >= S.eps1;
                    }
                    if (spin) emit(keep, A, sj, hv);
                    else emit(keep, sj, B, hv);
                }
            }
            for (int u0 = 0; u0 < pairs; u0 += 32) {
                int v = u0 + lane;
                int64_t e0 = 0;
                int len = 0, spin = 2, p = 0, q = 0;      // spin 0: alpha pair, 1: beta pair, 2: alpha and beta
                if (v < pairs) {
                    if (v < u_paa + u_pbb) {
                        spin = v < u_paa ? 0 : 1;
                        if (spin) v -= u_paa;
                        // pair rank v -> (x < y): y is the largest with y (y - 1) / 2 <= v
                        int y = (int)((1.0f + sqrtf(1.0f + 8.0f * (float)v)) * 0.5f);
                        while (y * (y - 1) / 2 > v) y--;
                        while ((y + 1) * y / 2 <= v) y++;
                        p = L.occ[spin][v - y * (y - 1) / 2];
                        q = L.occ[spin][y];
                    } else {
                        v -= u_paa + u_pbb;
                        p = L.occ[0][v / nb];
                        q = L.occ[1][v % nb];
                    }
                    const int64_t *off = spin == 2 ? S.os_off : S.ss_off;
                    const float *kf = spin == 2 ? S.os_kf : S.ss_kf;
                    e0 = __ldg(&off[p * n + q]);
                    int lo = 0, hi = (int)(__ldg(&off[p * n + q + 1]) - e0);
                    while (lo < hi) {                     // keys descend: first entry out of reach
                        const int mid = (lo + hi) >> 1;
                        if (key_bound(__ldg(&kf[e0 + mid])) * cmax < S.eps1) hi = mid;
                        else lo = mid + 1;
                    }
                    len = lo;
                }
                int incl = len;                           // inclusive prefix over the lanes
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int y = __shfl_up_sync(0xffffffffu, incl, o);
                    if (lane >= o) incl += y;
                }
                const int total = __shfl_sync(0xffffffffu, incl, 31);
                const int pq = p | (q << 8) | (spin << 16);
                for (int t0 = 0; t0 < total; t0 += 32) {
                    const int t = t0 + lane;
                    int src = 0;                          // the first lane with incl > t
#pragma unroll
                    for (int step = 16; step >= 1; step >>= 1) {
                        const int y = __shfl_sync(0xffffffffu, incl, src + step - 1);
                        if (y <= t) src += step;
                    }
                    src = min(src, 31);
                    const int64_t first = __shfl_sync(0xffffffffu, e0, src);
                    const int before = __shfl_sync(0xffffffffu, incl - len, src);
                    const int x = __shfl_sync(0xffffffffu, pq, src);
                    bool keep = false;
                    Str<W> a = A, b = B;
                    double hv = 0.0;
                    if (t < total) {
                        const int p1 = x & 255, q1 = (x >> 8) & 255, sp = x >> 16;
                        const int64_t e = first + (t - before);
                        const uint32_t rs = __ldg(sp == 2 ? &S.os_rs[e] : &S.ss_rs[e]);
                        hv = __ldg(sp == 2 ? &S.os_v[e] : &S.ss_v[e]);
                        const int r = (int)(rs & 0xFFFFu), s = (int)(rs >> 16);
                        // the strings the two holes p1, q1 and particles r, s belong to
                        const Str<W> &sa = sp == 1 ? B : A;
                        const Str<W> &sb = sp == 0 ? A : B;
                        keep = !has_bit(sa, r) && !has_bit(sb, s) && fabs(hv) * cmax >= S.eps1;
                        if (keep) {
                            int neg = 0;
                            if (sp == 2) {
                                flip_bit(a, p1);
                                flip_bit(b, q1);
                                if (FILL && PT)
                                    neg = bits_between<W>(a, min(p1, r), max(p1, r)) + bits_between<W>(b, min(q1, s), max(q1, s));
                                flip_bit(a, r);
                                flip_bit(b, s);
                            } else {
                                // p1 -> r, then q1 -> s on the intermediate string
                                Str<W> y = sa;
                                if (FILL && PT) neg = bits_between<W>(y, min(p1, r), max(p1, r));
                                flip_bit(y, p1);
                                flip_bit(y, r);
                                if (FILL && PT) neg += bits_between<W>(y, min(q1, s), max(q1, s));
                                flip_bit(y, q1);
                                flip_bit(y, s);
                                if (sp) b = y;
                                else a = y;
                            }
                            hv = flip_sign(hv, neg);
                        }
                    }
                    emit(keep, a, b, hv);
                }
            }
        }
        if (!FILL && lane == 0) S.cnt[i] = (unsigned long long)pos;
    }
}

// count pass over S's determinants and the offsets of their candidates; returns the total
template <int W, int KW, bool PT>
static int64_t count_candidates(shci_ctx *c, SelArgs &S, const DevInts &I, DevBuf<unsigned long long> &cnt,
                                DevBuf<int64_t> &off, DevBuf<int64_t> &tmp) {
    cudaStream_t st = c->st;
    const int64_t n = S.n_det;
    cnt.alloc((size_t)n + 1);
    off.alloc((size_t)n + 1);
    tmp.alloc((size_t)scan_tmp_len(n + 1));
    S.cnt = cnt.p;
    S.off = off.p;
    const int blocks = (int)std::min<int64_t>(ceil_div(n, SEL_THREADS / 32), (int64_t)c->n_sm * (2048 / SEL_THREADS));
    k_select<W, KW, false, PT><<<blocks, SEL_THREADS, 0, st>>>(S, I);
    KERNEL_CHECK();
    g_kernel_launches += 1;
    exclusive_scan<int64_t>(reinterpret_cast<const int64_t *>(cnt.p), off.p, n, tmp.p, st);
    int64_t total = 0;
    CUDA_TRY(cudaMemcpyAsync(&total, off.p + n, sizeof(int64_t), cudaMemcpyDeviceToHost, st));
    CUDA_TRY(cudaStreamSynchronize(st));
    return total;
}

template <int W, int KW, bool PT>
static void fill_candidates(shci_ctx *c, const SelArgs &S, const DevInts &I) {
    const int blocks = (int)std::min<int64_t>(ceil_div(S.n_det, SEL_THREADS / 32),
                                              (int64_t)c->n_sm * (2048 / SEL_THREADS));
    k_select<W, KW, true, PT><<<blocks, SEL_THREADS, 0, c->st>>>(S, I);
    KERNEL_CHECK();
    g_kernel_launches += 1;
}

// ---------------------------------------------------------------- unique, minus V

// Sorted candidates, 32 to a warp: masks[w] has a bit for each that is the
// first of its run and not in the sorted V; cnt[w] counts them.
template <int KW>
__global__ void __launch_bounds__(SEL_THREADS) k_sel_mark(const uint64_t *__restrict__ cand, int64_t total,
                                                         const uint64_t *__restrict__ vs, int64_t nv,
                                                         uint32_t *__restrict__ masks, int64_t *__restrict__ cnt) {
    const int lane = threadIdx.x & 31;
    const int64_t windows = (total + 31) >> 5, warps = (int64_t)gridDim.x * (SEL_THREADS / 32);
    for (int64_t w = ((int64_t)blockIdx.x * SEL_THREADS + threadIdx.x) >> 5; w < windows; w += warps) {
        const int64_t e = w * 32 + lane;
        bool keep = false;
        if (e < total) {
            const Key<KW> x = load_key<KW>(cand, e);
            keep = e == 0 || !(load_key<KW>(cand, e - 1) == x);
            keep = keep && !in_sorted<KW>(vs, nv, x);
        }
        const unsigned m = __ballot_sync(0xffffffffu, keep);
        if (lane == 0) {
            masks[w] = m;
            cnt[w] = __popc(m);
        }
    }
}

template <int W, int KW>
__global__ void __launch_bounds__(SEL_THREADS) k_sel_compact(const uint64_t *__restrict__ cand, int64_t total,
                                                            const uint32_t *__restrict__ masks,
                                                            const int64_t *__restrict__ pos, int n_orb,
                                                            uint64_t *__restrict__ out) {
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
        const int64_t w = e >> 5;
        const unsigned m = __ldg(&masks[w]), bit = 1u << (e & 31);
        if (!(m & bit)) continue;
        const int64_t o = __ldg(&pos[w]) + __popc(m & (bit - 1u));
        Str<W> a, b;
        split_key<W, KW>(load_key<KW>(cand, e), n_orb, a, b);
#pragma unroll
        for (int k = 0; k < W; k++) {
            out[o * 2 * W + k] = a.w[k];
            out[o * 2 * W + W + k] = b.w[k];
        }
    }
}

template <int W, int KW>
static void select_w(shci_ctx *c, int k, const double *cd, double eps1, DevBuf<uint64_t> &result, int64_t &n_new) {
    cudaStream_t st = c->st;
    const int64_t n = c->n_det;
    SelArgs S = sel_args(c, eps1);
    S.k = k;
    S.c = cd;
    const DevInts I = dev_ints(c);
    DevBuf<unsigned long long> cnt;
    DevBuf<int64_t> off, tmp;
    const int64_t total = count_candidates<W, KW, false>(c, S, I, cnt, off, tmp);
    c->stats.select_candidates = total;
    n_new = 0;
    if (total == 0) return;
    if (total > 0xFFFFFFFFll) throw ShciError{SHCI_ERR_INVALID, "too many candidates: raise eps1"};
    DevBuf<uint64_t> cand;
    cand.alloc((size_t)total * KW);
    S.out = cand.p;
    fill_candidates<W, KW, false>(c, S, I);
    radix_sort<KW>(cand.p, nullptr, total, c->sw, st, KeyMask<W, KW>(c->n_orb).w, RS_KEYS);
    DevBuf<uint64_t> vs;
    sorted_space<W, KW>(c, vs);
    const int64_t windows = ceil_div(total, 32);
    DevBuf<uint32_t> masks;
    DevBuf<int64_t> wcnt, pos, tmp2;
    masks.alloc((size_t)windows);
    wcnt.alloc((size_t)windows + 1);
    pos.alloc((size_t)windows + 1);
    tmp2.alloc((size_t)scan_tmp_len(windows + 1));
    const int gb = (int)std::min<int64_t>(ceil_div(total, SEL_THREADS), (int64_t)c->n_sm * 16);
    k_sel_mark<KW><<<gb, SEL_THREADS, 0, st>>>(cand.p, total, vs.p, n, masks.p, wcnt.p);
    KERNEL_CHECK();
    exclusive_scan<int64_t>(wcnt.p, pos.p, windows, tmp2.p, st);
    CUDA_TRY(cudaMemcpyAsync(&n_new, pos.p + windows, sizeof(int64_t), cudaMemcpyDeviceToHost, st));
    CUDA_TRY(cudaStreamSynchronize(st));
    result.alloc((size_t)std::max<int64_t>(n_new, 1) * 2 * W);
    k_sel_compact<W, KW><<<gb, SEL_THREADS, 0, st>>>(cand.p, total, masks.p, pos.p, c->n_orb, result.p);
    KERNEL_CHECK();
    g_kernel_launches += 2;
    CUDA_TRY(cudaStreamSynchronize(st));
}

// Runs F<W, KW>() for the context's strings: one sort word when both strings fit it.
#define DISPATCH_KEYS(c, CALL)                                  \
    do {                                                        \
        if ((c)->W == 1 && 2 * (c)->n_orb <= 64) { CALL(1, 1); } \
        else if ((c)->W == 1) { CALL(1, 2); }                   \
        else { CALL(2, 4); }                                    \
    } while (0)

// ---------------------------------------------------------------- second-order energy

// The sums a run of equal sorted determinants a is reduced to, and what they
// add to the result:
//   RUN_PT      num = sum of the terms: num^2 / (E_V - H_aa)
//   RUN_SAMPLE  S1, S2 over all terms and over those with magnitude >= eps:
//               (S1^2 + S2) / (E_V - H_aa) of each pair
//   RUN_PSTO    num over all terms and num_d over those with magnitude >= eps:
//               the correction (num^2 - num_d^2) / (E_V - H_aa), and its square
enum { RUN_PT = 0, RUN_SAMPLE = 1, RUN_PSTO = 2 };
template <int MODE>
struct RunSums {
    static constexpr int N = MODE == RUN_PT ? 1 : (MODE == RUN_SAMPLE ? 4 : 2);
};

struct RunArgs {
    const uint64_t *cand;                   // sorted keys of the terms' determinants
    const uint32_t *idx;                    // each one's term
    const double *t1, *t2, *mag;
    int64_t total;
    const uint64_t *vs;                     // V's sorted keys
    int64_t nv;
    double e_var, eps;
    double *part;                           // [blocks][2]
    unsigned long long *npart;              // [blocks]: determinants
};

template <int MODE>
__device__ __forceinline__ void run_terms(const RunArgs &A, int64_t e, double *v) {
    const uint32_t j = __ldg(&A.idx[e]);
    v[0] = __ldg(&A.t1[j]);
    if constexpr (MODE == RUN_SAMPLE) {
        v[1] = __ldg(&A.t2[j]);
        const bool big = __ldg(&A.mag[j]) >= A.eps;
        v[2] = big ? v[0] : 0.0;
        v[3] = big ? v[1] : 0.0;
    } else if constexpr (MODE == RUN_PSTO) {
        v[1] = __ldg(&A.mag[j]) >= A.eps ? v[0] : 0.0;
    }
}

// A warp takes 32 consecutive sorted elements: the runs that begin among them
// are summed by a segmented tree of shuffles, the last one's continuation by
// the whole warp, 128 elements at a time; the runs' keys and sums are queued
// and finished 32 at a time (is a in V, H_aa, the contribution).  A thread per
// run, adding up its terms one by one, took 27 ms for 1.8e8 terms and 18
// ms for a sample of 4e7, nearly all of it the longest runs' chains of
// dependent loads; this form 4.9 and 6.3.  The order of every
// sum is fixed.
template <int W, int KW, int MODE>
__global__ void __launch_bounds__(SEL_THREADS) k_run_reduce(RunArgs A, DevInts I) {
    constexpr int NS = RunSums<MODE>::N;
    constexpr int NW = SEL_THREADS / 32;
    __shared__ __align__(16) uint64_t qkey[NW][64 * KW];
    __shared__ double qsum[NW][64 * NS];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const unsigned lt = (1u << lane) - 1u;
    uint64_t *qk = qkey[wib];
    double *qs = qsum[wib];
    double acc0 = 0.0, acc1 = 0.0;
    unsigned long long cnt = 0;
    int qn = 0;
    auto finish = [&](int m) {                            // the first m (<= 32) queued runs
        if (lane < m) {
            const Key<KW> x = load_key<KW>(qk, lane);
            if (!in_sorted<KW>(A.vs, A.nv, x)) {
                Str<W> a, b;
                split_key<W, KW>(x, I.n, a, b);
                const double den = A.e_var - hii<W>(I, a, b);
                const double *v = qs + lane * NS;
                if constexpr (MODE == RUN_PT) {
                    acc0 += v[0] * v[0] / den;
                } else if constexpr (MODE == RUN_SAMPLE) {
                    acc0 += (v[0] * v[0] + v[1]) / den;
                    acc1 += (v[2] * v[2] + v[3]) / den;
                } else {
                    const double corr = (v[0] * v[0] - v[1] * v[1]) / den;
                    acc0 += corr;
                    acc1 += corr * corr;
                }
                cnt++;
            }
        }
    };
    const int64_t windows = (A.total + 31) >> 5, warps = (int64_t)gridDim.x * NW;
    for (int64_t w = ((int64_t)blockIdx.x * SEL_THREADS + threadIdx.x) >> 5; w < windows; w += warps) {
        const int64_t e = w * 32 + lane;
        const bool in = e < A.total;
        Key<KW> x{}, before{};
        if (in) x = load_key<KW>(A.cand, e);
        if (in && e > 0) before = load_key<KW>(A.cand, e - 1);
        const bool head = in && (e == 0 || !(x == before));
        const unsigned heads = __ballot_sync(0xffffffffu, head);
        if (heads == 0) continue;                         // inside a run that began earlier
        double v[NS];
#pragma unroll
        for (int s = 0; s < NS; s++) v[s] = 0.0;
        if (in && (heads & (lt | (1u << lane)))) run_terms<MODE>(A, e, v);
        const unsigned above = heads & ~(lt | (1u << lane));
        const int end = above ? __ffs(above) - 1 : 32;    // one past this lane's run within the window
        const int longest = __reduce_max_sync(0xffffffffu, head ? end - lane : 0);
        for (int d = 1; d < longest; d <<= 1) {
#pragma unroll
            for (int s = 0; s < NS; s++) {
                const double o = __shfl_down_sync(0xffffffffu, v[s], d);
                if (lane + d < end) v[s] += o;
            }
        }
        // the last run's elements beyond the window
        const int last = 31 - __clz(heads);
        const Key<KW> kx = shfl_key<KW>(x, last);
        int64_t f = w * 32 + 32;
        if (f < A.total && load_key<KW>(A.cand, f) == kx) {
            constexpr int U = 4;
            double tail[NS];
#pragma unroll
            for (int s = 0; s < NS; s++) tail[s] = 0.0;
            for (;; f += 32 * U) {
                bool same[U];
                double t[U][NS];
#pragma unroll
                for (int u = 0; u < U; u++) {
                    const int64_t ee = f + 32 * u + lane;
                    same[u] = ee < A.total && load_key<KW>(A.cand, ee) == kx;
                }
#pragma unroll
                for (int u = 0; u < U; u++) {
#pragma unroll
                    for (int s = 0; s < NS; s++) t[u][s] = 0.0;
                    if (same[u]) run_terms<MODE>(A, f + 32 * u + lane, t[u]);
                }
#pragma unroll
                for (int u = 0; u < U; u++)
#pragma unroll
                    for (int s = 0; s < NS; s++) tail[s] += t[u][s];
                if (!__all_sync(0xffffffffu, same[U - 1])) break;      // the run has ended
            }
#pragma unroll
            for (int s = 0; s < NS; s++) {
#pragma unroll
                for (int o = 16; o >= 1; o >>= 1) tail[s] += __shfl_xor_sync(0xffffffffu, tail[s], o);
                if (lane == last) v[s] += tail[s];
            }
        }
        if (head) {
            const int slot = qn + __popc(heads & lt);
            store_key<KW>(qk, slot, x);
#pragma unroll
            for (int s = 0; s < NS; s++) qs[slot * NS + s] = v[s];
        }
        qn += __popc(heads);
        __syncwarp();
        if (qn >= 32) {
            finish(32);
            __syncwarp();
            const int rest = qn - 32;
            if (lane < rest) {
                store_key<KW>(qk, lane, load_key<KW>(qk, 32 + lane));
#pragma unroll
                for (int s = 0; s < NS; s++) qs[lane * NS + s] = qs[(32 + lane) * NS + s];
            }
            qn = rest;
            __syncwarp();
        }
    }
    finish(qn);
    __shared__ double red[2][NW];
    __shared__ unsigned long long redc[NW];
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) {
        acc0 += __shfl_xor_sync(0xffffffffu, acc0, o);
        acc1 += __shfl_xor_sync(0xffffffffu, acc1, o);
        cnt += __shfl_xor_sync(0xffffffffu, cnt, o);
    }
    if (lane == 0) {
        red[0][wib] = acc0;
        red[1][wib] = acc1;
        redc[wib] = cnt;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double s0 = 0.0, s1 = 0.0;
        unsigned long long sc = 0;
        for (int y = 0; y < NW; y++) {
            s0 += red[0][y];
            s1 += red[1][y];
            sc += redc[y];
        }
        A.part[2 * blockIdx.x] = s0;
        A.part[2 * blockIdx.x + 1] = s1;
        A.npart[blockIdx.x] = sc;
    }
}

// The buffers of one batch (sample) of terms, kept from one to the next, and
// the result of its reduction.
struct TermWork {
    DevBuf<uint64_t> cand, vs;
    DevBuf<uint32_t> idx;
    DevBuf<double> t1, t2, mag, part;
    DevBuf<unsigned long long> npart, cnt;
    DevBuf<int64_t> off, tmp;
    std::vector<double> hp;
    std::vector<unsigned long long> hn;
    double sum0 = 0.0, sum1 = 0.0;
    int64_t dets = 0;
};

// Fill S's counted candidates (total > 0 of them), sort them by determinant
// and reduce their runs.
template <int W, int KW, int MODE>
static void reduce_terms(shci_ctx *c, SelArgs &S, const DevInts &I, int64_t total, double e_var, double eps,
                         TermWork &T) {
    cudaStream_t st = c->st;
    T.cand.alloc((size_t)total * KW);
    T.t1.alloc((size_t)total);
    T.idx.alloc((size_t)total);
    if (MODE != RUN_PT) T.mag.alloc((size_t)total);
    if (MODE == RUN_SAMPLE) T.t2.alloc((size_t)total);
    S.out = T.cand.p;
    S.terms = T.t1.p;
    S.terms2 = T.t2.p;
    S.mags = T.mag.p;
    fill_candidates<W, KW, true>(c, S, I);
    radix_sort<KW>(T.cand.p, T.idx.p, total, c->sw, st, KeyMask<W, KW>(c->n_orb).w, RS_POSITION);
    const int blocks = c->n_sm * 8;
    T.part.alloc((size_t)2 * blocks);
    T.npart.alloc((size_t)blocks);
    T.hp.resize(2 * blocks);
    T.hn.resize(blocks);
    RunArgs A{};
    A.cand = T.cand.p;
    A.idx = T.idx.p;
    A.t1 = T.t1.p;
    A.t2 = T.t2.p;
    A.mag = T.mag.p;
    A.total = total;
    A.vs = T.vs.p;
    A.nv = c->n_det;
    A.e_var = e_var;
    A.eps = eps;
    A.part = T.part.p;
    A.npart = T.npart.p;
    k_run_reduce<W, KW, MODE><<<blocks, SEL_THREADS, 0, st>>>(A, I);
    KERNEL_CHECK();
    g_kernel_launches += 1;
    CUDA_TRY(cudaMemcpyAsync(T.hp.data(), T.part.p, sizeof(double) * 2 * blocks, cudaMemcpyDeviceToHost, st));
    CUDA_TRY(cudaMemcpyAsync(T.hn.data(), T.npart.p, sizeof(unsigned long long) * blocks, cudaMemcpyDeviceToHost, st));
    CUDA_TRY(cudaStreamSynchronize(st));
    T.sum0 = T.sum1 = 0.0;
    T.dets = 0;
    for (int x = 0; x < blocks; x++) {
        T.sum0 += T.hp[2 * x];
        T.sum1 += T.hp[2 * x + 1];
        T.dets += (int64_t)T.hn[x];
    }
}

template <int W, int KW>
static double pt2_w(shci_ctx *c, const double *cd, double e_var, double eps2, int nbatch, int64_t &n_pert,
                    int &nbatch_used, int64_t &candidates) {
    SelArgs S = sel_args(c, eps2);
    S.c = cd;
    const DevInts I = dev_ints(c);
    TermWork T;
    // batches: enough that one batch's candidates and their sort fit a quarter of free memory
    constexpr double BYTES_PER_CAND = 2.0 * 8 * KW + 8 + 2 * 4;
    int64_t all = -1;                       // the count over every batch, where it was taken
    if (nbatch <= 0) {
        all = count_candidates<W, KW, true>(c, S, I, T.cnt, T.off, T.tmp);
        size_t fr = 0, tot = 0;
        CUDA_TRY(cudaMemGetInfo(&fr, &tot));
        const double budget = 0.25 * (double)fr;
        nbatch = (int)std::max<double>(1.0, std::ceil((double)all * BYTES_PER_CAND / budget));
        nbatch = std::max(nbatch, (int)((all + 0xFFFFFFFEll) / 0xFFFFFFFFll));
    }
    nbatch_used = nbatch;
    sorted_space<W, KW>(c, T.vs);
    double e2 = 0.0;
    n_pert = 0;
    candidates = 0;
    S.nbatch = nbatch;
    for (int b = 0; b < nbatch; b++) {
        S.batch = b;
        const int64_t total = nbatch == 1 && all >= 0 ? all
                                                      : count_candidates<W, KW, true>(c, S, I, T.cnt, T.off, T.tmp);
        candidates += total;
        if (total == 0) continue;
        if (total > 0xFFFFFFFFll) throw ShciError{SHCI_ERR_INVALID, "too many candidates in one batch: more batches"};
        reduce_terms<W, KW, RUN_PT>(c, S, I, total, e_var, 0.0, T);
        e2 += T.sum0;
        n_pert += T.dets;
    }
    return e2;
}

// ---------------------------------------------------------------- stochastic second-order energy

// sum |c_i| in a fixed order: per-block partials, then one block over them
__global__ void k_abs_partial(const double *__restrict__ c, int64_t n, double *__restrict__ part) {
    double s = 0.0;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        s += fabs(c[i]);
    __shared__ double red[SEL_THREADS / 32];
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < SEL_THREADS / 32; w++) t += red[w];
        part[blockIdx.x] = t;
    }
}

__global__ void k_sum_in_order(const double *__restrict__ part, int m, double *__restrict__ out) {
    if (threadIdx.x != 0 || blockIdx.x != 0) return;
    double t = 0.0;
    for (int b = 0; b < m; b++) t += part[b];
    *out = t;
}

// Walker's alias table for p_i = |c_i| / sum (Eq. 10), by Vose's two-list
// method: q_i = n p_i, the lists of small (q < 1) and large columns in
// ascending order, then pairs from the lists' ends.
__global__ void k_alias_split(const double *__restrict__ c, int64_t n, const double *__restrict__ sum,
                              double *__restrict__ q, int64_t *__restrict__ is_small) {
    const double scale = (double)n / *sum;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        q[i] = fabs(c[i]) * scale;
        is_small[i] = q[i] < 1.0 ? 1 : 0;
    }
}

// the lists, and the table's values for columns that are never paired: a large
// column keeps itself (probability 1), a small one its q and itself
__global__ void k_alias_lists(const double *__restrict__ q, int64_t n, const int64_t *__restrict__ pos,
                              uint32_t *__restrict__ small, uint32_t *__restrict__ large, double *__restrict__ prob,
                              int64_t *__restrict__ alias) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t s = pos[i];
        const bool is_small = q[i] < 1.0;
        if (is_small) small[s] = (uint32_t)i;
        else large[i - s] = (uint32_t)i;
        prob[i] = is_small ? q[i] : 1.0;
        alias[i] = i;
    }
}

// The pairing: the small column on top of its stack takes the large column g
// on top of the other as its alias, g keeps q_g + q_l - 1, and a g that falls
// below 1 goes onto the small stack.  Each step needs the one before it, but a
// demoted g is popped by the very next step, so both stacks are read strictly
// from their ends: one warp stages ALIAS_CH columns of each in shared memory,
// one lane runs the chain of additions over them, and the warp writes the
// aliases.  Bound by that chain (two dependent FP64 additions per column).
// With every access a dependent global load, 100,003 columns took 43.4 ms;
// this form 10.3.
constexpr int ALIAS_CH = 1024;

__global__ void __launch_bounds__(32) k_alias_pair(const double *__restrict__ q, const uint32_t *__restrict__ small,
                                                   const uint32_t *__restrict__ large, const int64_t *__restrict__ n_small,
                                                   int64_t n, double *__restrict__ prob, int64_t *__restrict__ alias) {
    __shared__ double sq[ALIAS_CH + 1], lq[ALIAS_CH];
    __shared__ uint32_t sidx[ALIAS_CH], lidx[ALIAS_CH], spair[ALIAS_CH];
    const int lane = threadIdx.x;
    int64_t ns = *n_small, nl = n - ns;                  // columns not yet staged
    int sc = 0, sk = 0, lc = 0, lk = 0;                  // staged and consumed
    bool have = false, demoted = false;                  // a large column in hand; a demoted one on top of the small stack
    double gq = 0.0, dq = 0.0;
    uint32_t gi = 0, di = 0;
    while (true) {
        if (sk == sc && ns > 0) {
            sc = (int)min((int64_t)ALIAS_CH, ns);
            for (int x = lane; x < sc; x += 32) {
                sidx[x] = small[ns - 1 - x];
                sq[x] = q[sidx[x]];
            }
            ns -= sc;
            sk = 0;
        }
        if (lk == lc && nl > 0) {
            lc = (int)min((int64_t)ALIAS_CH, nl);
            for (int x = lane; x < lc; x += 32) {
                lidx[x] = large[nl - 1 - x];
                lq[x] = q[lidx[x]];
            }
            nl -= lc;
            lk = 0;
        }
        __syncwarp();
        const int from = sk;
        if (lane == 0) {
            while (true) {
                if (!have) {
                    if (lk == lc) break;
                    gi = lidx[lk];
                    gq = lq[lk++];
                    have = true;
                }
                if (demoted) {
                    prob[di] = dq;
                    alias[di] = gi;
                    gq = (gq + dq) - 1.0;
                    demoted = false;
                } else {
                    if (sk == sc) break;
                    double next = sq[sk];
                    do {                                  // q_g >= 1 and q_l >= 0: the sign needs no test
                        const double l = next;
                        spair[sk] = gi;
                        next = sq[++sk];
                        gq = (gq + l) - 1.0;
                    } while (sk < sc && __double2hiint(gq) >= 0x3FF00000);
                }
                if (__double2hiint(gq) < 0x3FF00000) {    // below 1
                    demoted = true;
                    di = gi;
                    dq = gq;
                    have = false;
                }
            }
        }
        sk = __shfl_sync(0xffffffffu, sk, 0);
        lk = __shfl_sync(0xffffffffu, lk, 0);
        have = __shfl_sync(0xffffffffu, (int)have, 0);
        demoted = __shfl_sync(0xffffffffu, (int)demoted, 0);
        __syncwarp();
        for (int x = from + lane; x < sk; x += 32) alias[sidx[x]] = spair[x];
        __syncwarp();
        if ((!demoted && sk == sc && ns == 0) || (!have && lk == lc && nl == 0)) break;
    }
    // rounding leftovers keep themselves: the demoted column on top, the small columns never paired
    if (lane == 0 && demoted) prob[di] = 1.0;
    for (int x = sk + lane; x < sc; x += 32) prob[sidx[x]] = 1.0;
    for (int64_t x = lane; x < ns; x += 32) prob[small[x]] = 1.0;
}

// draw d: r = SplitMix64 output for the counter seed + (d + 1) * golden
// gamma; column = high 32 bits * n >> 32, uniform u = low 32 bits / 2^32;
// the column itself when u < prob[column], else its alias
__global__ void k_alias_draw(const double *__restrict__ prob, const int64_t *__restrict__ alias, int64_t n,
                             uint64_t seed, int64_t n_draws, int64_t *__restrict__ out) {
    for (int64_t d = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; d < n_draws;
         d += (int64_t)gridDim.x * blockDim.x) {
        uint64_t z = seed + (uint64_t)(d + 1) * 0x9E3779B97F4A7C15ull;
        z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
        z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
        z ^= z >> 31;
        const int64_t col = (int64_t)(((z >> 32) * (uint64_t)n) >> 32);
        const double u = (double)(uint32_t)z * 0x1p-32;
        out[d] = u < prob[col] ? col : alias[col];
    }
}

static double abs_sum(shci_ctx *c, const double *cd, int64_t n) {
    cudaStream_t st = c->st;
    const int nb = (int)std::min<int64_t>(ceil_div(n, SEL_THREADS), (int64_t)c->n_sm * 4);
    DevBuf<double> part, tot;
    part.alloc((size_t)nb);
    tot.alloc(1);
    k_abs_partial<<<nb, SEL_THREADS, 0, st>>>(cd, n, part.p);
    k_sum_in_order<<<1, 32, 0, st>>>(part.p, nb, tot.p);
    KERNEL_CHECK();
    g_kernel_launches += 2;
    double h = 0.0;
    CUDA_TRY(cudaMemcpyAsync(&h, tot.p, sizeof(double), cudaMemcpyDeviceToHost, st));
    CUDA_TRY(cudaStreamSynchronize(st));
    return h;
}

// sample prep: run heads of the sorted draws -> distinct index, count, and the
// per-determinant compact arrays (strings, c_i, w/p, w (n_d - 1)/p - w^2/p^2)
template <int W>
__global__ void k_sample_prep(const uint64_t *__restrict__ sorted, int64_t n_d, const int64_t *__restrict__ pos,
                              const uint64_t *__restrict__ dets, const double *__restrict__ c, double csum,
                              uint64_t *__restrict__ sdets, double *__restrict__ sc, double *__restrict__ f1,
                              double *__restrict__ f2) {
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n_d; e += (int64_t)gridDim.x * blockDim.x) {
        if (e > 0 && sorted[e - 1] == sorted[e]) continue;
        int64_t f = e + 1;
        while (f < n_d && sorted[f] == sorted[e]) f++;
        const int64_t i = (int64_t)sorted[e], u = pos[e];
        const double w = (double)(f - e), p = fabs(c[i]) / csum;
#pragma unroll
        for (int k = 0; k < 2 * W; k++) sdets[u * 2 * W + k] = dets[i * 2 * W + k];
        sc[u] = c[i];
        f1[u] = w / p;
        f2[u] = w * (double)(n_d - 1) / p - w * w / (p * p);
    }
}

__global__ void k_run_heads(const uint64_t *__restrict__ sorted, int64_t n, int64_t *__restrict__ flag) {
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x)
        flag[e] = (e == 0 || sorted[e - 1] != sorted[e]) ? 1 : 0;
}

// any draw that is out of range or has a zero coefficient?
__global__ void k_check_draws(const int64_t *__restrict__ draws, int64_t m, const double *__restrict__ c, int64_t n,
                              int *__restrict__ bad) {
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < m; e += (int64_t)gridDim.x * blockDim.x) {
        const int64_t v = draws[e];
        if (v < 0 || v >= n || c[v] == 0.0) *bad = 1;
    }
}

template <int W, int KW>
static void pt2_samples_w(shci_ctx *c, const double *cd, double e_var, double eps2, double eps2_d, int64_t n_d,
                          int n_samples, const int64_t *draws, double *out, int nbatch, const int *batch_of_sample) {
    cudaStream_t st = c->st;
    const int64_t n = c->n_det;
    const double csum = abs_sum(c, cd, n);
    if (!(csum > 0.0)) throw ShciError{SHCI_ERR_INVALID, "all coefficients are zero"};
    TermWork T;
    sorted_space<W, KW>(c, T.vs);
    const DevInts I = dev_ints(c);
    DevBuf<uint64_t> sorted, sdets;
    DevBuf<int64_t> flag, pos, tmp;
    DevBuf<double> sc, f1, f2;
    sorted.alloc((size_t)n_d);
    flag.alloc((size_t)n_d + 1);
    pos.alloc((size_t)n_d + 1);
    tmp.alloc((size_t)scan_tmp_len(n_d + 1));
    sdets.alloc((size_t)n_d * 2 * W);
    sc.alloc((size_t)n_d);
    f1.alloc((size_t)n_d);
    f2.alloc((size_t)n_d);
    uint64_t vary = 1;                      // bits of an index of V
    while ((int64_t)vary < n - 1) vary = 2 * vary + 1;
    const int gb = (int)std::min<int64_t>(ceil_div(n_d, SEL_THREADS), (int64_t)c->n_sm * 16);
    for (int smp = 0; smp < n_samples; smp++) {
        CUDA_TRY(cudaMemcpyAsync(sorted.p, draws + (int64_t)smp * n_d, sizeof(int64_t) * n_d,
                                 cudaMemcpyDeviceToDevice, st));
        radix_sort<1>(sorted.p, nullptr, n_d, c->sw, st, &vary, RS_KEYS);
        k_run_heads<<<gb, SEL_THREADS, 0, st>>>(sorted.p, n_d, flag.p);
        exclusive_scan<int64_t>(flag.p, pos.p, n_d, tmp.p, st);
        int64_t n_dist = 0;
        CUDA_TRY(cudaMemcpyAsync(&n_dist, pos.p + n_d, sizeof(int64_t), cudaMemcpyDeviceToHost, st));
        k_sample_prep<W><<<gb, SEL_THREADS, 0, st>>>(sorted.p, n_d, pos.p, c->dets.p, cd, csum, sdets.p, sc.p, f1.p,
                                                     f2.p);
        KERNEL_CHECK();
        g_kernel_launches += 2;
        CUDA_TRY(cudaStreamSynchronize(st));
        SelArgs S = sel_args(c, eps2);
        S.n_det = n_dist;
        S.dets = sdets.p;
        S.c = sc.p;
        S.nbatch = nbatch;
        S.batch = batch_of_sample ? batch_of_sample[smp] : 0;
        S.f1 = f1.p;
        S.f2 = f2.p;
        const int64_t total = count_candidates<W, KW, true>(c, S, I, T.cnt, T.off, T.tmp);
        const double norm = 1.0 / ((double)n_d * (double)(n_d - 1));
        if (total == 0) {
            out[2 * smp] = 0.0;
            out[2 * smp + 1] = 0.0;
            continue;
        }
        if (total > 0xFFFFFFFFll) throw ShciError{SHCI_ERR_INVALID, "too many terms in one sample: raise eps2"};
        reduce_terms<W, KW, RUN_SAMPLE>(c, S, I, total, e_var, eps2_d, T);
        out[2 * smp] = T.sum0 * norm;
        out[2 * smp + 1] = T.sum1 * norm;
    }
}

static void ensure_lists(shci_ctx *c) {
    if (!c->hb_valid) {
        build_hb_list(c, 1, c->hb_same);
        build_hb_list(c, 0, c->hb_opp);
        c->hb_valid = true;
    }
}

void pt2_samples(shci_ctx *c, const double *coef, double e_var, double eps2, double eps2_d, int64_t n_d,
                 int n_samples, const int64_t *draws, double *out, int mem, int nbatch, const int *batch_of_sample) {
    if (nbatch < 1 || nbatch > 1 << 20) throw ShciError{SHCI_ERR_INVALID, "n_batches must be in [1, 2^20]"};
    if (batch_of_sample)
        for (int sm = 0; sm < n_samples; sm++)
            if (batch_of_sample[sm] < 0 || batch_of_sample[sm] >= nbatch)
                throw ShciError{SHCI_ERR_INVALID, "batch index out of range"};
    if (!c->built) throw ShciError{SHCI_ERR_STATE, "build the connectivity first"};
    if (!(eps2 > 0.0) || !std::isfinite(eps2) || !(eps2_d >= eps2) || !std::isfinite(eps2_d))
        throw ShciError{SHCI_ERR_INVALID, "need 0 < eps2 <= eps2_d, finite"};
    if (!std::isfinite(e_var)) throw ShciError{SHCI_ERR_INVALID, "e_var must be finite"};
    if (n_d < 2 || n_samples < 1 || !coef || !draws || !out) throw ShciError{SHCI_ERR_INVALID, "bad sample arguments"};
    if (mem != SHCI_MEM_HOST && mem != SHCI_MEM_DEVICE) throw ShciError{SHCI_ERR_INVALID, "unknown mem_space"};
    if (c->n_orb > 128) throw ShciError{SHCI_ERR_INVALID, "up to 128 orbitals"};
    cudaStream_t st = c->st;
    ensure_lists(c);
    const int64_t n = c->n_det;
    const double *cd = coef;
    const int64_t *dd = draws;
    DevBuf<double> cbuf;
    DevBuf<int64_t> dbuf;
    if (mem == SHCI_MEM_HOST) {
        cbuf.alloc((size_t)n);
        CUDA_TRY(cudaMemcpyAsync(cbuf.p, coef, sizeof(double) * n, cudaMemcpyHostToDevice, st));
        cd = cbuf.p;
        dbuf.alloc((size_t)n_samples * n_d);
        CUDA_TRY(cudaMemcpyAsync(dbuf.p, draws, sizeof(int64_t) * n_samples * n_d, cudaMemcpyHostToDevice, st));
        dd = dbuf.p;
    }
    // every draw must index a determinant of V with a nonzero coefficient
    {
        DevBuf<int> bad;
        bad.alloc(1);
        CUDA_TRY(cudaMemsetAsync(bad.p, 0, sizeof(int), st));
        const int64_t m = (int64_t)n_samples * n_d;
        k_check_draws<<<(int)std::min<int64_t>(ceil_div(m, SEL_THREADS), (int64_t)c->n_sm * 16), SEL_THREADS, 0,
                        st>>>(dd, m, cd, n, bad.p);
        KERNEL_CHECK();
        g_kernel_launches += 1;
        int any = 0;
        CUDA_TRY(cudaMemcpyAsync(&any, bad.p, sizeof(int), cudaMemcpyDeviceToHost, st));
        CUDA_TRY(cudaStreamSynchronize(st));
        if (any) throw ShciError{SHCI_ERR_INVALID, "a draw is out of range or has a zero coefficient"};
    }
    std::vector<double> res((size_t)2 * n_samples);
#define CALL(W, KW) \
    pt2_samples_w<W, KW>(c, cd, e_var, eps2, eps2_d, n_d, n_samples, dd, res.data(), nbatch, batch_of_sample)
    DISPATCH_KEYS(c, CALL);
#undef CALL
    for (size_t e = 0; e < res.size(); e++) out[e] = res[e];
}

void alias_draw(shci_ctx *c, const double *coef, int64_t n_draws, uint64_t seed, int64_t *out, int mem) {
    if (!c->built) throw ShciError{SHCI_ERR_STATE, "build the connectivity first"};
    if (n_draws < 0 || !coef || (n_draws > 0 && !out)) throw ShciError{SHCI_ERR_INVALID, "bad draw arguments"};
    if (mem != SHCI_MEM_HOST && mem != SHCI_MEM_DEVICE) throw ShciError{SHCI_ERR_INVALID, "unknown mem_space"};
    cudaStream_t st = c->st;
    const int64_t n = c->n_det;
    if (n > 0xFFFFFFFFll) throw ShciError{SHCI_ERR_INVALID, "too many determinants for the sampler"};
    const double *cd = coef;
    DevBuf<double> cbuf;
    if (mem == SHCI_MEM_HOST) {
        cbuf.alloc((size_t)n);
        CUDA_TRY(cudaMemcpyAsync(cbuf.p, coef, sizeof(double) * n, cudaMemcpyHostToDevice, st));
        cd = cbuf.p;
    }
    const double csum = abs_sum(c, cd, n);
    if (!(csum > 0.0)) throw ShciError{SHCI_ERR_INVALID, "all coefficients are zero"};
    DevBuf<double> prob, q, sum;
    DevBuf<int64_t> alias, flag, pos, tmp, obuf;
    DevBuf<uint32_t> small, large;
    prob.alloc((size_t)n);
    q.alloc((size_t)n);
    sum.alloc(1);
    alias.alloc((size_t)n);
    flag.alloc((size_t)n + 1);
    pos.alloc((size_t)n + 1);
    tmp.alloc((size_t)scan_tmp_len(n + 1));
    small.alloc((size_t)n);
    large.alloc((size_t)n);
    CUDA_TRY(cudaMemcpyAsync(sum.p, &csum, sizeof(double), cudaMemcpyHostToDevice, st));
    const int gn = (int)std::min<int64_t>(ceil_div(n, SEL_THREADS), (int64_t)c->n_sm * 16);
    k_alias_split<<<gn, SEL_THREADS, 0, st>>>(cd, n, sum.p, q.p, flag.p);
    exclusive_scan<int64_t>(flag.p, pos.p, n, tmp.p, st);
    k_alias_lists<<<gn, SEL_THREADS, 0, st>>>(q.p, n, pos.p, small.p, large.p, prob.p, alias.p);
    k_alias_pair<<<1, 32, 0, st>>>(q.p, small.p, large.p, pos.p + n, n, prob.p, alias.p);
    KERNEL_CHECK();
    g_kernel_launches += 3;
    if (n_draws == 0) return;
    int64_t *o = out;
    if (mem == SHCI_MEM_HOST) {
        obuf.alloc((size_t)n_draws);
        o = obuf.p;
    }
    const int gb = (int)std::min<int64_t>(ceil_div(n_draws, SEL_THREADS), (int64_t)c->n_sm * 16);
    k_alias_draw<<<gb, SEL_THREADS, 0, st>>>(prob.p, alias.p, n, seed, n_draws, o);
    KERNEL_CHECK();
    g_kernel_launches += 1;
    if (mem == SHCI_MEM_HOST)
        CUDA_TRY(cudaMemcpyAsync(out, o, sizeof(int64_t) * n_draws, cudaMemcpyDeviceToHost, st));
    CUDA_TRY(cudaStreamSynchronize(st));
}

void pt2(shci_ctx *c, const double *coef, double e_var, double eps2, int nbatch, double *e2, int64_t *n_pert,
         int mem) {
    if (!c->built) throw ShciError{SHCI_ERR_STATE, "build the connectivity before the second-order energy"};
    if (!(eps2 > 0.0) || !std::isfinite(eps2)) throw ShciError{SHCI_ERR_INVALID, "eps2 must be positive and finite"};
    if (!std::isfinite(e_var)) throw ShciError{SHCI_ERR_INVALID, "e_var must be finite"};
    if (!coef || !e2) throw ShciError{SHCI_ERR_INVALID, "null pointer"};
    if (nbatch < 0 || nbatch > 1 << 20) throw ShciError{SHCI_ERR_INVALID, "n_batches must be in [0, 2^20]"};
    if (mem != SHCI_MEM_HOST && mem != SHCI_MEM_DEVICE) throw ShciError{SHCI_ERR_INVALID, "unknown mem_space"};
    if (c->n_orb > 128) throw ShciError{SHCI_ERR_INVALID, "up to 128 orbitals"};
    cudaStream_t st = c->st;
    cudaEvent_t e0, e1;
    CUDA_TRY(cudaEventCreate(&e0));
    CUDA_TRY(cudaEventCreate(&e1));
    CUDA_TRY(cudaEventRecord(e0, st));
    ensure_lists(c);
    const double *cd = coef;
    DevBuf<double> cbuf;
    if (mem == SHCI_MEM_HOST) {
        cbuf.alloc((size_t)c->n_det);
        CUDA_TRY(cudaMemcpyAsync(cbuf.p, coef, sizeof(double) * c->n_det, cudaMemcpyHostToDevice, st));
        cd = cbuf.p;
    }
    int64_t np = 0, cands = 0;
    int used = 0;
    double v = 0.0;
#define CALL(W, KW) v = pt2_w<W, KW>(c, cd, e_var, eps2, nbatch, np, used, cands)
    DISPATCH_KEYS(c, CALL);
#undef CALL
    *e2 = v;
    if (n_pert) *n_pert = np;
    CUDA_TRY(cudaEventRecord(e1, st));
    CUDA_TRY(cudaEventSynchronize(e1));
    float ms = 0.f;
    cudaEventElapsedTime(&ms, e0, e1);
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    c->stats.pt2_ms = ms;
    c->stats.pt2_batches = used;
    c->stats.pt2_terms = cands;
}

// Pseudo-stochastic step of the 3-step scheme: batches of the perturbative
// determinants (hash partition, at least 16) in order; after each batch the
// corrections seen so far give a mean and variance, the number of
// perturbative determinants is extrapolated from the batches done, and the
// loop stops when the standard deviation of the estimated sum of the
// unevaluated ones is below 0.4 target (all batches: exact, zero deviation).
template <int W, int KW>
static void psto_w(shci_ctx *c, const double *cd, double e_var, double eps_psto, double eps_dtm, int nbatch,
                   double target, double &est, double &err, int &done) {
    SelArgs S = sel_args(c, eps_psto);
    S.c = cd;
    S.nbatch = nbatch;
    const DevInts I = dev_ints(c);
    TermWork T;
    sorted_space<W, KW>(c, T.vs);
    double sum = 0.0, sum2 = 0.0;
    int64_t count = 0;
    est = 0.0;
    err = 0.0;
    done = 0;
    for (int b = 0; b < nbatch; b++) {
        S.batch = b;
        const int64_t total = count_candidates<W, KW, true>(c, S, I, T.cnt, T.off, T.tmp);
        if (total > 0xFFFFFFFFll) throw ShciError{SHCI_ERR_INVALID, "too many terms in one batch: more batches"};
        if (total > 0) {
            reduce_terms<W, KW, RUN_PSTO>(c, S, I, total, e_var, eps_dtm, T);
            sum += T.sum0;
            sum2 += T.sum1;
            count += T.dets;
        }
        done = b + 1;
        if (done == nbatch) {
            est = sum;
            err = 0.0;
            break;
        }
        const double n_est = (double)count * nbatch / done;             // perturbative determinants, all batches
        const double rest = n_est - (double)count;
        const double mean = count > 0 ? sum / count : 0.0;
        const double var = count > 1 ? std::max(0.0, (sum2 - count * mean * mean) / (count - 1)) : 0.0;
        est = sum + mean * rest;
        err = std::sqrt(var * rest);
        if (count > 1 && err < 0.4 * target) break;
    }
}

void pt2_3step(shci_ctx *c, const double *coef, double e_var, double eps2, double eps2_psto, double eps2_dtm,
               double target, int nbatch_psto, int nbatch_sto, int64_t n_d, int n_samples, uint64_t seed,
               shci_pt2_3step_t *out, int mem) {
    if (!out) throw ShciError{SHCI_ERR_INVALID, "null pointer"};
    if (!(eps2 > 0.0 && eps2 <= eps2_psto && eps2_psto <= eps2_dtm) || !std::isfinite(eps2_dtm))
        throw ShciError{SHCI_ERR_INVALID, "need 0 < eps2 <= eps2_psto <= eps2_dtm, finite"};
    if (!(target >= 0.0)) throw ShciError{SHCI_ERR_INVALID, "target error must be >= 0"};
    if (nbatch_psto < 16 || nbatch_psto > 1 << 20 || nbatch_sto < 1 || nbatch_sto > 1 << 20)
        throw ShciError{SHCI_ERR_INVALID, "need 16 <= pseudo-stochastic batches and 1 <= stochastic batches"};
    if (n_samples < 1 || n_d < 2) throw ShciError{SHCI_ERR_INVALID, "need n_samples >= 1 and n_d >= 2"};
    if (mem != SHCI_MEM_HOST && mem != SHCI_MEM_DEVICE) throw ShciError{SHCI_ERR_INVALID, "unknown mem_space"};
    cudaStream_t st = c->st;
    const double *cd = coef;
    DevBuf<double> cbuf;
    if (mem == SHCI_MEM_HOST) {
        cbuf.alloc((size_t)c->n_det);
        CUDA_TRY(cudaMemcpyAsync(cbuf.p, coef, sizeof(double) * c->n_det, cudaMemcpyHostToDevice, st));
        cd = cbuf.p;
    }
    *out = shci_pt2_3step_t{};
    // 1: deterministic at eps2_dtm (hash batches as memory requires)
    pt2(c, cd, e_var, eps2_dtm, 0, &out->dtm, nullptr, SHCI_MEM_DEVICE);
    // 2: pseudo-stochastic at eps2_psto, minus its eps2_dtm part
    ensure_lists(c);
    if (eps2_psto < eps2_dtm) {
#define CALL(W, KW)                                                                                            \
    psto_w<W, KW>(c, cd, e_var, eps2_psto, eps2_dtm, nbatch_psto, target, out->psto, out->psto_err, out->psto_batches)
        DISPATCH_KEYS(c, CALL);
#undef CALL
    }
    // 3: stochastic at eps2, minus its eps2_psto part; one batch per sample, drawn
    // from the SplitMix64 stream after the determinant draws, times the batch count
    if (eps2 < eps2_psto) {
        DevBuf<int64_t> draws;
        draws.alloc((size_t)n_samples * n_d);
        alias_draw(c, cd, (int64_t)n_samples * n_d, seed, draws.p, SHCI_MEM_DEVICE);
        std::vector<int> bsel(n_samples);
        for (int sm = 0; sm < n_samples; sm++) {
            uint64_t z = seed + (uint64_t)((int64_t)n_samples * n_d + sm + 1) * 0x9E3779B97F4A7C15ull;
            z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
            z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
            z ^= z >> 31;
            bsel[sm] = (int)(((z >> 32) * (uint64_t)nbatch_sto) >> 32);
        }
        std::vector<double> v((size_t)2 * n_samples);
        pt2_samples(c, cd, e_var, eps2, eps2_psto, n_d, n_samples, draws.p, v.data(), SHCI_MEM_DEVICE, nbatch_sto,
                    bsel.data());
        double mean = 0.0;
        for (int sm = 0; sm < n_samples; sm++) mean += nbatch_sto * (v[2 * sm] - v[2 * sm + 1]);
        mean /= n_samples;
        double var = 0.0;
        for (int sm = 0; sm < n_samples; sm++) {
            const double d = nbatch_sto * (v[2 * sm] - v[2 * sm + 1]) - mean;
            var += d * d;
        }
        out->sto = mean;
        out->sto_err = n_samples > 1 ? std::sqrt(var / (n_samples - 1) / n_samples) : 0.0;
    }
    out->e2 = out->dtm + out->psto + out->sto;
    out->e2_err = std::sqrt(out->psto_err * out->psto_err + out->sto_err * out->sto_err);
}

void pt2_semistochastic(shci_ctx *c, const double *coef, double e_var, double eps2, double eps2_d, int64_t n_d,
                        int n_samples, uint64_t seed, double *e2, double *e2_err, int mem) {
    if (!e2) throw ShciError{SHCI_ERR_INVALID, "null pointer"};
    if (n_samples < 1 || n_d < 2) throw ShciError{SHCI_ERR_INVALID, "need n_samples >= 1 and n_d >= 2"};
    // deterministic part at eps2_d (Eq. 8)
    double e2d = 0.0;
    pt2(c, coef, e_var, eps2_d, 0, &e2d, nullptr, mem);
    // stochastic part: the same samples at eps2 and at eps2_d (Eq. 9)
    DevBuf<int64_t> draws;
    draws.alloc((size_t)n_samples * n_d);
    const double *cd = coef;
    DevBuf<double> cbuf;
    if (mem == SHCI_MEM_HOST) {
        cbuf.alloc((size_t)c->n_det);
        CUDA_TRY(cudaMemcpyAsync(cbuf.p, coef, sizeof(double) * c->n_det, cudaMemcpyHostToDevice, c->st));
        cd = cbuf.p;
    }
    alias_draw(c, cd, (int64_t)n_samples * n_d, seed, draws.p, SHCI_MEM_DEVICE);
    std::vector<double> v((size_t)2 * n_samples);
    pt2_samples(c, cd, e_var, eps2, eps2_d, n_d, n_samples, draws.p, v.data(), SHCI_MEM_DEVICE, 1, nullptr);
    double mean = 0.0;
    for (int sm = 0; sm < n_samples; sm++) mean += v[2 * sm] - v[2 * sm + 1];
    mean /= n_samples;
    double var = 0.0;
    for (int sm = 0; sm < n_samples; sm++) {
        const double d = v[2 * sm] - v[2 * sm + 1] - mean;
        var += d * d;
    }
    *e2 = e2d + mean;
    if (e2_err) *e2_err = n_samples > 1 ? std::sqrt(var / (n_samples - 1) / n_samples) : 0.0;
}

void select_dets(shci_ctx *c, int k, const double *coef, double eps1, int64_t cap, uint64_t *out, int64_t *n_out,
                 int mem) {
    if (!c->built) throw ShciError{SHCI_ERR_STATE, "build the connectivity before selecting"};
    if (k < 1 || k > SHCI_MAX_K) throw ShciError{SHCI_ERR_INVALID, "k must be in [1, 8]"};
    if (!(eps1 > 0.0) || !std::isfinite(eps1)) throw ShciError{SHCI_ERR_INVALID, "eps1 must be positive and finite"};
    if (!coef || !n_out) throw ShciError{SHCI_ERR_INVALID, "null pointer"};
    if (cap < 0) throw ShciError{SHCI_ERR_INVALID, "cap must be >= 0"};
    if (mem != SHCI_MEM_HOST && mem != SHCI_MEM_DEVICE) throw ShciError{SHCI_ERR_INVALID, "unknown mem_space"};
    if (c->n_orb > 128) throw ShciError{SHCI_ERR_INVALID, "selection supports up to 128 orbitals"};
    cudaStream_t st = c->st;
    cudaEvent_t e0, e1;
    CUDA_TRY(cudaEventCreate(&e0));
    CUDA_TRY(cudaEventCreate(&e1));
    CUDA_TRY(cudaEventRecord(e0, st));
    if (!c->hb_valid) {
        build_hb_list(c, 1, c->hb_same);
        build_hb_list(c, 0, c->hb_opp);
        c->hb_valid = true;
    }
    const double *cd = coef;
    DevBuf<double> cbuf;
    if (mem == SHCI_MEM_HOST) {
        cbuf.alloc((size_t)k * c->n_det);
        CUDA_TRY(cudaMemcpyAsync(cbuf.p, coef, sizeof(double) * k * c->n_det, cudaMemcpyHostToDevice, st));
        cd = cbuf.p;
    }
    DevBuf<uint64_t> result;
    int64_t n_new = 0;
#define CALL(W, KW) select_w<W, KW>(c, k, cd, eps1, result, n_new)
    DISPATCH_KEYS(c, CALL);
#undef CALL
    *n_out = n_new;
    const int KW = 2 * c->W;
    if (n_new > 0 && cap > 0) {
        if (!out) throw ShciError{SHCI_ERR_INVALID, "null output pointer"};
        const int64_t m = std::min(cap, n_new);
        CUDA_TRY(cudaMemcpyAsync(out, result.p, sizeof(uint64_t) * m * KW,
                                 mem == SHCI_MEM_HOST ? cudaMemcpyDeviceToHost : cudaMemcpyDeviceToDevice, st));
    }
    CUDA_TRY(cudaEventRecord(e1, st));
    CUDA_TRY(cudaEventSynchronize(e1));
    float ms = 0.f;
    cudaEventElapsedTime(&ms, e0, e1);
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    c->stats.select_ms = ms;
}

}  // namespace shci
