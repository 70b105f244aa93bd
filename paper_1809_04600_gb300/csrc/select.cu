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
#include "move_tables.cuh"

namespace shci {

constexpr int SEL_THREADS = 256;

// ---------------------------------------------------------------- sorted double-excitation lists

// Tuple t = ((p n + q) n + r) n + s.  List 0 (same spin): p < q, r < s,
// {r, s} disjoint from {p, q}, magnitude |(pr|qs) - (ps|qr)|.  List 1
// (opposite spin, p and r alpha, q and s beta): r != p, s != q, magnitude
// |(pr|qs)|.  Entries with magnitude 0 never meet eps1 > 0 and are dropped.
// v is the element up to the parity of the electrons below p, q, r and s in
// the determinant: moving p -> r and then q -> s passes those strictly between
// each pair, i.e. the parities below the four orbitals and the order relations
// among them, which v's sign already holds.
__device__ __forceinline__ bool hb_entry(const DevInts &I, int same, int64_t t, int &slot, int &r, int &s,
                                         double &v) {
    const int n = I.n;
    s = (int)(t % n);
    r = (int)((t / n) % n);
    const int q = (int)((t / ((int64_t)n * n)) % n);
    const int p = (int)(t / ((int64_t)n * n * n));
    slot = p * n + q;
    if (same) {
        if (!(p < q && r < s) || r == p || r == q || s == p || s == q) return false;
        v = flip_sign(eri_get(I, p, r, q, s) - eri_get(I, p, s, q, r), (p < r) + (p < s) + (r < q) + (q < s));
    } else {
        if (r == p || s == q) return false;
        v = flip_sign(eri_get(I, p, r, q, s), (p < r) + (q < s));
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

// The key bits that n_orb orbitals can set.  One-word keys are sorted by them;
// longer ones have digits that are the same in every key where few orbitals are
// in use, and a reduction that finds them costs less than a pass (the rule of
// OrbMask in build.cu; 76 orbitals, selection from 9,001 determinants 3.70 to
// 3.45 ms, from 100,003 at a tighter threshold 15.55 to 15.37).
template <int W, int KW>
struct KeyMask {
    uint64_t w[KW];
    const uint64_t *known() const { return KW == 1 ? w : nullptr; }
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
    radix_sort<KW>(vs.p, nullptr, n, c->sw, c->st, KeyMask<W, KW>(c->n_orb).known(), RS_KEYS);
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
    // single moves from per-string tables (null: evaluated in full), and each
    // determinant's string indices
    const double *ma, *mb;
    const int32_t *ia, *ib;
};

// The tables of both spins' strings, owned by one call (move_tables.cuh).
struct MoveTables {
    DevBuf<double> a, b;
};

// Tabulate when that is less work than evaluating the moves of `rows`
// determinants (table entries against moves, both a sum over the electrons;
// a quarter, since the tables are written and read back) and takes at most a
// sixteenth of the free memory; otherwise S keeps evaluating each move.
template <int W>
static void tabulate_moves(shci_ctx *c, SelArgs &S, const DevInts &I, double rows, MoveTables &T, bool own) {
    const int n = c->n_orb;
    if (c->have_moves) {                    // the connectivity's own
        S.ma = c->move_a.p;
        S.mb = c->move_b.p;
        S.ia = c->ia.p;
        S.ib = c->ib.p;
        return;
    }
    if (!own || !c->h_even) return;
    const int64_t np = (int64_t)n * (n + 1) / 2;
    const double entries = (double)(c->Ua + c->Ub) * np;
    const double moves = rows * ((double)S.na * (n - S.na) + (double)S.nb * (n - S.nb));
    if (entries > 0.25 * moves) return;
    size_t fr = 0, tot = 0;
    CUDA_TRY(cudaMemGetInfo(&fr, &tot));
    if (entries * 16.0 > (double)fr / 16.0) return;
    make_move_tables<W>(c, I, T.a, T.b);
    S.ma = T.a.p;
    S.mb = T.b.p;
    S.ia = c->ia.p;
    S.ib = c->ib.p;
}

// f(true), and where the memory runs out f(false): without tables of the call's own
template <typename F>
static void with_tables(F f) {
    try {
        f(true);
    } catch (const ShciError &e) {
        if (e.code != SHCI_ERR_OOM) throw;
        cudaGetLastError();
        f(false);
    }
}

// The test |v| cmax >= eps without FP64 arithmetic where the answer is not
// close: against eps / cmax in FP32, widened by 2^-16 on both sides (three
// FP32 roundings), comparing the high words of |v|; FP64 decides in between,
// for infinities and NaN, and everywhere when the ratio leaves FP32's range.
struct Cut {
    double cmax, eps;
    float reach;                            // list keys below this are out of reach (0: none is)
    uint32_t no, yes;                       // high words: below `no` fails, above `yes` passes
};

__device__ __forceinline__ Cut make_cut(double eps, double cmax) {
    Cut t{cmax, eps, 0.0f, 0u, 0x7FF00000u};
    const float e = (float)eps, m = (float)cmax, x = e / m;
    if (e > 1e-30f && e < 1e30f && m > 1e-30f && m < 1e30f && x > 1e-30f && x < 1e30f) {
        t.reach = x * (1.0f - 0x1p-16f);
        auto high = [](float f) {                         // high word of (double)f, f positive and normal
            const uint32_t b = __float_as_uint(f);
            return (((b >> 23) + 896u) << 20) | ((b >> 3) & 0xFFFFFu);
        };
        t.no = high(t.reach);
        t.yes = high(x * (1.0f + 0x1p-16f));
    }
    return t;
}

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

// The exact comparison, out of line: as part of `passes` the compiler would
// turn the branch into predicated FP64 instructions that every element issues.
static __device__ __noinline__ bool passes_exactly(double v, double cmax, double eps) { return fabs(v) * cmax >= eps; }

__device__ __forceinline__ bool passes(const Cut &t, double v) {
    const uint32_t h = (uint32_t)__double2hiint(v) & 0x7FFFFFFFu;
    if (h < t.no) return false;
    if (h > t.yes && h < 0x7FF00000u) return true;
    return passes_exactly(v, t.cmax, t.eps);
}

// A determinant as the bits of its key: spin orbital o (alpha), beta(n) + o.
template <int W, int KW>
__device__ __forceinline__ int beta_bit(int n) { return KW == 1 ? n : 64 * W; }

template <int KW>
__device__ __forceinline__ void set_bit(Key<KW> &k, int x) {
    if constexpr (KW == 1) {
        k.w[0] |= 1ull << x;
    } else {
#pragma unroll
        for (int w = 0; w < KW; w++)
            if (w == (x >> 6)) k.w[w] |= 1ull << (x & 63);
    }
}

// bit x: the parity of the set bits below x within x's spin string (up to a
// constant per string, which the two orbitals of every move cancel)
template <int W, int KW>
__device__ __forceinline__ Key<KW> parity_below(const Key<KW> &d) {
    Key<KW> o;
#pragma unroll
    for (int w = 0; w < KW; w++) {
        uint64_t y = d.w[w] << 1;
#pragma unroll
        for (int s = 1; s < 64; s <<= 1) y ^= y << s;
        if (KW > 1 && (w % W) != 0 && (__popcll(d.w[w - 1]) & 1)) y = ~y;     // W <= 2: one lower word
        o.w[w] = y;
    }
    return o;
}

// parity of the number of bits set in both
template <int KW>
__device__ __forceinline__ int common_parity(const Key<KW> &a, const Key<KW> &b) {
    uint64_t x = 0;
#pragma unroll
    for (int w = 0; w < KW; w++) x ^= a.w[w] & b.w[w];
    return __popcll(x) & 1;
}

// Occupied and empty orbitals of both strings, ascending, and the double
// excitation lists in reach, of a warp's determinant.
struct SelWork {
    uint8_t occ[2][SHCI_MAX_ORB], vir[2][SHCI_MAX_ORB];
    int first[32];                          // index of a list's first entry minus those before it in the sequence
    int holes[32];                          // its pair: p | q << 8 (key bits), 0x10000 for an opposite-spin pair, beta 0x20000
};

template <int W>
__device__ __forceinline__ void list_orbitals(SelWork &L, int spin, const Str<W> &s, int n) {
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

// What k_select is run for: the selection, or the terms of the second-order
// energy and which of their values a fill pass writes.
enum { SEL_DETS = 0, SEL_TERMS = 1, SEL_SAMPLE = 2, SEL_MAGS = 3 };

// One warp per determinant.  First every single move (alpha then beta), a lane
// per move.  Then the double excitations: for 32 occupied pairs at a time a
// lane finds by bisection how many leading entries of its pair's sorted list
// can meet the threshold, and the warp takes those entries of all 32 lists as
// one sequence, 32 at a time (the starts of the lists among the 32, as bits,
// tell a lane its list), so that no lane waits for another's longer list and
// candidates leave as one contiguous, ordered run.  A candidate is the
// determinant's key with the holes' and particles' bits flipped, its sign the
// parity of those bits in the prefix-parity word.
// Walking one list per lane and reserving slots one by one took 17.7 ms
// (count) and 24.2 ms (fill) for the 1.8e8 terms of 200,003 determinants of 24
// orbitals (eps 1e-5); balanced, 5.5 and 7.8 with the FP64 pipe 75 % busy on
// thresholds and single moves; with those taken off it (Cut, k_move_tables)
// and bits instead of strings 2.6 and 3.4: bound by issue.
template <int W, int KW, bool FILL, int FOR>
__global__ void __launch_bounds__(SEL_THREADS) k_select(SelArgs S, DevInts I) {
    __shared__ SelWork work[SEL_THREADS / 32];
    const int lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u, le = lt | (1u << lane);
    SelWork &L = work[threadIdx.x >> 5];
    const int n = S.n, na = S.na, nb = S.nb;
    const int u_sa = na * (n - na), u_sb = nb * (n - nb);
    const int u_paa = na * (na - 1) / 2, u_pbb = nb * (nb - 1) / 2, u_pab = na * nb;
    const int pairs = u_paa + u_pbb + u_pab;
    const int beta = beta_bit<W, KW>(n);
    const int64_t warps = (int64_t)gridDim.x * (SEL_THREADS / 32);
    for (int64_t i = ((int64_t)blockIdx.x * SEL_THREADS + threadIdx.x) >> 5; i < S.n_det; i += warps) {
        double cmax = 0.0, ci = 0.0, f1 = 0.0, f2 = 0.0;
        if (FOR != SEL_DETS) {
            ci = __ldg(&S.c[i]);
            cmax = fabs(ci);
        } else {
            for (int l = 0; l < S.k; l++) cmax = fmax(cmax, fabs(__ldg(&S.c[(int64_t)l * S.n_det + i])));
        }
        if (FILL && FOR == SEL_SAMPLE) {
            f1 = __ldg(&S.f1[i]) * ci;
            f2 = __ldg(&S.f2[i]) * ci * ci;
        }
        int64_t pos = FILL ? __ldg(&S.off[i]) : 0;        // next slot, or candidates so far
        if (cmax > 0.0) {
            const Cut cut = make_cut(S.eps1, cmax);
            const Str<W> A = load_str<W>(S.dets, 2 * i), B = load_str<W>(S.dets, 2 * i + 1);
            const Key<KW> D = make_key<W, KW>(A, B, n);
            const Key<KW> PD = parity_below<W, KW>(D);
            // Record this round's candidates: the determinant with the bits of m flipped,
            // and v, its element up to the parity of m's bits.  Terms (FOR != SEL_DETS):
            // only determinants of the current hash batch.
            auto emit = [&](bool keep, const Key<KW> &m, double v) {
                Key<KW> x;
#pragma unroll
                for (int w = 0; w < KW; w++) x.w[w] = D.w[w] ^ m.w[w];
                if (FOR != SEL_DETS && S.nbatch > 1 && keep) {
                    Str<W> a, b;
                    split_key<W, KW>(x, n, a, b);
                    keep = det_batch<W>(a, b, S.nbatch) == S.batch;
                }
                const unsigned mask = __ballot_sync(0xffffffffu, keep);
                if (FILL && keep) {
                    const int64_t slot = pos + __popc(mask & lt);
                    store_key<KW>(S.out, slot, x);
                    if (FOR != SEL_DETS) {
                        const double hv = flip_sign(v, common_parity<KW>(PD, m));
                        if (FOR == SEL_SAMPLE) {
                            S.terms[slot] = f1 * hv;
                            S.terms2[slot] = f2 * hv * hv;
                        } else {
                            S.terms[slot] = hv * ci;
                        }
                        if (FOR != SEL_TERMS) S.mags[slot] = fabs(hv) * cmax;
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
                const int np = n * (n + 1) / 2;
                const double *own = nullptr, *other = nullptr;
                if (S.ma) {
                    const int64_t ua = __ldg(&S.ia[i]), ub = __ldg(&S.ib[i]);
                    own = spin ? S.mb + 2 * ub * np : S.ma + 2 * ua * np;
                    other = (spin ? S.ma + 2 * ua * np : S.mb + 2 * ub * np) + np;
                }
                for (int u0 = 0; u0 < units; u0 += 32) {
                    const int u = u0 + lane;
                    bool keep = false;
                    Key<KW> m{};
                    double v = 0.0;
                    if (u < units) {
                        const int x = u / nv;
                        const int p = L.occ[spin][x], r = L.vir[spin][u - x * nv];
                        set_bit(m, p + (spin ? beta : 0));
                        set_bit(m, r + (spin ? beta : 0));
                        if (own) {
                            const int pr = pair_idx(p, r);
                            v = flip_sign(__ldg(&own[pr]) + __ldg(&other[pr]), p < r);
                        } else {
                            const Str<W> &si = spin ? B : A;
                            Str<W> sj = si;
                            flip_bit(sj, p);
                            flip_bit(sj, r);
                            v = single_exc<W>(I, si, sj, spin ? A : B);
                            if (FILL) v = flip_sign(v, common_parity<KW>(PD, m));    // emit applies it once more
                        }
                        keep = passes(cut, v);
                    }
                    emit(keep, m, v);
                }
            }
            for (int u0 = 0; u0 < pairs; u0 += 32) {
                int v = u0 + lane;
                int e0 = 0, len = 0, holes = 0;
                if (v < pairs) {
                    int p, q;
                    const int64_t *off = S.ss_off;
                    const float *kf = S.ss_kf;
                    if (v < u_paa + u_pbb) {
                        const int spin = v < u_paa ? 0 : 1;
                        if (spin) v -= u_paa;
                        // pair rank v -> (x < y): y is the largest with y (y - 1) / 2 <= v
                        int y = (int)((1.0f + sqrtf(1.0f + 8.0f * (float)v)) * 0.5f);
                        while (y * (y - 1) / 2 > v) y--;
                        while ((y + 1) * y / 2 <= v) y++;
                        p = L.occ[spin][v - y * (y - 1) / 2];
                        q = L.occ[spin][y];
                        holes = spin ? 0x20000 : 0;
                    } else {
                        v -= u_paa + u_pbb;
                        const int x = v / nb;
                        p = L.occ[0][x];
                        q = L.occ[1][v - x * nb];
                        holes = 0x10000;
                        off = S.os_off;
                        kf = S.os_kf;
                    }
                    holes |= p | (q << 8);
                    const int64_t b = __ldg(&off[p * n + q]);
                    e0 = (int)b;                          // at most 128^4 / 2 entries
                    int lo = 0, hi = (int)(__ldg(&off[p * n + q + 1]) - b);
                    while (lo < hi) {                     // keys descend: first entry out of reach
                        const int mid = (lo + hi) >> 1;
                        if (__ldg(&kf[e0 + mid]) < cut.reach) hi = mid;
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
                const unsigned some = __ballot_sync(0xffffffffu, len > 0);
                __syncwarp();
                if (len > 0) {
                    const int at = __popc(some & lt);
                    L.first[at] = e0 - (incl - len);
                    L.holes[at] = holes;
                }
                __syncwarp();
                const int start = len > 0 ? incl - len : 0x40000000;
                int begun = 0;                            // lists that begin before this round
                for (int t0 = 0; t0 < total; t0 += 32) {
                    const int t = t0 + lane;
                    const unsigned rel = (unsigned)(start - t0);
                    const unsigned starts = __reduce_or_sync(0xffffffffu, rel < 32u ? 1u << rel : 0u);
                    const int src = begun + __popc(starts & le) - 1;
                    begun += __popc(starts);
                    bool keep = false;
                    Key<KW> m{};
                    double hv = 0.0;
                    if (t < total) {
                        const int h = L.holes[src], e = L.first[src] + t;
                        const bool opp = h & 0x10000;
                        const uint32_t rs = __ldg(opp ? &S.os_rs[e] : &S.ss_rs[e]);
                        hv = __ldg(opp ? &S.os_v[e] : &S.ss_v[e]);
                        const int o1 = h & 0x20000 ? beta : 0, o2 = h & 0x30000 ? beta : 0;   // key bits of the two spins
                        set_bit(m, (int)(rs & 0xFFFFu) + o1);
                        set_bit(m, (int)(rs >> 16) + o2);
                        bool free = true;                 // neither particle orbital is occupied
#pragma unroll
                        for (int w = 0; w < KW; w++) free = free && (m.w[w] & D.w[w]) == 0;
                        keep = free && passes(cut, hv);
                        set_bit(m, (h & 255) + o1);
                        set_bit(m, ((h >> 8) & 255) + o2);
                    }
                    emit(keep, m, hv);
                }
            }
        }
        if (!FILL && lane == 0) S.cnt[i] = (unsigned long long)pos;
    }
}

// count pass over S's determinants and the offsets of their candidates; returns the total
template <int W, int KW, bool TERMS>
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
    k_select<W, KW, false, TERMS ? SEL_TERMS : SEL_DETS><<<blocks, SEL_THREADS, 0, st>>>(S, I);
    KERNEL_CHECK();
    g_kernel_launches += 1;
    exclusive_scan<int64_t>(reinterpret_cast<const int64_t *>(cnt.p), off.p, n, tmp.p, st);
    int64_t total = 0;
    CUDA_TRY(cudaMemcpyAsync(&total, off.p + n, sizeof(int64_t), cudaMemcpyDeviceToHost, st));
    CUDA_TRY(cudaStreamSynchronize(st));
    return total;
}

template <int W, int KW, int FOR>
static void fill_candidates(shci_ctx *c, const SelArgs &S, const DevInts &I) {
    const int blocks = (int)std::min<int64_t>(ceil_div(S.n_det, SEL_THREADS / 32),
                                              (int64_t)c->n_sm * (2048 / SEL_THREADS));
    k_select<W, KW, true, FOR><<<blocks, SEL_THREADS, 0, c->st>>>(S, I);
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
static void select_w(shci_ctx *c, int k, const double *cd, double eps1, DevBuf<uint64_t> &result, int64_t &n_new,
                     bool tables) {
    cudaStream_t st = c->st;
    const int64_t n = c->n_det;
    SelArgs S = sel_args(c, eps1);
    S.k = k;
    S.c = cd;
    const DevInts I = dev_ints(c);
    MoveTables moves;
    tabulate_moves<W>(c, S, I, (double)n, moves, tables);
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
    fill_candidates<W, KW, SEL_DETS>(c, S, I);
    radix_sort<KW>(cand.p, nullptr, total, c->sw, st, KeyMask<W, KW>(c->n_orb).known(), RS_KEYS);
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
// run, adding up its terms one by one, took 27 ms for 1.8e8 terms and 18 ms
// for a sample of 5e7, nearly all of it the longest runs' chains of dependent
// loads; this form 4.8 and 5.5, with the FP64 pipe 66 and 81 % busy (the tree's
// additions, H_aa, the division) and HBM 52 and 33 %.  The order of every sum is fixed.
constexpr int RUN_CHUNK = 16;

template <int W, int KW, int MODE>
__global__ void __launch_bounds__(SEL_THREADS) k_run_reduce(RunArgs A, DevInts I) {
    constexpr int NS = RunSums<MODE>::N;
    constexpr int NW = SEL_THREADS / 32;
    __shared__ __align__(16) uint64_t qkey[NW][64 * KW];
    __shared__ double qsum[NW][64 * NS];
    __shared__ double ftab[NW][W == 1 ? 64 : SHCI_MAX_ORB];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const unsigned lt = (1u << lane) - 1u;
    uint64_t *qk = qkey[wib];
    double *qs = qsum[wib];
    double acc0 = 0.0, acc1 = 0.0;
    unsigned long long cnt = 0;
    int qn = 0;
    // H_aa of sorted runs: most of 32 consecutive ones share their beta string b
    // (its bits are the key's high ones), so the warp tabulates, once per b,
    // b's own energy and f_k = h_kk + sum_{l in b} J_kl; a run then adds f over
    // its alpha electrons and their pairs: 21 FP64 additions instead of 78 for
    // six electrons a spin.  Runs of a fourth string among the 32 sum in full.
    double *f = ftab[wib];
    Str<W> bcur{};
    double ecur = 0.0;
    bool have = false;
    auto diagonal = [&](bool need, const Str<W> &a, const Str<W> &b) {
        double e = 0.0;
        unsigned todo = __ballot_sync(0xffffffffu, need);
        for (int g = 0; todo != 0; g++) {
            if (g == 3) {
                if ((todo >> lane) & 1u) e = hii<W>(I, a, b);
                break;
            }
            Str<W> bg;
            bool cur = have, mine = (todo >> lane) & 1u;
#pragma unroll
            for (int k = 0; k < W; k++) {
                bg.w[k] = __shfl_sync(0xffffffffu, b.w[k], __ffs(todo) - 1);
                cur = cur && bg.w[k] == bcur.w[k];
                mine = mine && bg.w[k] == b.w[k];
            }
            if (!cur) {                                   // warp-uniform
                __syncwarp();
                double eb = 0.0;
                for (int k = lane; k < I.n; k += 32) {
                    const double hk = __ldg(&I.h[k * I.n + k]);
                    double v = hk;
                    for_bits_above<W>(bg, -1, [&](int l) { v += __ldg(&I.jdiag[k * I.n + l]); });
                    f[k] = v;
                    if (has_bit(bg, k)) {
                        eb += hk;
                        for_bits_above<W>(bg, k, [&](int l) { eb += __ldg(&I.jkdiag[k * I.n + l]); });
                    }
                }
#pragma unroll
                for (int o = 16; o >= 1; o >>= 1) eb += __shfl_xor_sync(0xffffffffu, eb, o);
                __syncwarp();
                bcur = bg;
                ecur = eb;
                have = true;
            }
            if (mine) {
                e = I.e_core + ecur;
                for_bits_above<W>(a, -1, [&](int k) {
                    e += f[k];
                    for_bits_above<W>(a, k, [&](int l) { e += __ldg(&I.jkdiag[k * I.n + l]); });
                });
            }
            todo &= ~__ballot_sync(0xffffffffu, mine);
        }
        return e;
    };
    auto finish = [&](int m) {                            // the first m (<= 32) queued runs
        Key<KW> x{};
        bool need = false;
        if (lane < m) {
            x = load_key<KW>(qk, lane);
            need = !in_sorted<KW>(A.vs, A.nv, x);
        }
        Str<W> a, b;
        split_key<W, KW>(x, I.n, a, b);
        const double haa = diagonal(need, a, b);
        if (need) {
            const double den = A.e_var - haa;
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
    };
    // RUN_CHUNK consecutive windows at a time: a warp's queued runs are neighbours
    const int64_t windows = (A.total + 31) >> 5, warps = (int64_t)gridDim.x * NW;
    const int64_t first = ((int64_t)blockIdx.x * SEL_THREADS + threadIdx.x) >> 5;
    for (int64_t step = 0;; step++) {
        const int64_t w = (step / RUN_CHUNK * warps + first) * RUN_CHUNK + step % RUN_CHUNK;
        if (w >= windows) break;
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
    constexpr int FOR = MODE == RUN_PT ? SEL_TERMS : (MODE == RUN_SAMPLE ? SEL_SAMPLE : SEL_MAGS);
    fill_candidates<W, KW, FOR>(c, S, I);
    radix_sort<KW>(T.cand.p, T.idx.p, total, c->sw, st, KeyMask<W, KW>(c->n_orb).known(), RS_POSITION);
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
                    int &nbatch_used, int64_t &candidates, bool tables) {
    SelArgs S = sel_args(c, eps2);
    S.c = cd;
    const DevInts I = dev_ints(c);
    MoveTables moves;
    tabulate_moves<W>(c, S, I, (double)c->n_det, moves, tables);
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

// Walker's alias table for p_i = |c_i| / sum (Eq. 10), built by Vose's
// two-list method: q_i = n p_i; the small column (q < 1) on top of its stack
// takes the large column g on top of the other as its alias, g keeps
// q_g + q_l - 1, and a g that falls below 1 goes onto the small stack.  Every
// step needs the rounded result of the one before it and no two can be
// exchanged, so this is one chain of n additions, and it runs on a host core.
// On the GPU 100,003 columns took one thread 43.4 ms (dependent loads), one
// warp that staged the columns in shared memory for one lane 10.3 ms (two
// dependent FP64 additions, a test and a branch per column), and the same in
// integers that give the additions' bits 12.8 to 14.9; the semistochastic
// energy of that space went from 61.5 ms with the last form to 50.7 with this.
static void alias_table(const double *c, int64_t n, double sum, double *prob, uint32_t *alias) {
    const double scale = (double)n / sum;
    std::vector<uint32_t> stack((size_t)n);              // the small columns
    int64_t ns = 0, nl = 0;
    for (int64_t i = 0; i < n; i++) {
        prob[i] = std::fabs(c[i]) * scale;
        alias[i] = (uint32_t)i;
        if (prob[i] < 1.0) ns++;
    }
    std::vector<uint32_t> large((size_t)(n - ns));
    ns = 0;
    for (int64_t i = 0; i < n; i++) {
        if (prob[i] < 1.0) stack[ns++] = (uint32_t)i;
        else large[nl++] = (uint32_t)i;
    }
    while (ns > 0 && nl > 0) {
        const uint32_t l = stack[--ns], g = large[--nl];
        alias[l] = g;                                    // prob[l] stays
        prob[g] = (prob[g] + prob[l]) - 1.0;
        if (prob[g] < 1.0) stack[ns++] = g;
        else nl++;
    }
    while (nl > 0) prob[large[--nl]] = 1.0;
    while (ns > 0) prob[stack[--ns]] = 1.0;              // rounding leftovers
}

// draw d: r = SplitMix64 output for the counter seed + (d + 1) * golden
// gamma; column = high 32 bits * n >> 32, uniform u = low 32 bits / 2^32;
// the column itself when u < prob[column], else its alias
__global__ void k_alias_draw(const double *__restrict__ prob, const uint32_t *__restrict__ alias, int64_t n,
                             uint64_t seed, int64_t n_draws, int64_t *__restrict__ out) {
    for (int64_t d = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; d < n_draws;
         d += (int64_t)gridDim.x * blockDim.x) {
        uint64_t z = seed + (uint64_t)(d + 1) * 0x9E3779B97F4A7C15ull;
        z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
        z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
        z ^= z >> 31;
        const int64_t col = (int64_t)(((z >> 32) * (uint64_t)n) >> 32);
        const double u = (double)(uint32_t)z * 0x1p-32;
        out[d] = u < prob[col] ? col : (int64_t)alias[col];
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
                              const uint64_t *__restrict__ dets, const int32_t *__restrict__ ia,
                              const int32_t *__restrict__ ib, const double *__restrict__ c, double csum,
                              uint64_t *__restrict__ sdets, int32_t *__restrict__ sia, int32_t *__restrict__ sib,
                              double *__restrict__ sc, double *__restrict__ f1, double *__restrict__ f2) {
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n_d; e += (int64_t)gridDim.x * blockDim.x) {
        if (e > 0 && sorted[e - 1] == sorted[e]) continue;
        int64_t f = e + 1;
        while (f < n_d && sorted[f] == sorted[e]) f++;
        const int64_t i = (int64_t)sorted[e], u = pos[e];
        const double w = (double)(f - e), p = fabs(c[i]) / csum;
#pragma unroll
        for (int k = 0; k < 2 * W; k++) sdets[u * 2 * W + k] = dets[i * 2 * W + k];
        sia[u] = ia[i];
        sib[u] = ib[i];
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
                          int n_samples, const int64_t *draws, double *out, int nbatch, const int *batch_of_sample,
                          bool tables) {
    cudaStream_t st = c->st;
    const int64_t n = c->n_det;
    const double csum = abs_sum(c, cd, n);
    if (!(csum > 0.0)) throw ShciError{SHCI_ERR_INVALID, "all coefficients are zero"};
    TermWork T;
    sorted_space<W, KW>(c, T.vs);
    const DevInts I = dev_ints(c);
    DevBuf<uint64_t> sorted, sdets;
    DevBuf<int64_t> flag, pos, tmp;
    DevBuf<int32_t> sia, sib;
    DevBuf<double> sc, f1, f2;
    sorted.alloc((size_t)n_d);
    flag.alloc((size_t)n_d + 1);
    pos.alloc((size_t)n_d + 1);
    tmp.alloc((size_t)scan_tmp_len(n_d + 1));
    sdets.alloc((size_t)n_d * 2 * W);
    sc.alloc((size_t)n_d);
    f1.alloc((size_t)n_d);
    f2.alloc((size_t)n_d);
    sia.alloc((size_t)n_d);
    sib.alloc((size_t)n_d);
    MoveTables moves;
    SelArgs S0 = sel_args(c, eps2);
    tabulate_moves<W>(c, S0, I, (double)std::min(n_d, n) * n_samples, moves, tables);
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
        k_sample_prep<W><<<gb, SEL_THREADS, 0, st>>>(sorted.p, n_d, pos.p, c->dets.p, c->ia.p, c->ib.p, cd, csum,
                                                     sdets.p, sia.p, sib.p, sc.p, f1.p, f2.p);
        KERNEL_CHECK();
        g_kernel_launches += 2;
        CUDA_TRY(cudaStreamSynchronize(st));
        SelArgs S = S0;
        S.ia = sia.p;
        S.ib = sib.p;
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
    pt2_samples_w<W, KW>(c, cd, e_var, eps2, eps2_d, n_d, n_samples, dd, res.data(), nbatch, batch_of_sample, tables)
    with_tables([&](bool tables) { DISPATCH_KEYS(c, CALL); });
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
    const double *cd = coef, *hc = coef;                 // on the device, on the host
    DevBuf<double> cbuf;
    std::vector<double> copy;
    if (mem == SHCI_MEM_HOST) {
        cbuf.alloc((size_t)n);
        CUDA_TRY(cudaMemcpyAsync(cbuf.p, coef, sizeof(double) * n, cudaMemcpyHostToDevice, st));
        cd = cbuf.p;
    } else {
        copy.resize((size_t)n);
        CUDA_TRY(cudaMemcpyAsync(copy.data(), coef, sizeof(double) * n, cudaMemcpyDeviceToHost, st));
        hc = copy.data();
    }
    const double csum = abs_sum(c, cd, n);               // waits for the stream: the copy is done
    if (!(csum > 0.0)) throw ShciError{SHCI_ERR_INVALID, "all coefficients are zero"};
    std::vector<double> hp((size_t)n);
    std::vector<uint32_t> ha((size_t)n);
    alias_table(hc, n, csum, hp.data(), ha.data());
    DevBuf<double> prob;
    DevBuf<uint32_t> alias;
    DevBuf<int64_t> obuf;
    prob.alloc((size_t)n);
    alias.alloc((size_t)n);
    CUDA_TRY(cudaMemcpyAsync(prob.p, hp.data(), sizeof(double) * n, cudaMemcpyHostToDevice, st));
    CUDA_TRY(cudaMemcpyAsync(alias.p, ha.data(), sizeof(uint32_t) * n, cudaMemcpyHostToDevice, st));
    if (n_draws == 0) {
        CUDA_TRY(cudaStreamSynchronize(st));
        return;
    }
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
#define CALL(W, KW) v = pt2_w<W, KW>(c, cd, e_var, eps2, nbatch, np, used, cands, tables)
    with_tables([&](bool tables) { DISPATCH_KEYS(c, CALL); });
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
                   double target, double &est, double &err, int &done, bool tables) {
    SelArgs S = sel_args(c, eps_psto);
    S.c = cd;
    S.nbatch = nbatch;
    const DevInts I = dev_ints(c);
    MoveTables moves;
    tabulate_moves<W>(c, S, I, (double)c->n_det * nbatch, moves, tables);
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
    psto_w<W, KW>(c, cd, e_var, eps2_psto, eps2_dtm, nbatch_psto, target, out->psto, out->psto_err, out->psto_batches, \
                  tables)
        with_tables([&](bool tables) { DISPATCH_KEYS(c, CALL); });
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

void select_dets(shci_ctx *c, int k, const double *coef, double eps1, int mem, int64_t *n_out,
                 const std::function<std::pair<uint64_t *, int64_t>(int64_t)> &place) {
    if (!c->built) throw ShciError{SHCI_ERR_STATE, "build the connectivity before selecting"};
    if (k < 1 || k > SHCI_MAX_K) throw ShciError{SHCI_ERR_INVALID, "k must be in [1, 8]"};
    if (!(eps1 > 0.0) || !std::isfinite(eps1)) throw ShciError{SHCI_ERR_INVALID, "eps1 must be positive and finite"};
    if (!coef || !n_out) throw ShciError{SHCI_ERR_INVALID, "null pointer"};
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
#define CALL(W, KW) select_w<W, KW>(c, k, cd, eps1, result, n_new, tables)
    with_tables([&](bool tables) { DISPATCH_KEYS(c, CALL); });
#undef CALL
    *n_out = n_new;
    const int KW = 2 * c->W;
    if (n_new > 0) {
        const std::pair<uint64_t *, int64_t> to = place(n_new);
        if (to.second > 0)
            CUDA_TRY(cudaMemcpyAsync(to.first, result.p, sizeof(uint64_t) * to.second * KW,
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
