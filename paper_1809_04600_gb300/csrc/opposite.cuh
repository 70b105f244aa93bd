// Opposite-spin double excitations (Sec. III, Algorithm 2) by bit masks over
// the alpha singles.
//
// Row (a, b) is connected to (k, kb) when k is an alpha single of a, kb a beta
// single of b, and (k, kb) is in V.  For 32 of a's singles k at a time, a CTA
// fills a table in shared memory over beta strings: M[kb] has bit s when
// (k_s, kb) is in V.  All rows of the group then look up their beta singles, a
// lane each: one word answers for 32 pairs, and every set bit is a connected
// pair.  (Of 1e6 selected determinants of 24 orbitals, a row has 91 x 91 pairs
// of singles, 1000 of them in V, while its alpha singles' groups have 28,000
// members: screening those 64 at a time by bitmaps over beta strings, 3,450
// words a row, took 21.6 ms to write H and 4.9 ms to count it; lookups pair by
// pair 51 and 18; this form 12.7 and 2.4.)  The bits go to a queue in
// shared memory and are evaluated 32 at a time: the pair's place among V's
// determinants by rank in the occupancy bitmap, the element from one entry of
// the integrals with the pair index and sign of the alpha single (once per
// group) and of the beta single (tabulated).
//
// Larger beta spaces take several tables, each over a range of OPP_RANGE
// strings.  A table pays where many rows share it and its singles are many:
// clearing it and reading the singles' members is one cost for all rows of the
// item.  Where that costs more than it saves (few alpha singles, or few rows,
// beside many members and several tables) the rows look their pairs of singles
// up in the occupancy bitmap one by one.  300,007 determinants over 3 alpha and
// 134,596 beta strings: product 78.9 ms by tables, 23.8 by lookups, 45.0 by the
// choice per alpha single in enumerate.cuh; count 66.4, 12.7 and 25.6.
#pragma once
#include "enumerate.cuh"
#include "prims.cuh"

namespace shci {

constexpr int OPP_ROWS = 1024;              // rows of an item, at most
constexpr int OPP_RANGE = 24576;            // beta strings per table: 96 KB, two CTAs per SM

// Rows of an item for n determinants: filling the tables takes about as long as
// scanning some 30 rows, but a small space has too few groups to spread over
// the GPU in large items.  About 16 items per SM, of 8 to 128 rows; spaces that
// have 64 items per SM of those take larger ones, because the groups, and with
// them the members read for a table, grow with V (76 orbitals, 31,500 strings a
// spin, 5e7 determinants: count pass with the same-spin ones 2.35 s at 128 rows,
// 1.06 at 1024; product 4.92 and 3.87; 1e7: 110 and 89 ms, 426 and 380).
inline int opp_item_rows(int64_t n, int n_sm) {
    int rows = 8;
    while (rows < OPP_ROWS && (int64_t)rows * (rows < 128 ? 32 : 128) * n_sm <= n) rows *= 2;
    return rows;
}

// the words of the table for U beta strings
__host__ __device__ inline int opp_table(int64_t U) { return (int)(U < OPP_RANGE ? U : OPP_RANGE); }

// dynamic shared memory: the table, then the rows' places
__host__ __device__ inline int opp_places(int64_t U) { return (opp_table(U) + 1) & ~1; }      // their word offset
inline size_t opp_smem(int rows, int64_t U) { return sizeof(uint32_t) * opp_places(U) + sizeof(int64_t) * rows; }
constexpr size_t OPP_SMEM_MAX = sizeof(int64_t) * OPP_ROWS + sizeof(uint32_t) * OPP_RANGE;

// Look the pairs of ns alpha singles up one by one instead of filling tables?
// rows x beta singles x ns lookups against, for each table, the singles' members
// and a word per row and beta single, and clearing all U words.  A cleared word
// takes 0.3 ps, the others 3 to 5 ps (the bitmap in L2 or not): the lookups are
// counted double, the cleared words as a sixteenth.  A row's lookups are one
// warp's, so fewer rows than warps take as long as that many.
__host__ __device__ inline int64_t opp_table_cost(int64_t rows, int64_t beta_singles, int64_t members, int64_t U) {
    return U / 16 + (U + OPP_RANGE - 1) / OPP_RANGE * (members + rows * beta_singles);
}
__host__ __device__ inline int64_t opp_lookup_cost(int64_t rows, int64_t beta_singles, int ns) {
    return 2 * (rows > ENUM_NW ? rows : ENUM_NW) * beta_singles * ns;
}
__host__ __device__ inline bool opp_direct(int64_t rows, int64_t beta_singles, int ns, int64_t members, int64_t U) {
    return opp_lookup_cost(rows, beta_singles, ns) < opp_table_cost(rows, beta_singles, members, U);
}

struct OppSmem {
    uint32_t queue[ENUM_NW][64];            // beta single << 5 | alpha single
    int64_t occ[32];                        // the singles' rows of the bitmap
    int pq[32];                             // alpha part: pair index << 1 | sign
    int members;                            // of the singles' groups
};

template <int MODE, int K>
struct OppRow {
    int64_t i, pos, sb;                     // determinant, next slot, first beta single
    int place;                              // its place in the group lists
    int found, qn;
    double ci;
    double acc[K > 0 ? K : 1];
};

template <int MODE, int K>
__device__ __forceinline__ void opp_flush(OppRow<MODE, K> &R, const EnumArgs &A, const DevInts &I, const OppSmem &S,
                                          const uint32_t *queue, int cnt) {
    const int lane = threadIdx.x & 31;
    bool on = lane < cnt;
    int32_t j = 0;
    double v = 0.0;
    if (on) {
        const uint32_t e = queue[lane];
        const int s = (int)(e & 31u);
        const int64_t t = R.sb + (e >> 5);
        const int2 b = __ldg(&A.bs_pair[t]);
        const OccCell o = occ_load(A.occ + S.occ[s], b.x >> 6);
        const int place = o.place + __popcll(o.bits & ((1ull << (b.x & 63)) - 1ull));
        if (MODE == ENUM_GRAD) on = place > R.place;      // each pair once
        else if (MODE != ENUM_SIGMA) j = __ldg(&A.ow_det[place]);
        else j = place;
        if (upper_only<MODE>(A)) on = (int64_t)j > R.i;
        if (MODE == ENUM_GRAD) j = place;
        if (!ModeOf<MODE>::count && on) {
            const int rs = b.y >> 1, pq = S.pq[s] >> 1, neg = (b.y & 1) + (S.pq[s] & 1);
            const int hi = pq > rs ? pq : rs, lo = pq > rs ? rs : pq;
            const int64_t slot = (int64_t)hi * (hi + 1) / 2 + lo;
            if (MODE == ENUM_GRAD) {
                const int rep = blockIdx.x % GRAD_REPLICAS;
                red_add(A.geri + rep * A.geri_len + slot, flip_sign(2.0 * R.ci * __ldg(&A.x_grouped[j]), neg));
            } else {
                v = flip_sign(__ldg(&I.eri[slot]), neg);
            }
        }
    }
    if (ModeOf<MODE>::count) {
        R.found += on ? 1 : 0;              // upper triangle only: the others count bits
        return;
    }
    if (ModeOf<MODE>::fill) {
        int64_t pos = R.pos + lane;
        int n = cnt;
        if (upper_only<MODE>(A)) {
            const unsigned m = __ballot_sync(0xffffffffu, on);
            pos = R.pos + __popc(m & ((1u << lane) - 1u));
            n = __popc(m);
        }
        if (on) {
            A.col[pos] = j;
            A.val[pos] = v;
        }
        R.pos += n;
    } else if (MODE == ENUM_SIGMA && on) {
        if (K == 2) {
            const double2 c2 = __ldg(reinterpret_cast<const double2 *>(A.x_grouped) + j);
            R.acc[0] = fma(v, c2.x, R.acc[0]);
            R.acc[K - 1] = fma(v, c2.y, R.acc[K - 1]);
        } else {
#pragma unroll
            for (int q = 0; q < K; q++) R.acc[q] = fma(v, __ldg(&A.x_grouped[(int64_t)j * K + q]), R.acc[q]);
        }
    }
}

// the first 32 queued pairs, and the rest moved up
template <int MODE, int K>
__device__ __forceinline__ void opp_flush_full(OppRow<MODE, K> &R, const EnumArgs &A, const DevInts &I, const OppSmem &S,
                                               uint32_t *queue) {
    const int lane = threadIdx.x & 31;
    opp_flush<MODE, K>(R, A, I, S, queue, 32);
    R.qn -= 32;
    const uint32_t keep = lane < R.qn ? queue[32 + lane] : 0u;
    __syncwarp();
    if (lane < R.qn) queue[lane] = keep;
    __syncwarp();
}

// one row's beta singles against the table of strings [k0, k0 + range), or (only
// with CHOICE: range 0) against the ns singles' rows of the bitmap
template <int MODE, int K, bool CHOICE>
__device__ __forceinline__ void opp_scan(OppRow<MODE, K> &R, const EnumArgs &A, const DevInts &I, const OppSmem &S,
                                         const uint32_t *M, uint32_t *queue, int n, int ns, int k0, int range) {
    const int lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u;
    for (int t0 = 0; t0 < n; t0 += 32) {
        const int t = t0 + lane;
        unsigned m = 0u;
        if (t < n) {
            const unsigned kb = (unsigned)(__ldg(&A.bs_pair[R.sb + t].x) - k0);
            if (kb < (unsigned)range) {
                m = M[kb];
            } else if (CHOICE && range == 0) {
#pragma unroll 4
                for (int s = 0; s < ns; s++)
                    m |= (unsigned)((__ldg(&A.occ[S.occ[s] + (kb >> 6)].bits) >> (kb & 63)) & 1ull) << s;
            }
        }
        if (ModeOf<MODE>::count && !upper_only<MODE>(A)) {
            R.found += __popc(m);
            continue;
        }
        // Rows of the upper triangle: the set bits lane by lane, 32 at a time, so that a
        // row's pairs of one beta string stand together.  Such determinants are near
        // one another in V as a selection orders it, and the product scatters into
        // them (24 orbitals, 1.2e5 determinants, one vector: 351 us by scans of the
        // groups, 328 in this order; 60,017: a bit at a time of every lane is as slow
        // as a random order, 236 us, this 217, ascending determinants 216).
        if (upper_only<MODE>(A) && !ModeOf<MODE>::count) {
            const int own = __popc(m), incl = warp_incl_scan(own), total = __shfl_sync(0xffffffffu, incl, 31);
            for (int q0 = 0; q0 < total; q0 += 32) {
                const int slot = q0 + lane;
                int q = 0;                                // the lane that holds bit `slot`: the first with incl > slot
#pragma unroll
                for (int step = 16; step >= 1; step >>= 1) {
                    const int v = __shfl_sync(0xffffffffu, incl, q + step - 1);
                    if (v <= slot) q += step;
                }
                q = min(q, 31);
                unsigned w = __shfl_sync(0xffffffffu, m, q);
                int nth = slot - __shfl_sync(0xffffffffu, incl - own, q), bit = 0;
#pragma unroll
                for (int half = 16; half >= 1; half >>= 1) {          // its nth set bit
                    const int c = __popc(w & ((1u << half) - 1u));
                    if (nth >= c) {
                        nth -= c;
                        w >>= half;
                        bit += half;
                    }
                }
                if (slot < total) queue[R.qn + lane] = ((uint32_t)(t0 + q) << 5) | (uint32_t)bit;
                R.qn += min(32, total - q0);
                __syncwarp();
                if (R.qn >= 32) opp_flush_full<MODE, K>(R, A, I, S, queue);
            }
            continue;
        }
        // a round takes one bit of every lane that has some left
        for (unsigned some = __ballot_sync(0xffffffffu, m != 0u); some; some = __ballot_sync(0xffffffffu, m != 0u)) {
            if (m) {
                queue[R.qn + __popc(some & lt)] = ((uint32_t)t << 5) | (uint32_t)(__ffs(m) - 1);
                m &= m - 1u;
            }
            R.qn += __popc(some);
            __syncwarp();
            if (R.qn >= 32) opp_flush_full<MODE, K>(R, A, I, S, queue);
        }
    }
    // the queue names this table's singles: empty it before they are replaced
    if (R.qn > 0) {
        opp_flush<MODE, K>(R, A, I, S, queue, R.qn);
        R.qn = 0;
        __syncwarp();
    }
}

// with the choice, as many CTAs per SM as the kernels without it reach by themselves
template <int MODE, int K, bool CHOICE>
struct OppMinBlocks {
    static constexpr int value = !CHOICE ? (MODE == ENUM_SIGMA && K > 4 ? 2 : 3)
                                         : (ModeOf<MODE>::count ? 6 : (MODE != ENUM_SIGMA || K <= 2 ? 5 : (K <= 5 ? 4 : 3)));
};

// CHOICE: tables or lookups for each 32 alpha singles (opp_direct), and nothing
// where they have no members.  Without it tables always: the choice costs 5 % of
// a product where it is never taken (24 orbitals, 60,017 determinants: 0.72 to
// 0.77 ms), so it is taken only where it saves a fifth of the whole pass
// (k_opp_costs).
template <int W, int MODE, int K, bool CHOICE>
__global__ void __launch_bounds__(ENUM_THREADS, OppMinBlocks<MODE, K, CHOICE>::value) k_opposite(EnumArgs A, DevInts I) {
    extern __shared__ uint32_t M[];         // [opp_table(Ub)], then [opp_rows] places
    __shared__ OppSmem S;
    __shared__ int item_sh;
    // fill: each row's next slot; count: pairs so far
    int64_t *const pos = reinterpret_cast<int64_t *>(M + opp_places(A.n_beta_str));
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t *queue = S.queue[warp];
    unsigned long long cand = 0;
    while (true) {
        __syncthreads();
        if (threadIdx.x == 0) item_sh = atomicAdd(A.work_counter, 1);
        __syncthreads();
        const int64_t item = item_sh;
        if (item >= A.n_items) break;
        const int a = A.item_group[item];
        const int64_t g_beg = A.ga_off[a], s_beg = A.as_off[a], s_end = A.as_off[a + 1];
        const int first = A.item_first[item];
        const int last = A.item_end ? A.item_end[item] : (int)(A.ga_off[a + 1] - g_beg);
        const int rows = min(last - first, A.opp_rows);
        const Str<W> Aa = load_str<W>(A.astr, a);
        if (ModeOf<MODE>::fill || ModeOf<MODE>::count) {
            for (int r = threadIdx.x; r < rows; r += ENUM_THREADS) {
                const int64_t i = A.row_det[g_beg + first + r];
                pos[r] = ModeOf<MODE>::fill ? A.rowptr[i] + A.part_off[i] : 0;
            }
        }
        for (int64_t s0 = s_beg; s0 < s_end; s0 += 32) {
            const int ns = (int)min((int64_t)32, s_end - s0);
            __syncthreads();
            if (threadIdx.x < ns) {
                const int k = A.as_idx[s0 + threadIdx.x];
                S.occ[threadIdx.x] = (int64_t)k * A.occ_words;
                int pq = 0, neg = 0;
                if (!ModeOf<MODE>::count) move_info<W>(Aa, load_str<W>(A.astr, k), pq, neg);
                S.pq[threadIdx.x] = (pq << 1) | (neg & 1);
            }
            bool direct = false;
            if constexpr (CHOICE) {
                if (warp == 0) {
                    const int k = lane < ns ? A.as_idx[s0 + lane] : -1;
                    const int len = __reduce_add_sync(0xffffffffu, k < 0 ? 0 : (int)(A.ow_off[k + 1] - A.ow_off[k]));
                    if (lane == 0) S.members = len;
                }
                __syncthreads();
                const int members = S.members;
                if (members == 0) continue;               // the same for all threads
                direct = opp_direct(rows, A.opp_beta_singles, ns, members, A.n_beta_str);
            }
            // looked up: one round without a table
            for (int64_t k0 = 0; k0 < (CHOICE && direct ? 1 : A.n_beta_str); k0 += OPP_RANGE) {
                const int range = CHOICE && direct ? 0 : (int)min((int64_t)OPP_RANGE, A.n_beta_str - k0);
                for (int e = threadIdx.x; e < range; e += ENUM_THREADS) M[e] = 0u;
                __syncthreads();
                // a warp per single: its members' bits
                for (int s = warp; s < (CHOICE && direct ? 0 : ns); s += ENUM_NW) {
                    const int k = A.as_idx[s0 + s];
                    const int64_t end = A.ow_off[k + 1];
                    for (int64_t p = A.ow_off[k] + lane; p < end; p += 32) {
                        const unsigned kb = (unsigned)(__ldg(&A.ow_ib[p]) - (int)k0);
                        if (kb < (unsigned)range) atomicOr(&M[kb], 1u << s);
                    }
                }
                __syncthreads();
                for (int r = warp; r < rows; r += ENUM_NW) {
                    OppRow<MODE, K> R;
                    R.i = A.row_det[g_beg + first + r];
                    R.place = (int)(g_beg + first + r);
                    const int b = A.ib[R.i];
                    R.sb = A.bs_off[b];
                    const int n = (int)(A.bs_off[b + 1] - R.sb);
                    R.pos = ModeOf<MODE>::fill ? pos[r] : 0;
                    R.found = 0;
                    R.qn = 0;
#pragma unroll
                    for (int q = 0; q < (K > 0 ? K : 1); q++) R.acc[q] = 0.0;
                    if (MODE == ENUM_GRAD) R.ci = A.x_grouped[R.place];
                    opp_scan<MODE, K, CHOICE>(R, A, I, S, M, queue, n, ns, (int)k0, range);
                    if (ModeOf<MODE>::count) {
                        const int f = __reduce_add_sync(0xffffffffu, R.found);
                        if (lane == 0) pos[r] += f;
                        if (k0 == 0) cand += lane == 0 ? (unsigned long long)n * ns : 0ull;
                    } else if (ModeOf<MODE>::fill) {
                        if (lane == 0) pos[r] = R.pos;
                    } else if (MODE == ENUM_SIGMA) {
                        double s;
                        const int q = warp_sum_many<(K > 0 ? K : 1)>(R.acc, s);
                        constexpr int P = K <= 1 ? 1 : (K <= 2 ? 2 : (K <= 4 ? 4 : 8));
                        if (q < K && (lane & (32 / P - 1)) == 0) A.y[R.i * K + q] += s;
                    }
                }
                __syncthreads();
            }
        }
        if (ModeOf<MODE>::count) {
            __syncthreads();
            for (int r = threadIdx.x; r < rows; r += ENUM_THREADS)
                A.cnt[A.row_det[g_beg + first + r]] = pos[r];
        }
    }
    if (ModeOf<MODE>::count && lane == 0 && cand) atomicAdd(A.cand, cand);
}

// Costs of the pass over all items, in opp_direct's units: sums[0] with tables
// only, sums[1] with the choice.  A warp per group.
static __global__ void k_opp_costs(const int64_t *__restrict__ off, int64_t n_groups, int rows_max,
                                   const int64_t *__restrict__ as_off, const int32_t *__restrict__ as_idx,
                                   int64_t beta_singles, int64_t U, unsigned long long *__restrict__ sums) {
    const int lane = threadIdx.x & 31;
    unsigned long long table = 0, least = 0;
    for (int64_t a = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; a < n_groups;
         a += ((int64_t)gridDim.x * blockDim.x) >> 5) {
        const int64_t g = off[a + 1] - off[a], items = (g + rows_max - 1) / rows_max;
        const int64_t rows = (g + items - 1) / items, s_end = as_off[a + 1];
        for (int64_t s0 = as_off[a]; s0 < s_end; s0 += 32) {
            const int ns = (int)min((int64_t)32, s_end - s0);
            const int k = lane < ns ? as_idx[s0 + lane] : -1;
            const int members = __reduce_add_sync(0xffffffffu, k < 0 ? 0 : (int)(off[k + 1] - off[k]));
            const int64_t t = opp_table_cost(rows, beta_singles, members, U), d = opp_lookup_cost(rows, beta_singles, ns);
            table += (unsigned long long)(items * t);
            least += (unsigned long long)(items * (d < t ? d : t));
        }
    }
    if (lane == 0 && table) {
        atomicAdd(&sums[0], table);
        atomicAdd(&sums[1], least);
    }
}

}  // namespace shci
