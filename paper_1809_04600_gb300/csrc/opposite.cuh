// Opposite-spin double excitations (Sec. III, Algorithm 2) by bitmap words.
//
// Row (a, b) is connected to (k, kb) when k is an alpha single of a, kb a beta
// single of b, and (k, kb) is in V.  The beta indices of V's members with
// alpha string k are kept as a list of the nonzero 64-bit words of their
// bitmap; a beta string's singles as a dense bitmap.  One AND of a word of k's
// list with the same word of b's bitmap therefore screens up to 64 candidates
// and names the connected ones.  Strings are numbered by decreasing number of
// determinants, so that a group's members fill few words.
//
// A CTA takes rows of one alpha group a: the words of all of a's alpha singles,
// with each word's alpha part (pair index, sign) and first member, are staged
// once in shared memory for all its rows; a warp takes a row, a lane a word.
// The set bits go to a queue in shared memory and are evaluated 32 at a time:
// the bit's rank in k's word gives the member, its rank in b's bitmap the beta
// part (pair index, sign) tabulated per beta single, and the element is one
// table entry with a sign.
#pragma once
#include "enumerate.cuh"

namespace shci {

constexpr int OPP_ROWS = 32;                // rows of an item (a full build; the incremental update's have ENUM_NW)
constexpr int OPP_TILE = 512;               // words staged at a time
constexpr int OPP_SINGLES = ENUM_THREADS;   // alpha singles laid out at a time
constexpr int OPP_QCAP = 512 + 32;          // queued matches per warp

struct OppSmem {
    unsigned long long word[OPP_TILE];
    int2 info[OPP_TILE];                    // word index, position of the word's first member
    int ctx[OPP_TILE];                      // alpha part: pair index << 1 | sign
    int start[OPP_SINGLES + 1];             // first word of each single of this part
    int64_t first[OPP_SINGLES];             // its words' place in the list
    int pq[OPP_SINGLES];
    uint16_t queue[ENUM_NW][OPP_QCAP];      // word << 6 | bit
};

template <int MODE, int K>
struct OppRow {
    int64_t i, found, pos;
    const unsigned long long *sb;           // b's singles bitmap
    const int32_t *sp;                      // singles before each word, from b's first entry
    int qn;
    double ci;
    double acc[K > 0 ? K : 1];
};

template <int MODE, int K>
__device__ __forceinline__ void opp_flush(OppRow<MODE, K> &R, const EnumArgs &A, const DevInts &I, const OppSmem &S,
                                          const uint16_t *queue, int cnt) {
    const int lane = threadIdx.x & 31;
    bool on = lane < cnt;
    int32_t j = 0;
    double v = 0.0;
    if (on) {
        const int e = queue[lane], t = e >> 6, bit = e & 63;
        const unsigned long long below = (1ull << bit) - 1ull;
        const int2 w = S.info[t];
        j = __ldg(&A.ow_det[w.y + __popcll(S.word[t] & below)]);
        if (upper_only<MODE>(A) || MODE == ENUM_GRAD) on = (int64_t)j > R.i;
        if (!ModeOf<MODE>::count && on) {
            const uint32_t b = __ldg(&A.bs_info[__ldg(&R.sp[w.x]) + __popcll(__ldg(&R.sb[w.x]) & below)]);
            const int c = S.ctx[t], rs = (int)(b >> 1), pq = c >> 1, neg = (int)(b & 1u) + (c & 1);
            const int hi = pq > rs ? pq : rs, lo = pq > rs ? rs : pq;
            const int64_t slot = (int64_t)hi * (hi + 1) / 2 + lo;
            if (MODE == ENUM_GRAD) {
                const int rep = blockIdx.x % GRAD_REPLICAS;
                red_add(A.geri + rep * A.geri_len + slot, flip_sign(2.0 * R.ci * __ldg(&A.x[j]), neg));
            } else {
                v = flip_sign(__ldg(&I.eri[slot]), neg);
            }
        }
    }
    if (ModeOf<MODE>::count) {
        R.found += on ? 1 : 0;              // upper triangle only: the others count words
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
            const double2 c2 = __ldg(reinterpret_cast<const double2 *>(A.x) + j);
            R.acc[0] = fma(v, c2.x, R.acc[0]);
            R.acc[K - 1] = fma(v, c2.y, R.acc[K - 1]);
        } else {
#pragma unroll
            for (int q = 0; q < K; q++) R.acc[q] = fma(v, __ldg(&A.x[(int64_t)j * K + q]), R.acc[q]);
        }
    }
}

// the staged words [0, n) against one row
template <int MODE, int K>
__device__ __forceinline__ void opp_scan(OppRow<MODE, K> &R, const EnumArgs &A, const DevInts &I, const OppSmem &S,
                                         uint16_t *queue, int n) {
    const int lane = threadIdx.x & 31;
    for (int t0 = 0; t0 < n; t0 += 32) {
        const int t = t0 + lane;
        unsigned long long m = 0ull;
        if (t < n) m = S.word[t] & __ldg(&R.sb[S.info[t].x]);
        const int c = __popcll(m);
        if (ModeOf<MODE>::count && !upper_only<MODE>(A)) {
            R.found += c;
            continue;
        }
        if (!__any_sync(0xffffffffu, c > 0)) continue;
        int incl = c;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        // all 32 lanes at once, or 8 at a time when their bits could overflow the queue
        const int total = __shfl_sync(0xffffffffu, incl, 31);
        const int step = total <= 512 ? 32 : 8;
        for (int g = 0; g < 32; g += step) {
            const int before = g == 0 ? 0 : __shfl_sync(0xffffffffu, incl, g - 1);
            const int last = __shfl_sync(0xffffffffu, incl, g + step - 1);
            if (lane >= g && lane < g + step) {
                int at = R.qn + incl - c - before;
                unsigned long long x = m;
                while (x) {
                    const int b = __ffsll((long long)x) - 1;
                    x &= x - 1;
                    queue[at++] = (uint16_t)((t << 6) | b);
                }
            }
            R.qn += last - before;
            __syncwarp();
            int done = 0;
            for (; R.qn - done >= 32; done += 32) opp_flush<MODE, K>(R, A, I, S, queue + done, 32);
            if (done) {
                const int rest = R.qn - done;
                const uint16_t keep = lane < rest ? queue[done + lane] : 0;
                __syncwarp();
                if (lane < rest) queue[lane] = keep;
                R.qn = rest;
            }
            __syncwarp();
        }
    }
    // the queue names staged words: empty it before they are replaced
    if (R.qn > 0) {
        opp_flush<MODE, K>(R, A, I, S, queue, R.qn);
        R.qn = 0;
        __syncwarp();
    }
}

// CTAs per SM (shared memory allows five); the on-the-fly product keeps its
// accumulators in registers
template <int MODE, int K>
struct OppMinBlocks {
    static constexpr int value = MODE == ENUM_SIGMA && K > 4 ? 3 : 5;
};

template <int W, int MODE, int K>
__global__ void __launch_bounds__(ENUM_THREADS, OppMinBlocks<MODE, K>::value) k_opposite(EnumArgs A, DevInts I) {
    __shared__ OppSmem S;
    __shared__ int item_sh, members_sh;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint16_t *queue = S.queue[warp];
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
        const int end = A.item_end ? min(A.item_end[item], first + ENUM_NW)
                                   : (int)min((int64_t)first + OPP_ROWS, A.ga_off[a + 1] - g_beg);
        const Str<W> Aa = load_str<W>(A.astr, a);
        auto begin = [&](OppRow<MODE, K> &R, int r) {
            R.i = A.row_det[g_beg + r];
            const int64_t b = A.ib[R.i];
            R.sb = A.sbm + b * A.sb_words;
            R.sp = A.sbp + b * A.sb_words;
            R.found = 0;
            R.qn = 0;
#pragma unroll
            for (int q = 0; q < (K > 0 ? K : 1); q++) R.acc[q] = 0.0;
            if (ModeOf<MODE>::fill) R.pos = A.rowptr[R.i] + A.part_off[R.i];
            if (MODE == ENUM_GRAD) R.ci = A.x[R.i];
        };
        auto finish = [&](OppRow<MODE, K> &R) {
            if (ModeOf<MODE>::count) {
                int64_t f = R.found;
#pragma unroll
                for (int o = 16; o >= 1; o >>= 1) f += __shfl_xor_sync(0xffffffffu, f, o);
                if (lane == 0) A.cnt[R.i] = f;
            } else if (MODE == ENUM_SIGMA) {
                double s;
                const int q = warp_sum_many<(K > 0 ? K : 1)>(R.acc, s);
                constexpr int P = K <= 1 ? 1 : (K <= 2 ? 2 : (K <= 4 ? 4 : 8));
                if (q < K && (lane & (32 / P - 1)) == 0) A.y[R.i * K + q] += s;
            }
        };
        // stage words [w0, w0 + n) of the singles [s0, s0 + OPP_SINGLES)
        auto stage = [&](int w0, int n) {
            int members = 0;
            for (int e = threadIdx.x; e < n; e += ENUM_THREADS) {
                const int w = w0 + e;
                int lo = 0, hi = OPP_SINGLES;             // the last single that starts at or before w
                while (hi - lo > 1) {
                    const int mid = (lo + hi) >> 1;
                    if (S.start[mid] <= w) lo = mid;
                    else hi = mid;
                }
                const int64_t at = S.first[lo] + (w - S.start[lo]);
                S.word[e] = __ldg(&A.ow_word[at]);
                S.info[e] = __ldg(&A.ow_info[at]);
                S.ctx[e] = S.pq[lo];
                if (ModeOf<MODE>::count) members += __popcll(S.word[e]);
            }
            if (ModeOf<MODE>::count && members) atomicAdd(&members_sh, members);
        };
        // lay out the words of singles [s0, s0 + OPP_SINGLES); returns their number
        auto layout = [&](int64_t s0) {
            int len = 0;
            if (s0 + threadIdx.x < s_end) {
                const int k = A.as_idx[s0 + threadIdx.x];
                const int64_t f = A.ow_off[k];
                len = (int)(A.ow_off[k + 1] - f);
                S.first[threadIdx.x] = f;
                int pq = 0, neg = 0;
                if (!ModeOf<MODE>::count && len > 0) move_info<W>(Aa, load_str<W>(A.astr, k), pq, neg);
                S.pq[threadIdx.x] = (pq << 1) | (neg & 1);
            }
            int total;
            const int before = block_excl_scan<int>(len, &total);
            S.start[threadIdx.x] = before;
            if (threadIdx.x == 0) S.start[OPP_SINGLES] = total;
            __syncthreads();
            return total;
        };
        OppRow<MODE, K> R;
        int total = layout(s_beg);
        if (s_end - s_beg <= OPP_SINGLES && total <= OPP_TILE) {
            // everything staged once for all the item's rows
            if (threadIdx.x == 0) members_sh = 0;
            __syncthreads();
            stage(0, total);
            __syncthreads();
            for (int r = first + warp; r < end; r += ENUM_NW) {
                begin(R, r);
                opp_scan<MODE, K>(R, A, I, S, queue, total);
                finish(R);
                cand += lane == 0 ? members_sh : 0;
            }
            continue;
        }
        for (int r0 = first; r0 < end; r0 += ENUM_NW) {
            const int r = r0 + warp;
            const bool valid = r < end;
            if (valid) begin(R, r);
            for (int64_t s0 = s_beg; s0 < s_end; s0 += OPP_SINGLES) {
                if (s0 != s_beg || r0 != first) {
                    __syncthreads();
                    total = layout(s0);
                }
                for (int w0 = 0; w0 < total; w0 += OPP_TILE) {
                    const int n = min(OPP_TILE, total - w0);
                    __syncthreads();
                    if (threadIdx.x == 0) members_sh = 0;
                    __syncthreads();
                    stage(w0, n);
                    __syncthreads();
                    if (valid) {
                        opp_scan<MODE, K>(R, A, I, S, queue, n);
                        cand += lane == 0 ? members_sh : 0;
                    }
                }
            }
            if (valid) finish(R);
        }
    }
    if (ModeOf<MODE>::count && lane == 0 && cand) atomicAdd(A.cand, cand);
}

}  // namespace shci
