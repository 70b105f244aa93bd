// Device-wide primitives: exclusive scan and a stable LSD radix sort of
// multi-word uint64 keys with uint32 payloads.  Used by the helper-list build.
#pragma once
#include "common.cuh"

namespace shci {

constexpr int SCAN_THREADS = 256;
constexpr int SCAN_ITEMS = 8;
constexpr int SCAN_TILE = SCAN_THREADS * SCAN_ITEMS;

template <typename T>
__device__ __forceinline__ T warp_incl_scan(T v) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        T u = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += u;
    }
    return v;
}

// exclusive scan of one value per thread across the block; returns the prefix,
// *total receives the block total
template <typename T>
__device__ __forceinline__ T block_excl_scan(T v, T *total) {
    __shared__ T warp_sums[33];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    T inc = warp_incl_scan(v);
    if (lane == 31) warp_sums[wid] = inc;
    __syncthreads();
    if (wid == 0) {
        T s = lane < nw ? warp_sums[lane] : T(0);
        T si = warp_incl_scan(s);
        if (lane < nw) warp_sums[lane] = si - s;
        if (lane == nw - 1) warp_sums[32] = si;
    }
    __syncthreads();
    T res = warp_sums[wid] + inc - v;
    *total = warp_sums[32];
    __syncthreads();
    return res;
}

template <typename T>
__global__ void k_scan_reduce(const T *__restrict__ in, int64_t n, T *__restrict__ block_sums) {
    int64_t base = (int64_t)blockIdx.x * SCAN_TILE + (int64_t)threadIdx.x * SCAN_ITEMS;
    T s = 0;
#pragma unroll
    for (int k = 0; k < SCAN_ITEMS; k++)
        if (base + k < n) s += in[base + k];
    T tot;
    block_excl_scan<T>(s, &tot);
    if (threadIdx.x == 0) block_sums[blockIdx.x] = tot;
}

// in-place exclusive scan of nb block sums by one block; block_sums[nb] = total
template <typename T>
__global__ void k_scan_blocksums(T *block_sums, int64_t nb) {
    T carry = 0;
    for (int64_t base = 0; base < nb; base += blockDim.x) {
        int64_t i = base + threadIdx.x;
        T v = i < nb ? block_sums[i] : T(0);
        T tot;
        T ex = block_excl_scan<T>(v, &tot);
        if (i < nb) block_sums[i] = ex + carry;
        carry += tot;
    }
    if (threadIdx.x == 0) block_sums[nb] = carry;
}

// OWN_PREFIX: block_sums holds plain sums and each block adds up those before
// its own (few blocks); otherwise they are already scanned.
template <typename T, bool OWN_PREFIX>
__global__ void k_scan_apply(const T *__restrict__ in, int64_t n, const T *__restrict__ block_sums,
                             T *__restrict__ out) {
    int64_t base = (int64_t)blockIdx.x * SCAN_TILE + (int64_t)threadIdx.x * SCAN_ITEMS;
    T v[SCAN_ITEMS];
    T s = 0;
#pragma unroll
    for (int k = 0; k < SCAN_ITEMS; k++) {
        v[k] = base + k < n ? in[base + k] : T(0);
        s += v[k];
    }
    T before;
    if (OWN_PREFIX) {
        T part = 0;
        for (unsigned b = threadIdx.x; b < blockIdx.x; b += SCAN_THREADS) part += block_sums[b];
        block_excl_scan<T>(part, &before);
    } else {
        before = block_sums[blockIdx.x];
    }
    T tot;
    T ex = block_excl_scan<T>(s, &tot) + before;
#pragma unroll
    for (int k = 0; k < SCAN_ITEMS; k++) {
        if (base + k < n) out[base + k] = ex;
        ex += v[k];
    }
    if (blockIdx.x == gridDim.x - 1 && threadIdx.x == blockDim.x - 1) out[n] = before + tot;
}

// Up to this many blocks every block sums the totals before it itself (at most
// two loads per thread) instead of a launch of its own doing so: the short
// scans of the helper lists are bound by their launches.
constexpr int64_t SCAN_OWN_PREFIX = 2 * SCAN_THREADS;

// out[0..n] = exclusive scan of in[0..n), out[n] = total.  `tmp` needs
// ceil(n / SCAN_TILE) + 1 elements.  in and out may alias.
template <typename T>
inline void exclusive_scan(const T *in, T *out, int64_t n, T *tmp, cudaStream_t st) {
    if (n == 0) {
        CUDA_TRY(cudaMemsetAsync(out, 0, sizeof(T), st));
        return;
    }
    int64_t nb = ceil_div(n, SCAN_TILE);
    if (nb > 1) {
        k_scan_reduce<T><<<(unsigned)nb, SCAN_THREADS, 0, st>>>(in, n, tmp);
        g_kernel_launches += 1;
    }
    if (nb <= SCAN_OWN_PREFIX) {
        k_scan_apply<T, true><<<(unsigned)nb, SCAN_THREADS, 0, st>>>(in, n, tmp, out);
    } else {
        k_scan_blocksums<T><<<1, 1024, 0, st>>>(tmp, nb);
        k_scan_apply<T, false><<<(unsigned)nb, SCAN_THREADS, 0, st>>>(in, n, tmp, out);
        g_kernel_launches += 1;
    }
    KERNEL_CHECK();
    g_kernel_launches += 1;
}

inline int64_t scan_tmp_len(int64_t n) { return ceil_div(n, SCAN_TILE) + 1; }

// ---------------------------------------------------------------- radix sort

constexpr int RS_THREADS = 256;                    // one thread per digit value in the tile-wide steps
constexpr int RS_WARPS = RS_THREADS / 32;

// 32-element rounds per warp: a tile's keys and payloads are reordered in
// shared memory before they are written, so that a digit's elements leave as
// one run; as many as 64 registers hold (four blocks per SM).
template <int KW>
struct RsTile {
    static constexpr int ROUNDS = KW == 1 ? 8 : (KW == 2 ? 5 : 3);
    static constexpr int N = RS_THREADS * ROUNDS;
};

// OR and AND of every key word: one atomic per block and word (an atomic per
// thread took 275 us of a 1e6-key sort's 390, all of it serialised on one L2 line).
template <int KW>
__global__ void __launch_bounds__(RS_THREADS) k_key_or_and(const uint64_t *__restrict__ keys, int64_t n,
                                                          unsigned long long *orand) {
    unsigned long long o[KW], a[KW];
#pragma unroll
    for (int w = 0; w < KW; w++) { o[w] = 0; a[w] = ~0ull; }
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
#pragma unroll
        for (int w = 0; w < KW; w++) { uint64_t k = keys[i * KW + w]; o[w] |= k; a[w] &= k; }
    }
    __shared__ unsigned long long so[RS_WARPS][KW], sa[RS_WARPS][KW];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
    for (int w = 0; w < KW; w++) {
#pragma unroll
        for (int d = 16; d >= 1; d >>= 1) {
            o[w] |= __shfl_xor_sync(0xffffffffu, o[w], d);
            a[w] &= __shfl_xor_sync(0xffffffffu, a[w], d);
        }
        if (lane == 0) { so[wid][w] = o[w]; sa[wid][w] = a[w]; }
    }
    __syncthreads();
    if (threadIdx.x < KW) {
        const int w = threadIdx.x;
        for (int x = 1; x < RS_WARPS; x++) { so[0][w] |= so[x][w]; sa[0][w] &= sa[x][w]; }
        atomicOr(&orand[w], so[0][w]);
        atomicAnd(&orand[KW + w], sa[0][w]);
    }
}

template <int KW>
__global__ void __launch_bounds__(RS_THREADS) k_rs_hist(const uint64_t *__restrict__ keys, int64_t n, int word,
                                                       int shift, uint32_t *__restrict__ hist, int64_t n_tiles) {
    __shared__ uint32_t h[256];
    h[threadIdx.x] = 0;
    __syncthreads();
    const int64_t base = (int64_t)blockIdx.x * RsTile<KW>::N;
#pragma unroll
    for (int r = 0; r < RsTile<KW>::ROUNDS; r++) {
        const int64_t i = base + r * RS_THREADS + threadIdx.x;
        if (i < n) atomicAdd(&h[(keys[i * KW + word] >> shift) & 255u], 1u);
    }
    __syncthreads();
    hist[(int64_t)threadIdx.x * n_tiles + blockIdx.x] = h[threadIdx.x];
}

// One digit's stable scatter of a tile: ranks by warp-wide matching, the tile
// reordered by digit in shared memory, then written in that order (a warp
// writes runs of one digit's consecutive slots).  Bound by HBM and by the
// loads' latency between the block's steps: 12 rounds at 95 registers (two
// blocks per SM) took 2.05 ms for a pass over 1.8e8 one-word keys with
// payloads, 8 rounds at 64 registers with the digit offsets and payloads
// loaded ahead of their use 1.02 ms (4.2 TB/s).
// vin == nullptr: an element's payload is its position; vout == nullptr: keys
// alone.
template <int KW>
__global__ void __launch_bounds__(RS_THREADS, 4) k_rs_scatter(const uint64_t *__restrict__ kin,
                                                          const uint32_t *__restrict__ vin,
                                                          uint64_t *__restrict__ kout, uint32_t *__restrict__ vout,
                                                          int64_t n, int word, int shift,
                                                          const uint32_t *__restrict__ offs, int64_t n_tiles) {
    constexpr int ROUNDS = RsTile<KW>::ROUNDS, TILE = RsTile<KW>::N;
    __shared__ uint32_t wcnt[RS_WARPS][256];
    __shared__ uint32_t gbase[256];                 // a digit's first global slot minus its first slot in the tile
    __shared__ uint64_t skey[TILE * KW];
    __shared__ uint32_t sval[TILE];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    for (int d = lane; d < 256; d += 32) wcnt[w][d] = 0;
    __syncwarp();
    const int64_t tile0 = (int64_t)blockIdx.x * TILE;
    const int64_t base = tile0 + (int64_t)w * (32 * ROUNDS);
    uint64_t key[ROUNDS][KW];
    uint32_t rank[ROUNDS], val[ROUNDS];
#pragma unroll
    for (int r = 0; r < ROUNDS; r++) {
        const int64_t i = base + r * 32 + lane;
#pragma unroll
        for (int q = 0; q < KW; q++) key[r][q] = i < n ? kin[i * KW + q] : 0ull;
    }
    const uint32_t off = offs[(int64_t)threadIdx.x * n_tiles + blockIdx.x];
    const unsigned lt = (1u << lane) - 1u;
    auto digit = [&](const uint64_t *k) {
        uint64_t x = k[0];
#pragma unroll
        for (int q = 1; q < KW; q++) x = word == q ? k[q] : x;
        return (int)((x >> shift) & 255u);
    };
#pragma unroll
    for (int r = 0; r < ROUNDS; r++) {
        const bool valid = base + r * 32 + lane < n;
        const int d = valid ? digit(key[r]) : 256 + lane;
        const unsigned peers = __match_any_sync(0xffffffffu, d);
        const uint32_t before = valid ? wcnt[w][d] : 0u;
        __syncwarp();
        if (valid && (peers & lt) == 0) wcnt[w][d] = before + __popc(peers);
        __syncwarp();
        rank[r] = before + __popc(peers & lt);
    }
    if (vout) {
#pragma unroll
        for (int r = 0; r < ROUNDS; r++) {
            const int64_t i = base + r * 32 + lane;
            val[r] = (i < n && vin) ? vin[i] : (uint32_t)i;
        }
    }
    __syncthreads();
    // per digit: exclusive prefix over the warps; then over the digits
    {
        const int d = threadIdx.x;
        uint32_t run = 0;
#pragma unroll
        for (int x = 0; x < RS_WARPS; x++) {
            const uint32_t t = wcnt[x][d];
            wcnt[x][d] = run;
            run += t;
        }
        uint32_t total;
        const uint32_t start = block_excl_scan<uint32_t>(run, &total);
        gbase[d] = off - start;
#pragma unroll
        for (int x = 0; x < RS_WARPS; x++) wcnt[x][d] += start;
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < ROUNDS; r++) {
        if (base + r * 32 + lane < n) {
            const uint32_t pos = wcnt[w][digit(key[r])] + rank[r];
#pragma unroll
            for (int q = 0; q < KW; q++) skey[pos * KW + q] = key[r][q];
            if (vout) sval[pos] = val[r];
        }
    }
    __syncthreads();
    const int cnt = (int)min((int64_t)TILE, n - tile0);
    for (int e = threadIdx.x; e < cnt; e += RS_THREADS) {
        const uint64_t *k = skey + (int64_t)e * KW;
        const uint32_t pos = gbase[digit(k)] + (uint32_t)e;
#pragma unroll
        for (int q = 0; q < KW; q++) kout[(int64_t)pos * KW + q] = k[q];
        if (vout) vout[pos] = sval[e];
    }
}

// Workspace for sorting up to n elements with KW-word keys.
struct SortWork {
    DevBuf<uint64_t> keys_alt;
    DevBuf<uint32_t> vals_alt;
    DevBuf<uint32_t> hist;
    DevBuf<uint32_t> scan_tmp;
    DevBuf<unsigned long long> orand;
};

__global__ static void k_rs_iota(uint32_t *__restrict__ v, int64_t n) {
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x)
        v[e] = (uint32_t)e;
}

// What the sort does with vals: carries them, sets them to each key's original
// position (the first pass writes them, nothing is read), or has none (vals unused).
enum { RS_VALS = 0, RS_POSITION = 1, RS_KEYS = 2 };

// Stable sort of (keys[n][KW], vals[n]) in place (ping-pong through ws).
// Word 0 is the least significant.  Digits that are equal for every key are
// skipped: those outside `may_vary` (per key word, where the caller knows the
// bits its keys can differ in), or those found by an OR/AND reduction over the
// keys and a read-back (may_vary == nullptr).
template <int KW>
inline void radix_sort(uint64_t *keys, uint32_t *vals, int64_t n, SortWork &ws, cudaStream_t st,
                       const uint64_t *may_vary = nullptr, int payload = RS_VALS) {
    if (n <= 1) {
        if (payload == RS_POSITION && n == 1) CUDA_TRY(cudaMemsetAsync(vals, 0, sizeof(uint32_t), st));
        return;
    }
    if (n > 0xFFFFFFFFll) throw ShciError{SHCI_ERR_INVALID, "radix_sort: too many elements"};
    int64_t n_tiles = ceil_div(n, RsTile<KW>::N);
    ws.keys_alt.alloc((size_t)n * KW);
    if (payload != RS_KEYS) ws.vals_alt.alloc((size_t)n);
    ws.hist.alloc((size_t)(256 * n_tiles + 1));
    ws.scan_tmp.alloc((size_t)scan_tmp_len(256 * n_tiles));
    uint64_t varying[KW];
    if (may_vary) {
        for (int w = 0; w < KW; w++) varying[w] = may_vary[w];
    } else {
        ws.orand.alloc(2 * KW);
        CUDA_TRY(cudaMemsetAsync(ws.orand.p, 0, sizeof(unsigned long long) * KW, st));
        CUDA_TRY(cudaMemsetAsync(ws.orand.p + KW, 0xFF, sizeof(unsigned long long) * KW, st));
        k_key_or_and<KW><<<(unsigned)std::min<int64_t>(ceil_div(n, RS_THREADS), 1024), RS_THREADS, 0, st>>>(keys, n,
                                                                                                          ws.orand.p);
        KERNEL_CHECK();
        g_kernel_launches += 1;
        unsigned long long oa[2 * KW];
        CUDA_TRY(cudaMemcpyAsync(oa, ws.orand.p, sizeof(oa), cudaMemcpyDeviceToHost, st));
        CUDA_TRY(cudaStreamSynchronize(st));
        for (int w = 0; w < KW; w++) varying[w] = oa[w] ^ oa[KW + w];
    }
    uint64_t *ka = keys, *kb = ws.keys_alt.p;
    uint32_t *va = payload == RS_KEYS ? nullptr : vals, *vb = payload == RS_KEYS ? nullptr : ws.vals_alt.p;
    bool first = true;
    for (int w = 0; w < KW; w++) {
        for (int shift = 0; shift < 64; shift += 8) {
            if (((varying[w] >> shift) & 255u) == 0) continue;
            k_rs_hist<KW><<<(unsigned)n_tiles, RS_THREADS, 0, st>>>(ka, n, w, shift, ws.hist.p, n_tiles);
            exclusive_scan<uint32_t>(ws.hist.p, ws.hist.p, 256 * n_tiles, ws.scan_tmp.p, st);
            k_rs_scatter<KW><<<(unsigned)n_tiles, RS_THREADS, 0, st>>>(
                ka, first && payload == RS_POSITION ? nullptr : va, kb, vb, n, w, shift, ws.hist.p, n_tiles);
            KERNEL_CHECK();
            g_kernel_launches += 2;
            first = false;
            std::swap(ka, kb);
            std::swap(va, vb);
        }
    }
    if (first && payload == RS_POSITION) {           // nothing to sort by
        k_rs_iota<<<(unsigned)std::min<int64_t>(ceil_div(n, RS_THREADS), 1024), RS_THREADS, 0, st>>>(vals, n);
        KERNEL_CHECK();
        g_kernel_launches += 1;
    }
    if (ka != keys) {
        CUDA_TRY(cudaMemcpyAsync(keys, ka, sizeof(uint64_t) * n * KW, cudaMemcpyDeviceToDevice, st));
        if (va) CUDA_TRY(cudaMemcpyAsync(vals, va, sizeof(uint32_t) * n, cudaMemcpyDeviceToDevice, st));
    }
}

}  // namespace shci
