// Device-wide exclusive scan and a stable LSD radix sort (the counting sorts
// that keep the store cell-ordered, Sections 2.1 and 2.3.3).
#include "kernels.h"

namespace cube {

namespace {

constexpr int SCAN_T = 1024;           // threads per scan block
constexpr int SCAN_ITEMS = 4;          // items per thread
constexpr int SCAN_TILE = SCAN_T * SCAN_ITEMS;

// SCAN_ITEMS = 4 consecutive items of one thread, as one 16-byte load when
// the array is 16-byte aligned and the four items exist
__device__ __forceinline__ void load4(const unsigned* __restrict__ in, int64_t base, int64_t n, bool vec,
                                      unsigned* v) {
    if (vec && base + 3 < n) {
        const uint4 q = *reinterpret_cast<const uint4*>(in + base);
        v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w;
    } else {
#pragma unroll
        for (int i = 0; i < SCAN_ITEMS; ++i) v[i] = base + i < n ? in[base + i] : 0u;
    }
}

// (member blockIdx.y of a batch: its arrays are `stride` bytes further on)
__global__ void k_scan_reduce(const unsigned* __restrict__ in, int64_t n, unsigned* __restrict__ bsum, bool vec,
                              Batch bt) {
    __shared__ unsigned sw[32];
    chain_wait();
    if (bt.ms && !bt.ms[blockIdx.y].active) return;
    const int m = slot_member(bt, blockIdx.y);
    in = moved(in, m * bt.stride);
    bsum = moved(bsum, m * bt.stride);
    unsigned v[SCAN_ITEMS];
    load4(in, (int64_t)blockIdx.x * SCAN_TILE + (int64_t)threadIdx.x * SCAN_ITEMS, n, vec, v);
    const unsigned s = v[0] + v[1] + v[2] + v[3];
    unsigned tot;
    block_inclusive_scan(s, sw, &tot);
    if (threadIdx.x == 0) bsum[blockIdx.x] = tot;
}

// exclusive scan of the block sums in place (single block, any count)
__global__ void k_scan_bsums(unsigned* bsum, int nb, unsigned* total_out, Batch bt) {
    __shared__ unsigned sw[32];
    chain_wait();
    if (bt.ms && !bt.ms[blockIdx.x].active) return;
    const int m = slot_member(bt, blockIdx.x);
    bsum = moved(bsum, m * bt.stride);
    total_out = moved(total_out, m * bt.stride);
    unsigned carry = 0;
    for (int base = 0; base < nb; base += SCAN_T) {
        int i = base + threadIdx.x;
        unsigned v = i < nb ? bsum[i] : 0u;
        unsigned tot;
        unsigned inc = block_inclusive_scan(v, sw, &tot);
        if (i < nb) bsum[i] = carry + inc - v;
        carry += tot;
    }
    if (threadIdx.x == 0 && total_out) *total_out = carry;
}

// SUMS: bsum holds the tiles' sums, not their scan: a block adds the ones
// before its own, and the last one writes the total to out[n]
template <bool SUMS>
__global__ void k_scan_down(const unsigned* in, int64_t n, const unsigned* __restrict__ bsum, unsigned* out,
                            bool vec, Batch bt) {
    __shared__ unsigned sw[32];
    chain_wait();
    if (bt.ms && !bt.ms[blockIdx.y].active) return;
    const int m = slot_member(bt, blockIdx.y);
    in = moved(in, m * bt.stride);
    bsum = moved(bsum, m * bt.stride);
    out = moved(out, m * bt.stride);
    const int64_t base = (int64_t)blockIdx.x * SCAN_TILE + (int64_t)threadIdx.x * SCAN_ITEMS;
    unsigned v[SCAN_ITEMS];
    load4(in, base, n, vec, v);
    const unsigned s = v[0] + v[1] + v[2] + v[3];
    unsigned tot, start;
    if (SUMS) {
        unsigned before = 0;
        for (int j = threadIdx.x; j < (int)blockIdx.x; j += SCAN_T) before += bsum[j];
        block_inclusive_scan(before, sw, &start);
    } else {
        start = bsum[blockIdx.x];
    }
    const unsigned inc = block_inclusive_scan(s, sw, &tot);
    if (SUMS && threadIdx.x == 0 && blockIdx.x == gridDim.x - 1) out[n] = start + tot;
    unsigned e[SCAN_ITEMS];
    e[0] = start + inc - s;
#pragma unroll
    for (int i = 1; i < SCAN_ITEMS; ++i) e[i] = e[i - 1] + v[i - 1];
    if (vec && base + 3 < n) {
        *reinterpret_cast<uint4*>(out + base) = make_uint4(e[0], e[1], e[2], e[3]);
    } else {
#pragma unroll
        for (int i = 0; i < SCAN_ITEMS; ++i)
            if (base + i < n) out[base + i] = e[i];
    }
}

__global__ void k_write_total(unsigned* out, int64_t n, const unsigned* total, Batch bt) {
    chain_wait();
    if (bt.ms && !bt.ms[blockIdx.x].active) return;
    const int m = slot_member(bt, blockIdx.x);
    moved(out, m * bt.stride)[n] = *moved(total, m * bt.stride);
}

// 64-bit sum and maximum of n 32-bit counts: out2[0] += sum, out2[1] = max(out2[1], max)
__global__ void k_count_totals(const unsigned* __restrict__ c, int64_t n, unsigned long long* out2) {
    chain_wait();
    unsigned long long s = 0;
    unsigned m = 0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        s += c[i];
        m = max(m, c[i]);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        s += __shfl_down_sync(0xffffffffu, s, o);
        m = max(m, __shfl_down_sync(0xffffffffu, m, o));
    }
    if ((threadIdx.x & 31) == 0) {
        atomicAdd(&out2[0], s);
        atomicMax(&out2[1], (unsigned long long)m);
    }
}

// ------------------------------------------------------------ radix sort
// Stable LSD radix sort of keys with the permutation that sorts them, at most
// 8 bits a pass (the bits split evenly).  A CTA takes a tile of 4096 consecutive items, a warp 512 of them in
// 16 rounds of 32: a round's items of one digit take consecutive ranks in lane
// order behind the warp's running count (match + popc, no barrier), the warps'
// counts are scanned per digit, and the tile is put in order in shared memory
// so that each digit's run goes out in consecutive addresses.  Bound by the
// latency of that chain: 64 registers and the largest shared-memory carve-out
// keep four CTAs a SM (two: 152-194 us).  16.7 M keys, us a pass: 136 with a
// block-wide ranking of every 256 items and scattered stores -> 96 the first
// pass, 110 the others; histogram 37 -> 13.
constexpr int RX_T = 256;
constexpr int RX_ITEMS = 16;
constexpr int RX_TILE = RX_T * RX_ITEMS;

__global__ void __launch_bounds__(RX_T) k_radix_hist(const unsigned* __restrict__ keys, int64_t n, int shift,
                                                     unsigned mask, int ntiles, unsigned* __restrict__ hist,
                                                     bool vec) {
    __shared__ unsigned h[256];
    chain_wait();
    h[threadIdx.x] = 0;
    __syncthreads();
    const int64_t base = (int64_t)blockIdx.x * RX_TILE;
    if (vec && base + RX_TILE <= n) {
        const uint4* k4 = reinterpret_cast<const uint4*>(keys + base);
        uint4 v[RX_ITEMS / 4];
#pragma unroll
        for (int i = 0; i < RX_ITEMS / 4; ++i) v[i] = k4[i * RX_T + threadIdx.x];
#pragma unroll
        for (int i = 0; i < RX_ITEMS / 4; ++i) {
            atomicAdd(&h[(v[i].x >> shift) & mask], 1u);
            atomicAdd(&h[(v[i].y >> shift) & mask], 1u);
            atomicAdd(&h[(v[i].z >> shift) & mask], 1u);
            atomicAdd(&h[(v[i].w >> shift) & mask], 1u);
        }
    } else {
        for (int i = 0; i < RX_ITEMS; ++i) {
            const int64_t idx = base + (int64_t)i * RX_T + threadIdx.x;
            if (idx < n) atomicAdd(&h[(keys[idx] >> shift) & mask], 1u);
        }
    }
    __syncthreads();
    if (threadIdx.x <= mask) hist[(int64_t)threadIdx.x * ntiles + blockIdx.x] = h[threadIdx.x];
}

// FIRST: the permutation so far is the identity (vin is not read)
template <bool FIRST>
__global__ void __launch_bounds__(RX_T, 4) k_radix_scatter(const unsigned* __restrict__ kin,
                                                        const unsigned* __restrict__ vin, int64_t n, int shift,
                                                        unsigned mask, int ntiles, const unsigned* __restrict__ hscan,
                                                        unsigned* __restrict__ kout, unsigned* __restrict__ vout) {
    constexpr int W = RX_T / 32;
    __shared__ unsigned wh[W][256];                          // per warp: a digit's count, then its first place
    __shared__ unsigned sk[RX_TILE], sv[RX_TILE];            // the tile in order
    __shared__ unsigned gs[256];                             // a digit's first address less its first place
    __shared__ unsigned sw[32];
    chain_wait();
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int64_t t0 = (int64_t)blockIdx.x * RX_TILE, base = t0 + w * (RX_ITEMS * 32) + lane;
    unsigned k[RX_ITEMS], rank[RX_ITEMS];
#pragma unroll
    for (int r = 0; r < RX_ITEMS; ++r) k[r] = base + r * 32 < n ? kin[base + r * 32] : 0u;
#pragma unroll
    for (int i = 0; i < W; ++i) wh[i][threadIdx.x] = 0u;
    __syncthreads();
#pragma unroll
    for (int r = 0; r < RX_ITEMS; ++r) {
        const bool act = base + r * 32 < n;
        const unsigned d = act ? (k[r] >> shift) & mask : 256u;
        // lanes of the same digit.  A match instruction costs more the more
        // values there are: the low digits of a pass over lattice order differ
        // all along a warp (117 us with a ballot per bit, 126 matched), the
        // higher ones hardly (113, 105)
        unsigned peers = 0xffffffffu;
        if (FIRST) {
#pragma unroll
            for (int b = 0; b < 9; ++b) {
                const bool bit = (d >> b) & 1u;
                const unsigned m = __ballot_sync(0xffffffffu, bit);
                peers &= bit ? m : ~m;
            }
        } else {
            peers = __match_any_sync(0xffffffffu, d);
        }
        const int leader = __ffs(peers) - 1;
        unsigned st = 0;
        if (lane == leader && act) {
            st = wh[w][d];
            wh[w][d] = st + (unsigned)__popc(peers);
        }
        rank[r] = __shfl_sync(0xffffffffu, st, leader) + (unsigned)__popc(peers & ((1u << lane) - 1u));
        __syncwarp();
    }
    __syncthreads();
    {
        const int d = threadIdx.x;
        unsigned t = 0, total;
#pragma unroll
        for (int i = 0; i < W; ++i) {
            const unsigned c = wh[i][d];
            wh[i][d] = t;
            t += c;
        }
        const unsigned first = block_inclusive_scan(t, sw, &total) - t;
#pragma unroll
        for (int i = 0; i < W; ++i) wh[i][d] += first;
        if (d <= (int)mask) gs[d] = hscan[(int64_t)d * ntiles + blockIdx.x] - first;
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < RX_ITEMS; ++r) {
        const int64_t idx = base + r * 32;
        if (idx < n) {
            const unsigned at = wh[w][(k[r] >> shift) & mask] + rank[r];
            sk[at] = k[r];
            sv[at] = FIRST ? (unsigned)idx : vin[idx];
        }
    }
    __syncthreads();
    const int cnt = (int)(n - t0 < RX_TILE ? n - t0 : RX_TILE);
    for (int i = threadIdx.x; i < cnt; i += RX_T) {
        const unsigned kk = sk[i];
        const unsigned at = gs[(kk >> shift) & mask] + (unsigned)i;
        if (at < (unsigned)n) {
            kout[at] = kk;
            vout[at] = sv[i];
        }
    }
}

}  // namespace

int scan_tmp_words(int64_t n) { return (int)((n + SCAN_TILE - 1) / SCAN_TILE) + 1; }

int scan_launches(int64_t n) { return (n + SCAN_TILE - 1) / SCAN_TILE <= 2048 ? 2 : 4; }

void exclusive_scan(const unsigned* in, unsigned* out, int64_t n, unsigned* tmp, cudaStream_t st, const Batch& bt) {
    int nb = (int)((n + SCAN_TILE - 1) / SCAN_TILE);
    if (nb == 0) nb = 1;
    unsigned* total = tmp + nb;
    // (members are whole multiples of 256 bytes apart: the same alignment)
    const bool vec = ((reinterpret_cast<uintptr_t>(in) | reinterpret_cast<uintptr_t>(out)) & 15) == 0;
    launch_chained(k_scan_reduce, dim3(nb, bt.members), SCAN_T, 0, st, in, n, tmp, vec, bt);
    // up to 2048 tiles (8 M items) the blocks add the earlier tiles' sums
    // themselves: two launches instead of four.  (A batch keeps the four.)
    if (nb <= 2048 && bt.members == 1 && !bt.ms) {
        launch_chained(k_scan_down<true>, dim3(nb), SCAN_T, 0, st, in, n, tmp, out, vec, bt);
        return;
    }
    launch_chained(k_scan_bsums, dim3(bt.members), SCAN_T, 0, st, tmp, nb, total, bt);
    launch_chained(k_scan_down<false>, dim3(nb, bt.members), SCAN_T, 0, st, in, n, tmp, out, vec, bt);
    launch_chained(k_write_total, dim3(bt.members), 1, 0, st, out, n, total, bt);
}

void count_totals(const unsigned* counts, int64_t n, unsigned long long* out2, cudaStream_t st) {
    const int64_t nb = (n + 255) / 256;
    launch_chained(k_count_totals, dim3((unsigned)(nb < 1024 ? (nb < 1 ? 1 : nb) : 1024)), 256, 0, st, counts, n, out2);
}

int64_t radix_tmp_words(int64_t n) {
    int64_t ntiles = (n + RX_TILE - 1) / RX_TILE;
    if (ntiles == 0) ntiles = 1;
    int64_t h = 256 * ntiles;
    return 2 * h + 1 + scan_tmp_words(h) + 2 * n + 8;     // + 8: the arrays of n begin on 16-byte boundaries
}

int radix_launches(int64_t n, int key_bits) {
    const int passes = (key_bits + 7) / 8, bits = (key_bits + passes - 1) / passes;
    return passes * (2 + scan_launches((n + RX_TILE - 1) / RX_TILE << bits));
}

unsigned* radix_sort_index(unsigned* keys, unsigned* perm, int64_t n, int key_bits, unsigned* tmp, cudaStream_t st,
                           unsigned** spare) {
    const int ntiles = (int)((n + RX_TILE - 1) / RX_TILE);
    const int64_t h = 256LL * ntiles;
    unsigned* hist = tmp;
    unsigned* hscan = hist + h;          // h + 1 entries (total at the end)
    unsigned* stmp = hscan + h + 1;
    unsigned* kalt = reinterpret_cast<unsigned*>((reinterpret_cast<uintptr_t>(stmp + scan_tmp_words(h)) + 15) & ~(uintptr_t)15);
    unsigned* valt = kalt + (n + 3) / 4 * 4;
    unsigned *ka = keys, *va = valt, *kb = kalt, *vb = perm;
    cudaFuncSetAttribute(k_radix_scatter<true>, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
    cudaFuncSetAttribute(k_radix_scatter<false>, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
    const int passes = (key_bits + 7) / 8, bits = (key_bits + passes - 1) / passes;
    const unsigned mask = (1u << bits) - 1u;
    for (int p = 0; p < passes; ++p) {
        const int shift = bits * p;
        const bool vec = (reinterpret_cast<uintptr_t>(ka) & 15) == 0;
        launch_chained(k_radix_hist, dim3(ntiles), RX_T, 0, st, ka, n, shift, mask, ntiles, hist, vec);
        exclusive_scan(hist, hscan, (int64_t)(mask + 1) * ntiles, stmp, st);
        if (p == 0) launch_chained(k_radix_scatter<true>, dim3(ntiles), RX_T, 0, st, ka, va, n, shift, mask, ntiles, hscan, kb, vb);
        else launch_chained(k_radix_scatter<false>, dim3(ntiles), RX_T, 0, st, ka, va, n, shift, mask, ntiles, hscan, kb, vb);
        std::swap(ka, kb);
        std::swap(va, vb);
    }
    spare[0] = ka;
    spare[1] = kb;
    spare[2] = vb;
    return va;
}

}  // namespace cube
