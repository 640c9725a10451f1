// Kernels on the compressed, cell-ordered particle store:
//   encode (Fig. fig.ic, Section 2.3.2), decode (Eqs. x, v), CIC deposit,
//   pass A (decode, CIC gather of -grad Phi, kick, re-encode, drift, new-cell
//   histograms; Figs. update_vp and update_xp first loop), cells (counts,
//   offsets and v_c of the new store from the scanned histograms), pass B
//   (identical drift, stable scatter by new cell,
//   Eq. chi / Eq. nu encode against the new v_c; Fig. update_xp second loop).
//
// The per-particle passes of a step run one CTA per storage brick: the brick's cells
// are contiguous in the store, so the CTA reads a contiguous particle range
// and finds each particle's cell by binary search in the brick's offsets.
#include <algorithm>

#include "kernels.h"

namespace cube {

namespace {

constexpr int T_BRICK = 256;                 // threads of the per-brick kernels
constexpr double PI_D = 3.141592653589793;   // nearest double to pi

__device__ __forceinline__ int upper_cell(const unsigned* off, int ncell, unsigned i) {
    // largest c in [0, ncell) with off[c] <= i  (off[ncell] > i)
    int lo = 0, hi = ncell;
    while (hi - lo > 1) {
        int mid = (lo + hi) >> 1;
        if (off[mid] <= i) lo = mid; else hi = mid;
    }
    return lo;
}

// Cells of a warp's 32 consecutive particles base + lane, from c0, the cell
// of particle base (off[c0] <= base < off[c0 + 1]; a brick's cells are
// contiguous and in order).  Lane j holds b_j = off[c0 + 1 + j] - base, which
// does not decrease with j, and the cell of particle base + l is
// c0 + #{j : b_j <= l}: a binary search over the lanes through shuffles.
// More than 32 cell starts within the round (empty cells) are finished by a
// walk.  *c_next is the cell of particle base + 32.  All 32 lanes call it,
// converged; every shuffle and vote below runs on all of them.
__device__ __forceinline__ int warp_cells(const unsigned* off, int ncell, unsigned base, int c0, int* c_next) {
    const unsigned lane = threadIdx.x & 31;
    const int cj = c0 + 1 + (int)lane;
    const unsigned b = cj < ncell ? off[cj] - base : 0xffffffffu;
    int k = 0;
#pragma unroll
    for (int st = 16; st >= 1; st >>= 1)
        k += __shfl_sync(0xffffffffu, b, k + st - 1) <= lane ? st : 0;
    const unsigned b31 = __shfl_sync(0xffffffffu, b, 31);    // by every lane, before any branch
    if (k == 31 && b31 <= lane) k = 32;
    int c = c0 + k;
    if (k == 32)
        while (c + 1 < ncell && off[c + 1] <= base + lane) ++c;
    const unsigned m = __ballot_sync(0xffffffffu, b <= 32u);
    int cn = c0 + __popc(m);
    if (m == 0xffffffffu)
        while (cn + 1 < ncell && off[cn + 1] <= base + 32) ++cn;
    *c_next = cn;
    return c;
}

// The particles [q0, q1) of a brick: each warp takes a contiguous share
// [*p0, *p1), a multiple of 32 but for the last.
__device__ __forceinline__ void brick_share(unsigned q0, unsigned q1, unsigned* p0, unsigned* p1) {
    const unsigned nw = blockDim.x >> 5;
    const unsigned share = ((q1 - q0 + nw * 32 - 1) / (nw * 32)) * 32;
    *p0 = q0 + min(q1 - q0, (threadIdx.x >> 5) * share);
    *p1 = min(q1, *p0 + share);
}

// the decode table of 2-byte codes through its corrections
template <int NV>
__device__ __forceinline__ VelTables vel_tables(const CodecDev& c, int lim) {
    return VelTables{c.dec, c.vdel, VelApprox{NV == 2 ? c.est[3] : 0.0f, NV == 2 ? c.est[4] : 0.0f, 2 * lim + 1},
                     lim};
}

// brick of a CTA launched on the (nb, nb, nb x members) grid: its
// coordinates and storage rank; *m the member of a batch
template <bool BAT>
__device__ __forceinline__ int grid_brick(const Geo& g, int* bx, int* by, int* bz, int* m) {
    *m = BAT ? (int)blockIdx.z / g.nb : 0;
    *bx = blockIdx.x;
    *by = blockIdx.y;
    *bz = (int)blockIdx.z - *m * g.nb;
    return *bx + g.nb * (*by + g.nb * *bz);
}

// One axis of the flattened (cell, brick) slot of a halo cell (flat_slot),
// for the brick at coordinate `me` on that axis and halo coordinate e in
// [0, Bh): the cell's home brick coordinate (bits 0-7), its coordinate in
// that brick (8-11), this brick's rank among the cell's candidate bricks
// (12-15), the number of candidates (16-19) and of candidate slots before
// the cell (20-23).  Bricks of 1, 2 or 4 cells and at most 256 bricks per
// side keep every field in range.
__device__ __forceinline__ unsigned halo_axis_desc(const Geo& g, int me, int e) {
    const int c = wrap1(me * g.B - 1 + e, g.Nc);
    const int lx = c & (g.B - 1), hbc = c >> g.lB;
    const int lo = lx == 0 ? wrap1(hbc - 1, g.nb) : -1;
    const int hi = lx == g.B - 1 ? wrap1(hbc + 1, g.nb) : -1;
    const int r = (hbc < me) + (lo >= 0 && lo < me) + (hi >= 0 && hi < me);
    return (unsigned)hbc | ((unsigned)lx << 8) | ((unsigned)r << 12) | ((unsigned)ncand(lx, g.B) << 16) |
           ((unsigned)ncand_before(lx) << 20);
}

// the flattened slot (flat_slot) and the storage rank (cell_rank) of the
// halo cell whose three axes have descriptions ax, ay, az
__device__ __forceinline__ void halo_slot(const Geo& g, unsigned ax, unsigned ay, unsigned az, int64_t* slot,
                                          int* rank_L) {
    const int S1 = g.Bh, S2 = S1 * S1;
    const int hb = (int)(ax & 255u) + g.nb * ((int)(ay & 255u) + g.nb * (int)(az & 255u));
    const int nc0 = (ax >> 16) & 15, nc1 = (ay >> 16) & 15, nc2 = (az >> 16) & 15;
    const int pre = (int)((az >> 20) & 15) * S2 + nc2 * ((int)((ay >> 20) & 15) * S1 + nc1 * (int)((ax >> 20) & 15));
    const int rank = ((int)((az >> 12) & 15) * nc1 + (int)((ay >> 12) & 15)) * nc0 + (int)((ax >> 12) & 15);
    *slot = (int64_t)hb * (S2 * S1) + pre + rank;
    *rank_L = (hb << (3 * g.lB)) + (int)((ax >> 8) & 15) + ((int)((ay >> 8) & 15) << g.lB) +
              ((int)((az >> 8) & 15) << (2 * g.lB));
}

__device__ __forceinline__ void brick_coords(const Geo& g, int brick, int* bx, int* by, int* bz) {
    *bx = brick % g.nb;
    *by = (brick / g.nb) % g.nb;
    *bz = brick / (g.nb * g.nb);
}

__device__ double block_sum_double(double v, double* sh) {
    // fixed-shape tree: deterministic for a given block size
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if (lane == 0) sh[w] = v;
    __syncthreads();
    double s = 0.0;
    if (threadIdx.x == 0)
        for (int i = 0; i < nw; ++i) s += sh[i];
    __syncthreads();
    return s;
}

__device__ __forceinline__ double snap_sigma_dev(double x) {
    // nearest 2^(m/16) in log2 (ties up), floor 2^-30
    x = fmax(x, 9.313225746154785e-10);
    double m = floor(16.0 * log2(x) + 0.5);
    return exp2(m / 16.0);
}

// ------------------------------------------------------------------ encode
// Bin of a position, floor(x scale) mod tot (tot = Nc 2^(8 n) <= 2^26, so it and
// every bin are exact in FP32): positions already in the box need neither the
// 64-bit conversion nor the modulo.  Non-finite positions give 0.
__device__ __forceinline__ int pos_bin(float x, float scale, int tot) {
    if (!isfinite(x)) return 0;
    const float f = x * scale;
    if (f >= 0.0f && f < (float)tot) return (int)f;
    long long b = __float2ll_rd(f) % tot;
    return (int)(b < 0 ? b + tot : b);
}

template <int NX>
__global__ void k_encode_keys(Geo g, const float* __restrict__ pos, unsigned* __restrict__ key, unsigned* counts,
                              unsigned* flags) {
    chain_wait();
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= g.Np) return;
    constexpr int nbits = 8 * NX;
    const float scale = ldexpf(1.0f, nbits - g.r);
    int cell[3];
    bool bad = false;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        const float x = pos[d * g.Np + i];
        bad |= !isfinite(x);
        cell[d] = pos_bin(x, scale, g.Nc << nbits) >> nbits;
    }
    const unsigned k = (unsigned)cell_rank(g, cell[0], cell[1], cell[2]);
    key[i] = k;
    // one atomic per run of lanes with one cell (neighbours in lattice order).
    // The lanes here are the warp's first `live`, whichever way each of them
    // took through pos_bin: the mask follows from the index, and the shuffle
    // and the ballot bring the lanes together.
    const int lane = threadIdx.x & 31;
    const int live = (int)min(g.Np - (i - lane), (int64_t)32);
    const unsigned act = 0xffffffffu >> (32 - live);
    const unsigned left = __shfl_up_sync(act, k, 1);
    const unsigned heads = __ballot_sync(act, lane == 0 || left != k);
    if ((heads >> lane) & 1u) {
        const unsigned after = lane == 31 ? 0u : heads & (0xfffffffeu << lane);
        const int end = after ? __ffs(after) - 1 : live;
        atomicAdd(&counts[k], (unsigned)(end - lane));
    }
    if (bad) atomicOr(flags, ERR_NONFINITE);
}

// Cells of a CTA of k_encode_vc and k_encode_codes: consecutive in storage order, so their
// particles are too, whatever the brick (the encode of 128^3 particles in bricks
// of one cell: 482 us with a CTA a brick -> 184; of 64 cells 183)
constexpr int ENC_CELLS = 64;

// A CTA's 64 cells may hold any number of particles (a halo in a cell).  Groups
// of more than ENC_BIG are cut at the multiples of ENC_RUN in storage order, and
// the runs taken by CTAs of their own from a list, so that no CTA works on more
// than ENC_BIG particles and no thread adds the squares of more than 64.  A run's
// slot is 2 c if it begins at c ENC_RUN and 2 c + 1 if its group begins inside
// that run: no two share one, and the scale's sum does not depend on the list's
// order.  Encode of 128^3 particles, a fifth of them in one cell: 4285 us by one CTA a
// group (695 with the global atomics before it) -> 335; of 256^3, 5% in one
// cell: 9065 (2134) -> 1160.  The three launches that find an empty list: 5 of
// 250 us, 14 of 1087.
constexpr unsigned ENC_RUN = 8192, ENC_BIG = 2 * ENC_RUN;
__host__ __device__ __forceinline__ int64_t crowded_slots(const Geo& g) { return 2 * (g.Np / ENC_RUN + 1); }

// the offsets of group G's cells in shared memory, off[0 .. *nc], and its
// particles [*q0, *q1)
__device__ __forceinline__ void stage_group(const Geo& g, const unsigned* __restrict__ offsets, int G, unsigned* off,
                                            int* nc, unsigned* q0, unsigned* q1) {
    const int L0 = G * ENC_CELLS;
    *nc = min(ENC_CELLS, g.Ncc - L0);
#pragma unroll 1
    for (int c = threadIdx.x; c <= *nc; c += blockDim.x) off[c] = offsets[L0 + c];
    __syncthreads();
    *q1 = min(off[*nc], (unsigned)g.Np);
    *q0 = min(off[0], *q1);
}
__device__ __forceinline__ void cut_to_run(unsigned slot, unsigned* q0, unsigned* q1) {
    const unsigned c = slot >> 1;
    *q0 = max(*q0, c * ENC_RUN);
    *q1 = min(*q1, (c + 1) * ENC_RUN);
}

// a crowded group's runs appended to the list and its cells' sums cleared, by its CTA
__device__ void list_runs(const Geo& g, const Crowded& cr, int G, int nc, unsigned q0, unsigned q1) {
    const unsigned c0 = q0 / ENC_RUN, n = (q1 - 1) / ENC_RUN - c0 + 1;
    __shared__ unsigned at;
    if (threadIdx.x == 0) at = atomicAdd(cr.count, n);
    for (int t = threadIdx.x; t < 3 * ENC_CELLS; t += blockDim.x)
        if (t % ENC_CELLS < nc) cr.vsum[(int64_t)(t / ENC_CELLS) * g.Ncc + G * ENC_CELLS + t % ENC_CELLS] = 0;
    __syncthreads();
    for (unsigned k = threadIdx.x; k < n; k += blockDim.x)
        cr.item[at + k] = make_uint2(G, 2 * (c0 + k) + (q0 > (c0 + k) * ENC_RUN ? 1u : 0u));
}

// One CTA per 64 cells of the sorted order: the particles' momenta are gathered
// once, written in storage order for the kernels that follow, and added up per
// cell in shared memory (exact fixed point); then v_c, and the cells' sum of
// squared offsets for a measured codec scale.  Crowded groups are only listed;
// the same kernel with RUNS then adds up their runs, CTA by CTA of the list, and
// k_encode_crowded finishes them.  (In one launch, the list's idle CTAs leave
// the groups unevenly over the SMs: 78 to 92 us against 66 for 512 groups of 4096
// particles.)  Six CTAs a SM, as k_encode_codes.  256^3 particles x1v1: this 182
// us and k_encode_codes 203, where 64-bit global atomics per particle, the
// measurement and the final gather took 215 + 28 + 58 + 398 us in four kernels;
// the whole encode with its sort 1540 -> 1087 us.
template <bool RUNS>
__global__ void __launch_bounds__(T_BRICK, 6) k_encode_vc(Geo g, const float* __restrict__ vel,
                                                          const unsigned* __restrict__ perm, StoreDev s, float* v0,
                                                          float* v1, float* v2, float* __restrict__ part, Crowded cr,
                                                          unsigned* flags) {
    __shared__ unsigned off[ENC_CELLS + 1];
    __shared__ unsigned vs[3 * ENC_CELLS * 2];               // {low, high} words
    __shared__ float svc[3 * ENC_CELLS];
    __shared__ double red[32];
    chain_wait();
    const unsigned lane = threadIdx.x & 31;
    float* vo[3] = {v0, v1, v2};
    const float* vi[3] = {vel, vel + g.Np, vel + 2 * g.Np};
    bool bad = false;
    const int nrun = RUNS ? (int)*cr.count : 0;
    for (int k = blockIdx.x; !RUNS || k < nrun; k += gridDim.x) {
        const uint2 item = RUNS ? cr.item[k] : make_uint2(blockIdx.x, 0u);
        const int G = (int)item.x, L0 = G * ENC_CELLS;
        if (RUNS) __syncthreads();                           // the last run's sums have been read
#pragma unroll 1
        for (int t = threadIdx.x; t < 6 * ENC_CELLS; t += blockDim.x) vs[t] = 0u;
        int nc;
        unsigned q0, q1, p0, p1;
        stage_group(g, s.offsets, G, off, &nc, &q0, &q1);
        if (RUNS) cut_to_run(item.y, &q0, &q1);
        if (!RUNS && cr.ctas > 0) {
            if (part && threadIdx.x == 0)
                for (int64_t i = G; i < crowded_slots(g); i += gridDim.x) cr.part[i] = 0.0f;
            if (q1 - q0 > ENC_BIG) {
                if (part && threadIdx.x == 0) part[G] = 0.0f;
                list_runs(g, cr, G, nc, q0, q1);
                return;
            }
        }
        brick_share(q0, q1, &p0, &p1);
        // 64 particles of the warp at a time, their loads in flight together
        float v[2][3];
        int cell[2] = {0, 0};
        int c0 = p0 < p1 ? upper_cell(off, nc, p0) : 0;
        for (unsigned base = p0; base < p1; base += 64) {
            unsigned i[2];
#pragma unroll
            for (int h = 0; h < 2; ++h) i[h] = base + 32 * h + lane < p1 ? perm[base + 32 * h + lane] : 0xffffffffu;
#pragma unroll
            for (int h = 0; h < 2; ++h)
#pragma unroll
                for (int d = 0; d < 3; ++d) v[h][d] = i[h] < (unsigned)g.Np ? vi[d][i[h]] : 0.0f;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const unsigned j = base + 32 * h + lane;
                int cnext;
                cell[h] = warp_cells(off, nc, base + 32 * h, c0, &cnext);
                c0 = cnext;
                if (j < p1)
#pragma unroll
                    for (int d = 0; d < 3; ++d) {
                        if (!isfinite(v[h][d])) {
                            bad = true;
                            v[h][d] = 0.0f;
                        }
                        vo[d][j] = v[h][d];
                        smem_add_u64(&vs[2 * (d * ENC_CELLS + cell[h])], (unsigned long long)vel_fix(v[h][d]));
                    }
            }
        }
        __syncthreads();
        for (int t = threadIdx.x; t < 3 * ENC_CELLS; t += blockDim.x) {
            const int d = t / ENC_CELLS, c = t % ENC_CELLS;
            if (c >= nc) continue;
            const unsigned long long sum = ((unsigned long long)vs[2 * t + 1] << 32) | vs[2 * t];
            const int64_t at = (int64_t)d * g.Ncc + L0 + c;
            if (RUNS) {
                if (sum) atomicAdd(reinterpret_cast<unsigned long long*>(&cr.vsum[at]), sum);
            } else {
                const float m = vel_unfix_mean((long long)sum, off[c + 1] - off[c]);
                svc[t] = m;
                s.vc[at] = m;
            }
        }
        if (RUNS) continue;
        if (part) {
            __syncthreads();
            float acc = 0.0f;
            auto add = [&](const float* x, int c) {
#pragma unroll
                for (int d = 0; d < 3; ++d) {
                    const float e = x[d] - svc[d * ENC_CELLS + c];
                    acc = __fmaf_rn(e, e, acc);
                }
            };
            if (p1 - p0 <= 64) {                             // the share is still in registers
#pragma unroll
                for (int h = 0; h < 2; ++h)
                    if (p0 + 32 * h + lane < p1) add(v[h], cell[h]);
            } else {
                c0 = upper_cell(off, nc, p0);
                for (unsigned base = p0; base < p1; base += 32) {
                    const unsigned j = base + lane;
                    int cnext;
                    const int c = warp_cells(off, nc, base, c0, &cnext);
                    c0 = cnext;
                    if (j < p1) {
                        const float x[3] = {vo[0][j], vo[1][j], vo[2][j]};
                        add(x, c);
                    }
                }
            }
            const double t = block_sum_double((double)acc, red);
            if (threadIdx.x == 0) part[G] = (float)t;
        }
        break;
    }
    if (bad) atomicOr(flags, ERR_NONFINITE);
}

// the crowded groups' v_c (written by a group's first run) and their runs' sums
// of squared offsets, each in its slot
__global__ void __launch_bounds__(T_BRICK) k_encode_crowded(Geo g, StoreDev s, const float* v0, const float* v1,
                                                            const float* v2, bool measure, Crowded cr) {
    __shared__ unsigned off[ENC_CELLS + 1];
    __shared__ float svc[3 * ENC_CELLS];
    __shared__ double red[32];
    chain_wait();
    const unsigned lane = threadIdx.x & 31, nrun = *cr.count;
    for (unsigned k = blockIdx.x; k < nrun; k += gridDim.x) {
        const uint2 item = cr.item[k];
        int nc;
        unsigned q0, q1, p0, p1;
        __syncthreads();                                     // the last run's tables have been read
        stage_group(g, s.offsets, (int)item.x, off, &nc, &q0, &q1);
        const bool first = item.y >> 1 == q0 / ENC_RUN;
        cut_to_run(item.y, &q0, &q1);
        for (int t = threadIdx.x; t < 3 * ENC_CELLS; t += blockDim.x) {
            const int d = t / ENC_CELLS, c = t % ENC_CELLS;
            if (c >= nc) continue;
            const int64_t at = (int64_t)d * g.Ncc + (int)item.x * ENC_CELLS + c;
            const float m = vel_unfix_mean(cr.vsum[at], off[c + 1] - off[c]);
            svc[t] = m;
            if (first) s.vc[at] = m;
        }
        if (!measure) continue;
        __syncthreads();
        brick_share(q0, q1, &p0, &p1);
        float acc = 0.0f;
        int c0 = p0 < p1 ? upper_cell(off, nc, p0) : 0;
        for (unsigned base = p0; base < p1; base += 32) {
            const unsigned j = base + lane;
            int cnext;
            const int c = warp_cells(off, nc, base, c0, &cnext);
            c0 = cnext;
            if (j >= p1) continue;
            const float x[3] = {v0[j], v1[j], v2[j]};
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                const float e = x[d] - svc[d * ENC_CELLS + c];
                acc = __fmaf_rn(e, e, acc);
            }
        }
        const double t = block_sum_double((double)acc, red);
        if (threadIdx.x == 0) cr.part[item.y] = (float)t;
    }
}

// The codec scale from the partial sums of squared offsets, by a block of 1024
// threads: strided FP32 sums per thread (coalesced loads, fixed order), then a
// fixed tree in FP64.  COMP: the additions' errors are added up beside them
// (the encode's many partial sums, of which it once had one a thread)
template <bool COMP>
__device__ __forceinline__ void sigma_body(const float* __restrict__ part, int nparts, double count, double ratio,
                                           double fixed, double* sigma_out) {
    __shared__ double sh[32];
    float acc = 0.0f, low = 0.0f;
    for (int i = threadIdx.x; i < nparts; i += 16 * blockDim.x) {
        float v[16];                                     // 16 loads in flight, added in order
#pragma unroll
        for (int k = 0; k < 16; ++k) {
            const int j = i + k * blockDim.x;
            v[k] = j < nparts ? part[j] : 0.0f;
        }
#pragma unroll
        for (int k = 0; k < 16; ++k) {                   // (+ 0 past the end changes nothing: acc >= 0)
            const float t = __fadd_rn(acc, v[k]);
            if (COMP) {                                  // Knuth's two-sum
                const float z = __fsub_rn(t, acc);
                low += __fadd_rn(__fsub_rn(acc, __fsub_rn(t, z)), __fsub_rn(v[k], z));
            }
            acc = t;
        }
    }
    double s = block_sum_double((double)acc + (double)low, sh);
    if (threadIdx.x == 0) {
        double x = fixed > 0.0 ? fixed : sqrt(s / count) * ratio;
        *sigma_out = snap_sigma_dev(x);
    }
}

template <bool COMP>
__global__ void k_sigma_finalize(const float* __restrict__ part, int nparts, double count, double ratio,
                                 double fixed, double* sigma_out, Batch bt) {
    chain_wait();
    const int slot = blockIdx.x;                             // slot of a batch
    if (bt.ms) {
        if (!bt.ms[slot].active) return;
        ratio = bt.ms[slot].ratio;
    }
    const int m = slot_member(bt, slot);
    sigma_body<COMP>(moved(part, m * bt.stride), nparts, count, ratio, fixed, moved(sigma_out, m * bt.stride));
}

// decode table, thresholds, scale constants and (1-byte codes,
// single block) the bucket table for the codec scale sg
__device__ void codec_tables_body(int lim, const double* __restrict__ tanv, const double* __restrict__ tanh_,
                                  double sg, float* __restrict__ dec, float* __restrict__ thr,
                                  float* __restrict__ est, unsigned char* __restrict__ vtab,
                                  signed char* __restrict__ vdel, int block, int nblocks) {
    const double s = sqrt(PI_D / (2.0 * sg * sg));
    const double gam = sqrt(2.0 * sg * sg / PI_D);
    const double m = (double)(2 * lim + 1);
    const VelApprox va{(float)(PI_D / (2.0 * m)), (float)gam, 2 * lim + 1};
    for (int k = block * blockDim.x + threadIdx.x; k <= lim + 1; k += nblocks * blockDim.x) {
        int ddec = 0;                                    // correction of the 2-byte decode table (vdel)
        if (k == 0) {
            dec[lim] = 0.0f;
            thr[0] = 0.0f;
            est[0] = (float)s;
            est[1] = (float)(m / PI_D);
            est[3] = va.c;
            est[4] = va.gam;
        } else if (k <= lim) {
            float dv = (float)(tanv[k] * gam);
            dec[lim + k] = dv;
            dec[lim - k] = -dv;
            const float tv = __double2float_ru(tanh_[k] / s);
            thr[k] = tv;
            if (vdel) ddec = __float_as_int(dv) - __float_as_int(tan_steps(k, va));
        } else {
            thr[lim + 1] = __int_as_float(0x7f800000);   // +inf
        }
        if (vdel) vdel[k] = vdelta(ddec);
    }
    if (vtab) {   // 1-byte codes (lim < 256), one block: the bucket table of nu_from_table
        __shared__ float sthr[256];
        __syncthreads();
        for (int k = threadIdx.x; k <= lim; k += blockDim.x) sthr[k] = thr[k];
        __syncthreads();
        const int key0 = (int)(__float_as_uint(sthr[1]) >> (23 - VT_B)) - 1;   // first bucket lies below thr[1]
        if (threadIdx.x == 0) est[2] = __int_as_float(key0);
        for (int i = threadIdx.x; i < VT_N; i += blockDim.x) {
            const float A = __uint_as_float((unsigned)(key0 + i) << (23 - VT_B));
            int lo = 0, hi = lim;                       // number of thresholds thr[1..lim] <= A
            while (lo < hi) {
                const int mid = (lo + hi + 1) >> 1;
                if (sthr[mid] <= A) lo = mid;
                else hi = mid - 1;
            }
            vtab[i] = (unsigned char)lo;
        }
    }
}

__global__ void k_codec_tables(int lim, const double* __restrict__ tanv, const double* __restrict__ tanh_,
                               const double* __restrict__ sigma, float* __restrict__ dec, float* __restrict__ thr,
                               float* __restrict__ est, unsigned char* __restrict__ vtab,
                               signed char* __restrict__ vdel, Batch bt) {
    chain_wait();
    const int slot = blockIdx.y;                             // slot of a batch
    if (bt.ms && !bt.ms[slot].active) return;
    const size_t o = slot_member(bt, slot) * bt.stride;
    codec_tables_body(lim, moved(tanv, o), moved(tanh_, o), *moved(sigma, o), moved(dec, o), moved(thr, o),
                      moved(est, o), moved(vtab, o), moved(vdel, o), blockIdx.x, gridDim.x);
}

// codes and ids in storage order, one CTA per 64 cells (RUNS: per listed run of
// a crowded group): positions and ids gathered by the permutation, momenta
// already in order.  Bound by that gather's latency, so six CTAs a SM: 40
// registers, which the two staging loops unrolled would raise to 48 (five CTAs:
// 45 us more at 256^3 particles).
template <int NX, int NV, bool RUNS>
__global__ void __launch_bounds__(T_BRICK) k_encode_codes(Geo g, const float* __restrict__ pos,
                                                          const float* __restrict__ v0, const float* __restrict__ v1,
                                                          const float* __restrict__ v2,
                                                          const unsigned* __restrict__ id_in,
                                                          const unsigned* __restrict__ perm, CodecDev cd, StoreDev s,
                                                          Crowded cr) {
    __shared__ unsigned off[ENC_CELLS + 1];
    __shared__ float svc[3 * ENC_CELLS];
    chain_wait();
    constexpr int nbits = 8 * NX, half = 1 << (nbits - 1), mask = (1 << nbits) - 1;
    const float scale = ldexpf(1.0f, nbits - g.r);
    const unsigned lane = threadIdx.x & 31;
    const CodeRows<NX> chi(s.chi, g.Np);
    const CodeRows<NV> nu_r(s.nu, g.Np);
    const float* vi[3] = {v0, v1, v2};
    const float* xi[3] = {pos, pos + g.Np, pos + 2 * g.Np};
    const int nrun = RUNS ? (int)*cr.count : 0;
    for (int k = blockIdx.x; !RUNS || k < nrun; k += gridDim.x) {
        const uint2 item = RUNS ? cr.item[k] : make_uint2(blockIdx.x, 0u);
        const int L0 = (int)item.x * ENC_CELLS;
        if (RUNS) __syncthreads();                           // the last run's tables have been read
#pragma unroll 1
        for (int t = threadIdx.x; t < 3 * ENC_CELLS; t += blockDim.x)
            if (L0 + t % ENC_CELLS < g.Ncc) svc[t] = s.vc[(int64_t)(t / ENC_CELLS) * g.Ncc + L0 + t % ENC_CELLS];
        int nc;
        unsigned q0, q1, p0, p1;
        stage_group(g, s.offsets, (int)item.x, off, &nc, &q0, &q1);
        if (RUNS) cut_to_run(item.y, &q0, &q1);
        else if (q1 - q0 > ENC_BIG) return;
        brick_share(q0, q1, &p0, &p1);
        if (!RUNS && p0 >= p1) return;
        const int key0 = NV == 1 ? __float_as_int(cd.est[2]) : 0;
        int c0 = p0 < p1 ? upper_cell(off, nc, p0) : 0;
        for (unsigned base = p0; base < p1; base += 64) {   // 64 particles' loads in flight
            float x[2][3], v[2][3];
            unsigned i[2], pid[2] = {0, 0};
#pragma unroll
            for (int h = 0; h < 2; ++h) i[h] = base + 32 * h + lane < p1 ? perm[base + 32 * h + lane] : 0xffffffffu;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const bool ok = i[h] < (unsigned)g.Np;
#pragma unroll
                for (int d = 0; d < 3; ++d) {
                    x[h][d] = ok ? xi[d][i[h]] : 0.0f;
                    v[h][d] = ok ? vi[d][base + 32 * h + lane] : 0.0f;
                }
                if (s.id && ok) pid[h] = id_in ? id_in[i[h]] : i[h];
            }
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const unsigned j = base + 32 * h + lane;
                int cnext;
                const int c = warp_cells(off, nc, base + 32 * h, c0, &cnext);
                c0 = cnext;
                if (j >= p1) continue;
                float dd[3];
                int nu[3];
#pragma unroll
                for (int d = 0; d < 3; ++d) {
                    chi.put(d, j, (pos_bin(x[h][d], scale, g.Nc << nbits) & mask) - half);
                    dd[d] = v[h][d] - svc[d * ENC_CELLS + c];
                    if (NV == 1) nu[d] = nu_from_table(dd[d], cd.thr, cd.vtab, key0, g.nulim);
                }
                if (NV == 2) nu_codes3(dd, cd.thr, g.nulim, cd.est[0], cd.est[1], nu);
#pragma unroll
                for (int d = 0; d < 3; ++d) nu_r.put(d, j, nu[d]);
                if (s.id) store_pid(s.id, j, g.nid, pid[h]);
            }
        }
        if (!RUNS) break;
    }
}

// ------------------------------------------------------------------ decode
// Bound by its 28 bytes written per particle.  Positions q 2^-s with the
// integer q = (cell << (8 n + 1)) + Q are rounded once: q < 2^19 for 1-byte
// codes is exact in FP32, q < 2^27 for 2-byte codes is rounded to nearest by
// u32_to_float_rn, and the scale is a power of two (the FP64 conversions of
// an FP64 product cost more than the stores here).  A CTA's life is a chain of
// loads, so a warp's first 64 particles are requested beside the brick's
// tables and the rest 64 at a time.  256^3 particles x1v1: 0.342 ms with FP64
// positions, a search per particle and tables in global memory -> 0.164 ms.
// A CTA takes 64 consecutive cells whatever the brick: one of side 4, eight of
// side 2 or 64 of side 1, whose cells' coordinates are staged (!B4).  128^3
// particles in bricks of one cell: 682 us with 256 threads a brick, 157 with 32 -> 45; with a
// fifth of them in one cell 2962, 6212 -> 803.  (The staging loops are not unrolled:
// 172 us instead of 163 at 256^3.)
constexpr int DEC_CELLS = 64;
template <int NX, int NV, bool B4>
__global__ void __launch_bounds__(T_BRICK) k_decode(Geo g, StoreDev s, CodecDev cd, float* __restrict__ pos,
                                                    float* __restrict__ vel, unsigned* __restrict__ id) {
    __shared__ unsigned off[DEC_CELLS + 1];
    __shared__ float svc[3 * DEC_CELLS];
    __shared__ float dec[NV == 1 ? 255 : 1];
    __shared__ unsigned where[B4 ? 1 : DEC_CELLS];            // x + 2^10 (y + 2^10 z) of the cells
    chain_wait();
    const int lim = g.nulim;
    const int L0 = blockIdx.x * DEC_CELLS, nc = B4 ? DEC_CELLS : min(DEC_CELLS, g.Ncc - L0);
#pragma unroll 1
    for (int i = threadIdx.x; i <= nc; i += blockDim.x) cp_async4(&off[i], &s.offsets[L0 + i]);
#pragma unroll 1
    for (int i = threadIdx.x; i < 3 * DEC_CELLS; i += blockDim.x)
        if (B4 || i % DEC_CELLS < nc)
            cp_async4(&svc[i], &s.vc[(int64_t)(i / DEC_CELLS) * g.Ncc + L0 + i % DEC_CELLS]);
    if (NV == 1)
#pragma unroll 1
        for (int i = threadIdx.x; i < 2 * lim + 1; i += blockDim.x) cp_async4(&dec[i], &cd.dec[i]);
    const unsigned q1 = min(s.offsets[L0 + nc], (unsigned)g.Np), q0 = min(s.offsets[L0], q1);
    unsigned p0, p1;
    brick_share(q0, q1, &p0, &p1);
    const unsigned lane = threadIdx.x & 31;
    const CodeRows<NX> chi(s.chi, g.Np);
    const CodeRows<NV> nu(s.nu, g.Np);
    int x[2][3], v[2][3];
    unsigned pid[2];
    auto load = [&](unsigned base) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const unsigned i = base + 32 * h + lane;
            if (i >= p1) continue;
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                x[h][d] = chi.get(d, i);
                v[h][d] = nu.get(d, i);
            }
            pid[h] = id && s.id ? load_pid(s.id, i, g.nid) : i;
        }
    };
    load(p0);
    int b[3];
    if (!B4 && (int)threadIdx.x < nc) {
        const int L = L0 + (int)threadIdx.x, lc = L & ((1 << (3 * g.lB)) - 1), bm = g.B - 1;
        brick_coords(g, L >> (3 * g.lB), &b[0], &b[1], &b[2]);
        where[threadIdx.x] = (unsigned)((b[0] << g.lB) + (lc & bm)) |
                             (unsigned)((b[1] << g.lB) + ((lc >> g.lB) & bm)) << 10 |
                             (unsigned)((b[2] << g.lB) + (lc >> (2 * g.lB))) << 20;
    }
    cp_async_wait_all();
    __syncthreads();
    if (p0 >= p1) return;
    const VelTables vt = vel_tables<NV>(cd, lim);
    if (B4) brick_coords(g, blockIdx.x, &b[0], &b[1], &b[2]);
    constexpr int nbits = 8 * NX, half = 1 << (nbits - 1);
    const float pscale = ldexpf(1.0f, g.r - nbits - 1);
    int c0 = upper_cell(off, nc, p0);
    for (unsigned base = p0;;) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const unsigned i = base + 32 * h + lane;
            int cnext;
            const int lc = warp_cells(off, nc, base + 32 * h, c0, &cnext);
            c0 = cnext;
            if (i < p1) {
#pragma unroll
                for (int d = 0; d < 3; ++d) {
                    const int c = B4 ? 4 * b[d] + ((lc >> (2 * d)) & 3) : (int)((where[lc] >> (10 * d)) & 1023u);
                    const unsigned q = ((unsigned)c << (nbits + 1)) + (unsigned)(2 * (x[h][d] + half) + 1);
                    const float f = NX == 1 ? __uint_as_float(0x4B000000u | q) - 8388608.0f : u32_to_float_rn(q);
                    pos[d * g.Np + i] = f * pscale;
                    const int k = max(-lim, min(lim, v[h][d]));
                    vel[d * g.Np + i] = svc[d * DEC_CELLS + lc] + (NV == 1 ? dec[k + lim] : vt.dec(k));
                }
                if (id) id[i] = pid[h];
            }
        }
        base += 64;
        if (base >= p1) break;
        load(base);
    }
}

// largest |p| over particles and axes of the store (momenta as decoded,
// v_c + tan-table offset), as the bits of a non-negative float (order-
// preserving as unsigned).  The table and the rounded sum grow with the code,
// so a cell's largest |p| along an axis is at its smallest or largest code:
// LPC lanes a cell take both over the cell's particles and two codes are
// decoded, not every particle's.  Cells of more than 8 LPC particles (haloes)
// are finished by their whole warp, so that no lane runs alone, and cells of
// more than SPEED_BIG by the whole CTA (128^3 particles, a fifth of them in one
// cell: 1566 us by a warp, 798 by a CTA a brick and a decode per particle -> 158).  A warp's
// life is a chain of loads (offsets, codes, table): LPC = 8 gives small stores
// their warps (one wave holds 64 of them per SM), LPC = 2 keeps large ones to
// few waves.  The call with its read-backs (25 us of
// them host and copies), 192^3 particles x1v1, clustered: 73 us with a CTA a
// brick, a search and a decode per particle -> 55 us; 32^3: 29.7 -> 26.4 us.
constexpr unsigned SPEED_BIG = 2048;
template <int NV, int LPC>
__global__ void __launch_bounds__(T_BRICK) k_max_speed(Geo g, StoreDev s, CodecDev cd,
                                                       unsigned* __restrict__ vmax_bits, Batch bt) {
    chain_wait();
    {                                                        // member of slot blockIdx.y of a batch
        const size_t o = slot_member(bt, blockIdx.y) * bt.stride;
        s = moved(s, o);
        cd = moved(cd, o);
        vmax_bits = moved(vmax_bits, o);
    }
    const int lane = threadIdx.x & 31;
    const int L = (blockIdx.x * T_BRICK + threadIdx.x) / LPC, sub = threadIdx.x % LPC;
    const CodeRows<NV> nu(s.nu, g.Np);
    constexpr int kNone = 0x7fffffff;
    unsigned i0 = 0, i1 = 0;
    float vc[3] = {0.0f, 0.0f, 0.0f};
    if (L < g.Ncc) {
        i1 = min(s.offsets[L + 1], (unsigned)g.Np);
        i0 = min(s.offsets[L], i1);
#pragma unroll
        for (int d = 0; d < 3; ++d) vc[d] = s.vc[(int64_t)d * g.Ncc + L];
    }
    int lo[3] = {kNone, kNone, kNone}, hi[3] = {-kNone, -kNone, -kNone};
    const unsigned e = min(i1, i0 + 8u * LPC);
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        const unsigned i = i0 + sub + k * LPC;
        if (i < e)
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                const int v = nu.get(d, i);
                lo[d] = min(lo[d], v);
                hi[d] = max(hi[d], v);
            }
    }
    const bool big = i1 - i0 > SPEED_BIG;
    for (unsigned more = __ballot_sync(0xffffffffu, sub == 0 && e < i1 && !big); more; more &= more - 1) {
        const int src = __ffs(more) - 1;
        const unsigned a = __shfl_sync(0xffffffffu, e, src), z = __shfl_sync(0xffffffffu, i1, src);
        int wl[3] = {kNone, kNone, kNone}, wh[3] = {-kNone, -kNone, -kNone};
#pragma unroll 4
        for (unsigned i = a + lane; i < z; i += 32)
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                const int v = nu.get(d, i);
                wl[d] = min(wl[d], v);
                wh[d] = max(wh[d], v);
            }
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            const int l = __reduce_min_sync(0xffffffffu, wl[d]), h = __reduce_max_sync(0xffffffffu, wh[d]);
            if (lane == src) {
                lo[d] = min(lo[d], l);
                hi[d] = max(hi[d], h);
            }
        }
    }
#pragma unroll
    for (int o = LPC / 2; o > 0; o >>= 1)
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            lo[d] = min(lo[d], __shfl_xor_sync(0xffffffffu, lo[d], o));
            hi[d] = max(hi[d], __shfl_xor_sync(0xffffffffu, hi[d], o));
        }
    float m = 0.0f;
    if (i0 < i1 && sub < 2)                                  // lane 0 decodes the smallest codes, lane 1 the largest
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            const int v = max(-g.nulim, min(g.nulim, sub ? hi[d] : lo[d]));
            m = fmaxf(m, fabsf(vc[d] + cd.dec[v + g.nulim]));
        }
    if (__syncthreads_or(big)) {                             // the rest of the CTA's big cells, one after the other
        __shared__ int list[T_BRICK / LPC], nbig;
        if (threadIdx.x == 0) nbig = 0;
        __syncthreads();
        if (big && sub == 0) list[atomicAdd(&nbig, 1)] = L;
        __syncthreads();
        for (int k = 0; k < nbig; ++k) {
            const int C = list[k];
            const unsigned z = min(s.offsets[C + 1], (unsigned)g.Np);
            int wl[3] = {kNone, kNone, kNone}, wh[3] = {-kNone, -kNone, -kNone};
#pragma unroll 4
            for (unsigned i = s.offsets[C] + 8u * LPC + threadIdx.x; i < z; i += T_BRICK)
#pragma unroll
                for (int d = 0; d < 3; ++d) {
                    const int v = nu.get(d, i);
                    wl[d] = min(wl[d], v);
                    wh[d] = max(wh[d], v);
                }
            // each warp's own extremes (it has some: SPEED_BIG is larger than a round)
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                const int l = __reduce_min_sync(0xffffffffu, wl[d]), h = __reduce_max_sync(0xffffffffu, wh[d]);
                const int v = max(-g.nulim, min(g.nulim, lane & 1 ? h : l));
                if (lane < 2) m = fmaxf(m, fabsf(s.vc[(int64_t)d * g.Ncc + C] + cd.dec[v + g.nulim]));
            }
        }
    }
    block_max_to(__float_as_uint(m), vmax_bits);
}

// ------------------------------------------------------------------ CIC deposit
// Owner computes: a CTA produces the density of its brick's fine nodes
// [o, o + F)^3 from the particles of the brick's cells and of the one-cell
// layer below it (a particle in fine cell i also feeds node i + 1).  Weights
// are integers (numerators over 2^s per axis) summed in int64, so the result
// is exact and independent of the summation order; rho = m * sum * 2^(-3s).
__device__ __forceinline__ float node_value(unsigned lo, unsigned hi) {
    return hi ? __ull2float_rn(((unsigned long long)hi << 32) | lo) : u32_to_float_rn(lo);
}

// slots of the per-particle cell table: bricks whose particles and layer
// fit look their cell up in it, larger ones (crowded late epochs) search
constexpr int DEP_QCAP = 2048;

// words of the deposit's node sums: the padded 32-bit tile of the common
// case, (F + 8) x (F + 2)^2 words, or F^3 {lo, hi} pairs, whichever is larger
__host__ __device__ __forceinline__ int dep_acc_words(int F) {
    const int fast = (F + 8) * (F + 2) * (F + 2);
    return fast > 2 * F * F * F ? fast : 2 * F * F * F;
}

template <int NX, int FC, bool BAT>
__global__ void __launch_bounds__(T_BRICK) k_deposit(Geo g, StoreDev s, float* __restrict__ mesh, float fscale,
                                                     long long* __restrict__ vsum, int* __restrict__ mig, Batch bt) {
    extern __shared__ unsigned long long dep_smem[];
    chain_wait();
    // FC > 0: the brick side in fine cells is the compile-time FC, else g.F
    const int lF = FC == 16 ? 4 : FC == 8 ? 3 : FC == 4 ? 2 : g.lF, F = 1 << lF, F3 = 1 << (3 * lF);
    const int E = g.B + 1, E3 = E * E * E;
    // node sums (block-uniform choice): when no sum can exceed 32 bits
    // ("small"), a padded tile of 32-bit words covering x in [-4, F + 4) and
    // y, z in [-1, F], so every corner of every contributing particle lies
    // inside it (no range checks) and rows start on 16-byte boundaries; else
    // [F3] {lo, hi} pairs over the brick's own nodes
    unsigned* acc = reinterpret_cast<unsigned*>(dep_smem);
    unsigned* cstart = acc + dep_acc_words(F);                       // [E3]
    unsigned* cpref = cstart + E3;                                   // [E3 + 1]
    int* cpack = reinterpret_cast<int*>(cpref + E3 + 1);             // [E3] packed cell offsets
    unsigned char* qcell = reinterpret_cast<unsigned char*>(cpack + E3);   // [DEP_QCAP] cell of each slot
    __shared__ unsigned wsum[T_BRICK / 32];
    int bx, by, bz, m;
    grid_brick<BAT>(g, &bx, &by, &bz, &m);
    if constexpr (BAT) {                                     // slot m of a batch
        if (bt.ms && !bt.ms[m].active) return;
        m = slot_member(bt, m);
        s = moved(s, m * bt.stride);
        mesh = moved(mesh, m * bt.stride);
    }
    const int c0[3] = {bx * g.B, by * g.B, bz * g.B};
    // the cells of the brick and of its one-cell layer below (E^3 <= 125 <=
    // one per thread), their particle counts scanned across the block
    unsigned cnt = 0;
    const int t = threadIdx.x;
    if (t < E3) {
        int ec[3];
        split3(t, E, div_magic(E), ec);
        const int lx = ec[0] - 1, ly = ec[1] - 1, lz = ec[2] - 1;
        const int L = cell_rank(g, wrap1(c0[0] + lx, g.Nc), wrap1(c0[1] + ly, g.Nc), wrap1(c0[2] + lz, g.Nc));
        const unsigned a = s.offsets[L];
        cstart[t] = a;
        cnt = s.offsets[L + 1] - a;
        cpack[t] = (lx + 1) | ((ly + 1) << 8) | ((lz + 1) << 16);
    }
    // node sums cleared while the offsets are in flight (both layouts)
    for (int u = threadIdx.x; u < dep_acc_words(F) / 4; u += blockDim.x)
        reinterpret_cast<uint4*>(acc)[u] = make_uint4(0u, 0u, 0u, 0u);
    {
        const int lane = t & 31, wp = t >> 5;
        unsigned v = cnt;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned u = __shfl_up_sync(0xffffffffu, v, o);
            if (lane >= o) v += u;
        }
        if (lane == 31) wsum[wp] = v;
        __syncthreads();
        for (int k = 0; k < wp; ++k) v += wsum[k];
        if (t < E3) {
            cpref[t + 1] = v;
            // this cell's slots of the per-particle cell table (used when
            // the brick's total fits it), before the barrier that publishes
            // the scan
            if (E3 <= 256)
                for (unsigned q = v - cnt, qe = min(v, (unsigned)DEP_QCAP); q < qe; ++q) qcell[q] = (unsigned char)t;
        }
        if (t == 0) cpref[0] = 0;
    }
    __syncthreads();
    // a step's deposit clears what its pass A accumulates into: the brick's
    // momentum sums, the largest migration and the number of crowded bricks
    if (!BAT && vsum) {
        const int nbc = g.B * g.B * g.B;
        const int64_t L0 = (int64_t)(bx + g.nb * (by + g.nb * bz)) * nbc;
        for (int i = t; i < 3 * nbc; i += T_BRICK) vsum[(int64_t)(i >> (3 * g.lB)) * g.Ncc + L0 + (i & (nbc - 1))] = 0;
        if (blockIdx.x + blockIdx.y + blockIdx.z == 0 && t < 2) mig[t] = 0;
    }
    const int nbits = 8 * NX, half = 1 << (nbits - 1);
    const int sb = g.sbits, wmask = (1 << sb) - 1, wone = 1 << sb;
    const unsigned total = min(cpref[E3], (unsigned)g.Np);   // bounded even for inconsistent offsets
    // a node's 32-bit sum of 1-byte-code weights (each < 2^(3 s)) cannot wrap
    // when fewer than 2^(32 - 3 s) particles feed the brick
    const bool small = 3 * sb < 32 && total < (1u << (32 - 3 * sb));
    const int ws = small ? 0 : 1;                                   // log2 words per node
    const bool table = total <= (unsigned)DEP_QCAP && E3 <= 256;    // block-uniform
    const int ox = c0[0] * g.R, oy = c0[1] * g.R, oz = c0[2] * g.R;
    if (NX == 1 && small && table) {
        // the common case: padded 32-bit tile, node (x, y, z) of the brick at
        // (x + 4) + DX ((y + 1) + DY (z + 1)); a particle's 8 corners at fixed
        // offsets from its base node, no range checks
        const int DX = F + 8, DY = F + 2, DXY = DX * DY;
        const int8_t* cx = reinterpret_cast<const int8_t*>(s.chi);
        const int8_t* cy = cx + g.Np;
        const int8_t* cz = cy + g.Np;
        const int shift = sb;
        // the next round's cell and codes are requested before this round's atomics
        int tn = 0, xn = 0, yn = 0, zn = 0;
        bool okn = false;
        auto fetch = [&](unsigned qq) {
            tn = qcell[qq];
            const unsigned ii = cstart[tn] + (qq - cpref[tn]);
            okn = ii < (unsigned)g.Np;
            if (okn) {
                xn = cx[ii];
                yn = cy[ii];
                zn = cz[ii];
            }
        };
        if (threadIdx.x < total) fetch(threadIdx.x);
        for (unsigned q = threadIdx.x; q < total; q += blockDim.x) {
            const int tc = tn, chx = xn, chy = yn, chz = zn;
            const bool ok = okn;
            if (q + blockDim.x < total) fetch(q + blockDim.x);
            if (!ok) continue;
            const int pk = cpack[tc];
            // Q = 2 (chi + 128) + 1: fine cell (Q >> sb) inside the coarse cell, weight Q & wmask
            const int Qx = 2 * chx + 257, Qy = 2 * chy + 257, Qz = 2 * chz + 257;
            const int nx = ((pk & 255) - 1) * g.R + (Qx >> shift);
            const int ny = (((pk >> 8) & 255) - 1) * g.R + (Qy >> shift);
            const int nz = ((pk >> 16) - 1) * g.R + (Qz >> shift);
            // a particle of the layer below more than one fine cell from the brick feeds none of its nodes
            if (min(nx, min(ny, nz)) < -1) continue;
            const unsigned wxn = Qx & wmask, wxm = wone - wxn;
            const unsigned wyn = Qy & wmask, wym = wone - wyn;
            const unsigned wzn = Qz & wmask, wzm = wone - wzn;
            const unsigned w00 = wym * wzm, w10 = wyn * wzm, w01 = wym * wzn, w11 = wyn * wzn;
            unsigned* a = acc + (nx + 4) + DX * ((ny + 1) + DY * (nz + 1));
            atomicAdd(a, wxm * w00);
            atomicAdd(a + 1, wxn * w00);
            atomicAdd(a + DX, wxm * w10);
            atomicAdd(a + DX + 1, wxn * w10);
            atomicAdd(a + DXY, wxm * w01);
            atomicAdd(a + DXY + 1, wxn * w01);
            atomicAdd(a + DXY + DX, wxm * w11);
            atomicAdd(a + DXY + DX + 1, wxn * w11);
        }
        __syncthreads();
        // the brick's rows (32-bit offsets: N^2 S < 2^31 for N <= 1024)
        float* mbase = mesh + ((int64_t)oz * g.N + oy) * g.S + ox;
        for (int t4 = threadIdx.x; t4 < F3 / 4; t4 += blockDim.x) {
            const int t = 4 * t4;
            const int x = t & (F - 1), y = (t >> lF) & (F - 1), z = t >> (2 * lF);
            const uint4 v = *reinterpret_cast<const uint4*>(&acc[(x + 4) + DX * ((y + 1) + DY * (z + 1))]);
            float4 f;
            if (max(max(v.x, v.y), max(v.z, v.w)) < (1u << 23)) {     // exact: 2^23 + u is a float
                f = make_float4(__uint_as_float(0x4B000000u | v.x) - 8388608.0f,
                                __uint_as_float(0x4B000000u | v.y) - 8388608.0f,
                                __uint_as_float(0x4B000000u | v.z) - 8388608.0f,
                                __uint_as_float(0x4B000000u | v.w) - 8388608.0f);
            } else {
                f = make_float4(u32_to_float_rn(v.x), u32_to_float_rn(v.y), u32_to_float_rn(v.z),
                                u32_to_float_rn(v.w));
            }
            *reinterpret_cast<float4*>(mbase + (unsigned)((z * g.N + y) * g.S + x)) =
                make_float4(f.x * fscale, f.y * fscale, f.z * fscale, f.w * fscale);
        }
        return;
    }
    for (unsigned q = threadIdx.x; q < total; q += blockDim.x) {
        const int t = table ? (int)qcell[q] : upper_cell(cpref, E3, q);
        const unsigned i = cstart[t] + (q - cpref[t]);
        if (i >= (unsigned)g.Np) continue;
        const int pk = cpack[t];
        const int l[3] = {(pk & 255) - 1, ((pk >> 8) & 255) - 1, (pk >> 16) - 1};
        int nd[3], wn[3], wm[3];
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            const int Q = 2 * (load_code<NX>(s.chi, d * g.Np + i) + half) + 1;
            nd[d] = l[d] * g.R + (Q >> sb);
            wn[d] = Q & wmask;
            wm[d] = wone - wn[d];
        }
        // a particle of the layer below more than one fine cell from the brick feeds none of its nodes
        if (nd[0] < -1 || nd[1] < -1 || nd[2] < -1) continue;
        // all 8 corners inside the brick's nodes: no per-corner range checks
        const bool inside = nd[0] >= 0 && nd[1] >= 0 && nd[2] >= 0 && nd[0] < F - 1 && nd[1] < F - 1 && nd[2] < F - 1;
#pragma unroll
        for (int dz = 0; dz < 2; ++dz) {
            const int z = nd[2] + dz;
            if (!inside && (z < 0 || z >= F)) continue;
#pragma unroll
            for (int dy = 0; dy < 2; ++dy) {
                const int y = nd[1] + dy;
                if (!inside && (y < 0 || y >= F)) continue;
#pragma unroll
                for (int dx = 0; dx < 2; ++dx) {
                    const int x = nd[0] + dx;
                    if (!inside && (x < 0 || x >= F)) continue;
                    unsigned* a = &acc[((((z << lF) + y) << lF) + x) << ws];
                    if (NX == 1) {   // weight numerators of 1-byte codes: product < 2^27
                        const unsigned w = (unsigned)(dz ? wn[2] : wm[2]) * (unsigned)(dy ? wn[1] : wm[1]) *
                                           (unsigned)(dx ? wn[0] : wm[0]);
                        if (small) {
                            atomicAdd(a, w);          // the 32-bit sum cannot wrap: no carry
                        } else {
                            const unsigned old = atomicAdd(a, w);
                            if (old + w < old) atomicAdd(a + 1, 1u);
                        }
                    } else {
                        const unsigned long long w = (unsigned long long)(dz ? wn[2] : wm[2]) *
                                                     (unsigned long long)(dy ? wn[1] : wm[1]) *
                                                     (unsigned long long)(dx ? wn[0] : wm[0]);
                        smem_add_u64(a, w);
                    }
                }
            }
        }
    }
    __syncthreads();
    // four consecutive x nodes per thread: one or two 16-byte shared loads,
    // one 16-byte store (F and the row stride S are multiples of 4)
    for (int t4 = threadIdx.x; t4 < F3 / 4; t4 += blockDim.x) {
        const int t = 4 * t4;
        const int x = t & (F - 1), y = (t >> lF) & (F - 1), z = t >> (2 * lF);
        // exact integer sum; one rounding when the scale is a power of two (mass 2^k)
        float4 v;
        if (small) {   // block-uniform: 32-bit sums of nodes t .. t + 3
            const uint4 a = reinterpret_cast<const uint4*>(acc)[t4];
            v = make_float4(u32_to_float_rn(a.x) * fscale, u32_to_float_rn(a.y) * fscale,
                            u32_to_float_rn(a.z) * fscale, u32_to_float_rn(a.w) * fscale);
        } else {
            const uint4 a = reinterpret_cast<const uint4*>(acc)[2 * t4];        // {lo, hi} of nodes t, t + 1
            const uint4 b = reinterpret_cast<const uint4*>(acc)[2 * t4 + 1];    // nodes t + 2, t + 3
            v = make_float4(node_value(a.x, a.y) * fscale, node_value(a.z, a.w) * fscale,
                            node_value(b.x, b.y) * fscale, node_value(b.z, b.w) * fscale);
        }
        *reinterpret_cast<float4*>(&mesh[((int64_t)(oz + z) * g.N + (oy + y)) * g.S + ox + x]) = v;
    }
}

// ------------------------------------------------------------------ pass A
// (bricks of more than PB_BIG particles are listed for pass B's whole-CTA path)
constexpr int PB_BIG = 1024;

// threads of a pass A CTA and the CTAs it keeps resident per SM
constexpr int PA_T = 256;
constexpr int PA_MINB = 4;

// One CTA per brick.  Shared memory: Phi tile of (F + 5)^3 fine nodes
// ([o - 2, o + F + 3) per axis, periodic), brick offsets, the histogram of
// destination cells over the brick and its one-cell halo (Bh^3 cells) with
// fixed-point momentum sums, and (1-byte velocities) the codec tables.
template <int NX, int NV, int FC, bool BAT>
__global__ void __launch_bounds__(PA_T, PA_MINB) k_passA(Geo g, StoreDev s, const float* __restrict__ phig,
                                                      const __grid_constant__ CUtensorMap tmap, int use_tma,
                                                      CodecDev cur, float kick, float dc, StepScratch w,
                                                      DriftDebug dbg, Batch bt) {
    extern __shared__ unsigned char pa_smem[];
    chain_wait();
    __shared__ __align__(8) unsigned long long tile_bar;
    // Phi tile: T x T rows (y, z: [o - 2, o + F + 3)) of TX = F + 8 nodes
    // (x: [o - 4, o + F + 4)), row stride TS = TX floats, read from the
    // ghosted Phi (no wrap): one TMA box, or 16-byte cp.async chunks
    // FC > 0: the brick side in fine cells is the compile-time FC (every
    // tile offset of the gather becomes an immediate), else g.F
    const int F = FC > 0 ? FC : g.F, T = F + 5, TX = F + 8, TS = TX, T3 = T * T * TS;
    const int nbc = g.B * g.B * g.B, Bh = g.Bh, H3 = Bh * Bh * Bh;
    const unsigned mBh = div_magic(Bh);
    const int lim = g.nulim;
    int bx, by, bz, m;
    const int brick = grid_brick<BAT>(g, &bx, &by, &bz, &m);
    if constexpr (BAT) {                                     // slot m of a batch
        if (bt.ms) {
            if (!bt.ms[m].active) return;
            kick = bt.ms[m].kick;
            dc = bt.ms[m].dc;
        }
        m = slot_member(bt, m);
        const size_t o = m * bt.stride;
        s = moved(s, o);
        phig = moved(phig, o);
        cur = moved(cur, o);
        w = moved(w, o);
    }
    const int ox = bx * F - 4, oy = by * F - 2, oz = bz * F - 2;      // tile origin
    long long* vs = reinterpret_cast<long long*>(pa_smem);                 // [3][H3]
    const unsigned sbase = smem_addr(pa_smem);
    float* tile = reinterpret_cast<float*>(pa_smem + (((sbase + 3 * H3 * 8 + 127) & ~127u) - sbase));   // [T3], 128-byte aligned
    if (use_tma) {
        if (threadIdx.x == 0) mbar_init(&tile_bar, 1);
        __syncthreads();
        if (threadIdx.x == 0) {
            mbar_expect_tx(&tile_bar, (unsigned)T3 * 4u);
            tma_load_4d(tile, &tmap, ox + PHIG_X0, oy + PHIG_Y0, oz + PHIG_Y0, m, &tile_bar);
        }
    }
    unsigned* hist = reinterpret_cast<unsigned*>(tile + T3);                // [H3]
    unsigned* sm_off = hist + H3;                                           // [nbc + 1]
    float* sdec = reinterpret_cast<float*>(sm_off + nbc + 1);               // NV == 1: [2 lim + 1]
    float* sthr = sdec + (NV == 1 ? 2 * lim + 1 : 0);                       // NV == 1: [lim + 2]
    float* svc = sthr + (NV == 1 ? lim + 2 : 0);                            // [3][nbc]: v_c of the brick
    unsigned char* stab = reinterpret_cast<unsigned char*>(svc + 3 * nbc);  // NV == 1: [VT_N] bucket table
    unsigned char* qcell = stab + (NV == 1 ? VT_N : 0);                     // [DEP_QCAP] cell of each particle
    const float* dec = cur.dec;
    const float* thr = cur.thr;
    int key0 = 0;
    if (NV == 1) {
        for (int t = threadIdx.x; t < 2 * lim + 1; t += blockDim.x) sdec[t] = cur.dec[t];
        for (int t = threadIdx.x; t < lim + 2; t += blockDim.x) sthr[t] = cur.thr[t];
        for (int t = threadIdx.x; t < VT_N / 4; t += blockDim.x)
            reinterpret_cast<unsigned*>(stab)[t] = reinterpret_cast<const unsigned*>(cur.vtab)[t];
        dec = sdec;
        thr = sthr;
        key0 = __float_as_int(cur.est[2]);
    }
    const int L0 = brick * nbc;
    for (int t = threadIdx.x; t < 3 * nbc; t += blockDim.x)
        cp_async4(&svc[t], &s.vc[(int64_t)(t >> (3 * g.lB)) * g.Ncc + L0 + (t & (nbc - 1))]);
    for (int c = threadIdx.x; c <= nbc; c += blockDim.x) sm_off[c] = s.offsets[L0 + c];
    for (int t = threadIdx.x; t < H3; t += blockDim.x) {
        hist[t] = 0u;
        vs[t] = 0;
        vs[H3 + t] = 0;
        vs[2 * H3 + t] = 0;
    }
    // per axis d and halo coordinate e in [0, Bh): the coarse cell's home
    // brick coordinate (bits 0-7), its coordinate in that brick (8-11), this
    // brick's rank among the cell's candidate bricks (12-15), the number of
    // candidates (16-19) and of candidate slots before the cell (20-23); the
    // flattened slot of a halo cell combines the three axes (flat_slot)
    __shared__ unsigned axis_desc[3 * 6];
    if (threadIdx.x < 3 * Bh) {
        const int d = threadIdx.x / Bh, ee = threadIdx.x - d * Bh;
        axis_desc[threadIdx.x] = halo_axis_desc(g, d == 0 ? bx : d == 1 ? by : bz, ee);
    }
    if (!use_tma) {
        // rows of TX = F + 8 nodes start on a 16-byte boundary: 4-node chunks;
        // thread t < RPI * CX owns chunk column cx of rows t / CX, + RPI, ...
        const int CX = TX >> 2, nrow = T * T, RPI = PA_T / CX;
        if (threadIdx.x < RPI * CX) {
            const int cx = threadIdx.x % CX;
            int row = threadIdx.x / CX;
            int z = row / T, y = row - z * T;
            const int dz = RPI / T, dy = RPI - dz * T;
            float* dst = tile + 4 * cx;
            for (; row < nrow; row += RPI) {
                cp_async16(dst + row * TS, phig + phig_index(g.N, ox + 4 * cx, oy + y, oz + z));
                y += dy;
                z += dz;
                if (y >= T) {
                    y -= T;
                    ++z;
                }
            }
        }
    }
    // the brick's particle range, and the first round's codes, requested
    // while the tile is in flight
    const unsigned q1 = min(s.offsets[L0 + nbc], (unsigned)g.Np);
    const unsigned q0 = min(s.offsets[L0], q1);
    unsigned i = q0 + threadIdx.x;
    if (threadIdx.x == 0 && q1 - q0 > (unsigned)PB_BIG) w.big[1 + atomicAdd(w.big, 1)] = brick;
    const CodeRows<NX> chi_r(s.chi, g.Np);
    const CodeRows<NV> nu_r(s.nu, g.Np);
    int nchi[3] = {0, 0, 0}, nnu[3] = {0, 0, 0};
    if (i < q1) {
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            nchi[d] = chi_r.get(d, i);
            nnu[d] = nu_r.get_nu(d, i, lim);
        }
    }
    // the cell of every particle of the brick, when they fit the table,
    // written while the tile is in flight (each thread reads its cells' bounds)
    const bool table = q1 - q0 <= (unsigned)DEP_QCAP;                  // block-uniform
    if (table)
        for (int c = threadIdx.x; c < nbc; c += blockDim.x)
            for (unsigned q = max(s.offsets[L0 + c], q0), qe = min(s.offsets[L0 + c + 1], q1); q < qe; ++q)
                qcell[q - q0] = (unsigned char)c;
    cp_async_wait_all();
    const bool tile_ok = !use_tma || mbar_wait_bounded(&tile_bar, 0);
    if (__syncthreads_or(!tile_ok)) {       // the tile copy never completed: report, drain, leave
        if (threadIdx.x == 0) atomicOr(w.flags, ERR_TIMEOUT);
        mbar_wait_bounded(&tile_bar, 0);
        return;
    }
    const float e0 = cur.est[0], e1 = cur.est[1];
    // 2-byte codes: the decode table through its L1-resident corrections
    const VelTables vt = vel_tables<NV>(cur, lim);
    const int nbits = 8 * NX, half = 1 << (nbits - 1);
    const int sb = g.sbits, wmask = (1 << sb) - 1;
    // the in-cell CIC weight (Q mod 2^sb) 2^-sb exactly from the bits of
    // 2^(23 - sb) + (Q mod 2^sb) 2^-sb
    const int wexp = (127 + 23 - sb) << 23;
    const float wbase = ldexpf(1.0f, 23 - sb);
    const float dcs = ldexpf(dc, nbits);           // drift in bins of the position code
    const float kick12 = kick * (-1.0f / 12.0f);   // the FD4 sums' 1/12 and the sign of -grad Phi
    float sacc = 0.0f;
    int mig = 0;
    bool migbad = false;
    const int TT = T * TS;   // z stride of the tile
    const int lB = g.lB, bm = g.B - 1;
    for (; i < q1; i += blockDim.x) {
        // this round's codes; the next round's are requested now
        const int cchi[3] = {nchi[0], nchi[1], nchi[2]}, cnu[3] = {nnu[0], nnu[1], nnu[2]};
        if (i + blockDim.x < q1) {
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                nchi[d] = chi_r.get(d, i + blockDim.x);
                nnu[d] = nu_r.get_nu(d, i + blockDim.x, lim);
            }
        }
        const int lc = table ? (int)qcell[i - q0] : upper_cell(sm_off, nbc, i);
        const int l[3] = {lc & bm, (lc >> lB) & bm, lc >> (2 * lB)};
        int Q[3], n[3];
        float w1[3], w0[3];
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            Q[d] = 2 * (cchi[d] + half) + 1;
            n[d] = (d == 0 ? 4 : 2) + (l[d] << g.r) + (Q[d] >> sb);
            w1[d] = __int_as_float(wexp | (Q[d] & wmask)) - wbase;
            w0[d] = 1.0f - w1[d];
        }
        // CIC gather of the FD4 gradient (56 nodes, read as 28 pairs of
        // x-adjacent nodes {o, o + 1}).  Near a uniform lattice every node
        // index is even, so a warp's loads would use the 16 even banks only; a
        // particle with odd n_y / 2 reads each pair in the other order, which
        // spreads a warp's loads over all 32 banks.  Columns along y and z
        // keep the swapped order and take the matching x weights (ca, cb);
        // rows along x are put back in order.  Two lines at a time in packed
        // FP32 pairs.
        const int base = (n[2] * T + n[1]) * TS + n[0];
        const int sh = (n[1] >> 1) & 1;
        const float* pa = tile + base + sh;
        const float* pb = tile + base + 1 - sh;
        const float ca = sh ? w1[0] : w0[0], cb = sh ? w0[0] : w1[0];   // x weights of the pa, pb values
        float2 gy2 = make_float2(0.0f, 0.0f), gz2 = make_float2(0.0f, 0.0f), gx2 = make_float2(0.0f, 0.0f);
#pragma unroll
        for (int b = 0; b < 2; ++b) {
            float2 r[6];
#pragma unroll
            for (int k = 0; k < 6; ++k) r[k] = make_float2(pa[b * TT + (k - 2) * TS], pb[b * TT + (k - 2) * TS]);
            gy2 = pfma(pk2(b ? w1[2] : w0[2]), fd4_cic_pair(r, w0[1], w1[1]), gy2);   // y columns at z + b
#pragma unroll
            for (int k = 0; k < 6; ++k) r[k] = make_float2(pa[b * TS + (k - 2) * TT], pb[b * TS + (k - 2) * TT]);
            gz2 = pfma(pk2(b ? w1[1] : w0[1]), fd4_cic_pair(r, w0[2], w1[2]), gz2);   // z columns at y + b
            // x rows at (y + a, z + b), a = 0, 1 in the two lanes, in natural order
#pragma unroll
            for (int k = 0; k < 6; k += 2) {
#pragma unroll
                for (int a = 0; a < 2; ++a) {
                    const int o = a * TS + b * TT + (k - 2);
                    const float u = pa[o], v = pb[o];
                    (a ? r[k].y : r[k].x) = sh ? v : u;
                    (a ? r[k + 1].y : r[k + 1].x) = sh ? u : v;
                }
            }
            gx2 = pfma(pmul(make_float2(w0[1], w1[1]), pk2(b ? w1[2] : w0[2])), fd4_cic_pair(r, w0[0], w1[0]), gx2);
        }
        // the gathered sums of 12 dPhi/dx_d; F = -sum / 12 is folded into the kick factor
        const float gsum[3] = {gx2.x + gx2.y, __fmaf_rn(ca, gy2.x, cb * gy2.y), __fmaf_rn(ca, gz2.x, cb * gz2.y)};
        // kick (update_vp): the code is decided on v - v_c + F K = offset + F K,
        // re-encoded against the same v_c; then the drift of the in-cell
        // offset Q / 2^(8n+1) by the decoded momentum, rounded once
        int e[3], nu1[3];
        float pv[3], un[3], dd[3];
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            dd[d] = __fmaf_rn(gsum[d], kick12, NV == 1 ? dec[cnu[d] + lim] : vt.dec(cnu[d]));
            if (NV == 1) nu1[d] = nu_from_table(dd[d], thr, stab, key0, lim);
        }
        if (NV == 2) nu_codes3(dd, cur.thr, lim, e0, e1, nu1);
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            nu_r.put(d, i, nu1[d]);
            const float off1 = NV == 1 ? dec[nu1[d] + lim] : vt.dec(nu1[d]);
            const float p2 = svc[(d << (3 * lB)) + lc] + off1;
            sacc = __fmaf_rn(off1, off1, sacc);
            const int sh1 = drift_bin(Q[d], p2, dcs, &un[d]) >> nbits;
            const int shc = max(-1, min(1, sh1));
            migbad |= sh1 != shc;
            mig |= shc & 1;                        // 1 if the particle changes cell along d
            e[d] = l[d] + shc + 1;
            pv[d] = p2;
        }

        const int ei = e[0] + Bh * (e[1] + Bh * e[2]);
        // per-lane shared-memory atomics (measured faster here than warp aggregation)
        atomicAdd(&hist[ei], 1u);
#pragma unroll
        for (int d = 0; d < 3; ++d)
            smem_add_u64(reinterpret_cast<unsigned*>(&vs[d * H3 + ei]), (unsigned long long)vel_fix(pv[d]));
        if (dbg.cell_old) {
            const int cg[3] = {bx * g.B + l[0], by * g.B + l[1], bz * g.B + l[2]};
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                dbg.cell_old[d * g.Np + i] = cg[d];
                dbg.u_new[d * g.Np + i] = ldexpf(un[d], -nbits);
                dbg.p[d * g.Np + i] = pv[d];
                dbg.force[d * g.Np + i] = gsum[d] * (-1.0f / 12.0f);
            }
        }
    }
    if (migbad) atomicOr(w.flags, ERR_MIGRATION);
    // the block's sum of squared offsets (a fixed tree: each warp's shuffle
    // tree, then the warps in order) and whether any particle changed cell,
    // finished by thread 0 after the barrier that also opens the write-out
    __shared__ float red[PA_T / 32];
    __shared__ unsigned redmig[PA_T / 32];
    {
        float v = sacc;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
        const unsigned wm = __reduce_or_sync(0xffffffffu, (unsigned)mig);
        if ((threadIdx.x & 31) == 0) {
            red[threadIdx.x >> 5] = v;
            redmig[threadIdx.x >> 5] = wm;
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        float tot = 0.0f;
        unsigned mm = 0u;
#pragma unroll
        for (int k = 0; k < PA_T / 32; ++k) {
            tot += red[k];
            mm |= redmig[k];
        }
        w.part[brick] = tot;
        if (mm) atomicMax(w.maxmig, (int)mm);
    }
    // each halo cell's slot in the flattened (cell, brick) order and its cell
    // rank, from the per-axis descriptions staged before the particle loop
    for (int t = threadIdx.x; t < H3; t += blockDim.x) {
        const unsigned h = hist[t];
        int ec[3];
        split3(t, Bh, mBh, ec);
        int64_t slot;
        int L;
        halo_slot(g, axis_desc[ec[0]], axis_desc[Bh + ec[1]], axis_desc[2 * Bh + ec[2]], &slot, &L);
        w.ghost[slot] = h;                                   // every slot has exactly one writer
        if (h) {
#pragma unroll
            for (int d = 0; d < 3; ++d)
                atomicAdd(reinterpret_cast<unsigned long long*>(&w.vsum_new[(int64_t)d * g.Ncc + L]),
                          (unsigned long long)vs[d * H3 + t]);
        }
    }
}

// ------------------------------------------------------------------ new cells
// After the exclusive scan of the flattened histograms, a cell's first slot
// holds offset*[c] and its slots span counts*[c] particles; v_c* = mean
// momentum of the cell's new particles (fixed point).
__device__ __forceinline__ void store_cell(const Geo& g, const StepScratch& w, int L, unsigned off, unsigned cnt,
                                           const long long* vs, unsigned* __restrict__ off_new,
                                           float* __restrict__ vc_new) {
    off_new[L] = off;
    w.counts_new[L] = cnt;
#pragma unroll
    for (int d = 0; d < 3; ++d) vc_new[(int64_t)d * g.Ncc + L] = vel_unfix_mean(vs[d], cnt);
}
// the end of the offsets, checked against the particle count
__device__ __forceinline__ void store_total(const Geo& g, const StepScratch& w, unsigned total,
                                            unsigned* __restrict__ off_new) {
    off_new[g.Ncc] = total;
    if (total != (unsigned)g.Np) atomicOr(w.flags, ERR_COUNT);
}

// the cells of a batch (blockIdx.y its slot)
__global__ void k_cells(Geo g, StepScratch w, unsigned* __restrict__ off_new, float* __restrict__ vc_new, Batch bt) {
    chain_wait();
    const int L = blockIdx.x * blockDim.x + threadIdx.x;
    if (L >= g.Ncc || (bt.ms && !bt.ms[blockIdx.y].active)) return;
    const int m = slot_member(bt, blockIdx.y);
    w = moved(w, m * bt.stride);
    off_new = moved(off_new, m * bt.stride);
    vc_new = moved(vc_new, m * bt.stride);
    const int lc = L & ((1 << (3 * g.lB)) - 1), bm = g.B - 1;
    const int l[3] = {lc & bm, (lc >> g.lB) & bm, lc >> (2 * g.lB)};
    const int64_t base = flat_base(g, L >> (3 * g.lB), l);
    const int n = ncand(l[0], g.B) * ncand(l[1], g.B) * ncand(l[2], g.B);
    const long long vs[3] = {w.vsum_new[L], w.vsum_new[(int64_t)g.Ncc + L], w.vsum_new[2 * (int64_t)g.Ncc + L]};
    const unsigned off = w.ghost[base];
    store_cell(g, w, L, off, w.ghost[base + n] - off, vs, off_new, vc_new);
    if (L == g.Ncc - 1) store_total(g, w, w.ghost[(int64_t)g.nbricks * (g.Bh * g.Bh * g.Bh)], off_new);
}

// A single context's step runs two kernels between its passes, over tiles of
// whole bricks (16, 64 or 128 of them: at most 4096 histogram slots, eight a
// thread, and 1024 cells, two a thread): k_step_sums adds each tile's slots up, k_step_cells starts from the
// sum of the tiles before its own (of many tiles, where that would add up tiles^2 / 2
// words, from a scan of the tile sums), scans its slots in place and, with the
// scanned values in shared memory, finishes the cells of its bricks.  The
// codec rides along: one block of the first kernel finds the next scale, a few
// blocks of the second build its tables.  Eight launches before (scale,
// tables, four of the scan, cells, and the clearing of the momentum sums, now
// in the deposit), each a few microseconds of launch and drain and the cells
// a second pass over the histograms: per step (with the clearing) 51 us at 32^3
// particles and 125 us at 256^3 -> 23 and 70 us.
constexpr int SC_T = 512, SC_ITEMS = 8;
__host__ __device__ __forceinline__ int tile_bricks(const Geo& g) { return g.B == 4 ? 16 : g.B == 2 ? 64 : 128; }
__host__ __device__ __forceinline__ int step_tiles(const Geo& g) {
    return (g.nbricks + tile_bricks(g) - 1) / tile_bricks(g);
}

// the eight slots of this thread in tile `tile` (zero past the last brick), of *count
__device__ __forceinline__ void tile_slots(const Geo& g, const unsigned* __restrict__ ghost, int tile, int* count,
                                           unsigned* v) {
    const int S3 = g.Bh * g.Bh * g.Bh, tb = tile_bricks(g);
    const int n = min(tb, g.nbricks - tile * tb) * S3, i = SC_ITEMS * (int)threadIdx.x;
    const unsigned* p = ghost + (int64_t)tile * tb * S3 + i;     // 16-byte aligned: tb S3 is a multiple of 4
    *count = n;
    if (i + SC_ITEMS <= n) {
        const uint4 a = reinterpret_cast<const uint4*>(p)[0], b = reinterpret_cast<const uint4*>(p)[1];
        v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
        v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
    } else {
#pragma unroll
        for (int k = 0; k < SC_ITEMS; ++k) v[k] = i + k < n ? p[k] : 0u;
    }
}

__global__ void __launch_bounds__(1024) k_step_sums(Geo g, StepScratch w, double ratio, double* sigma_out,
                                                    unsigned* __restrict__ tsum) {
    chain_wait();
    if (blockIdx.x == 0) {
        sigma_body<false>(w.part, g.nbricks, 3.0 * (double)g.Np, ratio, 0.0, sigma_out);
        return;
    }
    __shared__ unsigned sw[32];
    // two tiles a block, 512 threads each
    const int tile = 2 * ((int)blockIdx.x - 1) + ((int)threadIdx.x >= SC_T), t = threadIdx.x & (SC_T - 1);
    const int S3 = g.Bh * g.Bh * g.Bh, tb = tile_bricks(g);
    const int n = max(0, min(tb, g.nbricks - tile * tb)) * S3;
    const unsigned* p = w.ghost + (int64_t)tile * tb * S3;
    unsigned s = 0;
    for (int i = 4 * t; i < n; i += 4 * SC_T) {
        if (i + 3 < n) {
            const uint4 q = *reinterpret_cast<const uint4*>(p + i);
            s += q.x + q.y + q.z + q.w;
        } else {
            for (int k = i; k < n; ++k) s += p[k];
        }
    }
    s = __reduce_add_sync(0xffffffffu, s);
    if ((threadIdx.x & 31) == 0) sw[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x < 32) {
        s = sw[threadIdx.x];
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if ((threadIdx.x & 15) == 0) {
            const int k = 2 * ((int)blockIdx.x - 1) + ((int)threadIdx.x >> 4);
            if (k < step_tiles(g)) tsum[k] = s;
        }
    }
}

__global__ void __launch_bounds__(SC_T) k_step_cells(Geo g, StepScratch w, const unsigned* __restrict__ tsum,
                                                     unsigned* __restrict__ off_new, float* __restrict__ vc_new,
                                                     const double* __restrict__ tanv, const double* __restrict__ tanh_,
                                                     CodecDev next, int ntab, bool scanned) {
    chain_wait();
    if ((int)blockIdx.x < ntab) {                            // the next codec's tables
        codec_tables_body(g.nulim, tanv, tanh_, *next.sigma, next.dec, next.thr, next.est,
                          g.nnu == 1 ? next.vtab : nullptr, g.nnu == 1 ? nullptr : next.vdel, blockIdx.x, ntab);
        return;
    }
    __shared__ unsigned sw[32];
    __shared__ __align__(16) unsigned ex[SC_ITEMS * SC_T + 4];   // the tile's scanned slots and their end
    const int tile = blockIdx.x - ntab, tb = tile_bricks(g), S3 = g.Bh * g.Bh * g.Bh;
    const int nbc = 1 << (3 * g.lB), L0 = tile * tb * nbc, bm = g.B - 1;
    unsigned v[SC_ITEMS];
    int n;
    tile_slots(g, w.ghost, tile, &n, v);
    const int ncell = (n / S3) * nbc;
    // the momentum sums of this thread's cells (at most two), in flight during the scan
    long long vs[2][3];
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            const int c = (int)threadIdx.x + h * SC_T;
            vs[h][d] = c < ncell ? w.vsum_new[(int64_t)d * g.Ncc + L0 + c] : 0;
        }
    unsigned before = 0;
    if (scanned) before = threadIdx.x == 0 ? tsum[tile] : 0u;
    else
        for (int j = threadIdx.x; j < tile; j += SC_T) before += tsum[j];
    unsigned s = 0;
#pragma unroll
    for (int k = 0; k < SC_ITEMS; ++k) s += v[k];
    unsigned start, total;
    block_inclusive_scan(before, sw, &start);
    unsigned e = start + block_inclusive_scan(s, sw, &total) - s;
#pragma unroll
    for (int k = 0; k < SC_ITEMS; ++k) {
        const unsigned c = v[k];
        v[k] = e;
        e += c;
    }
    const int i = SC_ITEMS * (int)threadIdx.x;
    *reinterpret_cast<uint4*>(&ex[i]) = make_uint4(v[0], v[1], v[2], v[3]);
    *reinterpret_cast<uint4*>(&ex[i + 4]) = make_uint4(v[4], v[5], v[6], v[7]);
    if (threadIdx.x == 0) ex[SC_ITEMS * SC_T] = start + total;
    __syncthreads();
    // coalesced write-back; slots past the last are zero, so ex[n] holds the end as well
    unsigned* p = w.ghost + (int64_t)tile * tb * S3;
    for (int k = 4 * (int)threadIdx.x; k < n; k += 4 * SC_T) {
        if (k + 3 < n) *reinterpret_cast<uint4*>(p + k) = *reinterpret_cast<const uint4*>(&ex[k]);
        else
            for (int j = k; j < n; ++j) p[j] = ex[j];
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int c = (int)threadIdx.x + h * SC_T;
        if (c >= ncell) continue;
        const int lc = c & (nbc - 1);
        const int l[3] = {lc & bm, (lc >> g.lB) & bm, lc >> (2 * g.lB)};
        const int base = (int)flat_base(g, c >> (3 * g.lB), l);
        const int k = ncand(l[0], g.B) * ncand(l[1], g.B) * ncand(l[2], g.B);
        store_cell(g, w, L0 + c, ex[base], ex[base + k] - ex[base], vs[h], off_new, vc_new);
    }
    if (threadIdx.x == 0 && L0 + ncell == g.Ncc) store_total(g, w, start + total, off_new);
}

// ------------------------------------------------------------------ pass B
// Two splits, chosen by passB_all:
//
// Large stores: one warp per brick (8 bricks per CTA).
// The brick's particles are taken 32 at a time in index order; lanes moving
// to the same cell get consecutive slots in lane order from the cell's running
// start (match + popc), so the new order within a cell is the old index
// order.  No block barriers.  A brick holding more than PB_BIG particles
// (clustering: late epochs reach ~30x the mean) would make its warp the
// kernel's tail: pass A lists those bricks and the first CTAs of the grid take
// them whole.
//
// A whole CTA per brick, 256 particles per round: each warp's per-cell counts
// go to a shared table, and a lane's slot is the cell's running start + the
// counts of the lower warps + its rank in its warp, which is again the old
// index order.  Small stores take it because a warp's chain of 16 rounds is
// the whole kernel there, and bricks of side 4 with 2-byte velocities, whose
// rounds wait for their table reads.  Measured, us (warp a brick / CTA a brick), x1v1:
// 64 bricks 25.9 / 10.2, 512: 27.2 / 14.3, 1728: 30.0 / 27.0, 4096: 45.6 /
// 52.6, 13824: 102 / 159; x2v2: 64: 67 / 16, 512: 70 / 20, 1728: 78 / 42,
// 4096: 122 / 81, 13824: 367 / 250, 32768: 770 / 565.
constexpr int PB_WARPS = 8;

// what pass B needs of one particle: its new cell in the brick's halo
// region (ei), new position code and momentum
struct PbParticle {
    int ei;
    int chi[3];
    float pv[3];
};

// PID: 4 for 4-byte particle IDs (or none), 0 for the narrow widths of Geo::nid
template <int NX, int NV, int PID>
struct PassB {
    Geo g;
    const StoreDev& sn;
    CodeRows<NX> chi_n;
    CodeRows<NV> nu_n;
    const float* dec;
    const float* thr;
    const unsigned char* stab;
    int key0, lim;
    float dcs, e0, e1;     // dcs: the drift factor in bins of the position code (dc 2^(8n))

    // lc: the particle's coarse cell in the brick
    __device__ __forceinline__ PbParticle move(int lc, const float* svc, const int* cchi, const int* cnu) const {
        const int Bh = g.Bh;
        const int nbits = 8 * NX, half = 1 << (nbits - 1), bmask = (1 << nbits) - 1;
        const int l[3] = {lc & (g.B - 1), (lc >> g.lB) & (g.B - 1), lc >> (2 * g.lB)};
        PbParticle r;
        int e[3];
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            const int Q = 2 * (cchi[d] + half) + 1;
            const float p2 = svc[(d << (3 * g.lB)) + lc] + dec[cnu[d] + lim];
            float x;
            const int bin = drift_bin(Q, p2, dcs, &x);
            const int sh = max(-1, min(1, bin >> nbits));
            e[d] = l[d] + sh + 1;
            r.chi[d] = (bin & bmask) - half;
            r.pv[d] = p2;
        }
        r.ei = e[0] + Bh * (e[1] + Bh * e[2]);
        return r;
    }

    __device__ __forceinline__ void put(const PbParticle& q, const float* svn, unsigned pos, unsigned cid,
                                        unsigned* flags) const {
        const int H3 = g.Bh * g.Bh * g.Bh;
        if (pos >= (unsigned)g.Np) {
            atomicOr(flags, ERR_COUNT);
            return;
        }
        float dd[3];
        int nu[3];
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            chi_n.put(d, pos, q.chi[d]);
            dd[d] = q.pv[d] - svn[d * H3 + q.ei];
            if (NV == 1) nu[d] = nu_from_table(dd[d], thr, stab, key0, lim);
        }
        if (NV == 2) nu_codes3(dd, thr, lim, e0, e1, nu);
#pragma unroll
        for (int d = 0; d < 3; ++d) nu_n.put(d, pos, nu[d]);
        if (sn.id) {
            if (PID == 4) reinterpret_cast<unsigned*>(sn.id)[pos] = cid;
            else store_pid(sn.id, pos, g.nid, cid);
        }
    }
};

// brick offsets, v_c of the brick, running starts of the halo cells (this
// brick's slots of the scanned histograms) and v_c* of the halo region,
// staged by `nthr` threads from thread `t0`
__device__ __forceinline__ void passB_stage(const Geo& g, const StoreDev& so, const unsigned* __restrict__ ghost,
                                            const float* __restrict__ vc_new, int brick, int t0, int nthr,
                                            unsigned* sm_off, unsigned* run, float* svc, float* svn) {
    const int nbc = g.B * g.B * g.B, Bh = g.Bh, H3 = Bh * Bh * Bh;
    const unsigned mBh = div_magic(Bh);
    const int L0 = brick * nbc;
    int bx, by, bz;
    brick_coords(g, brick, &bx, &by, &bz);
    const int bc[3] = {bx, by, bz};
    for (int c = t0; c <= nbc; c += nthr) sm_off[c] = so.offsets[L0 + c];
    for (int t = t0; t < 3 * nbc; t += nthr) svc[t] = so.vc[(int64_t)(t >> (3 * g.lB)) * g.Ncc + L0 + (t & (nbc - 1))];
    // the 3 Bh (<= 18) per-axis descriptions of the halo coordinates, one per
    // lane of every warp, read by the others through shuffles
    const int lane = threadIdx.x & 31;
    unsigned dsc = 0u;
    if (lane < 3 * Bh) {
        const int d = lane / Bh;
        dsc = halo_axis_desc(g, bc[d], lane - d * Bh);
    }
    for (int base = t0 - lane; base < H3; base += nthr) {     // warp-uniform bounds
        const int t = base + lane;
        int e[3];
        split3(min(t, H3 - 1), Bh, mBh, e);
        const unsigned ax = __shfl_sync(0xffffffffu, dsc, e[0]);
        const unsigned ay = __shfl_sync(0xffffffffu, dsc, Bh + e[1]);
        const unsigned az = __shfl_sync(0xffffffffu, dsc, 2 * Bh + e[2]);
        if (t < H3) {
            int64_t slot;
            int L;
            halo_slot(g, ax, ay, az, &slot, &L);
            run[t] = ghost[slot];
#pragma unroll
            for (int d = 0; d < 3; ++d) svn[d * H3 + t] = vc_new[(int64_t)d * g.Ncc + L];
        }
    }
}

// One brick by the whole CTA, blockDim.x = 256 particles a round.  Shared
// words `sm`: [nbc + 1] offsets, [H3] running starts, [3][nbc] v_c, [3][H3]
// v_c*, [PB_WARPS][H3] per-warp cell counts.
template <int NX, int NV, int PID>
__device__ __forceinline__ void passB_cta_brick(const Geo& g, const PassB<NX, NV, PID>& pb, const StoreDev& so,
                                                const unsigned* __restrict__ ghost, const float* __restrict__ vc_new,
                                                int brick, unsigned* sm, unsigned* flags) {
    const int nbc = g.B * g.B * g.B, H3 = g.Bh * g.Bh * g.Bh, lim = g.nulim;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const CodeRows<NX> chi_o(so.chi, g.Np);
    const CodeRows<NV> nu_o(so.nu, g.Np);
    unsigned* sm_off = sm;
    unsigned* run = sm_off + nbc + 1;
    float* svc = reinterpret_cast<float*>(run + H3);
    float* svn = svc + 3 * nbc;
    unsigned* wcnt = reinterpret_cast<unsigned*>(svn + 3 * H3);
    // a round's codes and id, requested a round ahead (the first beside the staging)
    const unsigned p1 = min(so.offsets[brick * nbc + nbc], (unsigned)g.Np), p0 = min(so.offsets[brick * nbc], p1);
    int nchi[3] = {0, 0, 0}, nnu[3] = {0, 0, 0};
    unsigned nid = 0;
    auto fetch = [&](unsigned i) {
        if (i >= p1) return;
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            nchi[d] = chi_o.get(d, i);
            nnu[d] = nu_o.get(d, i);
        }
        if (pb.sn.id) nid = PID == 4 ? reinterpret_cast<const unsigned*>(so.id)[i] : load_pid(so.id, i, g.nid);
    };
    fetch(p0 + threadIdx.x);
    __syncthreads();                         // a previous brick's tables are no longer read
    for (int t = threadIdx.x; t < PB_WARPS * H3; t += blockDim.x) wcnt[t] = 0u;
    passB_stage(g, so, ghost, vc_new, brick, threadIdx.x, blockDim.x, sm_off, run, svc, svn);
    __syncthreads();
    for (unsigned base = p0; base < p1; base += blockDim.x) {
        const unsigned i = base + threadIdx.x;
        const bool act = i < p1;
        const unsigned am = __ballot_sync(0xffffffffu, act);
        PbParticle q{};
        unsigned peers = 0;
        const unsigned cid = nid;
        int leader = 0;
        if (act) {
            int cchi[3], cnu[3];
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                cchi[d] = nchi[d];
                cnu[d] = max(-lim, min(lim, nnu[d]));
            }
            fetch(i + blockDim.x);
            q = pb.move(upper_cell(sm_off, nbc, i), svc, cchi, cnu);
            peers = __match_any_sync(am, q.ei);
            leader = __ffs(peers) - 1;
            if (lane == leader) wcnt[warp * H3 + q.ei] = (unsigned)__popc(peers);
        }
        __syncthreads();
        unsigned start = 0, total = 0;
        bool last = true;
        if (act) {
            if (lane == leader) {
                start = run[q.ei];
#pragma unroll
                for (int v = 0; v < PB_WARPS; ++v) {
                    const unsigned c = wcnt[v * H3 + q.ei];
                    if (v < warp) start += c;
                    if (v > warp && c) last = false;
                    total += c;
                }
            }
            start = __shfl_sync(peers, start, leader);
        }
        __syncthreads();                     // every read of run and wcnt is done
        if (act) {
            if (lane == leader) {
                if (last) run[q.ei] += total;
                wcnt[warp * H3 + q.ei] = 0u;
            }
            pb.put(q, svn, start + (unsigned)__popc(peers & ((1u << lane) - 1u)), cid, flags);
        }
    }
}

// the split of pass B: a CTA per brick when the bricks' warps would fill less
// than 40% of the 40 resident per SM, or with 2-byte velocities when a brick
// holds some warps' worth of particles (bricks of side 4; a smaller brick's few
// particles leave most of a CTA idle: the step of 128^3 particles x2v2 with
// bricks of 8 cells takes 622 us by warps, of 64 cells 359 us by CTAs)
static bool passB_all(const Geo& g, int members) {
    return (int64_t)g.nbricks * members <= 16 * (int64_t)g.nsm || (g.nnu == 2 && g.Np >= 96 * (int64_t)g.nbricks);
}

// ALL: every brick by a whole CTA
template <int NX, int NV, bool BAT, int PID, bool ALL>
__global__ void __launch_bounds__(PB_WARPS * 32, 5) k_passB(Geo g, StoreDev so, StoreDev sn, CodecDev cur, CodecDev next,
                                                        float dc, const unsigned* __restrict__ ghost,
                                                        const float* __restrict__ vc_new, unsigned* flags,
                                                        const int* __restrict__ big, int nbig_ctas, Batch bt) {
    extern __shared__ unsigned pb_smem[];
    chain_wait();
    const int nbc = g.B * g.B * g.B, H3 = g.Bh * g.Bh * g.Bh;
    const int lim = g.nulim;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if constexpr (BAT) {                                     // slot blockIdx.y of a batch
        const int slot = blockIdx.y;
        if (bt.ms) {
            if (!bt.ms[slot].active) return;
            dc = bt.ms[slot].dc;
        }
        const size_t o = slot_member(bt, slot) * bt.stride;
        so = moved(so, o);
        sn = moved(sn, o);
        cur = moved(cur, o);
        next = moved(next, o);
        ghost = moved(ghost, o);
        vc_new = moved(vc_new, o);
        flags = moved(flags, o);
        big = moved(big, o);
    }
    const bool big_cta = !ALL && (int)blockIdx.x < nbig_ctas;
    const int nbig = big_cta ? big[0] : 0;
    if (big_cta && (int)blockIdx.x >= nbig) return;          // no crowded brick left for this CTA
    float* sdec = reinterpret_cast<float*>(pb_smem);                       // NV == 1: [2 lim + 1]
    float* sthr = sdec + (NV == 1 ? 2 * lim + 1 : 0);                       // NV == 1: [lim + 2]
    unsigned char* stab = reinterpret_cast<unsigned char*>(sthr + (NV == 1 ? lim + 2 : 0));   // NV == 1: [VT_N]
    unsigned* wbase = reinterpret_cast<unsigned*>(stab + (NV == 1 ? VT_N : 0));
    // (2-byte codes read the full tables here: the compact form of pass A
    // costs pass B more in instructions than its loads cost in latency)
    PassB<NX, NV, PID> pb{g, sn, CodeRows<NX>(sn.chi, g.Np), CodeRows<NV>(sn.nu, g.Np), cur.dec, next.thr, stab, 0, lim,
                     ldexpf(dc, 8 * NX), next.est[0], next.est[1]};
    const CodeRows<NX> chi_o(so.chi, g.Np);
    const CodeRows<NV> nu_o(so.nu, g.Np);
    if (NV == 1) {
        for (int t = threadIdx.x; t < 2 * lim + 1; t += blockDim.x) sdec[t] = cur.dec[t];
        for (int t = threadIdx.x; t < lim + 2; t += blockDim.x) sthr[t] = next.thr[t];
        for (int t = threadIdx.x; t < VT_N / 4; t += blockDim.x)
            reinterpret_cast<unsigned*>(stab)[t] = reinterpret_cast<const unsigned*>(next.vtab)[t];
        pb.dec = sdec;
        pb.thr = sthr;
        pb.key0 = __float_as_int(next.est[2]);
    }
    if constexpr (ALL) {
        passB_cta_brick<NX, NV, PID>(g, pb, so, ghost, vc_new, blockIdx.x, wbase, flags);
    } else {
        if (big_cta) {
            for (int k = blockIdx.x; k < nbig; k += nbig_ctas)
                passB_cta_brick<NX, NV, PID>(g, pb, so, ghost, vc_new, big[1 + k], wbase, flags);
            return;
        }
        __syncthreads();
        const int brick = ((int)blockIdx.x - nbig_ctas) * PB_WARPS + warp;
        if (brick >= g.nbricks) return;
        const int L0 = brick * nbc;
        const unsigned p1 = min(so.offsets[L0 + nbc], (unsigned)g.Np), p0 = min(so.offsets[L0], p1);
        if (p1 - p0 > (unsigned)PB_BIG) return;              // a crowded brick: taken by a whole CTA
        unsigned* sm_off = wbase + warp * (4 * nbc + 1 + 4 * H3);               // [nbc + 1] per warp
        unsigned* run = sm_off + nbc + 1;                                       // [H3] per warp
        float* svc = reinterpret_cast<float*>(run + H3);                        // [3][nbc]: v_c of the brick
        float* svn = svc + 3 * nbc;                                             // [3][H3]: v_c* of the halo region
        // the first round's codes and ids first, so their latency overlaps the staging
        int nchi[3] = {0, 0, 0}, nnu[3] = {0, 0, 0};
        unsigned nid = 0;
        if (p0 + lane < p1) {
    #pragma unroll
            for (int d = 0; d < 3; ++d) {
                nchi[d] = chi_o.get(d, p0 + lane);
                nnu[d] = nu_o.get_nu(d, p0 + lane, lim);
            }
            if (sn.id)
                nid = PID == 4 ? reinterpret_cast<const unsigned*>(so.id)[p0 + lane] : load_pid(so.id, p0 + lane, g.nid);
        }
        passB_stage(g, so, ghost, vc_new, brick, lane, 32, sm_off, run, svc, svn);
        __syncwarp();
        int c0 = upper_cell(sm_off, nbc, p0);      // the cell of each round's first particle
        for (unsigned base = p0; base < p1; base += 32) {
            const unsigned i = base + lane;
            const bool act = i < p1;
            const unsigned am = __ballot_sync(0xffffffffu, act);
            // this round's codes; the next round's are requested now
            const int cchi[3] = {nchi[0], nchi[1], nchi[2]}, cnu[3] = {nnu[0], nnu[1], nnu[2]};
            const unsigned cid = nid;
            if (i + 32 < p1) {
    #pragma unroll
                for (int d = 0; d < 3; ++d) {
                    nchi[d] = chi_o.get(d, i + 32);
                    nnu[d] = nu_o.get_nu(d, i + 32, lim);
                }
                if (sn.id)
                    nid = PID == 4 ? reinterpret_cast<const unsigned*>(so.id)[i + 32] : load_pid(so.id, i + 32, g.nid);
            }
            int cnext;
            const int lcell = warp_cells(sm_off, nbc, base, c0, &cnext);
            c0 = cnext;
            if (act) {
                const PbParticle q = pb.move(lcell, svc, cchi, cnu);
                const unsigned peers = __match_any_sync(am, q.ei);
                const int leader = __ffs(peers) - 1;
                unsigned start = 0;
                if (lane == leader) start = run[q.ei];
                start = __shfl_sync(peers, start, leader);
                if (lane == leader) run[q.ei] = start + (unsigned)__popc(peers);
                pb.put(q, svn, start + (unsigned)__popc(peers & ((1u << lane) - 1u)), cid, flags);
            }
            __syncwarp();
        }
    }
}

// Global sums of the current store (Section 2.3.3's bookkeeping): the
// momenta exactly as cube_decode returns them (v_c + decoded offset, FP32),
// each rounded to a multiple of 2^-24 and summed exactly in int64, so the
// result is independent of the summation order and within N 2^-25 of the
// exact sum of the decoded values; and the particle count as the sum of the
// cell counts.  One CTA per brick, one 64-bit atomic per warp and quantity.
template <int NV>
__global__ void __launch_bounds__(T_BRICK) k_store_sums(Geo g, StoreDev s, const float* __restrict__ dec,
                                                        long long* __restrict__ out4) {
    extern __shared__ unsigned sm_off[];
    const int nbc = g.B * g.B * g.B;
    const int L0 = blockIdx.x * nbc;
    for (int c = threadIdx.x; c <= nbc; c += blockDim.x) sm_off[c] = s.offsets[L0 + c];
    long long cnt = 0;
    for (int c = threadIdx.x; c < nbc; c += blockDim.x) cnt += s.counts[L0 + c];
    __syncthreads();
    const unsigned q1 = min(sm_off[nbc], (unsigned)g.Np);
    long long m[3] = {0, 0, 0};
    for (unsigned i = min(sm_off[0], q1) + threadIdx.x; i < q1; i += blockDim.x) {
        const int lc = upper_cell(sm_off, nbc, i);
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            const int nu = load_nu<NV>(s.nu, d * g.Np + i, g.nulim);
            m[d] += vel_fix(s.vc[(int64_t)d * g.Ncc + L0 + lc] + dec[nu + g.nulim]);
        }
    }
    // warp sums, then the block's in shared memory, then one atomic per sum and block
    __shared__ long long part[4][T_BRICK / 32];
    long long v[4] = {m[0], m[1], m[2], cnt};
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v[k] += __shfl_down_sync(0xffffffffu, v[k], o);
        if (lane == 0) part[k][wid] = v[k];
    }
    __syncthreads();
    if (threadIdx.x < 4) {
        long long t = 0;
        for (int i = 0; i < (int)(blockDim.x >> 5); ++i) t += part[threadIdx.x][i];
        if (t) atomicAdd(reinterpret_cast<unsigned long long*>(&out4[threadIdx.x]), (unsigned long long)t);
    }
}

template <int NX, int NV>
struct Disp {
    static void passA(const Geo& g, const StoreDev& s, const float* phig, const CUtensorMap& tmap, int use_tma,
                      const CodecDev& cur, float kick, float dc, const StepScratch& w, const DriftDebug& dbg,
                      size_t sm, cudaStream_t st, const Batch& bt) {
        const dim3 grid(g.nb, g.nb, g.nb * bt.members);
        const bool bat = bt.members > 1 || bt.ms;
        if (g.F == 16) {
            if (bat) launch_chained(k_passA<NX, NV, 16, true>, grid, PA_T, sm, st, g, s, phig, tmap, use_tma, cur, kick, dc, w, dbg, bt);
            else launch_chained(k_passA<NX, NV, 16, false>, grid, PA_T, sm, st, g, s, phig, tmap, use_tma, cur, kick, dc, w, dbg, bt);
        } else {
            if (bat) launch_chained(k_passA<NX, NV, 0, true>, grid, PA_T, sm, st, g, s, phig, tmap, use_tma, cur, kick, dc, w, dbg, bt);
            else launch_chained(k_passA<NX, NV, 0, false>, grid, PA_T, sm, st, g, s, phig, tmap, use_tma, cur, kick, dc, w, dbg, bt);
        }
    }
    static void passB(const Geo& g, const StoreDev& so, const StoreDev& sn, const CodecDev& cur,
                      const CodecDev& next, float dc, const unsigned* ghost, const float* vcn, unsigned* flags,
                      const int* big, size_t sm, size_t sm_cta, cudaStream_t st, const Batch& bt) {
        const bool narrow = g.nid == 1 || g.nid == 2, bat = bt.members > 1 || bt.ms;
        if (passB_all(g, bt.members)) {
            const dim3 gb(g.nbricks, bt.members);
            if (bat && narrow) launch_chained(k_passB<NX, NV, true, 0, true>, gb, PB_WARPS * 32, sm_cta, st, g, so, sn, cur, next, dc, ghost, vcn, flags, big, 0, bt);
            else if (bat) launch_chained(k_passB<NX, NV, true, 4, true>, gb, PB_WARPS * 32, sm_cta, st, g, so, sn, cur, next, dc, ghost, vcn, flags, big, 0, bt);
            else if (narrow) launch_chained(k_passB<NX, NV, false, 0, true>, gb, PB_WARPS * 32, sm_cta, st, g, so, sn, cur, next, dc, ghost, vcn, flags, big, 0, bt);
            else launch_chained(k_passB<NX, NV, false, 4, true>, gb, PB_WARPS * 32, sm_cta, st, g, so, sn, cur, next, dc, ghost, vcn, flags, big, 0, bt);
            return;
        }
        // CTAs for crowded bricks first (at most Np / (PB_BIG + 1) of them exist)
        const int nbig_ctas = (int)std::min<int64_t>(2 * g.nsm, g.Np / (PB_BIG + 1));
        const dim3 gb(nbig_ctas + (g.nbricks + PB_WARPS - 1) / PB_WARPS, bt.members);
        if (bat && narrow) launch_chained(k_passB<NX, NV, true, 0, false>, gb, PB_WARPS * 32, sm, st, g, so, sn, cur, next, dc, ghost, vcn, flags, big, nbig_ctas, bt);
        else if (bat) launch_chained(k_passB<NX, NV, true, 4, false>, gb, PB_WARPS * 32, sm, st, g, so, sn, cur, next, dc, ghost, vcn, flags, big, nbig_ctas, bt);
        else if (narrow) launch_chained(k_passB<NX, NV, false, 0, false>, gb, PB_WARPS * 32, sm, st, g, so, sn, cur, next, dc, ghost, vcn, flags, big, nbig_ctas, bt);
        else launch_chained(k_passB<NX, NV, false, 4, false>, gb, PB_WARPS * 32, sm, st, g, so, sn, cur, next, dc, ghost, vcn, flags, big, nbig_ctas, bt);
    }
};

template <int NX, int NV>
void set_smem_attrs() {
    static bool done = false;
    if (done) return;
    const int lim = 200 * 1024;
    cudaFuncSetAttribute(k_passA<NX, NV, 0, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
    cudaFuncSetAttribute(k_passA<NX, NV, 16, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
    cudaFuncSetAttribute(k_passA<NX, NV, 0, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
    cudaFuncSetAttribute(k_passA<NX, NV, 16, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
    cudaFuncSetAttribute(k_passB<NX, NV, false, 4, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
    cudaFuncSetAttribute(k_passB<NX, NV, true, 4, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
    cudaFuncSetAttribute(k_passB<NX, NV, false, 0, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
    cudaFuncSetAttribute(k_passB<NX, NV, true, 0, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
    cudaFuncSetAttribute(k_deposit<NX, 0, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
    cudaFuncSetAttribute(k_deposit<NX, 16, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
    cudaFuncSetAttribute(k_deposit<NX, 0, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
    cudaFuncSetAttribute(k_deposit<NX, 16, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
    done = true;
}

// one word of every listed member of a batch set to zero
__global__ void k_zero_slot_words(unsigned* p, Batch bt) {
    chain_wait();
    for (int i = threadIdx.x; i < bt.members; i += blockDim.x) moved(p, slot_member(bt, i) * bt.stride)[0] = 0u;
}

// every entry of the 2-byte decode table as VelTables rebuilds it, and the
// codes of nu_codes3 at and just below every threshold, of a NaN, of infinity and of 0, against the tables
__global__ void k_check_vel_tables(int lim, CodecDev c, long long* out2) {
    const VelTables vt = vel_tables<2>(c, lim);
    long long bad = 0, whole = 0;
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k <= lim; k += gridDim.x * blockDim.x) {
        bad += __float_as_int(vt.dec(k)) != __float_as_int(c.dec[lim + k]);
        bad += k > 0 && __float_as_int(vt.dec(-k)) != __float_as_int(c.dec[lim - k]);
        whole += c.vdel[k] == -128;
        if (k > 0) {
            const float t = c.thr[k], below = __int_as_float(__float_as_int(t) - 1);
            const float d[3] = {t, -t, below};
            int nu[3];
            nu_codes3(d, c.thr, lim, c.est[0], c.est[1], nu);
            bad += nu[0] != k || nu[1] != -k || nu[2] != k - 1;
        } else {
            const float nan = __int_as_float(0x7fffffff), inf = __int_as_float(0x7f800000), d[3] = {nan, -inf, 0.0f};
            int nu[3];
            nu_codes3(d, c.thr, lim, c.est[0], c.est[1], nu);
            bad += nu[0] != 0 || nu[1] != -lim || nu[2] != 0;
        }
    }
    block_sum_to(bad, &out2[0]);
    block_sum_to(whole, &out2[1]);
}

// the step's cleared scratch of every stepped member of a batch: the
// fixed-point momentum sums [3][Ncc] and the migration / crowded-brick words
__global__ void k_batch_clear(int64_t n64, long long* __restrict__ vsum, int* __restrict__ mig, Batch bt) {
    chain_wait();
    if (bt.ms && !bt.ms[blockIdx.y].active) return;
    const int m = slot_member(bt, blockIdx.y);
    vsum = moved(vsum, m * bt.stride);
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < n64; t += (int64_t)gridDim.x * blockDim.x)
        vsum[t] = 0;
    if (blockIdx.x == 0 && threadIdx.x < 2) moved(mig, m * bt.stride)[threadIdx.x] = 0;
}

__global__ void __launch_bounds__(256) k_section_copy(const __grid_constant__ SectionCopy c) {
    const int64_t t0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, nt = (int64_t)gridDim.x * blockDim.x;
    if (blockIdx.x == 0) {
        if (c.header_to && threadIdx.x < 16) {
            unsigned w = c.header[threadIdx.x];
            if (threadIdx.x >= 14 && c.sigma_from) w = reinterpret_cast<const unsigned*>(c.sigma_from)[threadIdx.x - 14];
            reinterpret_cast<unsigned*>(c.header_to)[threadIdx.x] = w;
        }
        if (c.sigma_to && threadIdx.x == 0) *c.sigma_to = c.sigma;
        if ((int)threadIdx.x < c.nzero) c.zero[threadIdx.x] = 0u;
        if (c.zero64 && threadIdx.x < 2) c.zero64[threadIdx.x] = 0;
    }
    for (int s = 0; s < c.n; ++s) {
        const int64_t q = c.bytes[s] >> 4;
        const uint4* a = reinterpret_cast<const uint4*>(c.src[s]);
        uint4* b = reinterpret_cast<uint4*>(c.dst[s]);
        int64_t i = t0;
        for (; i + 3 * nt < q; i += 4 * nt) {                // four 16-byte loads in flight
            const uint4 v0 = a[i], v1 = a[i + nt], v2 = a[i + 2 * nt], v3 = a[i + 3 * nt];
            b[i] = v0;
            b[i + nt] = v1;
            b[i + 2 * nt] = v2;
            b[i + 3 * nt] = v3;
        }
        for (; i < q; i += nt) b[i] = a[i];
        if (t0 < (c.bytes[s] & 15)) c.dst[s][16 * q + t0] = c.src[s][16 * q + t0];
    }
}

}  // namespace

// ------------------------------------------------------------------ launchers
void launch_section_copy(const SectionCopy& c, cudaStream_t st) {
    int64_t total = 0;
    for (int s = 0; s < c.n; ++s) total += c.bytes[s];
    const int64_t nb = (total / 64 + 255) / 256;
    k_section_copy<<<(unsigned)std::min<int64_t>(152 * 8, std::max<int64_t>(1, nb)), 256, 0, st>>>(c);
}

void launch_batch_clear(const Geo& g, long long* vsum, int* maxmig, cudaStream_t st, const Batch& bt) {
    const int64_t n = 3 * (int64_t)g.Ncc;
    launch_chained(k_batch_clear, dim3((unsigned)std::min<int64_t>(1024, (n + 255) / 256), bt.members), 256, 0, st, n,
                   vsum, maxmig, bt);
}

static inline int nblk(int64_t n, int t) { return (int)((n + t - 1) / t); }

// scratch of the crowded groups; none where no group can be crowded
Crowded encode_crowded(const Geo& g, unsigned* count, unsigned* items, long long* vsum, float* part) {
    return Crowded{count, reinterpret_cast<uint2*>(items), vsum, part + encode_groups(g),
                   g.Np > ENC_BIG ? (int)std::min<int64_t>(crowded_slots(g), 4 * g.nsm) : 0};
}

int64_t encode_partials(const Geo& g) { return encode_groups(g) + crowded_slots(g); }

void launch_encode_keys(const Geo& g, const float* pos, unsigned* key, unsigned* counts, unsigned* flags,
                        cudaStream_t st) {
    const dim3 grid(nblk(g.Np, 256));
    if (g.nchi == 1) launch_chained(k_encode_keys<1>, grid, 256, 0, st, g, pos, key, counts, flags);
    else launch_chained(k_encode_keys<2>, grid, 256, 0, st, g, pos, key, counts, flags);
}

int encode_groups(const Geo& g) { return nblk(g.Ncc, ENC_CELLS); }

int launch_encode_vc(const Geo& g, const float* vel, const unsigned* perm, const StoreDev& s, float* const* vsorted,
                     float* part, const Crowded& cr, unsigned* flags, cudaStream_t st) {
    launch_chained(k_encode_vc<false>, dim3(encode_groups(g)), T_BRICK, 0, st, g, vel, perm, s, vsorted[0], vsorted[1],
                   vsorted[2], part, cr, flags);
    if (cr.ctas == 0) return 1;
    launch_chained(k_encode_vc<true>, dim3(cr.ctas), T_BRICK, 0, st, g, vel, perm, s, vsorted[0], vsorted[1], vsorted[2],
                   part, cr, flags);
    launch_chained(k_encode_crowded, dim3(cr.ctas), T_BRICK, 0, st, g, s, vsorted[0], vsorted[1], vsorted[2],
                   part != nullptr, cr);
    return 3;
}

void launch_sigma_finalize(const float* part, int nparts, double count, double ratio, double fixed,
                           double* sigma_out, bool comp, cudaStream_t st, const Batch& bt) {
    launch_chained(comp ? k_sigma_finalize<true> : k_sigma_finalize<false>, dim3(bt.members), 1024, 0, st, part, nparts,
                   count, ratio, fixed, sigma_out, bt);
}

void launch_codec_tables(int nulim, const double* tanv, const double* tanh_, const CodecDev& c, cudaStream_t st,
                         const Batch& bt) {
    // 1-byte codes (nulim 127) fit one block, which also builds the bucket table
    const bool one = nulim + 2 <= 256;
    launch_chained(k_codec_tables, dim3(nblk(nulim + 2, 256), bt.members), 256, 0, st, nulim, tanv, tanh_, c.sigma, c.dec, c.thr,
                                                                          c.est, one ? c.vtab : nullptr,
                                                                          one ? nullptr : c.vdel, bt);
}

template <int NX, int NV>
static int encode_codes(const Geo& g, const float* pos, const float* const* vsorted, const unsigned* id_in,
                        const unsigned* perm, const CodecDev& c, const StoreDev& s, const Crowded& cr, cudaStream_t st) {
    launch_chained(k_encode_codes<NX, NV, false>, dim3(encode_groups(g)), T_BRICK, 0, st, g, pos, vsorted[0], vsorted[1],
                   vsorted[2], id_in, perm, c, s, cr);
    if (cr.ctas == 0) return 1;
    launch_chained(k_encode_codes<NX, NV, true>, dim3(cr.ctas), T_BRICK, 0, st, g, pos, vsorted[0], vsorted[1],
                   vsorted[2], id_in, perm, c, s, cr);
    return 2;
}

int launch_encode_codes(const Geo& g, const float* pos, const float* const* vsorted, const unsigned* id_in,
                        const unsigned* perm, const CodecDev& c, const StoreDev& s, const Crowded& cr,
                        cudaStream_t st) {
    if (g.nchi == 1 && g.nnu == 1) return encode_codes<1, 1>(g, pos, vsorted, id_in, perm, c, s, cr, st);
    if (g.nchi == 1) return encode_codes<1, 2>(g, pos, vsorted, id_in, perm, c, s, cr, st);
    if (g.nnu == 1) return encode_codes<2, 1>(g, pos, vsorted, id_in, perm, c, s, cr, st);
    return encode_codes<2, 2>(g, pos, vsorted, id_in, perm, c, s, cr, st);
}

void launch_max_speed(const Geo& g, const StoreDev& s, const CodecDev& c, unsigned* vmax_bits, cudaStream_t st,
                      const Batch& bt) {
    if (bt.members == 1 && !bt.ms) cudaMemsetAsync(vmax_bits, 0, sizeof(unsigned), st);
    else launch_chained(k_zero_slot_words, dim3(1), 256, 0, st, vmax_bits, bt);
    // one wave of 64 warps per SM holds eight lanes a cell: small stores
    const bool wide = (int64_t)g.Ncc * bt.members * 8 <= (int64_t)64 * 32 * g.nsm;
    const dim3 grid(nblk((int64_t)g.Ncc * (wide ? 8 : 2), T_BRICK), bt.members);
    if (g.nnu == 1 && wide) launch_chained(k_max_speed<1, 8>, grid, T_BRICK, 0, st, g, s, c, vmax_bits, bt);
    else if (g.nnu == 1) launch_chained(k_max_speed<1, 2>, grid, T_BRICK, 0, st, g, s, c, vmax_bits, bt);
    else if (wide) launch_chained(k_max_speed<2, 8>, grid, T_BRICK, 0, st, g, s, c, vmax_bits, bt);
    else launch_chained(k_max_speed<2, 2>, grid, T_BRICK, 0, st, g, s, c, vmax_bits, bt);
}

template <int NX, int NV>
static void decode(const Geo& g, const StoreDev& s, const CodecDev& c, float* pos, float* vel, unsigned* id,
                   cudaStream_t st) {
    const dim3 grid(nblk(g.Ncc, DEC_CELLS));
    if (g.B == 4) launch_chained(k_decode<NX, NV, true>, grid, T_BRICK, 0, st, g, s, c, pos, vel, id);
    else launch_chained(k_decode<NX, NV, false>, grid, T_BRICK, 0, st, g, s, c, pos, vel, id);
}

void launch_decode(const Geo& g, const StoreDev& s, const CodecDev& c, float* pos, float* vel, unsigned* id,
                   cudaStream_t st) {
    if (g.nchi == 1 && g.nnu == 1) decode<1, 1>(g, s, c, pos, vel, id, st);
    else if (g.nchi == 1) decode<1, 2>(g, s, c, pos, vel, id, st);
    else if (g.nnu == 1) decode<2, 1>(g, s, c, pos, vel, id, st);
    else decode<2, 2>(g, s, c, pos, vel, id, st);
}

static size_t deposit_smem(const Geo& g) {
    const int E = g.B + 1, E3 = E * E * E;
    return (size_t)dep_acc_words(g.F) * 4 + (size_t)(3 * E3 + 1) * 4 + DEP_QCAP;
}

void launch_deposit(const Geo& g, const StoreDev& s, float* mesh, double scale, cudaStream_t st, const Batch& bt,
                    const StepScratch* step) {
    size_t sm = deposit_smem(g);
    const bool f16 = g.F == 16, bat = bt.members > 1 || bt.ms;
    const dim3 grid(g.nb, g.nb, g.nb * bt.members);
    const float fs = (float)scale;
    long long* vs = step ? step->vsum_new : nullptr;
    int* mig = step ? step->maxmig : nullptr;
    if (g.nchi == 1) {
        set_smem_attrs<1, 1>(); set_smem_attrs<1, 2>();
        if (f16) {
            if (bat) launch_chained(k_deposit<1, 16, true>, grid, T_BRICK, sm, st, g, s, mesh, fs, vs, mig, bt);
            else launch_chained(k_deposit<1, 16, false>, grid, T_BRICK, sm, st, g, s, mesh, fs, vs, mig, bt);
        } else {
            if (bat) launch_chained(k_deposit<1, 0, true>, grid, T_BRICK, sm, st, g, s, mesh, fs, vs, mig, bt);
            else launch_chained(k_deposit<1, 0, false>, grid, T_BRICK, sm, st, g, s, mesh, fs, vs, mig, bt);
        }
    } else {
        set_smem_attrs<2, 1>(); set_smem_attrs<2, 2>();
        if (f16) {
            if (bat) launch_chained(k_deposit<2, 16, true>, grid, T_BRICK, sm, st, g, s, mesh, fs, vs, mig, bt);
            else launch_chained(k_deposit<2, 16, false>, grid, T_BRICK, sm, st, g, s, mesh, fs, vs, mig, bt);
        } else {
            if (bat) launch_chained(k_deposit<2, 0, true>, grid, T_BRICK, sm, st, g, s, mesh, fs, vs, mig, bt);
            else launch_chained(k_deposit<2, 0, false>, grid, T_BRICK, sm, st, g, s, mesh, fs, vs, mig, bt);
        }
    }
}

static size_t passA_smem(const Geo& g) {
    const int T = g.F + 5, TS = g.F + 8, H3 = g.Bh * g.Bh * g.Bh, nbc = g.B * g.B * g.B;
    // + 128: the tile is placed on a 128-byte boundary at run time
    size_t sm = (size_t)3 * H3 * 8 + 128 + (size_t)T * T * TS * 4 + (size_t)H3 * 4 + (size_t)(nbc + 1) * 4;
    if (g.nnu == 1) sm += (size_t)(3 * g.nulim + 3) * 4 + VT_N;
    sm += (size_t)3 * nbc * 4 + DEP_QCAP;
    return (sm + 15) & ~(size_t)15;
}

void launch_passA(const Geo& g, const StoreDev& s, const float* phig, const CUtensorMap* tmap, const CodecDev& cur,
                  float kick, float dc, const StepScratch& w, const DriftDebug& dbg, cudaStream_t st,
                  const Batch& bt) {
    size_t sm = passA_smem(g);
    static const CUtensorMap none{};
    const CUtensorMap& tm = tmap ? *tmap : none;
    const int use = tmap != nullptr;
    if (g.nchi == 1 && g.nnu == 1) { set_smem_attrs<1, 1>(); Disp<1, 1>::passA(g, s, phig, tm, use, cur, kick, dc, w, dbg, sm, st, bt); }
    else if (g.nchi == 1) { set_smem_attrs<1, 2>(); Disp<1, 2>::passA(g, s, phig, tm, use, cur, kick, dc, w, dbg, sm, st, bt); }
    else if (g.nnu == 1) { set_smem_attrs<2, 1>(); Disp<2, 1>::passA(g, s, phig, tm, use, cur, kick, dc, w, dbg, sm, st, bt); }
    else { set_smem_attrs<2, 2>(); Disp<2, 2>::passA(g, s, phig, tm, use, cur, kick, dc, w, dbg, sm, st, bt); }
}

void launch_cells(const Geo& g, const StepScratch& w, unsigned* off_new, float* vc_new, cudaStream_t st,
                  const Batch& bt) {
    launch_chained(k_cells, dim3(nblk(g.Ncc, 256), bt.members), 256, 0, st, g, w, off_new, vc_new, bt);
}

// Beyond STEP_TILES tiles their sums are scanned in two more launches, us of the
// three (every tile adding up the ones before it / scanned): 4096 tiles 57 /
// 62, 6912 139 / 141, 16384 319 / 310, 55296 1166 / 1002, 131072 (a mesh of
// 512^3 at ratio 1, a step of 28 ms) 3470 / 2352.
constexpr int STEP_TILES = 8192;
int step_scan_launches(const Geo& g) { return step_tiles(g) > STEP_TILES ? scan_launches(step_tiles(g)) : 0; }

int step_tmp_words(const Geo& g) {
    const int n = step_tiles(g);
    return n > STEP_TILES ? n + 1 + scan_tmp_words(n) : n;
}

void launch_step_scan(const Geo& g, unsigned* tmp, cudaStream_t st) {
    const int n = step_tiles(g);
    if (n > STEP_TILES) exclusive_scan(tmp, tmp, n, tmp + n + 1, st);
}

void launch_step_sums(const Geo& g, const StepScratch& w, double ratio, double* sigma_out, unsigned* tmp,
                      cudaStream_t st) {
    launch_chained(k_step_sums, dim3(1 + (step_tiles(g) + 1) / 2), 1024, 0, st, g, w, ratio, sigma_out, tmp);
}

void launch_step_cells(const Geo& g, const StepScratch& w, unsigned* off_new, float* vc_new, const double* tanv,
                       const double* tanh, const CodecDev& next, const unsigned* tmp, cudaStream_t st) {
    const int ntab = g.nnu == 1 ? 1 : nblk(g.nulim + 2, SC_T);
    launch_chained(k_step_cells, dim3(ntab + step_tiles(g)), SC_T, 0, st, g, w, tmp, off_new, vc_new, tanv, tanh, next, ntab,
                   step_tiles(g) > STEP_TILES);
}

// `words` of a CTA's brick tables after the staged 1-byte codec tables
static size_t passB_smem(const Geo& g, int words) {
    size_t sm = (size_t)words * 4;
    if (g.nnu == 1) sm += (size_t)(3 * g.nulim + 3) * 4 + VT_N;
    return (sm + 15) & ~(size_t)15;
}

void launch_passB(const Geo& g, const StoreDev& so, const StoreDev& sn, const CodecDev& cur, const CodecDev& next,
                  float dc, const StepScratch& w, cudaStream_t st, const Batch& bt) {
    const size_t sm = passB_smem(g, PB_WARPS * (4 * g.B * g.B * g.B + 1 + 4 * g.Bh * g.Bh * g.Bh));
    const size_t sm_cta = passB_smem(g, 4 * g.B * g.B * g.B + 1 + (4 + PB_WARPS) * g.Bh * g.Bh * g.Bh);
    const float* vcn = sn.vc;
    if (g.nchi == 1 && g.nnu == 1) { set_smem_attrs<1, 1>(); Disp<1, 1>::passB(g, so, sn, cur, next, dc, w.ghost, vcn, w.flags, w.big, sm, sm_cta, st, bt); }
    else if (g.nchi == 1) { set_smem_attrs<1, 2>(); Disp<1, 2>::passB(g, so, sn, cur, next, dc, w.ghost, vcn, w.flags, w.big, sm, sm_cta, st, bt); }
    else if (g.nnu == 1) { set_smem_attrs<2, 1>(); Disp<2, 1>::passB(g, so, sn, cur, next, dc, w.ghost, vcn, w.flags, w.big, sm, sm_cta, st, bt); }
    else { set_smem_attrs<2, 2>(); Disp<2, 2>::passB(g, so, sn, cur, next, dc, w.ghost, vcn, w.flags, w.big, sm, sm_cta, st, bt); }
}

void launch_check_vel_tables(int lim, const CodecDev& c, long long* out2, cudaStream_t st) {
    cudaMemsetAsync(out2, 0, 2 * sizeof(long long), st);
    k_check_vel_tables<<<nblk(lim + 2, 256), 256, 0, st>>>(lim, c, out2);
}

void launch_store_sums(const Geo& g, const StoreDev& s, const float* dec, long long* out4, cudaStream_t st) {
    size_t sm = (size_t)(g.B * g.B * g.B + 1) * sizeof(unsigned);
    cudaMemsetAsync(out4, 0, 4 * sizeof(long long), st);
    if (g.nnu == 1) k_store_sums<1><<<g.nbricks, T_BRICK, sm, st>>>(g, s, dec, out4);
    else k_store_sums<2><<<g.nbricks, T_BRICK, sm, st>>>(g, s, dec, out4);
}

}  // namespace cube
