// Internal launch interface between libcube's host code and its kernels.
#pragma once

#include <string>
#include <type_traits>
#include <utility>

#include <cuda.h>

#include "cube_common.cuh"

namespace cube {

// ------------------------------------------------------------ chained launches
// A step is a chain of short kernels, each reading what the one before wrote.
// launch_chained lets the next kernel's launch overlap the running one
// (programmatic dependent launch): its CTAs come up as the predecessor's exit,
// and chain_wait() holds them until the predecessor has completed and its
// writes are visible.  Every CTA of a kernel launched this way calls
// chain_wait() before it touches anything that an earlier kernel of the stream
// reads or writes (tables uploaded once at creation may be read before), and
// before it returns, so completion stays transitive along the chain.  Steps of
// 32^3, 64^3 (x1v2), 128^3 and 256^3 particles: runs 766 -> 636, 640 -> 519, 1787
// -> 1656 and 6683 -> 6599 us.  (An early griddepcontrol.launch_dependents
// lets the successor's waiting CTAs take the slots of the running kernel: 7535
// us at 256^3.)
__device__ __forceinline__ void chain_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
template <class... P, class... A>
inline void launch_chained(void (*kernel)(P...), dim3 grid, unsigned block, size_t smem, cudaStream_t st, A&&... args) {
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, kernel, std::forward<A>(args)...);
}

// inclusive scan of one value per thread over the block; returns the
// inclusive prefix, writes the block total to *total
__device__ __forceinline__ unsigned block_inclusive_scan(unsigned v, unsigned* smem_warp, unsigned* total) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int nw = blockDim.x >> 5;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        unsigned t = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += t;
    }
    if (lane == 31) smem_warp[w] = v;
    __syncthreads();
    if (w == 0) {
        unsigned s = lane < nw ? smem_warp[lane] : 0u;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            unsigned t = __shfl_up_sync(0xffffffffu, s, o);
            if (lane >= o) s += t;
        }
        if (lane < nw) smem_warp[lane] = s;
    }
    __syncthreads();
    unsigned add = w > 0 ? smem_warp[w - 1] : 0u;
    unsigned tot = smem_warp[nw - 1];
    __syncthreads();
    *total = tot;
    return v + add;
}

// ------------------------------------------------------------ batches
// A batched launch steps several members (simulations with the same
// geometry) at once: member m's device buffers are member 0's plus m * stride
// bytes, so every kernel of the step takes one extra grid dimension over the
// members and moves its pointers by m * stride.  A single context is the
// batch of one (members 1, stride 0, no per-member table).
struct MemberStep {
    float kick, dc;     // the step's kick factor and drift per coarse cell
    double ratio;       // momentum growth ratio of the codec-scale update
    int active;         // 0: the slot steps nothing (its kernels return at once)
    int member;         // the member this grid slot steps
};
// A launch's grid has one slot per listed member: with a per-member table,
// slot i steps member ms[i].member (a batch step lists only the members it
// moves, so members that sit it out cost no CTAs); without one, slot i is
// member i.  host_members mirrors ms[i].member for launches issued member by
// member from the host (null: slot i is member i).
struct Batch {
    int members;                 // slots of the launch
    size_t stride;               // bytes between consecutive members' buffers
    const MemberStep* ms;        // [members] (device) or null
    const int* host_members;     // [members] (host) or null
};
__host__ __device__ __forceinline__ int slot_member(const Batch& bt, int slot) {
#ifdef __CUDA_ARCH__
    return bt.ms ? bt.ms[slot].member : slot;
#else
    return bt.host_members ? bt.host_members[slot] : slot;
#endif
}
template <class T>
__host__ __device__ __forceinline__ T* moved(T* p, size_t off) {
    return p ? reinterpret_cast<T*>(reinterpret_cast<char*>(const_cast<typename std::remove_const<T>::type*>(p)) + off)
             : p;
}

// ------------------------------------------------------------ cube_api.cu
void set_last_error(const std::string& msg);     // message for cube_last_error()

// ------------------------------------------------------------ k_scan.cu
int scan_tmp_words(int64_t n);
int scan_launches(int64_t n);              // kernels of exclusive_scan for one context
void exclusive_scan(const unsigned* in, unsigned* out, int64_t n, unsigned* tmp, cudaStream_t st,
                    const Batch& bt = Batch{1, 0, nullptr, nullptr});
// out2[0] += 64-bit sum, out2[1] = max(out2[1], maximum) of n counts
void count_totals(const unsigned* counts, int64_t n, unsigned long long* out2, cudaStream_t st);
int64_t radix_tmp_words(int64_t n);
int radix_launches(int64_t n, int key_bits);   // kernels of radix_sort_index
// the permutation that sorts keys[n] by their low key_bits bits (stable), in
// `perm` or `tmp`; *spare: three other arrays of n words, free afterwards
// (the keys are overwritten)
unsigned* radix_sort_index(unsigned* keys, unsigned* perm, int64_t n, int key_bits, unsigned* tmp, cudaStream_t st,
                           unsigned** spare);

// ------------------------------------------------------------ k_store.cu
struct StoreDev {
    unsigned* counts;   // [Ncc]
    unsigned* offsets;  // [Ncc + 1]
    float* vc;          // [3][Ncc]
    void* chi;          // [3][Np]
    void* nu;           // [3][Np]
    void* id;           // [Np] particle IDs of Geo::nid bytes (1, 2 or 4), or null
};

struct CodecDev {
    float* dec;         // [2 lim + 1]: dec[nu + lim] = tan(pi nu / M) * sqrt(2 sigma^2 / pi)
    float* thr;         // [lim + 2]: encode thresholds (Eq. nu, cube_common.cuh)
    float* est;         // [8]: s and M/pi (nu_codes3); [2] the first bucket key of vtab (int bits);
                        // [3], [4]: pi / (2M) and 1 / s of the 2-byte tables' approximation (VelApprox)
    unsigned char* vtab;   // [VT_N] (1-byte codes): code at the start of each bucket of |d| (see nu_from_table)
    double* sigma;      // device scalar
    signed char* vdel;     // [lim + 2] (2-byte codes): corrections of dec to tan_steps (VelTables)
};

struct DriftDebug {
    int* cell_old;      // [3][Np] or null
    float* u_new;       // [3][Np]
    float* p;           // [3][Np]
    float* force;       // [3][Np]: gathered -grad Phi before the kick
};

struct StepScratch {
    unsigned* counts_new;   // [Ncc]
    long long* vsum_new;    // [3][Ncc]
    unsigned* ghost;        // [nbricks * Bh^3 + 1]: per-brick histograms in flattened
                            // (cell, brick) order, scanned in place into starts
    float* part;            // [max(nbricks, blocks)] partial sums
    unsigned* flags;        // device error flags
    int* maxmig;            // largest |cell shift| of the step
    int* big;               // [1 + nbricks]: number of bricks with more than PB_BIG
                            // particles, then their indices (listed by pass A)
};

// the same buffers of the member `off` bytes further on
__host__ __device__ __forceinline__ StoreDev moved(const StoreDev& s, size_t off) {
    return StoreDev{moved(s.counts, off), moved(s.offsets, off), moved(s.vc, off), moved(s.chi, off),
                    moved(s.nu, off), moved(s.id, off)};
}
__host__ __device__ __forceinline__ CodecDev moved(const CodecDev& c, size_t off) {
    return CodecDev{moved(c.dec, off), moved(c.thr, off), moved(c.est, off), moved(c.vtab, off), moved(c.sigma, off),
                    moved(c.vdel, off)};
}
__host__ __device__ __forceinline__ StepScratch moved(const StepScratch& w, size_t off) {
    return StepScratch{moved(w.counts_new, off), moved(w.vsum_new, off), moved(w.ghost, off), moved(w.part, off),
                       moved(w.flags, off), moved(w.maxmig, off), moved(w.big, off)};
}
// a batch of one: a single context's launch
constexpr Batch kSingle{1, 0, nullptr, nullptr};

// Groups of cells that the encode splits over several CTAs (k_store.cu): the
// list of their runs, {group, slot}, and its length (cleared by the caller); their cells' momentum sums
// [3][Ncc]; the runs' sums of squared offsets, by slot.  ctas: CTAs for
// the list (0: no group can be crowded, and nothing else is used)
struct Crowded {
    unsigned* count;
    uint2* item;
    long long* vsum;
    float* part;
    int ctas;
};
// items: two words a slot, 4 (Np / 8192 + 1) in all; part: encode_partials(g) words
Crowded encode_crowded(const Geo& g, unsigned* count, unsigned* items, long long* vsum, float* part);
int64_t encode_partials(const Geo& g);
// sort keys (cell ranks) and cell counts of float positions
void launch_encode_keys(const Geo& g, const float* pos, unsigned* key, unsigned* counts, unsigned* flags,
                        cudaStream_t st);
// the particles' momenta in storage order (three rows of Np), v_c of every
// cell, and (part not null) the sums of squared offsets from v_c of
// encode_groups runs of cells; the kernels launched
int encode_groups(const Geo& g);
int launch_encode_vc(const Geo& g, const float* vel, const unsigned* perm, const StoreDev& s, float* const* vsorted,
                     float* part, const Crowded& cr, unsigned* flags, cudaStream_t st);
// (comp: many partial sums, added with their errors)
void launch_sigma_finalize(const float* part, int nparts, double count, double ratio, double fixed,
                           double* sigma_out, bool comp, cudaStream_t st,
                           const Batch& bt = Batch{1, 0, nullptr, nullptr});
void launch_codec_tables(int nulim, const double* tanv, const double* tanh, const CodecDev& c, cudaStream_t st,
                         const Batch& bt = Batch{1, 0, nullptr, nullptr});
int launch_encode_codes(const Geo& g, const float* pos, const float* const* vsorted, const unsigned* id_in,
                         const unsigned* perm, const CodecDev& c, const StoreDev& s, const Crowded& cr,
                         cudaStream_t st);
void launch_decode(const Geo& g, const StoreDev& s, const CodecDev& c, float* pos, float* vel, unsigned* id,
                   cudaStream_t st);
// (step: the step's scratch that pass A accumulates into, cleared by the way, or null)
void launch_deposit(const Geo& g, const StoreDev& s, float* mesh, double scale, cudaStream_t st,
                    const Batch& bt = Batch{1, 0, nullptr, nullptr}, const StepScratch* step = nullptr);
// phig: ghosted Phi; tmap: TMA map of phig with the brick's tile as its box, or NULL (cp.async loads)
// (tmap: a 4-D map over (x, y, z, member) of the members' ghosted Phi)
void launch_passA(const Geo& g, const StoreDev& s, const float* phig, const CUtensorMap* tmap, const CodecDev& cur,
                  float kick, float dc, const StepScratch& w, const DriftDebug& dbg, cudaStream_t st,
                  const Batch& bt = Batch{1, 0, nullptr, nullptr});
// a batch step's cleared scratch (momentum sums, migration words) of its stepped members
void launch_batch_clear(const Geo& g, long long* vsum, int* maxmig, cudaStream_t st, const Batch& bt);
// a single context's kernels between the passes: the histograms' tile sums and
// the next codec scale, the tile sums' scan (many tiles only), then the scanned histograms, the new cells' counts,
// offsets and v_c, and the next codec's tables.  tmp: step_tmp_words words
int step_tmp_words(const Geo& g);
void launch_step_sums(const Geo& g, const StepScratch& w, double ratio, double* sigma_out, unsigned* tmp,
                      cudaStream_t st);
int step_scan_launches(const Geo& g);
void launch_step_scan(const Geo& g, unsigned* tmp, cudaStream_t st);
void launch_step_cells(const Geo& g, const StepScratch& w, unsigned* off_new, float* vc_new, const double* tanv,
                       const double* tanh, const CodecDev& next, const unsigned* tmp, cudaStream_t st);
// the new cells of a batch, from the scanned histograms
void launch_cells(const Geo& g, const StepScratch& w, unsigned* off_new, float* vc_new, cudaStream_t st,
                  const Batch& bt);
void launch_passB(const Geo& g, const StoreDev& s_old, const StoreDev& s_new, const CodecDev& cur,
                  const CodecDev& next, float dc, const StepScratch& w, cudaStream_t st,
                  const Batch& bt = Batch{1, 0, nullptr, nullptr});
// Up to five arrays copied in one launch (a checkpoint's sections): array i is
// bytes[i] long, both ends 16-byte aligned.  By the way, any of: a 64-byte
// header written to `header_to` with *sigma_from at byte 56; sigma_to = sigma;
// zero[0 .. nzero) and zero64[0 .. 1] cleared.
struct SectionCopy {
    char* dst[5];
    const char* src[5];
    int64_t bytes[5];
    int n;
    char* header_to;
    unsigned header[16];
    const double* sigma_from;
    double* sigma_to;
    double sigma;
    unsigned* zero;
    int nzero;
    long long* zero64;
};
void launch_section_copy(const SectionCopy& c, cudaStream_t st);
// sums over the current store: out[0..2] momentum of the decoded particles in
// 2^-24 fixed point, out[3] the particle count (sum of the cell counts)
void launch_store_sums(const Geo& g, const StoreDev& s, const float* dec, long long* out4, cudaStream_t st);
// 2-byte codes: out2[0] entries of dec that VelTables rebuilds differently and thresholds that nu_codes3
// decides differently, out2[1] entries read whole
void launch_check_vel_tables(int lim, const CodecDev& c, long long* out2, cudaStream_t st);

// uncompressed FP32 particles (k_raw.cu)
void launch_raw_encode(const Geo& g, const float* pos, const float* vel, const unsigned* id_in, float* P, float* V,
                       unsigned* I, unsigned* flags, cudaStream_t st);
void launch_raw_deposit(const Geo& g, const float* P, float* mesh, float mass, cudaStream_t st);
void launch_raw_kick_drift(const Geo& g, float* P, float* V, const float* phi, float kick, float drift,
                           unsigned* flags, cudaStream_t st);
void launch_raw_momentum(const Geo& g, const float* V, long long* out3, cudaStream_t st);
void launch_iota(unsigned* out, int64_t n, cudaStream_t st);
void launch_raw_max_speed(const Geo& g, const float* V, unsigned* vmax_bits, cudaStream_t st);
// largest |p| of the store (float bits), of every listed member of a batch
void launch_max_speed(const Geo& g, const StoreDev& s, const CodecDev& c, unsigned* vmax_bits, cudaStream_t st,
                      const Batch& bt = Batch{1, 0, nullptr, nullptr});

// ------------------------------------------------------------ k_fft.cu
struct FftPlan {
    int N;              // transform length along every axis
    float2* tw;         // [N] e^{-2 pi i k / N}
    float* k2;          // [N] (2 pi f / N)^2, f the signed frequency of index i
    float* wdec;        // [N] sinc(pi f / N)^(-2 p)  (deconvolution factor per axis)
    double* wpk;        // [N] sinc(pi f / N)^(-4)    (P(k) window correction per axis)
};

bool fft_size_supported(int N);                                                    // compiled mesh sizes
void fft_x_r2c(const FftPlan& p, float* mesh, int S, cudaStream_t st,
               const Batch& bt = Batch{1, 0, nullptr, nullptr});                                      // rows: r2c
void fft_y(const FftPlan& p, float* mesh, int S, bool inverse, cudaStream_t st,
           const Batch& bt = Batch{1, 0, nullptr, nullptr});                                          // y columns
void fft_z(const FftPlan& p, float* mesh, int S, float g0, bool green, cudaStream_t st,
           const Batch& bt = Batch{1, 0, nullptr, nullptr});                                          // z (+ Green, inverse)
void fft_x_c2r(const FftPlan& p, float* mesh, int S, float* phig, cudaStream_t st,
               const Batch& bt = Batch{1, 0, nullptr, nullptr});                                      // rows: c2r into ghosted Phi
int pk_blocks(int N);
void launch_pk_bin(const FftPlan& p, const float* mesh, int S, int nbins, double* part, cudaStream_t st);
void launch_pk_reduce(const FftPlan& p, const double* part, int nbins, double pfac, double kfund, double* k, double* pk,
                      double* nm, cudaStream_t st);
void launch_unpad(const float* mesh, int N, int S, float* out, cudaStream_t st);
// largest |component| of the FD4 gradient / 12 of the ghosted potential over
// all mesh nodes (float bits): an upper bound of every particle's force
// component, which the gather interpolates from these values with CIC weights
void launch_grad_max(const float* phig, int N, unsigned* out_bits, cudaStream_t st);
void launch_unpad_phig(const float* phig, int N, float* out, cudaStream_t st);

}  // namespace cube
