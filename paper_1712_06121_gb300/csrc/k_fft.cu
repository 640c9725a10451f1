// 3-D real FFT Poisson solve on the fine mesh and the power-spectrum binning.
//
// Mesh layout: real rho / Phi as rows of N floats with row stride S = N + 4
// (z-major, then y); in place, the r2c result is rows of N/2 + 1 complex
// (kx = 0..N/2) with complex stride S/2.  Transforms are unnormalised; the
// 1/N^3 of the inverse is folded into the Green's function.
//
// Each kernel transforms one tile of 16 columns of length n in shared memory
// with a mixed-radix (8, 4, 2, 3) Stockham autosort FFT: every pass reads each
// element once and writes it once, through registers.
//   x sweep : 16 rows per CTA, r2c / c2r by the even-odd packing into an
//             N/2-point complex transform (layout [k][row pair], XOR-swizzled so
//             row-wise and column-wise accesses are both conflict-free)
//   y sweep : 16 consecutive kx columns of one z-slab
//   z sweep : 16 consecutive kx columns of one ky line; forward, times
//             -(3/2) Om / k^2 / W(k)^p / N^3, inverse, in one pass.
//
// The sweeps are bound by instruction issue before they are bound by memory,
// so a thread transforms two columns at once: a tile element is (re, re, im,
// im) of a column pair, one 16-byte access, and every operation is one packed
// FP32 instruction on the pair; twiddles (one address and one load for both
// columns) are staged as (re, re, im, im) too.  Each lane of a packed operation
// is rounded as the scalar one, and sums of products are written as the fused
// operations the scalar expressions contract to, so the results are those of
// one column at a time, bit for bit.  512^3, us, one column a thread with two
// barriers a pass -> this: x r2c 210 -> 184, y 222 -> 209, z 373 -> 322, inverse
// y 234 -> 206, c2r 234 -> 227; 384^3: 113 -> 107, 119 -> 92, 180 -> 146, 115 ->
// 84, 111 -> 108.
#include <cmath>

#include "kernels.h"

namespace cube {

namespace {

constexpr int NC = 16;          // columns per tile
constexpr int NP = NC / 2;      // column pairs per tile
constexpr int LOG_NP = 3;

// Threads of a CTA: one radix-8 butterfly of a column pair each, at least a
// warp; launch bounds keep 64 registers a thread (1024 threads per SM)
constexpr int fft_threads(int n) { return n < 32 ? 32 : n > 1024 ? 1024 : n; }
constexpr int fft_blocks(int n) { return 1024 / fft_threads(n) > 16 ? 16 : 1024 / fft_threads(n); }

// a pair of complex numbers: (re, re), (im, im) of two columns
struct C2 {
    float2 x, y;
};
__device__ __forceinline__ C2 c2(float4 f) { return C2{make_float2(f.x, f.y), make_float2(f.z, f.w)}; }
__device__ __forceinline__ float4 pack4(const C2& a) { return make_float4(a.x.x, a.x.y, a.y.x, a.y.y); }
// two complex numbers in memory order (re0, im0, re1, im1)
__device__ __forceinline__ C2 from_columns(float4 f) { return C2{make_float2(f.x, f.z), make_float2(f.y, f.w)}; }
__device__ __forceinline__ float4 to_columns(const C2& a) { return make_float4(a.x.x, a.y.x, a.x.y, a.y.y); }
__device__ __forceinline__ C2 from_rows(float2 a, float2 b) { return C2{make_float2(a.x, b.x), make_float2(a.y, b.y)}; }
__device__ __forceinline__ float2 row_of(const C2& a, int r) {
    return r ? make_float2(a.x.y, a.y.y) : make_float2(a.x.x, a.y.x);
}
__device__ __forceinline__ C2 cadd(const C2& a, const C2& b) { return C2{padd(a.x, b.x), padd(a.y, b.y)}; }
__device__ __forceinline__ C2 csub(const C2& a, const C2& b) { return C2{psub(a.x, b.x), psub(a.y, b.y)}; }
// a + r b and a - r b, r = -i (forward) or +i (inverse)
template <bool INV>
__device__ __forceinline__ C2 cadd_rot(const C2& a, const C2& b) {
    return INV ? C2{psub(a.x, b.y), padd(a.y, b.x)} : C2{padd(a.x, b.y), psub(a.y, b.x)};
}
template <bool INV>
__device__ __forceinline__ C2 csub_rot(const C2& a, const C2& b) {
    return cadd_rot<!INV>(a, b);
}
// f a, each lane by its own factor; scalar products, which nothing fuses
__device__ __forceinline__ C2 scaled(const C2& a, float2 f) {
    return C2{make_float2(__fmul_rn(a.x.x, f.x), __fmul_rn(a.x.y, f.y)),
              make_float2(__fmul_rn(a.y.x, f.x), __fmul_rn(a.y.y, f.y))};
}
// a w (forward) or a w* (inverse), w the same for both columns.  One product of
// each sum is rounded first: of the imaginary part the second, or (YX) the first
template <bool INV, bool YX = INV>
__device__ __forceinline__ C2 cmul_tw(const C2& a, float2 w) {
    const float2 wx = pk2(w.x), wy = pk2(w.y), nwy = pk2(-w.y);
    const float2 im = YX ? pfma(a.y, wx, pmul(a.x, INV ? nwy : wy)) : pfma(a.x, INV ? nwy : wy, pmul(a.y, wx));
    return C2{INV ? pfma(a.x, wx, pmul(a.y, wy)) : pfma(a.x, wx, pmul(a.y, nwy)), im};
}

// w a or (CONJ) w* a, the product's terms in the order of a scalar w a
template <bool CONJ>
__device__ __forceinline__ C2 cmul_by(float2 w, const C2& a) {
    const float2 wx = pk2(w.x), wy = pk2(w.y), nwy = pk2(-w.y);
    return CONJ ? C2{pfma(wx, a.x, pmul(wy, a.y)), pfma(wx, a.y, pmul(nwy, a.x))}
                : C2{pfma(wx, a.x, pmul(nwy, a.y)), pfma(wx, a.y, pmul(wy, a.x))};
}

// Tile layout: element k of column (row) pair p at k NP + p, or, swizzled (x
// sweeps), at k NP + (p ^ ((k ^ (k >> 3)) mod NP)).  A 16-byte access is served
// eight lanes at a time: eight pairs of one k fill a 128-byte row, and with the
// swizzle so do eight values of k of one pair, whether consecutive or with the
// strides of the Stockham passes.
template <bool SWZ>
__device__ __forceinline__ int sidx(int k, int p) {
    return SWZ ? (k << LOG_NP) + (p ^ ((k ^ (k >> 3)) & (NP - 1))) : (k << LOG_NP) + p;
}

// sidx(k_lo + k_hi, p) from base = sidx(k_lo, p) when the set bits of the
// compile-time k_hi lie above those of k_lo: the swizzle is XOR-linear in k,
// so the sum is base XOR a constant plus a constant (one logic op and an
// immediate offset per access)
template <bool SWZ>
__device__ __forceinline__ int sidx_add(int base, int k_hi) {
    return SWZ ? (base ^ ((k_hi ^ (k_hi >> 3)) & (NP - 1))) + (k_hi << LOG_NP) : base + (k_hi << LOG_NP);
}

constexpr bool pow2(int x) { return x > 0 && (x & (x - 1)) == 0; }

template <int RAD, bool INV>
__device__ __forceinline__ void dft(C2* v);

// the radix-4 DFTs of a[m] = x[m] + x[m + 4] and of b[m] w8^m, b[m] = x[m] -
// x[m + 4], w8 = e^{-+ 2 pi i / 8}: the even and odd outputs of a radix-8 DFT.
// w8^2 is a rotation, and with w8 b1 = r (u1, w1), w8^3 b3 = r (u3, w3) the
// sum and difference are formed as r u1 + (r u3) and so on, one rounding
// after a product.
template <bool INV>
__device__ __forceinline__ void dft8_tail(C2* a, const C2* b, C2* v) {
    const float2 r = pk2(0.70710678118654752f), n = pk2(-0.70710678118654752f);
    dft<4, INV>(a);
    const float2 u1 = INV ? psub(b[1].x, b[1].y) : padd(b[1].x, b[1].y);
    const float2 w1 = INV ? padd(b[1].x, b[1].y) : psub(b[1].y, b[1].x);
    const float2 u3 = INV ? padd(b[3].x, b[3].y) : psub(b[3].y, b[3].x);    // inverse: -u3
    const float2 w3 = INV ? psub(b[3].x, b[3].y) : padd(b[3].x, b[3].y);    // forward: -w3
    const float2 ru = pmul(INV ? n : r, u3), nu = pmul(INV ? r : n, u3);
    const float2 rw = pmul(INV ? r : n, w3), nw = pmul(INV ? n : r, w3);
    const C2 s{pfma(r, u1, ru), pfma(r, w1, rw)}, d{pfma(r, u1, nu), pfma(r, w1, nw)};
    const C2 a0 = cadd_rot<INV>(b[0], b[2]), a1 = csub_rot<INV>(b[0], b[2]);
#pragma unroll
    for (int k = 0; k < 4; ++k) v[2 * k] = a[k];
    v[1] = cadd(a0, s);
    v[3] = cadd_rot<INV>(a1, d);
    v[5] = csub(a0, s);
    v[7] = csub_rot<INV>(a1, d);
}

template <int RAD, bool INV>
__device__ __forceinline__ void dft(C2* v) {
    if (RAD == 2) {
        const C2 a = v[0], b = v[1];
        v[0] = cadd(a, b);
        v[1] = csub(a, b);
    } else if (RAD == 3) {
        const float h = 0.86602540378443865f;   // sqrt(3)/2
        const C2 t1 = cadd(v[1], v[2]), d = csub(v[1], v[2]);
        const C2 t2 = C2{pfma(pk2(-0.5f), t1.x, v[0].x), pfma(pk2(-0.5f), t1.y, v[0].y)};
        v[0] = cadd(v[0], t1);
        // t2 -+ i h d
        const float2 p = pk2(h), m = pk2(-h);
        const C2 up = C2{pfma(m, d.y, t2.x), pfma(p, d.x, t2.y)}, dn = C2{pfma(p, d.y, t2.x), pfma(m, d.x, t2.y)};
        v[1] = INV ? up : dn;
        v[2] = INV ? dn : up;
    } else if (RAD == 4) {
        const C2 a0 = cadd(v[0], v[2]), a1 = csub(v[0], v[2]);
        const C2 b0 = cadd(v[1], v[3]), b1 = csub(v[1], v[3]);
        v[0] = cadd(a0, b0);
        v[1] = cadd_rot<INV>(a1, b1);
        v[2] = csub(a0, b0);
        v[3] = csub_rot<INV>(a1, b1);
    } else {   // 8 = 2 x 4
        C2 a[4], b[4];
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            a[m] = cadd(v[m], v[m + 4]);
            b[m] = csub(v[m], v[m + 4]);
        }
        dft8_tail<INV>(a, b, v);
    }
}

// the radices 8, 4, 2, 3 taken greedily
constexpr int radix_of(int rem) { return rem % 8 == 0 ? 8 : rem % 4 == 0 ? 4 : rem % 2 == 0 ? 2 : 3; }

// one Stockham pass of radix R over the tile of length n, span Ns; twiddles
// come from a table of TWN = n * TWM entries e^{-2 pi i k / TWN}
template <int n, int Ns, int R, int TWM, bool INV, bool SWZ, int T>
__device__ __forceinline__ void fft_pass(float4* buf, const float2* tw) {
    constexpr int nq = n / R;
    constexpr int nbf = nq * NP;
    constexpr int KMAX = (nbf + T - 1) / T;
    constexpr int step = TWM * (n / (Ns * R));
    constexpr bool lin = pow2(nq) && pow2(Ns) && pow2(R);   // bit-disjoint element offsets
    C2 v[KMAX][R];
#pragma unroll
    for (int q = 0; q < KMAX; ++q) {
        const int b = threadIdx.x + q * T;
        if (nbf % T == 0 || b < nbf) {
            const int p = b & (NP - 1), j = b >> LOG_NP;
            const int base = sidx<SWZ>(j, p);
#pragma unroll
            for (int m = 0; m < R; ++m)
                v[q][m] = c2(buf[lin ? sidx_add<SWZ>(base, m * nq) : sidx<SWZ>(j + m * nq, p)]);
        }
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < KMAX; ++q) {
        const int b = threadIdx.x + q * T;
        if (nbf % T == 0 || b < nbf) {
            const int p = b & (NP - 1), j = b >> LOG_NP;
            const int k = j % Ns;
            if (Ns > 1) {                                  // span 1: all twiddles are 1
#pragma unroll
                for (int m = 1; m < R; ++m) v[q][m] = cmul_tw<INV>(v[q][m], tw[k * m * step]);
            }
            dft<R, INV>(v[q]);
            const int idxD = (j / Ns) * Ns * R + k;
            const int base = sidx<SWZ>(idxD, p);
#pragma unroll
            for (int m = 0; m < R; ++m)
                buf[lin ? sidx_add<SWZ>(base, m * Ns) : sidx<SWZ>(idxD + m * Ns, p)] = pack4(v[q][m]);
        }
    }
    __syncthreads();
}

// all passes from span Ns on
template <int n, int Ns, int TWM, bool INV, bool SWZ, int T>
__device__ __forceinline__ void tile_fft(float4* buf, const float2* tw) {
    if constexpr (Ns < n) {
        constexpr int R = radix_of(n / Ns);
        static_assert((n / Ns) % R == 0, "length must be 2^a 3^b");
        fft_pass<n, Ns, R, TWM, INV, SWZ, T>(buf, tw);
        tile_fft<n, Ns * R, TWM, INV, SWZ, T>(buf, tw);
    }
}

// passes from span Ns up to (not including) the last
template <int n, int Ns, int TWM, bool INV, bool SWZ, int T>
__device__ __forceinline__ void tile_fft_but_last(float4* buf, const float2* tw) {
    constexpr int R = radix_of(n / Ns);
    if constexpr (Ns * R < n) {
        fft_pass<n, Ns, R, TWM, INV, SWZ, T>(buf, tw);
        tile_fft_but_last<n, Ns * R, TWM, INV, SWZ, T>(buf, tw);
    }
}

template <int n, int ns0 = 1>
constexpr int last_span() {   // span of the last pass of tile_fft<n, ns0, ...>
    int ns = ns0;
    while (ns * radix_of(n / ns) != n) ns *= radix_of(n / ns);
    return ns;
}

// ---- column tiles, in place
// A pass's butterfly writes its results where it read its inputs, so passes
// are separated by one barrier and hold nothing across it.  With radices R_1 ..
// R_q (P_i = R_1 .. R_i), pass i turns digit d_i of the input index
// sum d_l n / P_l into digit k_i of the output index sum k_l P_{l-1}, at the
// slot whose digits are the k's done and the d's to do.  Forward transforms
// weigh digit l by P_{l-1} (the output ends in natural order), inverse ones by
// n / P_l (the input begins in natural order).  A slot is a 128-byte row of 8
// pairs, so every order of the butterflies is free of bank conflicts; those of
// one twiddle are neighbours.
constexpr int rad(int n, int i) {                // R_i
    for (int l = 1; l < i; ++l) n /= radix_of(n);
    return radix_of(n);
}
constexpr int pre(int n, int i) {                // P_i
    int p = 1;
    for (int l = 1; l <= i; ++l) p *= rad(n, l);
    return p;
}
constexpr int npass(int n) {
    int q = 0;
    for (int m = n; m > 1; m /= radix_of(m)) ++q;
    return q;
}
// sum_{l = 1 .. I} k_l n / P_l of kk = sum k_l P_{l-1}
template <int n, int I>
__device__ __forceinline__ int rev_k(int kk) {
    if constexpr (I == 0) return 0;
    else return rev_k<n, I - 1>(kk) + (kk / pre(n, I - 1)) % rad(n, I) * (n / pre(n, I));
}
// sum_{l = 2 .. I} d_l P_{l-1} of j = sum_{l >= 2} d_l n / P_l
template <int n, int I>
__device__ __forceinline__ int rev_d(int j) {
    if constexpr (I <= 1) return 0;
    else return rev_d<n, I - 1>(j) + (j / (n / pre(n, I))) % rad(n, I) * pre(n, I - 1);
}
// slot of butterfly j's input 0 in pass I, and the distance to the next
template <int n, int I, bool INV>
__device__ __forceinline__ int slot0(int kk, int dd) {
    return INV ? rev_k<n, I - 1>(kk) + dd : kk + pre(n, I) * dd;
}
template <int n, int I, bool INV>
constexpr int slot_step() {
    return INV ? n / pre(n, I) : pre(n, I - 1);
}

// runs fn(pair, butterfly) over the tile's butterflies of radix R
template <int n, int R, int T, class Fn>
__device__ __forceinline__ void for_butterflies(Fn fn) {
    constexpr int nbf = n / R * NP;
#pragma unroll
    for (int b0 = 0; b0 < nbf; b0 += T) {
        const int b = b0 + threadIdx.x;
        if (nbf % T == 0 || b < nbf) fn(b & (NP - 1), b >> LOG_NP);
    }
}

// inputs of butterfly (kk, dd) of pass I, times their twiddles, transformed
template <int n, int I, bool INV, bool YX = INV>
__device__ __forceinline__ void butterfly(const float4* buf, const float2* tw, int p, int kk, int dd, C2* v) {
    constexpr int R = rad(n, I), step = n / pre(n, I);
    const float4* s = buf + (slot0<n, I, INV>(kk, dd) << LOG_NP) + p;
#pragma unroll
    for (int m = 0; m < R; ++m) v[m] = c2(s[(m * slot_step<n, I, INV>()) << LOG_NP]);
    if (I > 1) {                                           // pass 1: all twiddles are 1
#pragma unroll
        for (int m = 1; m < R; ++m) v[m] = cmul_tw<INV, YX>(v[m], tw[kk * m * step]);
    }
}

// pass I in shared memory
template <int n, int I, bool INV, int T>
__device__ __forceinline__ void col_pass(float4* buf, const float2* tw) {
    constexpr int R = rad(n, I), D = n / pre(n, I);
    for_butterflies<n, R, T>([&](int p, int j) {
        const int kk = j / D, dd = j % D;
        C2 v[R];
        butterfly<n, I, INV>(buf, tw, p, kk, dd, v);
        dft<R, INV>(v);
        float4* s = buf + (slot0<n, I, INV>(kk, dd) << LOG_NP) + p;
#pragma unroll
        for (int m = 0; m < R; ++m) s[(m * slot_step<n, I, INV>()) << LOG_NP] = pack4(v[m]);
    });
    __syncthreads();
}
// passes I .. L
template <int n, int I, int L, bool INV, int T>
__device__ __forceinline__ void col_passes(float4* buf, const float2* tw) {
    if constexpr (I <= L) {
        col_pass<n, I, INV, T>(buf, tw);
        col_passes<n, I + 1, L, INV, T>(buf, tw);
    }
}

// First pass (no twiddles) of a column tile straight from global memory:
// element r of pair p (columns c and c + 1) is the 16 bytes at src[r rs + p ps],
// zero from pair np on (a last column without a partner is paired with the
// row's padding slot, whose values go nowhere).  pack_off > 0: column 0 of pair
// 0 becomes X + i Y, X its own values and Y those of the column pack_off
// further (two real sequences in one complex transform).  Ends with a barrier.
template <int n, bool INV, int T>
__device__ __forceinline__ void col_load(float4* buf, const float2* __restrict__ src, int64_t rs, int ps, int np,
                                         int pack_off = 0) {
    constexpr int R = rad(n, 1), nq = n / R;
    for_butterflies<n, R, T>([&](int p, int j) {
        const bool ok = p < np;
        const float2* s = src + (int64_t)j * rs + p * ps;
        float4 f[R];
#pragma unroll
        for (int m = 0; m < R; ++m)
            f[m] = ok ? *reinterpret_cast<const float4*>(s + (int64_t)m * nq * rs) : make_float4(0.f, 0.f, 0.f, 0.f);
        if (pack_off > 0 && p == 0)
#pragma unroll
            for (int m = 0; m < R; ++m) {
                const float2 y = s[(int64_t)m * nq * rs + pack_off];
                f[m].x -= y.y;
                f[m].y += y.x;
            }
        C2 v[R];
#pragma unroll
        for (int m = 0; m < R; ++m) v[m] = from_columns(f[m]);
        dft<R, INV>(v);
        float4* d = buf + ((INV ? j : rev_d<n, npass(n)>(j)) << LOG_NP) + p;
#pragma unroll
        for (int m = 0; m < R; ++m) d[(m * slot_step<n, 1, INV>()) << LOG_NP] = pack4(v[m]);
    });
    __syncthreads();
}

// Last pass of a column tile: results go straight to dst[k rs + p ps] for pairs
// below np.  split_off > 0: column 0 of pair 0 holds x + i y of two real
// sequences; x goes to column 0 and y to the column split_off further, both as
// (value, 0).
template <int n, bool INV, int T>
__device__ __forceinline__ void col_store(const float4* buf, const float2* tw, float2* dst, int64_t rs, int ps,
                                          int np, int split_off = 0) {
    constexpr int q = npass(n), R = rad(n, q), nq = n / R;
    for_butterflies<n, R, T>([&](int p, int j) {
        C2 v[R];
        butterfly<n, q, INV>(buf, tw, p, j, 0, v);
        dft<R, INV>(v);
        float2* d = dst + (int64_t)j * rs + p * ps;
        if (split_off > 0 && p == 0) {
#pragma unroll
            for (int m = 0; m < R; ++m) {
                *reinterpret_cast<float4*>(d + (int64_t)m * nq * rs) = make_float4(v[m].x.x, 0.f, v[m].x.y, v[m].y.y);
                d[(int64_t)m * nq * rs + split_off] = make_float2(v[m].y.x, 0.f);
            }
        } else if (p < np) {
#pragma unroll
            for (int m = 0; m < R; ++m) *reinterpret_cast<float4*>(d + (int64_t)m * nq * rs) = to_columns(v[m]);
        }
    });
}

// The last forward pass, times post(element, pair) (the Green's function), in
// place (natural order).  Where the last forward and the first inverse pass
// have the same radix (8), both act on the same elements: FUSE runs the first
// inverse pass before the results are written.
template <int n, bool FUSE, int T, class Post>
__device__ __forceinline__ void col_pass_post(float4* buf, const float2* tw, Post post) {
    constexpr int q = npass(n), R = rad(n, q), nq = n / R;
    static_assert(!FUSE || R == rad(n, 1), "one radix");
    for_butterflies<n, R, T>([&](int p, int j) {
        C2 v[R];
        butterfly<n, q, false, FUSE>(buf, tw, p, j, 0, v);
        dft<R, false>(v);
#pragma unroll
        for (int m = 0; m < R; ++m) v[m] = scaled(v[m], post(j + m * nq, p));
        if (FUSE) dft<R, true>(v);
        float4* s = buf + (j << LOG_NP) + p;
#pragma unroll
        for (int m = 0; m < R; ++m) s[(m * nq) << LOG_NP] = pack4(v[m]);
    });
    __syncthreads();
}

// first radix of the row transforms: never the whole length, so that the
// first (load) and last (store) passes are distinct
template <int n>
constexpr int x_first_radix() {
    return radix_of(n) < n ? radix_of(n) : (n % 4 == 0 && n > 4 ? 4 : 2);
}

// `bytes` (a multiple of 16) from the 16-byte aligned p into L2.  A row sweep's
// tile is one run of 16 rows; requesting the tile that this SM's next wave of
// CTAs will load keeps HBM busy while the resident ones compute (512^3: x r2c
// 184 -> 177 us, c2r 227 -> 193; 384^3: 107 -> 90, 108 -> 92; the column sweeps'
// 128-byte pieces gain nothing from it)
__device__ __forceinline__ void l2_prefetch(const void* p, unsigned bytes) {
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(bytes) : "memory");
}

// twiddle table into shared memory; the tile's first barrier publishes it
template <int N, int T>
__device__ __forceinline__ void load_tw(float2* stw, const float2* __restrict__ tw) {
#pragma unroll
    for (int i = threadIdx.x; i < N; i += T) stw[i] = __ldg(&tw[i]);
}

// ------------------------------------------------------------ x sweeps
// NC = 16 rows per CTA, two a thread.  The first and last passes run with
// threads along the row (j fastest), so they read and write global memory in
// coalesced runs; the middle passes run across the 8 row pairs.

// First pass (span 1) of the n = N/2-point transforms of rows row0 .. row0 +
// NC - 1, straight from global memory.  PACK (c2r): the input row holds the
// half spectrum X[0 .. n] and the transform input is Z[k] = E + i O with
// E = X[k] + X*[n-k], O = W^-k (X[k] - X*[n-k]), W = e^{-2 pi i / N} (twiddles
// read from global memory: the shared copy may still be in flight).
template <int n, int R, bool INV, bool PACK, int T>
__device__ __forceinline__ void xpass_load(float4* buf, const float* mesh, int64_t row0, int S,
                                           const float2* __restrict__ gtw) {
    constexpr int nq = n / R;
    constexpr int nbf = nq * NP;
    constexpr int KMAX = (nbf + T - 1) / T;
#pragma unroll
    for (int q = 0; q < KMAX; ++q) {
        const int b = threadIdx.x + q * T;
        if (nbf % T == 0 || b < nbf) {
            const int j = b % nq, p = b / nq;
            const float2* r0 = reinterpret_cast<const float2*>(mesh + (row0 + 2 * p) * S);
            const float2* r1 = reinterpret_cast<const float2*>(mesh + (row0 + 2 * p + 1) * S);
            C2 v[R];
#pragma unroll
            for (int m = 0; m < R; ++m) {
                const int k = j + m * nq;
                if (!PACK) {
                    v[m] = from_rows(r0[k], r1[k]);
                } else {
                    const C2 xk = from_rows(r0[k], r1[k]), xm = from_rows(r0[n - k], r1[n - k]);
                    const C2 e{padd(xk.x, xm.x), psub(xk.y, xm.y)}, d{psub(xk.x, xm.x), padd(xk.y, xm.y)};
                    const C2 o = cmul_by<true>(gtw[k], d);
                    v[m] = C2{psub(e.x, o.y), padd(e.y, o.x)};
                }
            }
            dft<R, INV>(v);
            const int base = sidx<true>(j * R, p);
#pragma unroll
            for (int m = 0; m < R; ++m) buf[pow2(R) ? sidx_add<true>(base, m) : sidx<true>(j * R + m, p)] = pack4(v[m]);
        }
    }
    __syncthreads();
}

// Last pass (span n / R) of the row transforms of N = 2n reals, straight to
// the ghosted copy of Phi: every row lands at its place and, within the
// ghost layers, at its periodic images (rows y < 3 also at y + N, y >= N - 2
// also at y - N, the same in z; x < 4 also at x + N, x >= N - 4 at x - N).
template <int n, int Ns, int R, int TWM, bool INV, int T>
__device__ __forceinline__ void xpass_store(const float4* buf, const float2* tw, float* phig, int64_t row0) {
    constexpr int N = 2 * n;
    constexpr int nq = n / R;
    static_assert(nq == Ns, "the last pass has span n / R");
    constexpr int nbf = nq * NP;
    constexpr int KMAX = (nbf + T - 1) / T;
    constexpr int step = TWM * (n / (Ns * R));
#pragma unroll
    for (int q = 0; q < KMAX; ++q) {
        const int b = threadIdx.x + q * T;
        if (nbf % T == 0 || b < nbf) {
            const int j = b % nq, p = b / nq;
            C2 v[R];
            const int base = sidx<true>(j, p);
#pragma unroll
            for (int m = 0; m < R; ++m)
                v[m] = c2(buf[pow2(nq) ? sidx_add<true>(base, m * nq) : sidx<true>(j + m * nq, p)]);
            if (Ns > 1) {
#pragma unroll
                for (int m = 1; m < R; ++m) v[m] = cmul_tw<INV>(v[m], tw[j * m * step]);
            }
            dft<R, INV>(v);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int64_t r = row0 + 2 * p + h;
                const int z = (int)(r / N), y = (int)(r - (int64_t)z * N);
                // element k = j + m Ns holds reals 2k, 2k + 1; k < 2 only for m = 0,
                // k >= n - 2 only for m = R - 1 (Ns >= 2)
                auto put = [&](int yy, int zz) {
                    float2* row = reinterpret_cast<float2*>(phig + phig_index(N, 0, yy, zz));
#pragma unroll
                    for (int m = 0; m < R; ++m) row[j + m * Ns] = row_of(v[m], h);
                    if (j < 2) row[j + n] = row_of(v[0], h);
                    if (j >= Ns - 2) row[j + (R - 1) * Ns - n] = row_of(v[R - 1], h);
                };
                put(y, z);
                const bool gy = y < 3 || y >= N - 2, gz = z < 3 || z >= N - 2;
                if (gy || gz) {                  // rows with periodic images in the ghost layers
                    const int y2 = y < 3 ? y + N : y - N, z2 = z < 3 ? z + N : z - N;
                    if (gy) put(y2, z);
                    if (gz) put(y, z2);
                    if (gy && gz) put(y2, z2);
                }
            }
        }
    }
}

// r2c: the N reals of a row as N/2 complex z[k] = x[2k] + i x[2k+1], an
// N/2-point FFT Z, then X[k] = (Z[k] + Z*[h-k])/2 - i W^k (Z[k] - Z*[h-k])/2
template <int N, bool BAT>
__global__ void __launch_bounds__(fft_threads(N / 2), fft_blocks(N / 2))
    k_fft_x_r2c(float* mesh, int S, const float2* __restrict__ tw, Batch bt) {
    extern __shared__ float4 fsm[];
    if constexpr (BAT) {                                     // slot blockIdx.y of a batch
        if (bt.ms && !bt.ms[blockIdx.y].active) {
            chain_wait();
            return;
        }
        mesh = moved(mesh, slot_member(bt, blockIdx.y) * bt.stride);
    }
    constexpr int h = N / 2, T = fft_threads(h);
    float4* buf = fsm;                                       // [h][NP]
    float2* stw = reinterpret_cast<float2*>(buf + h * NP);   // [N]
    load_tw<N, T>(stw, tw);
    const int64_t row0 = (int64_t)blockIdx.x * NC;
    chain_wait();
    if (threadIdx.x == 0) {
        const int64_t r = row0 + (int64_t)152 * fft_blocks(h) * NC;
        if (r < (int64_t)N * N) l2_prefetch(mesh + r * S, NC * S * 4);
    }
    constexpr int R1 = x_first_radix<h>();
    xpass_load<h, R1, false, false, T>(buf, mesh, row0, S, tw);
    tile_fft<h, R1, 2, false, true, T>(buf, stw);
    // X[k] and X[h - k] from Z[k] and Z[h - k], k = 0 .. h / 2: threads along k
    // of one row pair, the self-paired k = h / 2 of the 8 pairs last
    for (int t = threadIdx.x; t < (h / 2) * NP + NP; t += T) {
        const bool mid = t >= (h / 2) * NP;
        const int k = mid ? h / 2 : t % (h / 2), p = mid ? t - (h / 2) * NP : t / (h / 2);
        float2* d0 = reinterpret_cast<float2*>(mesh + (row0 + 2 * p) * S);
        float2* d1 = reinterpret_cast<float2*>(mesh + (row0 + 2 * p + 1) * S);
        const C2 zk = c2(buf[sidx<true>(k % h, p)]);
        const C2 zm = c2(buf[sidx<true>((h - k) % h, p)]);
        const float2 hf = pk2(0.5f);
        {
            const C2 e{pmul(hf, padd(zk.x, zm.x)), pmul(hf, psub(zk.y, zm.y))};
            const C2 o{pmul(hf, psub(zk.x, zm.x)), pmul(hf, padd(zk.y, zm.y))};   // (Z - Z*) / 2
            const C2 wo = cmul_by<false>(stw[k], o);
            const C2 x{padd(e.x, wo.y), psub(e.y, wo.x)};                         // e - i wo
            d0[k] = row_of(x, 0);
            d1[k] = row_of(x, 1);
        }
        if (k != h - k) {
            const int km = h - k;
            const C2 e{pmul(hf, padd(zm.x, zk.x)), pmul(hf, psub(zm.y, zk.y))};
            const C2 o{pmul(hf, psub(zm.x, zk.x)), pmul(hf, padd(zm.y, zk.y))};
            const C2 wo = cmul_by<false>(stw[km], o);
            const C2 x{padd(e.x, wo.y), psub(e.y, wo.x)};
            d0[km] = row_of(x, 0);
            d1[km] = row_of(x, 1);
        }
    }
}

// c2r: the packing above inverted inside the first pass, the N/2-point
// inverse FFT, and the last pass writing the row's N reals
template <int N, bool BAT>
__global__ void __launch_bounds__(fft_threads(N / 2), fft_blocks(N / 2))
    k_fft_x_c2r(const float* mesh, int S, const float2* __restrict__ tw, float* __restrict__ phig, Batch bt) {
    extern __shared__ float4 fsm[];
    if constexpr (BAT) {                                     // slot blockIdx.y of a batch
        if (bt.ms && !bt.ms[blockIdx.y].active) {
            chain_wait();
            return;
        }
        const int m = slot_member(bt, blockIdx.y);
        mesh = moved(mesh, m * bt.stride);
        phig = moved(phig, m * bt.stride);
    }
    constexpr int h = N / 2, T = fft_threads(h);
    float4* buf = fsm;                                       // [h][NP]
    float2* stw = reinterpret_cast<float2*>(buf + h * NP);   // [N]
    load_tw<N, T>(stw, tw);
    const int64_t row0 = (int64_t)blockIdx.x * NC;
    chain_wait();
    if (threadIdx.x == 0) {
        const int64_t r = row0 + (int64_t)152 * fft_blocks(h) * NC;
        if (r < (int64_t)N * N) l2_prefetch(mesh + r * S, NC * S * 4);
    }
    constexpr int R1 = x_first_radix<h>();
    xpass_load<h, R1, true, true, T>(buf, mesh, row0, S, tw);
    tile_fft_but_last<h, R1, 2, true, true, T>(buf, stw);
    constexpr int Ns = last_span<h, R1>();
    xpass_store<h, Ns, h / Ns, 2, true, T>(buf, stw, phig, row0);
}

// ------------------------------------------------------------ y sweep
// The tile's first pass reads global memory and its last pass writes it:
// shared memory holds only the intermediate passes.  Columns kx = 0 and
// kx = N/2 are real before the forward sweep and after the inverse one, so
// they share one complex column (x + i y) in tile 0, and N/2 / NC tiles
// cover the N/2 + 1 columns.  Forward, tile 0 separates the two transforms
// by Hermitian symmetry, A(k) = (Z(k) + Z*(N-k)) / 2, B(k) = (Z(k) - Z*(N-k)) / 2i.
template <int N>
constexpr int ntile_x() { return (N / 2 + NC - 1) / NC; }

template <int N, bool INV, bool BAT>
__global__ void __launch_bounds__(fft_threads(N), fft_blocks(N))
    k_fft_y(float* mesh, int S, const float2* __restrict__ tw, Batch bt) {
    extern __shared__ float4 fsm[];
    if constexpr (BAT) {                                     // slot blockIdx.z of a batch
        if (bt.ms && !bt.ms[blockIdx.z].active) {
            chain_wait();
            return;
        }
        mesh = moved(mesh, slot_member(bt, blockIdx.z) * bt.stride);
    }
    constexpr int h = N / 2, T = fft_threads(N);
    float4* buf = fsm;
    float2* stw = reinterpret_cast<float2*>(buf + N * NP);
    load_tw<N, T>(stw, tw);
    chain_wait();
    const int Sc = S / 2;
    const int c0 = blockIdx.x * NC;
    float2* slab = reinterpret_cast<float2*>(mesh) + (int64_t)blockIdx.y * N * Sc;
    constexpr int q = npass(N);
    const int np = h % NC == 0 ? NP : min(NP, (h - c0) / 2), packed = blockIdx.x == 0 ? h : 0;
    col_load<N, INV, T>(buf, slab + c0, Sc, 2, np, packed);
    if (INV || blockIdx.x > 0) {
        col_passes<N, 2, q - 1, INV, T>(buf, stw);
        col_store<N, INV, T>(buf, stw, slab + c0, Sc, 2, np, packed);
    } else {
        col_passes<N, 2, q, INV, T>(buf, stw);
        for (int t = threadIdx.x; t < N * NP; t += T) {
            const int p = t & (NP - 1), ky = t >> LOG_NP;
            if (2 * p >= h) continue;
            float2* row = slab + (int64_t)ky * Sc;
            const C2 z = c2(buf[sidx<false>(ky, p)]);
            float4 f = to_columns(z);
            if (p == 0) {
                const float2 zk = row_of(z, 0), zm = row_of(c2(buf[sidx<false>((N - ky) % N, 0)]), 0);
                f.x = 0.5f * (zk.x + zm.x);
                f.y = 0.5f * (zk.y - zm.y);
                row[h] = make_float2(0.5f * (zk.y + zm.y), 0.5f * (zm.x - zk.x));
            }
            *reinterpret_cast<float4*>(row + 2 * p) = f;
        }
    }
}

// ------------------------------------------------------------ z sweep (+ Green)
// Green's function -(3/2) Om / k^2 / W(k)^p / N^3 of a pair's columns, kz = z
struct GreenPost {
    const float2* tab;           // (k^2, window factor) of each index
    float g0;
    int kx0, ky0;                // pair p: columns kx0 + 2 p, + 1 at ky0, or (edge) column kx0 at ky0 + p
    bool edge;
    __device__ __forceinline__ float at(float2 x, float2 y, float2 z, bool origin) const {
        const float kk = x.x + y.x + z.x;
        // approximate division: within 2 ulp for kk below 2^126 (here kk < 3 pi^2)
        return origin ? 0.0f : __fdividef(g0, kk) * (x.y * y.y * z.y);
    }
    __device__ __forceinline__ float2 operator()(int z, int p) const {
        const int kx = edge ? kx0 : kx0 + 2 * p, ky = edge ? ky0 + p : ky0;
        const float4 x = *reinterpret_cast<const float4*>(&tab[kx]);
        const float2 y = tab[ky], tz = tab[z];
        return make_float2(at(make_float2(x.x, x.y), y, tz, kx == 0 && ky == 0 && z == 0),
                           at(make_float2(x.z, x.w), y, tz, false));
    }
};

// Tiles of 16 consecutive kx at one ky.  The column kx = N/2 would fill a tile
// of its own with one column of 16 at every ky, so up to N = 384 it goes, for
// eight consecutive ky at a time, into edge tiles, the first of the grid (z of
// 12 meshes of 128^3 55 -> 50 us, 192^3 20.5 -> 18.6, 256^3 41 -> 38, 384^3 145
// -> 139; at 512^3 the edge tiles' scattered 16-byte pieces cost more than the
// 6% they save: 312 -> 320).
template <int N>
constexpr int nedge() { return N <= 384 ? N / NP : 0; }
template <int N>
constexpr int ntile_z() { return nedge<N>() ? ntile_x<N>() : (N / 2 + NC) / NC; }
template <int N>
constexpr int ztiles() { return nedge<N>() + ntile_z<N>() * N; }

template <int N, int MODE, bool BAT>   // MODE 0: forward only, 1: forward, Green, inverse
__global__ void __launch_bounds__(fft_threads(N), fft_blocks(N))
    k_fft_z(float* mesh, int S, const float2* __restrict__ tw, const float* __restrict__ k2,
            const float* __restrict__ wdec, float g0, Batch bt) {
    extern __shared__ float4 fsm[];
    if constexpr (BAT) {                                     // slot blockIdx.y of a batch
        if (bt.ms && !bt.ms[blockIdx.y].active) {
            chain_wait();
            return;
        }
        mesh = moved(mesh, slot_member(bt, blockIdx.y) * bt.stride);
    }
    constexpr int h = N / 2, T = fft_threads(N), q = npass(N);
    float4* buf = fsm;
    float2* stw = reinterpret_cast<float2*>(buf + N * NP);
    float2* green = stw + N;     // [N + NC]: a last pair's padding column stays inside
    load_tw<N, T>(stw, tw);
    const int Sc = S / 2;
    const int64_t zs = (int64_t)N * Sc;
    constexpr int ne = nedge<N>(), ncol = ne ? h : h + 1;    // columns of the 16-column tiles
    const bool edge = (int)blockIdx.x < ne;
    const int t = (int)blockIdx.x - ne;
    const int ky = edge ? (int)blockIdx.x * NP : t / ntile_z<N>(), c0 = edge ? h : t % ntile_z<N>() * NC;
    const int ps = edge ? Sc : 2, np = ne && h % NC == 0 ? NP : edge ? NP : min(NP, (ncol - c0 + 1) / 2);
    float2* base = reinterpret_cast<float2*>(mesh) + (int64_t)ky * Sc + c0;
    if (MODE == 1)
        for (int i = threadIdx.x; i < N + NC; i += T)
            green[i] = i < N ? make_float2(__ldg(&k2[i]), __ldg(&wdec[i])) : make_float2(1.0f, 1.0f);
    chain_wait();
    col_load<N, false, T>(buf, base, zs, ps, np);
    col_passes<N, 2, q - 1, false, T>(buf, stw);
    if (MODE == 1) {
        const GreenPost gp{green, g0, c0, ky, edge};
        constexpr bool fuse = rad(N, 1) == rad(N, q);
        col_pass_post<N, fuse, T>(buf, stw, gp);
        col_passes<N, fuse ? 2 : 1, q - 1, true, T>(buf, stw);
        col_store<N, true, T>(buf, stw, base, zs, ps, np);
    } else {
        col_store<N, false, T>(buf, stw, base, zs, ps, np);
    }
}

// ------------------------------------------------------------ largest force component
// max over mesh nodes and axes of |8 (f(+1) - f(-1)) - (f(+2) - f(-2))| / 12 of
// the ghosted potential (the FD4 gradient the force gather interpolates), as
// the bits of a non-negative float
__global__ void k_grad_max(const float* __restrict__ phig, int N, unsigned* __restrict__ out_bits) {
    const int64_t n3 = (int64_t)N * N * N;
    const int64_t sy = phig_nx(N), sz = sy * phig_ny(N);
    float m = 0.0f;
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < n3; t += (int64_t)gridDim.x * blockDim.x) {
        const int x = (int)(t % N), y = (int)((t / N) % N), z = (int)(t / ((int64_t)N * N));
        const float* c = phig + phig_index(N, x, y, z);
        const float gx = 8.0f * (c[1] - c[-1]) - (c[2] - c[-2]);
        const float gy = 8.0f * (c[sy] - c[-sy]) - (c[2 * sy] - c[-2 * sy]);
        const float gz = 8.0f * (c[sz] - c[-sz]) - (c[2 * sz] - c[-2 * sz]);
        m = fmaxf(m, fmaxf(fabsf(gx), fmaxf(fabsf(gy), fabsf(gz))));
    }
    const unsigned b = __reduce_max_sync(0xffffffffu, __float_as_uint(m / 12.0f));
    if ((threadIdx.x & 31) == 0 && b) atomicMax(out_bits, b);
}

// ------------------------------------------------------------ power spectrum
// Sums over the shells i = 1 .. nb, i - 1/2 <= |n| < i + 1/2, of the mode
// weights, weight * |n| and weight * |delta_k|^2 / W^2.
//
// FP64 issues at 1/64 of the FP32 rate here, and FP64 shared atomics are a
// compare-and-swap loop, so neither is in the loop: sums are triples of floats
// (the exact rounding errors of the values in a second word, those of the
// second in a third: the two-sum of Knuth and the FMA product, cascaded as in
// Ogita, Rump and Oishi's DotK, about 2^-70 relative), converted to FP64 once
// per CTA, so no sum has fewer bits than in FP64.  Largest error over meshes of
// 16^3 to 512^3 with known modes, |k| / P: FP64 atomics 1.8e-15 / 1.7e-15, pairs
// of floats (2^-47 an addition) 1.3e-15 / 6.7e-15, triples 4.1e-16 / 3.7e-16.
// The modes are scaled by 2^12, which keeps the error words in range for every
// mode from 2^-62 to 2^30 (a mesh of mean 1 has none larger).  A warp takes the
// rows (|ky|, |kz|) that share their weights and shells, up to four of them
// (+-ky, +-kz), 32 consecutive kx at a time; along kx the shell index never decreases, so equal shells are
// runs of lanes: a segmented scan adds each run and its last lane alone adds it
// to the warp's own bins, without atomics and in a fixed order.  Rows are left
// as soon as they leave the last shell.  512^3 mesh, 256 bins: 4.23 ms with
// FP64 sums and shared atomics -> 0.185 ms (pairs: 0.136 ms), 65% of the issue
// slots; the reduction over blocks 0.170 ms (one thread per bin) -> 0.012 ms
// (one warp per bin).
constexpr int PK_WARPS = 8;
constexpr float PK_SCALE = 4096.0f;

// a sum as h + l + m, and two of them side by side (float2)
struct Triple {
    float h, l, m;
};
struct Triple2 {
    float2 h, l, m;
};
// a + b = a + (returned error), exactly
__device__ __forceinline__ float2 two_sum(float2& a, float2 b) {
    const float2 s = padd(a, b), z = psub(s, a);
    const float2 e = padd(psub(a, psub(s, z)), psub(b, z));
    a = s;
    return e;
}
__device__ __forceinline__ float two_sum(float& a, float b) {
    const float s = __fadd_rn(a, b), z = __fsub_rn(s, a);
    const float e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, z)), __fsub_rn(b, z));
    a = s;
    return e;
}
__device__ __forceinline__ void add(Triple2& t, const Triple2& b) {
    const float2 e0 = two_sum(t.h, b.h);
    const float2 e1 = two_sum(t.l, b.l);
    const float2 e2 = two_sum(t.l, e0);
    t.m = padd(t.m, padd(b.m, padd(e1, e2)));
}
__device__ __forceinline__ void add(Triple& t, const Triple& b) {
    const float e0 = two_sum(t.h, b.h);
    const float e1 = two_sum(t.l, b.l);
    const float e2 = two_sum(t.l, e0);
    t.m = __fadd_rn(t.m, __fadd_rn(b.m, __fadd_rn(e1, e2)));
}
// t += x^2 (the square exactly: q and its error)
__device__ __forceinline__ void add_square(Triple2& t, float2 x) {
    const float2 q = pmul(x, x), e = pfma(x, x, make_float2(-q.x, -q.y));
    const float2 e0 = two_sum(t.h, q);
    const float2 e1 = two_sum(t.l, e);
    const float2 e2 = two_sum(t.l, e0);
    t.m = padd(t.m, padd(e1, e2));
}
// a b: the products down to the third word, their errors down to the second
__device__ __forceinline__ Triple mul(const Triple& a, const Triple& b) {
    Triple r;
    r.h = __fmul_rn(a.h, b.h);
    r.l = __fmaf_rn(a.h, b.h, -r.h);
    const float p = __fmul_rn(a.h, b.l), q = __fmul_rn(a.l, b.h);
    float m = __fadd_rn(__fmaf_rn(a.h, b.l, -p), __fmaf_rn(a.l, b.h, -q));
    m = __fmaf_rn(a.l, b.l, __fmaf_rn(a.h, b.m, __fmaf_rn(a.m, b.h, m)));
    const float e0 = two_sum(r.l, p);
    const float e1 = two_sum(r.l, q);
    r.m = __fadd_rn(m, __fadd_rn(e0, e1));
    return r;
}
__device__ __forceinline__ Triple triple(double x) {
    const float h = (float)x;
    const double d = x - (double)h;
    const float l = (float)d;
    return Triple{h, l, (float)(d - (double)l)};
}
__device__ __forceinline__ double value(const Triple& t) { return (double)t.h + ((double)t.l + (double)t.m); }

// shell of the integer n2 = |n|^2 <= 3 (N / 2)^2: |n| is never within 1.4e-4 of
// a half-integer (n2 = i^2 + i lies 1/8 / i below one) and the correctly
// rounded root within 3e-5 of |n| (checked for every n2 up to N = 1024)
__device__ __forceinline__ int pk_shell(float n2, float* root) {
    *root = __fsqrt_rn(n2);
    return __float2int_rn(*root);
}

__global__ void __launch_bounds__(PK_WARPS * 32) k_pk_bin(const float* __restrict__ mesh, int N, int S, int nb,
                                                          int nbins, const double* __restrict__ wpk,
                                                          double* __restrict__ part) {
    extern __shared__ Triple pk_smem[];
    const int M = N / 2 + 1, Sc = S / 2;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    Triple* wt = pk_smem;                                        // [M] window weights
    Triple* sp = wt + M;                                         // [PK_WARPS][nb] power
    Triple* sk = sp + PK_WARPS * nb;                             // [PK_WARPS][nb] |n|
    unsigned* sc = reinterpret_cast<unsigned*>(sk + PK_WARPS * nb);   // [PK_WARPS][nb] weights
    for (int i = threadIdx.x; i < M; i += blockDim.x) wt[i] = triple(wpk[i]);
    for (int i = threadIdx.x; i < PK_WARPS * nb; i += blockDim.x) {
        sp[i] = sk[i] = Triple{0.0f, 0.0f, 0.0f};
        sc[i] = 0u;
    }
    __syncthreads();
    Triple* wp = sp + warp * nb - 1;                             // bins from shell 1
    Triple* wk = sk + warp * nb - 1;
    unsigned* wc = sc + warp * nb - 1;
    const float2* base = reinterpret_cast<const float2*>(mesh);
    const int nw = gridDim.x * PK_WARPS;
    for (int it = blockIdx.x * PK_WARPS + warp; it < M * M; it += nw) {
        const int b = it / M, a = it - b * M;                    // |kz|, |ky|
        const int ay = a > 0 && a < N / 2 ? N - a : a, bz = b > 0 && b < N / 2 ? N - b : b;
        const bool ry = ay != a, rz = bz != b;                   // the mirrored rows exist
        const float2* r0 = base + ((int64_t)b * N + a) * Sc;
        const float2* r1 = base + ((int64_t)b * N + ay) * Sc;
        const float2* r2 = base + ((int64_t)bz * N + a) * Sc;
        const float2* r3 = base + ((int64_t)bz * N + ay) * Sc;
        const float rows = (ry ? 2.0f : 1.0f) * (rz ? 2.0f : 1.0f);
        const float c2 = (float)(a * a + b * b);
        const Triple wab = mul(wt[a], wt[b]);
        const float2 zero = make_float2(0.0f, 0.0f);
        float2 n0, n1, n2v, n3;
        auto fetch = [&](int kx) {
            const bool ok = kx < M;
            n0 = ok ? r0[kx] : zero;
            n1 = ok && ry ? r1[kx] : zero;
            n2v = ok && rz ? r2[kx] : zero;
            n3 = ok && ry && rz ? r3[kx] : zero;
        };
        fetch(lane);
        for (int kx0 = 0; kx0 < M; kx0 += 32) {
            float root;
            if (pk_shell(c2 + (float)(kx0 * kx0), &root) > nb) break;     // the rest of the row lies outside
            const float2 v0 = n0, v1 = n1, v2 = n2v, v3 = n3;
            const int kx = kx0 + lane;
            if (kx0 + 32 < M) fetch(kx + 32);
            // real and imaginary parts side by side, then together
            const float2 sc2 = pk2(PK_SCALE);
            const float2 y = pmul(sc2, v0), y2 = pmul(y, y);
            Triple2 s2{y2, pfma(y, y, make_float2(-y2.x, -y2.y)), zero};
            if (ry) add_square(s2, pmul(sc2, v1));
            if (rz) add_square(s2, pmul(sc2, v2));
            if (ry && rz) add_square(s2, pmul(sc2, v3));
            Triple p{s2.h.x, s2.l.x, s2.m.x};
            add(p, Triple{s2.h.y, s2.l.y, s2.m.y});
            p = mul(p, wt[min(kx, M - 1)]);
            const float mult = kx == 0 || kx == N / 2 ? 1.0f : 2.0f;
            const float q2 = c2 + (float)(kx * kx);              // exact: < 2^24
            int shell = pk_shell(q2, &root);
            if (kx >= M) shell = 0x7fffffff;
            // |n| = root + l + x: q2 - root^2 is exact, then (root + l + x)^2 = q2
            const float inv = shell > 0 ? __fdividef(0.5f, root) : 0.0f;
            const float d = __fmaf_rn(-root, root, q2), l = __fmul_rn(d, inv);
            const float x = __fmul_rn(__fmaf_rn(-2.0f * root, l, d) - __fmul_rn(l, l), inv);
            // power and |n| side by side
            const float2 mu = pk2(mult);
            Triple2 t{pmul(mu, make_float2(p.h, root)), pmul(mu, make_float2(p.l, l)), pmul(mu, make_float2(p.m, x))};
            // runs of equal shells
            const int before = __shfl_up_sync(0xffffffffu, shell, 1);
            const unsigned heads = __ballot_sync(0xffffffffu, lane == 0 || shell != before);
            const int head = 31 - __clz((int)(heads & (0xffffffffu >> (31 - lane))));
            for (int o = 1; o < 32; o <<= 1) {
                const bool in = lane - o >= head;
                if (!__any_sync(0xffffffffu, in)) break;         // no run is longer than o
                auto up = [&](float2 v) {
                    return make_float2(__shfl_up_sync(0xffffffffu, v.x, o), __shfl_up_sync(0xffffffffu, v.y, o));
                };
                const Triple2 u{up(t.h), up(t.l), up(t.m)};
                if (in) add(t, u);
            }
            const bool tail = lane == 31 || ((heads >> (lane + 1)) & 1u);
            if (tail && shell >= 1 && shell <= nb) {
                const Triple w = mul(Triple{t.h.x, t.l.x, t.m.x}, wab), ap = wp[shell], ak = wk[shell];
                Triple2 acc{make_float2(ap.h, ak.h), make_float2(ap.l, ak.l), make_float2(ap.m, ak.m)};
                add(acc, Triple2{make_float2(w.h, rows * t.h.y), make_float2(w.l, rows * t.l.y),
                                 make_float2(w.m, rows * t.m.y)});
                wp[shell] = Triple{acc.h.x, acc.l.x, acc.m.x};
                wk[shell] = Triple{acc.h.y, acc.l.y, acc.m.y};
                const int len = lane - head + 1;
                const int cnt = 2 * len - (kx0 + head == 0) - (kx == N / 2);
                wc[shell] += (unsigned)cnt * (unsigned)rows;
            }
            __syncwarp();
        }
    }
    __syncthreads();
    double* out = part + (int64_t)blockIdx.x * 3 * nbins;
    for (int i = threadIdx.x; i < nb; i += blockDim.x) {
        Triple2 s{make_float2(0.0f, 0.0f), make_float2(0.0f, 0.0f), make_float2(0.0f, 0.0f)};
        double c = 0.0;
        for (int w = 0; w < PK_WARPS; ++w) {
            const Triple vp = sp[w * nb + i], vk = sk[w * nb + i];
            c += (double)sc[w * nb + i];
            add(s, Triple2{make_float2(vp.h, vk.h), make_float2(vp.l, vk.l), make_float2(vp.m, vk.m)});
        }
        out[i] = c;
        out[nbins + i] = value(Triple{s.h.y, s.l.y, s.m.y});
        out[2 * nbins + i] = value(Triple{s.h.x, s.l.x, s.m.x}) * (1.0 / ((double)PK_SCALE * PK_SCALE));
    }
}

// shells that can hold modes: up to the corner |n| = sqrt(3) N / 2 < 7 N / 8
__host__ __device__ __forceinline__ int pk_used_bins(int N, int nbins) { return min(nbins, 7 * N / 8); }

// window weights, and each warp's sums of nb bins
size_t pk_bytes(int N, int nb) {
    return (size_t)(N / 2 + 1) * sizeof(Triple) + (size_t)PK_WARPS * nb * (2 * sizeof(Triple) + sizeof(unsigned));
}

// one warp per bin: the blocks' sums in a fixed order; bins from nb on lie
// beyond the mesh's corner and hold no mode
__global__ void k_pk_reduce(const double* __restrict__ part, int nblocks, int nb, int nbins, double pfac, double kfund,
                            double* k, double* pk, double* nm) {
    const int b = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (b >= nbins) return;
    double w = 0, ks = 0, ps = 0;
    if (b < nb)
        for (int j = lane; j < nblocks; j += 32) {
            const double* p = part + (int64_t)j * 3 * nbins;
            w += p[b];
            ks += p[nbins + b];
            ps += p[2 * nbins + b];
        }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        w += __shfl_down_sync(0xffffffffu, w, o);
        ks += __shfl_down_sync(0xffffffffu, ks, o);
        ps += __shfl_down_sync(0xffffffffu, ps, o);
    }
    if (lane == 0) {
        nm[b] = w;
        k[b] = w > 0 ? kfund * ks / w : nan("");
        pk[b] = w > 0 ? pfac * ps / w : nan("");
    }
}

// The N^3 values of an array with padded rows (row (z, y) starts at
// src + (z ny + y) rs), packed: one row a warp, 16 bytes a lane when `out`
// allows it (N, rs and the padded rows' starts are multiples of 4 floats).
// Bound by its reads and writes; 384^3: 0.171 ms (mesh) and 0.242 ms
// (ghosted Phi) with one value a thread and 64-bit divisions ->
// 0.063 ms; the density needs no copy where its rows can be written packed.
__global__ void __launch_bounds__(256) k_unpad(const float* __restrict__ src, int N, int rs, int ny,
                                               float* __restrict__ out, bool vec) {
    const int lane = threadIdx.x & 31;
    const int nrow = N * N;
    for (int row = blockIdx.x * 8 + (threadIdx.x >> 5); row < nrow; row += gridDim.x * 8) {
        const int z = row / N, y = row - z * N;
        const float* s = src + ((int64_t)z * ny + y) * rs;
        float* o = out + (int64_t)row * N;
        if (vec)
            for (int x = lane; x < N / 4; x += 32) reinterpret_cast<float4*>(o)[x] = reinterpret_cast<const float4*>(s)[x];
        else
            for (int x = lane; x < N; x += 32) o[x] = s[x];
    }
}

// twiddles (N) + tile (n x NP pairs)
size_t tile_smem(int N, int n) { return (size_t)N * sizeof(float2) + (size_t)n * NP * sizeof(float4); }
// the z sweep's, with the Green's function tables
size_t ztile_smem(int N) { return tile_smem(N, N) + (size_t)2 * (N + NC) * sizeof(float); }

template <int N>
struct Sweeps {
    template <bool BAT>
    static void attrs_for() {
        if constexpr (BAT && !(N <= 256)) return;
        else {
        const int big = (int)tile_smem(N, N), half = (int)tile_smem(N, N / 2), bigz = (int)ztile_smem(N);
        cudaFuncSetAttribute(k_fft_x_r2c<N, BAT>, cudaFuncAttributeMaxDynamicSharedMemorySize, half);
        cudaFuncSetAttribute(k_fft_x_c2r<N, BAT>, cudaFuncAttributeMaxDynamicSharedMemorySize, half);
        cudaFuncSetAttribute(k_fft_y<N, false, BAT>, cudaFuncAttributeMaxDynamicSharedMemorySize, big);
        cudaFuncSetAttribute(k_fft_y<N, true, BAT>, cudaFuncAttributeMaxDynamicSharedMemorySize, big);
        cudaFuncSetAttribute(k_fft_z<N, 0, BAT>, cudaFuncAttributeMaxDynamicSharedMemorySize, bigz);
        cudaFuncSetAttribute(k_fft_z<N, 1, BAT>, cudaFuncAttributeMaxDynamicSharedMemorySize, bigz);
        }
    }
    // instances with a member dimension exist for the small meshes, where a
    // step is launch-bound; a batch of larger meshes is launched member by member
    static constexpr bool kBatchable = N <= 256;
    static void attrs() {
        static bool done = false;
        if (done) return;
        attrs_for<false>();
        if constexpr (kBatchable) attrs_for<true>();
        done = true;
    }
    // a batch (several members or a per-member table) takes the instances with a member dimension
    static bool batched(const Batch& bt) { return bt.members > 1 || bt.ms != nullptr; }
    // slot by slot from the host: the members the launch lists
    template <class Fn>
    static void per_member(const Batch& bt, Fn fn) {
        for (int i = 0; i < bt.members; ++i) fn((size_t)slot_member(bt, i) * bt.stride);
    }
    static void x_r2c(const FftPlan& p, float* mesh, int S, cudaStream_t st, const Batch& bt) {
        attrs();
        if constexpr (kBatchable) {
            if (batched(bt)) {
                launch_chained(k_fft_x_r2c<N, true>, dim3((N * N) / NC, bt.members), fft_threads(N / 2), tile_smem(N, N / 2), st, mesh, S,
                                                                                                         p.tw, bt);
                return;
            }
        }
        per_member(bt, [&](size_t o) {
            launch_chained(k_fft_x_r2c<N, false>, (N * N) / NC, fft_threads(N / 2), tile_smem(N, N / 2), st, moved(mesh, o), S, p.tw, kSingle);
        });
    }
    static void y(const FftPlan& p, float* mesh, int S, bool inv, cudaStream_t st, const Batch& bt) {
        attrs();
        const size_t sm = tile_smem(N, N);
        if constexpr (kBatchable) {
            if (batched(bt)) {
                const dim3 gy(ntile_x<N>(), N, bt.members);
                if (inv) launch_chained(k_fft_y<N, true, true>, gy, fft_threads(N), sm, st, mesh, S, p.tw, bt);
                else launch_chained(k_fft_y<N, false, true>, gy, fft_threads(N), sm, st, mesh, S, p.tw, bt);
                return;
            }
        }
        const dim3 gy(ntile_x<N>(), N);
        per_member(bt, [&](size_t o) {
            if (inv) launch_chained(k_fft_y<N, true, false>, gy, fft_threads(N), sm, st, moved(mesh, o), S, p.tw, kSingle);
            else launch_chained(k_fft_y<N, false, false>, gy, fft_threads(N), sm, st, moved(mesh, o), S, p.tw, kSingle);
        });
    }
    static void z(const FftPlan& p, float* mesh, int S, float g0, bool green, cudaStream_t st, const Batch& bt) {
        attrs();
        const size_t sm = ztile_smem(N);
        if constexpr (kBatchable) {
            if (batched(bt)) {
                const dim3 gz(ztiles<N>(), bt.members);
                if (green) launch_chained(k_fft_z<N, 1, true>, gz, fft_threads(N), sm, st, mesh, S, p.tw, p.k2, p.wdec, g0, bt);
                else launch_chained(k_fft_z<N, 0, true>, gz, fft_threads(N), sm, st, mesh, S, p.tw, p.k2, p.wdec, g0, bt);
                return;
            }
        }
        const dim3 gz(ztiles<N>());
        per_member(bt, [&](size_t o) {
            if (green) launch_chained(k_fft_z<N, 1, false>, gz, fft_threads(N), sm, st, moved(mesh, o), S, p.tw, p.k2, p.wdec, g0, kSingle);
            else launch_chained(k_fft_z<N, 0, false>, gz, fft_threads(N), sm, st, moved(mesh, o), S, p.tw, p.k2, p.wdec, g0, kSingle);
        });
    }
    static void x_c2r(const FftPlan& p, float* mesh, int S, float* phig, cudaStream_t st, const Batch& bt) {
        attrs();
        if constexpr (kBatchable) {
            if (batched(bt)) {
                launch_chained(k_fft_x_c2r<N, true>, dim3((N * N) / NC, bt.members), fft_threads(N / 2), tile_smem(N, N / 2), st, mesh, S,
                                                                                                         p.tw, phig, bt);
                return;
            }
        }
        per_member(bt, [&](size_t o) {
            launch_chained(k_fft_x_c2r<N, false>, (N * N) / NC, fft_threads(N / 2), tile_smem(N, N / 2), st, moved(mesh, o), S, p.tw,
                                                                                     moved(phig, o), kSingle);
        });
    }
};

// mesh sizes with compiled sweeps: 2^a and 3 * 2^a from 16 to 1024
#define CUBE_FFT_SIZES(X) X(16) X(24) X(32) X(48) X(64) X(96) X(128) X(192) X(256) X(384) X(512) X(768) X(1024)

}  // namespace

bool fft_size_supported(int N) {
    switch (N) {
#define CASE(n) case n:
        CUBE_FFT_SIZES(CASE)
#undef CASE
        return true;
        default: return false;
    }
}

#define DISPATCH()                                       \
    switch (p.N) {                                       \
        CUBE_FFT_SIZES(DCASE)                            \
        default: break;                                  \
    }

void fft_x_r2c(const FftPlan& p, float* mesh, int S, cudaStream_t st, const Batch& bt) {
#define DCASE(n) case n: Sweeps<n>::x_r2c(p, mesh, S, st, bt); break;
    DISPATCH()
#undef DCASE
}

void fft_y(const FftPlan& p, float* mesh, int S, bool inverse, cudaStream_t st, const Batch& bt) {
#define DCASE(n) case n: Sweeps<n>::y(p, mesh, S, inverse, st, bt); break;
    DISPATCH()
#undef DCASE
}

void fft_z(const FftPlan& p, float* mesh, int S, float g0, bool green, cudaStream_t st, const Batch& bt) {
#define DCASE(n) case n: Sweeps<n>::z(p, mesh, S, g0, green, st, bt); break;
    DISPATCH()
#undef DCASE
}

void fft_x_c2r(const FftPlan& p, float* mesh, int S, float* phig, cudaStream_t st, const Batch& bt) {
#define DCASE(n) case n: Sweeps<n>::x_c2r(p, mesh, S, phig, st, bt); break;
    DISPATCH()
#undef DCASE
}

// three CTAs per SM, each warp with at least one group of rows
int pk_blocks(int N) {
    const int M = N / 2 + 1;
    return min(3 * 152, (M * M + PK_WARPS - 1) / PK_WARPS);
}

void launch_pk_bin(const FftPlan& p, const float* mesh, int S, int nbins, double* part, cudaStream_t st) {
    const int nb = pk_used_bins(p.N, nbins);
    // the limit is the kernel's, not this launch's: always the largest mesh's, so
    // that a call on another thread cannot lower it between here and the launch
    cudaFuncSetAttribute(k_pk_bin, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)pk_bytes(1024, pk_used_bins(1024, 1024)));
    k_pk_bin<<<pk_blocks(p.N), PK_WARPS * 32, pk_bytes(p.N, nb), st>>>(mesh, p.N, S, nb, nbins, p.wpk, part);
}

void launch_pk_reduce(const FftPlan& p, const double* part, int nbins, double pfac, double kfund, double* k, double* pk,
                      double* nm, cudaStream_t st) {
    k_pk_reduce<<<(nbins + 3) / 4, 128, 0, st>>>(part, pk_blocks(p.N), pk_used_bins(p.N, nbins), nbins, pfac, kfund, k,
                                                pk, nm);
}

void launch_grad_max(const float* phig, int N, unsigned* out_bits, cudaStream_t st) {
    cudaMemsetAsync(out_bits, 0, sizeof(unsigned), st);
    k_grad_max<<<4 * 152, 256, 0, st>>>(phig, N, out_bits);
}

static void unpad(const float* src, int N, int rs, int ny, float* out, cudaStream_t st) {
    const bool vec = (reinterpret_cast<uintptr_t>(out) & 15) == 0;
    k_unpad<<<(N * N + 7) / 8, 256, 0, st>>>(src, N, rs, ny, out, vec);
}

void launch_unpad_phig(const float* phig, int N, float* out, cudaStream_t st) {
    unpad(phig + phig_index(N, 0, 0, 0), N, phig_nx(N), phig_ny(N), out, st);
}

void launch_unpad(const float* mesh, int N, int S, float* out, cudaStream_t st) { unpad(mesh, N, S, N, out, st); }

}  // namespace cube
