// m2l_oz.cu -- the FP64 and FP32 M2L (S|R part of Eq. 2.21) on the GB300 tensor cores.
//
// GB300 runs FP64 at about 1/60 of its FP32 rate, and the double-precision M2L on the FP64 pipe was
// bound by it (the folded rotation form 88 % busy at p = 10, the dense many-column form at p = 8).
// Here each double is cut into OZ_S = 8 signed 8-bit digits (the error-free transformation of Ozaki,
// Ogita, Oishi and Rump, "Error-free transformations of matrix multiplication", 2012), every digit is
// an exact bf16, and the products of digits are summed exactly: a digit product is at most 2^14 units,
// so that the sums over K = 2 p^2 <= 200 stay below the 24 bits that FP32 tensor memory holds.
//
//   S|R[R][K] 2^(s_K - er_R) = sum_i T_i[R][K] 2^(-7 - 8 i),   C[K][col] 2^(-s_K - ec_col) likewise,
//   Y[R][col] = 2^(er_R + ec_col) sum_{d = 0..7} sum_{i + j = d} T_i C_j   (d > 7 is below 2^-64).
//
// s_K (one power of two per degree, domain and level) balances the matrices, whose entries grow like
// double factorials of the degrees while the expansions shrink; er (per matrix row) and ec (per source
// column) bring the largest entries to [1/2, 1).  The diagonals d = 0..4 have a tensor-memory accumulator
// each (exact); d = 5..7 share one, whose FP32 rounding is below 2^-60.  The six sums are added without
// error in FP32 pairs and rounded once to a double.  Measured on pair results against quad
// precision (rms relative error, torus of 3840 nodes): p = 8 8e-17 and p = 10 3e-16, where the FP64 sums
// of the dense form have 5e-16 and the rotation form 1e-8 (a seven-digit form had 6e-16 and 1.5e-15).
//
// The digits are fixed-point: an entry is held to 2^-63 of the largest balanced one of its matrix row or source
// column, and the products with i + j > 7 are left out.  An FP64 entry more than 2^-10 below the largest has fewer
// bits than a double (a single-precision one more than 2^-7 below, with four digits: 2^-31), so that the error is
// small against the norm of a row's products, not against each of them.  The balance by degree keeps the
// entries that matter within that range.
//
// A single-precision product takes the first four digits of the same images and four digits of its sources
// (2^-31 of the largest entry), ten products in four exact accumulators, added once in FP32: more exact than
// the FP32 sums it replaces (product errors against FP64, torus of 9216 nodes: p = 8, 16 right-hand sides
// 5.1e-7 with the dense sums, 1.3e-7; p = 10, 3 right-hand sides 1.2e-7 with the rotation form, 1.0e-7), and
// faster at every size (a whole product: sphere of 642 nodes 135 -> 104 us, 40962 nodes p = 10 1.69 -> 1.03 ms,
// torus of 9216 nodes with 16 right-hand sides 8.3 -> 2.4 ms).
//
// S|S and R|R between levels run the same way in double precision: the children of a level grouped by octant
// (torus of 9216 nodes, 16 right-hand sides, p = 8: M2M 2.18 and L2L 2.4 ms on the FP64 pipe, product 16.8 ms,
// now 13.2; p = 10, three right-hand sides: in rotation form 6.19 ms and 5e-13 from the dense form, now 4.63 ms
// and 2e-16).  In single precision the forms on the FP32 pipe are as fast (10242 nodes, p = 10: product 0.41
// ms, 0.45 in digits; 9216 nodes, three right-hand sides: 1.28, 1.15) and stay.
//
// The FF pairs of one level and offset share a matrix; their columns (W per pair) follow one another
// and are cut into tiles of N columns, the N of the MMAs (FP64: 80, six accumulators of 80 columns fill tensor
// memory; FP32: 128, four accumulators); the matrix rows are its M = 128 (one row tile for p <= 8, two for p = 10).  The results go to
// Y[pair][column], which k_l2l_reduce sums per target.
#include <algorithm>
#include <string>

#include "fmbem_internal.cuh"
#include "tc_ptx.cuh"

namespace {

constexpr int OZ_S = 8;      // digits per double
constexpr int OZ_SLOTS = 4;  // operand ring: one K block of 16 each
constexpr int OZ_FILL = 3;   // producer warps
constexpr int OZ_EPI = 16;   // epilogue warps
constexpr int OZ_NONFINITE = 1 << 20;  // exponent marking a column or row with an Inf or a NaN
constexpr uint32_t OZ_A_BYTES = OZ_S * TC_M * 32u;  // the matrix digits of one K block
template <typename R>
struct Oz;
template <>
struct Oz<double> {
    static constexpr int S = OZ_S;  // digits
    static constexpr int N = 80;    // pair columns per tile
    static constexpr int ACC = 6;   // accumulators: d = 0, 1, 2, 3, 4 and 5..7
};
template <>
struct Oz<float> {
    static constexpr int S = 4, N = 128, ACC = 4;  // d = 0..3
};
template <typename R>
constexpr uint32_t oz_a_bytes = Oz<R>::S * TC_M * 32u;
template <typename R>
constexpr uint32_t oz_slot_bytes = oz_a_bytes<R> + Oz<R>::S * Oz<R>::N * 32u;
template <typename R>
constexpr int oz_row = Oz<R>::S * 32;  // bytes of a source column's digits in one K block
constexpr int OZ_MAX_LEVELS = 12;
constexpr int OZ_THREADS = 32 * (OZ_FILL + 1 + OZ_EPI);
static_assert(OZ_SLOTS == 4 && OZ_FILL == 3 && OZ_EPI == 16 && OZ_S == 8 && Oz<double>::ACC * Oz<double>::N <= 512 &&
                  Oz<float>::ACC * Oz<float>::N <= 512,
              "ring arithmetic, tensor-memory lanes of the epilogue warps, digit arithmetic, tensor memory");

// byte offset of the 16-byte chunk c (0, 1) of a row in the 32-byte-swizzled K-major layout
__host__ __device__ __forceinline__ uint32_t sw32_chunk(int row, int c) {
    return (uint32_t)(row * 32 + ((c ^ (row >> 2)) & 1) * 16);
}
// shared-memory matrix descriptor, K-major, 32-byte swizzle: 8-row groups 256 bytes apart
__device__ __forceinline__ uint64_t smem_desc_sw32(uint32_t saddr) {
    uint64_t d = (uint64_t)((saddr & 0x3FFFFu) >> 4);
    d |= (uint64_t)1 << 16;
    d |= (uint64_t)(256 >> 4) << 32;
    d |= (uint64_t)1 << 46;
    d |= (uint64_t)6 << 61;
    return d;
}

struct OzLevels {  // first box of each level (levels 2..lmax), for the level of a box
    int lmax;
    int64_t off[OZ_MAX_LEVELS + 2];
};

// exponent e with |x| < 2^e for the larger of two doubles (zero: very small; Inf, NaN: OZ_NONFINITE)
__device__ __forceinline__ int oz_exp2(double a, double b) {
    const int ea = (__double2hiint(a) >> 20) & 0x7ff, eb = (__double2hiint(b) >> 20) & 0x7ff;
    const int e = max(ea, eb);
    if (e == 0x7ff) return OZ_NONFINITE;
    if (e == 0) return a == 0.0 && b == 0.0 ? -OZ_NONFINITE : -1022;
    return e - 1022;
}

__device__ __forceinline__ int oz_exp2(float a, float b) {
    const int ea = (__float_as_int(a) >> 23) & 0xff, eb = (__float_as_int(b) >> 23) & 0xff;
    const int e = max(ea, eb);
    if (e == 0xff) return OZ_NONFINITE;
    if (e == 0) return a == 0.f && b == 0.f ? -OZ_NONFINITE : -126;
    return e - 126;
}

// the digits of x 2^shift (|x 2^shift| < 1), each as the bf16 bits of digit 2^(-7 - 8 i); a float has
// 24 bits, so that 2^31 times it is an int
__device__ __forceinline__ void oz_digits(float x, int shift, uint16_t *out) {
    constexpr int S = Oz<float>::S;
    int m = __float2int_rn(ldexpf(x, shift + 8 * S - 1));
#pragma unroll
    for (int i = S - 1; i >= 0; --i) {
        const int dgt = i > 0 ? (int)(int8_t)(m & 0xff) : m;
        // (m - dgt may pass 2^31 - 1 by less than 2^7: the last digits' carry into the first)
        if (i > 0) m = (m >> 8) + (dgt < 0 ? 1 : 0);
        const float f = (float)dgt * __int_as_float((127 - 7 - 8 * i) << 23);
        out[i] = (uint16_t)(__float_as_uint(f) >> 16);
    }
}
__device__ __forceinline__ void oz_digits(double x, int shift, uint16_t *out) {
    long long m = __double2ll_rn(ldexp(x, shift + 8 * OZ_S - 1));
#pragma unroll
    for (int i = OZ_S - 1; i >= 0; --i) {
        const int dgt = i > 0 ? (int)(int8_t)(m & 0xff) : (int)m;
        if (i > 0) m = (m - dgt) >> 8;
        const float f = (float)dgt * __int_as_float((127 - 7 - 8 * i) << 23);
        out[i] = (uint16_t)(__float_as_uint(f) >> 16);  // at most 8 significant bits: exact
    }
}

// s_K per (domain, level) and degree n: minus half the exponent of the largest entry between
// coefficients of degree n, over all 316 offsets, less n / 4 (expansions of surface nodes shrink a
// little faster with the degree than that; measured 1.3 to 2 times more exact than without); grid
// (matrix sets, degree)
__global__ void k_oz_balance(const c64 *T, int p, int lmax, int *bal) {
    const int set = blockIdx.x, n = blockIdx.y, p2 = p * p;
    const int d = set / (lmax - 1), l = 2 + set % (lmax - 1), w = 2 * n + 1;
    const c64 *M = T + m2l_matrix(d, l, 0, lmax) * p2 * p2;
    int e = -OZ_NONFINITE;
    for (int i = threadIdx.x; i < 316 * w * w; i += blockDim.x) {
        const int o = i / (w * w), c = n * n + (i / w) % w, r = n * n + i % w;
        const c64 t = M[((int64_t)o * p2 + c) * p2 + r];
        const int x = oz_exp2(t.re, t.im);
        if (x < OZ_NONFINITE) e = max(e, x);
    }
    __shared__ int best;
    if (threadIdx.x == 0) best = -OZ_NONFINITE;
    __syncthreads();
    atomicMax(&best, e);
    __syncthreads();
    if (threadIdx.x == 0) bal[set * p + n] = best > -OZ_NONFINITE ? -(best >> 1) - n / 4 : 0;
}

__device__ __forceinline__ int oz_degree(int q) {
    int n = 0;
    while ((n + 1) * (n + 1) <= q) ++n;
    return n;
}

// exponent by which the sources of degree n are scaled down: s_K for multipole expansions; for the local
// expansions of R|R, which grow where the multipole ones shrink, the opposite, less the same n / 4
__device__ __forceinline__ int oz_scale_of(const int *bal, int n, bool local) {
    return local ? -bal[n] - n / 2 : bal[n];
}

// digit images of the matrices of one kind (per of them per domain and level l0 .. l0 + nlev - 1, T's set of a
// domain having lmax + 1 levels; sources of level lsrc ..): block per matrix; per (row tile, K block) eight
// digit blocks of 128 rows x 16 K in the 32-byte-swizzled K-major layout, real-form rows 2r + a as in m2l_tc.cu
__global__ void __launch_bounds__(256) k_oz_images(const c64 *T, int p, int lmax, int per, int l0, int nlev, int lsrc, bool local,
                                                   int mt, int kblocks, const int *bal, unsigned char *img, int *er) {
    const int64_t mat = blockIdx.x;
    const int set = (int)(mat / per), o = (int)(mat % per), p2 = p * p;
    const int d = set / nlev, l = set % nlev;
    const c64 *M = T + (((int64_t)d * (lmax + 1) + l0 + l) * per + o) * p2 * p2;
    bal += (d * (lmax - 1) + lsrc - 2 + l) * p;
    __shared__ int s_er[400], s_bal[400];
    for (int c = threadIdx.x; c < p2; c += blockDim.x) s_bal[c] = oz_scale_of(bal, oz_degree(c), local);
    __syncthreads();
    for (int r = threadIdx.x; r < p2; r += blockDim.x) {
        int e = -OZ_NONFINITE;
        for (int c = 0; c < p2; ++c) {
            const c64 t = M[(int64_t)c * p2 + r];
            const int x = oz_exp2(t.re, t.im);
            e = max(e, x == OZ_NONFINITE ? x : x + s_bal[c]);
        }
        if (e < -OZ_NONFINITE / 2) e = 0;
        if (e > OZ_NONFINITE / 2) e = OZ_NONFINITE;
        s_er[r] = e;
        er[mat * p2 + r] = e;
    }
    __syncthreads();
    unsigned char *out = img + mat * (int64_t)mt * kblocks * OZ_A_BYTES;
    const int chunks = kblocks * 2;  // 16-byte chunks (eight K values) of a row
    for (int i = threadIdx.x; i < mt * TC_M * chunks; i += blockDim.x) {
        const int R = i / chunks, ch = i % chunks, kb = ch >> 1, r = R >> 1, a = R & 1;
        uint16_t w[OZ_S][8];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int c = ch * 4 + j;
            c64 t = {0.0, 0.0};
            int sh = 0;
            if (r < p2 && c < p2 && s_er[r] != OZ_NONFINITE) {
                t = M[(int64_t)c * p2 + r];
                sh = s_bal[c] - s_er[r];
            }
            uint16_t u[OZ_S], v[OZ_S];
            oz_digits(a == 0 ? t.re : t.im, sh, u);    // [[Re, -Im], [Im, Re]]
            oz_digits(a == 0 ? -t.im : t.re, sh, v);
#pragma unroll
            for (int k = 0; k < OZ_S; ++k) {
                w[k][2 * j] = u[k];
                w[k][2 * j + 1] = v[k];
            }
        }
        unsigned char *blk = out + ((int64_t)(R / TC_M) * kblocks + kb) * OZ_A_BYTES;
        const uint32_t at = sw32_chunk(R % TC_M, ch & 1);
#pragma unroll
        for (int k = 0; k < OZ_S; ++k)
            *reinterpret_cast<uint4 *>(blk + k * (TC_M * 32) + at) =
                make_uint4(w[k][0] | (uint32_t)w[k][1] << 16, w[k][2] | (uint32_t)w[k][3] << 16,
                           w[k][4] | (uint32_t)w[k][5] << 16, w[k][6] | (uint32_t)w[k][7] << 16);
    }
}

// digits of the expansions, columns col0 .. col0 + W - 1 of the boxes b0 .. b0 + nb - 1 (levels >= 2): a warp
// per (domain, box, column) row; row (d nbox + box) W + c holds per K block its digit rows of 32
// bytes, and ec its exponent
template <typename R>
__global__ void __launch_bounds__(256) k_oz_split(const cx<R> *C, const OzLevels L, int64_t b0, int64_t nb, bool local,
                                                  int64_t nbox, int64_t ncols, int col0, int W, int ndom, int p, int kblocks,
                                                  const int *bal, unsigned char *out, int *ec) {
    const int lane = threadIdx.x & 31, p2 = p * p;
    const int64_t i = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
    if (i >= (int64_t)ndom * nb * W) return;
    const int c = (int)(i % W);
    const int64_t b = b0 + (i / W) % nb;
    const int d = (int)(i / W / nb);
    int l = 2;
    while (l < L.lmax && L.off[l + 1] <= b) ++l;
    const int *s = bal + (d * (L.lmax - 1) + l - 2) * p;
    const cx<R> *x = C + (((int64_t)d * nbox + b) * ncols + col0 + c) * p2;
    constexpr int Q = 4;  // p^2 <= 100 coefficients over 32 lanes
    cx<R> v[Q];
    int sc[Q], e = -OZ_NONFINITE;
#pragma unroll
    for (int k = 0; k < Q; ++k) {
        const int q = lane + 32 * k;
        v[k] = q < p2 ? x[q] : cx<R>{R(0), R(0)};
        sc[k] = q < p2 ? oz_scale_of(s, oz_degree(q), local) : 0;
        const int y = oz_exp2(v[k].re, v[k].im);
        e = max(e, abs(y) == OZ_NONFINITE ? y : y - sc[k]);
    }
    for (int o = 16; o > 0; o >>= 1) e = max(e, __shfl_xor_sync(0xffffffffu, e, o));
    const bool bad = e > OZ_NONFINITE / 2;
    if (e < -OZ_NONFINITE / 2 || bad) e = 0;
    const int64_t row = ((int64_t)d * nbox + b) * W + c;
    if (lane == 0) ec[row] = bad ? OZ_NONFINITE : e;
    constexpr int S = Oz<R>::S;
    unsigned char *o = out + row * (int64_t)kblocks * oz_row<R>;
#pragma unroll
    for (int k = 0; k < Q; ++k) {
        const int q = lane + 32 * k;
        if (q >= kblocks * 8) break;
        uint16_t a[S], b2[S];
        oz_digits(bad ? R(0) : v[k].re, -sc[k] - e, a);
        oz_digits(bad ? R(0) : v[k].im, -sc[k] - e, b2);
        unsigned char *w = o + (q >> 3) * oz_row<R> + (q & 7) * 4;
#pragma unroll
        for (int j = 0; j < S; ++j) *reinterpret_cast<uint32_t *>(w + j * 32) = a[j] | (uint32_t)b2[j] << 16;
    }
}

struct OzP {
    int64_t nbox, y_dom;
    int64_t mat_dom, mat0;  // matrices of a domain, and of its first group
    int W, p2, kblocks;     // columns per pair of this window, K blocks of 16
    int ndom, mt, ngroup;
};
template <typename R>
__host__ __device__ __forceinline__ int oz_tiles(int64_t pairs, int W) {
    return (int)((pairs * W + Oz<R>::N - 1) / Oz<R>::N);
}

// unit v of a launch (row tile fastest, so that concurrent CTAs share source digits, then the tiles of
// a group, which share a matrix): domain, row tile, group (level, offset) and its columns
struct OzTile {
    int d, mt, g, n;     // n columns of the tile
    int64_t pair0;       // first pair (pair_e position) of the group
    int col0;            // first column within the group
};
template <typename R>
__device__ __forceinline__ OzTile oz_tile(const OzP &P, int v, int ntile, const int *first, const int32_t *group) {
    OzTile t;
    t.mt = v % P.mt;
    v /= P.mt;
    t.d = v / ntile;
    v -= t.d * ntile;
    int lo = 0, hi = P.ngroup;  // the group with first[g] <= v < first[g + 1]
    while (hi - lo > 1) {
        const int m = (lo + hi) >> 1;
        if (first[m] <= v) lo = m;
        else hi = m;
    }
    t.g = lo;
    t.pair0 = group[lo];
    t.col0 = (v - first[lo]) * Oz<R>::N;
    t.n = (int)min((int64_t)Oz<R>::N, (int64_t)(group[lo + 1] - t.pair0) * P.W - t.col0);
    return t;
}

// 2^k (s + w + r) as a double by FP32 and integer operations: an FP64 addition keeps a quarter of the SM
// busy for 64 cycles here, and with two of them per result the sums took longer than the MMAs.  The three
// floats become a head h, a tail g of at most half its ulp and a rest e2, and g and e2 are added to the
// bits of h's double in quarters of its last place (within 0.8 of which the result is).  FP64 where the
// sum nearly cancels, and where k is out of the doubles' range (OZ_NONFINITE and beyond: an Inf or a NaN).
__device__ __noinline__ double oz_compose_far(float s, float w, float r, int k) {
    if (k > OZ_NONFINITE / 2) return __longlong_as_double(0x7ff8000000000000ll);
    return ldexp(((double)s + (double)w) + (double)r, k);
}
__device__ __forceinline__ float oz_two_sum(float a, float b, float &err) {
    const float s = a + b, t = s - a;
    err = (a - (s - t)) + (b - t);
    return s;
}
__device__ __forceinline__ double oz_compose(float s, float w, float r, int k) {
    float e1, e2, g;
    const float h1 = oz_two_sum(s, w, e1), t = oz_two_sum(e1, r, e2), h = oz_two_sum(h1, t, g);
    if (!(fabsf(e2) <= fabsf(h) * 5.8207661e-11f) || abs(k) > 800) return oz_compose_far(s, w, r, k);  // 2^-34
    const int b = __float_as_int(h), eh = (b >> 23) & 0xff, bg = __float_as_int(g), eg = (bg >> 23) & 0xff;
    // |g| in quarters of 2^(exponent of h - 52): 24 bits times 2^7, shifted right by eh - eg - 24 >= 0
    int q = (int)(((uint32_t)(bg & 0x7fffff) | 0x800000u) << 7 >> min(max(eh - eg - 24, 0), 31));
    if (eg == 0) q = 0;
    const float quarter = __int_as_float(min(127 + 54 + 127 - eh, 254) << 23);
    int x = __float_as_int(__fmaf_rn(e2, quarter, 12582912.f)) - 0x4b400000;  // |e2| is below 2^21 quarters
    if (b < 0) x = -x;
    x += (b ^ bg) < 0 ? -q : q;
    // below a power of two the last place is half as large
    const int add = (b & 0x7fffff) == 0 && x < 0 ? (x + 1) >> 1 : (x + 2) >> 2;
    const long long mag = ((long long)(((b & 0x7fffffff) >> 3) + ((896 + k) << 20)) << 32 | (uint32_t)(b << 29)) + add;
    return eh == 0 ? 0.0 : __longlong_as_double(mag | (long long)(b & 0x80000000) << 32);
}

// x 2^k as a float (NaN where k holds the mark OZ_NONFINITE)
__device__ __forceinline__ float oz_scale(float x, int k) {
    if (k > OZ_NONFINITE / 2) return __int_as_float(0x7fc00000);
    const int h = min(max(k >> 1, -126), 126), g = min(max(k - h, -126), 126);
    return x * __int_as_float((127 + h) << 23) * __int_as_float((127 + g) << 23);
}

// Persistent, one CTA per SM (20 warps, five to a scheduler).  Warps 0-2 fill the ring, each every third K
// block of the CTA's sequence of tiles (the digit image by bulk copy, the gathered source digits by 16-byte
// cp.async), the pairs of their next tile already on the way; warp 3 issues the MMAs; warps 4-19 empty the
// accumulators (three floats per result in registers), free tensor memory for the next tile, and then
// compose the doubles and store them beside that tile's MMAs (eight epilogue warps with twice the columns,
// and twice the unrolled code, took longer over it than the MMAs).
template <typename R>
__global__ void __launch_bounds__(OZ_THREADS, 1)
    k_m2l_oz(const OzP P, const int32_t *__restrict__ group, const int2 *__restrict__ pairs,
             const unsigned char *__restrict__ Cdig, const int *__restrict__ ec, const unsigned char *__restrict__ img,
             const int *__restrict__ er, R *Y, int *err, int *err_host) {
    constexpr int S = Oz<R>::S, N = Oz<R>::N, ACC = Oz<R>::ACC;
    constexpr uint32_t A_BYTES = oz_a_bytes<R>;
    extern __shared__ unsigned char smem_raw[];
    __shared__ uint64_t full[OZ_SLOTS], empty[OZ_SLOTS], done, tfree, fin;
    __shared__ uint32_t tmem_slot;
    __shared__ volatile int s_abort;
    __shared__ int rowid[OZ_FILL][N];  // per producer warp: digit row of each pair column (-1: none)
    __shared__ int s_part[OZ_THREADS / 32];
    __shared__ int first[(OZ_MAX_LEVELS - 2) * 316 + 1];  // tiles before each group
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t sbase = (smem_u32(smem_raw) + 1023u) & ~1023u;
    auto give_up = [&] {
        atomicExch(err, 1);
        *(volatile int *)err_host = 1;
        s_abort = 1;
    };
    if (threadIdx.x == 0) {
        for (int s = 0; s < OZ_SLOTS; ++s) {
            mbar_init(&full[s], 33);  // the filling warp's 32 lanes + the bulk copy's expect_tx
            mbar_init(&empty[s], 1);
        }
        mbar_init(&done, 1);
        mbar_init(&tfree, 32 * OZ_EPI);
        mbar_init(&fin, 1);
        s_abort = *(volatile int *)err;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0)
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)), "r"(512)
                     : "memory");
    {  // prefix sum of the groups' tiles
        const int per = (P.ngroup + OZ_THREADS - 1) / OZ_THREADS, g0 = min(threadIdx.x * per, P.ngroup);
        const int g1 = min(g0 + per, P.ngroup);
        int sum = 0;
        for (int g = g0; g < g1; ++g) sum += oz_tiles<R>(group[g + 1] - group[g], P.W);
        int inc = sum;
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += y;
        }
        if (lane == 31) s_part[warp] = inc;
        __syncthreads();
        int at = inc - sum;
        for (int w = 0; w < warp; ++w) at += s_part[w];
        for (int g = g0; g < g1; ++g) {
            first[g] = at;
            at += oz_tiles<R>(group[g + 1] - group[g], P.W);
        }
        if (g0 < g1 && g1 == P.ngroup) first[P.ngroup] = at;
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = tmem_slot;
    const int ntile = first[P.ngroup], nunit = ntile * P.ndom * P.mt;
    int last = -1;  // a producer warp's last K block

    if (warp < OZ_FILL) {
        // ------------------------------------------------------------------ producers
        // source boxes of a tile's columns lane, lane + 32, ..
        constexpr int NSRC = (N + 31) / 32;
        auto sources = [&](const OzTile &t, int *src) {
#pragma unroll
            for (int k = 0; k < NSRC; ++k) {
                const int m = lane + 32 * k;
                src[k] = m < t.n ? pairs[t.pair0 + (t.col0 + m) / P.W].x : -1;
            }
        };
        int src[NSRC];
        OzTile t;
        if ((int)blockIdx.x < nunit) {
            t = oz_tile<R>(P, blockIdx.x, ntile, first, group);
            sources(t, src);
        }
        int u = 0, turn = 0;  // K blocks of the CTA's sequence, u mod OZ_FILL
        bool stop = false;
        for (int v = blockIdx.x; v < nunit && !stop; v += gridDim.x) {
            __syncwarp();
#pragma unroll
            for (int k = 0; k < NSRC; ++k) {
                const int m = lane + 32 * k, c = (t.col0 + m) % P.W;
                if (m < N)
                    rowid[warp][m] = src[k] >= 0 ? (int)(((int64_t)t.d * P.nbox + src[k]) * P.W + c) : -1;
            }
            __syncwarp();
            const OzTile cur = t;
            if (v + (int)gridDim.x < nunit) {
                t = oz_tile<R>(P, v + gridDim.x, ntile, first, group);
                sources(t, src);
            }
            const int n_pad = (cur.n + 15) & ~15;
            const int64_t mat = cur.d * P.mat_dom + P.mat0 + cur.g;
            const unsigned char *A = img + (mat * P.mt + cur.mt) * P.kblocks * (int64_t)OZ_A_BYTES;
            for (int kb = 0; kb < P.kblocks; ++kb, ++u, turn = turn == OZ_FILL - 1 ? 0 : turn + 1) {
                if (turn != warp) continue;
                const int slot = u & 3;
                const uint32_t sA = sbase + (uint32_t)slot * oz_slot_bytes<R>, sB = sA + A_BYTES;
                bool ok = u < OZ_SLOTS || mbar_wait(&empty[slot], (uint32_t)((u >> 2) - 1) & 1u);
                ok = __all_sync(0xffffffffu, ok && !s_abort);
                if (!ok) {
                    if (lane == 0) give_up();
                    stop = true;
                    break;
                }
                if (lane == 0) {
                    mbar_arrive_expect_tx(&full[slot], A_BYTES);
                    bulk_load(sA, A + (int64_t)kb * OZ_A_BYTES, A_BYTES, &full[slot]);
                }
                // a column's 32 S bytes of digits: 2 S lanes each, S columns a lane in one go
                constexpr int CPW = 16 / S;  // columns of the warp at once
                const int part = lane & (2 * S - 1), dg = part >> 1, ch = part & 1;
                const unsigned char *src0 = Cdig + (int64_t)kb * oz_row<R> + part * 16;
                const uint32_t dst0 = sB + (uint32_t)dg * (N * 32u), stride = (uint32_t)P.kblocks * oz_row<R>;
                for (int m0 = lane / (2 * S); m0 < n_pad; m0 += 16) {
                    int row[S];
#pragma unroll
                    for (int k = 0; k < S; ++k) row[k] = rowid[warp][m0 + CPW * k];
#pragma unroll
                    for (int k = 0; k < S; ++k)
                        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst0 + sw32_chunk(m0 + CPW * k, ch)),
                                     "l"(src0 + (uint64_t)(uint32_t)max(row[k], 0) * stride), "r"(row[k] >= 0 ? 16 : 0)
                                     : "memory");
                }
                asm volatile("cp.async.wait_all;" ::: "memory");
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&full[slot])) : "memory");
                last = u;
            }
        }
    } else if (warp == OZ_FILL) {
        // ------------------------------------------------------------------ MMA issuer
        // the whole warp runs the loop, so that descriptors stay in uniform registers (issued by one
        // divergent lane, an MMA cost 95 cycles, twice its operands' shared-memory reads); one elected
        // lane issues
        uint32_t leader;
        asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}\n" : "=r"(leader));
        bool ok = true;
        int u = 0, nt = 0;
        for (int v = blockIdx.x; v < nunit && ok; v += gridDim.x) {
            // (one answer for the whole warp: the flag may be raised between two lanes' reads of it)
            if (__any_sync(0xffffffffu, s_abort)) break;
            const OzTile t = oz_tile<R>(P, v, ntile, first, group);
            const uint32_t idesc = idesc_bf16((t.n + 15) & ~15);
            if (nt > 0) ok = __all_sync(0xffffffffu, mbar_wait(&tfree, (uint32_t)(nt - 1) & 1u));
            if (!ok) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            for (int kb = 0; kb < P.kblocks; ++kb, ++u) {
                const int s = u & 3;
                ok = __all_sync(0xffffffffu, mbar_wait(&full[s], (uint32_t)(u >> 2) & 1u));
                if (!ok) break;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint32_t sA = sbase + (uint32_t)s * oz_slot_bytes<R>;
                const uint64_t da = smem_desc_sw32(sA), db = smem_desc_sw32(sA + A_BYTES);
                // a digit of the matrix against every digit it meets, held in the collector after the
                // first; the smallest products first, so that the shared accumulator loses least
#pragma unroll
                for (int i = 0; i < S; ++i)
#pragma unroll
                    for (int j = S - 1 - i; j >= 0; --j) {
                        const int dd = i + j;
                        const uint32_t acc = tmem + (uint32_t)((dd < ACC ? dd : ACC - 1) * N);
                        const bool head = i == 0 && (dd < ACC - 1 || dd == S - 1);
                        const uint64_t a = da + (uint64_t)((i * (TC_M * 32)) >> 4), b = db + (uint64_t)((j * (N * 32)) >> 4);
                        const uint32_t add = head && kb == 0 ? 0u : 1u;
                        if (i == S - 1) mma_bf16_if<0>(leader, acc, a, b, idesc, add);
                        else if (j == S - 1 - i) mma_bf16_if<1>(leader, acc, a, b, idesc, add);
                        else if (j > 0) mma_bf16_if<2>(leader, acc, a, b, idesc, add);
                        else mma_bf16_if<3>(leader, acc, a, b, idesc, add);
                    }
                if (leader) mma_commit(&empty[s]);
                __syncwarp();
            }
            if (ok && leader) mma_commit(&done);
            __syncwarp();
            ++nt;
        }
        if (leader) {  // arrives once every MMA issued above has completed
            if (nt > 0) mma_commit(&fin);
            else asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&fin)) : "memory");
            if (!ok) give_up();
        }
        __syncwarp();
    } else {
        // ------------------------------------------------------------------ epilogue warps 4..19
        // warp: accumulator lanes 32 (warp mod 4) .., columns 16 b + 4 sub + j (b < NG, j < 4)
        const int quarter = warp & 3, sub = (warp - 4) >> 2;
        constexpr int NG = N / 16;
        static_assert(4 * NG <= 32, "a lane per column of the warp");
        int nt = 0;
        for (int v = blockIdx.x; v < nunit; v += gridDim.x) {
            const OzTile t = oz_tile<R>(P, v, ntile, first, group);
            const int64_t mat = t.d * P.mat_dom + P.mat0 + t.g;
            const int rr = t.mt * TC_M + quarter * 32 + lane;
            const bool rows = t.mt * TC_M + quarter * 32 < 2 * P.p2, row_ok = rr < 2 * P.p2;
            const int eR = row_ok ? er[mat * P.p2 + (rr >> 1)] : 0;
            // lane i knows column i of this warp's 4 NG: its row of Y and its exponent
            const int m = 16 * (lane >> 2) + 4 * sub + (lane & 3);
            int yr = -1, ex = 0;
            if (m < t.n && lane < 4 * NG) {
                const int2 pr = pairs[t.pair0 + (t.col0 + m) / P.W];
                const int c = (t.col0 + m) % P.W;
                yr = pr.y * P.W + c;
                ex = ec[((int64_t)t.d * P.nbox + pr.x) * P.W + c];
            }
            bool ok = !s_abort && mbar_wait(&done, (uint32_t)nt & 1u);
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) {
                if (lane == 0) give_up();
                break;
            }
            ++nt;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const int ng = rows ? (t.n - 4 * sub + 15) / 16 : 0;  // this warp's column groups in use
            constexpr bool DBL = sizeof(R) == 8;
            float hi[4 * NG], mi[DBL ? 4 * NG : 1], lo[DBL ? 4 * NG : 1];
#pragma unroll
            for (int b = 0; b < NG; ++b) {
                if (b < ng) {
                    uint32_t a[ACC][4];
#pragma unroll
                    for (int k = 0; k < ACC; ++k) {
                        const uint32_t ta = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(k * N + 16 * b + 4 * sub);
                        asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
                                     : "=r"(a[k][0]), "=r"(a[k][1]), "=r"(a[k][2]), "=r"(a[k][3])
                                     : "r"(ta));
                    }
                    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        if constexpr (!DBL) {  // the smallest first
                            hi[4 * b + j] = __uint_as_float(a[0][j]) + (__uint_as_float(a[1][j]) +
                                            (__uint_as_float(a[2][j]) + __uint_as_float(a[3][j])));
                        } else {
                            const float d0 = __uint_as_float(a[0][j]), d1 = __uint_as_float(a[1][j]);
                            const float d3 = __uint_as_float(a[3][j]);
                            const float s = d0 + d1, sb = s - d0;                         // s + e = d0 + d1
                            const float e = (d0 - (s - sb)) + (d1 - sb);
                            const float l = e + __uint_as_float(a[2][j]);                 // exact: within 24 bits
                            const float m = l + d3, mb = m - l;                           // m + .. = l + d3
                            const float x = ((l - (m - mb)) + (d3 - mb)) + __uint_as_float(a[4][j]);  // exact
                            const float w = m + x, wb = w - m;                            // w + .. = m + x
                            hi[4 * b + j] = s;
                            mi[4 * b + j] = w;
                            lo[4 * b + j] = ((m - (w - wb)) + (x - wb)) + __uint_as_float(a[5][j]);
                        }
                    }
                }
            }
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&tfree)) : "memory");
            R *Yd = Y + (int64_t)t.d * P.y_dom + rr;
#pragma unroll
            for (int b = 0; b < NG; ++b) {
                if (b < ng) {
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const int i = 4 * b + j;
                        const int o = __shfl_sync(0xffffffffu, yr, i);
                        const int k = __shfl_sync(0xffffffffu, ex, i) + eR;
                        R x;
                        if constexpr (DBL) x = oz_compose(hi[i], mi[i], lo[i], k);
                        else x = oz_scale(hi[i], k);
                        if (row_ok && o >= 0) Yd[(int64_t)o * (2 * P.p2)] = x;
                    }
                }
            }
        }
    }
    __syncwarp();
    __syncthreads();
    // After an abort (which any warp may have raised, also after the producers were through) no bulk copy may be in
    // flight when the CTA ends: wait (bounded) for each producer warp's last two.  Those before them have landed, as
    // the last one's slot was free only after the MMAs of the K block OZ_SLOTS earlier.
    if (warp < OZ_FILL && lane == 0 && s_abort)
        for (int u = max(last - OZ_FILL, last % OZ_FILL); u >= 0 && u <= last; u += OZ_FILL)
            if (!mbar_wait(&full[u & 3], (uint32_t)(u >> 2) & 1u)) give_up();
    if (threadIdx.x == 0 && !mbar_wait(&fin, 0)) give_up();
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0) {
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
}

__global__ void k_oz_pairs(int64_t n, const int32_t *pair_e, const int32_t *ff_src, int2 *out) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i < n) out[i] = make_int2(ff_src[pair_e[i]], pair_e[i]);
}

int oz_kblocks(int p2) { return (2 * p2 + 15) / 16; }
int oz_mt(int p2) { return (2 * p2 + TC_M - 1) / TC_M; }

}  // namespace

// even p in 4..10: K = 2 p^2 <= 200 keeps the digit sums exact (a diagonal of five products of at most 2^14 units
// per K, 2 p^2 5 2^14 < 2^24).  Odd p would be as exact (images and digits are padded with zeros to whole K
// blocks); they have not been measured and keep the rotation and dense forms
bool m2l_oz_supported(const fmbem *h) {
    return h->p >= 4 && h->p <= 10 && h->p % 2 == 0 && h->lmax >= 2 && h->lmax < OZ_MAX_LEVELS && !h->opt.fp32_only;
}

// digit images of every S|R matrix of levels 2..l_max; not built when they would take more than an
// eighth of the free device memory (the FP64 pipe's kernels then remain)
void build_oz_tables(fmbem *h, cudaStream_t s) {
    const int p2 = h->p2, kb = oz_kblocks(p2), mt = oz_mt(p2), sets = (h->Jf + 1) * (h->lmax - 1);
    const int64_t nmat = (int64_t)sets * 316, bytes = nmat * mt * kb * (int64_t)OZ_A_BYTES;
    size_t free_b = 0, total_b = 0;
    CK(cudaMemGetInfo(&free_b, &total_b));
    if (h->n_ff <= 0 || h->tc_err == nullptr || (size_t)bytes > free_b / 8) return;
    h->oz_group = (int32_t *)dev_alloc(h, sizeof(int32_t) * h->h_group_beg.size());
    CK(cudaMemcpyAsync(h->oz_group, h->h_group_beg.data(), sizeof(int32_t) * h->h_group_beg.size(), cudaMemcpyHostToDevice, s));
    h->oz_pairs = dev_alloc(h, sizeof(int2) * h->n_ff);
    k_oz_pairs<<<(unsigned)((h->n_ff + 255) / 256), 256, 0, s>>>(h->n_ff, h->pair_e, h->ff_src, (int2 *)h->oz_pairs);
    CKL("k_oz_pairs");
    h->oz_bal = (int *)dev_alloc(h, sizeof(int) * sets * h->p);
    h->oz_er = (int *)dev_alloc(h, sizeof(int) * nmat * p2);
    h->oz_img = dev_alloc(h, bytes);
    CK(cudaHostAlloc((void **)&h->oz_err_host, sizeof(int), cudaHostAllocMapped));
    *h->oz_err_host = 0;
    k_oz_balance<<<dim3((unsigned)sets, (unsigned)h->p), 256, 0, s>>>(h->T_m2l64, h->p, h->lmax, h->oz_bal);
    CKL("k_oz_balance");
    k_oz_images<<<(unsigned)nmat, 256, 0, s>>>(h->T_m2l64, h->p, h->lmax, 316, 2, h->lmax - 1, 2, false, mt, kb, h->oz_bal,
                                               (unsigned char *)h->oz_img, h->oz_er);
    CKL("k_oz_images");
    if (h->lmax < 3) return;
    // S|S and R|R between levels: the children of levels 3.. by octant (source and result rows per entry)
    if (h->rmm_entry == nullptr) build_rot_mm_lists(h, s);
    if (h->n_rmm == 0) return;
    std::vector<int32_t> cnt((size_t)8 * (h->lmax - 2), 0), entry(h->nbox);
    std::vector<uint64_t> key(h->nbox);
    std::vector<int32_t> par(h->nbox);
    CK(cudaMemcpyAsync(key.data(), h->box_key, sizeof(uint64_t) * h->nbox, cudaMemcpyDeviceToHost, s));
    CK(cudaMemcpyAsync(par.data(), h->box_parent, sizeof(int32_t) * h->nbox, cudaMemcpyDeviceToHost, s));
    CK(cudaMemcpyAsync(entry.data(), h->rmm_entry, sizeof(int32_t) * h->nbox, cudaMemcpyDeviceToHost, s));
    CK(cudaStreamSynchronize(s));
    std::vector<int2> up(h->n_rmm), down(h->n_rmm);
    for (int l = 3; l <= h->lmax; ++l)
        for (int64_t g = h->lev[l].off; g < h->lev[l].off + h->lev[l].n; ++g) {
            const int row = entry[g] - (int)h->h_rmm_first[l];
            up[entry[g]] = make_int2((int)g, row);
            down[entry[g]] = make_int2(par[g], row);
            ++cnt[(size_t)(l - 3) * 8 + (key[g] & 7)];
        }
    h->h_oz_ogroup.assign(1, 0);
    for (const int32_t c : cnt) h->h_oz_ogroup.push_back(h->h_oz_ogroup.back() + c);
    h->oz_ogroup = (int32_t *)dev_alloc(h, sizeof(int32_t) * h->h_oz_ogroup.size());
    h->oz_up = dev_alloc(h, sizeof(int2) * up.size());
    h->oz_down = dev_alloc(h, sizeof(int2) * down.size());
    CK(cudaMemcpyAsync(h->oz_ogroup, h->h_oz_ogroup.data(), sizeof(int32_t) * h->h_oz_ogroup.size(), cudaMemcpyHostToDevice, s));
    CK(cudaMemcpyAsync(h->oz_up, up.data(), sizeof(int2) * up.size(), cudaMemcpyHostToDevice, s));
    CK(cudaMemcpyAsync(h->oz_down, down.data(), sizeof(int2) * down.size(), cudaMemcpyHostToDevice, s));
    CK(cudaStreamSynchronize(s));
    const int64_t noct = (int64_t)(h->Jf + 1) * (h->lmax - 2) * 8;
    for (int k = 0; k < 2; ++k) {
        h->oz_oer[k] = (int *)dev_alloc(h, sizeof(int) * noct * p2);
        h->oz_oimg[k] = dev_alloc(h, noct * mt * kb * (int64_t)OZ_A_BYTES);
        k_oz_images<<<(unsigned)noct, 256, 0, s>>>(k == 0 ? h->T_mm64 : h->T_ll64, h->p, h->lmax, 8, 3, h->lmax - 2, k == 0 ? 3 : 2,
                                                   k == 1, mt, kb, h->oz_bal, (unsigned char *)h->oz_oimg[k], h->oz_oer[k]);
        CKL("k_oz_images");
    }
}

// real numbers of Y per domain for a window of W columns, and bytes of the window's digits and exponents
int64_t oz_y_dom(const fmbem *h, int W) { return h->n_ff * W * 2 * h->p2; }
template <typename R>
size_t oz_digit_bytes(const fmbem *h, int W) {
    const size_t rows = (size_t)(h->Jf + 1) * h->nbox * W;
    return rows * oz_kblocks(h->p2) * oz_row<R> + rows * sizeof(int);
}
template size_t oz_digit_bytes<double>(const fmbem *, int);
template size_t oz_digit_bytes<float>(const fmbem *, int);

// the digits of the boxes b0 .. b0 + nb - 1 of X, then the products of the groups' matrices and pairs
template <typename R>
static void oz_products(fmbem *h, const cx<R> *X, int64_t b0, int64_t nb, bool local, cx<R> *Y, int64_t y_dom, int64_t nr,
                        int col0, int W, int ngroup, const int32_t *h_group, const int32_t *group, const void *pairs,
                        const void *img, const int *er, int64_t mat_dom, int64_t mat0, cudaStream_t s) {
    const int p2 = h->p2, kb = oz_kblocks(p2), ndom = h->Jf + 1;
    OzP P{};
    P.nbox = h->nbox;
    P.y_dom = y_dom;
    P.mat_dom = mat_dom;
    P.mat0 = mat0;
    P.W = W;
    P.p2 = p2;
    P.kblocks = kb;
    P.ndom = ndom;
    P.mt = oz_mt(p2);
    P.ngroup = ngroup;
    int64_t tiles = 0;
    for (int g = 0; g < ngroup; ++g) tiles += oz_tiles<R>(h_group[g + 1] - h_group[g], W);
    if (tiles == 0) return;
    OzLevels L{};
    L.lmax = h->lmax;
    for (int l = 2; l <= h->lmax; ++l) L.off[l] = h->lev[l].off;
    L.off[h->lmax + 1] = h->nbox;
    const int64_t rows = (int64_t)ndom * nb * W;
    unsigned char *dig = (unsigned char *)h->oz_dig;
    int *ec = (int *)(dig + (size_t)ndom * h->nbox * W * kb * oz_row<R>);
    k_oz_split<R><<<(unsigned)((rows + 7) / 8), 256, 0, s>>>(X, L, b0, nb, local, h->nbox, 3 * nr, col0, W, ndom, h->p, kb,
                                                             h->oz_bal, dig, ec);
    CKL("k_oz_split");
    const size_t smem = OZ_SLOTS * (size_t)oz_slot_bytes<R> + 1024;
    CK(cudaFuncSetAttribute(k_m2l_oz<R>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    int dev = 0, nsm = 0;
    CK(cudaGetDevice(&dev));
    CK(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
    // an odd grid: a CTA then alternates between the row tiles, of which the second is the shorter
    const int64_t grid = std::min<int64_t>(tiles * ndom * P.mt, (nsm - 1) | 1);
    k_m2l_oz<R><<<(unsigned)grid, OZ_THREADS, smem, s>>>(P, group, (const int2 *)pairs, dig, ec, (const unsigned char *)img, er,
                                                         (R *)Y, h->tc_err, h->oz_err_host);
    CKL("k_m2l_oz");
}

// the S|R products of every level and domain for columns col0 .. col0 + W - 1 of C (3 n_rhs columns)
// into Y[d][CSR position][W][p^2] (domains oz_y_dom apart)
template <typename R>
void run_m2l_oz(fmbem *h, const cx<R> *C, cx<R> *Y, int64_t nr, int col0, int W, cudaStream_t s) {
    if (h->n_ff <= 0) return;
    const int64_t b0 = h->lev[2].off;
    oz_products<R>(h, C, b0, h->nbox - b0, false, Y, oz_y_dom(h, W), nr, col0, W, (h->lmax - 1) * 316, h->h_group_beg.data(),
                   h->oz_group, h->oz_pairs, h->oz_img, h->oz_er, (int64_t)(h->lmax - 1) * 316, 0, s);
}
// the S|S products of the children of level l (up: X their multipole expansions) or the R|R products of their
// parents' local expansions X, into Y[d][entry of the level][W][p^2] (domains n W p^2 complex values apart)
void run_oct_oz(fmbem *h, bool up, int l, const c64 *X, c64 *Y, int64_t nr, int col0, int W, cudaStream_t s) {
    const LevelInfo &S = h->lev[up ? l : l - 1];
    oz_products<double>(h, X, S.off, S.n, !up, Y, h->lev[l].n * W * 2 * h->p2, nr, col0, W, 8, h->h_oz_ogroup.data() + (l - 3) * 8,
                        h->oz_ogroup + (l - 3) * 8, up ? h->oz_up : h->oz_down, h->oz_oimg[up ? 0 : 1], h->oz_oer[up ? 0 : 1],
                        (int64_t)(h->lmax - 2) * 8, (int64_t)(l - 3) * 8, s);
}
template void run_m2l_oz<double>(fmbem *, const c64 *, c64 *, int64_t, int, int, cudaStream_t);
template void run_m2l_oz<float>(fmbem *, const c32 *, c32 *, int64_t, int, int, cudaStream_t);

// a wait of this M2L that ran out on an earlier product of this handle
void check_oz_err(fmbem *h, cudaStream_t s) {
    if (h->oz_err_host == nullptr || *(volatile int *)h->oz_err_host == 0) return;
    *(volatile int *)h->oz_err_host = 0;
    CK(cudaMemsetAsync(h->tc_err, 0, sizeof(int), s));
    throw fmbem_error{FMBEM_ERR_DEVICE_TIMEOUT, "tensor-core M2L (8-bit digits): an mbarrier wait timed out"};
}
