// k_layout.cu -- gauge ingest, two-link build, vector pack/unpack, norms.
//
//   ingest      canonical FP64 U[t][z][y][x][mu][3][3] -> sublattice planes
//               (bit-exact permutation; U_t is never read)
//   build       W_i(x) = U_i(x) U_i(x+i) in FP64 (Sec. 2), rounded to nearest
//               into the chosen W storage (Sec. 3: computed once, reused)
//   pack        caller vectors (FP64/FP32, canonical) -> packed storage
//   unpack      packed storage -> caller layout, with FP64 |psi|^2 partial sums
//   norms       fixed-order reduction of the partial sums (deterministic)
//
// Packed U layout: block b = t * 8 + sub, direction d, entry k = 0..8:
//   Up[((b * 3 + d) * 9 + k) * Ps + i]  (double2 = one complex entry)
#include <cooperative_groups.h>

#include <algorithm>
#include <type_traits>

#include "layout_plan.h"
#include "tls_dev.cuh"
#include "tls_internal.h"

namespace tls {

namespace {

struct Coords {
    int x, y, z;
};

// Site i of sublattice `sub` -> spatial coordinates.
__device__ __forceinline__ Coords coords_of(const SubGeom &g, int sub, int i)
{
    int xq = i % g.hx;
    int r = i / g.hx;
    int yq = r % g.hy;
    int zq = r / g.hy;
    Coords c;
    c.x = 2 * xq + (sub & 1);
    c.y = 2 * yq + ((sub >> 1) & 1);
    c.z = 2 * zq + ((sub >> 2) & 1);
    return c;
}

// CTA = a run of up to kIngestSites sites of one canonical x-row.  The links come in entry by entry
// (27 consecutive complex numbers a site, coalesced; host memory over C2C included), go through
// shared memory and leave plane by plane, the even sites of the run and then the odd ones, so that
// a plane is written in runs of 16-byte words instead of one word per site and plane.  HBM-bound:
// tls_load_gauge at 48^3 x 64 (device links, 0.15 ms of it cudaMalloc) 2.1 ms before, 1.6
// now.
constexpr int kIngestSites = 64;
__global__ void __launch_bounds__(256) k_ingest_gauge(const double *__restrict__ U, int nd, double2 *__restrict__ Up,
                                                      SubGeom g, int Lx, int Ly, int Lz, int runs)
{
    __shared__ double2 sm[27][kIngestSites + 1];
    const int64_t row = blockIdx.x / runs;  // (t, z, y)
    const int x0 = (int)(blockIdx.x - row * runs) * kIngestSites;
    const int n = min(kIngestSites, Lx - x0), h = n / 2;  // x0 and n are even
    const int y = (int)(row % Ly);
    const int64_t r2 = row / Ly;
    const int z = (int)(r2 % Lz), t = (int)(r2 / Lz);
    const double2 *src = reinterpret_cast<const double2 *>(U) + (row * Lx + x0) * nd * 9;
    for (int k = threadIdx.x; k < n * 27; k += blockDim.x) {
        const int x = k / 27, e = k - x * 27;
        sm[e][(x & 1) * h + (x >> 1)] = src[(int64_t)x * nd * 9 + e];
    }
    __syncthreads();
    const int sub = ((y & 1) << 1) | ((z & 1) << 2);
    const int i0 = ((z >> 1) * g.hy + (y >> 1)) * g.hx + x0 / 2;
    for (int k = threadIdx.x; k < n * 27; k += blockDim.x) {
        const int e = k / n, pos = k - e * n;
        const int par = pos >= h;
        Up[((int64_t)(t * 8 + (sub | par)) * 27 + e) * g.Ps + i0 + pos - par * h] = sm[e][pos];
    }
}

// Short rows: CTA = an even number of rows, kIngestSites sites or a little less, consecutive in the
// caller's array.  They leave sublattice by sublattice, rows of the same y parity one behind
// the other in its planes.  A CTA of its own for a row of two sites moves 54 words
// (2 x 48 x 48 x 48: 329 us for a load and release, 277 with a thread per word before that,
// 254 now).
__global__ void __launch_bounds__(256) k_ingest_rows(const double *__restrict__ U, int nd, double2 *__restrict__ Up,
                                                     SubGeom g, int Lx, int Ly, int Lz, int rows, int64_t nrow)
{
    __shared__ double2 sm[27][kIngestSites + 1];
    const int64_t row0 = (int64_t)blockIdx.x * rows;  // (t, z, y); even
    const int n = (int)min((int64_t)rows, nrow - row0) * Lx;
    const double2 *src = reinterpret_cast<const double2 *>(U) + row0 * Lx * nd * 9;
    for (int k = threadIdx.x; k < n * 27; k += blockDim.x) {
        const int s = k / 27, e = k - s * 27;
        sm[e][s] = src[(int64_t)s * nd * 9 + e];
    }
    __syncthreads();
    const int q = n / 4;  // sites of a sublattice
    for (int k = threadIdx.x; k < n * 27; k += blockDim.x) {
        const int e = k / n, pos = k - e * n, c = pos / q, r = pos - c * q;  // c: parities of x and y
        const int rl = 2 * (r / g.hx) + (c >> 1), xq = r % g.hx;
        const int64_t row = row0 + rl;
        const int y = (int)(row % Ly);
        const int64_t r2 = row / Ly;
        const int z = (int)(r2 % Lz), t = (int)(r2 / Lz);
        Up[((int64_t)(t * 8 + (c | (z & 1) << 2)) * 27 + e) * g.Ps + ((z >> 1) * g.hy + (y >> 1)) * g.hx + xq] =
            sm[e][rl * Lx + 2 * xq + (c & 1)];
    }
}

__global__ void k_export_gauge(const double2 *__restrict__ Up, double *__restrict__ out, SubGeom g, int Lx, int Ly,
                               int Lz, int64_t total)
{
    int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= total) return;
    const int i = (int)(idx % g.Vs);
    const int64_t r = idx / g.Vs;
    const int d = (int)(r % 3);
    const int b = (int)(r / 3);
    const int t = b >> 3, sub = b & 7;
    Coords c = coords_of(g, sub, i);
    const int64_t site = (((int64_t)t * Lz + c.z) * Ly + c.y) * Lx + c.x;
    double2 *dst = reinterpret_cast<double2 *>(out) + (site * 3 + d) * 9;
    const double2 *src = Up + ((int64_t)b * 3 + d) * 9 * g.Ps + i;
#pragma unroll
    for (int k = 0; k < 9; ++k) dst[k] = src[k * g.Ps];
}

// W_d(x) = U_d(x) U_d(x + d).  In sublattice terms x + d flips bit d of the
// sublattice index, and the half coordinate advances (with wrap) only when
// the coordinate was odd.
template <int WF, bool ONE = false>
__global__ void k_build_twolink(const double2 *__restrict__ Up, char *__restrict__ W, SubGeom g, int64_t total,
                                int *err)
{
    int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= total) return;
    const int i = (int)(idx % g.Vs);
    const int64_t r = idx / g.Vs;
    const int d = (int)(r % 3);
    const int b = (int)(r / 3);
    const int sub = b & 7;
    int fw[3], bw[3];
    sub_neighbours(g, i, fw, bw);
    const int odd = (sub >> d) & 1;
    const int ip = odd ? fw[d] : i;
    const int bp = (b & ~7) | (sub ^ (1 << d));
    const double2 *A = Up + ((int64_t)b * 3 + d) * 9 * g.Ps + i;
    const double2 *B = Up + ((int64_t)bp * 3 + d) * 9 * g.Ps + ip;
    double2 a[9], bb[9];
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        a[k] = A[k * g.Ps];
        bb[k] = B[k * g.Ps];
    }
    double w[18];
    if constexpr (ONE) {  // one-link field: U_d(x) itself
#pragma unroll
        for (int k = 0; k < 9; ++k) {
            w[2 * k] = a[k].x;
            w[2 * k + 1] = a[k].y;
        }
    } else {
#pragma unroll
    for (int rr = 0; rr < 3; ++rr)
#pragma unroll
        for (int cc = 0; cc < 3; ++cc) {
            double re = 0.0, im = 0.0;
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const double2 x = a[rr * 3 + k], y = bb[k * 3 + cc];
                re = fma(x.x, y.x, re);
                re = fma(-x.y, y.y, re);
                im = fma(x.x, y.y, im);
                im = fma(x.y, y.x, im);
            }
            w[2 * (rr * 3 + cc)] = re;
            w[2 * (rr * 3 + cc) + 1] = im;
        }
    }
    char *blk = W + ((int64_t)b * 3 + d) * g.Ps * wfmt_bytes(WF);
    if constexpr (WF == W_F32_8) {
        if (!WFmt<WF>::store(blk, g.Ps, i, w)) atomicOr(err, DERR_RECON8);
    } else {
        WFmt<WF>::store(blk, g.Ps, i, w);
    }
}

// --------------------------------------------------------------------------
// The product rounded to FP32 without the FP64 pipe.
//
// k_build_twolink is bound by the FP64 pipe, which runs at 1/75 of the FP32 FMA
// rate here (64^3 x 96: 16.3 ms against 2.4 ms for its bytes).  This form gives
// the same bits from FP32 arithmetic wherever that decides the rounding, and
// takes the FP64 chain of k_build_twolink for the elements where it does not.
//
// Split: each double |v| <= 1.125 becomes v0 + v1 + v2 with v0 a multiple of
// 2^-10, v1 of 2^-21 (|v1| <= 2^-11) and |v2| <= 1.5 * 2^-22, off by less than
// 2^-45 (taken from the bits of the double: no FP64 instruction).
// Products, six per real part, by the sum of the slice indices:
//   S0 = sum a0 b0                       multiples of 2^-20 below 8: exact in FP32
//   S1 = sum a0 b1 + a1 b0               multiples of 2^-31 below 2^-7: exact
//   S2 = sum a0 b2 + a1 b1 + a2 b0 + a1 b2 + a2 b1   below 2^-17, 30 roundings of
//                                        at most 2^-42 each
// S0 + S1 is renormalised exactly to h + l (two-sum) and l += S2.  The error of
// h + l (roundings of S2 and l, the split, a2 b2) and of the FP64 chain itself add
// up to less than T = 2^-36, so when RN(h + (l - T)) == RN(h + (l + T)) every value
// in between, the FP64 chain's among them, rounds to that float.  The rest (about
// 0.3 % of the elements of random SU(3) links; all of a matrix with an entry above
// 1.125, an infinity or a NaN) is recomputed.
// A matrix costs about 660 packed FP32 and 550 integer instructions of a warp;
// slices of A stay in registers, those of B are made column by column.
// tls_build_twolink at 48^3 x 64 with the links released: 6.3 ms before, 3.5 ms now, of
// which 1.1 ms is cudaFree of the links (about 0.7 ms are the bytes at the copy rate).
// --------------------------------------------------------------------------
struct Slices {
    float2 s[3];  // (re, im) of the three slices
};

// The leading 24 bits of v (truncated) and the next 23: v = f + g up to 2^-46 |v|.
__device__ __forceinline__ void split_bits(double v, float &f, float &g, unsigned &top)
{
    const unsigned hi = (unsigned)__double2hiint(v), lo = (unsigned)__double2loint(v);
    const unsigned mag = hi & 0x7fffffffu, sign = hi & 0x80000000u;
    top = max(top, mag);
    const unsigned fb = ((mag - (896u << 20)) << 3) | (lo >> 29);
    const unsigned base = ((fb & 0x7f800000u) - (23u << 23)) | sign;
    const bool tiny = mag < ((1023u - 60u) << 20);  // below 2^-60: taken as zero
    f = tiny ? 0.0f : __uint_as_float(fb | sign);
    g = tiny ? 0.0f : __uint_as_float(base | ((lo >> 6) & 0x7fffffu)) - __uint_as_float(base);
}

__device__ __forceinline__ Slices split3(double2 v, unsigned &top)
{
    float2 f, g;
    split_bits(v.x, f.x, g.x, top);
    split_bits(v.y, f.y, g.y, top);
    Slices o;
    const float2 m0 = make_float2(12288.0f, 12288.0f), n0 = make_float2(-12288.0f, -12288.0f);  // 1.5 * 2^13: units of 2^-10
    const float2 m1 = make_float2(6.0f, 6.0f), n1 = make_float2(-6.0f, -6.0f);                  // 1.5 * 2^2: units of 2^-21
    const float2 neg = make_float2(-1.0f, -1.0f);
    o.s[0] = __fadd2_rn(__fadd2_rn(f, m0), n0);
    const float2 r = __ffma2_rn(o.s[0], neg, f);  // exact
    o.s[1] = __fadd2_rn(__fadd2_rn(r, m1), n1);
    o.s[2] = __fadd2_rn(__ffma2_rn(o.s[1], neg, r), g);
    return o;
}

__device__ __forceinline__ bool is_zero(double2 v)
{
    return (((unsigned)__double2hiint(v.x) | (unsigned)__double2hiint(v.y)) << 1 | (unsigned)__double2loint(v.x) |
            (unsigned)__double2loint(v.y)) == 0;
}

// Element e (of the real and imaginary parts of the stored rows) of site i.
__device__ __forceinline__ void put_element(char *blk, int64_t Ps, int i, int e, float f)
{
    if (e < 16)
        reinterpret_cast<float *>(reinterpret_cast<float4 *>(blk) + (e >> 2) * Ps + i)[e & 3] = f;
    else
        reinterpret_cast<float *>(blk + 4 * Ps * 16)[2 * i + (e & 1)] = f;
}

// Writes the undecided elements all of whose products have a zero factor (diagonal links, the free
// field): +0, as in the FP64 chain.  Returns the others.  Such elements are undecided
// because T itself decides their rounding; through the chain the free field took 1.6 times as long
// as with FP64 alone (48^3 x 16: 1934 us against 1184; 837 so).  A call, so that its registers are
// not the kernel's.
template <int ROWS>
__device__ __noinline__ unsigned put_zeros(const double2 *A, const double2 *B, char *blk, int64_t Ps, int i, unsigned bad)
{
    unsigned za = 0, zb = 0, left = 0;  // zero entries
#pragma unroll 1
    for (int k = 0; k < 9; ++k) {
        if (k < ROWS * 3) za |= is_zero(A[k * Ps]) ? 1u << k : 0u;
        zb |= is_zero(B[k * Ps]) ? 1u << k : 0u;
    }
#pragma unroll 1
    for (; bad; bad &= bad - 1) {
        const int e = __ffs(bad) - 1, r = e / 6, c = (e - 6 * r) >> 1;
        const unsigned zr = za >> (3 * r), zc = (zb >> c & 1u) | (zb >> (c + 2) & 2u) | (zb >> (c + 4) & 4u);
        if (((zr | zc) & 7u) == 7u)
            put_element(blk, Ps, i, e, 0.0f);
        else
            left |= 1u << e;
    }
    return left;
}

// ROWS = 3 (W f32-18) or 2 (f32-12: rows 1-2 are stored).
template <int ROWS>
__global__ void __launch_bounds__(128, 4) k_build_split(const double2 *__restrict__ Up, char *__restrict__ W, SubGeom g,
                                                        int64_t total)
{
    constexpr int WB = ROWS == 3 ? wfmt_bytes(W_F32_18) : wfmt_bytes(W_F32_12);
    const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= total) return;
    const int i = (int)(idx % g.Vs);
    const int64_t rr = idx / g.Vs;
    const int d = (int)(rr % 3);
    const int b = (int)(rr / 3);
    const int sub = b & 7;
    int fw[3], bw[3];
    sub_neighbours(g, i, fw, bw);
    const int ip = ((sub >> d) & 1) ? fw[d] : i;
    const int bp = (b & ~7) | (sub ^ (1 << d));
    const double2 *A = Up + ((int64_t)b * 3 + d) * 9 * g.Ps + i;
    const double2 *B = Up + ((int64_t)bp * 3 + d) * 9 * g.Ps + ip;
    unsigned top = 0;
    Slices a[ROWS * 3];
#pragma unroll
    for (int k = 0; k < ROWS * 3; ++k) a[k] = split3(A[k * g.Ps], top);
    float w[ROWS * 6];
    unsigned bad = 0;
    const float T = 1.0f / 68719476736.0f;  // 2^-36
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        float2 s[ROWS][3];
#pragma unroll
        for (int r = 0; r < ROWS; ++r)
#pragma unroll
            for (int q = 0; q < 3; ++q) s[r][q] = make_float2(0.f, 0.f);
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const Slices y = split3(B[(k * 3 + c) * g.Ps], top);
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                const float2 p = y.s[j], t = make_float2(-p.y, p.x);  // i p
#pragma unroll
                for (int r = 0; r < ROWS; ++r)
#pragma unroll
                    for (int q = 0; q < 3; ++q) {
                        if (q + j > 3) continue;
                        const float2 x = a[r * 3 + k].s[q];
                        float2 &acc = s[r][q + j > 2 ? 2 : q + j];
                        acc = __ffma2_rn(make_float2(x.x, x.x), p, acc);
                        acc = __ffma2_rn(make_float2(x.y, x.y), t, acc);
                    }
            }
        }
#pragma unroll
        for (int r = 0; r < ROWS; ++r) {
            const float2 neg = make_float2(-1.f, -1.f);
            const float2 h = __fadd2_rn(s[r][0], s[r][1]);
            const float2 v = __ffma2_rn(s[r][0], neg, h);  // two-sum: l = (S0 - (h - v)) + (S1 - v)
            const float2 u = __ffma2_rn(v, neg, h);
            float2 l = __fadd2_rn(__ffma2_rn(u, neg, s[r][0]), __ffma2_rn(v, neg, s[r][1]));
            l = __fadd2_rn(l, s[r][2]);
            const float2 up = __fadd2_rn(h, __fadd2_rn(l, make_float2(T, T)));
            const float2 dn = __fadd2_rn(h, __fadd2_rn(l, make_float2(-T, -T)));
            const int e = 2 * (r * 3 + c);
            w[e] = up.x;
            w[e + 1] = up.y;
            bad |= (up.x == dn.x ? 0u : 1u << e) | (up.y == dn.y ? 0u : 2u << e);
        }
    }
    if (top > 0x3FF20000u) bad = (1u << (6 * ROWS)) - 1u;  // an entry above 1.125
    char *blk = W + ((int64_t)b * 3 + d) * g.Ps * WB;
    float4 *q4 = reinterpret_cast<float4 *>(blk);
#pragma unroll
    for (int k = 0; k < ROWS * 6 / 4; ++k)
        q4[k * g.Ps + i] = make_float4(w[4 * k], w[4 * k + 1], w[4 * k + 2], w[4 * k + 3]);
    if constexpr (ROWS == 3) reinterpret_cast<float2 *>(blk + 4 * g.Ps * 16)[i] = make_float2(w[16], w[17]);
    if (__popc(bad) >= 6 && top <= 0x3FF20000u) bad = put_zeros<ROWS>(A, B, blk, g.Ps, i, bad);
    while (bad) {  // undecided elements: the FP64 chain of k_build_twolink
        const int e = __ffs(bad) - 1;
        bad &= bad - 1;
        const int r = e / 6, c = (e - 6 * r) >> 1;
        double acc = 0.0;
        for (int k = 0; k < 3; ++k) {
            const double2 x = A[(r * 3 + k) * g.Ps], y = B[(k * 3 + c) * g.Ps];
            acc = (e & 1) ? fma(x.x, y.y, acc) : fma(x.x, y.x, acc);
            acc = (e & 1) ? fma(x.y, y.x, acc) : fma(-x.y, y.y, acc);
        }
        put_element(blk, g.Ps, i, e, __double2float_rn(acc));
    }
}

// The links rounded to FP32, a slice as one block of gc with its sites in canonical order.
__global__ void __launch_bounds__(128) k_links_slices(const double2 *__restrict__ Up, char *__restrict__ L1, SubGeom g,
                                                      SubGeom gc, int64_t total)
{
    const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= total) return;
    const int c = (int)(idx % gc.Vs);
    const int64_t r = idx / gc.Vs;
    const int d = (int)(r % 3), t = (int)(r / 3);
    const int x = c % gc.hx, y = c / gc.hx % gc.hy, z = c / gc.hx / gc.hy;
    const int sub = (x & 1) | ((y & 1) << 1) | ((z & 1) << 2);
    const int i = ((z >> 1) * g.hy + (y >> 1)) * g.hx + (x >> 1);
    const double2 *A = Up + ((int64_t)(t * 8 + sub) * 3 + d) * 9 * g.Ps + i;
    double w[18];
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        const double2 v = A[k * g.Ps];
        w[2 * k] = v.x;
        w[2 * k + 1] = v.y;
    }
    WFmt<W_F32_18>::store(L1 + ((int64_t)t * 3 + d) * gc.Ps * wfmt_bytes(W_F32_18), gc.Ps, c, w);
}

template <int WF>
__global__ void k_export_twolink(const char *__restrict__ W, double *__restrict__ out, SubGeom g, int Lx, int Ly,
                                 int Lz, int64_t total)
{
    int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= total) return;
    const int i = (int)(idx % g.Vs);
    const int64_t r = idx / g.Vs;
    const int d = (int)(r % 3);
    const int b = (int)(r / 3);
    const int t = b >> 3, sub = b & 7;
    Coords c = coords_of(g, sub, i);
    const int64_t site = (((int64_t)t * Lz + c.z) * Ly + c.y) * Lx + c.x;
    typedef typename WFmt<WF>::R R;
    cpx<R> m[9];
    WFmt<WF>::load(W + ((int64_t)b * 3 + d) * g.Ps * wfmt_bytes(WF), g.Ps, i, m);
    double *dst = out + ((site * 3 + d) * 9) * 2;
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        dst[2 * k] = (double)m[k].re;
        dst[2 * k + 1] = (double)m[k].im;
    }
}

// Planar vectors (one vector per launch, persistent forms).  A thread moves the two
// sites x = 2 x', 2 x' + 1 of a canonical row: 48 (FP64: 96) contiguous bytes of the
// caller's vector against one site in each of two sublattice blocks, where consecutive
// lanes are consecutive sites.  HBM-bound; 48^3 x 64, one vector: pack 0.062 ms, unpack
// 0.160 ms with a thread per site (whose 24-byte pieces lie 48 bytes apart), 0.055 and 0.053 now.
// AL: the caller's vectors are 16-byte aligned.
template <typename IO, int VP, bool PACK, bool AL>
__global__ void __launch_bounds__(256) k_move_planar(std::conditional_t<PACK, const IO, IO> *__restrict__ canon, int64_t cvs,
                                                     std::conditional_t<PACK, char, const char> *__restrict__ packed,
                                                     int64_t pvs, SubGeom g, int Ly, int Lz, int t_first, int64_t total)
{
    const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= total) return;
    const int xq = (int)(idx % g.hx);
    const int64_t row = idx / g.hx;
    const int y = (int)(row % Ly);
    const int64_t r2 = row / Ly;
    const int z = (int)(r2 % Lz), ts = (int)(r2 / Lz);
    const int sub0 = ((y & 1) << 1) | ((z & 1) << 2);
    const int i = ((z >> 1) * g.hy + (y >> 1)) * g.hx + xq;
    auto *p = canon + ((int64_t)blockIdx.y * cvs + ((int64_t)t_first * Lz * Ly + row) * (2 * g.hx) + 2 * xq) * 6;
    auto *s = packed + (int64_t)blockIdx.y * pvs + (int64_t)(ts * 8 + sub0) * g.Ps * vfmt_bytes(VP);
    typedef typename VFmt<VP>::R R;
    constexpr int NV = 16 / sizeof(IO);  // reals per 16-byte word
    union {
        float4 q4[3];
        IO v[12];
    } w4;
    IO v[12];
    if constexpr (PACK) {
#pragma unroll
        for (int k = 0; k < 12; k += NV) {
            if constexpr (AL) {
                w4.q4[0] = *reinterpret_cast<const float4 *>(p + k);
#pragma unroll
                for (int j = 0; j < NV; ++j) v[k + j] = w4.v[j];
            } else {
#pragma unroll
                for (int j = 0; j < NV; ++j) v[k + j] = p[k + j];
            }
        }
    }
#pragma unroll
    for (int par = 0; par < 2; ++par) {
        cpx<R> c[3];
        auto *blk = s + (int64_t)par * g.Ps * vfmt_bytes(VP);
        if constexpr (PACK) {
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                c[k].re = (R)v[6 * par + 2 * k];
                c[k].im = (R)v[6 * par + 2 * k + 1];
            }
            VFmt<VP>::template store<false>(blk, g.Ps, i, c);
        } else {
            VFmt<VP>::template load<false>(blk, g.Ps, i, c);
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                v[6 * par + 2 * k] = (IO)c[k].re;
                v[6 * par + 2 * k + 1] = (IO)c[k].im;
            }
        }
    }
    if constexpr (!PACK) {
#pragma unroll
        for (int k = 0; k < 12; k += NV) {
            if constexpr (AL) {
#pragma unroll
                for (int j = 0; j < NV; ++j) w4.v[j] = v[k + j];
                *reinterpret_cast<float4 *>(p + k) = w4.q4[0];
            } else {
#pragma unroll
                for (int j = 0; j < NV; ++j) p[k + j] = v[k + j];
            }
        }
    }
}

// One CTA per vector sums its partials in a fixed order.
__global__ void __launch_bounds__(256) k_reduce_norms(const double *__restrict__ partials, int nparts,
                                                      double *__restrict__ norms)
{
    __shared__ double red[256];
    const int v = blockIdx.x;
    double acc = 0.0;
    for (int k = threadIdx.x; k < nparts; k += blockDim.x) acc += partials[(int64_t)v * nparts + k];
    red[threadIdx.x] = acc;
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if ((int)threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) norms[v] = red[0];
}

// FP64 records: CTA = (nvec, spb); threadIdx.x = vector, threadIdx.y = site.
template <typename IO, int VP>
__global__ void k_pack_il(const IO *__restrict__ src, int64_t svs, char *__restrict__ dst, SubGeom g, int Lx, int Ly,
                          int Lz, int t_first, int64_t nsite, int rec_n, int rec_v0)
{
    const int64_t s = (int64_t)blockIdx.x * blockDim.y + threadIdx.y;
    if (s >= nsite) return;
    const int v = threadIdx.x;
    const int b = (int)(s / g.Vs);
    const int i = (int)(s - (int64_t)b * g.Vs);
    const int t = t_first + (b >> 3), sub = b & 7;
    Coords c = coords_of(g, sub, i);
    const int64_t site = (((int64_t)t * Lz + c.z) * Ly + c.y) * Lx + c.x;
    const IO *p = src + ((int64_t)v * svs + site) * 6;
    typedef typename VRec<VP>::R R;
    cpx<R> val[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        val[k].re = (R)p[2 * k];
        val[k].im = (R)p[2 * k + 1];
    }
    VRec<VP>::store(dst + (int64_t)b * g.Ps * rec_n * vfmt_bytes(VP) + (int64_t)i * rec_n * VRec<VP>::SB, g.Ps * rec_n,
                    rec_v0 + v, val);
}

template <typename IO, int VP>
__global__ void k_unpack_il(const char *__restrict__ src, IO *__restrict__ dst, int64_t dvs, SubGeom g, int Lx,
                            int Ly, int Lz, int t_first, int64_t nsite, int rec_n, int rec_v0)
{
    const int64_t s = (int64_t)blockIdx.x * blockDim.y + threadIdx.y;
    if (s >= nsite) return;
    const int v = threadIdx.x;
    const int b = (int)(s / g.Vs);
    const int i = (int)(s - (int64_t)b * g.Vs);
    const int t = t_first + (b >> 3), sub = b & 7;
    Coords c = coords_of(g, sub, i);
    const int64_t site = (((int64_t)t * Lz + c.z) * Ly + c.y) * Lx + c.x;
    typedef typename VRec<VP>::R R;
    cpx<R> val[3];
    VRec<VP>::load(src + (int64_t)b * g.Ps * rec_n * vfmt_bytes(VP) + (int64_t)i * rec_n * VRec<VP>::SB, g.Ps * rec_n,
                   rec_v0 + v, val);
    IO *p = dst + ((int64_t)v * dvs + site) * 6;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        p[2 * k] = (IO)val[k].re;
        p[2 * k + 1] = (IO)val[k].im;
    }
}

// Partial sums of |psi|^2 of canonical vectors, per (vector, slice, part): part p of slice s of
// vector v goes to partials[v * part_stride + part_off + s * kNormPartsPerSlice + p].  A part is
// S strided subsets of the reals of its slice, 256 sums each, added up subset by subset and then as
// a tree: S depends on the slice alone (norm_subsets), so a norm does not depend on the call
// it is part of.  CL: a cluster of S CTAs, one subset each; otherwise one CTA takes all S, its sums
// independent of one another.  The same bits.
// Bound by the FP64 adds of the SMs in use.  With norms of one slice of 48^3, 3 vectors, a call
// takes 22 us longer with clusters, 38 with one CTA per part; 24 FP32 vectors on 16 slices 1056 and
// 998 us.  Small slices have one subset: a thread of four CTAs would have one or two reals and
// the tree cost more than the sums (16^3 x 32, 72 vectors: 811 us with clusters, 269 now).
constexpr int kNormSplit = 4;

// v summed over the CTA in the order of a tree over the thread index; thread 0 has the sum.
__device__ __forceinline__ double norm_tree(double v, double red[256])
{
    const int t = threadIdx.x;
    red[t] = v;
    __syncthreads();
    if (t < 128) red[t] = v += red[t + 128];
    __syncthreads();
    if (t < 64) red[t] = v += red[t + 64];
    __syncthreads();
    if (t < 32) {
        v += red[t + 32];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    }
    return v;
}

template <typename IO, int S, bool CL>
__device__ __forceinline__ void norm_partials(const IO *__restrict__ base, int64_t vstride, int64_t slice_sites,
                                              double *__restrict__ partials, int64_t part_stride, int64_t part_off)
{
    constexpr int R = CL ? 1 : S;                            // subsets of this CTA
    constexpr int kCtas = kNormPartsPerSlice * (CL ? S : 1);  // of a slice
    __shared__ double red[256];
    const int v = blockIdx.y;
    const int sl = blockIdx.x / kCtas, part = blockIdx.x - sl * kCtas;
    const IO *p = base + ((int64_t)v * vstride + (int64_t)sl * slice_sites) * 6;
    const int64_t n = slice_sites * 6;
    constexpr int64_t step = (int64_t)kNormPartsPerSlice * S * 256;
    double acc[R];
#pragma unroll
    for (int r = 0; r < R; ++r) acc[r] = 0.0;
    int64_t k = (int64_t)part * R * 256 + threadIdx.x;
#pragma unroll(R > 1 ? 2 : 8)
    for (; k + (R - 1) * 256 < n; k += step)
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const double x = (double)p[k + r * 256];
            acc[r] = fma(x, x, acc[r]);
        }
    if constexpr (R > 1) {
#pragma unroll
        for (int r = 0; r < R; ++r)
            if (k + r * 256 < n) {
                const double x = (double)p[k + r * 256];
                acc[r] = fma(x, x, acc[r]);
            }
    }
    double sum = acc[0];
    if constexpr (CL) {
        cooperative_groups::cluster_group cl = cooperative_groups::this_cluster();
        red[threadIdx.x] = sum;
        cl.sync();
        if (cl.block_rank() == 0)
            for (int r = 1; r < S; ++r) sum += *cl.map_shared_rank(red + threadIdx.x, r);
        cl.sync();  // no CTA leaves or reuses its sums while they are read
        if (cl.block_rank() != 0) return;
    } else {
#pragma unroll
        for (int r = 1; r < R; ++r) sum += acc[r];
    }
    sum = norm_tree(sum, red);
    if (threadIdx.x == 0) partials[(int64_t)v * part_stride + part_off + blockIdx.x / (CL ? S : 1)] = sum;
}

template <typename IO, int S>
__global__ void __launch_bounds__(256)
    k_norm_partials(const IO *__restrict__ base, int64_t vstride, int64_t slice_sites, double *__restrict__ partials,
                    int64_t part_stride, int64_t part_off)
{
    norm_partials<IO, S, false>(base, vstride, slice_sites, partials, part_stride, part_off);
}

template <typename IO>
__global__ void __cluster_dims__(kNormSplit, 1, 1) __launch_bounds__(256)
    k_norm_partials_cl(const IO *__restrict__ base, int64_t vstride, int64_t slice_sites, double *__restrict__ partials,
                       int64_t part_stride, int64_t part_off)
{
    norm_partials<IO, kNormSplit, true>(base, vstride, slice_sites, partials, part_stride, part_off);
}

// Copies the interleaved records of one x'-row (hx sites starting at site r of
// block b, all rec_n vectors) between global memory and a shared-memory row
// of the same layout (colour planes hx * rec_n elements apart), 16 bytes per
// thread and step.  to_smem selects the direction.
template <int VP>
__device__ __forceinline__ void row_copy(unsigned char *smr, const void *gbase, int b, int r, const SubGeom &g, int hx,
                                         int rec_n, bool to_smem)
{
    constexpr int SB = VRec<VP>::SB;
    const int segB = hx * rec_n * SB;  // one colour (or the whole row for 16-bit records)
    const int nseg = il_planes(VP) ? 3 : 1;
    char *blk = (char *)gbase + (int64_t)b * g.Ps * rec_n * vfmt_bytes(VP);
    for (int c = 0; c < nseg; ++c) {
        uint4 *gs = reinterpret_cast<uint4 *>(blk + ((int64_t)c * g.Ps + r) * rec_n * SB);
        uint4 *ss = reinterpret_cast<uint4 *>(smr + c * segB);
        if (to_smem)
            for (int k = threadIdx.x; k < segB / 16; k += blockDim.x) ss[k] = gs[k];
        else
            for (int k = threadIdx.x; k < segB / 16; k += blockDim.x) gs[k] = ss[k];
    }
}

// Row transposes between the canonical layout and the interleaved records.
// One CTA per canonical x-row (t, z, y): the row's Lx sites are two x'-rows
// of hx records groups in sublattices (x even) and (x odd), each a contiguous
// segment of hx * nvec records.  Both segments go through shared memory so
// that the global side of either layout is read and written in contiguous
// runs (nvec canonical rows of Lx sites, two record segments).
template <typename IO, int VP>
__global__ void __launch_bounds__(256) k_unpack_rows(const char *__restrict__ src, IO *__restrict__ dst, int64_t dvs,
                                                     SubGeom g, int Lx, int Ly, int Lz, int t_first, int nvec,
                                                     int rec_n, int rec_v0)
{
    extern __shared__ __align__(16) unsigned char smr[];
    constexpr int VBY = vfmt_bytes(VP);
    const int y = blockIdx.x % Ly, z = blockIdx.x / Ly;
    const int ts = blockIdx.y;
    const int hx = g.hx;
    const int sub0 = ((y & 1) << 1) | ((z & 1) << 2);
    const int r = ((z >> 1) * g.hy + (y >> 1)) * hx;
    const int segB = hx * rec_n * VBY;
    // stage both x'-rows (all rec_n records) with 16-byte loads
    for (int par = 0; par < 2; ++par) row_copy<VP>(smr + par * segB, src, ts * 8 + (sub0 | par), r, g, hx, rec_n, true);
    __syncthreads();
    typedef typename VRec<VP>::R R;
    const int64_t site0 = (((int64_t)(t_first + ts) * Lz + z) * Ly + y) * Lx;
    for (int k = threadIdx.x; k < nvec * Lx; k += blockDim.x) {
        const int v = k / Lx, x = k - v * Lx;
        cpx<R> val[3];
        VRec<VP>::load(reinterpret_cast<const char *>(smr) + (x & 1) * segB + (x >> 1) * rec_n * VRec<VP>::SB, hx * rec_n,
                       rec_v0 + v, val);
        IO *p = dst + ((int64_t)v * dvs + site0 + x) * 6;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            p[2 * c] = (IO)val[c].re;
            p[2 * c + 1] = (IO)val[c].im;
        }
    }
}

template <typename IO, int VP>
__global__ void __launch_bounds__(256) k_pack_rows(const IO *__restrict__ src, int64_t svs, char *__restrict__ dst,
                                                   SubGeom g, int Lx, int Ly, int Lz, int t_first, int nvec, int rec_n,
                                                   int rec_v0)
{
    extern __shared__ __align__(16) unsigned char smr[];
    constexpr int VBY = vfmt_bytes(VP);
    const int y = blockIdx.x % Ly, z = blockIdx.x / Ly;
    const int ts = blockIdx.y;
    const int hx = g.hx;
    const int sub0 = ((y & 1) << 1) | ((z & 1) << 2);
    const int r = ((z >> 1) * g.hy + (y >> 1)) * hx;
    const int segB = hx * rec_n * VBY;
    const bool partial = nvec != rec_n;
    if (partial) {  // keep the records of the other slots: start from the current segments
        for (int par = 0; par < 2; ++par)
            row_copy<VP>(smr + par * segB, dst, ts * 8 + (sub0 | par), r, g, hx, rec_n, true);
        __syncthreads();
    }
    typedef typename VRec<VP>::R R;
    const int64_t site0 = (((int64_t)(t_first + ts) * Lz + z) * Ly + y) * Lx;
    for (int k = threadIdx.x; k < nvec * Lx; k += blockDim.x) {
        const int v = k / Lx, x = k - v * Lx;
        const IO *p = src + ((int64_t)v * svs + site0 + x) * 6;
        cpx<R> val[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            val[c].re = (R)p[2 * c];
            val[c].im = (R)p[2 * c + 1];
        }
        VRec<VP>::store(reinterpret_cast<char *>(smr) + (x & 1) * segB + (x >> 1) * rec_n * VRec<VP>::SB, hx * rec_n,
                        rec_v0 + v, val);
    }
    __syncthreads();
    for (int par = 0; par < 2; ++par)
        row_copy<VP>(smr + par * segB, dst, ts * 8 + (sub0 | par), r, g, hx, rec_n, false);
}

// --------------------------------------------------------------------------
// Pack and unpack of the FP32 and 16-bit interleaved records, by vector pairs.
// A thread moves one record pair of one site: two canonical colour vectors of 24
// (FP64 caller: 48) bytes each against one 16-byte word per colour, or one 32-byte
// record.  CTA = one or several canonical x-rows (pair_split); consecutive lanes take up
// to four pairs of a site, then the next site, so that the records of the even and of the
// odd sites of the row are written in runs (nvg = 8: contiguous, 256 bytes per colour and
// warp) and the canonical side is read in runs of eight sites per vector, every
// sector in full.  Both sides go straight between global memory and registers.
// HBM-bound: 48^3 x 32, 24 vectors, FP32 1.00 / 1.33 ms (pack / unpack) with the
// rows staged in shared memory one vector at a time, 0.58 / 0.82 now (4.1 GB moved); FP16
// 2.14 / 1.30, now 0.50 / 0.64.
// grid.z: vector groups (column kernel), rec_n records each; record rec_v0 + v of a
// group holds vector v.  A pair of which the caller owns one vector only leaves the
// other half alone.  AL: the caller's vectors are aligned to a complex number.
// --------------------------------------------------------------------------
// Site i of an interleaved block, in units of rec_n * SB bytes: the colour
// planes of the block, or (rc) of each x'-row, one row behind the other.
template <int VP> __device__ __forceinline__ int64_t il_site(const SubGeom &g, int i, bool rc)
{
    if (!rc || !il_planes(VP)) return i;
    const int row = i / g.hx;
    return (int64_t)row * 2 * g.hx + i;
}

template <typename IO, bool AL> __device__ __forceinline__ void io_load(const IO *p, IO v[6])
{
    if constexpr (AL && sizeof(IO) == 4) {
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const float2 q = reinterpret_cast<const float2 *>(p)[c];
            v[2 * c] = q.x;
            v[2 * c + 1] = q.y;
        }
    } else if constexpr (AL) {
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const double2 q = reinterpret_cast<const double2 *>(p)[c];
            v[2 * c] = q.x;
            v[2 * c + 1] = q.y;
        }
    } else {
#pragma unroll
        for (int k = 0; k < 6; ++k) v[k] = p[k];
    }
}

template <typename IO, bool AL> __device__ __forceinline__ void io_store(IO *p, const cpx<float> x[3])
{
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        if constexpr (AL && sizeof(IO) == 4)
            reinterpret_cast<float2 *>(p)[c] = make_float2(x[c].re, x[c].im);
        else if constexpr (AL)
            reinterpret_cast<double2 *>(p)[c] = make_double2((double)x[c].re, (double)x[c].im);
        else {
            p[2 * c] = (IO)x[c].re;
            p[2 * c + 1] = (IO)x[c].im;
        }
    }
}

struct PairArgs {
    int64_t vs;            // canonical vector stride in sites
    int Lx, Ly, Lz, t_first;
    int nvec, rec_n, rec_v0;
    int64_t gstride;       // bytes between the fields of two groups
    bool rc, whole;        // rows contiguous; blocks are whole slices
    PairSplit sp;
};

template <typename IO, int VP, bool PACK, bool AL>
__global__ void __launch_bounds__(256) k_move_pairs(std::conditional_t<PACK, const IO, IO> *__restrict__ canon,
                                                    std::conditional_t<PACK, char, const char> *__restrict__ recs,
                                                    SubGeom g, PairArgs a)
{
    const int ts = blockIdx.y;
    const int first = blockIdx.z * a.rec_n;  // vectors of the groups before this one
    const int nv = min(a.nvec - first, a.rec_n);
    const int u0 = a.rec_v0 >> 1, T = ((a.rec_v0 + nv + 1) >> 1) - u0;
    const int64_t sb = (int64_t)a.rec_n * VRec<VP>::SB;
    const int cs = (int)((a.rc ? g.hx : g.Ps) * a.rec_n);
    const int C = a.sp.pairs, per = a.Lx * C, rowI = per * a.sp.chunks;
    for (int k = threadIdx.x; k < a.sp.rows * rowI; k += blockDim.x) {
        const int rl = k / rowI, j = k - rl * rowI;      // row, item of the row
        const int ch = j / per, i = j - ch * per;        // chunk of pairs, item of the chunk
        const int x = i / C, t = ch * C + i - x * C;     // site, pair
        const int yz = blockIdx.x * a.sp.rows + rl;
        if (t >= T || yz >= a.Ly * a.Lz) continue;
        const int y = yz % a.Ly, z = yz / a.Ly, u = u0 + t;
        const int sub0 = ((y & 1) << 1) | ((z & 1) << 2);
        const int r = a.whole ? (z * g.hy + y) * g.hx : ((z >> 1) * g.hy + (y >> 1)) * g.hx;
        const int64_t site0 = (((int64_t)(a.t_first + ts) * a.Lz + z) * a.Ly + y) * a.Lx;
        const int64_t row = il_site<VP>(g, r, a.rc);
        const int v0 = 2 * u - a.rec_v0;
        const bool on0 = v0 >= 0, on1 = v0 + 1 < nv;
        const int b = a.whole ? ts : ts * 8 + (sub0 | (x & 1));
        auto *s = recs + blockIdx.z * a.gstride + ((int64_t)b * g.Ps * a.rec_n) * vfmt_bytes(VP) +
                  (row + (a.whole ? x : x >> 1)) * sb;
        auto *p = canon + ((int64_t)(first + v0) * a.vs + site0 + x) * 6;
        const int64_t next = a.vs * 6;
        cpx<float> q[2][3];
        if constexpr (PACK) {
            IO w[2][6];
            if (on0) io_load<IO, AL>(p, w[0]);
            if (on1) io_load<IO, AL>(p + next, w[1]);
#pragma unroll
            for (int j = 0; j < 2; ++j)
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    q[j][c].re = (float)w[j][2 * c];
                    q[j][c].im = (float)w[j][2 * c + 1];
                }
            if (on0 && on1)
                VRec<VP>::store2(s, cs, u, q[0], q[1]);
            else if (on0)
                VRec<VP>::store(s, cs, 2 * u, q[0]);
            else
                VRec<VP>::store(s, cs, 2 * u + 1, q[1]);
        } else {
            VRec<VP>::load2(s, cs, u, q[0], q[1]);
            if (on0) io_store<IO, AL>(p, q[0]);
            if (on1) io_store<IO, AL>(p + next, q[1]);
        }
    }
}

template <typename IO, bool PACK>
cudaError_t move_pairs(const void *canon, char *recs, int prec, const SubGeom &g, int nsl, int ngrp, const PairArgs &a,
                       cudaStream_t s)
{
    const dim3 grid((unsigned)((a.Ly * a.Lz + a.sp.rows - 1) / a.sp.rows), nsl, ngrp);
    if (nsl > 65535 || ngrp > 65535) return cudaErrorInvalidConfiguration;
    const bool al = reinterpret_cast<uintptr_t>(canon) % (2 * sizeof(IO)) == 0;
    auto go = [&](auto k_al, auto k) {
        if (al)
            k_al<<<grid, 256, 0, s>>>((IO *)canon, recs, g, a);
        else
            k<<<grid, 256, 0, s>>>((IO *)canon, recs, g, a);
        return cudaGetLastError();
    };
    switch (prec) {
    case P_F32: return go(k_move_pairs<IO, P_F32, PACK, true>, k_move_pairs<IO, P_F32, PACK, false>);
    case P_F16: return go(k_move_pairs<IO, P_F16, PACK, true>, k_move_pairs<IO, P_F16, PACK, false>);
    case P_BF16: return go(k_move_pairs<IO, P_BF16, PACK, true>, k_move_pairs<IO, P_BF16, PACK, false>);
    default: return cudaErrorNotSupported;
    }
}

inline int spb_of(int nvec) { return std::max(1, 256 / nvec); }

inline unsigned nblocks(int64_t n, int t) { return (unsigned)((n + t - 1) / t); }

template <typename IO, bool PACK>
cudaError_t move_planar(const void *canon, int64_t cvs, char *packed, int prec, int64_t pvs, const SubGeom &g,
                        const int L[4], int t_first, int nsl, int nvec, cudaStream_t s)
{
    const int64_t total = (int64_t)nsl * L[2] * L[1] * g.hx;
    const dim3 grid(nblocks(total, 256), nvec);
    const bool al = reinterpret_cast<uintptr_t>(canon) % 16 == 0;
    auto go = [&](auto k_al, auto k) {
        if (al)
            k_al<<<grid, 256, 0, s>>>((IO *)canon, cvs, packed, pvs, g, L[1], L[2], t_first, total);
        else
            k<<<grid, 256, 0, s>>>((IO *)canon, cvs, packed, pvs, g, L[1], L[2], t_first, total);
        return cudaGetLastError();
    };
    switch (prec) {
    case P_F64: return go(k_move_planar<IO, P_F64, PACK, true>, k_move_planar<IO, P_F64, PACK, false>);
    case P_F32: return go(k_move_planar<IO, P_F32, PACK, true>, k_move_planar<IO, P_F32, PACK, false>);
    case P_F16: return go(k_move_planar<IO, P_F16, PACK, true>, k_move_planar<IO, P_F16, PACK, false>);
    case P_BF16: return go(k_move_planar<IO, P_BF16, PACK, true>, k_move_planar<IO, P_BF16, PACK, false>);
    default: return cudaErrorNotSupported;
    }
}

}  // namespace

cudaError_t launch_ingest_gauge(const double *U, int nd, double *Up, const SubGeom &g, const int L[4], cudaStream_t s)
{
    const int64_t nrow = (int64_t)L[1] * L[2] * L[3];
    const int rows = ingest_rows(L[0], kIngestSites, nrow);
    if (rows > 0) {
        k_ingest_rows<<<(unsigned)((nrow + rows - 1) / rows), 256, 0, s>>>(U, nd, reinterpret_cast<double2 *>(Up), g, L[0],
                                                                          L[1], L[2], rows, nrow);
        return cudaGetLastError();
    }
    const int runs = (L[0] + kIngestSites - 1) / kIngestSites;
    const int64_t blocks = (int64_t)L[1] * L[2] * L[3] * runs;
    if (blocks == 0) return cudaSuccess;
    k_ingest_gauge<<<(unsigned)blocks, 256, 0, s>>>(U, nd, reinterpret_cast<double2 *>(Up), g, L[0], L[1], L[2], runs);
    return cudaGetLastError();
}

cudaError_t launch_export_gauge(const double *Up, double *out, const SubGeom &g, const int L[4], cudaStream_t s)
{
    const int64_t total = (int64_t)L[3] * 8 * 3 * g.Vs;
    if (total == 0) return cudaSuccess;
    k_export_gauge<<<nblocks(total, 256), 256, 0, s>>>(reinterpret_cast<const double2 *>(Up), out, g, L[0], L[1],
                                                       L[2], total);
    return cudaGetLastError();
}

cudaError_t launch_build_twolink(const double *Up, char *W, int wfmt, const SubGeom &g, int nblk, int *err,
                                 cudaStream_t s)
{
    const int64_t total = (int64_t)nblk * 3 * g.Vs;
    if (total == 0) return cudaSuccess;
    const double2 *u = reinterpret_cast<const double2 *>(Up);
    const unsigned nb = nblocks(total, 128);
    switch (wfmt) {
    case W_F64_18: k_build_twolink<W_F64_18><<<nb, 128, 0, s>>>(u, W, g, total, err); break;
    case W_F32_18: k_build_split<3><<<nb, 128, 0, s>>>(u, W, g, total); break;
    case W_F32_12: k_build_split<2><<<nb, 128, 0, s>>>(u, W, g, total); break;
    case W_F32_8: k_build_twolink<W_F32_8><<<nb, 128, 0, s>>>(u, W, g, total, err); break;
    case W_F16_18: k_build_twolink<W_F16_18><<<nb, 128, 0, s>>>(u, W, g, total, err); break;
    case W_F16_12: k_build_twolink<W_F16_12><<<nb, 128, 0, s>>>(u, W, g, total, err); break;
    case W_BF16_18: k_build_twolink<W_BF16_18><<<nb, 128, 0, s>>>(u, W, g, total, err); break;
    case W_BF16_12: k_build_twolink<W_BF16_12><<<nb, 128, 0, s>>>(u, W, g, total, err); break;
    default: return cudaErrorNotSupported;
    }
    return cudaGetLastError();
}

cudaError_t launch_build_links(const double *Up, char *L1, int wfmt, const SubGeom &g, int nblk, cudaStream_t s)
{
    const int64_t total = (int64_t)nblk * 3 * g.Vs;
    if (total == 0) return cudaSuccess;
    const double2 *u = reinterpret_cast<const double2 *>(Up);
    const unsigned nb = nblocks(total, 128);
    switch (wfmt) {
    case W_F64_18: k_build_twolink<W_F64_18, true><<<nb, 128, 0, s>>>(u, L1, g, total, nullptr); break;
    default: return cudaErrorNotSupported;
    }
    return cudaGetLastError();
}

cudaError_t launch_build_links_slices(const double *Up, char *L1, const SubGeom &g, const SubGeom &gc, int nsl,
                                      cudaStream_t s)
{
    const int64_t total = (int64_t)nsl * 3 * gc.Vs;
    if (total == 0) return cudaSuccess;
    k_links_slices<<<nblocks(total, 128), 128, 0, s>>>(reinterpret_cast<const double2 *>(Up), L1, g, gc, total);
    return cudaGetLastError();
}

cudaError_t launch_export_twolink(const char *W, int wfmt, double *out, const SubGeom &g, const int L[4],
                                  cudaStream_t s)
{
    const int64_t total = (int64_t)L[3] * 8 * 3 * g.Vs;
    if (total == 0) return cudaSuccess;
    const unsigned nb = nblocks(total, 128);
    switch (wfmt) {
    case W_F64_18: k_export_twolink<W_F64_18><<<nb, 128, 0, s>>>(W, out, g, L[0], L[1], L[2], total); break;
    case W_F32_18: k_export_twolink<W_F32_18><<<nb, 128, 0, s>>>(W, out, g, L[0], L[1], L[2], total); break;
    case W_F32_12: k_export_twolink<W_F32_12><<<nb, 128, 0, s>>>(W, out, g, L[0], L[1], L[2], total); break;
    case W_F32_8: k_export_twolink<W_F32_8><<<nb, 128, 0, s>>>(W, out, g, L[0], L[1], L[2], total); break;
    case W_F16_18: k_export_twolink<W_F16_18><<<nb, 128, 0, s>>>(W, out, g, L[0], L[1], L[2], total); break;
    case W_F16_12: k_export_twolink<W_F16_12><<<nb, 128, 0, s>>>(W, out, g, L[0], L[1], L[2], total); break;
    case W_BF16_18: k_export_twolink<W_BF16_18><<<nb, 128, 0, s>>>(W, out, g, L[0], L[1], L[2], total); break;
    case W_BF16_12: k_export_twolink<W_BF16_12><<<nb, 128, 0, s>>>(W, out, g, L[0], L[1], L[2], total); break;
    default: return cudaErrorNotSupported;
    }
    return cudaGetLastError();
}

cudaError_t launch_pack_vectors(const void *src, int io_prec, int64_t src_vstride_sites, char *dst, int prec,
                                int64_t dst_vstride, const SubGeom &g, const int L[4], int t_first, int nsl,
                                int nvec, cudaStream_t s)
{
    if ((int64_t)nsl * 8 * g.Vs == 0 || nvec == 0) return cudaSuccess;
    if (io_prec == P_F64)
        return move_planar<double, true>(src, src_vstride_sites, dst, prec, dst_vstride, g, L, t_first, nsl, nvec, s);
    if (io_prec == P_F32)
        return move_planar<float, true>(src, src_vstride_sites, dst, prec, dst_vstride, g, L, t_first, nsl, nvec, s);
    return cudaErrorNotSupported;
}

cudaError_t launch_unpack_vectors(const char *src, int prec, int64_t src_vstride, void *dst, int io_prec,
                                  int64_t dst_vstride_sites, const SubGeom &g, const int L[4], int t_first,
                                  int nsl, int nvec, cudaStream_t s)
{
    if ((int64_t)nsl * 8 * g.Vs == 0 || nvec == 0) return cudaSuccess;
    char *p = const_cast<char *>(src);
    if (io_prec == P_F64)
        return move_planar<double, false>(dst, dst_vstride_sites, p, prec, src_vstride, g, L, t_first, nsl, nvec, s);
    if (io_prec == P_F32)
        return move_planar<float, false>(dst, dst_vstride_sites, p, prec, src_vstride, g, L, t_first, nsl, nvec, s);
    return cudaErrorNotSupported;
}

static bool rows_transpose_ok(const SubGeom &g, int rec_n, int prec, const int L[4])
{
    // each colour plane's (or the 16-bit row's) segment is copied in 16-byte words
    const int colB = g.hx * rec_n * il_site_bytes(prec);
    const int rowB = g.hx * rec_n * vfmt_bytes(prec);
    return colB % 16 == 0 && 2 * rowB <= 48 * 1024 && (int64_t)L[1] * L[2] <= 0x7fffffff;
}

// FP64 records: whole rows through shared memory where they fit, else site by site.
template <typename IO>
static cudaError_t move_f64(bool pack, const void *canon, int64_t vs, char *recs, const SubGeom &g, const int L[4],
                            int t_first, int nsl, int nvec, int rec_n, int rec_v0, cudaStream_t s)
{
    if (rows_transpose_ok(g, rec_n, P_F64, L)) {
        const dim3 grid((unsigned)(L[1] * L[2]), nsl);
        const int smem = 2 * g.hx * rec_n * vfmt_bytes(P_F64);
        if (pack)
            k_pack_rows<IO, P_F64><<<grid, 256, smem, s>>>((const IO *)canon, vs, recs, g, L[0], L[1], L[2], t_first, nvec,
                                                          rec_n, rec_v0);
        else
            k_unpack_rows<IO, P_F64><<<grid, 256, smem, s>>>(recs, (IO *)canon, vs, g, L[0], L[1], L[2], t_first, nvec,
                                                            rec_n, rec_v0);
        return cudaGetLastError();
    }
    const int spb = spb_of(nvec);
    const int64_t nsite = (int64_t)nsl * 8 * g.Vs;
    const dim3 block(nvec, spb), grid(nblocks(nsite, spb));
    if (pack)
        k_pack_il<IO, P_F64><<<grid, block, 0, s>>>((const IO *)canon, vs, recs, g, L[0], L[1], L[2], t_first, nsite, rec_n,
                                                    rec_v0);
    else
        k_unpack_il<IO, P_F64><<<grid, block, 0, s>>>(recs, (IO *)canon, vs, g, L[0], L[1], L[2], t_first, nsite, rec_n,
                                                      rec_v0);
    return cudaGetLastError();
}

template <bool PACK>
static cudaError_t move_il(const void *canon, int io_prec, int64_t vs, char *recs, int prec, const SubGeom &g,
                           const int L[4], int t_first, int nsl, int nvec, int rec_n, int rec_v0, cudaStream_t s, bool rc, bool whole)
{
    if ((int64_t)nsl * 8 * g.Vs == 0 || nvec == 0) return cudaSuccess;
    const int ngrp = rc && rec_v0 == 0 ? (nvec + rec_n - 1) / rec_n : 1;
    if (nvec > 256 || rec_v0 < 0 || (ngrp == 1 && rec_v0 + nvec > rec_n)) return cudaErrorInvalidValue;
    if (io_prec != P_F64 && io_prec != P_F32) return cudaErrorNotSupported;
    if (prec == P_F64) {
        if (rc || whole) return cudaErrorNotSupported;
        return io_prec == P_F64
                   ? move_f64<double>(PACK, canon, vs, recs, g, L, t_first, nsl, nvec, rec_n, rec_v0, s)
                   : move_f64<float>(PACK, canon, vs, recs, g, L, t_first, nsl, nvec, rec_n, rec_v0, s);
    }
    const int T = ((rec_v0 + std::min(nvec, rec_n) + 1) >> 1) - (rec_v0 >> 1);  // pairs of the largest group
    const PairArgs a{vs, L[0], L[1], L[2], t_first, nvec, rec_n, rec_v0, (int64_t)nsl * (whole ? 1 : 8) * g.Ps * rec_n * vfmt_bytes(prec),
                     rc, whole, pair_split(T, L[0], L[1] * L[2])};
    return io_prec == P_F64 ? move_pairs<double, PACK>(canon, recs, prec, g, nsl, ngrp, a, s)
                            : move_pairs<float, PACK>(canon, recs, prec, g, nsl, ngrp, a, s);
}

cudaError_t launch_pack_il(const void *src, int io_prec, int64_t src_vstride_sites, char *dst, int prec,
                           const SubGeom &g, const int L[4], int t_first, int nsl, int nvec, int rec_n, int rec_v0,
                           cudaStream_t s, bool rc, bool whole)
{
    return move_il<true>(src, io_prec, src_vstride_sites, dst, prec, g, L, t_first, nsl, nvec, rec_n, rec_v0, s, rc, whole);
}

cudaError_t launch_unpack_il(const char *src, int prec, void *dst, int io_prec, int64_t dst_vstride_sites,
                             const SubGeom &g, const int L[4], int t_first, int nsl, int nvec, int rec_n, int rec_v0,
                             cudaStream_t s, bool rc, bool whole)
{
    return move_il<false>(dst, io_prec, dst_vstride_sites, const_cast<char *>(src), prec, g, L, t_first, nsl, nvec, rec_n,
                          rec_v0, s, rc, whole);
}

template <typename IO>
static cudaError_t norm_launch(const void *base, int64_t vstride_sites, int64_t slice_sites, int nsl, int nvec,
                               double *partials, int64_t part_stride, int64_t part_off, cudaStream_t s)
{
    const IO *p = (const IO *)base;
    const dim3 one(nsl * kNormPartsPerSlice, nvec), split(nsl * kNormPartsPerSlice * kNormSplit, nvec);
    if (norm_subsets(slice_sites, kNormSplit) == 1)
        k_norm_partials<IO, 1><<<one, 256, 0, s>>>(p, vstride_sites, slice_sites, partials, part_stride, part_off);
    else if (norm_cluster(nsl, nvec))
        k_norm_partials_cl<IO><<<split, 256, 0, s>>>(p, vstride_sites, slice_sites, partials, part_stride, part_off);
    else
        k_norm_partials<IO, kNormSplit><<<one, 256, 0, s>>>(p, vstride_sites, slice_sites, partials, part_stride, part_off);
    return cudaGetLastError();
}

cudaError_t launch_norm_partials(const void *base, int io_prec, int64_t vstride_sites, int64_t slice_sites, int nsl,
                                 int nvec, double *partials, int64_t part_stride, int64_t part_off, cudaStream_t s)
{
    if (nvec == 0 || nsl == 0) return cudaSuccess;
    if ((int64_t)nsl * kNormPartsPerSlice * kNormSplit > 0x7fffffff || nvec > 65535) return cudaErrorInvalidValue;
    if (io_prec == P_F64)
        return norm_launch<double>(base, vstride_sites, slice_sites, nsl, nvec, partials, part_stride, part_off, s);
    if (io_prec == P_F32)
        return norm_launch<float>(base, vstride_sites, slice_sites, nsl, nvec, partials, part_stride, part_off, s);
    return cudaErrorNotSupported;
}

cudaError_t launch_reduce_norms(const double *partials, int nparts, int nvec, double *norms, cudaStream_t s)
{
    if (nvec == 0) return cudaSuccess;
    k_reduce_norms<<<nvec, 256, 0, s>>>(partials, nparts, norms);
    return cudaGetLastError();
}

}  // namespace tls
