// k_ape.cu -- APE smearing of the spatial links (gauge-smeared links in place
// of U_mu, Sec. 2, the remark after Eq. tlSmear).
//
// One step, every link from the previous iterate (out of place):
//   V_mu(x) = (1 - a) U_mu(x) + (a/4) sum_{nu != mu, spatial} [
//       U_nu(x) U_mu(x+nu) U_nu(x+mu)^dag + U_nu(x-nu)^dag U_mu(x-nu) U_nu(x-nu+mu) ]
//   U'_mu(x) = P(V_mu(x))
// P is the projection onto SU(3): the unitary polar factor of V by Newton's
// iteration X <- (X + X^-dag) / 2 (at most 100 steps), then multiplied by
// exp(-i phi / 3) with phi = arg det X in (-pi, pi].  All results are FP64 on the
// packed links (sublattice layout, double2 planes).  A singular V or an iteration
// that does not settle sets DERR_PROJECT and leaves that link unchanged.
//
// The FP64 pipe bounds the kernel (1/75 of the FP32 rate), so what counts is the
// number of FP64 instructions per link: products accumulate by FMA (864 for the
// eight of the staples, 1250 with separate adds); a Newton step takes about 155
// (280 with two divisions, separate adds and an explicit change); the end of the
// iteration is seen from |det X|^2, which the step has anyway, and stops where the
// next step changes nothing (about 5 steps for smooth links, 7 when the change
// itself had to fall below 1e-12); and the cube root of the determinant starts
// from FP32.  Three steps at 32^3 x 32: 47.1 ms before, 25.9 ms now.
#include "tls_dev.cuh"
#include "tls_internal.h"

namespace tls {
namespace {

struct M3 {
    double2 e[9];  // row-major complex 3x3
};

__device__ __forceinline__ double2 cm(double2 a, double2 b)
{
    return make_double2(fma(a.x, b.x, -a.y * b.y), fma(a.x, b.y, a.y * b.x));
}

// acc + a b and acc - a b
__device__ __forceinline__ double2 cfma(double2 a, double2 b, double2 acc)
{
    return make_double2(fma(-a.y, b.y, fma(a.x, b.x, acc.x)), fma(a.y, b.x, fma(a.x, b.y, acc.y)));
}
__device__ __forceinline__ double2 cfms(double2 a, double2 b, double2 acc)
{
    return make_double2(fma(a.y, b.y, fma(-a.x, b.x, acc.x)), fma(-a.y, b.x, fma(-a.x, b.y, acc.y)));
}

// c + a b
__device__ __forceinline__ M3 mul_add(const M3 &a, const M3 &b, M3 c)
{
#pragma unroll
    for (int r = 0; r < 3; ++r)
#pragma unroll
        for (int s = 0; s < 3; ++s)
#pragma unroll
            for (int k = 0; k < 3; ++k) c.e[r * 3 + s] = cfma(a.e[r * 3 + k], b.e[k * 3 + s], c.e[r * 3 + s]);
    return c;
}

__device__ __forceinline__ M3 mul(const M3 &a, const M3 &b)
{
    M3 c;
#pragma unroll
    for (int r = 0; r < 3; ++r)
#pragma unroll
        for (int s = 0; s < 3; ++s) {
            double2 acc = cm(a.e[r * 3], b.e[s]);
            acc = cfma(a.e[r * 3 + 1], b.e[3 + s], acc);
            c.e[r * 3 + s] = cfma(a.e[r * 3 + 2], b.e[6 + s], acc);
        }
    return c;
}

__device__ __forceinline__ M3 dag(const M3 &a)
{
    M3 d;
#pragma unroll
    for (int r = 0; r < 3; ++r)
#pragma unroll
        for (int s = 0; s < 3; ++s) d.e[r * 3 + s] = make_double2(a.e[s * 3 + r].x, -a.e[s * 3 + r].y);
    return d;
}

// Cofactor C_rs of a 3x3 complex matrix: with cyclic indices the sign is built in.
__device__ __forceinline__ double2 cofactor(const M3 &m, int r, int s)
{
    const int r0 = (r + 1) % 3, r1 = (r + 2) % 3, s0 = (s + 1) % 3, s1 = (s + 2) % 3;
    return cfms(m.e[r0 * 3 + s1], m.e[r1 * 3 + s0], cm(m.e[r0 * 3 + s0], m.e[r1 * 3 + s1]));
}

__device__ __forceinline__ double2 det(const M3 &m)
{
    return cfma(m.e[2], cofactor(m, 0, 2), cfma(m.e[1], cofactor(m, 0, 1), cm(m.e[0], cofactor(m, 0, 0))));
}

// z^(-1/3) of a unit complex number, the branch exp(-i phi / 3), phi = arg z in (-pi, pi]:
// from FP32, then two Newton steps w <- w (4 - z w^3) / 3 (errors 1e-7, 1e-14, below 1e-16).
__device__ __forceinline__ double2 inv_cbrt(double2 z)
{
    const float phi = atan2f((float)z.y, (float)z.x) * (1.0f / 3.0f);
    float sn, cn;
    sincosf(phi, &sn, &cn);
    double2 w = make_double2((double)cn, -(double)sn);
#pragma unroll
    for (int it = 0; it < 2; ++it) {
        const double2 w3z = cm(cm(cm(w, w), w), z);
        w = cm(w, make_double2(fma(-1.0 / 3.0, w3z.x, 4.0 / 3.0), -1.0 / 3.0 * w3z.y));
    }
    return w;
}

// From the first step on the singular values are 1 + e with e >= 0 and a step takes e to
// e^2 / 2; |det X|^2 - 1 is then twice the sum of the e.  Below 2e-8 the step being made
// leaves e <= 5e-17.
__device__ bool project_su3(M3 &x)
{
    bool done = false;
    for (int it = 0; it < 100 && !done; ++it) {
        M3 c;
#pragma unroll
        for (int r = 0; r < 3; ++r)
#pragma unroll
            for (int s = 0; s < 3; ++s) c.e[r * 3 + s] = cofactor(x, r, s);
        const double2 d = cfma(x.e[2], c.e[2], cfma(x.e[1], c.e[1], cm(x.e[0], c.e[0])));
        const double n2 = fma(d.x, d.x, d.y * d.y);
        if (!(n2 > 0.0)) return false;
        done = it > 0 && fabs(n2 - 1.0) < 2e-8;
        // X^-dag = (adj X / det X)^dag: element (r, s) = conj(C_rs / det)
        double2 rd;  // 1 / (2 det)
        if (n2 > 1e-280) {
            const double h = 0.5 / n2;
            rd = make_double2(d.x * h, -d.y * h);
        } else {  // h would overflow
            rd = make_double2(0.5 * (d.x / n2), -0.5 * (d.y / n2));
        }
#pragma unroll
        for (int k = 0; k < 9; ++k) {
            const double re = fma(-c.e[k].y, rd.y, fma(c.e[k].x, rd.x, 0.5 * x.e[k].x));
            const double im = fma(-c.e[k].x, rd.y, fma(-c.e[k].y, rd.x, 0.5 * x.e[k].y));
            x.e[k] = make_double2(re, im);
        }
    }
    if (!done) return false;
    const double2 ph = inv_cbrt(det(x));
#pragma unroll
    for (int k = 0; k < 9; ++k) x.e[k] = cm(x.e[k], ph);
    return true;
}

// Site reached from (block b, site i) by one step along spatial direction d
// (dir = +1 or -1): the sublattice bit d flips; the half coordinate moves only
// when leaving an odd coordinate forwards or an even one backwards.
__device__ __forceinline__ void step1(const SubGeom &g, int &b, int &i, int d, int dir)
{
    const int sub = b & 7;
    const int odd = (sub >> d) & 1;
    const int h[3] = {g.hx, g.hy, g.hz};
    int q[3];
    q[0] = i % g.hx;
    const int r = i / g.hx;
    q[1] = r % g.hy;
    q[2] = r / g.hy;
    if (dir > 0 && odd) q[d] = q[d] + 1 == h[d] ? 0 : q[d] + 1;
    if (dir < 0 && !odd) q[d] = q[d] == 0 ? h[d] - 1 : q[d] - 1;
    b = (b & ~7) | (sub ^ (1 << d));
    i = (q[2] * g.hy + q[1]) * g.hx + q[0];
}

__device__ __forceinline__ M3 load_link(const double2 *__restrict__ U, const SubGeom &g, int b, int i, int d)
{
    M3 m;
    const double2 *p = U + ((int64_t)b * 3 + d) * 9 * g.Ps + i;
#pragma unroll
    for (int k = 0; k < 9; ++k) m.e[k] = p[(int64_t)k * g.Ps];
    return m;
}

// One thread per (block, site, direction mu).
__global__ void __launch_bounds__(128) k_ape_step(const double2 *__restrict__ U, double2 *__restrict__ out, SubGeom g,
                                                  int64_t total, double a, int *err)
{
    const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= total) return;
    const int i = (int)(idx % g.Vs);
    const int64_t r = idx / g.Vs;
    const int mu = (int)(r % 3);
    const int b = (int)(r / 3);
    M3 st;
#pragma unroll
    for (int k = 0; k < 9; ++k) st.e[k] = make_double2(0.0, 0.0);
    for (int nu = 0; nu < 3; ++nu) {
        if (nu == mu) continue;
        // forward staple U_nu(x) U_mu(x+nu) U_nu(x+mu)^dag
        int bn = b, in_ = i, bm = b, im = i;
        step1(g, bn, in_, nu, +1);
        step1(g, bm, im, mu, +1);
        st = mul_add(mul(load_link(U, g, b, i, nu), load_link(U, g, bn, in_, mu)), dag(load_link(U, g, bm, im, nu)), st);
        // backward staple U_nu(x-nu)^dag U_mu(x-nu) U_nu(x-nu+mu)
        int bb = b, ib = i;
        step1(g, bb, ib, nu, -1);
        int bd = bb, id = ib;
        step1(g, bd, id, mu, +1);
        st = mul_add(mul(dag(load_link(U, g, bb, ib, nu)), load_link(U, g, bb, ib, mu)), load_link(U, g, bd, id, nu), st);
    }
    const M3 u = load_link(U, g, b, i, mu);
    M3 v;
#pragma unroll
    for (int k = 0; k < 9; ++k)
        v.e[k] = make_double2(fma(1.0 - a, u.e[k].x, 0.25 * a * st.e[k].x), fma(1.0 - a, u.e[k].y, 0.25 * a * st.e[k].y));
    const bool ok = project_su3(v);
    if (!ok) atomicOr(err, DERR_PROJECT);
    const M3 &w = ok ? v : u;
    double2 *p = out + ((int64_t)b * 3 + mu) * 9 * g.Ps + i;
#pragma unroll
    for (int k = 0; k < 9; ++k) p[(int64_t)k * g.Ps] = w.e[k];
}

}  // namespace

cudaError_t launch_ape_step(const double *U, double *out, const SubGeom &g, int nblk, double a, int *err,
                            cudaStream_t s)
{
    const int64_t total = (int64_t)nblk * 3 * g.Vs;
    const unsigned nb = (unsigned)((total + 127) / 128);
    k_ape_step<<<nb, 128, 0, s>>>(reinterpret_cast<const double2 *>(U), reinterpret_cast<double2 *>(out), g, total, a,
                                  err);
    return cudaGetLastError();
}

}  // namespace tls
