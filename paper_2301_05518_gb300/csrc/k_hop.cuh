// k_hop.cuh -- one-link Gaussian smearing step on the interleaved layout.
//
// Sec. 2, Eq. 2-3: psi' = psi + alpha H psi with the one-link hopping operator
//   H psi(x) = sum_mu [ U_mu(x) psi(x + mu) + U_mu^dag(x - mu) psi(x - mu) ]
// (Eq. 3 with C = 1).  A +-1 hop flips bit mu of the spatial parity, so in the
// sublattice layout it reaches the record group of the neighbouring block
// (slice, sub ^ (1 << mu)); the half coordinate moves only when the source
// coordinate is odd (forward) or even (backward):
//   x + mu: block sub ^ bit, site  bit_mu(sub) ? forward(i) : i
//   x - mu: block sub ^ bit, site  bit_mu(sub) ? i : backward(i)
// The links U_mu are stored in a W-format field (rounded U, same planes).
#pragma once

#include "k_stencil.cuh"

namespace tls {

template <int VP, int WF, int VB>
__global__ void __launch_bounds__(512) k_hop_il(const char *__restrict__ L1, const char *__restrict__ in,
                                                char *__restrict__ out, const double *__restrict__ alpha,
                                                SubGeom g, int nvec)
{
    typedef typename VRec<VP>::R R;
    constexpr int WB = wfmt_bytes(WF);
    constexpr int VBY = vfmt_bytes(VP);
    const int t = threadIdx.x, T = nvec / VB;
    const int xq = blockIdx.x * blockDim.y + threadIdx.y;
    if (xq >= g.hx) return;
    const int yq = blockIdx.y;
    const int blk = blockIdx.z / g.hz;
    const int zq = blockIdx.z - blk * g.hz;
    const int sub = blk & 7, bt = blk & ~7;
    const int sy = g.hx, sz = g.hx * g.hy;
    const int i = zq * sz + yq * sy + xq;
    int fw[3], bw[3];
    fw[0] = xq == g.hx - 1 ? i - (g.hx - 1) : i + 1;
    bw[0] = xq == 0 ? i + (g.hx - 1) : i - 1;
    fw[1] = yq == g.hy - 1 ? i - (g.hy - 1) * sy : i + sy;
    bw[1] = yq == 0 ? i + (g.hy - 1) * sy : i - sy;
    fw[2] = zq == g.hz - 1 ? i - (g.hz - 1) * sz : i + sz;
    bw[2] = zq == 0 ? i + (g.hz - 1) * sz : i - sz;
    const unsigned rstride = (unsigned)nvec * VRec<VP>::SB;  // site stride
    const int cs = g.Ps * nvec;                                    // colour planes
    auto recs = [&](int b) { return in + (int64_t)b * g.Ps * nvec * VBY; };
    auto links = [&](int b, int d) { return L1 + ((int64_t)b * 3 + d) * g.Ps * WB; };
    cpx<R> acc[VB][3];
#pragma unroll
    for (int k = 0; k < VB; ++k)
#pragma unroll
        for (int c = 0; c < 3; ++c) acc[k][c].re = acc[k][c].im = R(0);
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        const int odd = (sub >> d) & 1;
        const int nb = bt | (sub ^ (1 << d));
        const int i_f = odd ? fw[d] : i;
        const int i_b = odd ? i : bw[d];
        cpx<R> m[9], p[VB][3];
        WFmt<WF>::load(links(blk, d), g.Ps, i, m);
        RecGroup<VP, VB>::load(recs(nb) + (unsigned)i_f * rstride, cs, t, T, p);
#pragma unroll
        for (int k = 0; k < VB; ++k) mv_add(m, p[k], acc[k]);
        WFmt<WF>::load(links(nb, d), g.Ps, i_b, m);
        RecGroup<VP, VB>::load(recs(nb) + (unsigned)i_b * rstride, cs, t, T, p);
#pragma unroll
        for (int k = 0; k < VB; ++k) mdv_add(m, p[k], acc[k]);
    }
    cpx<R> c[VB][3], o[VB][3];
    RecGroup<VP, VB>::load(recs(blk) + (unsigned)i * rstride, cs, t, T, c);
#pragma unroll
    for (int k = 0; k < VB; ++k) {
        const R a = (R)alpha[il_vec<VP, VB>(t, T, k)];
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            o[k][q].re = fma(a, acc[k][q].re, c[k][q].re);
            o[k][q].im = fma(a, acc[k][q].im, c[k][q].im);
        }
    }
    RecGroup<VP, VB>::store(out + (int64_t)blk * g.Ps * nvec * VBY + (unsigned)i * rstride, cs, t, T, o);
}

template <int VP, int WF, int VB> cudaError_t hop_launch(const StepArgs &a)
{
    const int tx = a.nvec / VB;
    const int spb = il_spb(tx, a.threads);
    dim3 block(tx, spb);
    dim3 grid((a.g.hx + spb - 1) / spb, a.g.hy, (unsigned)a.g.hz * a.nblk);
    if (grid.y > 65535 || grid.z > 65535) return cudaErrorInvalidConfiguration;
    k_hop_il<VP, WF, VB><<<grid, block, 0, a.stream>>>(a.W, a.in, a.out, a.alpha, a.g, a.nvec);
    return cudaGetLastError();
}

// --------------------------------------------------------------------------
// The same step with vector-pair arithmetic and TMA-staged links (FP32 and
// 16-bit storage; bitwise equal to k_hop_il).  One CTA per whole x'-row and
// group of vectors, as the two-link row kernel (k_ilt.cuh): the leader copies
// the six link rows the row needs (U_mu of the row itself and of the rows one
// step back, which lie in the neighbouring blocks) into shared memory with
// cp.async.bulk, the remainder plane from the 16-byte boundary at or before
// the row, so that rows of any length take this path.  Each thread takes NP
// vector pairs at one x' and requests its first records before the wait.
// Bound by the latency of the record loads and the L1 pipe, like the two-link
// row kernel; k_hop_il spent its time on scalar FMAs and on loading every link
// once per thread (32^3 x 64, 12 FP32 vectors: 1.22 ms per step, now 0.38).
// --------------------------------------------------------------------------

// Shared-memory bytes of one link row: 16-byte planes, then the remainder with room for its alignment.
__host__ __device__ inline int hop_row_bytes(int hx) { return 4 * hx * 16 + (hx * 8 + 15) / 16 * 16 + 16; }

// The NP vector pairs of thread t (of T per site) at site pointer s.
template <int VP, int NP>
__device__ __forceinline__ void hop_load(const char *s, int cs, int t, int T, float2 re[NP][3], float2 im[NP][3])
{
    if constexpr (VP != P_F32) {
#pragma unroll
        for (int j = 0; j < NP; ++j) VRec<VP>::load_pairs(s, t + j * T, re[j], im[j]);
    } else if constexpr (NP == 2) {
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            float2 r2[2], i2[2];
            VRec<P_F32>::load4g_pairs(s, cs, t, c, r2, i2);
            re[0][c] = r2[0];
            re[1][c] = r2[1];
            im[0][c] = i2[0];
            im[1][c] = i2[1];
        }
    } else {
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const float4 q = reinterpret_cast<const float4 *>(s)[t + (int64_t)c * (cs >> 1)];
            re[0][c] = make_float2(q.x, q.y);
            im[0][c] = make_float2(q.z, q.w);
        }
    }
}

template <int VP, int NP>
__global__ void __launch_bounds__(256, 3) k_hop_rows(const char *__restrict__ L1, const char *__restrict__ in,
                                                     char *__restrict__ out, const float *__restrict__ alphaf, SubGeom g,
                                                     int nvec, int *err)
{
    constexpr int WB = wfmt_bytes(W_F32_18), VBY = vfmt_bytes(VP);
    extern __shared__ __align__(128) unsigned char hop_sm[];
    __shared__ int w_ok;
    uint64_t *bar = reinterpret_cast<uint64_t *>(hop_sm);
    char *ws = reinterpret_cast<char *>(hop_sm) + 128;
    const int hx = g.hx, rowB = hop_row_bytes(hx);
    const int yq = blockIdx.y;
    // the eight sublattices of a plane one after another: the neighbouring blocks' rows are
    // read while they are in L2 (a slice of 24 vectors at 48^3 does not stay there whole)
    const int sub = blockIdx.z & 7, zt = blockIdx.z >> 3;
    const int blk = zt / g.hz * 8 + sub, zq = zt % g.hz;
    const int k = threadIdx.y, t = blockIdx.x * blockDim.x + threadIdx.x, T = nvec / (2 * NP);
    const int sy = hx, sz = hx * g.hy;
    const int row = zq * sz + yq * sy, i = row + k;
    const bool ox = sub & 1, oy = (sub >> 1) & 1, oz = (sub >> 2) & 1;
    const int yp = yq == g.hy - 1 ? 0 : yq + 1, ym = yq == 0 ? g.hy - 1 : yq - 1;
    const int zp = zq == g.hz - 1 ? 0 : zq + 1, zm = zq == 0 ? g.hz - 1 : zq - 1;
    const int km = k == 0 ? hx - 1 : k - 1;
    // rows (first sites) of the backward links: x, y, z
    const int rbx = row, rby = zq * sz + (oy ? yq : ym) * sy, rbz = (oz ? zq : zm) * sz + yq * sy;
    const bool leader = threadIdx.x == 0 && threadIdx.y == 0;
    if (leader) {
        mbar_init(bar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        unsigned total = 0;
#pragma unroll
        for (int q = 0; q < 6; ++q) {
            const int r = q == 1 ? rbx : q == 3 ? rby : q == 5 ? rbz : row;
            total += (unsigned)(4 * hx * 16 + ((((r * 8) & 15) + hx * 8 + 15) & ~15));
        }
        mbar_expect_tx(bar, total);
#pragma unroll
        for (int q = 0; q < 6; ++q) {
            const int d = q >> 1, r = q == 1 ? rbx : q == 3 ? rby : q == 5 ? rbz : row;
            const int b = q & 1 ? blk ^ (1 << d) : blk;
            const char *src = L1 + ((int64_t)b * 3 + d) * g.Ps * WB;
            char *dst = ws + q * rowB;
#pragma unroll
            for (int j = 0; j < 4; ++j)
                bulk_load(dst + j * hx * 16, src + ((int64_t)j * g.Ps + r) * 16, (unsigned)(hx * 16), bar);
            const int mis = (r * 8) & 15;
            bulk_load(dst + 4 * hx * 16, src + 4 * g.Ps * 16 + (int64_t)r * 8 - mis, (unsigned)((mis + hx * 8 + 15) & ~15),
                      bar);
        }
    }
    grid_dep_launch();
    grid_dep_wait();  // the links do not change between steps, the records do
    const int64_t blkB = g.Ps * nvec * VBY;
    const unsigned rstride = (unsigned)nvec * VRec<VP>::SB;  // site stride
    const int cs = g.Ps * nvec;                              // colour planes
    auto src = [&](int q) {  // records of hop q
        const int d = q >> 1;
        int s;
        if (q == 0) s = ox ? (k == hx - 1 ? row : i + 1) : i;
        else if (q == 1) s = ox ? i : row + km;
        else if (q == 2) s = oy ? zq * sz + yp * sy + k : i;
        else if (q == 3) s = rby + k;
        else if (q == 4) s = oz ? zp * sz + yq * sy + k : i;
        else s = rbz + k;
        return in + (int64_t)(blk ^ (1 << d)) * blkB + (unsigned)s * (int64_t)rstride;
    };
    float2 re[NP][3], im[NP][3], aR[NP][3], aI[NP][3];
    hop_load<VP, NP>(src(0), cs, t, T, re, im);
#pragma unroll
    for (int j = 0; j < NP; ++j)
#pragma unroll
        for (int r = 0; r < 3; ++r) aR[j][r] = aI[j][r] = make_float2(0.f, 0.f);
    // The leader waits for the copies; on a timeout it waits once more (bounded), so that the CTA
    // does not retire while its copies are in flight.
    if (leader) {
        const bool okw = ilt_wait(bar, 0u);
        w_ok = okw;
        if (!okw) {
            atomicOr(err, DERR_TIMEOUT);
            ilt_wait(bar, 0u);
        }
    }
    __syncthreads();
    if (!w_ok) return;
#pragma unroll
    for (int q = 0; q < 6; ++q) {
        if (q > 0) hop_load<VP, NP>(src(q), cs, t, T, re, im);
        const bool dag = q & 1;
        const char *w = ws + q * rowB;
        const int r = q == 1 ? rbx : q == 3 ? rby : q == 5 ? rbz : row;
        const int wk = q == 1 && !ox ? km : k;
        const float2 *last = reinterpret_cast<const float2 *>(w + 4 * hx * 16 + ((r * 8) & 15));
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            float2 ng[NP];
#pragma unroll
            for (int j = 0; j < NP; ++j)
                ng[j] = dag ? make_float2(-re[j][c].x, -re[j][c].y) : make_float2(-im[j][c].x, -im[j][c].y);
#pragma unroll
            for (int rr = 0; rr < 3; ++rr) {
                const int e = dag ? c * 3 + rr : rr * 3 + c;
                const float2 f = e < 8 ? reinterpret_cast<const float2 *>(w)[((e >> 1) * hx + wk) * 2 + (e & 1)] : last[wk];
                const float2 wr = make_float2(f.x, f.x), wi = make_float2(f.y, f.y);
#pragma unroll
                for (int j = 0; j < NP; ++j) {
                    aR[j][rr] = __ffma2_rn(wr, re[j][c], aR[j][rr]);
                    aR[j][rr] = __ffma2_rn(wi, dag ? im[j][c] : ng[j], aR[j][rr]);
                    aI[j][rr] = __ffma2_rn(wr, im[j][c], aI[j][rr]);
                    aI[j][rr] = __ffma2_rn(wi, dag ? ng[j] : re[j][c], aI[j][rr]);
                }
            }
        }
    }
    hop_load<VP, NP>(in + (int64_t)blk * blkB + (unsigned)i * (int64_t)rstride, cs, t, T, re, im);
    char *so = out + (int64_t)blk * blkB + (unsigned)i * (int64_t)rstride;
#pragma unroll
    for (int j = 0; j < NP; ++j) {
        // pair j of the thread: F32 threads own adjacent pairs, 16-bit ones pairs T apart
        const int u = VP == P_F32 ? NP * t + j : t + j * T;
        const float2 a2 = *reinterpret_cast<const float2 *>(alphaf + 2 * u);
#pragma unroll
        for (int r = 0; r < 3; ++r) {
            re[j][r] = __ffma2_rn(a2, aR[j][r], re[j][r]);
            im[j][r] = __ffma2_rn(a2, aI[j][r], im[j][r]);
        }
        if constexpr (VP != P_F32) VRec<VP>::store_pairs(so, u, re[j], im[j]);
    }
    if constexpr (VP == P_F32) {
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            if constexpr (NP == 2) {
                const float2 r2[2] = {re[0][c], re[1][c]}, i2[2] = {im[0][c], im[1][c]};
                VRec<P_F32>::store4g_pairs(so, cs, t, c, r2, i2);
            } else {
                reinterpret_cast<float4 *>(so)[t + (int64_t)c * (cs >> 1)] =
                    make_float4(re[0][c].x, re[0][c].y, im[0][c].x, im[0][c].y);
            }
        }
    }
}

// cudaErrorNotSupported: no CTA shape (rows longer than 256 sites).
template <int VP, int NP> cudaError_t hop_rows_launch(const StepArgs &a)
{
    const int nvg = ilt_group(a.nvec, 2 * NP, a.g.hx, 0);
    const int smem = 128 + 6 * hop_row_bytes(a.g.hx);
    if (!a.err || !a.alphaf || nvg == 0 || smem > (48 << 10)) return cudaErrorNotSupported;
    dim3 block(nvg / (2 * NP), a.g.hx), grid(a.nvec / nvg, a.g.hy, (unsigned)a.g.hz * a.nblk);
    if (grid.y > 65535 || grid.z > 65535) return cudaErrorInvalidConfiguration;
    return launch_dep(a.dep, k_hop_rows<VP, NP>, grid, block, smem, a.stream, a.W, a.in, a.out, a.alphaf, a.g, a.nvec,
                      a.err);
}

// Link fields are FP64-18 for FP64 vectors and FP32-18 otherwise.
template <int VP> cudaError_t hop_dispatch(const StepArgs &a)
{
    constexpr int WF = VP == P_F64 ? W_F64_18 : W_F32_18;
    if (a.wfmt != WF) return cudaErrorNotSupported;
    if (a.nvec < 1 || a.nvec > 256) return cudaErrorInvalidValue;
    if constexpr (VP != P_F64) {
        // FP32 and 16-bit records come in pairs: a.nvec is even.  Two pairs per thread where the
        // rows then still fill a warp (as row_tile, measured on the two-link rows)
        const bool two = a.nvec % 4 == 0 && a.nvec / 4 * a.g.hx >= (VP == P_F32 ? 20 : 64);
        const cudaError_t e = two ? hop_rows_launch<VP, 2>(a) : hop_rows_launch<VP, 1>(a);
        if (e != cudaErrorNotSupported) return e;
    }
    const int vb = (a.vb == 2 && a.nvec % 2 == 0) ? 2 : 1;
    if (vb == 2) return hop_launch<VP, WF, 2>(a);
    return hop_launch<VP, WF, 1>(a);
}

}  // namespace tls
