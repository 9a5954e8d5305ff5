// k_col.cuh -- multi-RHS smearing step marching along z' through a TMA-fed ring.
//
// The step of Sec. 2 (Eq. tlSmear with Eq. tlLapl1) on the grouped interleaved
// layout: the vectors are split into groups of nvg (even), each group an
// interleaved field of its own (VRec), one behind the other.  The per-vector
// FMA sequence is that of site_step: results are bitwise equal to every other
// kernel of the library.
//
// Work decomposition: a tile is ny whole x'-rows of one (slice, sublattice)
// block and one vector group, marched through a segment of z'-planes; a
// consumer thread owns one vector pair of one (x', y') column and keeps
// psi(z'-1), psi(z') and psi(z'+1) of its column in registers.  One producer
// warp streams planes into a ring of shared-memory units, completion counted on
// one mbarrier per unit; consumer warps hand a unit back through a second one.
// Records are laid out row by row (colour planes inside a row), so that the rows
// of a unit are one to three plain bulk copies; the 16-byte planes of the W rows
// come as boxes of a tensor map.  Few copies per unit matter: issuing one costs
// the producer about 120 cycles, and with one copy per colour and W plane (29
// per unit) the producer, not the memory, set the time of the kernel.
// No CTA barrier runs after the start, CTAs are persistent (tile after tile,
// the ring never drains), and the next unit is in flight while one is used.
//
// Unit u of a tile carries the records of plane z0 + u + 1 (rows y0 - 1 ..
// y0 + ny, halo rows included; the first and the last of a segment need no
// halo) and the W rows of plane z0 + u; plane k uses unit k (W of the plane,
// psi(k+1)) and unit k - 1 (psi of the plane's x and y neighbours, W_z(k-1)).
//
// HOP: the one-link step on whole slices (slice_geom), in which its hops are +-1 steps too.
//
// Every wait is bounded: one that runs out sets DERR_TIMEOUT and the CTA's
// abort flag; the producer then waits (bounded) for its copies in flight
// before the CTA ends.
#pragma once

#include <cuda.h>

#include "col_plan.h"
#include "k_ilt.cuh"

namespace tls {

// The matrix at q (16-byte planes n sites apart) with its remainder at r.
template <int WF> __device__ __forceinline__ void col_w(const char *q, int n, const char *r, cpx<float> m[9])
{
    if constexpr (WF == W_F32_18) {
        const float4 *p = reinterpret_cast<const float4 *>(q);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const float4 v = p[k * n];
            m[2 * k].re = v.x; m[2 * k].im = v.y;
            m[2 * k + 1].re = v.z; m[2 * k + 1].im = v.w;
        }
        const float2 v = *reinterpret_cast<const float2 *>(r);
        m[8].re = v.x;
        m[8].im = v.y;
    } else if constexpr (wfmt_bytes(WF) % 16 == 0) {
        WFmt<WF>::load(q, n, 0, m);
    } else {
        WFmt<WF>::load_split(q, n, r, 0, m);
    }
}

// acc += W v (DAG: W^dag v) for a vector pair; lane by lane the FMA sequence of mv_add / mdv_add.
template <bool DAG>
__device__ __forceinline__ void col_hop(const cpx<float> m[9], const float2 re[3], const float2 im[3], float2 aR[3],
                                        float2 aI[3])
{
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const float2 ng = DAG ? make_float2(-re[c].x, -re[c].y) : make_float2(-im[c].x, -im[c].y);
#pragma unroll
        for (int r = 0; r < 3; ++r) {
            const cpx<float> w = DAG ? m[c * 3 + r] : m[r * 3 + c];
            const float2 wr = make_float2(w.re, w.re), wi = make_float2(w.im, w.im);
            aR[r] = __ffma2_rn(wr, re[c], aR[r]);
            aR[r] = __ffma2_rn(wi, DAG ? im[c] : ng, aR[r]);
            aI[r] = __ffma2_rn(wr, im[c], aI[r]);
            aI[r] = __ffma2_rn(wi, DAG ? ng : re[c], aI[r]);
        }
    }
}

// A pair's record in shared memory: colour planes cs bytes apart (F32) or one 32-byte record (16-bit).
template <int VP>
__device__ __forceinline__ void col_rec(const char *s, int cs, float2 re[3], float2 im[3])
{
    if constexpr (VP == P_F32) {
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const float4 q = *reinterpret_cast<const float4 *>(s + c * cs);
            re[c] = make_float2(q.x, q.y);
            im[c] = make_float2(q.z, q.w);
        }
    } else {
        VRec<VP>::template load_pairs<false>(s, 0, re, im);
    }
}

__device__ __forceinline__ bool col_wait(uint64_t *bar, unsigned parity, volatile int *abort)
{
    for (long long n = 0; !mbar_try_wait_sleep(bar, parity, 20000u);)
        if (++n > kIltWaitPolls || *abort) return false;
    return true;
}

struct ColTile {
    int grp, blk, z0, n, y0, nyl;
};

// ngrp: vector groups that have tiles (serving: those with an active slot).
__device__ __forceinline__ ColTile col_tile(int tile, int ngrp, const ColPlan &p, const SubGeom &g)
{
    ColTile t;
    t.grp = tile % ngrp;
    int r = tile / ngrp;
    const int yt = r % p.nyt;
    r /= p.nyt;
    const int seg = r % p.nseg;
    t.blk = r / p.nseg;
    t.z0 = (int)((int64_t)seg * g.hz / p.nseg);
    t.n = (int)((int64_t)(seg + 1) * g.hz / p.nseg) - t.z0;
    t.y0 = (int)((int64_t)yt * g.hy / p.nyt);
    t.nyl = (int)((int64_t)(yt + 1) * g.hy / p.nyt) - t.y0;
    return t;
}

template <int VP, int WF, bool ACT, bool HOP = false>
__global__ void __launch_bounds__(kColMaxThreads, 1)
    k_step_col(const char *__restrict__ W, const char *__restrict__ in, char *__restrict__ out,
               const float *__restrict__ alphaf, const int *__restrict__ active, SubGeom g, ColPlan p, int64_t gstride,
               int *err, const __grid_constant__ CUtensorMap mapW, const __grid_constant__ CUtensorMap mapH)
{
    static_assert(VP != P_F64, "packed FP32 pairs only");
    constexpr int WB = wfmt_bytes(WF), NQ = WB / 16, REM = WB % 16;
    constexpr int VBY = vfmt_bytes(VP);
    constexpr int UB = VP == P_F32 ? 16 : 32;  // bytes of one pair in a colour plane / record
    extern __shared__ __align__(128) unsigned char col_sm[];
    uint64_t *full = reinterpret_cast<uint64_t *>(col_sm), *empty = full + kColMaxUnits;
    volatile int *abort = reinterpret_cast<volatile int *>(col_sm + 120);
    char *recs = reinterpret_cast<char *>(col_sm) + 128;
    char *ws = recs + p.units * p.recB;
    const int hx = g.hx, hy = g.hy, hz = g.hz;
    const int rowB = hx * p.nvg * VBY;              // one row of records
    const int tid = threadIdx.x, lane = tid & 31;
    if (tid == 0) {
        for (int k = 0; k < p.units; ++k) {
            mbar_init(full + k, 1);
            mbar_init(empty + k, p.threads / 32);
        }
        *abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    // Serving: only the groups with an active slot have tiles, so that the CTAs share them evenly
    // whatever their number (skipped tile by tile, a stride of 152 CTAs over 4 groups left half the
    // CTAs without work when two groups were active).
    __shared__ int act_grp[ACT ? kColMaxGroups + 1 : 1];  // their indices, then their number
    if constexpr (ACT) {
        if (tid < 32) {
            int n = 0;
            for (int g0 = 0; g0 < p.ngrp; g0 += 32) {
                const int grp = g0 + lane;
                bool any = false;
                if (grp < p.ngrp)
                    for (int v = 0; v < p.nvg; ++v) any = any || active[grp * p.nvg + v] != 0;
                const unsigned m = __ballot_sync(0xffffffffu, any);
                if (any) act_grp[n + __popc(m & ((1u << lane) - 1u))] = grp;
                n += __popc(m);
            }
            if (lane == 0) act_grp[kColMaxGroups] = n;
        }
    }
    __syncthreads();
    grid_dep_launch();
    grid_dep_wait();
    const int ngrp = ACT ? act_grp[kColMaxGroups * ACT] : p.ngrp;
    const int ntile = ACT ? p.ntile / p.ngrp * ngrp : p.ntile;
    auto tile_at = [&](int tile) {
        ColTile t = col_tile(tile, ngrp, p, g);
        if constexpr (ACT) t.grp = act_grp[t.grp];
        return t;
    };

    if (tid >= p.threads) {
        // ---- producer warp: one copy of the unit per lane.
        // kinds: 0 main rows, 1 row y0 - 1 and 2 row y0 + ny wrapped around; 3 W_x, 4 W_y, 5 W_z boxes,
        // 6 W_y row y0 - 1; 7..10 remainders of x, y halo row, y, z.  What does not change from plane to
        // plane is worked out once per tile: the loop below is on the kernel's critical path.
        const int nb = p.w.nb;
        int kind = 99, idx = 0;
        if (lane < 3)
            kind = lane;
        else if (lane < 3 + 3 * nb) {
            kind = 3 + (lane - 3) / nb;
            idx = (lane - 3) % nb;
        } else if (lane < 4 + 3 * nb)
            kind = 6;
        else if (REM > 0 && lane < 8 + 3 * nb)
            kind = 7 + lane - (4 + 3 * nb);
        const bool rec = kind < 3, box = kind >= 3 && kind < 7, rem = kind >= 7 && kind < 99;
        const bool halo = kind == 6 || kind == 8;
        const int wdir = kind == 3 || kind == 7 ? 0 : kind == 5 || kind == 10 ? 2 : 1;
        const bool dyn = REM > 0 && (hx * REM) % 16 != 0;  // remainder rows not on 16-byte boundaries
        const uint32_t slotB = rec ? p.recB : p.wB;
        const int wof = kind == 3 ? p.w.oX : kind == 4 ? p.w.oY : kind == 5 ? p.w.oZ : kind == 6 ? p.w.oYh
                        : kind == 7 ? p.w.oRx : kind == 8 ? p.w.oRyh : kind == 9 ? p.w.oRy : p.w.oRz;
        const uint32_t dst0 = smem_addr(rec ? recs : ws + wof + idx * p.w.boxB);
        const void *map = kind == 6 ? &mapH : &mapW;
        const int64_t planeB = rec ? (int64_t)hy * rowB : (int64_t)hy * hx * REM;
        int slot = 0, issued = 0;
        unsigned phase = 1;  // empty[] parity to wait for: the first pass through the ring does not wait
        bool ok = true;
        for (int tile = blockIdx.x; tile < ntile && ok; tile += gridDim.x) {
            const ColTile t = tile_at(tile);
            const int ym = t.y0 == 0 ? hy - 1 : t.y0 - 1;
            const bool up = t.y0 > 0, dn = t.y0 + t.nyl < hy;  // halo rows next to the main rows
            const char *src0 = nullptr;
            uint32_t dst = dst0;
            unsigned n = 0;
            int x0 = 0, zc = 0;
            if (rec) {
                const int y = kind == 0 ? t.y0 - (up ? 1 : 0) : kind == 1 ? hy - 1 : 0;
                const int l = kind == 0 ? (up ? 0 : 1) : kind == 1 ? 0 : t.nyl + 1;
                const int rows = kind == 0 ? t.nyl + (up ? 1 : 0) + (dn ? 1 : 0) : (kind == 1 ? up : dn) ? 0 : 1;
                src0 = in + t.grp * gstride + (int64_t)t.blk * g.Ps * p.nvg * VBY + (int64_t)y * rowB;
                dst += l * rowB;
                n = (unsigned)(rows * rowB);
            } else if (box) {
                x0 = 2 * hx * (halo ? ym : t.y0 + idx * p.w.br);
                zc = t.blk * 3 + wdir;
                n = (unsigned)(NQ * (halo ? 1 : p.w.br) * hx * 16);
            } else if (rem) {
                src0 = W + (((int64_t)t.blk * 3 + wdir) * WB + NQ * 16) * g.Ps + (int64_t)(halo ? ym : t.y0) * hx * REM;
                n = (unsigned)((halo ? 1 : t.nyl) * hx * REM);
            }
            unsigned total = __reduce_add_sync(0xffffffffu, n);
            for (int u = -2; u < t.n; ++u) {
                if (issued >= p.units) {
                    ok = col_wait(empty + slot, phase, abort);
                    ok = __all_sync(0xffffffffu, ok);
                    if (!ok) break;
                }
                int z = t.z0 + u + (rec ? 1 : 0);  // records run one plane ahead of W
                z = z < 0 ? z + hz : z >= hz ? z - hz : z;
                const char *src = src0 + z * planeB;
                unsigned m = rec || u >= 0 || (u == -1 && wdir == 2) ? n : 0u;
                unsigned bytes = total;
                if (dyn || u < 0) {
                    if (REM > 0 && rem && m) {  // from the 16-byte boundary at or before the first site
                        const unsigned mis = (unsigned)reinterpret_cast<uintptr_t>(src) & 15u;
                        src -= mis;
                        m = (mis + m + 15u) & ~15u;
                    }
                    bytes = __reduce_add_sync(0xffffffffu, m);
                }
                if (lane == 0) mbar_expect_tx(full + slot, bytes);
                __syncwarp();
                if (m) {
                    const uint32_t d = dst + slot * slotB;
                    if (box)
                        tensor_load_3d(d, map, x0 + z * (2 * hx * hy), 0, zc, full + slot);
                    else
                        bulk_load_s(d, src, m, full + slot);
                }
                ++issued;
                if (++slot == p.units) {
                    slot = 0;
                    phase ^= 1;
                }
            }
        }
        if (!ok) {  // the copies in flight land before the shared memory is given back
            if (lane == 0) atomicOr(err, DERR_TIMEOUT);
            *abort = 1;
            for (int q = max(0, issued - p.units); q < issued; ++q) ilt_wait(full + q % p.units, (q / p.units) & 1);
        }
        return;
    }

    // ---- consumers: one vector pair of one column
    const int T = p.nvg / 2;
    const int tp = tid % T, sl = tid / T;
    const int yl = sl / hx, xl = sl - yl * hx;
    const int xp = xl == hx - 1 ? 0 : xl + 1, xm = xl == 0 ? hx - 1 : xl - 1;
    const int sb = T * UB;                  // one site of one colour
    const int cs = hx * sb;                 // one colour of a row
    const int oC = (yl + 1) * rowB + xl * sb + tp * UB;
    const int dXp = (xp - xl) * sb, dXm = (xm - xl) * sb;
    // this thread's matrices in a unit: 16-byte planes (pn sites apart) and remainders
    const int pn = p.w.br * hx;
    const int wo = yl / p.w.br * p.w.boxB + (yl % p.w.br * hx + xl) * 16;
    const int ylm = max(yl - 1, 0);
    const int oWx = p.w.oX + wo, oWxm = oWx + (xm - xl) * 16, oWy = p.w.oY + wo, oWz = p.w.oZ + wo;
    const int wyb = yl == 0 ? p.w.oYh + xl * 16 : p.w.oY + ylm / p.w.br * p.w.boxB + (ylm % p.w.br * hx + xl) * 16;
    const int pnb = yl == 0 ? hx : pn;
    const int oRx = p.w.oRx + sl * REM, oRxm = oRx + (xm - xl) * REM, oRy = p.w.oRy + sl * REM, oRz = p.w.oRz + sl * REM;
    const int oRyb = yl == 0 ? p.w.oRyh + xl * REM : oRy - hx * REM;
    const bool dyn = REM > 0 && (hx * REM) % 16 != 0;  // remainder rows not on 16-byte boundaries
    int slot = 0;      // unit in use
    unsigned phase = 0;
    auto acquire = [&]() -> bool {
        const bool ok = col_wait(full + slot, phase, abort);
        if (__all_sync(0xffffffffu, ok)) return true;
        if (lane == 0) atomicOr(err, DERR_TIMEOUT);
        *abort = 1;
        return false;
    };
    auto release = [&](int s) {
        __syncwarp();
        if (lane == 0) mbar_arrive(empty + s);
    };
    auto next = [&]() {
        if (++slot == p.units) {
            slot = 0;
            phase ^= 1;
        }
    };
    for (int tile = blockIdx.x; tile < ntile; tile += gridDim.x) {
        const ColTile t = tile_at(tile);
        const bool mine = yl < t.nyl;
        const int v = t.grp * p.nvg + 2 * tp;
        const float2 a2 = *reinterpret_cast<const float2 *>(alphaf + v);
        const bool on0 = !ACT || active[v] != 0, on1 = !ACT || active[v + 1] != 0;
        // psi of the thread's column in planes k - 1, k, k + 1: three register sets whose roles rotate
        float2 pR[3][3], pI[3][3];
        if (!acquire()) return;
        if (mine) col_rec<VP>(recs + slot * p.recB + oC, cs, pR[0], pI[0]);
        release(slot);
        next();
        if (!acquire()) return;
        if (mine) col_rec<VP>(recs + slot * p.recB + oC, cs, pR[1], pI[1]);
        int prev = slot;
        next();
        // the thread's record of the first plane of the tile
        char *so = out + t.grp * gstride + (int64_t)t.blk * g.Ps * p.nvg * VBY + (int64_t)(t.z0 * hy + t.y0 + yl) * rowB +
                   xl * sb + tp * UB;
        int site = (t.z0 * hy + t.y0) * hx;  // first site of the tile's plane
        const int ym = t.y0 == 0 ? hy - 1 : t.y0 - 1;
        int mz = dyn ? (((t.z0 == 0 ? hz - 1 : t.z0 - 1) * hy + t.y0) * hx * REM) & 15 : 0;
        auto plane = [&](const float2 (&zmR)[3], const float2 (&zmI)[3], const float2 (&cR)[3],
                         const float2 (&cI)[3], float2 (&zpR)[3], float2 (&zpI)[3]) -> bool {
            if (!acquire()) return false;
            if (mine) {
                const char *rc = recs + prev * p.recB + oC, *rn = recs + slot * p.recB + oC;
                const char *wc = ws + slot * p.wB, *wp = ws + prev * p.wB;
                int mx = 0, mh = 0;  // misalignment of the remainder pieces of this plane
                if (dyn) {
                    mx = (site * REM) & 15;
                    mh = ((site + (ym - t.y0) * hx) * REM) & 15;
                }
                float2 aR[3], aI[3], re[3], im[3];
#pragma unroll
                for (int r = 0; r < 3; ++r) aR[r] = aI[r] = make_float2(0.f, 0.f);
                cpx<float> m[9];
                col_rec<VP>(rc + dXp, cs, re, im);
                col_w<WF>(wc + oWx, pn, wc + oRx + mx, m);
                if constexpr (VP == P_F32) {
                    // a hop's operands are requested before the hop before it is applied (48^3 x 32, 24
                    // vectors: 0.925 -> 0.919 ms; 16-bit records lose by it, 1.037 -> 1.077)
                    float2 nr[3], ni[3];
                    cpx<float> n[9];
                    col_rec<VP>(rc + dXm, cs, nr, ni);
                    col_w<WF>(wc + oWxm, pn, wc + oRxm + mx, n);
                    col_hop<false>(m, re, im, aR, aI);
                    col_rec<VP>(rc + rowB, cs, re, im);
                    col_w<WF>(wc + oWy, pn, wc + oRy + mx, m);
                    col_hop<true>(n, nr, ni, aR, aI);
                    col_rec<VP>(rc - rowB, cs, nr, ni);
                    col_w<WF>(wc + wyb, pnb, wc + oRyb + (yl == 0 ? mh : mx), n);
                    col_hop<false>(m, re, im, aR, aI);
                    col_rec<VP>(rn, cs, zpR, zpI);
                    col_w<WF>(wc + oWz, pn, wc + oRz + mx, m);
                    col_hop<true>(n, nr, ni, aR, aI);
                } else {
                    col_hop<false>(m, re, im, aR, aI);
                    col_rec<VP>(rc + dXm, cs, re, im);
                    col_w<WF>(wc + oWxm, pn, wc + oRxm + mx, m);
                    col_hop<true>(m, re, im, aR, aI);
                    col_rec<VP>(rc + rowB, cs, re, im);
                    col_w<WF>(wc + oWy, pn, wc + oRy + mx, m);
                    col_hop<false>(m, re, im, aR, aI);
                    col_rec<VP>(rc - rowB, cs, re, im);
                    col_w<WF>(wc + wyb, pnb, wc + oRyb + (yl == 0 ? mh : mx), m);
                    col_hop<true>(m, re, im, aR, aI);
                    col_rec<VP>(rn, cs, zpR, zpI);
                    col_w<WF>(wc + oWz, pn, wc + oRz + mx, m);
                }
                col_hop<false>(m, zpR, zpI, aR, aI);
                col_w<WF>(wp + oWz, pn, wp + oRz + mz, m);
                col_hop<true>(m, zmR, zmI, aR, aI);
                mz = mx;
                const float2 m6 = make_float2(-6.f, -6.f);
#pragma unroll
                for (int r = 0; r < 3; ++r) {
                    re[r] = __ffma2_rn(a2, HOP ? aR[r] : __ffma2_rn(m6, cR[r], aR[r]), cR[r]);
                    im[r] = __ffma2_rn(a2, HOP ? aI[r] : __ffma2_rn(m6, cI[r], aI[r]), cI[r]);
                }
                if (on0 && on1) {
                    if constexpr (VP == P_F32) {
#pragma unroll
                        for (int c = 0; c < 3; ++c)
                            *reinterpret_cast<float4 *>(so + c * cs) = make_float4(re[c].x, re[c].y, im[c].x, im[c].y);
                    } else {
                        VRec<VP>::store_pairs(so, 0, re, im);
                    }
                } else if (on0 || on1) {
                    cpx<float> o[3];
#pragma unroll
                    for (int c = 0; c < 3; ++c) {
                        o[c].re = on0 ? re[c].x : re[c].y;
                        o[c].im = on0 ? im[c].x : im[c].y;
                    }
                    VRec<VP>::store(so, hx * p.nvg, on0 ? 0 : 1, o);
                }
            }
            release(prev);
            prev = slot;
            next();
            site += hy * hx;
            so += (int64_t)hy * rowB;
            return true;
        };
        for (int k = 0; k < t.n; k += 3) {
            if (!plane(pR[0], pI[0], pR[1], pI[1], pR[2], pI[2])) return;
            if (k + 1 >= t.n) break;
            if (!plane(pR[1], pI[1], pR[2], pI[2], pR[0], pI[0])) return;
            if (k + 2 >= t.n) break;
            if (!plane(pR[2], pI[2], pR[0], pI[0], pR[1], pI[1])) return;
        }
        release(prev);
    }
}

// Tensor map of the 16-byte W planes: [3 nblk block directions][planes][Ps sites of
// two doubles], boxes of all planes of `sites` consecutive sites.
bool col_map(CUtensorMap &m, const char *W, const SubGeom &g, int nblk, int wb, int sites);

template <int VP, int WF> cudaError_t col_launch(const StepArgs &a)
{
    if constexpr (VP == P_F64 || WF == W_F64_18) {
        return cudaErrorNotSupported;
    } else {
        if (!a.err || !a.alphaf) return cudaErrorNotSupported;
        ColPlan p{};
        if (!col_of_tile(a.g, a.nblk, a.nvec, vfmt_bytes(VP), wfmt_bytes(WF), a.tile, p)) return cudaErrorNotSupported;
        const int64_t gstride = (int64_t)a.nblk * a.g.Ps * p.nvg * vfmt_bytes(VP);
        auto kern = a.active ? k_step_col<VP, WF, true> : k_step_col<VP, WF, false>;
        if constexpr (WF == W_F32_18) {
            if (a.hop) kern = k_step_col<VP, WF, false, true>;
        }
        // always the same value: the attribute belongs to the function, other threads may launch it too
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kColMaxSmem);
        int occ = 0;
        if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, p.threads + 32, p.smem);
        if (e != cudaSuccess) return e;
        if (occ < 1) return cudaErrorNotSupported;
        CUtensorMap mw, mh;
        if (!col_map(mw, a.W, a.g, a.nblk, wfmt_bytes(WF), p.w.br * a.g.hx) ||
            !col_map(mh, a.W, a.g, a.nblk, wfmt_bytes(WF), a.g.hx))
            return cudaErrorNotSupported;
        const int grid = std::min(p.ntile, a.num_sms * occ);
        return launch_dep(a.dep, kern, dim3(grid), dim3(p.threads + 32), p.smem, a.stream, a.W, a.in, a.out, a.alphaf,
                          a.active, a.g, p, gstride, a.err, mw, mh);
    }
}

template <int VP> cudaError_t col_dispatch(const StepArgs &a)
{
    switch (a.wfmt) {
    case W_F32_18: return col_launch<VP, W_F32_18>(a);
    case W_F32_12: return col_launch<VP, W_F32_12>(a);
    case W_F32_8:
        if constexpr (VP == P_F32) return col_launch<VP, W_F32_8>(a);
        else return cudaErrorNotSupported;
    case W_F16_18:
        if constexpr (VP == P_F16) return col_launch<VP, W_F16_18>(a);
        else return cudaErrorNotSupported;
    case W_F16_12:
        if constexpr (VP == P_F16) return col_launch<VP, W_F16_12>(a);
        else return cudaErrorNotSupported;
    case W_BF16_18:
        if constexpr (VP == P_BF16) return col_launch<VP, W_BF16_18>(a);
        else return cudaErrorNotSupported;
    case W_BF16_12:
        if constexpr (VP == P_BF16) return col_launch<VP, W_BF16_12>(a);
        else return cudaErrorNotSupported;
    default: return cudaErrorNotSupported;
    }
}

}  // namespace tls
