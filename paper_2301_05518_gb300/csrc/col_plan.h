// col_plan.h -- tile shapes and shared-memory geometry of the column kernel (k_col.cuh).
#pragma once

#include <stdint.h>

#include <algorithm>
#include <cmath>

#include "tls_types.h"

namespace tls {

constexpr int kColMaxUnits = 6;
constexpr int kColMaxSmem = 226 * 1024;  // of 227 KB, beside the serving form's list of groups
constexpr int kColMaxGroups = 128;   // vector groups: at most 256 vectors in pairs
constexpr int kColMaxThreads = 512;  // consumers and the producer warp: 16 warps of 128 registers

TLS_HD inline int up16(int n) { return (n + 15) & ~15; }

// W rows of a unit, wb bytes per matrix.  The 16-byte words come as boxes of all
// planes of br rows (one tensor copy each): nb boxes for the ny rows of W_x, of
// W_y and of W_z, and a one-row box for row y0 - 1 of W_y.  The remainder planes
// come as four plain pieces (x; y halo row; y; z), each with 16 spare bytes for
// its alignment.
struct ColW {
    int br, nb;                   // rows per box, boxes per direction
    int boxB, haloB;              // their shared-memory bytes (128-byte aligned)
    int oX, oYh, oY, oZ;          // box offsets in the unit
    int oRx, oRyh, oRy, oRz;      // remainder pieces
    int bytes;
};

inline ColW col_w_plan(int wb, int hx, int ny)
{
    auto up = [](int n) { return (n + 127) & ~127; };
    const int nq = wb / 16, rem = wb % 16;
    ColW w{};
    w.br = 1;
    for (int r = 2; r <= ny; ++r)
        if (ny % r == 0 && r * hx * 2 <= 256) w.br = r;  // a box row holds at most 256 doubles
    w.nb = ny / w.br;
    w.boxB = up(nq * w.br * hx * 16);
    w.haloB = up(nq * hx * 16);
    w.oX = 0;
    w.oYh = w.nb * w.boxB;
    w.oY = w.oYh + w.haloB;
    w.oZ = w.oY + w.nb * w.boxB;
    w.oRx = w.oZ + w.nb * w.boxB;
    const int p = rem ? up16(ny * hx * rem) + 16 : 0, h = rem ? up16(hx * rem) + 16 : 0;
    w.oRyh = w.oRx + p;
    w.oRy = w.oRyh + h;
    w.oRz = w.oRy + p;
    w.bytes = up(w.oRz + p);
    return w;
}

// Shared-memory geometry of one tile shape (bytes).
struct ColPlan {
    int nvg, ny, nseg, threads;  // vectors per group, rows per tile, z' segments, consumer threads (whole warps)
    int ngrp, nyt, ntile;
    int units;                   // ring units
    int recB, wB, smem;          // one unit's records, one unit's W rows, the CTA's total
    ColW w;
};

inline int col_smem(const ColPlan &p) { return 128 + p.units * (p.recB + p.wB); }

// The tile shape: nvg vectors per group, ny rows, nseg segments, at most `units` ring units (0: as
// many as fit).  False: no fit.  Fewer than three units are no ring: a consumer keeps the unit
// before the one it waits for, and the producer runs one further.
// w: col_w_plan of the tile's rows, if the caller has it.
inline bool col_shape(const SubGeom &g, int nblk, int nvec, int vby, int wb, int nvg, int ny, int nseg, int units,
                      ColPlan &out, const ColW *w = nullptr)
{
    ColPlan p{};
    if (nvg < 2 || (nvg & 1) || ny < 1 || ny > g.hy || nseg < 1 || nseg > g.hz) return false;
    if (units != 0 && units < 3) return false;
    if (ny > 255) return false;  // a tune entry holds the rows in eight bits
    p.nvg = nvg;
    p.ngrp = (nvec + nvg - 1) / nvg;
    if (p.ngrp > kColMaxGroups) return false;
    p.nyt = (g.hy + ny - 1) / ny;
    p.ny = (g.hy + p.nyt - 1) / p.nyt;
    p.nseg = nseg;
    const int64_t act = (int64_t)(nvg / 2) * p.ny * g.hx;
    if (act > kColMaxThreads - 32) return false;
    p.threads = (int)((act + 31) / 32 * 32);
    const int64_t recB = (int64_t)(p.ny + 2) * g.hx * nvg * vby;
    p.recB = (int)((recB + 127) / 128 * 128);
    p.w = w ? *w : col_w_plan(wb, g.hx, p.ny);
    p.wB = p.w.bytes;
    if (g.hx > 128 || p.w.nb > 8) return false;
    p.units = (int)((kColMaxSmem - 128) / (p.recB + p.wB));
    if (p.units < 3) return false;
    p.units = std::min(p.units, units ? std::min(units, kColMaxUnits) : kColMaxUnits);
    p.smem = col_smem(p);
    const int64_t nt = (int64_t)p.ngrp * p.nyt * nseg * nblk;
    if (nt > 0x7fffffff) return false;
    p.ntile = (int)nt;
    out = p;
    return true;
}

// Estimated time of one step (us) of the column kernel with tile shape p, fitted to
// 1100 measured (lattice, vectors, shape) points on a GB300 (within 10 % for most;
// the shape it picks is within 5 % of the best one measured, except on lattices
// whose step takes a few launches' time anyway).  A unit of the busiest SM takes the
// largest of: the arithmetic, 356 + 650 w cycles for w consumer warps on one
// scheduler; the copies, 36.5 bytes per cycle; and, with d units in flight, 1/d of
// a copy's latency of 2350 cycles plus its transfer.  A tile of n planes takes n + 2
// units; the whole cannot beat the memory.  A thread rebuilds W for one vector pair
// only, so W formats that need arithmetic cost it more than the row kernel; groups of
// two or four vectors measured about an eighth above the fit.  A shape that its largest term alone
// puts at `limit` or above gets that as its estimate.
inline double col_estimate(const ColPlan &p, const SubGeom &g, int nblk, int vby, int wb, int num_sms, double limit)
{
    const int warps = p.threads / 32;
    int occ = 1;
    while ((occ + 1) * (warps + 1) <= 16 && (occ + 1) * (p.smem + 1024) <= 228 * 1024) ++occ;
    const int eff = std::min(occ, (p.ntile + num_sms - 1) / num_sms);
    const double rounds = (p.ntile + num_sms * eff - 1) / (num_sms * eff);
    const double fmt = (wb == 72 ? 1.0 : wb == 48 || wb == 36 ? 1.15 : wb == 24 ? 1.7 : 4.0) * (p.nvg <= 4 ? 1.12 : 1.0);
    const double unit = p.recB + p.wB;
    const double comp = (356 + 650.0 * ((warps * eff + 3) / 4)) * (vby == 16 ? 1.145 : 1.0) * fmt;
    const double copy = eff * unit / 36.5, lat = (2350 + unit / 36.5) / (p.units - 2);
    const double dram = (double)nblk * g.Vs * (3.0 * wb + 2.0 * vby * p.ngrp * p.nvg) / 6.4e6;
    const double units = 1 + (rounds > 1 ? 0.005 : 0.03) * (p.units - 3);
    auto total = [&](double t) { return std::max(rounds * ((double)g.hz / p.nseg + 2) * t / 2060, dram) * units + 3.5; };
    const double low = total(std::max(std::max(comp, copy), lat));
    if (low >= limit) return low;
    auto p6 = [](double x) { return x * x * x * x * x * x; };
    return total(std::cbrt(std::sqrt(p6(comp) + p6(copy) + p6(lat))));
}

// The same for the row kernel (k_ilt.cuh): 0.03 + 0.0105 n ns per site for n vectors
// in fours (0.0125 n above 24, 0.0165 n where a row's vectors take several CTAs), 0.02 +
// 0.015 n otherwise (48^3 x 32: 3 / 5 / 12 / 24 / 72 vectors 224 / 394 / 578 / 1018 / 3510
// us; 64^3 x 24: 8 / 24 vectors 595 / 1624 us; rows of 48, 24 vectors 0.0170 n), 1.75 times that where its TMA copies do not apply (50^3 x 16, 24 vectors: 884
// us), with the arithmetic of the W formats shared by four vectors (24 vectors at
// 48^3 x 32, row / column kernel: f32-18 1018 / 927, f32-12 1103 / 1065, f32-8 1699 /
// above 2600, 16-bit vectors with f32-18 1203 / 1037, with f16-12 1393 / 1414 us).
// Rows (CTAs of the row kernel): one starts about every nanosecond (16^3 x 32: 16384 of them,
// 17.7 us per step with 3 vectors).
inline double row_ctas(const SubGeom &g, int nblk) { return (double)nblk * g.hy * g.hz; }

inline double row_estimate(const SubGeom &g, int nblk, int nvec, int vby, int wb)
{
    const int n = (nvec + 1) & ~1;
    const double fmt = wb == 48 ? 1.08 : wb == 32 ? 1.65 : wb == 24 ? 1.15 : 1.0;
    const bool split = n / 4 * g.hx > 256;  // the vectors of a row take several CTAs
    const double site = n % 4 ? 0.02 + 0.015 * n : split ? 0.0165 * n : n > 24 ? 0.0125 * n : 0.03 + 0.0105 * n;
    const bool tma = (g.hx * (wb % 16)) % 16 == 0;
    const double us = (double)nblk * g.Vs * site * 1e-3 * (tma ? 1.0 : 1.75) * (vby == 16 ? 1.2 : 1.0) * fmt;
    return std::max(us, row_ctas(g, nblk) * 1e-3) + 2;
}

// All vectors in one launch of the planar kernel, two or four a thread: reads W once, has
// no rows to keep whole, but pays for unused lanes of its four vectors (16^3 x 32, 2 / 3 / 4
// vectors: 7.0 / 11.3 / 13.9 us per step against 12.1 / 17.7 / 17.7; 48^3 x 32: 202 / 375 /
// 460 against 186 / 231 / 231; 32^3 x 16, 2 FP16 vectors with W f16-12: 27 against 47).
// A candidate for two vectors, and for up to four where the row kernel is bound by starting
// its CTAs.  Not for the 8-real W, whose reconstruction rounds differently there.
inline bool planar_ok(const SubGeom &g, int nblk, int nvec, int wb)
{
    return wb != 32 && (nvec == 2 || (nvec > 2 && nvec <= 4 && row_ctas(g, nblk) > 8000));
}

inline double planar_estimate(const SubGeom &g, int nblk, int nvec, int vby, int wb)
{
    const double sites = (double)nblk * g.Vs;
    const double site = nvec == 2 ? 0.06 : nvec == 3 ? 0.108 : 0.132;
    const double l2 = sites * (3.0 * wb + 2.0 * vby * nvec) < 60e6 ? 0.7 : 1.0;  // stays in L2
    return sites * site * l2 * (wb == 48 ? 1.15 : 1.0) * (vby == 16 ? 0.9 : 1.0) * 1e-3 + 2.5;
}

// The best tile shapes by that estimate, best first (at most `most`).  nvg divides
// the vectors into equal groups with at most a third of padding (exact: none).
// Runs in every call without a tune entry, before anything is enqueued: what a shape shares with
// others is worked out once and most shapes are dropped by the largest term of their estimate
// (48^3, one slice, 24 vectors 40 -> 5 us on an x86 host; 4 x 48 x 48, 72 vectors 103 -> 13).
inline int col_plans(const SubGeom &g, int nblk, int nvec, int vby, int wb, int num_sms, ColPlan *best, double *us,
                     int most, bool exact = false)
{
    int n = 0;
    const int n2 = (nvec + 1) & ~1;
    for (int last = 0, nyt = 1; nyt <= g.hy; ++nyt) {
        const int ny = (g.hy + nyt - 1) / nyt;
        if (ny == last) continue;
        last = ny;
        if ((int64_t)ny * g.hx > kColMaxThreads - 32) continue;
        const ColW w = col_w_plan(wb, g.hx, ny);
        for (int nvg = 2; nvg <= 24 && nvg <= n2; nvg += 2) {
            if ((nvec + nvg - 1) / nvg * nvg * 3 > 4 * n2 || (exact && nvec % nvg)) continue;
            ColPlan p;
            if (!col_shape(g, nblk, nvec, vby, wb, nvg, ny, 1, 0, p, &w)) continue;
            const int most_units = p.units, tiles = p.ntile;
            for (int nseg = 1; nseg <= 4 && nseg * 4 <= g.hz; nseg *= 2) {
                if ((int64_t)tiles * nseg > 0x7fffffff) break;
                p.nseg = nseg;
                p.ntile = tiles * nseg;
                for (int units : {most_units, 3}) {  // three: more CTAs per SM
                    p.units = units;
                    p.smem = col_smem(p);
                    const double limit = n < most ? 1e300 : us[n - 1];
                    const double e = col_estimate(p, g, nblk, vby, wb, num_sms, limit);
                    if (n == most && e >= limit) continue;
                    int at = n < most ? n++ : most - 1;
                    for (; at > 0 && us[at - 1] > e; --at) {
                        best[at] = best[at - 1];
                        us[at] = us[at - 1];
                    }
                    best[at] = p;
                    us[at] = e;
                    if (most_units == 3) break;
                }
            }
        }
    }
    return n;
}

// Whether buffers of have[k] bytes can grow to need[k] under an HBM cap (0: none) with `used` bytes
// in use, the old ones counted.  Known before a buffer is given up: a call that tried the padded
// groups of the column kernel and failed freed, allocated and cleared its buffers each time.
inline bool workspace_fits(uint64_t used, uint64_t cap, int n, const uint64_t *have, const uint64_t *need)
{
    for (int k = 0; k < n; ++k)
        if (need[k] > have[k]) used += need[k] - have[k];
    return cap == 0 || used <= cap;
}

// tile[] of the tune entry for a shape: 9 selects the column kernel.
inline void col_tile_of(const ColPlan &p, int tile[3])
{
    tile[0] = p.nvg;
    tile[1] = 9;
    tile[2] = p.ny | p.nseg << 8 | p.units << 16;
}

// The shape of such an entry.  False: no fit.
inline bool col_of_tile(const SubGeom &g, int nblk, int nvec, int vby, int wb, const int tile[3], ColPlan &out)
{
    return col_shape(g, nblk, nvec, vby, wb, tile[0], tile[2] & 255, std::max(1, (tile[2] >> 8) & 255), tile[2] >> 16, out);
}

// Row kernel parameters without a tune entry: tile[], returns the vectors per thread.
// More than 24 vectors go through CTAs of 24 where that divides them (72 vectors at
// 48^3 x 24: 2.41 ms against 2.64 with 36 a CTA); rows are asked into L2 ahead (tile[2])
// where a step's data do not stay there (64^3 x 24, 24 vectors: 1.61 against 1.64 ms;
// 16^3 x 32, 2 vectors: 21 against 19 us).  Four vectors per thread where the rows then still
// fill a warp (32^3 x 64 / 48^3 x 32, 3 vectors: 16 / 24 threads, 180 / 224 us with four and
// 142 / 290 with two); 16-bit records want twice the threads (12 vectors, 48 threads: 434
// against 369 us; 24 vectors, 144 threads: 1203 against 1507).
inline int row_tile(const SubGeom &g, int nblk, int nvec, int vby, int tile[3])
{
    const int n = (nvec + 1) & ~1;
    tile[0] = n > 24 && n % 24 == 0 ? 24 : 0;
    tile[1] = 6;
    tile[2] = (double)nblk * g.Vs * (216.0 + 2.0 * vby * n) > 120e6 ? -1 : 0;
    return n % 4 == 0 && n / 4 * g.hx >= (vby == 16 ? 64 : 20) ? 4 : 2;
}

// Vectors per thread of the planar kernel when it takes several at once.
inline int planar_vb(int storage, int nvec)
{
    const int cap = storage == P_F64 ? 4 : 8;
    int vb = 2;
    while (vb < cap && vb < nvec) vb *= 2;
    return vb;
}

// Share of the lanes of a warp at work in the FP64 multi-RHS kernel (nvec threads per site, a
// strip of one row per CTA of at most 256 threads).  The FP64 pipe bounds it, so idle lanes cost
// their share, and one vector per launch, which has none, reads W more often for nothing lost
// (32^3 x 16, 3 vectors: 48 of 64 lanes, 779 us per step against 597; 4 vectors: 779 against 796).
inline double il_f64_lanes(int nvec, int hx)
{
    const int n = nvec < 256 ? nvec : 256;
    int spb = std::max(1, 256 / n);
    for (int s = spb; s >= 1; --s)
        if ((s * n) % 32 == 0) {
            spb = s;
            break;
        }
    spb = std::min(spb, hx);
    const int strips = (hx + spb - 1) / spb;  // the last one may be short, its CTA is not
    const double threads = (double)strips * ((spb * n + 31) / 32 * 32);
    return (double)hx * n / threads;
}

}  // namespace tls
