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

// Sites per CTA for the interleaved kernels: nvec * spb <= threads, with a
// whole number of warps when possible.
inline int il_spb(int nvec, int threads)
{
    if (threads <= 0) threads = 256;
    int spb = std::max(1, threads / nvec);
    for (int s = spb; s >= 1; --s)
        if ((s * nvec) % 32 == 0) return s;
    return spb;
}

// Shared-memory bytes of a CTA of the row kernel: the mbarrier (128 bytes) and the five W rows.
inline int row_smem(int hx, int wb) { return 128 + 5 * hx * wb; }
constexpr int kRowMaxSmem = 48 << 10;

// Whether its TMA staging applies: every plane segment of a W row starts and ends on a
// 16-byte boundary (the remainder plane has 4 or 8 bytes per site).
inline bool row_tma(int hx, int wb) { return (hx * (wb % 16)) % 16 == 0; }

// Vectors per CTA of the row kernel: `want` if it is a multiple of vb dividing nvec, else the
// largest such count with (count / vb) * hx <= 256 threads.  0: no fit.
inline int row_group(int nvec, int vb, int hx, int want)
{
    auto fits = [&](int n) { return n >= vb && n % vb == 0 && nvec % n == 0 && (n / vb) * hx <= 256; };
    if (want > 0 && fits(want)) return want;
    for (int n = nvec; n >= vb; n -= vb)
        if (fits(n)) return n;
    return 0;
}

// Estimated time of one step (us) of the other kernels, fitted to 1600 measured (lattice, slices,
// vectors, storage, W format) problems on a GB300: cubes of 8 to 64 and boxes of 4 to 64, even and odd
// rows, 1 to 64 slices, 2 to 96 vectors.  Each is a latency of the step and, per warp of
// an SM, a time that depends on the formats (us; two and four vectors a thread), beside
// the bytes at 6.6 TB/s and what a CTA costs by itself.  Spread of estimate / measurement:
// 10 % for the interleaved kernels, 13 % for the row and the planar one.
enum StepFmt { SF_32_18, SF_32_12, SF_32_8, SF_32_18_H, SF_16_18, SF_16_12, SF_N };  // W (_H: 16-bit vectors)

inline int step_fmt(int vby, int wb)
{
    switch (wb) {
    case 72: return vby == 16 ? SF_32_18_H : SF_32_18;
    case 48: return SF_32_12;
    case 32: return SF_32_8;
    case 36: return SF_16_18;
    default: return SF_16_12;
    }
}

inline double step_bytes(const SubGeom &g, int nblk, int n, int vby, int wb)
{
    return (double)nblk * g.Vs * (3.0 * wb + 2.0 * vby * n);
}

// Plain interleaved kernel (k_step_il), n vectors (an even number): any row, no staging.
inline double il_estimate(const SubGeom &g, int nblk, int n, int vby, int wb, int num_sms)
{
    static const double per_warp[SF_N][2] = {{.109, .252}, {.092, .198}, {.202, .324}, {.105, .269}, {.109, .235}, {.129, .225}};
    const int vb = n % 4 ? 2 : 4, tx = n / vb, spb = std::max(1, std::min(il_spb(tx, 256), g.hx));
    const double warps = (double)((g.hx + spb - 1) / spb) * g.hy * g.hz * nblk * ((tx * spb + 31) / 32);
    return 5.2 + (wb == 32 ? 2.0 : 0.0) + step_bytes(g, nblk, n, vby, wb) / 9.0e6 +
           per_warp[step_fmt(vby, wb)][vb / 4] * warps / num_sms;
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

// Row kernel with the parameters of row_tile; where its copies do not apply, the packed kernel
// (k_step_ilx) that runs instead.  Where the vectors of a row do not divide, a CTA is left with one
// pair or two and copies the five W rows for them: no candidate then (44^3, one slice, 26
// vectors with W f32-12: 103 us against 51 with the interleaved kernel).
inline double row_estimate(const SubGeom &g, int nblk, int n, int vby, int wb, int num_sms)
{
    static const double per_warp[SF_N][2] = {{.145, .223}, {.149, .233}, {.254, .358}, {.148, .255}, {.161, .284}, {.171, .291}};
    static const double packed[SF_N][2] = {{.028, .042}, {.05, .08}, {.2, .3}, {.071, .150}, {.089, .155}, {.093, .185}};
    int tile[3];
    const int vb = row_tile(g, nblk, n, vby, tile), f = step_fmt(vby, wb);
    const double rows = (double)nblk * g.hy * g.hz;
    const int nvg = row_group(n, vb, g.hx, tile[0]);
    if (row_tma(g.hx, wb) && nvg > 0 && row_smem(g.hx, wb) <= kRowMaxSmem) {
        if (nvg < 8 && nvg < n) return 1e300;
        const double ctas = rows * (n / nvg);
        const double a = per_warp[f][vb / 4] * ctas * ((nvg / vb * g.hx + 31) / 32) / num_sms;
        const double b = 1.3e-4 * ctas, w = 0.116e-6 * ctas * g.hx * 5 * wb;  // starting them; their W rows from L2
        return (wb == 32 ? 4.0 : 2.3) + std::sqrt(a * a + b * b + w * w);
    }
    const int tx = n / vb, spb = std::max(1, std::min(std::min(il_spb(tx, 256), g.hx), 56));
    const double ctas = rows * ((g.hx + spb - 1) / spb);
    return 5.4 + step_bytes(g, nblk, n, vby, wb) / 3.5e6 + 7.2e-4 * ctas +
           packed[f][vb / 4] * ctas * ((tx * spb + 31) / 32) / num_sms;
}

// Vectors per thread of the planar kernel when it takes several at once.
inline int planar_vb(int storage, int nvec)
{
    const int cap = storage == P_F64 ? 4 : 8;
    int vb = 2;
    while (vb < cap && vb < nvec) vb *= 2;
    return vb;
}

// All vectors in one launch of the planar kernel, two or four a thread: reads W once, has no rows
// to keep whole, but pays for unused lanes of its four vectors.  For two to four vectors; not for
// the 8-real W, whose reconstruction rounds differently there.
inline double planar_estimate(const SubGeom &g, int nblk, int nvec, int vby, int wb, int num_sms)
{
    static const double per_warp[SF_N][2] = {{.254, .523}, {.317, .585}, {0, 0}, {.298, .468}, {.273, .473}, {.246, .456}};
    if (wb == 32 || nvec < 2 || nvec > 4) return 1e300;
    const double warps = (double)(((int64_t)nblk * g.Vs + 31) / 32);
    const double a = per_warp[step_fmt(vby, wb)][nvec > 2] * warps / num_sms, b = 1.6 * nvec;
    return 2.5 + 1.07 * std::pow(std::pow(a, 1.46) + std::pow(b, 1.46), 1 / 1.46);
}

// What the fit of col_estimate leaves out when kernels are compared, from the same 1600 problems
// (spread 15 %): tiles of one or two warps and 16-bit records take longer, W f32-8 less.
inline double col_bias(const ColPlan &p, int vby, int wb)
{
    return (p.threads <= 32 ? 1.34 : p.threads <= 64 ? 1.12 : 1.0) * (vby == 16 ? 1.075 : 1.0) * (wb == 32 ? 0.9 : 1.0);
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

// tile[] of the tune entry for a shape: 9 selects the column kernel.
inline void col_tile_of(const ColPlan &p, int tile[3])
{
    tile[0] = p.nvg;
    tile[1] = 9;
    tile[2] = p.ny | p.nseg << 8 | p.units << 16;
}

// The kernel of a call without a tune entry: the cheapest by these estimates.  In short steps, where
// they are least sure, the plain kernel gets 5 % of credit: it was the only one before the others
// came in.  Chosen by earlier estimates, which knew neither it nor rows off 16 bytes, 266 of the 1600 problems ran more than 10 % slower
// than with it (up to 2.0 times), now 10 (up to 1.3); the mean over all is 1.32 times its rate, 1.26
// before.
enum StepKind { STEP_IL, STEP_ROW, STEP_COL, STEP_PLANAR };

struct StepPlan {
    int kind, vb;  // vb 0: the kernel's own rule
    int tile[3];
    ColPlan col;
};

// n of the call's nvec vectors are packed at a time; exact: no padded groups; planar: the planar kernel
// is possible.
inline StepPlan plan_step(const SubGeom &g, int nblk, int nvec, int n, int vby, int wb, int num_sms, bool exact, bool planar)
{
    StepPlan s{};
    const int n2 = (n + 1) & ~1;
    double best = il_estimate(g, nblk, n2, vby, wb, num_sms);
    if (best < 40) best *= 0.95;
    s.kind = STEP_IL;
    const double row = row_estimate(g, nblk, n2, vby, wb, num_sms);
    if (row < best) {
        best = row;
        s.kind = STEP_ROW;
    }
    const double pl = planar ? planar_estimate(g, nblk, nvec, vby, wb, num_sms) : 1e300;
    if (pl < best) {
        best = pl;
        s.kind = STEP_PLANAR;
    }
    double us = 0;
    if (col_plans(g, nblk, exact ? n2 : n, vby, wb, num_sms, &s.col, &us, 1, exact) > 0 &&
        us * col_bias(s.col, vby, wb) < best)
        s.kind = STEP_COL;
    if (s.kind == STEP_ROW) s.vb = row_tile(g, nblk, n, vby, s.tile);
    if (s.kind == STEP_PLANAR) s.tile[1] = 10;
    if (s.kind == STEP_COL) {
        s.vb = 2;
        col_tile_of(s.col, s.tile);
    }
    return s;
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

// The shape of such an entry.  False: no fit.
inline bool col_of_tile(const SubGeom &g, int nblk, int nvec, int vby, int wb, const int tile[3], ColPlan &out)
{
    return col_shape(g, nblk, nvec, vby, wb, tile[0], tile[2] & 255, std::max(1, (tile[2] >> 8) & 255), tile[2] >> 16, out);
}

// FP64 steps.  The FP64 pipe of an SM takes 1.82 us for the step of a warp (32 sites and vectors),
// so what counts is the warps on the busiest SM, beside what a launch costs; fitted to 110 measured
// problems (one slice of 8^3 to 48^3, 8^3 x 8 to 32^3 x 16, odd rows, 2 to 30 vectors), within 10 %.
// One launch per vector and step: small lattices run three threads a site in CTAs of one warp.
inline double f64_single_estimate(const SubGeom &g, int nblk, int nvec, int num_sms)
{
    const int64_t sites = (int64_t)nblk * g.Vs;
    auto per_sm = [&](int64_t n) { return (double)((n + num_sms - 1) / num_sms); };
    const int64_t rows = (sites + 31) / 32 * 3;
    const double one = sites > (int64_t)4 * 32 * num_sms ? 3 + 1.82 * 4 * per_sm((sites + 127) / 128)
                       : rows <= 2 * num_sms             ? 4.2
                                                         : std::max(9.3, 3 + 0.62 * per_sm(rows));
    return nvec * one;
}

// All vectors in one launch (k_step_il, one vector a thread): strips of a row, whose last one may be
// short.  Idle lanes cost their share (32^3 x 16, 3 vectors: 48 of 64 lanes, 778 us against 598
// one by one), launches theirs (8^3, one slice, 12 vectors: 12.6 us against 47.7).
inline double f64_il_estimate(const SubGeom &g, int nblk, int nvec, int num_sms)
{
    double us = 0;
    for (int v = 0; v < nvec; v += 256) {
        const int n = std::min(nvec - v, 256), spb = std::min(il_spb(n, 256), g.hx);
        const int full = g.hx / spb, rest = g.hx - full * spb;
        const double warps = (double)full * ((spb * n + 31) / 32) + (rest * n + 31) / 32;  // of a row
        const int strips = full + (rest > 0);
        const int64_t ctas = (int64_t)strips * g.hy * g.hz * nblk;
        us += std::max(12.4, 4 + 1.82 * ((ctas + num_sms - 1) / num_sms) * warps / strips);
    }
    return us;
}

}  // namespace tls
