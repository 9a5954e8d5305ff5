"""The planner's rules on the host (csrc/col_plan.h, layout_plan.h; no GPU): compiled with g++ behind a few C functions."""

import ctypes
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2301_05518_gb300", "csrc")

GLUE = r"""
#include "col_plan.h"
#include "layout_plan.h"
using namespace tls;
static SubGeom geom(const int *h) { return SubGeom{h[0], h[1], h[2], h[0] * h[1] * h[2], (h[0] * h[1] * h[2] + 31) / 32 * 32}; }
static int out_of(const ColPlan &p, int *o)
{
    const int v[] = {p.nvg, p.ny, p.nseg, p.units, p.smem, p.ntile, p.threads};
    for (int k = 0; k < 7; ++k) o[k] = v[k];
    return 1;
}
extern "C" {
int entry_shape(const int *h, int nblk, int nvec, int vby, int wb, const int *tile, int *o)
{
    ColPlan p;
    return col_of_tile(geom(h), nblk, nvec, vby, wb, tile, p) ? out_of(p, o) : 0;
}
int best_shapes(const int *h, int nblk, int nvec, int vby, int wb, int most, int *tiles, int *o)
{
    ColPlan p[8] = {};
    double us[8];
    const int n = col_plans(geom(h), nblk, nvec, vby, wb, 152, p, us, most);
    for (int k = 0; k < n; ++k) {
        col_tile_of(p[k], tiles + 3 * k);
        out_of(p[k], o + 7 * k);
    }
    return n;
}
double estimate(const int *h, int nblk, int nvec, int vby, int wb, const int *tile)
{
    ColPlan p;
    return col_of_tile(geom(h), nblk, nvec, vby, wb, tile, p) ? col_estimate(p, geom(h), nblk, vby, wb, 152, 1e300) : 1e300;
}
int planned(const int *h, int nblk, int nvec, int vby, int wb, int exact, int planar, int *tile)
{
    const StepPlan s = plan_step(geom(h), nblk, nvec, nvec, vby, wb, 152, exact, planar);
    for (int k = 0; k < 3; ++k) tile[k] = s.tile[k];
    return s.kind;
}
double f64_us(const int *h, int nblk, int nvec, int single)
{
    return single ? f64_single_estimate(geom(h), nblk, nvec, 152) : f64_il_estimate(geom(h), nblk, nvec, 152);
}
int link_rows(int Lx, long long nrow) { return ingest_rows(Lx, 64, nrow); }
void split(int T, int Lx, int nrow, int *o)
{
    const PairSplit p = pair_split(T, Lx, nrow);
    o[0] = p.rows;
    o[1] = p.chunks;
    o[2] = p.pairs;
}
int fits(unsigned long long used, unsigned long long cap, int n, const unsigned long long *have, const unsigned long long *need)
{
    return workspace_fits(used, cap, n, (const uint64_t *)have, (const uint64_t *)need);
}
}
"""


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    d = tmp_path_factory.mktemp("plan")
    (d / "glue.cpp").write_text(GLUE)
    subprocess.check_call(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-I" + CSRC, "-o", str(d / "plan.so"),
                           str(d / "glue.cpp")])
    lib = ctypes.CDLL(str(d / "plan.so"))
    lib.estimate.restype = lib.f64_us.restype = ctypes.c_double
    return lib


def ints(*v):
    return (ctypes.c_int * len(v))(*v)


def entry(plan, h, nvec, nvg, ny, nseg, units, vby=24, wb=72, nblk=8):
    o = ints(*[0] * 7)
    ok = plan.entry_shape(ints(*h), nblk, nvec, vby, wb, ints(nvg, 9, ny | nseg << 8 | units << 16), o)
    return list(o) if ok else None


@pytest.mark.parametrize("units,want", [(0, 6), (3, 3), (5, 5), (6, 6), (9, 6), (1, None), (2, None), (-1, None), (-3, None)])
def test_ring_units_of_an_entry(plan, units, want):
    """Fewer than three units are no ring: such a shape does not fit (the planner takes over)."""
    got = entry(plan, (4, 4, 4), 8, 8, 2, 1, units)
    assert (got and got[3]) == want
    if got:
        assert 0 < got[4] <= 226 * 1024


@pytest.mark.parametrize("hy,hz,nblk,vby,wb", [(256, 4, 152, 24, 32), (256, 4, 1024, 24, 32), (256, 4, 152, 24, 24),
                                               (480, 32, 304, 24, 24), (24, 24, 8, 24, 72), (17, 9, 40, 16, 24)])
@pytest.mark.parametrize("nvec", [2, 4, 24])
def test_planned_shape_is_the_launched_shape(plan, hy, hz, nblk, vby, wb, nvec):
    """Shapes travel to the kernel as tune entries: what the planner chose is what the entry says, also
    where a tile could take more rows than an entry can hold (2 x 512 x 8 sites a slice)."""
    hx = 1 if hy > 100 else hy
    tiles, o = ints(*[0] * 24), ints(*[0] * 56)
    n = plan.best_shapes(ints(hx, hy, hz), nblk, nvec, vby, wb, 3, tiles, o)
    assert n > 0
    for k in range(n):
        q = ints(*[0] * 7)
        assert plan.entry_shape(ints(hx, hy, hz), nblk, nvec, vby, wb, ints(*tiles[3 * k:3 * k + 3]), q) == 1
        assert list(q) == o[7 * k:7 * k + 7]


@pytest.mark.parametrize("used,cap,have,need,want", [
    (100, 0, [0, 0], [1 << 40, 1 << 40], True),       # no cap
    (100, 120, [40, 40], [50, 50], True),             # both grow by ten: 120 in use
    (100, 119, [40, 40], [50, 50], False),
    (100, 100, [40, 40], [40, 10], True),             # nothing grows, nothing shrinks
    (100, 104, [40, 40], [10, 45], False),            # a buffer that is larger than needed stays
    (100, 105, [40, 40], [10, 45], True)])
def test_padding_is_decided_before_a_buffer_is_freed(plan, used, cap, have, need, want):
    arr = ctypes.c_ulonglong * len(have)
    assert bool(plan.fits(ctypes.c_ulonglong(used), ctypes.c_ulonglong(cap), len(have), arr(*have), arr(*need))) == want


@pytest.mark.parametrize("T", [1, 2, 3, 4, 5, 9, 12, 13, 24, 36, 128])
@pytest.mark.parametrize("Lx,nrow", [(2, 4), (4, 2304), (12, 1296), (48, 2304), (66, 6), (512, 4)])
def test_pair_split_fills_the_threads(plan, T, Lx, nrow):
    """Every pair has a place, at most four lie side by side, and a CTA of 256 threads is at least half
    full unless the whole slice has less work or a chunk of another pair does not fit."""
    p = ints(0, 0, 0)
    plan.split(T, Lx, nrow, p)
    rows, chunks, pairs = p
    assert chunks * pairs >= T > (chunks - 1) * pairs and 1 <= pairs <= 4
    assert 1 <= rows <= nrow
    items = chunks * pairs * Lx
    assert rows == 1 or rows * items <= 256
    assert rows * items > 128 or rows == nrow


@pytest.mark.parametrize("h,nblk,nvec", [((24, 24, 24), 8, 24), ((24, 24, 24), 256, 72), ((2, 24, 24), 8, 72), ((5, 17, 3), 40, 7),
                                         ((1, 9, 8), 512, 3), ((33, 4, 16), 8, 30), ((8, 64, 64), 1, 12)])
@pytest.mark.parametrize("vby,wb", [(24, 72), (16, 24)])
def test_search_finds_the_best_shapes(plan, h, nblk, nvec, vby, wb):
    """Shapes dropped early by a lower bound are none of the best three: against the full list, each shape
    estimated without a limit."""
    every = set()
    for nvg in range(2, 26, 2):
        if -(-nvec // nvg) * nvg * 3 > 4 * ((nvec + 1) & ~1) or nvg > ((nvec + 1) & ~1):
            continue
        for ny in {-(-h[1] // t) for t in range(1, h[1] + 1)}:
            for nseg in (1, 2, 4):
                if nseg * 4 <= h[2]:
                    for units in (0, 3):
                        got = entry(plan, h, nvec, nvg, ny, nseg, units, vby, wb, nblk)
                        if got:
                            every.add((got[0], 9, got[1] | got[2] << 8 | got[3] << 16))
    times = sorted(plan.estimate(ints(*h), nblk, nvec, vby, wb, ints(*t)) for t in every)
    tiles, o = ints(*[0] * 24), ints(*[0] * 56)
    n = plan.best_shapes(ints(*h), nblk, nvec, vby, wb, 3, tiles, o)
    assert n == min(3, len(times))
    for k in range(n):
        t = tuple(tiles[3 * k:3 * k + 3])
        assert t in every and plan.estimate(ints(*h), nblk, nvec, vby, wb, ints(*t)) == times[k]


IL, ROW, COL, PLANAR = range(4)


# measured us per step (interleaved / row or its stand-in / column / planar), a GB300: kernels within 10 % of the best
@pytest.mark.parametrize("h,nblk,nvec,vby,wb,good", [
    ((22, 22, 22), 8, 26, 24, 48, {IL, COL}),      # 51 / 103 / 48: the row kernel is left one pair a CTA
    ((13, 2, 21), 336, 46, 24, 32, {IL}),          # 293 / 567 / 508
    ((17, 17, 17), 8, 4, 24, 72, {IL, COL}),       # 8.2 / 14.5 / 8.7 / 11.1: rows off 16 bytes
    ((13, 13, 13), 264, 53, 16, 24, {IL}),         # 609 / 732 / 791
    ((29, 29, 29), 40, 6, 16, 24, {IL}),           # 119 / 181 / 154 / 255
    ((24, 24, 24), 512, 24, 24, 72, {COL}),        # 3980 / 1950 / 1800
    ((32, 32, 32), 128, 24, 24, 48, {ROW, COL}),   # 2126 / 1188 / 1232
    ((16, 16, 16), 256, 24, 24, 32, {ROW}),        # 573 / 450
    ((8, 8, 8), 8, 6, 16, 36, {ROW}),              # 6.1 / 2.8 / 10.4
    ((14, 14, 14), 40, 2, 24, 72, {ROW, PLANAR}),  # 12.7 / 9.5 / 16.0 / 8.1
])
def test_planned_kernel_is_a_good_one(plan, h, nblk, nvec, vby, wb, good):
    assert plan.planned(ints(*h), nblk, nvec, vby, wb, 0, 1, ints(0, 0, 0)) in good


@pytest.mark.parametrize("vby,wb", [(24, 72), (24, 48), (24, 32), (16, 72), (16, 48), (16, 36), (16, 24)])
def test_plan_is_launchable(plan, vby, wb):
    """Over sizes and counts: a planned column shape fits as it is written down, padded groups only where
    they are allowed, the planar kernel only where it is possible."""
    for h in ((1, 1, 1), (1, 300, 2), (3, 7, 5), (17, 4, 9), (24, 24, 24), (150, 3, 2)):
        for nblk in (1, 8, 200):
            for nvec in (1, 2, 3, 5, 24, 31, 96, 256):
                for exact in (0, 1):
                    t = ints(0, 0, 0)
                    kind = plan.planned(ints(*h), nblk, nvec, vby, wb, exact, 0, t)
                    assert kind in (IL, ROW, COL)
                    if kind == COL:
                        o = ints(*[0] * 7)
                        assert t[1] == 9 and plan.entry_shape(ints(*h), nblk, nvec, vby, wb, t, o) == 1
                        assert not exact or ((nvec + 1) & ~1) % t[0] == 0
                    else:
                        assert t[1] == (6 if kind == ROW else 0)


# half extents, blocks, then vectors and measured us per step: one launch per vector / one for all
F64 = [
    ((4, 4, 4), 8, [(2, 7.9, 12.4), (3, 12.1, 12.5), (6, 23.9, 12.4), (12, 47.7, 12.6), (24, 95.5, 12.6), (30, 119.5, 12.5)]),
    ((6, 6, 6), 8, [(2, 8.0, 12.4), (3, 12.3, 12.5), (6, 24.6, 12.5), (12, 52.0, 14.5), (24, 107.8, 22.8), (30, 140.7, 25.0)]),
    ((8, 8, 8), 8, [(2, 17.3, 12.6), (3, 27.2, 12.3), (6, 55.4, 18.6), (12, 110.9, 24.8), (24, 221.3, 47.4), (30, 276.2, 61.8)]),
    ((12, 12, 12), 8, [(2, 19.1, 18.8), (3, 28.8, 33.1), (6, 57.5, 47.4), (12, 114.6, 76.2), (24, 228.9, 140.5), (30, 286.1, 176.7)]),
    ((16, 16, 16), 128, [(2, 399.2, 392.3), (3, 598.4, 778.1), (6, 1195.4, 1164.5), (12, 2391.1, 2322.2), (24, 4780.5, 4636.6), (30, 5977.0, 6177.9)]),
    ((4, 4, 4), 64, [(2, 17.1, 16.4), (3, 26.9, 16.4), (6, 55.2, 16.4), (12, 110.6, 30.8), (24, 220.3, 43.2), (30, 275.6, 53.6)]),
    ((24, 24, 24), 8, [(2, 94.6, 119.6), (3, 141.9, 176.7), (6, 283.1, 283.2), (12, 566.2, 505.9), (24, 1131.5, 983.1), (30, 1414.1, 1308.6)]),
    ((8, 8, 8), 64, [(2, 37.4, 53.6), (3, 55.8, 53.7), (6, 111.2, 104.7), (12, 221.6, 154.1), (24, 442.7, 295.3), (30, 553.1, 391.9)]),
    ((3, 5, 7), 32, [(2, 15.0, 18.7), (3, 26.0, 18.9), (6, 56.5, 18.7), (12, 113.6, 33.1), (24, 227.0, 47.5), (30, 282.9, 47.6)]),
    ((6, 6, 6), 192, [(2, 50.9, 90.6), (3, 76.7, 90.7), (6, 154.1, 168.8), (12, 306.7, 252.6), (24, 613.7, 417.7), (30, 766.4, 498.2)]),
]


@pytest.mark.parametrize("h,nblk,times", F64)
def test_f64_choice(plan, h, nblk, times):
    """One FP64 vector per launch or all in one: the choice is within 10 % of the better one (a launch's
    time: within 5 us)."""
    for nvec, single, together in times:
        a, b = plan.f64_us(ints(*h), nblk, nvec, 1), plan.f64_us(ints(*h), nblk, nvec, 0)
        chosen = single if a < b else together
        assert chosen <= max(1.1 * min(single, together), min(single, together) + 5), (nvec, a, b, single, together)


@pytest.mark.parametrize("Lx,nrow,want", [(2, 110592, 32), (4, 55296, 16), (6, 100000, 10), (8, 100000, 0), (48, 100000, 0),
                                          (2, 512, 0), (2, 304 * 32, 32), (2, 304 * 32 - 2, 0)])
def test_short_rows_of_links_share_a_cta(plan, Lx, nrow, want):
    assert plan.link_rows(Lx, ctypes.c_longlong(nrow)) == want
