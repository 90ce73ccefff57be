"""The host-side plans of the kernels that march several steps along strips
(csrc/lbm_plan.cu), built for the CPU: the strips cover every lattice, and planning one
takes time in proportion to its size."""
import ctypes
import os
import subprocess
import time

import numpy as np
import pytest

from paper_1307_4703_gb300 import workloads as W

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1307_4703_gb300", "csrc")
PORT, SIDE, LANE = 1 << 16, 1 << 17, 18  # kPairPort, kPairSide, kPairLaneBit
FP32, FP16 = 0, 1
SHAPES = {FP32: ((6, 304, 152), (4, 456, 152)), FP16: ((8, 304, 152), (6, 304, 152))}  # warps, resident blocks, SMs
SCALAR = (9, 304, 152)
LEVELS = 3
SINGLE_WARPS = 2432

# Tiles as lbm_create makes them: from a row's first fluid node on, in steps of 128
# nodes, or by 128-node segments where the last one would run past the padded row.
SHIM = r"""
#include <cstring>
#include "lbm_plan.h"
using namespace lbm;
static StripPlan p;
static std::vector<uint2> tiles;
extern "C" {
void make_tiles(const uint8_t* solid, int nx, int ny, int pitch)
{
    auto S = [&](int x, int y) { return x < 0 || y < 0 || x >= nx || y >= ny || solid[size_t(y) * nx + x]; };
    tiles.clear();
    for (int y = 0; y < ny; ++y)
        for (int gran : {kTileStart, kTileNodes}) {
            const size_t first = tiles.size();
            bool fits = true, scattered = false;
            int t0 = -1, q0 = 0, q1 = 0, wall = -1;
            auto push = [&] {
                tiles.push_back(make_uint2((unsigned(y) << kColBits) | unsigned(t0 / kTileStart),
                                           unsigned(q0) | (unsigned(q1) << 8) | (scattered ? kWallTile : 0u)));
            };
            for (int x = 0; x < nx && fits; ++x) {
                if (S(x, y)) continue;
                if (t0 < 0 || x >= t0 + kTileNodes) {
                    if (t0 >= 0) push();
                    t0 = x / gran * gran;
                    if (t0 + kTileNodes > pitch) fits = false;
                    q0 = (x - t0) / 4;
                    wall = -1;
                    scattered = false;
                }
                q1 = (x - t0) / 4;
                scattered |= wall >= 0 && q1 > wall;
                bool link = false;
                for (int dy = -1; dy <= 1; ++dy)
                    for (int dx = -1; dx <= 1; ++dx) link |= S(x + dx, y + dy);
                if (link && q1 > q0) wall = q1;
            }
            if (fits) {
                if (t0 >= 0) push();
                break;
            }
            tiles.resize(first);
        }
}
void make_plan(int nx, int ny, int pitch, const int* port_x, int levels, int precision, int rescale, const int* shapes,
               int n_shapes, long long single_warps, double* out)
{
    std::vector<RowBC> bc(size_t(2) * ny, RowBC{-1, 0, 0.f, 0.f});
    for (int k = 0; k < 2 * ny; ++k) bc[size_t(k)].x = port_x[k];
    PairShape s[2] = {};
    for (int k = 0; k < n_shapes; ++k) s[k] = {shapes[3 * k], shapes[3 * k + 1], shapes[3 * k + 2]};
    p = levels ? plan_scalar(tiles, bc, nx, ny, pitch, levels, s[0].warps, s[0].resident)
               : plan_pairs(tiles, bc, nx, ny, pitch, precision, rescale, s, n_shapes, single_warps);
    out[0] = double(tiles.size());
    out[1] = double(p.items.size());
    out[2] = p.grid;
    out[3] = p.warps;
    out[4] = p.work;
    out[5] = p.worth;
}
void get_plan(int* items, int* first)
{
    std::memcpy(items, p.items.data(), p.items.size() * sizeof(int4));
    std::memcpy(first, p.block_first.data(), p.block_first.size() * sizeof(int));
}
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("plan")
    shim, so = d / "shim.cpp", d / "plan.so"
    shim.write_text(SHIM)
    include = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, "-I", include, "-x", "c++",
                    os.path.join(CSRC, "lbm_plan.cu"), str(shim), "-o", str(so)], check=True)
    return ctypes.CDLL(str(so))


def _ptr(a):
    return a.ctypes.data_as(ctypes.c_void_p)


class Plan:
    def __init__(self, lib, solid, ports=(), levels=0, precision=FP32, rescale=False, shapes=None):
        solid = np.ascontiguousarray(np.asarray(solid) != 0, dtype=np.uint8)
        self.ny, self.nx = solid.shape
        self.pitch = (self.nx + 127) // 128 * 128
        self.port_x = np.full((2, self.ny), -1, np.int32)
        for q in ports:
            self.port_x[q["side"], q["y0"]:q["y1"]] = q["x"]
        shapes = np.array(shapes or ([SCALAR] if levels else SHAPES[precision]), np.int32)
        lib.make_tiles(_ptr(solid), self.nx, self.ny, self.pitch)
        out = np.zeros(6)
        t = time.perf_counter()
        lib.make_plan(self.nx, self.ny, self.pitch, _ptr(self.port_x), levels, precision, int(rescale), _ptr(shapes),
                      len(shapes), ctypes.c_longlong(SINGLE_WARPS), _ptr(out))
        self.seconds = time.perf_counter() - t
        self.tiles, n, self.grid, self.warps, self.work, self.worth = int(out[0]), int(out[1]), int(out[2]), int(out[3]), \
            out[4], bool(out[5])
        self.items = np.zeros((n, 4), np.int32)
        self.first = np.zeros(self.grid + 1, np.int32)
        lib.get_plan(_ptr(self.items), _ptr(self.first))


def _check(p, solid, halo, resident):
    """Blocks in one wave, each with strips; a strip's lanes and the rows and lanes around
    them lie in the lattice; ports that it or its neighbour rows hold are announced; and
    every fluid node is written by one strip, no node by two."""
    assert p.grid <= resident and p.first[0] == 0 and p.first[-1] == len(p.items)
    assert np.all(np.diff(p.first) > 0)
    cover = np.zeros((p.ny, p.pitch), np.int32)
    for x0, lanes, ya, yb in p.items.tolist():
        l0, l1 = lanes & 0xFF, (lanes >> 8) & 0xFF
        assert 0 <= x0 and x0 % 4 == 0 and x0 + 128 <= p.pitch and l0 <= l1 <= 31 and 0 <= ya < yb <= p.ny
        assert l0 > 0 or x0 == 0  # a neighbouring lane, or the lattice's edge
        assert l1 < 31 or x0 + 128 >= p.nx
        near = p.port_x[:, max(ya - halo, 0):yb + halo]
        assert not np.any((near >= x0) & (near < x0 + 128)) or lanes & PORT
        cover[ya:yb, x0 + 4 * l0:x0 + 4 * l1 + 4] += 1
    assert cover.max() == 1 and np.all(cover[:, :p.nx][np.asarray(solid) == 0] == 1)


@pytest.mark.parametrize("seed", range(12))
def test_strips_cover_the_lattice(lib, seed):
    r = np.random.default_rng(seed)
    for _ in range(12):
        nx, ny = int(r.integers(1, 900)), int(r.integers(1, 120))
        kind = r.integers(4)
        if kind == 0:    # scattered cells, few to nearly all
            solid = r.random((ny, nx)) < r.choice([0.03, 0.2, 0.5, 0.7, 0.97])
        elif kind == 1:  # two blocks of rows, each of its own columns
            solid = np.ones((ny, nx), bool)
            m = int(r.integers(ny + 1))
            for rows in (slice(0, m), slice(m, ny)):
                a, b = sorted(r.integers(0, nx + 1, 2))
                solid[rows, a:b] = False
        elif kind == 2:  # channels
            solid = np.zeros((ny, nx), bool)
            solid[3::int(r.integers(4, 20))] = True
        else:            # pillars
            solid = np.zeros((ny, nx), bool)
            step = int(r.integers(8, 40))
            for k in range(step // 3):
                for j in range(step // 3):
                    solid[k::step, j::step] = True
        if solid.all():
            continue
        ports = [dict(side=0, x=int(r.integers(nx)), y0=0, y1=max(1, ny // 3))] if r.integers(2) else []
        resident = int(r.integers(1, 600))
        warps = int(r.choice([4, 6, 8]))
        _check(Plan(lib, solid, ports, shapes=[(warps, resident, 1 + resident // 2)]), solid, 1, resident)
        _check(Plan(lib, solid, ports, levels=LEVELS, shapes=[(9, resident, 1)]), solid, LEVELS - 1, resident)


def test_planning_time_follows_the_size(lib):
    """A row's spans and strips are walked once: a lattice 256 times as wide and as many
    times lower takes about as long (strips times spans a row made it 11 times as long)."""
    cells = np.random.default_rng(1).random(1 << 22) < 0.9

    def seconds(nx):
        return min(Plan(lib, cells.reshape(-1, nx), levels=k).seconds for k in (0, LEVELS, 0, LEVELS, 0))
    assert seconds(131072) < 4 * seconds(512)


@pytest.mark.parametrize("share", [0.2, 0.5, 0.7])
@pytest.mark.parametrize("nx,ny", [(2001, 1003), (4096, 2048)])
def test_dense_lattices_stay_in_long_strips(lib, nx, ny, share):
    """Scattered cells: strips as long as a block's share of the lattice, whatever part of it
    is solid (half solid fell into pieces of five rows).  A strip writes 120 of its 128
    columns and computes halo rows above and below it, so with at least ten strips a block's
    length apart the work is that of the tiles times the cost of an iteration (28 / 16,
    scalar 24 / 16), 128 / 120 and a tenth for the ends."""
    solid = np.random.default_rng(3).random((ny, nx)) < share
    for levels, cost in ((0, 28 / 16), (LEVELS, 24 / 16)):
        for precision in (FP32, FP16) if not levels else (FP32,):
            p = Plan(lib, solid, levels=levels, precision=precision)
            assert len(p.items) <= 2 * p.grid
            assert p.work < cost * 128 / 120 * 1.2 * p.tiles


def _pillars(nx, ny, step, side):
    solid = np.zeros((ny, nx), np.uint8)
    for y in range(4, ny - 8, step):
        for x in range(4 + (y // step % 2) * step // 2, nx - 8, step):
            solid[y:min(y + side, ny - 4), x:min(x + side, nx - 4)] = 1
    return solid


def test_two_steps_a_launch_where_they_are_faster(lib):
    """FP32, by the measured times a step that csrc/lbm_plan.cu gives: channel chips and
    lattices of scattered cells take two steps a launch, pillars whose strips fall into
    pieces only on large lattices."""
    for prob in (W.config_small(), W.config_full_chip(), W.config_adjoint_chip(), W.config_large_chip(2000, 1000)):
        assert Plan(lib, prob["solid"], prob["ports"]).worth, prob["name"]
    for nx, ny in ((1001, 517), (2001, 1003)):
        for share in (0.03, 0.2, 0.5, 0.7):
            assert Plan(lib, np.random.default_rng(5).random((ny, nx)) < share).worth, (nx, ny, share)
    for nx, ny, step, side, worth in ((2001, 1003, 24, 10, True), (3000, 1500, 24, 10, True), (700, 400, 24, 10, False),
                                      (900, 600, 24, 10, False), (1001, 517, 24, 10, False), (700, 400, 12, 6, False)):
        ports = W.random_case(5, nx, ny, solid_frac=0.0)[0]["ports"]
        assert Plan(lib, _pillars(nx, ny, step, side), ports).worth == worth, (nx, ny, step, side)


def test_other_launches_where_they_are_faster(lib):
    """16-bit storage, ports of the rescaling kinds and scalar-only steps, as above: islands
    of a few nodes, walls every ninth row and rows of narrow channels go one step a launch,
    though their neighbours in kind do not."""
    nx, ny = 2001, 1003
    prob = W.random_case(5, nx, ny, solid_frac=0.95)[0]
    assert not Plan(lib, prob["solid"], prob["ports"], levels=LEVELS).worth
    for share in (0.03, 0.5, 0.7):
        solid = np.random.default_rng(5).random((ny, nx)) < share
        assert Plan(lib, solid, levels=LEVELS).worth and Plan(lib, solid, precision=FP16).worth
    y = np.arange(ny)[:, None] + np.zeros(nx, int)
    inner = np.zeros((ny, nx), bool)
    inner[:, 4:-4] = True
    ports = W.random_case(5, nx, ny, solid_frac=0.0)[0]["ports"]
    rows, channels = (y % 9 == 4) & inner, (y % 40 >= 12) & inner
    assert not Plan(lib, rows, ports, precision=FP16).worth
    assert not Plan(lib, channels, ports, rescale=True).worth
    assert Plan(lib, channels, ports).worth
    chip = W.config_large_chip()
    for precision in (FP32, FP16):
        for rescale in (False, True):
            assert Plan(lib, chip["solid"], chip["ports"], precision=precision, rescale=rescale).worth


@pytest.mark.parametrize("n,seed", [(3, 1), (4, W.SEED + 4), (4, 2), (16, 1)])
def test_small_batches_take_two_steps_a_launch(lib, n, seed):
    """Batches as lbm_create_batch stacks them (one solid row between chips): two steps a
    launch are the faster way from three chips on."""
    probs = W.config_batch(n, seed=seed)
    nx = max(q["nx"] for q in probs)
    rows, ports, y = [], [], 0
    for k, q in enumerate(probs):
        if k:
            rows.append(np.ones((1, nx), np.uint8))
            y += 1
        m = np.ones((q["ny"], nx), np.uint8)
        m[:, :q["nx"]] = q["solid"]
        rows.append(m)
        ports += [dict(r, y0=r["y0"] + y, y1=r["y1"] + y) for r in q["ports"]]
        y += q["ny"]
    assert Plan(lib, np.concatenate(rows), ports).worth
