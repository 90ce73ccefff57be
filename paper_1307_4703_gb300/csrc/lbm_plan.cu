// lbm_plan.cu -- host-side plans of the kernels that march several steps along
// strips (lbm_pair.cu, the levels kernel of lbm_scalar.cu): strips of the lattice
// and their split over the blocks of one wave.
#include <algorithm>
#include <vector>

#include "lbm_plan.h"


namespace lbm {
namespace {

// Strips begin and end on multiples of this many columns: whole 32-byte
// sectors of FP32 rows (at multiples of 4 the large chip took 45.6 against 44.7
// us a step, its blocks sharing sectors).
constexpr int kAlign = 8;

struct Span {
    int b, e;  // columns [b, e)
};

// A strip's columns: lanes l0 .. l1 of the 128 columns from x0 are written.
struct Strip {
    int x0, l0, l1;
    int begin() const { return x0 + 4 * l0; }
    int end() const { return x0 + 4 * (l1 + 1); }
};

// Strips that cover the spans from the left.  A strip writes its lanes
// 1 .. 30: lanes 0 and 31 are computed for the second step of their
// neighbours only, except at the lattice's own edges.
std::vector<Strip> cover(const std::vector<Span>& spans, int nx, int pitch)
{
    std::vector<Strip> out;
    for (const Span& s : spans) {
        int p = s.b;
        while (p < s.e) {
            if (!out.empty() && p < out.back().end()) {
                p = out.back().end();
                continue;
            }
            p = p / kAlign * kAlign;
            const int x0 = std::min(std::max(p - 4, 0), pitch - kTileNodes);
            int l1 = x0 + kTileNodes >= nx ? 31 : 30;
            if (l1 == 30) l1 = (x0 + 124) / kAlign * kAlign / 4 - x0 / 4 - 1;
            const Strip t{x0, (p - x0) / 4, l1};
            out.push_back(t);
            p = t.end();
        }
    }
    return out;
}

// Which of `strips` a row's spans touch (both in order of their columns, one walk
// over them), how many, and whether they cover all of the spans.
int touched(const std::vector<Strip>& strips, const std::vector<Span>& spans, std::vector<char>& hit, bool& covered)
{
    int hits = 0;
    size_t k = 0;
    hit.assign(strips.size(), 0);
    for (size_t n = 0; n < strips.size(); ++n) {
        while (k < spans.size() && spans[k].e <= strips[n].begin()) ++k;
        if (k == spans.size()) break;
        if (spans[k].b < strips[n].end()) {
            hit[n] = 1;
            ++hits;
        }
    }
    covered = true;
    k = 0;
    for (const Span& s : spans)
        for (int p = s.b; p < s.e;) {
            while (k < strips.size() && strips[k].end() <= p) ++k;
            if (k == strips.size() || strips[k].begin() > p) {
                covered = false;
                return hits;
            }
            p = strips[k].end();
        }
    return hits;
}

// What a strip's rows hold.  The costs are of an iteration of the march (of the
// two coupled steps, of the scalar-only steps), measured on the 4096 x 2048 chip
// and the batch of 64 chips (the splits that were fastest): side walls add the
// side lanes' work, ports that of a lane that completes its node alone while
// its warp waits, and walls anywhere a wait for the nodes' own values in global
// memory.  (Ports of two coupled steps at 24 instead of 22: 1024 x 768 6.2 us a step
// against 5.4, 64 chips 77.6 against 77.0; at 20 2000 x 1000 10.7 against 10.4.)
enum Kind { kPlain, kSide, kScattered, kPort, kScatteredPort };
constexpr int kPairCost[5] = {16, 18, 28, 22, 33};
constexpr int kPairRescaleCost[5] = {16, 18, 28, 30, 42};  // with ports of the rescaling kinds (22: 4096 x 2048 44 us, here 39)
constexpr int kScalarCost[5] = {16, 20, 24, 28, 32};
// What an iteration of two coupled steps takes next to a plain one (16), by least
// squares over some hundred lattices, FP32 and 16-bit alike (the costs above are
// those of the fastest splits).
constexpr int kPairTime[5] = {16, 17, 21, 22, 25};

struct Run {
    Strip t;
    int ya, yb;
    Kind kind;
    int side;   // kPairSide and the lanes along the walls
    int rough;  // rows with scattered walls
};

constexpr int kBandRows = 8;  // rows that must gain from new strips before the strips change

// Consecutive rows [ya, yb) whose fluid covers the same columns (whole quads).
struct Rows {
    int ya, yb;
    std::vector<Span> spans;
    std::vector<Strip> own;  // the strips that cover them alone
};

std::vector<Rows> row_groups(const std::vector<uint2>& tiles, int nx, int ny, int pitch)
{
    std::vector<Rows> out;
    std::vector<Span> spans;
    size_t t = 0;
    for (int y = 0; y < ny; ++y) {
        spans.clear();
        for (; t < tiles.size() && int(tiles[t].x >> kColBits) == y; ++t) {
            const int x0 = int(tiles[t].x & ((1u << kColBits) - 1)) * kTileStart;
            const Span s{x0 + 4 * int(tiles[t].y & 0xFFu), x0 + 4 * int((tiles[t].y >> 8) & 0xFFu) + 4};
            if (!spans.empty() && spans.back().e == s.b) spans.back().e = s.e;
            else spans.push_back(s);
        }
        if (!out.empty() && out.back().spans.size() == spans.size() &&
            std::equal(spans.begin(), spans.end(), out.back().spans.begin(),
                       [](const Span& a, const Span& b) { return a.b == b.b && a.e == b.e; }))
            out.back().yb = y + 1;
        else
            out.push_back({y, y + 1, spans, {}});
    }
    const int parts = parts_for((long long)out.size() * (pitch / kTileNodes), 1 << 14, (long long)out.size());
    const bool ok = over_parts(parts, [&](int k) {
        for (size_t g = out.size() * size_t(k) / size_t(parts); g < out.size() * size_t(k + 1) / size_t(parts); ++g)
            out[g].own = cover(out[g].spans, nx, pitch);
    });
    if (!ok) throw std::bad_alloc();
    return out;
}

std::vector<Run> strip_runs(const std::vector<Rows>& groups)
{
    std::vector<Run> runs;
    std::vector<Strip> cur;
    std::vector<int> open;  // index of each strip's run in `runs`, -1 = none
    std::vector<char> hit, ahead;
    for (size_t k = 0; k < groups.size(); ++k) {
        const Rows& g = groups[k];
        bool covered = false;
        const int hits = touched(cur, g.spans, hit, covered);
        bool fresh = g.spans.empty() || !covered;
        if (!fresh) {  // would other strips do with fewer, and for long enough?
            int gain = 0;
            for (size_t n = k; n < groups.size() && gain < kBandRows; ++n) {
                bool c = false;
                if (groups[n].spans.empty() ||
                    (n == k ? hits : touched(cur, groups[n].spans, ahead, c)) <= int(groups[n].own.size()))
                    break;
                gain += groups[n].yb - groups[n].ya;
            }
            fresh = gain >= kBandRows;
        }
        if (fresh) {
            cur = g.own;
            open.assign(cur.size(), -1);
            touched(cur, g.spans, hit, covered);
        }
        for (size_t n = 0; n < cur.size(); ++n) {
            if (!hit[n]) open[n] = -1;
            else if (open[n] >= 0) runs[size_t(open[n])].yb = g.yb;
            else {
                open[n] = int(runs.size());
                runs.push_back({cur[n], g.ya, g.yb, kPlain, 0, 0});
            }
        }
    }
    return runs;
}

// Runs split where they start or stop holding port nodes or side walls, and
// their kinds: scattered walls where more than half of the rows have some
// within the strip (kWallTile).  Parts of scattered walls in a row stay one run:
// in dense lattices side walls come and go every few rows, and each part's
// neighbour rows are computed once more (4096 x 2048, half solid: 15200 strips
// instead of 331, a scalar-only step 88.9 us instead of 40.6, 65.8 one step a
// launch; two coupled steps in FP16 184 a step instead of 102, 154 one by one).
std::vector<Run> split_kinds(const std::vector<Run>& runs, const std::vector<Rows>& groups,
                             const std::vector<uint2>& tiles, const std::vector<RowBC>& bc, int ny, int halo)
{
    std::vector<int> group_of(static_cast<size_t>(ny));
    for (size_t k = 0; k < groups.size(); ++k)
        for (int y = groups[k].ya; y < groups[k].yb; ++y) group_of[size_t(y)] = int(k);
    // first columns of the tiles with scattered walls, row after row
    std::vector<int> walls, first_wall;
    for (const uint2& t : tiles)
        if (t.y & kWallTile) {
            first_wall.resize(size_t(t.x >> kColBits) + 1, int(walls.size()));
            walls.push_back(int(t.x & ((1u << kColBits) - 1)) * kTileStart);
        }
    first_wall.resize(size_t(ny) + 1, int(walls.size()));
    std::vector<int> port_cols;
    for (const RowBC& b : bc)
        if (b.x >= 0 && (port_cols.empty() || port_cols.back() != b.x)) port_cols.push_back(b.x);
    std::sort(port_cols.begin(), port_cols.end());
    auto split_run = [&](const Run& r, std::vector<Run>& out) {
        const int x0 = r.t.x0, x1 = x0 + kTileNodes;
        // the lanes where the row's fluid begins and ends within the strip; -1: more than two
        auto side = [&](int y) {
            int lanes = 0, n = 0;
            const std::vector<Span>& spans = groups[size_t(group_of[size_t(y)])].spans;
            auto s = std::lower_bound(spans.begin(), spans.end(), x0, [](const Span& a, int x) { return a.e <= x; });
            for (; s != spans.end() && s->b < x1 && n < 3; ++s) {
                if (s->b >= x0 && n++ < 2) lanes |= (s->b - x0) / 4 << (kPairLaneBit + 5 * (n - 1));
                if (s->e <= x1 && n++ < 2) lanes |= (s->e - 4 - x0) / 4 << (kPairLaneBit + 5 * (n - 1));
            }
            return n == 1 || n == 2 ? lanes | kPairSide : n ? -1 : 0;
        };
        const auto col = std::lower_bound(port_cols.begin(), port_cols.end(), x0);
        const bool any_port = col != port_cols.end() && *col < x1;
        auto port = [&](int y) {
            if (!any_port) return false;
            for (int yy = std::max(y - halo, 0); yy <= std::min(y + halo, ny - 1); ++yy)
                for (int s = 0; s < 2; ++s) {
                    const int px = bc[size_t(s) * ny + yy].x;
                    if (px >= x0 && px < x1) return true;
                }
            return false;
        };
        auto scattered = [&](int y) {
            const auto end = walls.begin() + first_wall[size_t(y) + 1];
            const auto w = std::upper_bound(walls.begin() + first_wall[size_t(y)], end, x0 - kTileNodes);
            return w != end && *w < x1;
        };
        for (int y = r.ya; y < r.yb;) {
            const bool ports = port(y);
            const int first = side(y);
            bool same = first >= 0;
            int last = group_of[size_t(y)], lanes = first, rough = 0, e = y;
            for (; e < r.yb && port(e) == ports; ++e) {
                if (group_of[size_t(e)] != last) {
                    last = group_of[size_t(e)];
                    lanes = side(e);
                    if ((lanes != 0) != (first != 0)) break;
                    same &= lanes == first;
                }
                rough += scattered(e);
            }
            const bool walls_anywhere = 2 * rough > e - y || !same;
            const Kind kind = ports ? (walls_anywhere ? kScatteredPort : kPort)
                              : walls_anywhere ? kScattered : first ? kSide : kPlain;
            const int walls_at = same ? first : 0;
            Run* const before = y > r.ya ? &out.back() : nullptr;
            if (before && before->kind == kind && (kind == kScattered || kind == kScatteredPort)) {
                before->yb = e;
                before->rough += rough;
                if (before->side != walls_at) before->side = 0;
            } else {
                out.push_back({r.t, y, e, kind, walls_at, rough});
            }
            y = e;
        }
    };
    long long rows = 0;
    for (const Run& r : runs) rows += r.yb - r.ya;
    const int parts = parts_for(rows, 1 << 14, (long long)runs.size());
    std::vector<std::vector<Run>> done(static_cast<size_t>(parts));
    const bool ok = over_parts(parts, [&](int k) {
        for (size_t n = runs.size() * size_t(k) / size_t(parts); n < runs.size() * size_t(k + 1) / size_t(parts); ++n)
            split_run(runs[n], done[size_t(k)]);
    });
    if (!ok) throw std::bad_alloc();
    std::vector<Run> out = std::move(done[0]);
    for (size_t k = 1; k < done.size(); ++k) out.insert(out.end(), done[k].begin(), done[k].end());
    return out;
}

// The runs cut into items of whole iterations, block after block, with at
// most `m` units of cost a block; returns the blocks this takes.
int split(const std::vector<Run>& runs, const int (&costs)[5], int halo, int W, int m, StripPlan* out)
{
    int blocks = 1, left = m, time = 0;
    if (out) {
        out->items.clear();
        out->block_first.assign(1, 0);
    }
    auto next_block = [&]() {
        ++blocks;
        left = m;
        time = 0;
        if (out) out->block_first.push_back(int(out->items.size()));
    };
    for (const Run& r : runs) {
        const int cost = costs[r.kind];
        // (an iteration is as slow as its slowest row: scattered walls in half of the
        // rows are in 0.7 of the iterations)
        const int rows = r.yb - r.ya, base = kPairTime[r.kind];
        const int more = kPairTime[r.kind >= kPort ? kScatteredPort : kScattered] - base;
        const int step = base + more * std::min(7 * r.rough, 5 * rows) / (5 * rows);
        for (int y = r.ya; y < r.yb;) {
            if (left < m && left / cost * W - 2 * halo < std::min(r.yb - y, W)) next_block();
            const int h = std::min(r.yb - y, std::max(left / cost * W - 2 * halo, 1));
            const int iterations = (h + 2 * halo + W - 1) / W;
            left -= iterations * cost;
            time += iterations * step;
            if (out) {
                out->time = std::max(out->time, time);
                out->items.push_back(make_int4(r.t.x0, r.t.l0 | (r.t.l1 << 8) | (r.kind >= kPort ? kPairPort : 0) | r.side, y, y + h));
            }
            y += h;
        }
    }
    if (out) out->block_first.push_back(int(out->items.size()));
    return blocks;
}

}  // namespace

namespace {
// Strips of the runs over one wave of `resident` blocks.
StripPlan plan(const std::vector<Run>& runs, const int (&costs)[5], int halo, int warps, int resident)
{
    StripPlan out;
    long long cost = 0;
    int least = 0;
    for (const Run& r : runs) {
        cost += (long long)((r.yb - r.ya + 2 * halo + warps - 1) / warps) * costs[r.kind];
        least = std::max(least, costs[r.kind] * ((1 + 2 * halo + warps - 1) / warps));
    }
    // the least cost of the costliest block for which one wave holds the blocks
    int m = int(std::max<long long>(least, cost / resident));
    while (split(runs, costs, halo, warps, m, nullptr) > resident) m += std::max(1, m / 64);
    split(runs, costs, halo, warps, m, &out);
    out.grid = int(out.block_first.size()) - 1;
    out.longest = m;
    // the work of the launch in plain rows of 128 nodes, blocks that end early included
    out.work = double(out.grid) * warps * m / costs[kPlain];
    return out;
}

double scattered_tiles(const std::vector<uint2>& tiles)
{
    double n = 0.;
    for (const uint2& t : tiles) n += (t.y & kWallTile) != 0;
    return n;
}

// A single step's time, us: of n tiles in one wave, in several, at the rate of
// memory, and what each tile of scattered walls adds.  These fits and those of the
// several-steps launches' times are within some 15 % over 340 lattices.
struct SingleTime {
    double wave, per_tile, waves, per_tile_waves, memory, wall;
};
constexpr SingleTime kSingle[2][2] = {  // FP32 and 16-bit storage; the second with ports of the rescaling kinds
    {{3.2, 0.95e-3, 4.0, 1.25e-3, 2.1e-3, 0.5e-3}, {4.1, 0.87e-3, 3.2, 1.54e-3, 2.3e-3, 0.5e-3}},
    {{4.7, 0.2e-3, 2.9, 1.02e-3, 1.33e-3, 1.0e-3}, {5.0, 0.3e-3, 3.3, 1.17e-3, 1.5e-3, 1.0e-3}}};
constexpr SingleTime kSingleScalar = {2.5, 0.36e-3, 2.0, 0.6e-3, 0.875e-3, 0.1e-3};
double single_step(const SingleTime& f, const std::vector<uint2>& tiles, long long warps)
{
    const double n = double(tiles.size());
    const double t = (long long)tiles.size() <= warps ? f.wave + f.per_tile * n : f.waves + f.per_tile_waves * n;
    return std::max(t, f.memory * n) + f.wall * scattered_tiles(tiles);
}

std::vector<Run> runs_of(const std::vector<uint2>& tiles, const std::vector<RowBC>& bc, int nx, int ny, int pitch, int halo)
{
    const std::vector<Rows> groups = row_groups(tiles, nx, ny, pitch);
    return split_kinds(strip_runs(groups), groups, tiles, bc, ny, halo);
}
}  // namespace

StripPlan plan_pairs(const std::vector<uint2>& tiles, const std::vector<RowBC>& bc, int nx, int ny, int pitch,
                     int precision, bool rescale, const PairShape* shapes, int n_shapes, long long single_warps)
{
    // The block shape: the one whose longest block is over first.  FP32, 2 blocks of 6
    // warps an SM or 3 of 4: an iteration of 4 warps takes 0.96 of one of 6 on a full
    // SM.  us a step, 6 / 4 warps: equal lengths 4096 x 2048 38.0 / 35.5, 64 chips 77.0 /
    // 74.7, 1300 x 800 6.9 / 6.6; 99 to 112 (1001 x 517 with obstacles) 9.4 / 10.9, 44 to
    // 48 (1024 x 768) 5.4 / 6.1.  16-bit, 2 blocks of 8 or of 6: 0.75 to 0.80 of the time.
    // 8 / 6 warps: 36 to 44 (1024 x 768) 5.16 / 4.86, 32 to 36 (1024 x 512) 4.92 / 4.13, 64
    // to 80 (2000 x 1000) 9.07 / 8.66, 208 to 273 (4096 x 2048) 28.1 / 28.7, 452 to 585
    // (64 chips) 60.9 / 63.1.  A block that has an SM to itself is faster still (FP32 400
    // x 300, 136 / 271 blocks: 2.64 / 3.08; 256 x 128, 54 / 101 blocks: 2.57 / 2.50).
    const bool f32 = precision == kFP32;
    const std::vector<Run> runs = runs_of(tiles, bc, nx, ny, pitch, 1);
    StripPlan p;
    int resident = 0;
    bool alone = false;  // every block of p has an SM to itself
    double best = 0.;
    for (int k = 0; k < n_shapes; ++k) {
        const PairShape& s = shapes[k];
        StripPlan q = plan(runs, rescale ? kPairRescaleCost : kPairCost, 1, s.warps, s.resident);
        q.warps = s.warps;
        const double time = q.longest * (k == 0 ? 1. : f32 ? 0.96 : 0.78);
        const bool spread = q.grid <= s.sms;
        if (k > 0 && (alone != spread ? alone : time >= best)) continue;
        best = time;
        alone = spread;
        resident = s.resident;
        p = std::move(q);
    }
    // Where single steps are the better choice: where obstacles break the rows into
    // pieces, each with its neighbours' rows around it.  Strips that leave half the
    // blocks' room idle are always the shorter way; elsewhere the longest block's time
    // is set against a single step's.  The margins are those that leave the least time
    // on the table: FP32 strips of much more work than the tiles' have to be ahead by a
    // tenth, those of few scattered walls may seem as much behind (batches of 3 and 4
    // chips 5.6 / 5.4, 5.5 / 5.2), and with rescaling ports they gain from the third
    // tile of a single step's warps on.  us a step, single / two-step launches: FP32 256
    // x 128 3.6 / 2.3, 1024 x 512 5.24 / 4.60, 1024 x 768 7.1 / 5.4, 4096 x 2048 59.5 /
    // 35.5; random cells, 3 and 70 % solid, 1001 x 517 10.5 / 9.5 and 12.2 / 9.6, 2001 x
    // 1003 40.7 / 32.4 and 51.3 / 36.5; pillars of 10 cells 24 apart, whose strips fall
    // into pieces of a dozen rows, 2001 x 1003 39.3 / 31.4 but 900 x 600 9.5 / 10.9 and 700
    // x 400 5.7 / 8.6; with rescaling ports 4096 x 2048 54.4 / 39.0, 1024 x 768 7.2 / 7.6,
    // channels of 12 rows in 40 2001 x 1003 14.1 / 18.7.  FP16 256 x 128 4.8 / 2.4, 1024 x
    // 768 5.6 / 4.9, 4096 x 2048 36.2 / 28.1, half solid 154 / 102; walls every ninth row
    // 2001 x 1003 21.4 / 26.3.
    const bool idle = 2 * p.grid <= resident;
    const double n = double(tiles.size()), work = p.work / (2. * n);
    double margin = 1.1, two;
    if (f32) {
        if (rescale) margin = (long long)tiles.size() <= 2 * single_warps ? 0. : 1.;
        else margin = work >= 1.5 ? 0.9 : 8. * scattered_tiles(tiles) < n ? 1.15 : 1.06;
        two = (rescale ? (p.warps == 4 ? 0.157 : 0.155) : (p.warps == 4 ? 0.126 : 0.131)) * p.time;
    } else {
        two = (rescale ? 0.7 : 0.2) + (p.warps == 6 ? 0.109 : rescale ? 0.147 : 0.138) * p.time;
    }
    p.worth = idle || two < margin * single_step(kSingle[f32 ? 0 : 1][rescale], tiles, single_warps);
    // With the state between the steps stored as well (a gradient's recomputation):
    // ahead on lattices that leave the GPU idle (a gradient over 150 steps of 256 x 128
    // 1605 -> 1447 us, 512 x 256 1270 -> 1210) and on those of more than two rounds of a
    // single step's tiles (2048 x 1024 3.70 -> 3.51 ms, 4096 x 2048 6.34 -> 6.04); between
    // them a draw (1024 x 512 3161 / 3194 us, 1500 x 900 2313 / 2322).
    p.worth_keep = idle || (p.worth && (long long)tiles.size() > 2 * single_warps);
    return p;
}

// Worth it unless the lattice is mostly solid: us a step, one step a launch / three,
// scattered cells 3 and 70 % solid 1001 x 517 4.5 / 4.2 and 4.8 / 4.4, 2001 x 1003 13.7 / 9.7
// and 14.2 / 10.1, 4096 x 2048 61.4 / 39.0; 95 % solid, islands of a few nodes, 2001 x 1003
// 9.5 / 35.4; walls every ninth row there 11.8 / 13.2; at worst, pillars of 10 cells 24
// apart, 1001 x 517 4.2 / 4.7.
StripPlan plan_scalar(const std::vector<uint2>& tiles, const std::vector<RowBC>& bc, int nx, int ny, int pitch, int levels,
                      int warps, int resident)
{
    StripPlan p = plan(runs_of(tiles, bc, nx, ny, pitch, levels - 1), kScalarCost, levels - 1, warps, resident);
    // (a single step's wave is 16 warps an SM, here two blocks)
    p.worth = 0.0607 * p.longest < 1.05 * single_step(kSingleScalar, tiles, 8ll * resident);
    return p;
}

}  // namespace lbm
