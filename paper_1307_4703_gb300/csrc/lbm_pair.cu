// lbm_pair.cu -- two coupled time steps in one launch (temporal blocking).
//
// A block marches along y over a strip of 128 columns.  Per iteration each of
// its W warps takes one row through the first step (populations pulled from
// the source buffer, result kept in a ring of W + 2 rows in shared memory) and
// then one row, a row behind, through the second step (pulled from the ring,
// result stored to the destination buffer): the state between the two steps
// never goes to memory, which halves the bytes a step moves.  The lanes at
// the strip's sides and the rows above and below its end are computed by the
// neighbouring strips too (their first step only), so blocks never wait for
// each other.  The arithmetic of each node is collide_quad on values rounded
// to the storage type, as in the single-step kernels: the same bits.
//
// What bounds it: memory first (363 MB a launch on the 4096 x 2048 chip, FP32,
// which HBM takes 54 us for, against 71), then the barriers' and shared memory's
// turns at 12 warps an SM, which shared memory (FP32: a staged row and 1.3 to 1.5
// ring rows a warp) and registers allow; 42% of the issue slots are used, 55% in
// 16-bit storage at 16 warps.  So nothing in the loop waits for global memory:
//   - the rows the W warps pull from come as 14 tensor copies a block and
//     iteration (one box of W rows a plane, each at the plane's own row
//     offset), shared between the warps and asked for as soon as every warp
//     has pulled its row, under the second step's arithmetic;
//   - wall-link words, port entries, relaxation rates and the side lanes' own
//     diagonal populations come by per-lane asynchronous copies an iteration
//     ahead (a load into a register an iteration ahead is waited for at once:
//     2100 of 4400 cycles a row);
//   - a strip along a side wall names the two lanes at it, and these bounce
//     back from the staged rows (from global memory, such strips took 1.5
//     times as long as the others and set the launch's length).
// Steps of the 4096 x 2048 chip, us: FP32 59.5 one by one, 35.5 here; FP16
// 36.2 -> 28.1; 64 chips in a batch 111 -> 74.7 (FP32).  FP32 blocks are of 6
// warps (2 an SM) or 4 (3 an SM), 16-bit blocks of 8 or 6 (2 an SM), whichever the
// strips of a lattice suit (plan_pairs).  Tried: the second step's rows written by bulk copies from
// shared memory (50.4 against 46.7 us at that stage: 14 copies a row by one warp
// are slow to issue); rows copied lane by lane (cp.async: FP32 the same, FP16
// 34.7 against 30.5 us); 5 x 2 (40.1 where 6 x 2 took 38.0) and 12 x 1 (59 us) for
// FP32; 4 x 4 (27.9 against 28.1 us, 1024 x 768 5.6 against 4.9), 5 x 3 (29.6), 7 x 2
// (30.8), 9 x 2 and 10 x 2 (43 and 45: 96 registers spill) for 16-bit.
#include <algorithm>

#include <cudaTypedefs.h>

#include "lbm_device.cuh"

namespace lbm {
namespace {

// Resident blocks per SM of W warps: what shared memory and registers allow.
constexpr int pair_blocks(int W) { return W == 4 ? 3 : 2; }
template <typename T>
constexpr int kBoxCols = sizeof(T) == 4 ? 136 : 144;  // columns of a staged row: the strip's 128, a halo of at least one
                                                      // on each side, from a 16-byte boundary on

// A ring row: 14 plane rows of the strip's first step, its wall-link words,
// relaxation rates and port entries.
template <typename T>
struct alignas(16) RingRow {
    T pl[kPlanes][kTileNodes];
    unsigned links[kTileNodes / 4];
    RowBC bc[2];
    float2 rates;
    float2 pad;
};
// What a warp copies for its row of the next iteration beside the boxes.
template <typename T>
struct alignas(16) RowStage {
    unsigned links[kTileNodes / 4];  // wall-link words, lanes l0 - 1 .. l1 + 1
    RowBC bc[2];                     // the row's port entries, for strips that hold port nodes
    T side[2][4][4];                 // the side lanes' own quads of planes 5 .. 8
    float2 rates;                    // the row's relaxation rates (batches)
    float2 pad;
};
template <typename T, int W>
struct alignas(128) PairSmem {
    struct alignas(128) Box {
        T row[W][kBoxCols<T>];
    } box[kPlanes];    // the W rows each plane is pulled from
    RowStage<T> stage[W];
    RingRow<T> ring[W + 2];
    uint64_t full;     // the boxes have arrived
    uint64_t done;     // the iteration's first-step rows are in the ring
    uint64_t read;     // the iteration's second steps have read the ring
};
template <typename T, int W>
constexpr bool smem_aligned()
{
    using S = PairSmem<T, W>;
    using R = RingRow<T>;
    using G = RowStage<T>;
    return offsetof(S, box) % 128 == 0 && sizeof(typename S::Box) % 128 == 0 && offsetof(S, stage) % 16 == 0 &&
           offsetof(S, ring) % 16 == 0 && offsetof(S, full) % 8 == 0 && offsetof(S, done) % 8 == 0 &&
           offsetof(S, read) % 8 == 0 && offsetof(R, links) % 16 == 0 && offsetof(R, bc) % 16 == 0 &&
           offsetof(R, rates) % 8 == 0 && sizeof(R) % 16 == 0 && offsetof(G, bc) % 16 == 0 &&
           offsetof(G, side) % 16 == 0 && offsetof(G, rates) % 8 == 0 && sizeof(G) % 16 == 0;
}
static_assert(smem_aligned<float, 4>() && smem_aligned<float, 6>() && smem_aligned<__half, 6>() &&
                  smem_aligned<__half, 8>(),
              "targets of vector accesses, copies and barriers");
static_assert(sizeof(PairSmem<__half, 6>) == sizeof(PairSmem<__nv_bfloat16, 6>) &&
                  sizeof(PairSmem<__half, 8>) == sizeof(PairSmem<__nv_bfloat16, 8>),
              "one 16-bit layout");

// Column of x0 in a staged row (x0 is a multiple of 4).
template <typename T>
__device__ __forceinline__ int box_offset(int x0)
{
    return sizeof(T) == 4 ? 4 : 4 + (~x0 & 4);
}

template <typename T>
__device__ __forceinline__ void cp_async_quad(T* dst, const T* src)
{
    if constexpr (sizeof(T) == 4) cp_async16(dst, src);
    else cp_async8(dst, src);
}

struct PairStrip {
    int x0, l0, l1, ya, yb;
    bool port, side;
    int s0, s1;  // side: the lanes along a side wall
    PairStrip() = default;
    __device__ __forceinline__ explicit PairStrip(int4 it)
        : x0(it.x), l0(it.y & 0xFF), l1((it.y >> 8) & 0xFF), ya(it.z), yb(it.w), port(it.y & kPairPort), side(it.y & kPairSide),
          s0((it.y >> kPairLaneBit) & 31), s1((it.y >> (kPairLaneBit + 5)) & 31)
    {
    }
    // row of the march's j-th row (the first step takes rows ya - 1 .. yb)
    __device__ __forceinline__ int row(int j, int reverse) const { return reverse ? yb - j : ya - 1 + j; }
};

// The lane's quads of the 14 planes at the pull sources, from row r of the
// boxes.
template <typename T, int W>
__device__ __forceinline__ void pull_staged(float4 (&v)[kPlanes], const PairSmem<T, W>& sm, int r, int offset, int lane)
{
#pragma unroll
    for (int p = 0; p < kPlanes; ++p) {
        const T* row = &sm.box[p].row[r][offset + 4 * lane];
        float4 r = Codec<T>::lds4(row, 0.f);
        if (src_col(p) == 1) {
            float w = __shfl_up_sync(kFull, r.w, 1);
            if (lane == 0) w = Codec<T>::lds1(row - 1, 0.f);
            r = make_float4(w, r.x, r.y, r.z);
        } else if (src_col(p) == 2) {
            float e = __shfl_down_sync(kFull, r.x, 1);
            if (lane == 31) e = Codec<T>::lds1(row + 4, 0.f);
            r = make_float4(r.y, r.z, r.w, e);
        }
        v[p] = r;
    }
}

// Completion of the open port node k of a lane's quad.  kRescale: the lattice
// has ports of the rescaling kinds, whose completion is a call (complete_port);
// kernels without it are 2 to 6 % faster (4096 x 2048 in FP32 39.4 -> 39.0 us a
// step, FP16 30.1 -> 29.3; 256 x 128 2.70 -> 2.60, FP16 2.97 -> 2.79, before the
// packed arithmetic).
template <bool kRescale, int k, typename T>
__device__ __forceinline__ void port_at(float4 (&v)[kPlanes], bool west, const RowBC& b, const StepArgs& a, const T* S,
                                        long long oC)
{
    float f[9], g[5];
#pragma unroll
    for (int i = 0; i < 9; ++i) f[i] = at(v[i], k);
#pragma unroll
    for (int i = 0; i < 5; ++i) g[i] = at(v[9 + i], k);
    port_node<kRescale>(f, g, west, b, a, S, oC + k);
#pragma unroll
    for (int i = 0; i < 9; ++i) at(v[i], k) = f[i];
#pragma unroll
    for (int i = 0; i < 5; ++i) at(v[9 + i], k) = g[i];
}

// Completion of the open port nodes among a lane's quad; bc: the row's west
// and east port entries.
template <bool kRescale, typename T>
__device__ __forceinline__ void port_pass(float4 (&v)[kPlanes], int x0, const RowBC* bc, const StepArgs& a, const T* S,
                                          long long oC)
{
#pragma unroll 1
    for (int side = 0; side < 2; ++side) {
        const RowBC b = side == 0 ? bc[0] : bc[1];
        if (b.x < x0 || b.x >= x0 + 4 || !valve_open(a, b.chan_kind)) continue;
        switch (b.x - x0) {
        case 0: port_at<kRescale, 0>(v, side == 0, b, a, S, oC); break;
        case 1: port_at<kRescale, 1>(v, side == 0, b, a, S, oC); break;
        case 2: port_at<kRescale, 2>(v, side == 0, b, a, S, oC); break;
        default: port_at<kRescale, 3>(v, side == 0, b, a, S, oC); break;
        }
    }
}

// Halfway bounce-back as bounce_back, its loads in three groups (a wall to
// the west, to the east, above or below): the loads of a group are in flight
// together, so a row along a side wall waits for one of them and not for
// each link's in turn.
template <int kFirst, int kCount, typename T>
__device__ __forceinline__ void bounce_group(float4 (&v)[kPlanes], unsigned lk, unsigned wall, const T* S, long long P,
                                             long long oC)
{
    // the links of group kFirst: 1, 5, 8 (west), 3, 6, 7 (east) or 2, 4 (below, above)
    constexpr int d[3] = {kFirst, kFirst == 1 ? 5 : kFirst == 3 ? 6 : 4, kFirst == 1 ? 8 : 7};
    unsigned any = 0;
#pragma unroll
    for (int n = 0; n < kCount; ++n) any |= 1u << (d[n] - 1);
    if (!(wall & any)) return;
    float4 own[kCount], ownc[kCount];
#pragma unroll
    for (int n = 0; n < kCount; ++n) {
        own[n] = Codec<T>::ld4(S + opp(d[n]) * P + oC, 0.f);
        if (d[n] <= 4) ownc[n] = Codec<T>::ld4(S + (9 + opp(d[n])) * P + oC, 0.f);
    }
#pragma unroll
    for (int n = 0; n < kCount; ++n)
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const bool link = (lk >> (8 * k + d[n] - 1)) & 1u;
            at(v[d[n]], k) = link ? at(own[n], k) : at(v[d[n]], k);
            if (d[n] <= 4) at(v[9 + d[n]], k) = link ? at(ownc[n], k) : at(v[9 + d[n]], k);
        }
}

template <typename T>
__device__ __forceinline__ void bounce_groups(float4 (&v)[kPlanes], unsigned lk, unsigned groups, const T* S, long long P,
                                              long long oC)
{
    unsigned wall = 0;  // union of the wall links of the fluid nodes
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const unsigned lb = (lk >> (8 * k)) & 0xFFu;
        if (lb != kSolid) wall |= lb;
    }
    wall &= groups;
    if (!wall) return;
    bounce_group<1, 3>(v, lk, wall, S, P, oC);
    bounce_group<3, 3>(v, lk, wall, S, P, oC);
    bounce_group<2, 2>(v, lk, wall, S, P, oC);
}

// Bounce-back at walls to the west and east for a strip's side lane, from its
// warp's row of the boxes (r; c: the lane's first column in it), which holds
// the populations along the row, and its stage, which holds the diagonal ones.
template <typename T, int W>
__device__ __forceinline__ void bounce_side(float4 (&v)[kPlanes], unsigned lk, const RowStage<T>& st, const PairSmem<T, W>& sm, int r,
                                            int c, int n)
{
    const float4 f1 = Codec<T>::lds4(&sm.box[1].row[r][c], 0.f), f3 = Codec<T>::lds4(&sm.box[3].row[r][c], 0.f);
    const float4 g1 = Codec<T>::lds4(&sm.box[10].row[r][c], 0.f), g3 = Codec<T>::lds4(&sm.box[12].row[r][c], 0.f);
    const float4 f5 = Codec<T>::lds4(st.side[n][0], 0.f), f6 = Codec<T>::lds4(st.side[n][1], 0.f);
    const float4 f7 = Codec<T>::lds4(st.side[n][2], 0.f), f8 = Codec<T>::lds4(st.side[n][3], 0.f);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const unsigned lb = lk >> (8 * k);
        if (lb & 0x01u) at(v[1], k) = at(f3, k), at(v[10], k) = at(g3, k);
        if (lb & 0x04u) at(v[3], k) = at(f1, k), at(v[12], k) = at(g1, k);
        if (lb & 0x10u) at(v[5], k) = at(f7, k);
        if (lb & 0x20u) at(v[6], k) = at(f8, k);
        if (lb & 0x40u) at(v[7], k) = at(f5, k);
        if (lb & 0x80u) at(v[8], k) = at(f6, k);
    }
}

// Walls and ports of the lane's pulled quads; S, P and oC: the nodes' own
// stored populations.
template <bool kRescale, typename T>
__device__ __forceinline__ void complete_quad(const StepArgs& a, bool port, float4 (&v)[kPlanes], unsigned lk,
                                              unsigned groups, int x0, const RowBC* bc, const T* S, long long P, long long oC)
{
    bounce_groups<T>(v, lk, groups, S, P, oC);
    if (port) port_pass<kRescale, T>(v, x0, bc, a, S, oC);
}

// Collisions of the lane's quad.
template <bool kRescale, typename T>
__device__ __forceinline__ void collide_row(const StepArgs& a, float4 (&v)[kPlanes], unsigned lk, float2 omega, bool& bad)
{
    QuadAcc q;
    // packed arithmetic spills in 16-bit storage beside the rescaling call (34.4
    // against 32.1 us a step at 4096 x 2048)
    constexpr bool kPacked = !kRescale || kStoresF32<T>;
    collide_quad<T, true, false, kRescale, kPacked>(v, lk, 0, RowBC{}, RowBC{}, a, static_cast<const T*>(nullptr), 0, omega,
                                                    q);
    bad |= q.bad;
}

template <typename T, bool kRescale, int W, bool kKeep>
__global__ void __launch_bounds__(32 * W, pair_blocks(W))
    coupled_step_pair(const PairArgs p, const __grid_constant__ CUtensorMap map)
{
    constexpr int R = W + 2;
    extern __shared__ __align__(128) unsigned char pair_smem[];
    PairSmem<T, W>& sm = *reinterpret_cast<PairSmem<T, W>*>(pair_smem);
    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    const int reverse = p.first.reverse, pitch = p.first.pitch, ny = p.first.ny;
    const T* const src = reinterpret_cast<const T*>(p.first.src);
    const long long P = p.first.plane;
    RowStage<T>& stage = sm.stage[warp];
    bool bad = false;
    bool late = false;  // a wait gave up: nothing is copied or waited for any more

    if (threadIdx.x == 0) {
        mbar_init(&sm.full, W);
        mbar_init(&sm.done, W);
        mbar_init(&sm.read, W);
        mbar_fence_init();
    }
    int i = p.block_first[blockIdx.x];
    const int i_end = p.block_first[blockIdx.x + 1];
    PairStrip st(p.items[i]);
    __syncthreads();
    grid_dependency_sync();

    // warp w asks for planes w, w + W, ... of an iteration whose first march
    // row is j: the W rows each plane is pulled from (rows outside the lattice
    // arrive as zeros, which no fluid node uses)
    auto issue_boxes = [&](const PairStrip& s, int j) {
        if (lane != 0) return;
        const int y = reverse ? s.row(j + W - 1, 1) : s.row(j, 0);  // lowest row
        const int x = s.x0 - box_offset<T>(s.x0);
        mbar_arrive_expect_tx(&sm.full, uint32_t((kPlanes - warp + W - 1) / W) * uint32_t(W * kBoxCols<T> * sizeof(T)));
        for (int q = warp; q < kPlanes; q += W) {
            const int dy = (0x0864 >> q) & 1 ? -1 : (0x2190 >> q) & 1;  // planes 2, 5, 6, 11 and 4, 7, 8, 13 (src_row)
            tensor_g2s(&sm.box[q], &map, x, y + dy, q, &sm.full);
        }
    };
    // and copies what else its own row y needs
    auto issue_row = [&](const PairStrip& s, int y) {
        const long long row = (long long)y * pitch + s.x0;
        if (lane >= s.l0 - 1 && lane <= s.l1 + 1) cp_async4(&stage.links[lane], p.first.links + row + 4 * lane);
        if (s.port && lane < 2) cp_async16(&stage.bc[lane], p.first.rowbc + (lane == 0 ? y : ny + y));
        if (s.side && lane < 8)
            cp_async_quad(&stage.side[lane >> 2][lane & 3][0],
                          src + (5 + (lane & 3)) * P + row + 4 * (lane < 4 ? s.s0 : s.s1));
        if (p.first.rates != nullptr && lane == 8) cp_async8(&stage.rates, p.first.rates + y);
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    // march rows outside the lattice or past the strip's end are not computed
    auto live = [&](const PairStrip& s, int j) {
        const int y = s.row(j, reverse);
        return j < s.yb - s.ya + 2 && y >= 0 && y < ny;
    };
    auto rates_of = [&](const StepArgs& a, const float2& row) {
        return a.rates != nullptr ? row : make_float2(a.omega_f, a.omega_g);
    };

    unsigned issued = 1;  // iterations whose boxes were asked for
    issue_boxes(st, 0);
    bool here = live(st, warp);
    if (here) issue_row(st, st.row(warp, reverse));

    int base = 0;   // first march row of the iteration
    int sp = warp;  // ring slot of the warp's march row
    // Iteration t.  Every warp waits for every phase of the three barriers, so
    // none of them can run more than one phase ahead of a waiting warp.
    for (unsigned t = 0;; ++t) {
        const int rows = st.yb - st.ya;
        const int j = base + warp, y = st.row(j, reverse);
        const int sc = sp >= 1 ? sp - 1 : R - 1;
        const int sq = sc >= 1 ? sc - 1 : R - 1;  // slots of the rows j - 1 and j - 2
        // the next iteration, of this strip or of the block's next one
        PairStrip nst = st;
        int nbase = base + W;
        bool more = true;
        if (nbase >= rows + 2) {
            nbase = 0;
            more = i + 1 < i_end;
            if (more) nst = PairStrip(p.items[i + 1]);
        }
        const bool next = more && live(nst, nbase + warp);

        // ---- free flight of the first step, and its walls at the side lanes ----
        float4 v[kPlanes];
        unsigned lk = 0xFFFFFFFFu;
        RowBC bc[2];
        float2 rates;
        const bool at_side = st.side && (lane == st.s0 || lane == st.s1);
        if (!late) late = !mbar_wait(&sm.full, t & 1u);
        if (here) {
            asm volatile("cp.async.wait_group 0;" ::: "memory");
            __syncwarp();
            const int r = reverse ? W - 1 - warp : warp, c = box_offset<T>(st.x0);
            pull_staged<T>(v, sm, r, c, lane);
            if (lane >= st.l0 - 1 && lane <= st.l1 + 1) lk = stage.links[lane];
            if (st.port) {
                bc[0] = stage.bc[0];
                bc[1] = stage.bc[1];
            }
            rates = stage.rates;
            if (at_side) bounce_side(v, lk, stage, sm, r, c + 4 * lane, lane == st.s0 ? 0 : 1);
        }
        late = __any_sync(kFull, late);
        if (next && !late) issue_row(nst, nst.row(nbase + warp, reverse));  // the warp's stage is free again

        // ---- first step of row j, into the ring once the second steps of
        //      the iteration before have read it ----
        if (lk != 0xFFFFFFFFu) {
            complete_quad<kRescale>(p.first, st.port, v, lk, at_side ? 0x0Au : 0xFFu, st.x0 + 4 * lane, bc, src, P,
                          (long long)y * pitch + st.x0 + 4 * lane);
            collide_row<kRescale, T>(p.first, v, lk, rates_of(p.first, rates), bad);
            if constexpr (kKeep) {  // the state between the steps, of the rows and lanes the second step writes
                if (y >= st.ya && y < st.yb && lane >= st.l0 && lane <= st.l1) {
                    T* const M = static_cast<T*>(p.mid) + (long long)y * pitch + st.x0 + 4 * lane;
#pragma unroll
                    for (int q = 0; q < kPlanes; ++q) Codec<T>::st4(M + q * P, v[q], 0.f);
                }
            }
        }
        if (t > 0 && !late) late = !mbar_wait(&sm.read, (t - 1) & 1u);
        if (here) {
            RingRow<T>& out = sm.ring[sp];
            out.links[lane] = lk;
            if (lane == 0) {
                out.rates = rates;
                if (st.port) {
                    out.bc[0] = bc[0];
                    out.bc[1] = bc[1];
                }
            }
            if (lk != 0xFFFFFFFFu) {
#pragma unroll
                for (int q = 0; q < kPlanes; ++q) Codec<T>::st4(&out.pl[q][4 * lane], v[q], 0.f);
            }
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(&sm.done);

        // ---- second step of row j - 1 ----
        if (!late) late = !mbar_wait(&sm.done, t & 1u);
        if (more && !late) {  // every warp has pulled its row from the boxes
            issue_boxes(nst, nbase);
            ++issued;
        }
        const int y2 = st.row(j - 1, reverse);
        const RingRow<T>& rC = sm.ring[sc];
        lk = 0xFFFFFFFFu;
        if (j >= 2 && j <= rows + 1) {
            const RingRow<T>& rS = sm.ring[reverse ? sp : sq];
            const RingRow<T>& rN = sm.ring[reverse ? sq : sp];
            if (lane >= st.l0 && lane <= st.l1) lk = rC.links[lane];
            rates = rC.rates;
#pragma unroll
            for (int q = 0; q < kPlanes; ++q) {
                const RingRow<T>& row = src_row(q) == 0 ? rC : src_row(q) == 1 ? rS : rN;
                float4 r = Codec<T>::lds4(&row.pl[q][4 * lane], 0.f);
                // the values shifted in at lanes 0 and 31 are never used: those lanes
                // are computed for their neighbours only, or lie at a wall
                if (src_col(q) == 1) r = make_float4(__shfl_up_sync(kFull, r.w, 1), r.x, r.y, r.z);
                else if (src_col(q) == 2) r = make_float4(r.y, r.z, r.w, __shfl_down_sync(kFull, r.x, 1));
                v[q] = r;
            }
            if (lk != 0xFFFFFFFFu)
                complete_quad<kRescale>(p.second, st.port, v, lk, 0xFFu, st.x0 + 4 * lane, rC.bc,
                              reinterpret_cast<const Shared<T>*>(&rC.pl[0][0]), kTileNodes, 4 * lane);
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(&sm.read);
        if (lk != 0xFFFFFFFFu) {
            collide_row<kRescale, T>(p.second, v, lk, rates_of(p.second, rates), bad);
            T* __restrict__ D = reinterpret_cast<T*>(p.second.dst) + (long long)y2 * pitch + st.x0 + 4 * lane;
#pragma unroll
            for (int q = 0; q < kPlanes; ++q) Codec<T>::st4(D + q * P, v[q], 0.f);
        }
        if (!more) break;
        if (nbase == 0) ++i;
        st = nst;
        base = nbase;
        here = next;
        sp += W;
        if (sp >= R) sp -= R;
    }
    if (late) {
        // no copy may still be writing this block's shared memory at exit
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        mbar_wait(&sm.full, (issued - 1) & 1u);
        atomicOr(p.first.err, 2u);
    }
    if (__any_sync(kFull, bad) && lane == 0) atomicOr(p.first.err, 1u);
}

template <typename T, bool kRescale, int W, bool kKeep = false>
cudaError_t launch(const PairArgs& p, const CUtensorMap& map, int grid, cudaStream_t s)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(32 * W);
    cfg.dynamicSmemBytes = sizeof(PairSmem<T, W>);
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, coupled_step_pair<T, kRescale, W, kKeep>, p, map);
}

template <typename T, bool kRescale, int W, bool kKeep = false>
cudaError_t occupancy(int* per_sm)
{
    cudaError_t e = cudaFuncSetAttribute(coupled_step_pair<T, kRescale, W, kKeep>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         int(sizeof(PairSmem<T, W>)));
    if (e == cudaSuccess)
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(per_sm, coupled_step_pair<T, kRescale, W, kKeep>, 32 * W,
                                                          sizeof(PairSmem<T, W>));
    return e;
}

// f.template operator()<T, kRescale, W>() of the instance that a launch takes.
template <typename T, int kFew, int kMany, typename F>
cudaError_t instance_of(bool rescale, int warps, const F& f)
{
    if (warps == kFew) return rescale ? f.template operator()<T, true, kFew>() : f.template operator()<T, false, kFew>();
    return rescale ? f.template operator()<T, true, kMany>() : f.template operator()<T, false, kMany>();
}
template <typename F>
cudaError_t instance(int precision, bool rescale, int warps, const F& f)
{
    if (precision == kFP16) return instance_of<__half, 6, 8>(rescale, warps, f);
    if (precision == kBF16) return instance_of<__nv_bfloat16, 6, 8>(rescale, warps, f);
    return instance_of<float, 4, 6>(rescale, warps, f);
}
struct Occupancy {
    int* per_sm;
    template <typename T, bool kRescale, int W>
    cudaError_t operator()() const
    {
        return occupancy<T, kRescale, W>(per_sm);
    }
};
struct Launch {
    const PairArgs& p;
    const CUtensorMap& map;
    int grid;
    cudaStream_t s;
    template <typename T, bool kRescale, int W>
    cudaError_t operator()() const
    {
        if constexpr (sizeof(T) == 4 && !kRescale)
            if (p.mid != nullptr) return launch<T, kRescale, W, true>(p, map, grid, s);
        return launch<T, kRescale, W>(p, map, grid, s);
    }
};

}  // namespace

cudaError_t pair_occupancy(int precision, bool rescale, int warps, int* per_sm)
{
    return instance(precision, rescale, warps, Occupancy{per_sm});
}

cudaError_t pair_keep_occupancy(int warps, int* per_sm)
{
    return warps == 4 ? occupancy<float, false, 4, true>(per_sm) : occupancy<float, false, 6, true>(per_sm);
}

cudaError_t rows_tensor_map(CUtensorMap* map, void* base, int planes, int ny, int pitch, int elem, int cols, int rows)
{
    // looked up once: the driver's entry point, without linking against it
    static const PFN_cuTensorMapEncodeTiled_v12000 encode = [] {
        void* fn = nullptr;
        cudaDriverEntryPointQueryResult found;
        const cudaError_t e = cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &found);
        return e == cudaSuccess && found == cudaDriverEntryPointSuccess
                   ? reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(fn)
                   : nullptr;
    }();
    if (!encode) return cudaErrorNotSupported;
    const cuuint64_t dims[3] = {cuuint64_t(pitch), cuuint64_t(ny), cuuint64_t(planes)};
    const cuuint64_t strides[2] = {cuuint64_t(pitch) * elem, cuuint64_t(pitch) * cuuint64_t(ny) * elem};
    const cuuint32_t box[3] = {cuuint32_t(cols), cuuint32_t(rows), 1};
    const cuuint32_t steps[3] = {1, 1, 1};
    const CUresult r = encode(map, elem == 4 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_UINT16, 3, base,
                              dims, strides, box, steps, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                              CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

cudaError_t pair_tensor_map(CUtensorMap* map, void* pop, int ny, int pitch, int precision, int warps)
{
    const bool f32 = precision == kFP32;
    return rows_tensor_map(map, pop, kPlanes, ny, pitch, f32 ? 4 : 2, f32 ? kBoxCols<float> : kBoxCols<__half>, warps);
}

cudaError_t launch_step_pair(const PairArgs& p, const CUtensorMap& map, int grid, int warps, int precision, bool rescale,
                             cudaStream_t s)
{
    const cudaError_t e = instance(precision, rescale, warps, Launch{p, map, grid, s});
    if (e != cudaSuccess) return e;
    return cudaGetLastError();
}

}  // namespace lbm
