// lbm_scalar.cu -- scalar-only steps on a stored velocity field.
//
// The paper's own workflow (section "Results"): the flow reaches its steady
// state quickly, so the stationary velocity field of each valve state is
// computed once and the advection-diffusion solver reads it, with a larger
// time step for the scalar (the field is rescaled by the ratio of the time
// steps).  A step of the scalar lattice is pull-stream of g with bounce-back,
// held concentration / do-nothing at open ports, and BGK relaxation towards
// the equilibrium of Eq. cdeequilibrium with the stored (scaled) velocity.
// The kernels of one step (scalar_frozen_regs, scalar_frozen_bulk) read 5 scalar
// populations and the 2 velocity components per fluid node and write 5
// populations: 48 bytes, against 112 for the coupled step.
// scalar_frozen_levels takes three steps a launch, which move that once.
#include "lbm_device.cuh"

namespace lbm {
namespace {

// Completion of an open port node, node n of the pair g (node k of its quad),
// with velocity ux, uy.  Returns true for an outlet node.
template <typename Own>
__device__ __forceinline__ bool scalar_port(float2 (&p)[5], int n, bool west, const RowBC& b, float ux, float uy,
                                            const ScalarArgs& a, const Own& own, int k)
{
    float g[5];
#pragma unroll
    for (int i = 0; i < 5; ++i) g[i] = at(p[i], n);
    const int gi = west ? 1 : 3;
    const int kind = (b.chan_kind >> 8) & 0xFF;
    if (kind == 0) {  // held concentration
        float others = 0.f;
#pragma unroll
        for (int i = 0; i < 5; ++i)
            if (i != gi) others += g[i];
        g[gi] = b.c - others;
    } else {          // do-nothing
        g[gi] = own(gi, k);
        if (kind == 3) {  // the paper's inlet: scaled to C_in
            const float Cs = ((g[0] + g[1]) + (g[2] + g[3])) + g[4];
            if (Cs > 0.f) {
                const float gc = b.c / Cs;
#pragma unroll
                for (int i = 0; i < 5; ++i) g[i] *= gc;
            } else {
                const float c1 = a.wg1 * b.c, cx = c1 * a.inv_cs2g * ux, cy = c1 * a.inv_cs2g * uy;
                g[0] = b.c - 4.f * c1;
                g[1] = c1 + cx;
                g[3] = c1 - cx;
                g[2] = c1 + cy;
                g[4] = c1 - cy;
            }
        }
    }
#pragma unroll
    for (int i = 0; i < 5; ++i) at(p[i], n) = g[i];
    return kind != 0 && kind != 3;
}

// Ports and relaxation of one lane's quad.  v: the pulled scalar populations,
// walls bounced back, on entry, the post-collision ones on exit; ux4, uy4: the
// stored field at the quad; own(i, k): the stored population i of node k; sc,
// sq: the quad's scalar and outlet-flux sums.  kPorts = false: none of the
// nodes is a port; kAllFluid: none of them is solid either (the selects of the
// solid nodes are a third of the instructions).  The relaxation takes two nodes
// an instruction (packed arithmetic: the levels kernel 13.4 -> 13.0 us a step).
template <bool kPorts, bool kAllFluid = false, typename Own>
__device__ __forceinline__ void scalar_nodes(float4 (&v)[5], unsigned lk, int x0, const RowBC& bw, const RowBC& be,
                                             float4 ux4, float4 uy4, const ScalarArgs& a, const Own& own, float& tc,
                                             float& tq, bool& bad)
{
    const bool open_w = kPorts && bw.x >= 0 && ((a.open_mask >> (bw.chan_kind & 31)) & 1u);
    const bool open_e = kPorts && be.x >= 0 && ((a.open_mask >> (be.chan_kind & 31)) & 1u);
    const float2 wg = two(a.omega_g);
#pragma unroll
    for (int h = 0; h < 4; h += 2) {
        float2 g[5];
        const float2 ux = mul2(two(a.u_scale), make_float2(at(ux4, h), at(ux4, h + 1)));
        const float2 uy = mul2(two(a.u_scale), make_float2(at(uy4, h), at(uy4, h + 1)));
        bool fluid[2], pressure_node[2] = {false, false};
#pragma unroll
        for (int n = 0; n < 2; ++n) {
            const int k = h + n;
            fluid[n] = kAllFluid || ((lk >> (8 * k)) & 0xFFu) != kSolid;
#pragma unroll
            for (int i = 0; i < 5; ++i) at(g[i], n) = fluid[n] ? at(v[i], k) : 0.f;
            const int xk = x0 + k;
            const bool pw = open_w && bw.x == xk;
            const bool pe = !pw && open_e && be.x == xk;
            if (pw || pe) pressure_node[n] = scalar_port(g, n, pw, pw ? bw : be, at(ux, n), at(uy, n), a, own, k);
        }
        // the node form's arithmetic on two nodes an instruction, its products fused
        // into sums as the compiler fuses them there
        const float2 C = add2(add2(add2(g[0], g[1]), add2(g[2], g[3])), g[4]);
        const float2 c1 = mul2(two(a.wg1), C), ci = mul2(c1, two(a.inv_cs2g)), nci = mul2(c1, two(-a.inv_cs2g));
        g[0] = fma2(wg, sub2(fma2(two(-4.f), c1, C), g[0]), g[0]);
        g[1] = fma2(wg, sub2(fma2(ci, ux, c1), g[1]), g[1]);
        g[3] = fma2(wg, sub2(fma2(nci, ux, c1), g[3]), g[3]);
        g[2] = fma2(wg, sub2(fma2(ci, uy, c1), g[2]), g[2]);
        g[4] = fma2(wg, sub2(fma2(nci, uy, c1), g[4]), g[4]);
        if (a.decay != 0.f) {  // reaction term R = -k C of Eq. cde, as w_i R
            const float2 R = mul2(two(-a.decay), C);
            g[0] = fma2(two(a.wg0), R, g[0]);
#pragma unroll
            for (int i = 1; i < 5; ++i) g[i] = fma2(two(a.wg1), R, g[i]);
        }
#pragma unroll
        for (int n = 0; n < 2; ++n) {
#pragma unroll
            for (int i = 0; i < 5; ++i) at(v[i], h + n) = at(g[i], n);
            if (!fluid[n]) continue;
            bad |= !(fabsf(at(C, n)) < INFINITY);
            tc += at(C, n);
            if (pressure_node[n]) tq += at(C, n) * at(ux, n);
        }
    }
}

// Bounce-back, ports, relaxation and stores of one lane's quad.  v: the
// streamed scalar populations; sc, sq: the lane's scalar and outlet-flux sums.
__device__ __forceinline__ void scalar_quad(float4 (&v)[5], unsigned lk, int x0, const RowBC& bw, const RowBC& be,
                                            float4 ux4, float4 uy4, const ScalarArgs& a, const float* S, long long P,
                                            long long oC, KahanF& sc, KahanF& sq, bool& bad)
{
    // ---- no-flux walls: halfway bounce-back of g ----
    unsigned wall = 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const unsigned lb = (lk >> (8 * k)) & 0xFFu;
        if (lb != kSolid) wall |= lb;
    }
#pragma unroll
    for (int i = 1; i <= 4; ++i) {
        if (wall & (1u << (i - 1))) {
            const float4 own = ldg4(S + opp(i) * P + oC);
#pragma unroll
            for (int k = 0; k < 4; ++k)
                if ((lk >> (8 * k + i - 1)) & 1u) at(v[i], k) = at(own, k);
        }
    }
    float tc = 0.f, tq = 0.f;
    scalar_nodes<true>(v, lk, x0, bw, be, ux4, uy4, a, [&](int i, int k) { return __ldg(S + i * P + oC + k); }, tc, tq, bad);
    sc.add(tc);
    if (tq != 0.f) sq.add(tq);
#pragma unroll
    for (int i = 0; i < 5; ++i) stg4(a.dst + i * P + oC, v[i]);
}

// The block's scalar and outlet-flux sums into slots 1 and 3 of its
// partials (and the bookkeeping of the slots of the coupled step's grid).
__device__ __forceinline__ void scalar_partials(const ScalarArgs& a, const KahanF& sc, const KahanF& sq)
{
    if (a.partials == nullptr) return;  // a step whose diagnostics nothing reads (uniform over the grid)
    __shared__ DF red[32][2];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const DF s1 = warp_sum(sc.pair()), s3 = warp_sum(sq.pair());
    if (lane == 0) {
        red[warp][0] = s1;
        red[warp][1] = s3;
    }
    __syncthreads();
    if (threadIdx.x < 2) {
        DF sum = red[0][threadIdx.x];
        for (int w = 1; w < int(blockDim.x >> 5); ++w) sum = df_add(sum, red[w][threadIdx.x]);
        a.partials[blockIdx.x * 4 + 1 + 2 * threadIdx.x] = make_float2(sum.hi, sum.lo);
        for (int b = blockIdx.x + gridDim.x; b < a.n_partials; b += gridDim.x)
            a.partials[b * 4 + 1 + 2 * threadIdx.x] = make_float2(0.f, 0.f);
        // blocks beyond the last coupled step's grid hold no fluid partial
        if (int(blockIdx.x) >= a.fluid_blocks) a.partials[blockIdx.x * 4 + 2 * threadIdx.x] = make_float2(0.f, 0.f);
    }
}

// The kernel: a producer warp streams each tile's 5 scalar plane rows
// (with the halos of the shifted directions), its 2 stored velocity rows,
// its wall-link bytes and port entries into a ring of shared-memory stages
// with cp.async.bulk copies completing on mbarriers; consumer warps compute
// from shared memory.  The same stage ring as the coupled step's
// coupled_step_bulk (each consumer owns its stages; bounded waits set bit 1
// of the error word).
struct __align__(16) ScalarStage {
    float pl[5][kRowFloats];
    float u[2][kTileNodes];
    unsigned links[kTileNodes / 4];
    RowBC bc[2];
    uint2 tile;
    uint2 pad;
};
static_assert(sizeof(ScalarStage) % 16 == 0 && offsetof(ScalarStage, u) % 16 == 0 &&
                  offsetof(ScalarStage, links) % 16 == 0 && offsetof(ScalarStage, bc) % 16 == 0,
              "bulk-copy targets");

__global__ void __launch_bounds__(kBulkMaxThreads, 2) scalar_frozen_bulk(const ScalarArgs a, int per)
{
    extern __shared__ __align__(128) unsigned char smem[];
    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    const int nc = (blockDim.x >> 5) - 1;  // consumer warps; the last warp produces
    const int n_stages = nc * per;
    ScalarStage* st = reinterpret_cast<ScalarStage*>(smem);
    uint64_t* full = reinterpret_cast<uint64_t*>(smem + size_t(n_stages) * sizeof(ScalarStage));
    uint64_t* empty = full + n_stages;
    const long long P = a.plane;
    const float* __restrict__ S = a.src;
    const int G = int(gridDim.x);
    const int n_items = int(blockIdx.x) < a.n_tiles ? (a.n_tiles - 1 - int(blockIdx.x)) / G + 1 : 0;

    if (threadIdx.x == 0) {
        for (int s = 0; s < n_stages; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        mbar_fence_init();
    }
    __syncthreads();
    grid_dependency_sync();

    KahanF sc, sq;
    bool bad = false;
    if (warp == nc) {
        // producer: lane l owns stage (l % nc) * per + l / nc (see coupled_step_bulk)
        const bool mine = lane < n_stages;
        const int s = (lane % nc) * per + lane / nc;
        int last_use = -1;
        for (int batch = 0, base = 0; base < n_items; ++batch, base += n_stages) {
            const int j = base + lane;
            bool good = true;
            if (mine && j < n_items) {
                const uint2 tile = tile_at(a.tiles, a.n_tiles, int(blockIdx.x) + j * G, a.reverse);
                if (batch > 0 && !mbar_wait(&empty[s], uint32_t(batch - 1) & 1u)) {
                    good = false;
                } else {
                    const int y = int(tile.x >> kColBits);
                    const int x0 = tile_x0(tile);
                    const int q0 = int(tile.y & 0xFFu), q1 = int((tile.y >> 8) & 0xFFu);
                    const int us = x0 + 4 * q0, ue = x0 + 4 * q1 + 4;
                    const int ss = us - 4 > 0 ? us - 4 : 0;
                    const int se = ue + 4 < a.pitch ? ue + 4 : a.pitch;
                    const long long rC = (long long)y * a.pitch;
                    const long long rS = (long long)(y > 0 ? y - 1 : y) * a.pitch;
                    const long long rN = (long long)(y + 1 < a.ny ? y + 1 : y) * a.pitch;
                    // directions 0, 2, 4 copy the lanes' span, 1 and 3 one quad more on
                    // each side; the two velocity rows the lanes' span
                    const uint32_t bytes = uint32_t(5 * (ue - us) + 2 * (se - ss)) * 4u + kTileNodes + 2 * sizeof(RowBC);
                    st[s].tile = tile;
                    mbar_arrive_expect_tx(&full[s], bytes);
#pragma unroll
                    for (int i = 0; i < 5; ++i) {
                        const int p = 9 + i;
                        const long long r = src_row(p) == 0 ? rC : src_row(p) == 1 ? rS : rN;
                        const int b = src_col(p) == 0 ? us : ss;
                        const int e = src_col(p) == 0 ? ue : se;
                        bulk_g2s(&st[s].pl[i][b - x0 + 4], S + i * P + r + b, uint32_t(e - b) * 4u, &full[s]);
                    }
                    bulk_g2s(&st[s].u[0][us - x0], a.ux + rC + us, uint32_t(ue - us) * 4u, &full[s]);
                    bulk_g2s(&st[s].u[1][us - x0], a.uy + rC + us, uint32_t(ue - us) * 4u, &full[s]);
                    bulk_g2s(st[s].links, a.links + rC + x0, kTileNodes, &full[s]);
                    bulk_g2s(&st[s].bc[0], a.rowbc + y, sizeof(RowBC), &full[s]);
                    bulk_g2s(&st[s].bc[1], a.rowbc + a.ny + y, sizeof(RowBC), &full[s]);
                    last_use = batch;
                }
            }
            if (!__all_sync(kFull, good)) {
                if (lane == 0) atomicOr(a.err, 2u);
                break;
            }
        }
        if (mine && last_use >= 0 && !mbar_wait(&full[s], uint32_t(last_use) & 1u)) atomicOr(a.err, 2u);
        __syncwarp();
    } else {
        for (int k = 0, j = warp; j < n_items; ++k, j += nc) {
            const int s = warp * per + k % per;
            const uint32_t use = uint32_t(k / per);
            if (!__all_sync(kFull, mbar_wait(&full[s], use & 1u))) {
                if (lane == 0) atomicOr(a.err, 2u);
                break;
            }
            const ScalarStage& sg = st[s];
            const uint2 tile = sg.tile;
            const int y = int(tile.x >> kColBits);
            const int x0 = tile_x0(tile) + 4 * lane;
            const long long oC = (long long)y * a.pitch + x0;
            const unsigned lk = sg.links[lane];
            const bool act = lk != 0xFFFFFFFFu;
            const RowBC bw = sg.bc[0], be = sg.bc[1];
            float4 v[5], ux4 = make_float4(0.f, 0.f, 0.f, 0.f), uy4 = ux4;
            if (act) {
#pragma unroll
                for (int i = 0; i < 5; ++i) {
                    const float* row = sg.pl[i] + 4 * lane;
                    const float4 c = *reinterpret_cast<const float4*>(row + 4);
                    if (src_col(9 + i) == 0) v[i] = c;
                    else if (src_col(9 + i) == 1) v[i] = make_float4(row[3], c.x, c.y, c.z);
                    else v[i] = make_float4(c.y, c.z, c.w, row[8]);
                }
                ux4 = *reinterpret_cast<const float4*>(&sg.u[0][4 * lane]);
                uy4 = *reinterpret_cast<const float4*>(&sg.u[1][4 * lane]);
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&empty[s]);  // the stage may be refilled
            if (act) scalar_quad(v, lk, x0, bw, be, ux4, uy4, a, S, P, oC, sc, sq, bad);
        }
        if (__any_sync(kFull, bad) && lane == 0) atomicOr(a.err, 1u);
    }
    scalar_partials(a, sc, sq);
}

// The register variant: each warp pulls its tile's five scalar planes with
// 128-bit loads and warp shuffles (as coupled_step_regs does for all
// fourteen) and the stored field of its nodes; 20 live floats per lane
// instead of 56 leave room for many warps per SM, which keep the loads in
// flight without a shared-memory pipeline.
__global__ void __launch_bounds__(128) scalar_frozen_regs(const ScalarArgs a)
{
    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    const int wpb = blockDim.x >> 5;
    const long long P = a.plane;
    const float* __restrict__ S = a.src;
    KahanF sc, sq;
    bool bad = false;
    grid_dependency_sync();
    for (int t = blockIdx.x * wpb + warp; t < a.n_tiles; t += gridDim.x * wpb) {
        const uint2 tile = tile_at(a.tiles, a.n_tiles, t, a.reverse);
        const int y = int(tile.x >> kColBits);
        const int x0 = tile_x0(tile) + 4 * lane;
        const long long oC = (long long)y * a.pitch + x0;
        const long long oS = (long long)(y > 0 ? y - 1 : y) * a.pitch + x0;
        const long long oN = (long long)(y + 1 < a.ny ? y + 1 : y) * a.pitch + x0;
        const int halo_w = x0 > 0 ? -1 : 0;
        const int halo_e = x0 + 4 < a.pitch ? 4 : 3;
        const unsigned lk = __ldg(reinterpret_cast<const unsigned*>(a.links + oC));
        // loads from the tile's fluid range, beside the wall-link word (see
        // load_range)
        const LoadRange r = load_range(tile, lane);
        float4 v[5];
        pull_quad<false, float, 9, 5>(v, S, P, oC, oS, oN, halo_w, halo_e, r.own, r.west, r.east, lane);
        const float4 ux4 = r.own ? ldg4(a.ux + oC) : make_float4(0.f, 0.f, 0.f, 0.f);
        const float4 uy4 = r.own ? ldg4(a.uy + oC) : make_float4(0.f, 0.f, 0.f, 0.f);
        const bool act = lk != 0xFFFFFFFFu;
        if (!act) continue;
        const RowBC bw = a.rowbc[y];
        const RowBC be = a.rowbc[a.ny + y];
        scalar_quad(v, lk, x0, bw, be, ux4, uy4, a, S, P, oC, sc, sq, bad);
    }
    if (__any_sync(kFull, bad) && lane == 0) atomicOr(a.err, 1u);
    scalar_partials(a, sc, sq);
}

// ---------------------------------------------------------------------------
// Several steps in one launch
// ---------------------------------------------------------------------------
// kLevels steps of one valve word in one launch, as coupled_step_pair takes
// two (lbm_pair.cu): a block marches along y over a strip of 128 columns, W
// rows an iteration; level l takes a row l - 1 rows behind level 1, from the
// ring of rows level l - 1 has left in shared memory, and the last level
// stores to the destination buffer.  Strips repeat each other's columns and
// rows at their sides and ends, so blocks never wait for each other.  Each
// level spoils one column more from the strip's outer lanes inwards, up to
// kLevels - 2 of the four of a side lane, none of them stored.
// What bounds it: three levels move 49 MB a step on the 4096 x 2048 chip (161
// MB one by one), which HBM would take 8 us for; the levels' turns (barrier,
// gather from shared memory, arithmetic) at 18 warps an SM take 12.5 us (24.8 us
// one step a launch, at 0.95 of the HBM rate; 1024 x 768 3.9 -> 2.7, 256 x 128 2.5 ->
// 1.5).  Nine warps a block are what shared memory holds twice: 8 x 2 takes 13.0 us
// (2000 x 1000 4.6 against 4.2; 1001 x 517 with obstacles 3.7 against 4.1), 10 x 2,
// whose second block no longer fits, 16.6.  Tried before the packed arithmetic
// (8 x 2: 13.4 us): four levels (19.2-20.6 us: shared memory for 10 or 12 warps
// only), five (24.4), 6 warps x 3 blocks (16.7 where 8 x 2 took 16.5), 4 x 4 (17.3).
constexpr int kLevels = kScalarLevels, kScalarW = kScalarWarps;
constexpr int kScalarBox = kTileNodes + 8;  // columns of a staged row: from x0 - 4 on
struct ScalarRow {
    float pl[5][kTileNodes];
};
struct alignas(16) ScalarInfo {  // what every level needs of a row beside populations
    float u[2][kTileNodes];
    unsigned links[kTileNodes / 4];
    RowBC bc[2];
};
struct alignas(128) ScalarSmem {
    struct alignas(128) Box {
        float row[kScalarW][kScalarBox];
    } box[7];                                  // five scalar planes, each at its pull offset, and u_x, u_y
    ScalarRow ring[kLevels - 1][kScalarW + 2];  // ring l - 1: rows of level l
    ScalarInfo info[kScalarW + kLevels - 1];
    struct alignas(16) Stage {
        unsigned links[kTileNodes / 4];
        RowBC bc[2];
    } stage[kScalarW];
    uint64_t full;  // the boxes have arrived
    uint64_t step;  // every warp has left its row of a level: kLevels - 1 phases an iteration
};
static_assert(offsetof(ScalarSmem, ring) % 16 == 0 && offsetof(ScalarSmem, info) % 16 == 0 &&
                  offsetof(ScalarSmem, stage) % 16 == 0 && offsetof(ScalarSmem, full) % 8 == 0 &&
                  sizeof(ScalarSmem::Box) % 128 == 0 && sizeof(ScalarInfo) % 16 == 0 && sizeof(ScalarRow) % 16 == 0 &&
                  offsetof(ScalarInfo, links) % 16 == 0 && offsetof(ScalarInfo, bc) % 16 == 0,
              "targets of vector accesses, copies and barriers");
static_assert(kLevels >= 3 && kLevels <= 5, "with two levels a row would be rewritten while it may still be read");

// Free flight of one lane's quad from three rows (lanes 0 and 31 take no
// value from beyond the strip: see above).
template <typename RowOf>
__device__ __forceinline__ void pull_rows(float4 (&v)[5], const RowOf& row, int lane)
{
#pragma unroll
    for (int i = 0; i < 5; ++i) {
        float4 r = *reinterpret_cast<const float4*>(row(i) + 4 * lane);
        if (src_col(i) == 1) r = make_float4(__shfl_up_sync(kFull, r.w, 1), r.x, r.y, r.z);
        else if (src_col(i) == 2) r = make_float4(r.y, r.z, r.w, __shfl_down_sync(kFull, r.x, 1));
        v[i] = r;
    }
}

__device__ __forceinline__ void bounce_link(float4& v, unsigned lk, int i, const float4& own)
{
#pragma unroll
    for (int k = 0; k < 4; ++k) at(v, k) = (lk >> (8 * k + i - 1)) & 1u ? at(own, k) : at(v, k);
}

__global__ void __launch_bounds__(32 * kScalarW, kScalarBlocks)
    scalar_frozen_levels(const ScalarArgs a, const int4* items, const int* block_first,
                         const __grid_constant__ CUtensorMap map, const __grid_constant__ CUtensorMap umap)
{
    constexpr int W = kScalarW, K = kLevels, R = W + 2, RI = W + K - 1;
    extern __shared__ __align__(128) unsigned char smem[];
    ScalarSmem& sm = *reinterpret_cast<ScalarSmem*>(smem);
    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    const int reverse = a.reverse, pitch = a.pitch, ny = a.ny;
    const long long P = a.plane;
    ScalarSmem::Stage& stage = sm.stage[warp];
    bool bad = false, late = false;

    if (threadIdx.x == 0) {
        mbar_init(&sm.full, 1);
        mbar_init(&sm.step, W);
        mbar_fence_init();
    }
    int i = block_first[blockIdx.x];
    const int i_end = block_first[blockIdx.x + 1];
    int4 st = items[i];
    __syncthreads();
    grid_dependency_sync();

    // march row j of the strip's level 1: rows ya - (K - 1) .. yb + K - 2
    auto row_of = [&](const int4& s, int j) { return reverse ? s.w + K - 2 - j : s.z - (K - 1) + j; };
    auto total = [&](const int4& s) { return s.w - s.z + 2 * (K - 1); };
    auto inside = [&](int y) { return y >= 0 && y < ny; };
    auto issue_boxes = [&](const int4& s, int j) {
        if (threadIdx.x != 0) return;
        const int y = reverse ? row_of(s, j + W - 1) : row_of(s, j);  // lowest row
        mbar_arrive_expect_tx(&sm.full, uint32_t(7 * W * kScalarBox * sizeof(float)));
#pragma unroll
        for (int q = 0; q < 5; ++q)
            tensor_g2s(&sm.box[q], &map, s.x - 4, y - (src_row(q) == 1) + (src_row(q) == 2), 9 + q, &sm.full);
        for (int q = 0; q < 2; ++q) tensor_g2s(&sm.box[5 + q], &umap, s.x - 4, y, q, &sm.full);
    };
    auto issue_row = [&](const int4& s, int y) {
        const int l0 = s.y & 0xFF, l1 = (s.y >> 8) & 0xFF;
        if (lane >= l0 - 1 && lane <= l1 + 1)
            cp_async4(&stage.links[lane], a.links + (long long)y * pitch + s.x + 4 * lane);
        if ((s.y & kPairPort) && lane < 2) cp_async16(&stage.bc[lane], a.rowbc + (lane == 0 ? y : ny + y));
        asm volatile("cp.async.commit_group;" ::: "memory");
    };

    unsigned issued = 1, phase = 0;
    issue_boxes(st, 0);
    bool here = inside(row_of(st, warp)) && warp < total(st);
    if (here) issue_row(st, row_of(st, warp));

    int base = 0;             // first march row of the iteration
    int sp = warp, ip = warp;  // ring and info slots of the warp's level-1 row
    for (unsigned t = 0;; ++t) {
        const int j = base + warp, n_rows = total(st);
        const int l0 = st.y & 0xFF, l1 = (st.y >> 8) & 0xFF;
        const bool port = st.y & kPairPort;
        const int x0 = st.x + 4 * lane;
        int4 nst = st;
        int nbase = base + W;
        bool more = true;
        if (nbase >= n_rows) {
            nbase = 0;
            more = i + 1 < i_end;
            if (more) nst = items[i + 1];
        }
        const int yn = row_of(nst, nbase + warp);
        const bool next = more && nbase + warp < total(nst) && inside(yn);

        // ---- level 1, from the boxes ----
        if (!late) late = !mbar_wait(&sm.full, t & 1u);
        float4 v[5], ux4, uy4;
        unsigned lk = 0xFFFFFFFFu;
        RowBC bc[2];
        const int y1 = row_of(st, j), r = reverse ? W - 1 - warp : warp;
        if (here) {
            asm volatile("cp.async.wait_group 0;" ::: "memory");
            __syncwarp();
            auto row = [&](int q) { return &sm.box[q].row[r][4]; };
            pull_rows(v, row, lane);
            if (lane == 0) v[1].x = sm.box[1].row[r][3];
            if (lane == 31) v[3].w = sm.box[3].row[r][4 + kTileNodes];
            ux4 = *reinterpret_cast<const float4*>(row(5) + 4 * lane);
            uy4 = *reinterpret_cast<const float4*>(row(6) + 4 * lane);
            if (lane >= l0 - 1 && lane <= l1 + 1) lk = stage.links[lane];
            if (port) {
                bc[0] = stage.bc[0];
                bc[1] = stage.bc[1];
            }
        }
        late = __any_sync(kFull, late);
        if (next && !late) issue_row(nst, yn);
        ScalarInfo& info = sm.info[ip];
        if (here) {
            // this warp was the slot's last reader (level K of the iteration before)
            *reinterpret_cast<float4*>(&info.u[0][4 * lane]) = ux4;
            *reinterpret_cast<float4*>(&info.u[1][4 * lane]) = uy4;
            info.links[lane] = lk;
            if (port && lane < 2) info.bc[lane] = lane == 0 ? bc[0] : bc[1];
        }
        const bool open1 = __all_sync(kFull, lk == 0u || lk == 0xFFFFFFFFu);  // a row without walls
        if (lk != 0xFFFFFFFFu && open1) {
            float tc = 0.f, tq = 0.f;
            bool b = false;
            scalar_nodes<false, true>(v, lk, x0, RowBC{}, RowBC{}, ux4, uy4, a, [](int, int) { return 0.f; }, tc, tq, b);
            bad |= b && lane >= l0 && lane <= l1;
        } else if (lk != 0xFFFFFFFFu) {
            // walls: along the row from the box, which holds the row's own values of
            // directions 1 and 3; across it from global memory
            const float4 g1 = *reinterpret_cast<const float4*>(&sm.box[1].row[r][4 + 4 * lane]);
            const float4 g3 = *reinterpret_cast<const float4*>(&sm.box[3].row[r][4 + 4 * lane]);
            unsigned wall = 0;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const unsigned lb = (lk >> (8 * k)) & 0xFFu;
                if (lb != kSolid) wall |= lb;
            }
            if (wall & 0x5u) {
                bounce_link(v[1], lk, 1, g3);
                bounce_link(v[3], lk, 3, g1);
            }
            if (wall & 0xAu) {
                const long long o = (long long)y1 * pitch + x0;
                const float4 g4 = ldg4(a.src + 4 * P + o), g2 = ldg4(a.src + 2 * P + o);
                bounce_link(v[2], lk, 2, g4);
                bounce_link(v[4], lk, 4, g2);
            }
            float tc = 0.f, tq = 0.f;
            bool b = false;
            auto own = [&](int q, int k) { return q == 1 ? at(g1, k) : at(g3, k); };
            if (port) scalar_nodes<true>(v, lk, x0, bc[0], bc[1], ux4, uy4, a, own, tc, tq, b);
            else scalar_nodes<false>(v, lk, x0, RowBC{}, RowBC{}, ux4, uy4, a, own, tc, tq, b);
            bad |= b && lane >= l0 && lane <= l1;
        }
        if (lk != 0xFFFFFFFFu) {
            ScalarRow& out = sm.ring[0][sp];
#pragma unroll
            for (int q = 0; q < 5; ++q) *reinterpret_cast<float4*>(&out.pl[q][4 * lane]) = v[q];
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(&sm.step);
        if (!late) late = !mbar_wait(&sm.step, phase & 1u);
        ++phase;
        if (more && !late) {  // every warp has pulled its row from the boxes
            issue_boxes(nst, nbase);
            ++issued;
        }

        // ---- levels 2 .. K: row j - (l - 1) from the ring of level l - 1 ----
#pragma unroll
        for (int l = 2; l <= K; ++l) {
            const int jl = j - (l - 1), yl = row_of(st, jl);
            const bool on = j >= 2 * (l - 1) && j < n_rows && inside(yl);
            int sc = sp - (l - 1), ic = ip - (l - 1);  // slots of row j - (l - 1)
            if (sc < 0) sc += R;
            if (ic < 0) ic += RI;
            const int sa = sc == R - 1 ? 0 : sc + 1, sb = sc == 0 ? R - 1 : sc - 1;  // rows one on and one back
            lk = 0xFFFFFFFFu;
            if (on) {
                const ScalarRow* ring = sm.ring[l - 2];
                const ScalarInfo& in = sm.info[ic];
                const ScalarRow& rS = ring[reverse ? sa : sb];
                const ScalarRow& rN = ring[reverse ? sb : sa];
                const ScalarRow& rC = ring[sc];
                auto row = [&](int q) { return src_row(q) == 0 ? rC.pl[q] : src_row(q) == 1 ? rS.pl[q] : rN.pl[q]; };
                pull_rows(v, row, lane);
                const int w = l < K ? 1 : 0;
                if (lane >= l0 - w && lane <= l1 + w) lk = in.links[lane];
                ux4 = *reinterpret_cast<const float4*>(&in.u[0][4 * lane]);
                uy4 = *reinterpret_cast<const float4*>(&in.u[1][4 * lane]);
                float tc = 0.f, tq = 0.f;
                bool b = false;
                if (__all_sync(kFull, lk == 0u || lk == 0xFFFFFFFFu)) {
                    if (lk == 0u)
                        scalar_nodes<false, true>(v, lk, x0, RowBC{}, RowBC{}, ux4, uy4, a, [](int, int) { return 0.f; }, tc,
                                                  tq, b);
                } else if (lk != 0xFFFFFFFFu) {
                    unsigned wall = 0;
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const unsigned lb = (lk >> (8 * k)) & 0xFFu;
                        if (lb != kSolid) wall |= lb;
                    }
                    if (wall & 0xFu) {
#pragma unroll
                        for (int q = 1; q <= 4; ++q)
                            bounce_link(v[q], lk, q, *reinterpret_cast<const float4*>(&rC.pl[opp(q)][4 * lane]));
                    }
                    auto own = [&](int q, int k) { return rC.pl[q][4 * lane + k]; };
                    if (port) scalar_nodes<true>(v, lk, x0, in.bc[0], in.bc[1], ux4, uy4, a, own, tc, tq, b);
                    else scalar_nodes<false>(v, lk, x0, RowBC{}, RowBC{}, ux4, uy4, a, own, tc, tq, b);
                }
                bad |= b && lane >= l0 && lane <= l1 && yl >= st.z && yl < st.w;
            }
            if (l < K) {
                if (lk != 0xFFFFFFFFu) {
                    ScalarRow& out = sm.ring[l - 1][sc];
#pragma unroll
                    for (int q = 0; q < 5; ++q) *reinterpret_cast<float4*>(&out.pl[q][4 * lane]) = v[q];
                }
                __syncwarp();
                if (lane == 0) mbar_arrive(&sm.step);
                if (!late) late = !mbar_wait(&sm.step, phase & 1u);
                ++phase;
            } else if (lk != 0xFFFFFFFFu) {
                float* const D = a.dst + (long long)yl * pitch + x0;
#pragma unroll
                for (int q = 0; q < 5; ++q) stg4(D + q * P, v[q]);
            }
        }
        if (!more) break;
        if (nbase == 0) ++i;
        st = nst;
        base = nbase;
        here = next;
        sp += W;
        if (sp >= R) sp -= R;
        ip += W;
        if (ip >= RI) ip -= RI;
    }
    if (late) {
        // no copy may still be writing this block's shared memory at exit
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        mbar_wait(&sm.full, (issued - 1) & 1u);
        atomicOr(a.err, 2u);
    }
    if (__any_sync(kFull, bad) && lane == 0) atomicOr(a.err, 1u);
}

// Velocity of the stored populations (f as deviations) into two planes.
__global__ void velocity_of_state(const float* pop, const uint8_t* links, long long plane, int n, float* ux,
                                  float* uy)
{
    for (long long o = blockIdx.x * (long long)blockDim.x + threadIdx.x; o < plane;
         o += (long long)gridDim.x * blockDim.x) {
        float vx = 0.f, vy = 0.f;
        if (links[o] != kSolid) {
            float f[9];
#pragma unroll
            for (int i = 0; i < 9; ++i) f[i] = pop[i * plane + o];
            const float rho = 1.f + (((f[0] + f[1]) + (f[2] + f[3])) + ((f[4] + f[5]) + (f[6] + f[7])) + f[8]);
            vx = ((f[1] - f[3]) + (f[5] - f[6]) + (f[8] - f[7])) / rho;
            vy = ((f[2] - f[4]) + (f[5] + f[6]) - (f[7] + f[8])) / rho;
        }
        ux[o] = vx;
        uy[o] = vy;
    }
    (void)n;
}

}  // namespace

size_t scalar_bulk_smem_bytes(int stages)
{
    return size_t(stages) * (sizeof(ScalarStage) + 2 * sizeof(uint64_t));
}

cudaError_t launch_scalar_step_bulk(const ScalarArgs& a, int grid, int consumers, int per, cudaStream_t s)
{
    static_assert(kBulkMaxThreads >= 32 * 8, "block of up to 7 consumers and a producer");
    cudaError_t e = cudaFuncSetAttribute(scalar_frozen_bulk, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         int(scalar_bulk_smem_bytes(kMaxStages)));
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(32 * (consumers + 1));
    cfg.dynamicSmemBytes = scalar_bulk_smem_bytes(consumers * per);
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    e = cudaLaunchKernelEx(&cfg, scalar_frozen_bulk, a, per);
    if (e != cudaSuccess) return e;
    return cudaGetLastError();
}

cudaError_t scalar_bulk_occupancy(int consumers, int per, int* blocks_per_sm)
{
    cudaError_t e = cudaFuncSetAttribute(scalar_frozen_bulk, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         int(scalar_bulk_smem_bytes(kMaxStages)));
    if (e != cudaSuccess) return e;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, scalar_frozen_bulk, 32 * (consumers + 1),
                                                         scalar_bulk_smem_bytes(consumers * per));
}

cudaError_t launch_scalar_step_regs(const ScalarArgs& a, int grid, int block, cudaStream_t s)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cudaError_t e = cudaLaunchKernelEx(&cfg, scalar_frozen_regs, a);
    if (e != cudaSuccess) return e;
    return cudaGetLastError();
}

cudaError_t scalar_regs_occupancy(int block, int* blocks_per_sm)
{
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, scalar_frozen_regs, block, 0);
}

int scalar_level_warps() { return kScalarW; }

cudaError_t scalar_tensor_map(CUtensorMap* map, void* base, int planes, int ny, int pitch)
{
    return rows_tensor_map(map, base, planes, ny, pitch, sizeof(float), kScalarBox, kScalarW);
}

cudaError_t scalar_levels_occupancy(int* blocks_per_sm)
{
    cudaError_t e = cudaFuncSetAttribute(scalar_frozen_levels, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         int(sizeof(ScalarSmem)));
    if (e != cudaSuccess) return e;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, scalar_frozen_levels, 32 * kScalarW,
                                                         sizeof(ScalarSmem));
}

cudaError_t launch_scalar_levels(const ScalarArgs& a, const int4* items, const int* block_first, int grid,
                                 const CUtensorMap& map, const CUtensorMap& umap, cudaStream_t s)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(32 * kScalarW);
    cfg.dynamicSmemBytes = sizeof(ScalarSmem);
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cudaError_t e = cudaLaunchKernelEx(&cfg, scalar_frozen_levels, a, items, block_first, map, umap);
    if (e != cudaSuccess) return e;
    return cudaGetLastError();
}

cudaError_t launch_velocity_of_state(const float* pop, const uint8_t* links, long long plane, float* ux, float* uy,
                                     cudaStream_t s)
{
    const int block = 256;
    const long long want = (plane + block - 1) / block;
    velocity_of_state<<<int(want < 65536 ? want : 65536), block, 0, s>>>(pop, links, plane, 0, ux, uy);
    return cudaGetLastError();
}

}  // namespace lbm
