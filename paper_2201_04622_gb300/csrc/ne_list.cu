// ne_list.cu -- neighbour-list build of the multi-kernel path.
//
// Rebuild of the candidate list of every replica whose flag is set (or of all
// replicas, when forced), in two launches (three with a replica above
// SORT_IN_BLOCK atoms, four of them forced) that return at once when there is
// nothing to do:
//   k_nl_cells  reference positions (the lattice sites at the start of a run,
//               the current positions after an atom strayed more than
//               skin / 2), wrapped and binned into cells of edge > r_c + skin.
//               One thread per atom over all SMs; the block that finishes a
//               replica's last tile forms its cell starts and writes the atoms
//               sorted by cell, each cell's by index, so the order does not
//               depend on the atomics.  Replicas above SORT_IN_BLOCK are
//               sorted, and in a forced build scattered, by launches over all
//               SMs (k_nl_sort, k_nl_scatter);
//   k_nl_list   for each atom the atoms of the 27 surrounding cells (all atoms
//               when the box holds < 3 cells per axis) within r_c + skin,
//               minimum image, FP32 distances with a 1e-3 A margin so that
//               rounding never drops a pair.
#include <type_traits>

#include "ne_internal.cuh"

namespace {

constexpr int CELL_THREADS = 1024;
constexpr int CELL_TILES = CELL_THREADS / NE_TILE;

// replicas above this size have their cells sorted by a launch of its own
// (k_nl_sort): with one block's pass over 70,304 atoms the FP64 energy call
// took 1049 us, with the launch 973; below, the launch, paid at every step,
// costs more than it saves
constexpr int SORT_IN_BLOCK = 16384;

// Atoms first, first + step, ... (in cell order) of a replica into the sorted
// copy: an atom's place in its cell is the number of lower indices there.
__device__ __forceinline__ void rank_cells(const DevBatch& B, int rep, int first, int step)
{
    const RepDev& P = B.rep[rep];
    const int n = P.n, off = P.off;
    const int* start = B.cstart + P.cell_off + rep;
    for (int p = first; p < n; p += step) {
        const int a = B.craw[off + p];
        const int c = __ldcg(&B.cellof[off + a]);
        const float4 x = __ldcg(&B.pbuild[off + a]);
        const int lo = start[c], hi = start[c + 1];
        int r = 0;
#pragma unroll 4
        for (int q = lo; q < hi; ++q) r += B.craw[off + q] < a;
        B.csort[off + lo + r] = make_float4(x.x, x.y, x.z, __int_as_float(a));
    }
}

// Cell starts and the atoms by cell (and, for a replica that one block sorts,
// the sorted copy) of one replica whose atoms are all counted, by the whole
// block.
__device__ void sort_cells(const DevBatch& B, int rep, bool scatter, int* s_warp)
{
    const RepDev& P = B.rep[rep];
    const int tid = threadIdx.x, n = P.n, off = P.off;
    const int ncell = P.nc[0] * P.nc[1] * P.nc[2];
    int* start = B.cstart + P.cell_off + rep;  // ncell + 1 entries
    int* count = B.ccount + P.cell_off;
    // exclusive scan of the counts: each thread a contiguous chunk of cells,
    // warp scans over the chunk totals, then over the warps
    const int per = (ncell + CELL_THREADS - 1) / CELL_THREADS;
    const int c0 = min(ncell, tid * per), c1 = min(ncell, c0 + per);
    int tot = 0;
    for (int c = c0; c < c1; ++c) tot += __ldcg(&count[c]);
    int inc = tot;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, inc, o);
        if ((tid & 31) >= o) inc += v;
    }
    if ((tid & 31) == 31) s_warp[tid >> 5] = inc;
    __syncthreads();
    if (tid < 32) {
        int v = s_warp[tid];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int w = __shfl_up_sync(0xffffffffu, v, o);
            if (tid >= o) v += w;
        }
        s_warp[tid] = v;
    }
    __syncthreads();
    int run = inc - tot + (tid >= 32 ? s_warp[(tid >> 5) - 1] : 0);
    for (int c = c0; c < c1; ++c) {
        const int k = __ldcg(&count[c]);
        start[c] = run;
        run += k;
        count[c] = 0;  // zero for the next build
    }
    if (tid == 0) start[ncell] = n;
    if (!scatter) return;
    __syncthreads();
    for (int a0 = tid; a0 < n; a0 += 8 * CELL_THREADS) {
        int c[8], k[8];  // eight atoms in flight: the chain is cell -> start -> store
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const int a = min(a0 + q * CELL_THREADS, n - 1);
            c[q] = __ldcg(&B.cellof[off + a]);
            k[q] = __ldcg(&B.cslot[off + a]);
        }
#pragma unroll
        for (int q = 0; q < 8; ++q) k[q] += start[c[q]];
#pragma unroll
        for (int q = 0; q < 8; ++q)
            if (a0 + q * CELL_THREADS < n) B.craw[off + k[q]] = a0 + q * CELL_THREADS;
    }
    __syncthreads();
    if (n <= SORT_IN_BLOCK) rank_cells(B, rep, tid, CELL_THREADS);
}

// Bound by latency: one thread per atom does the FP64 wrap and one atomic,
// then the finishing block scans and scatters its replica's atoms.  Before, one
// 512-thread block counted, scanned and sorted each cell by insertion (176 us
// for 65,536 atoms, 40 us for 2000) and one thread an atom walked its cells
// (176 and 253 us).  Whole calls, before and with this build: energy and forces of
// 70,304 atoms in FP64 1232 -> 973 us, energy and gradients of 65,536 atoms 1504
// -> 1091 us, the 200-step spring fit of 2000 atoms at 1400 K 17.0 -> 13.6 ms.
// The image index and, where the cells are wide enough (bin64), the cell in FP32
// took another 8 us of FP64 out.
__global__ void __launch_bounds__(CELL_THREADS) k_nl_cells(DevBatch B, int force, int from_sites)
{
    __shared__ int s_warp[32];
    __shared__ int s_done[CELL_TILES];  // replica whose last tile this block finished, or -1
    const int tl = threadIdx.x / NE_TILE;
    const int tile = blockIdx.x * CELL_TILES + tl;
    ne_chain();
    // (after the wait: in a single-point call the kernel before this one is
    // k_setup, which writes the table)
    const int rep = tile < B.n_tiles ? B.tile_rep[tile] : 0;
    const bool go = tile < B.n_tiles && (force || B.flags[rep] != 0);
    if (!__syncthreads_or(go)) return;
    const RepDev& P = B.rep[rep];
    const int a = (tile - P.tile0) * NE_TILE + threadIdx.x % NE_TILE;
    if (go && a < P.n) {
        const int i = P.off + a;
        const double* X = from_sites ? B.x0 : B.x;
        double w[3];
        float wf[3];
        for (int d = 0; d < 3; ++d) {
            w[d] = X[3 * i + d];
            ne_wrap(w[d], wf[d], P.L[d], P.iLf[d]);
        }
        const float4 p = make_float4(wf[0], wf[1], wf[2], __int_as_float(a));
        B.pbuild[i] = p;
        if (!from_sites) {  // what the pair passes read
            B.pos32[i] = make_float4(p.x, p.y, p.z, __int_as_float(0));
            if (B.pos64) B.pos64[i] = ned4{w[0], w[1], w[2], 0.0};
        }
        if (P.nc[0] == 0) {
            B.csort[i] = p;  // all pairs: the atoms in index order
        } else {
            int c3[3];
            for (int d = 0; d < 3; ++d) {
                const int q = P.bin64 ? (int)(w[d] * P.invL[d] * P.nc[d]) : (int)(wf[d] * P.iLf[d] * (float)P.nc[d]);
                c3[d] = min(max(q, 0), P.nc[d] - 1);
            }
            const int c = (c3[0] * P.nc[1] + c3[1]) * P.nc[2] + c3[2];
            B.cellof[i] = c;
            B.cslot[i] = atomicAdd(&B.ccount[P.cell_off + c], 1);
        }
    }
    __syncthreads();
    if (threadIdx.x % NE_TILE == 0) {
        int done = -1;
        if (go) {
            __threadfence();  // this tile's writes before its ticket
            if (atomicAdd(&B.nl_done[rep], 1u) == (unsigned)P.ntile - 1u) {
                __threadfence();
                B.nl_done[rep] = 0u;
                B.flags[rep] = 0;  // every tile has read it
                B.building[rep] = 1;
                atomicAdd(B.rebuilds, 1ull);
                if (P.nc[0] != 0) done = rep;
            }
        }
        s_done[tl] = done;
    }
    __syncthreads();
    for (int q = 0; q < CELL_TILES; ++q) {
        if (s_done[q] >= 0) sort_cells(B, s_done[q], !(force && B.rep[s_done[q]].n > SORT_IN_BLOCK), s_warp);
        __syncthreads();
    }
}

// the scatter of a forced build of large replicas (the finishing block's own
// takes ~20 us at 65,536 atoms; inside a run, where builds are rare, the launch
// would cost every step)
__global__ void __launch_bounds__(256) k_nl_scatter(DevBatch B)
{
    ne_chain();
    const int tile = blockIdx.x * (256 / NE_TILE) + threadIdx.x / NE_TILE;
    if (tile >= B.n_tiles) return;
    const int rep = B.tile_rep[tile];
    const RepDev& P = B.rep[rep];
    const int a = (tile - P.tile0) * NE_TILE + threadIdx.x % NE_TILE;
    if (P.nc[0] == 0 || P.n <= SORT_IN_BLOCK || a >= P.n) return;
    B.craw[P.off + (B.cstart + P.cell_off + rep)[B.cellof[P.off + a]] + B.cslot[P.off + a]] = a;
}

__global__ void __launch_bounds__(256) k_nl_sort(DevBatch B)
{
    ne_chain();
    const int tile = blockIdx.x * (256 / NE_TILE) + threadIdx.x / NE_TILE;
    if (tile >= B.n_tiles) return;
    const int rep = B.tile_rep[tile];
    const RepDev& P = B.rep[rep];
    if (!B.building[rep] || P.nc[0] == 0 || P.n <= SORT_IN_BLOCK) return;
    rank_cells(B, rep, (tile - P.tile0) * NE_TILE + threadIdx.x % NE_TILE, P.ntile * NE_TILE);
}

// G lanes per atom walk its 27 cells: the z neighbours of a cell are one run
// of the sorted copy (two at the box edge), so the lanes read consecutive
// 16-byte entries, and a ballot packs the lanes' hits in order.  Bound by
// instructions (72 % issue): a run's image is known from its cells, so a
// candidate is three differences and a test, without a nearest-image rounding
// (20 replicas with a 2.6 A skin, ~2000 candidates an atom: 191 -> 123 us).
constexpr int LIST_THREADS = 256;

template <int G>
__device__ void list_block(const DevBatch& B, int blk, int rep)
{
    constexpr int AT = LIST_THREADS / G, SUB = NE_TILE / AT;
    const int tile = blk / SUB;
    if (!B.building[rep]) return;
    const RepDev& P = B.rep[rep];
    const int lane = threadIdx.x % G;
    const int a = (tile - P.tile0) * NE_TILE + (blk % SUB) * AT + threadIdx.x / G;
    const bool valid = a < P.n;
    const int off = P.off, i = off + (valid ? a : 0);
    const float L0 = P.Lf[0], L1 = P.Lf[1], L2 = P.Lf[2];
    const float iL0 = P.iLf[0], iL1 = P.iLf[1], iL2 = P.iLf[2];
    const float rl = sqrtf((float)P.rlist2) + 1e-3f;
    const float rl2 = rl * rl;
    const float4 pi = B.pbuild[i];
    int* const row = B.nbr + (size_t)i * NE_NMAX;
    const int gsh = (threadIdx.x & 31) / G * G;  // this atom's first lane in the warp
    const unsigned gmask = G == 32 ? 0xffffffffu : ((1u << G) - 1u);
    int cnt = 0;
    // entries [lo, hi) of the sorted copy (empty for a lane group with no atom)
    // that lie `code` box lengths off; ALL: each at its nearest image instead
    auto scan = [&](auto all, int lo, int hi, int code, float px, float py, float pz) {
        const int trips = __reduce_max_sync(0xffffffffu, (unsigned)(hi > lo ? (hi - lo + G - 1) / G : 0));
        for (int t = 0; t < trips; ++t) {
            const int p = lo + t * G + lane;
            bool hit = false;
            int b = 0;
            if (p < hi) {
                const float4 pj = B.csort[off + p];
                b = __float_as_int(pj.w);
                float dx = pj.x - px, dy = pj.y - py, dz = pj.z - pz;
                if constexpr (all.value) {
                    const float n0 = rintf(dx * iL0), n1 = rintf(dy * iL1), n2 = rintf(dz * iL2);
                    dx -= L0 * n0;
                    dy -= L1 * n1;
                    dz -= L2 * n2;
                    code = NE_IMG_NONE - (int)(9.f * n0 + 3.f * n1 + n2);
                }
                hit = dx * dx + dy * dy + dz * dz < rl2 && b != a;
            }
            const unsigned m = (__ballot_sync(0xffffffffu, hit) >> gsh) & gmask;
            const int at = cnt + __popc(m & ((1u << lane) - 1u));
            if (hit && at < NE_NMAX) row[at] = (off + b) | (int)((unsigned)code << NE_IMG_SHIFT);
            cnt += __popc(m);
        }
    };
    if (P.nc[0] == 0) {
        scan(std::true_type(), 0, valid ? P.n : 0, 0, pi.x, pi.y, pi.z);
    } else {
        const int nc0 = P.nc[0], nc1 = P.nc[1], nc2 = P.nc[2];
        const int* start = B.cstart + P.cell_off + rep;
        const int c = valid ? B.cellof[i] : 0;
        const int cx = c / (nc1 * nc2), cy = (c / nc2) % nc1, cz = c % nc2;
        // z cells cz - 1 .. cz + 1 in order: [z0, z1) and, across the edge,
        // [z2, z3); the image of each run is that of its cells
        int z0 = cz - 1, z1 = cz + 2, z3 = 0, sz0 = 0, sz1 = 0;
        if (cz == 0) z0 = nc2 - 1, z1 = nc2, z3 = 2, sz0 = -1;
        if (cz == nc2 - 1) z1 = nc2, z3 = 1, sz1 = 1;
#pragma unroll 1
        for (int r = 0; r < 9; ++r) {
            const int x = cx + r / 3 - 1, y = cy + r % 3 - 1;
            const int sx = x < 0 ? -1 : (x >= nc0 ? 1 : 0), sy = y < 0 ? -1 : (y >= nc1 ? 1 : 0);
            const int o = ((x - sx * nc0) * nc1 + y - sy * nc1) * nc2;
            const int code = NE_IMG_NONE + 9 * sx + 3 * sy;
            const float px = pi.x - (float)sx * L0, py = pi.y - (float)sy * L1;
            scan(std::false_type(), valid ? start[o + z0] : 0, valid ? start[o + z1] : 0, code + sz0, px, py,
                 pi.z - (float)sz0 * L2);
            if (__any_sync(0xffffffffu, z3 > 0)) {
                const bool two = valid && z3 > 0;
                scan(std::false_type(), two ? start[o] : 0, two ? start[o + z3] : 0, code + sz1, px, py,
                     pi.z - (float)sz1 * L2);
            }
        }
    }
    if (valid && lane == 0) {
        if (cnt > NE_NMAX) ne_set_status(B.status, ST_ENEIGH);
        B.ncnt[i] = min(cnt, NE_NMAX);
    }
}

// a few blocks an SM take the atoms in turn: a launch with nothing to build is
// over sooner than with a block for every 8 or 32 atoms
template <int G>
__global__ void __launch_bounds__(LIST_THREADS) k_nl_list(DevBatch B)
{
    constexpr int SUB = NE_TILE * G / LIST_THREADS;
    int blk = blockIdx.x, rep = B.tile_rep[blk / SUB];
    ne_chain();
    for (;;) {
        list_block<G>(B, blk, rep);
        blk += gridDim.x;
        if (blk >= B.n_tiles * SUB) break;
        rep = B.tile_rep[blk / SUB];
    }
}

}  // namespace

namespace ne {

void launch_nl_build(const DevBatch& B, int force, int from_sites, cudaStream_t st)
{
    ne_launch(k_nl_cells, (B.n_tiles + CELL_TILES - 1) / CELL_TILES, CELL_THREADS, 0, st, B, force, from_sites);
    const auto grid = [&](int want) { return want < 6 * B.sms ? want : 6 * B.sms; };
    if (force && B.n_max > SORT_IN_BLOCK)
        ne_launch(k_nl_scatter, (B.n_tiles + 3) / 4, 256, 0, st, B);
    if (B.n_max > SORT_IN_BLOCK)
        ne_launch(k_nl_sort, (B.n_tiles + 3) / 4, 256, 0, st, B);
    // a warp an atom up to 8192 atoms (a quarter of a million threads, one
    // wave), eight lanes above: fewer idle lanes at the ends of the short runs.
    // Whole mixed energy calls in us with 32 and with 8: 2000 atoms 63-66, 76; 4056
    // 72, 82; 8192 90, 96; 12,288 109, 102; 16,000 124, 114; 35,152 154, 123
    if (B.n_tot <= 8192)
        ne_launch(k_nl_list<32>, grid(B.n_tiles * (NE_TILE * 32 / LIST_THREADS)), LIST_THREADS, 0, st, B);
    else
        ne_launch(k_nl_list<8>, grid(B.n_tiles * (NE_TILE * 8 / LIST_THREADS)), LIST_THREADS, 0, st, B);
}

}  // namespace ne
