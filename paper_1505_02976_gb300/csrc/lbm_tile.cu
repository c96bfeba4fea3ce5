// lbm_tile.cu -- two time steps of an FP32 lattice in one launch.
//
// One step moves every population through HBM once in each direction, and the
// one-step kernels run at that bound.  Here a block computes a tile of the
// lattice twice: step 1 on the tile and a ring of one node around it, from
// global memory into shared memory, and step 2 on the tile, from shared
// memory back to global memory.  The populations cross HBM once for two steps;
// the price is the ring (2 columns of 64 and 2 rows of 10 computed
// twice).
//
// A warp takes one row of 64 columns, each lane two x-neighbours, and runs
// the packed form of the node update.  The tile's first output column X0 is
// even.  Step 1 works on the pairs (X0 - 1 + 2l, X0 + 2l): the values pulled
// from the left or right start at an even column and are one aligned 64-bit
// load, those pulled from the same column two 32-bit loads.  Step 2 works on
// the pairs (X0 + 2l, X0 + 2l + 1), and in the tile's shared rows (which start
// at column X0 - 1) its pulls are aligned in the same way and its stores to
// global memory are aligned 64-bit ones.  Step 1 writes only to shared memory
// and step 2 only reads there, so one block barrier separates them.
//
// Bound: neither pipe alone.  2048^2: 285 + 236 MB of DRAM traffic and 69 M
// warp instructions a launch, issue 49 % active with 18 warps an SM, DRAM at
// 4.4 TB/s; 58.8 us a step in the timed loop (71 GLUPS) against 85 us (49) of
// the one-step kernels, which are at 0.98 of measured HBM; 4096^2 222 us (76)
// against 342; 1024 x 513 periodic 9.0 us against 9.3 of the global-load kernel;
// 1000 x 777 with a porosity field off tau = 1 16.6 us against 17.2 (12.7 and
// 24 before the node update was rearranged).
// Copying the pulls into the shared rows asynchronously (cp.async, every row of
// a warp in flight at once) took as long at 2048^2 and 3 to 8 % longer below
// 1024^2 (more instructions for the same bytes).
//
// Wall nodes are updated one per thread by the same code as in the one-step
// kernels (wall_node_tau1 / wall_node_generic) from global or shared memory.
// Tiles split the columns and rows evenly, so that every tile is at least
// three nodes wide and tall and x_f, x_ff of its wall nodes lie inside.
#include <math.h>
#include <string.h>

#include <vector>

#include "lbm_step.cuh"

namespace lbm {

constexpr int kTileCols = 64;                  // columns of a shared row (the tile and its ring)
constexpr int kTilePairs = kTileCols / 2 - 1;  // output pairs of a tile, at most

// Shape of a launch: output rows of a tile (at most; tiles split the rows
// evenly), warps that take its rows, warps beside them for the wall nodes
// (0: the same warps, afterwards).
struct TileShape {
    int rows, warps, wall_warps;
};
// Large lattices: two rows a warp, four blocks an SM.  Fewer, taller tiles
// leave fewer blocks in different phases (18 rows, 10 warps: 61.1 against 58.3
// us a step at 2048^2), more resident warps leave too little of the SM's
// memory as L1 for the loads in flight (25 warps: 70).
constexpr TileShape kTileLarge = {8, 5, 0};
// Lattices that do not fill the GPU: the step lasts as long as one block, so
// every warp has one row, and the wall nodes' long chain runs beside the rows
// (201^2: 2.8 us a step against 5.1 with the large shape, 3.6 without the wall
// warps; 32^2: 2.5 against 3.9).  The line lies at one and a half waves of its
// blocks: 384^2 (448 tiles) 5.0 against 5.7 us, 512^2 (774 tiles) 7.2 against 5.8.
constexpr TileShape kTileSmall = {6, 8, 2};
constexpr int kTileSmallWaves = 3;             // in SMs: at most 3 x 152 tiles
// x_f and x_ff of a tile's wall rows and their ring: three rows at least, which
// an even split of eight or more rows into tiles of at most four has
static_assert(kTileLarge.rows >= 4 && kTileSmall.rows >= 4, "tiles are at least three rows tall");
constexpr int kTileMaxThreads = 32 * (kTileSmall.warps + kTileSmall.wall_warps);
constexpr int kTileRowElems = NPLANES * kTileCols;

__host__ __device__ constexpr size_t tile_smem(int rows) { return (size_t)(rows + 2) * kTileRowElems * sizeof(float); }
// what a launch may ask for without the function's opt-in, beside the batch
// kernel's constants (43 520 bytes and about 1.5 KB)
static_assert(tile_smem(kTileLarge.rows) + sizeof(KConst<float>) + sizeof(PairConst) <= 48 * 1024 &&
                  kTileSmall.rows <= kTileLarge.rows,
              "a tile's shared rows fit 48 KB");

__device__ __forceinline__ float2 ld2(const float* p) { return *reinterpret_cast<const float2*>(p); }

// Pulled values of a wall node's source from the tile's shared rows.
struct TileSource {
    const float* slots;
    int xr, yr;  // lattice position of the first shared row's first column
    __device__ __forceinline__ void operator()(const KConst<float>&, int x, int y, Pops<float>& P) const {
        const float* s = slots + (y - yr) * kTileRowElems + (x - xr);
#pragma unroll
        for (int i = 1; i < 9; ++i) P.f[i] = s[-cy_of(i) * kTileRowElems + (i - 1) * kTileCols - cx_of(i)];
#pragma unroll
        for (int i = 0; i < 9; ++i) P.h[i] = s[-cy_of(i) * kTileRowElems + (8 + i) * kTileCols - cx_of(i)];
        P.f[0] = 0.f;
    }
};

template <bool TAU1>
__device__ __noinline__ void tile_wall_1(const KConst<float>& k, const float* __restrict__ src, float* slot, float* mid,
                                         int x, int y) {
    float fo[9], ho[9];
    if constexpr (TAU1) wall_node_tau1(k, GlobalSource<float, float>{src}, x, y, fo, ho);
    else wall_node_generic(k, GlobalSource<float, float>{src}, x, y, fo, ho);
#pragma unroll
    for (int i = 1; i < 9; ++i) slot[(i - 1) * kTileCols] = fo[i];
#pragma unroll
    for (int i = 0; i < 9; ++i) slot[(8 + i) * kTileCols] = ho[i];
    if (mid) store_node(k, mid, (long long)y * k.pitch + x, fo, ho);
}

template <bool TAU1>
__device__ __noinline__ void tile_wall_2(const KConst<float>& k, TileSource src, float* __restrict__ dst, int x, int y) {
    float fo[9], ho[9];
    if constexpr (TAU1) wall_node_tau1(k, src, x, y, fo, ho);
    else wall_node_generic(k, src, x, y, fo, ho);
    store_node(k, dst, (long long)y * k.pitch + x, fo, ho);
}

// The wall nodes of columns x0 .. x1 - 1, rows y0 .. y1 - 1, numbered: the S
// and N rows, then the W and E columns without them.
struct TileWalls {
    int x0, x1, y0, y1, nS, nN, nW, nE;
    __device__ __forceinline__ TileWalls(const KConst<float>& k, int x0_, int x1_, int y0_, int y1_)
        : x0(x0_), x1(x1_), y0(y0_), y1(y1_) {
        const bool wx = k.bc[SW] != BC_PERIODIC, wy = k.bc[SS] != BC_PERIODIC;
        const bool S = wy && y0 == 0, N = wy && y1 == k.ny;
        nS = S ? x1 - x0 : 0;
        nN = N ? x1 - x0 : 0;
        const int inner = y1 - y0 - (S ? 1 : 0) - (N ? 1 : 0);
        nW = wx && x0 == 0 ? inner : 0;
        nE = wx && x1 == k.nx ? inner : 0;
    }
    __device__ __forceinline__ int count() const { return nS + nN + nW + nE; }
    __device__ __forceinline__ void at(int n, int& x, int& y) const {
        const int first = nS ? y0 + 1 : y0;
        if (n < nS) { x = x0 + n; y = y0; return; }
        n -= nS;
        if (n < nN) { x = x0 + n; y = y1 - 1; return; }
        n -= nN;
        if (n < nW) { x = x0; y = first + n; return; }
        x = x1 - 1;
        y = first + n - nW;
    }
};

// Two steps of one tile: output columns X0 .. X1 - 1 (X0 even), rows Y0 .. Y1 - 1.
// mid (or nullptr): where the state after the first step goes as well.
template <bool EPS_FIELD, bool TAU1>
__device__ __forceinline__ void tile_two_steps(const KConst<float>& k, const PairConst& pc, const float* __restrict__ src,
                                               float* __restrict__ mid, float* __restrict__ dst, float* slots,
                                               int X0, int X1, int Y0, int Y1, int warps, bool hot) {
    // the first `warps` warps take the rows; the others, if there are any, the wall nodes
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int wall_threads = (int)blockDim.x > 32 * warps ? (int)blockDim.x - 32 * warps : (int)blockDim.x;
    const int wall_thread = (int)(blockDim.x - 1 - threadIdx.x);
    const bool wx = k.bc[SW] != BC_PERIODIC, wy = k.bc[SS] != BC_PERIODIC;
    const int nx = k.nx, ny = k.ny, pl = k.plane32, pitch = k.pitch;
    // step 1: the tile and its ring, as far as the lattice goes
    const int ya = wy ? max(Y0 - 1, 0) : Y0 - 1, yb = wy ? min(Y1 + 1, ny) : Y1 + 1;
    const int xa = wx ? max(X0 - 1, 0) : X0 - 1, xb = wx ? min(X1 + 1, nx) : X1 + 1;
    {
        const int x = X0 - 1 + 2 * lane;  // the pair x, x + 1
        const bool va = x >= (wx ? max(xa, 1) : xa) && x < (wx ? min(xb, nx - 1) : xb);
        const bool vb = x + 1 >= (wx ? max(xa, 1) : xa) && x + 1 < (wx ? min(xb, nx - 1) : xb);
        // columns of the loads: at a wall the values of clamped columns are
        // not used; on a periodic side they wrap, and a pair stays a pair
        // unless nx is odd (split)
        auto col = [&](int c) { return wx ? min(max(c, 0), nx - 1) : (c < 0 ? c + nx : (c >= nx ? c - nx : c)); };
        const bool split = !wx && (nx & 1) && (X0 == 0 || X1 + 2 >= nx);
        const int last = pitch - 2;
        // (a lane beyond the ring repeats its last pair)
        const int xe = min(x, X1 + 1 - ((X1 + 1 - x) & 1));
        const unsigned cl = wx || split ? min(max(xe - 1, 0), last) : col(xe - 1);
        const unsigned cr = wx || split ? min(max(xe + 1, 0), last) : col(xe + 1);
        const unsigned c0 = col(xe), c1 = col(xe + 1), cm = col(xe - 1), c2 = col(min(xe + 2, X1 + 2));
        for (int yy = warp < warps ? ya + warp : yb; yy < yb; yy += warps) {
            const int y = wy ? yy : (yy < 0 ? yy + ny : (yy >= ny ? yy - ny : yy));
            if (wy && (y == 0 || y == ny - 1)) continue;
            const unsigned rm = (y == 0 ? ny - 1 : y - 1) * pitch, r0 = y * pitch, rp = (y == ny - 1 ? 0 : y + 1) * pitch;
            float2 f[9], h[9], fo[9], ho[9];
            auto row = [&](int i) { return cy_of(i) > 0 ? rm : (cy_of(i) < 0 ? rp : r0); };
            if (!split) {
                auto load = [&](int i, int plane) {
                    const float* s = src + plane * pl;
                    const unsigned r = row(i);
                    return cx_of(i) > 0 ? ld2(s + (r + cl)) : (cx_of(i) < 0 ? ld2(s + (r + cr)) : make_float2(s[r + c0], s[r + c1]));
                };
#pragma unroll
                for (int i = 1; i < 9; ++i) f[i] = load(i, i - 1);
#pragma unroll
                for (int i = 0; i < 9; ++i) h[i] = load(i, 8 + i);
            } else {
                auto load = [&](int i, int plane) {
                    const float* s = src + plane * pl;
                    const unsigned r = row(i);
                    return cx_of(i) > 0 ? make_float2(s[r + cm], s[r + c0])
                                        : (cx_of(i) < 0 ? make_float2(s[r + c1], s[r + c2]) : make_float2(s[r + c0], s[r + c1]));
                };
#pragma unroll
                for (int i = 1; i < 9; ++i) f[i] = load(i, i - 1);
#pragma unroll
                for (int i = 0; i < 9; ++i) h[i] = load(i, 8 + i);
            }
            Cell<float2> c;
            if constexpr (EPS_FIELD) {
                const float* e = k.eps_field + (long long)y * nx;
                c = field_cell(pc, make_float2(e[c0], e[c1]));
            } else {
                c = pc.cell;
            }
            core_interior<TAU1>(pc, c, eps_ay(k, pc, c, y), f, h, fo, ho);
            if ((va && !lfinite(ho[0].x)) || (vb && !lfinite(ho[0].y))) atomicOr(k.flag, 1);
            if (mid && yy >= Y0 && yy < Y1) {
                float* m = mid + (y * pitch + x);
                if (va && x >= X0) {
#pragma unroll
                    for (int i = 1; i < 9; ++i) m[(i - 1) * pl] = fo[i].x;
#pragma unroll
                    for (int i = 0; i < 9; ++i) m[(8 + i) * pl] = ho[i].x;
                }
                if (vb && x + 1 < X1) {
#pragma unroll
                    for (int i = 1; i < 9; ++i) m[(i - 1) * pl + 1] = fo[i].y;
#pragma unroll
                    for (int i = 0; i < 9; ++i) m[(8 + i) * pl + 1] = ho[i].y;
                }
            }
            float* d = slots + (yy - Y0 + 1) * kTileRowElems + 2 * lane;
            if (va && vb) {
#pragma unroll
                for (int i = 1; i < 9; ++i) *reinterpret_cast<float2*>(d + (i - 1) * kTileCols) = fo[i];
#pragma unroll
                for (int i = 0; i < 9; ++i) *reinterpret_cast<float2*>(d + (8 + i) * kTileCols) = ho[i];
            } else if (va || vb) {
                d += va ? 0 : 1;
#pragma unroll
                for (int i = 1; i < 9; ++i) d[(i - 1) * kTileCols] = va ? fo[i].x : fo[i].y;
#pragma unroll
                for (int i = 0; i < 9; ++i) d[(8 + i) * kTileCols] = va ? ho[i].x : ho[i].y;
            }
        }
        const TileWalls W(k, xa, xb, ya, yb);
        const int nw = W.count();
        for (int n = wall_thread < wall_threads ? wall_thread : nw; n < nw; n += wall_threads) {
            int X, Y;
            W.at(n, X, Y);
            float* slot = slots + (Y - Y0 + 1) * kTileRowElems + (X - X0 + 1);
            float* own = X >= X0 && X < X1 && Y >= Y0 && Y < Y1 ? mid : nullptr;
            if (!wx) X = X < 0 ? X + nx : (X >= nx ? X - nx : X);
            if (!wy) Y = Y < 0 ? Y + ny : (Y >= ny ? Y - ny : Y);
            tile_wall_1<TAU1>(k, src, slot, own, X, Y);
        }
    }
    __syncthreads();
    // step 2: the tile
    {
        const int x = X0 + 2 * lane;
        const bool in = lane < kTilePairs && x < X1;
        const bool va = in && !(wx && (x == 0 || x == nx - 1)), vb = in && x + 1 < X1 && !(wx && x + 1 == nx - 1);
        const int l = min(lane, kTilePairs - 1);
        for (int y = warp < warps ? Y0 + warp : Y1; y < Y1; y += warps) {
            if (wy && (y == 0 || y == ny - 1)) continue;
            // the pair's left neighbour column is 2 l of the shared row
            const float* s0 = slots + (y - Y0 + 1) * kTileRowElems + 2 * l;
            float2 f[9], h[9], fo[9], ho[9];
            auto load = [&](int i, int plane) {
                const float* s = s0 + (plane * kTileCols - cy_of(i) * kTileRowElems);
                return cx_of(i) > 0 ? ld2(s) : (cx_of(i) < 0 ? ld2(s + 2) : make_float2(s[1], s[2]));
            };
#pragma unroll
            for (int i = 1; i < 9; ++i) f[i] = load(i, i - 1);
#pragma unroll
            for (int i = 0; i < 9; ++i) h[i] = load(i, 8 + i);
            Cell<float2> c;
            if constexpr (EPS_FIELD) {
                const float* e = k.eps_field + (long long)y * nx;
                c = field_cell(pc, make_float2(e[min(x, nx - 1)], e[min(x + 1, nx - 1)]));
            } else {
                c = pc.cell;
            }
            core_interior<TAU1>(pc, c, eps_ay(k, pc, c, y), f, h, fo, ho);
            if ((va && !lfinite(ho[0].x)) || (vb && !lfinite(ho[0].y))) atomicOr(k.flag, 1);
            float* d = dst + (y * pitch + x);
            if (va && vb) {
                if (hot) {
                    uint64_t pol;
                    asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(pol));
#pragma unroll
                    for (int i = 1; i < 9; ++i)
                        asm volatile("st.global.L2::cache_hint.v2.f32 [%0], {%1, %2}, %3;" ::"l"(d + (i - 1) * pl),
                                     "f"(fo[i].x), "f"(fo[i].y), "l"(pol) : "memory");
#pragma unroll
                    for (int i = 0; i < 9; ++i)
                        asm volatile("st.global.L2::cache_hint.v2.f32 [%0], {%1, %2}, %3;" ::"l"(d + (8 + i) * pl),
                                     "f"(ho[i].x), "f"(ho[i].y), "l"(pol) : "memory");
                } else {
#pragma unroll
                    for (int i = 1; i < 9; ++i) *reinterpret_cast<float2*>(d + (i - 1) * pl) = fo[i];
#pragma unroll
                    for (int i = 0; i < 9; ++i) *reinterpret_cast<float2*>(d + (8 + i) * pl) = ho[i];
                }
            } else if (va || vb) {
                d += va ? 0 : 1;
#pragma unroll
                for (int i = 1; i < 9; ++i) d[(i - 1) * pl] = va ? fo[i].x : fo[i].y;
#pragma unroll
                for (int i = 0; i < 9; ++i) d[(8 + i) * pl] = va ? ho[i].x : ho[i].y;
            }
        }
        const TileWalls W(k, X0, X1, Y0, Y1);
        const int nw = W.count();
        for (int n = wall_thread < wall_threads ? wall_thread : nw; n < nw; n += wall_threads) {
            int X, Y;
            W.at(n, X, Y);
            tile_wall_2<TAU1>(k, TileSource{slots, X0 - 1, Y0 - 1}, dst, X, Y);
        }
    }
}

// An axis of `size` nodes split into n tiles of whole units: q units each,
// one more in the first r.
struct TileSplit {
    int n, q, r, unit, size;
    __host__ __device__ __forceinline__ int begin(int b) const {
        const int at = (b * q + min(b, r)) * unit;
        return at < size ? at : size;
    }
};

template <bool EPS_FIELD, bool TAU1>
__global__ void __launch_bounds__(kTileMaxThreads, 2)
k_tile(const __grid_constant__ KConst<float> k, const __grid_constant__ PairConst pc, const float* __restrict__ src, float* __restrict__ mid,
       float* __restrict__ dst, TileSplit sx, TileSplit sy, int warps, bool early, uint32_t launch) {
    extern __shared__ __align__(16) float slots[];
    // early: let the next launch's blocks in as soon as this one's have all
    // started.  Small lattices' blocks do it only once the previous launch is
    // done: otherwise a queue of later launches takes their places on the SMs
    // (128^2 2.9 -> 2.6 us a step; 2048^2 58 -> 60, so large ones keep it).
    if (early) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    // bottom-up and top-down in turn, so that a launch first reads the rows
    // the previous one wrote last, while they are in L2
    const int by = (launch & 1u) ? (int)(gridDim.y - 1 - blockIdx.y) : (int)blockIdx.y;
    const int X0 = sx.begin(blockIdx.x), X1 = sx.begin(blockIdx.x + 1), Y0 = sy.begin(by), Y1 = sy.begin(by + 1);
    const bool hot = (long long)(gridDim.y - blockIdx.y) * (Y1 - Y0) * k.nx <= k.l2_hot;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (!early) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    tile_two_steps<EPS_FIELD, TAU1>(k, pc, src, mid, dst, slots, X0, X1, Y0, Y1, warps, hot);
}

// ------------------------------------------------------------- moment state
// One step of the FP32 moment state (lbm_moment.cu) over the same tiles: the
// moments of the tile and its ring are expanded into populations in the shared
// rows (two x-neighbours a lane, packed), and the tile's new moments computed
// from their pulls.  Wall nodes expand like any other; their new state is the
// boundary state of x_f's new moments, one wall node a thread.
// Against warps that march up strips of columns (k_step_m), which expand fewer
// nodes twice but keep only one row a warp in flight: 64^2 3.7 against 6.1 us a
// step, 201^2 4.0 / 7.6, 512^2 7.2 / 11.3, 1024 x 777 15.1 / 18.9, but 2048^2 73.9 /
// 72.4 and 3000 x 2900 145 / 139: the line lies between, at 16 tiles an SM.
__device__ __noinline__ void tile_wall_m(const KConst<float>& k, TileSource src, float* __restrict__ dst, int x, int y) {
    const WallInfo w = classify(k, x, y);
    Pops<float> P;
    src(k, w.xs, w.ys, P);
    const Cell<float> c = node_cell(k, w.xs, w.ys);
    float m[kMPlanes];
    stored_moments(k, c, core_moments(k, c, eps_ay(k, k, c, w.ys), P.f, P.h), m);
    m[MUX] = k.u_bc[w.uside][0];
    m[MUY] = k.u_bc[w.uside][1];
    if (w.tside >= 0) {
        m[MTH] = lsub(k.T_bc[w.tside], k.T0);
    } else {
        Pops<float> Q;
        src(k, w.xff, w.yff, Q);
        m[MTH] = lmul(lfma(4.f, m[MTH], -core_theta(k, core_hsum(Q.h))), 1.f / 3.f);
        if (w.fixgx) m[MGX] = 0.f;
        if (w.fixgy) m[MGY] = 0.f;
    }
    if (!isfinite(m[MTH] + m[MP])) atomicOr(k.flag, 1);
    float* d = dst + ((long long)y * k.pitch + x);
#pragma unroll
    for (int q = 0; q < kMPlanes; ++q) d[q * k.plane] = m[q];
}

template <bool EPS_FIELD, bool SOURCES>
__global__ void __launch_bounds__(kTileMaxThreads, 2)
k_tile_m(const __grid_constant__ KConst<float> k, const __grid_constant__ PairConst pc, const float* __restrict__ src,
         float* __restrict__ dst, TileSplit sx, TileSplit sy, int warps, bool early) {
    extern __shared__ __align__(16) float slots[];
    if (early) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int X0 = sx.begin(blockIdx.x), X1 = sx.begin(blockIdx.x + 1), Y0 = sy.begin(blockIdx.y), Y1 = sy.begin(blockIdx.y + 1);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const bool wx = k.bc[SW] != BC_PERIODIC, wy = k.bc[SS] != BC_PERIODIC;
    const int nx = k.nx, ny = k.ny, pl = k.plane32, pitch = k.pitch;
    const int ya = wy ? max(Y0 - 1, 0) : Y0 - 1, yb = wy ? min(Y1 + 1, ny) : Y1 + 1;
    const int xa = wx ? max(X0 - 1, 0) : X0 - 1, xb = wx ? min(X1 + 1, nx) : X1 + 1;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (!early) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    auto cell_of = [&](int y, unsigned c0, unsigned c1) {
        if constexpr (EPS_FIELD) {
            const float* e = k.eps_field + (long long)y * nx;
            return field_cell(pc, make_float2(e[c0], e[c1]));
        } else {
            return pc.cell;
        }
    };
    {
        const int x = X0 - 1 + 2 * lane;
        const bool va = x >= xa && x < xb, vb = x + 1 >= xa && x + 1 < xb;
        auto col = [&](int c) { return wx ? min(max(c, 0), nx - 1) : (c < 0 ? c + nx : (c >= nx ? c - nx : c)); };
        const int xe = min(x, X1);  // (a lane beyond the ring repeats its end)
        const unsigned c0 = col(xe), c1 = col(min(x + 1, X1));
        for (int yy = warp < warps ? ya + warp : yb; yy < yb; yy += warps) {
            const int y = wy ? yy : (yy < 0 ? yy + ny : (yy >= ny ? yy - ny : yy));
            const unsigned r = y * pitch;
            float2 m[kMPlanes], fo[9], ho[9];
#pragma unroll
            for (int q = 0; q < kMPlanes; ++q) {
                const float* s = src + q * pl;
                m[q] = make_float2(s[r + c0], s[r + c1]);
            }
            const Cell<float2> c = cell_of(y, c0, c1);
            expand_moments<SOURCES>(pc, c, eps_ay(k, pc, c, y), m, fo, ho);
            float* d = slots + (yy - Y0 + 1) * kTileRowElems + 2 * lane;
            if (va && vb) {
#pragma unroll
                for (int i = 1; i < 9; ++i) *reinterpret_cast<float2*>(d + (i - 1) * kTileCols) = fo[i];
#pragma unroll
                for (int i = 0; i < 9; ++i) *reinterpret_cast<float2*>(d + (8 + i) * kTileCols) = ho[i];
            } else if (va || vb) {
                d += va ? 0 : 1;
#pragma unroll
                for (int i = 1; i < 9; ++i) d[(i - 1) * kTileCols] = va ? fo[i].x : fo[i].y;
#pragma unroll
                for (int i = 0; i < 9; ++i) d[(8 + i) * kTileCols] = va ? ho[i].x : ho[i].y;
            }
        }
    }
    __syncthreads();
    {
        const int x = X0 + 2 * lane;
        const bool in = lane < kTilePairs && x < X1;
        const bool va = in && !(wx && (x == 0 || x == nx - 1)), vb = in && x + 1 < X1 && !(wx && x + 1 == nx - 1);
        const int l = min(lane, kTilePairs - 1);
        for (int y = warp < warps ? Y0 + warp : Y1; y < Y1; y += warps) {
            if (wy && (y == 0 || y == ny - 1)) continue;
            const float* s0 = slots + (y - Y0 + 1) * kTileRowElems + 2 * l;
            float2 f[9], h[9], m[kMPlanes];
            auto load = [&](int i, int plane) {
                const float* s = s0 + (plane * kTileCols - cy_of(i) * kTileRowElems);
                return cx_of(i) > 0 ? ld2(s) : (cx_of(i) < 0 ? ld2(s + 2) : make_float2(s[1], s[2]));
            };
#pragma unroll
            for (int i = 1; i < 9; ++i) f[i] = load(i, i - 1);
#pragma unroll
            for (int i = 0; i < 9; ++i) h[i] = load(i, 8 + i);
            const Cell<float2> c = cell_of(y, min(x, nx - 1), min(x + 1, nx - 1));
            stored_moments(pc, c, core_moments(pc, c, eps_ay(k, pc, c, y), f, h), m);
            const float2 check = ladd(ladd(m[MTH], m[MUX]), m[MUY]);
            if ((va && !lfinite(check.x)) || (vb && !lfinite(check.y))) atomicOr(k.flag, 1);
            float* d = dst + (y * pitch + x);
            if (va && vb) {
#pragma unroll
                for (int q = 0; q < kMPlanes; ++q) *reinterpret_cast<float2*>(d + q * pl) = m[q];
            } else if (va || vb) {
                d += va ? 0 : 1;
#pragma unroll
                for (int q = 0; q < kMPlanes; ++q) d[q * pl] = va ? m[q].x : m[q].y;
            }
        }
        const int wall_threads = (int)blockDim.x > 32 * warps ? (int)blockDim.x - 32 * warps : (int)blockDim.x;
        const int wall_thread = (int)(blockDim.x - 1 - threadIdx.x);
        const TileWalls W(k, X0, X1, Y0, Y1);
        const int nw = W.count();
        for (int n = wall_thread < wall_threads ? wall_thread : nw; n < nw; n += wall_threads) {
            int X, Y;
            W.at(n, X, Y);
            tile_wall_m(k, TileSource{slots, X0 - 1, Y0 - 1}, dst, X, Y);
        }
    }
}

// Two steps of a batch of FP32 cavities walled on all four sides: block i takes
// tile i of the list (cavity by cavity, tiles of the large shape) and reads the
// cavity's constants from shared memory (128 cavities of 64^2 to 512^2: 54.5
// GLUPS against 44 of the staged one-step kernel).  TAU1: every cavity has tau_f = tau_T =
// 1 (with both forms in one kernel the registers spill).
template <bool TAU1>
__global__ void __launch_bounds__(32 * kTileLarge.warps, 4)
k_tile_batch(const BatchCavity<float>* __restrict__ cav, const PairConst* __restrict__ pair,
             const TileItem* __restrict__ items, const float* __restrict__ src, float* __restrict__ dst) {
    extern __shared__ __align__(16) float slots[];
    __shared__ KConst<float> k;
    __shared__ PairConst pc;
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const TileItem w = items[blockIdx.x];
    // written once, before any step: may be read before the previous step is done
    auto fetch = [](auto& to, const auto& from) {
        const int* a = reinterpret_cast<const int*>(&from);
        int* b = reinterpret_cast<int*>(&to);
        for (int q = threadIdx.x; q < (int)(sizeof(to) / sizeof(int)); q += 32 * kTileLarge.warps) b[q] = a[q];
    };
    fetch(k, cav[w.cavity].k);
    fetch(pc, pair[w.cavity]);
    const long long off = cav[w.cavity].offset;
    __syncthreads();
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (TAU1 || (k.omf == 0.f && k.omT == 0.f))
        tile_two_steps<false, true>(k, pc, src + off, nullptr, dst + off, slots, w.x0, w.x1, w.y0, w.y1, kTileLarge.warps, false);
    else
        tile_two_steps<false, false>(k, pc, src + off, nullptr, dst + off, slots, w.x0, w.x1, w.y0, w.y1, kTileLarge.warps, false);
}

// The fewest tiles of at most `most` units.
static TileSplit tile_split(int size, int unit, int most) {
    const int u = (size + unit - 1) / unit, n = (u + most - 1) / most;
    return {n, u / n, u % n, unit, size};
}

template <bool E, bool T>
static cudaError_t launch_tile(cudaLaunchConfig_t& cfg, const KConst<float>& k, const float* src, float* mid,
                               float* dst, const TileSplit& sx, const TileSplit& sy, int warps, bool early, uint32_t launch) {
    const PairConst pc = make_pair_const(k, 1.0f);
    return cudaLaunchKernelEx(&cfg, k_tile<E, T>, k, pc, src, mid, dst, sx, sy, warps, early, launch);
}

std::vector<TileItem> tile_items(int cavity, int nx, int ny) {
    const TileSplit sx = tile_split(nx, 2, kTilePairs), sy = tile_split(ny, 1, kTileLarge.rows);
    std::vector<TileItem> v;
    for (int j = 0; j < sy.n; ++j)
        for (int i = 0; i < sx.n; ++i) v.push_back({cavity, sx.begin(i), sx.begin(i + 1), sy.begin(j), sy.begin(j + 1)});
    return v;
}

void make_pair_consts(const BatchCavity<float>* cav, int n, std::vector<unsigned char>* out) {
    out->resize((size_t)n * sizeof(PairConst));
    for (int c = 0; c < n; ++c) {
        const PairConst q = make_pair_const(cav[c].k, 1.0f);
        memcpy(out->data() + (size_t)c * sizeof(PairConst), &q, sizeof(q));
    }
}
size_t pair_const_bytes() { return sizeof(PairConst); }

cudaError_t launch_two_steps_batch(const BatchCavity<float>* cav, const void* pair, const TileItem* items, int n_items,
                                   bool tau1, const float* src, float* dst, cudaStream_t st) {
    if (n_items < 1) return cudaErrorInvalidValue;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)n_items);
    cfg.blockDim = dim3(32 * kTileLarge.warps);
    cfg.dynamicSmemBytes = tile_smem(kTileLarge.rows);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return tau1 ? cudaLaunchKernelEx(&cfg, k_tile_batch<true>, cav, (const PairConst*)pair, items, src, dst)
                : cudaLaunchKernelEx(&cfg, k_tile_batch<false>, cav, (const PairConst*)pair, items, src, dst);
}

template <bool E, bool S>
static cudaError_t launch_tile_m(cudaLaunchConfig_t& cfg, const KConst<float>& k, const float* src, float* dst,
                                 const TileSplit& sx, const TileSplit& sy, int warps, bool early) {
    const PairConst pc = make_pair_const(k, 1.0f);
    return cudaLaunchKernelEx(&cfg, k_tile_m<E, S>, k, pc, src, dst, sx, sy, warps, early);
}

bool moment_tiles_preferred(const KConst<float>& k, int sms) {
    return two_steps_supported(k) &&
           (long long)tile_split(k.nx, 2, kTilePairs).n * tile_split(k.ny, 1, kTileLarge.rows).n <= 16LL * sms;
}

cudaError_t launch_step_m_tiles(const KConst<float>& k, const float* src, float* dst, bool sources, int sms, cudaStream_t st) {
    if (!two_steps_supported(k)) return cudaErrorInvalidValue;
    const TileSplit sx = tile_split(k.nx, 2, kTilePairs);
    const bool small = (long long)sx.n * tile_split(k.ny, 1, kTileSmall.rows).n <= (long long)kTileSmallWaves * sms;
    const TileShape shape = small ? kTileSmall : kTileLarge;
    const TileSplit sy = tile_split(k.ny, 1, shape.rows);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)sx.n, (unsigned)sy.n);
    cfg.blockDim = dim3((unsigned)(32 * (shape.warps + shape.wall_warps)));
    cfg.dynamicSmemBytes = tile_smem(shape.rows);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (k.eps_field)
        return sources ? launch_tile_m<true, true>(cfg, k, src, dst, sx, sy, shape.warps, !small)
                       : launch_tile_m<true, false>(cfg, k, src, dst, sx, sy, shape.warps, !small);
    return sources ? launch_tile_m<false, true>(cfg, k, src, dst, sx, sy, shape.warps, !small)
                   : launch_tile_m<false, false>(cfg, k, src, dst, sx, sy, shape.warps, !small);
}

bool two_steps_supported(const KConst<float>& k) { return k.nx >= 8 && k.ny >= 8; }

cudaError_t launch_two_steps(const KConst<float>& k, const float* src, float* mid, float* dst, uint32_t launch, int sms,
                             cudaStream_t st) {
    if (!two_steps_supported(k)) return cudaErrorInvalidValue;
    const TileSplit sx = tile_split(k.nx, 2, kTilePairs);
    const bool small = (long long)sx.n * tile_split(k.ny, 1, kTileSmall.rows).n <= (long long)kTileSmallWaves * sms;
    const TileShape shape = small ? kTileSmall : kTileLarge;
    const TileSplit sy = tile_split(k.ny, 1, shape.rows);
    const int warps = shape.warps;
    const bool early = !small;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)sx.n, (unsigned)sy.n);
    cfg.blockDim = dim3((unsigned)(32 * (shape.warps + shape.wall_warps)));
    cfg.dynamicSmemBytes = tile_smem(shape.rows);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    const bool tau1 = k.omf == 0.f && k.omT == 0.f;
    if (k.eps_field) return tau1 ? launch_tile<true, true>(cfg, k, src, mid, dst, sx, sy, warps, early, launch) : launch_tile<true, false>(cfg, k, src, mid, dst, sx, sy, warps, early, launch);
    return tau1 ? launch_tile<false, true>(cfg, k, src, mid, dst, sx, sy, warps, early, launch) : launch_tile<false, false>(cfg, k, src, mid, dst, sx, sy, warps, early, launch);
}

}  // namespace lbm
