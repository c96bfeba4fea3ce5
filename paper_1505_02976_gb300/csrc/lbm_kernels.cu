// lbm_kernels.cu -- the fused step kernel of a single lattice.
//
// k_step: one thread per node, pull streaming from the ping buffer, all the
// per-node arithmetic of the step in registers, and one write of the 17
// post-collision planes to the pong buffer.  Wall nodes take the NEES rebuild
// inside the same launch (an out-of-line path that pulls the populations of
// the wall node's fluid neighbour x_f instead of its own).  It steps FP64
// lattices, FP16 lattices with a periodic side, and what FP32 lattices do not
// take in pairs (lbm_tile.cu) where rows cannot be staged (lbm_step_tma.cu); and
// FP32 and FP16 lattices on which it is selected (lbm_set_step_staging).
#include <math.h>

#include <atomic>

#include "lbm_step.cuh"

namespace lbm {

// The fused step: one thread per node.  The first `wall_blocks` blocks take the
// wall nodes in perimeter order (the NEES path), the others the interior nodes
// row by row, bx blocks a row: a warp then runs one of the two paths, where a
// warp with both would run them one after the other, and the wall nodes'
// longer chain starts first.  TAU1: tau_f = tau_T = 1 (the paper's default,
// Sec. 4), where the (1 - 1/tau) terms vanish.
// FP64 is bound by its pipe (two lanes a cycle and SM): 700 x 517 takes 128 us a
// step, 0.98 of the measured FP64 rate for its 183 FP64 instructions a node.
// Before the root and the reciprocal took their second iteration (2 % of every
// FP64 figure here): 126 us, 165 with the wall nodes inside the rows' warps, 267
// with the direction-by-direction arithmetic too; blocks of one warp end most
// evenly (130 us in blocks of four).  A lattice that leaves SMs empty is bound by one
// warp's chain, and blocks of one warp put every warp on an SM of its own: 32^2
// 8.6 us a step (10.0 in blocks of four; 17.3 with the wall nodes inside, 38
// before), 7.1 with SPLIT (below).
// One block's share: block b of the numbering above.  PART: lbm_step.cuh.
template <class R, class S, bool EPS_FIELD, bool TAU1, int PART>
__device__ __forceinline__ void step_block(const KConst<R>& k, const S* __restrict__ src, S* __restrict__ dst, unsigned b,
                                           int wall_blocks, int bx, uint32_t step) {
    if ((int)b < wall_blocks) {
        const int n = (int)(b * blockDim.x + threadIdx.x);
        if (n >= perimeter_nodes(k)) return;
        int x, y;
        perimeter_node(k, n, x, y);
        if constexpr (PART == 0) wall_update(k, src, dst, x, y, step);
        else wall_update_tau1<R, S, PART>(k, src, dst, x, y, step);
        return;
    }
    b -= wall_blocks;
    const int y = (int)(b / (unsigned)bx);
    const int x = (int)((b - (unsigned)y * bx) * blockDim.x + threadIdx.x);
    if (x >= k.nx || is_wall(k, x, y)) return;
    interior_update<R, S, EPS_FIELD, TAU1, PART>(k, src, dst, x, y, step);
}

// SPLIT (FP64, tau = 1): two blocks for each share, one for the flow and one for
// the thermal planes.  They repeat what both need, but each has the shorter
// chain, and a small lattice's step lasts as long as the longest chain: 32^2 8.6
// -> 7.1 us a step, 80^2 (250 shares) 8.8 -> 8.2, but 100^2 (425) 9.1 -> 9.6, so up
// to two shares an SM.
template <class R, class S, bool EPS_FIELD, bool TAU1, bool SPLIT>
__global__ void __launch_bounds__(kStepBlock, StepOccupancy<R>::blocks)
k_step(const __grid_constant__ KConst<R> k, const S* __restrict__ src, S* __restrict__ dst, int wall_blocks, int bx,
       uint32_t step) {
    // Programmatic dependent launch: wait here until the previous step's grid
    // has completed and its writes are visible (no-op without the launch
    // attribute), then let the next step's blocks be scheduled while this grid
    // runs.  Both are hardware-managed; nothing spins.  The other order lets a
    // whole queue of later steps take their places on the SMs: FP64 80^2 8.9 us
    // a step against 19.4.
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if constexpr (SPLIT) {
        const unsigned b = blockIdx.x >> 1;
        if (blockIdx.x & 1u) step_block<R, S, EPS_FIELD, TAU1, 1>(k, src, dst, b, wall_blocks, bx, step);
        else step_block<R, S, EPS_FIELD, TAU1, 2>(k, src, dst, b, wall_blocks, bx, step);
    } else {
        step_block<R, S, EPS_FIELD, TAU1, 0>(k, src, dst, blockIdx.x, wall_blocks, bx, step);
    }
}

template <class R, class S>
__global__ void k_init(const __grid_constant__ KConst<R> k, S* __restrict__ dst,
                       const double* __restrict__ T, const double* __restrict__ ux,
                       const double* __restrict__ uy, double T_init) {
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y;
    if (x >= k.nx) return;
    const long long c = (long long)y * k.nx + x;
    State<R> s;
    s.th = R((T ? T[c] : T_init) - double(k.T0));
    s.ux = ux ? R(ux[c]) : R(0);
    s.uy = uy ? R(uy[c]) : R(0);
    s.p = R(0);
    s.Fx = s.Fy = R(0);
    s.Sxx = s.Sxy = s.Syy = R(0);
    s.gx = s.gy = R(0);
    EqTerms<R> e;
    eq_terms(k, cell_consts(k, node_eps(k, x, y)), s, e);
    store_node(k, dst, (long long)y * k.pitch + x, e.fe, e.he);
}

// ------------------------------------------------------------------ launchers

// Multiprocessors of the current device (asked once per device).
static int device_sms() {
    constexpr int kMaxDev = 64;
    static std::atomic<int> known[kMaxDev];  // 0: not asked yet (any thread may ask)
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 1;
    if (dev < kMaxDev && (sms = known[dev].load(std::memory_order_relaxed)) > 0) return sms;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1) return 1;
    if (dev < kMaxDev) known[dev].store(sms, std::memory_order_relaxed);
    return sms;
}

template <class R, class S>
cudaError_t launch_step(const KConst<R>& k, const S* src, S* dst, uint32_t step, cudaStream_t st) {
    cudaLaunchConfig_t cfg = {};
    // blocks of one warp in FP64, and while whole blocks would not fill the GPU twice
    const long long full = (long long)((k.nx + kStepBlock - 1) / kStepBlock) * k.ny;
    const int block = sizeof(R) == 8 || full < 2LL * device_sms() ? 32 : kStepBlock;
    const int bx = (k.nx + block - 1) / block, wall_blocks = (perimeter_nodes(k) + block - 1) / block;
    const bool tau1 = k.omf == R(0) && k.omT == R(0);
    const long long shares = wall_blocks + (long long)bx * k.ny;
    const bool split = sizeof(R) == 8 && tau1 && shares <= 2LL * device_sms();
    cfg.gridDim = dim3((unsigned)(split ? 2 * shares : shares));
    cfg.blockDim = dim3((unsigned)block);
    // The blocks of a dependent launch fill SM after SM up to the kernel's
    // occupancy (12 or more blocks of one warp), which leaves SMs idle where the
    // grid is smaller, and in the last round where that is less than half full:
    // unused shared memory keeps each SM to its share of the blocks, in rounds of
    // one size.  FP64 130^2 13.2 -> 12.0, 201^2 21.6 -> 18.9 us a step in one round
    // (with fewer than four blocks an SM the launches overlap less and it costs
    // 0.5 us, and four would need more than the 48 KB a launch may ask for
    // unasked); 243 x 240 29.0 -> 25.9, 261 x 258 32.5 -> 29.4, 279 x 276 34.9 -> 31.0 in
    // two, 351 x 348 48.4 -> 46.4 in three.  Where the last round is fuller, or
    // holds an eighth of the SMs' number or less, it costs up to 7 % (333 x 330
    // periodic: 41.9 -> 44.7); beyond three rounds it changes nothing.
    const long long sms = device_sms(), per = (cfg.gridDim.x + sms - 1) / sms;
    const long long rounds = (per + 11) / 12, last = per - 12 * (rounds - 1), over = cfg.gridDim.x - 12 * (rounds - 1) * sms;
    const bool spread = sizeof(R) == 8 && per >= 5 && (rounds == 1 ? last < 12 : rounds <= 3 && last <= 6 && over > sms / 8);
    const long long resident = (per + rounds - 1) / rounds;
    cfg.dynamicSmemBytes = spread ? (size_t)(227 / resident - 1) * 1024 : 0;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    auto go = [&](auto kernel) { return cudaLaunchKernelEx(&cfg, kernel, k, src, dst, wall_blocks, bx, step); };
    if constexpr (sizeof(R) == 8)
        if (split) return k.eps_field ? go(k_step<R, S, true, true, true>) : go(k_step<R, S, false, true, true>);
    if (k.eps_field) return tau1 ? go(k_step<R, S, true, true, false>) : go(k_step<R, S, true, false, false>);
    return tau1 ? go(k_step<R, S, false, true, false>) : go(k_step<R, S, false, false, false>);
}

template <class R, class S>
cudaError_t launch_init(const KConst<R>& k, S* dst, const double* T, const double* ux,
                        const double* uy, double T_init, cudaStream_t st) {
    k_init<R, S><<<row_grid(k.nx, k.ny, 128), 128, 0, st>>>(k, dst, T, ux, uy, T_init);
    return cudaGetLastError();
}

#define LBM_INSTANTIATE(R, S)                                                                        \
    template cudaError_t launch_step<R, S>(const KConst<R>&, const S*, S*, uint32_t, cudaStream_t);  \
    template cudaError_t launch_init<R, S>(const KConst<R>&, S*, const double*, const double*,      \
                                           const double*, double, cudaStream_t);

LBM_INSTANTIATE(double, double)
LBM_INSTANTIATE(float, float)
LBM_INSTANTIATE(float, __half)

}  // namespace lbm
