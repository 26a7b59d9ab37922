// The single-lattice step with two x-adjacent sites per thread (pair_update in lbm_kernels.cu):
// every lattice with halfway walls, ping-pong and AA, in a translation unit of its own.
// lbm_pair_first.cu compiles the ping-pong steps a second time with other L2 hints.
#define LBM_DEVICE_ONLY
#include "lbm_kernels.cu"

namespace lbm {
namespace {

// Registers per thread (ptxas cap), measured on the GB300 at 64-thread blocks; us a step at 96 /
// 104 / 112 / 120 / 128 where tried: FP32 64^3 7.14 / 7.67 / 7.23 / 7.47 / 7.36, D3Q15 channel
// 192x48x48 10.2 / 10.9 / 10.6 / 10.4 / 10.5; odd rows (63x61x59) 7.64 / 8.06 / 7.69 / 7.43 / 7.50;
// FP16 channel 256x64x64 23.7 (96), 24.7 (104), 26.1 (112), 23.8 (128); FP16 odd rows 127^3 51.5 /
// 53.9 / 52.2 / 51.9 / 52.2, channel 255x64x64 28.3 / 28.6 / 27.6 / 27.2 / 27.5; BF16 field cavity 64^3
// 8.02 / 7.85 / 7.73 / 7.88 / 7.75, 128^3 49.9 / 51.9 / 51.9 / 51.8 / 51.9, 127^3 57.0 / 55.7 / 55.7 /
// 55.6 / 55.5 (with a field 96 gains at large even sizes alone); FP32 field 256^3 512 at 112-128, 571
// at 144; enthalpy 64^3 9.2 / 8.7 / 8.2 / 7.9 / 7.9.
template <bool HET, class S, bool ENTH, bool VEC>
constexpr int pair_regs() {
    return ENTH ? 128 : HET ? (S::kScaled ? 120 : 128) : S::kScaled ? 96 : VEC ? 96 : 120;
}

// The pair of a thread; false past the end of the lattice.
__device__ __forceinline__ bool pair_of_thread(const KParams& p, const PairGrid& w, int* xa, int* y, int* z) {
    if (w.dense) {
        const unsigned t = (unsigned)sweep_block(blockIdx.x, gridDim.x, p.reverse) * blockDim.x + threadIdx.x;
        const unsigned row = w.pairs.div(t);
        *z = (int)w.ny.div(row);
        *y = (int)row - *z * p.ny;
        *xa = 2 * (int)(t - row * w.pairs.d);
        return *z < p.nz;
    }
    *xa = 2 * (sweep_block(blockIdx.x, gridDim.x, p.reverse) * blockDim.x + threadIdx.x);
    *y = sweep_block(blockIdx.y, gridDim.y, p.reverse) * blockDim.y + threadIdx.y;
    *z = sweep_block(blockIdx.z, gridDim.z, p.reverse);
    return true;
}

// Where rows and slabs divide into blocks of 2^k pairs along x and whole rows along y, a 3D grid
// gives each thread its pair without a division; elsewhere (PairGrid::dense) pairs are numbered
// row by row over the whole lattice, so that no lane idles: with blocks of 2^k pairs along x, a 96^3 cavity idled a
// quarter of its lanes.  Measured (GB300, cavity n^3, us a step, 2^k blocks -> dense rows and
// paired face rows): FP32 32: 3.6 -> 3.1, 40: 4.8 -> 3.5, 64: 7.7 -> 7.2, 80: 18.5 -> 13.9,
// 96: 29.0 -> 26.1; FP16 96: 25.9 -> 20.0, 160: 126 -> 86.6.
template <bool HET, bool OUTF, class S, bool ENTH, class L, bool VEC>
__global__ void __maxnreg__((pair_regs<HET, S, ENTH, VEC>()))
    step_pair_kernel(const __grid_constant__ KParams p, const __grid_constant__ Planes pl,
                     const __grid_constant__ PairGrid w) {
    dependent_launch_prologue();
    int xa, y, z;
    const bool valid = pair_of_thread(p, w, &xa, &y, &z);
    const int mode = warp_pair_mode(p, xa, y, z, valid);
    if (valid) pair_update<HET, OUTF, S, ENTH, L, VEC>(pl, p, xa, y, z, mode, xa + 1 < p.nx);
}

#ifndef LBM_L2_FIRST
// The two steps of the AA scheme (aa_pair_pull, aa_pair_local), swept in alternate directions like
// the ping-pong steps: with one copy, twice the lattice stays in L2.  Measured (GB300, us a step,
// one site per thread -> here): 64^3 11.2 -> 7.5, 96^3 38.2 -> 20.7, 127^3 77 -> 61.6, 160^3 156 ->
// 117.8 (129 before the alternate sweep), 192^3 235 -> 205.7, field 160^3 176 -> 124.5.  Registers of
// the pull step, 160^3 at 96 / 104 / 112 / 128: 126.7 / 122.6 / 119.5 / 117.8.
template <bool HET, bool VEC>
__global__ void __maxnreg__(128)
    aa_pair_pull_kernel(const __grid_constant__ KParams p, const __grid_constant__ Planes pl,
                        const __grid_constant__ PairGrid w) {
    dependent_launch_prologue();
    int xa, y, z;
    const bool valid = pair_of_thread(p, w, &xa, &y, &z);
    const int mode = warp_pair_mode(p, xa, y, z, valid);
    if (valid) aa_pair_pull<HET, VEC>(p, pl, xa, y, z, mode, xa + 1 < p.nx);
}
template <bool HET, bool VEC>
__global__ void __maxnreg__(HET ? 128 : 96)
    aa_pair_local_kernel(const __grid_constant__ KParams p, const __grid_constant__ Planes pl,
                         const __grid_constant__ PairGrid w) {
    dependent_launch_prologue();
    int xa, y, z;
    if (pair_of_thread(p, w, &xa, &y, &z)) aa_pair_local<HET, VEC>(p, pl, xa, y, z, xa + 1 < p.nx);
}
#endif

// Grid of one thread per pair: 3D where rows and slabs divide into its blocks, else dense.
PairGrid pair_launch(const KParams& p, dim3* grid, dim3* block) {
    const unsigned nt = p.block_threads >= 32 && p.block_threads <= kBlock ? p.block_threads : 64;
    PairGrid w;
    w.pairs = FastDiv((unsigned)(p.nx + 1) / 2);
    w.ny = FastDiv((unsigned)p.ny);
    const unsigned n = w.pairs.d * (unsigned)(p.ny * p.nz);
    const unsigned bx = (unsigned)block_x_of((int)w.pairs.d, (int)nt), by = nt / bx;
    w.dense = w.pairs.d % bx != 0 || p.ny % by != 0;
    *block = w.dense ? dim3(nt) : dim3(bx, by);
    *grid = w.dense ? dim3((n + nt - 1) / nt) : dim3(w.pairs.d / bx, p.ny / by, p.nz);
    return w;
}

}  // namespace

#ifndef LBM_L2_FIRST
cudaError_t launch_aa_pair(const KParams& p, bool local, const Planes& pl, bool pdl, cudaStream_t st) {
    dim3 grid, block;
    const PairGrid w = pair_launch(p, &grid, &block);
    const bool het = p.phi_field != nullptr;
    auto run = [&](auto k) { return launch_kernel(pdl, k, grid, block, 0, st, p, pl, w); };
    if (p.nx % 2 == 0) {
        if (local) return het ? run(aa_pair_local_kernel<true, true>) : run(aa_pair_local_kernel<false, true>);
        return het ? run(aa_pair_pull_kernel<true, true>) : run(aa_pair_pull_kernel<false, true>);
    }
    if (local) return het ? run(aa_pair_local_kernel<true, false>) : run(aa_pair_local_kernel<false, false>);
    return het ? run(aa_pair_pull_kernel<true, false>) : run(aa_pair_pull_kernel<false, false>);
}

cudaError_t launch_step_pair(const KParams& p, bool outflow, const Planes& pl, bool pdl,
                             cudaStream_t st) {
#else
cudaError_t launch_step_pair_first(const KParams& p, bool outflow, const Planes& pl, bool pdl,
                                   cudaStream_t st) {
#endif
    dim3 grid, block;
    const PairGrid w = pair_launch(p, &grid, &block);
    const bool het = p.phi_field != nullptr, vec = p.nx % 2 == 0;
    if (p.enthalpy)  // FP32, uniform medium, no outflow (validated on the host)
        return vec ? launch_kernel(pdl, step_pair_kernel<false, false, StoreF32o, true, D3Q19, true>, grid,
                                   block, 0, st, p, pl, w)
                   : launch_kernel(pdl, step_pair_kernel<false, false, StoreF32o, true, D3Q19, false>, grid,
                                   block, 0, st, p, pl, w);
    auto go = [&](auto tag, auto lat, auto v) {
        using S = decltype(tag);
        using L = decltype(lat);
        constexpr bool V = decltype(v)::value;
        // formats with every load hinted: 16 bits with a porosity field, D3Q15; without a field the
        // FP16 kernel with an outflow has no register for a policy (ld_pop), and the 16-bit kernels but
        // FP16 without an outflow load their temperatures inline (ldT2)
        constexpr bool kQ15 = L::kQ == 15, kHalf = std::is_same<typename S::T, __half>::value;
        using H = typename std::conditional<kL2First && (S::kScaled || kQ15), HintAll<S>, S>::type;
        using B = typename std::conditional<S::kScaled && !kHalf, PinT<S>, S>::type;
        using U = typename std::conditional<kL2First && kQ15, HintAll<S>, B>::type;
        using P = typename std::conditional<kL2First && kHalf, HintStream<S>, PinT<S>>::type;
        using O = typename std::conditional<S::kScaled, P, U>::type;
        auto k = het ? (outflow ? step_pair_kernel<true, true, H, false, L, V>
                                : step_pair_kernel<true, false, H, false, L, V>)
                     : (outflow ? step_pair_kernel<false, true, O, false, L, V>
                                : step_pair_kernel<false, false, U, false, L, V>);
        return launch_kernel(pdl, k, grid, block, 0, st, p, pl, w);
    };
    auto pick = [&](auto v) {
        if (p.qf == 15) return go(StoreF32o{}, D3Q15{}, v);  // FP32 storage (validated on the host)
        if (p.storage == 1) return go(StoreF16o{}, D3Q19{}, v);
        if (p.storage == 2) return go(StoreBF16o{}, D3Q19{}, v);
        return go(StoreF32o{}, D3Q19{}, v);
    };
    return vec ? pick(std::true_type{}) : pick(std::false_type{});
}

}  // namespace lbm
