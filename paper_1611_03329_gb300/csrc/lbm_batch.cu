// Batched steps: one launch per time step for a group of lattices of the same kernel variant.
#define LBM_DEVICE_ONLY
#include "lbm_kernels.cu"

namespace lbm {
namespace {

// Batched step: one flat grid over the blocks of many lattices.  blk_lat[b] names the lattice
// of block b; the lattice's parameters and planes are read in place through the read-only
// cache (uniform over the block).  A block covers `rows` consecutive z-planes of one
// (x-segment, y-band) column, so the lookup is paid once per `rows` site updates.  L and NEE
// as in step_kernel: the D3Q15 flow lattice, node walls (a node-wall site takes nee_site).
template <bool HET, bool OUTF, class S, bool ENTH = false, class L = D3Q19, bool NEE = false>
__global__ void __launch_bounds__(kBlock, kStepMinBlocks - 1)
    batch_step_kernel(const BatchLattice* __restrict__ tab,
                      const unsigned short* __restrict__ blk_lat, int flip, int rows) {
    dependent_launch_prologue();
    const BatchLattice* B = tab + __ldg(blk_lat + blockIdx.x);
    const KParams& p = B->p;
    const Planes& pl = B->pl[B->cur ^ flip];
    const int bx = B->bx, gx = B->gx, gy = B->gy;
    const int local = (int)blockIdx.x - B->block_begin;
    const int by = blockDim.x / bx;
    const int tx = threadIdx.x & (bx - 1), ty = threadIdx.x / bx;
    const int bxi = local % gx, rest = local / gx;
    const int x = bxi * bx + tx;
    const int y = (rest % gy) * by + ty;
    const int z0 = (rest / gy) * rows;
    const bool valid = x < p.nx && y < p.ny;
    for (int r = 0; r < rows; ++r) {
        const int z = z0 + r;
        if (z >= p.nz) break;  // uniform over the block
        const unsigned nb = (NEE && valid) ? nee_bits(p, x, y, z) : 0u;  // node-wall site
        // every lane of the warp reaches the votes; only the valid lanes update a site (the
        // site update itself holds no warp-wide vote)
        const int mode = warp_gather_mode(p, x, y, z, valid && nb == 0u);
        if (!valid) continue;
        float f[L::kQ], g[kQT];
        const int s = x + p.nx * (y + p.ny * z);
        if constexpr (NEE) {
            if (nb) {
                nee_site<HET, true, S, L>(pl, p, x, y, z, s, nb, f, g);
#pragma unroll
                for (int i = 0; i < L::kQ; ++i) stp<S>(pl, p, i, s, f[i]);
#pragma unroll
                for (int i = 0; i < kQT; ++i) stg_dev<S>(pl, p, i, s, g[i], 0.0f);
                continue;
            }
        }
        gather_site<OUTF, S, L>(pl, p, x, y, z, s, mode, f, g);
        finish_site<HET, OUTF, S, ENTH, L>(pl, p, x, y, z, s, f, g);
    }
}

// Batched step with two x-adjacent sites per thread: the lattices of a group whose rows are all
// even (VEC) or all odd, halfway walls, 32-bit plane offsets.  Pairs are numbered row by row over
// each lattice (PairGrid) and a block takes `rows` runs of blockDim.x consecutive pairs of one
// lattice, so the lattice lookup is paid once per `rows` updates and no lane idles but at a
// lattice's end; each pair is updated by pair_update, as step_pair_kernel updates it, bit for bit.
// The parameters come from the lattice table in global memory, not from the constant bank, and
// take registers of their own: 128 per thread (16 warps per SM) keeps its spills to a few bytes
// (at the single kernel's 96-104 it spilled 200-400 bytes).
template <bool HET, bool OUTF, class S, bool ENTH, class L, bool VEC>
__global__ void __maxnreg__(128)
    batch_pair_kernel(const BatchLattice* __restrict__ tab,
                      const unsigned short* __restrict__ blk_lat, int flip, int rows) {
    dependent_launch_prologue();
    const BatchLattice* B = tab + __ldg(blk_lat + blockIdx.x);
    const KParams& p = B->p;
    const Planes& pl = B->pl[B->cur ^ flip];
    const FastDiv pairs = B->w.pairs, fy = B->w.ny;
    unsigned t = ((unsigned)blockIdx.x - (unsigned)B->block_begin) * (unsigned)rows * blockDim.x + threadIdx.x;
    for (int r = 0; r < rows; ++r, t += blockDim.x) {
        const unsigned row = pairs.div(t);
        const int z = (int)fy.div(row), y = (int)row - z * p.ny;
        const int xa = 2 * (int)(t - row * pairs.d);
        const bool valid = z < p.nz;
        const int mode = warp_pair_mode(p, xa, y, z, valid);
        if (valid) pair_update<HET, OUTF, S, ENTH, L, VEC>(pl, p, xa, y, z, mode, xa + 1 < p.nx);
    }
}

// Batched AA step: one flat grid over the blocks of the AA lattices of a group (FP32, D3Q19,
// no outflow), each lattice in its own phase.  Lattice L runs a pull step when
// (L->cur ^ flip) is 0 (its copy in the swapped layout) and a local step otherwise; L->pl[0] =
// (in: permuted, out: identity) and L->pl[1] = (in: identity, out: permuted) are the plane
// tables of its single copy, and pl[0] doubles as the local step's permuted input table.  The
// block -> site mapping is that of batch_step_kernel.
template <bool HET>
__global__ void __launch_bounds__(kBlock, kStepMinBlocks - 1)
    batch_aa_kernel(const BatchLattice* __restrict__ tab,
                    const unsigned short* __restrict__ blk_lat, int flip, int rows) {
    dependent_launch_prologue();
    const BatchLattice* L = tab + __ldg(blk_lat + blockIdx.x);
    const KParams& p = L->p;
    const bool local = ((L->cur ^ flip) & 1) != 0;  // uniform over the block
    const int bx = L->bx, gx = L->gx, gy = L->gy;
    const int loc = (int)blockIdx.x - L->block_begin;
    const int by = blockDim.x / bx;
    const int tx = threadIdx.x & (bx - 1), ty = threadIdx.x / bx;
    const int bxi = loc % gx, rest = loc / gx;
    const int x = bxi * bx + tx;
    const int y = (rest % gy) * by + ty;
    const int z0 = (rest / gy) * rows;
    const bool valid = x < p.nx && y < p.ny;
    for (int r = 0; r < rows; ++r) {
        const int z = z0 + r;
        if (z >= p.nz) break;  // uniform over the block
        // every lane reaches the votes; only the valid lanes update a site
        const int mode = warp_gather_mode(p, x, y, z, valid);
        if (!valid) continue;
        if (local) aa_local_site<HET>(p, L->pl[1], L->pl[0], x, y, z);
        else aa_pull_site<HET>(p, L->pl[0], x, y, z, mode);
    }
}

// The same with two sites per thread, in the runs of pairs of batch_pair_kernel.
template <bool HET, bool VEC>
__global__ void __maxnreg__(128)
    batch_aa_pair_kernel(const BatchLattice* __restrict__ tab,
                         const unsigned short* __restrict__ blk_lat, int flip, int rows) {
    dependent_launch_prologue();
    const BatchLattice* B = tab + __ldg(blk_lat + blockIdx.x);
    const KParams& p = B->p;
    const bool local = ((B->cur ^ flip) & 1) != 0;  // uniform over the block
    const FastDiv pairs = B->w.pairs, fy = B->w.ny;
    unsigned t = ((unsigned)blockIdx.x - (unsigned)B->block_begin) * (unsigned)rows * blockDim.x + threadIdx.x;
    for (int r = 0; r < rows; ++r, t += blockDim.x) {
        const unsigned row = pairs.div(t);
        const int z = (int)fy.div(row), y = (int)row - z * p.ny;
        const int xa = 2 * (int)(t - row * pairs.d);
        const bool valid = z < p.nz;
        const int mode = warp_pair_mode(p, xa, y, z, valid);
        if (!valid) continue;
        if (local) aa_pair_local<HET, VEC>(p, B->pl[1], xa, y, z, xa + 1 < p.nx);
        else aa_pair_pull<HET, VEC>(p, B->pl[0], xa, y, z, mode, xa + 1 < p.nx);
    }
}

}  // namespace

cudaError_t launch_batch_step(const BatchLattice* tab, const unsigned short* blk_lat, int nblocks,
                              int block_threads, int rows, const BatchVariant& g, int flip, bool pdl,
                              cudaStream_t st) {
    if (nblocks <= 0) return cudaSuccess;
    auto run = [&](auto k) {
        return launch_kernel(pdl, k, dim3((unsigned)nblocks), dim3((unsigned)block_threads), 0, st, tab,
                             blk_lat, flip, rows);
    };
    if (g.nee) {  // node walls: FP32 storage, no outflow (validated on the host)
        if (g.qf == 15) return g.het ? run(batch_step_kernel<true, false, StoreF32, false, D3Q15, true>)
                                     : run(batch_step_kernel<false, false, StoreF32, false, D3Q15, true>);
        return g.het ? run(batch_step_kernel<true, false, StoreF32, false, D3Q19, true>)
                     : run(batch_step_kernel<false, false, StoreF32, false, D3Q19, true>);
    }
    if (g.pair) {  // halfway walls, 32-bit plane offsets
        auto go = [&](auto tag, auto lat, auto v) {
            using S = decltype(tag);
            using L = decltype(lat);
            constexpr bool V = decltype(v)::value;
            if (g.het) return g.outflow ? run(batch_pair_kernel<true, true, S, false, L, V>)
                                        : run(batch_pair_kernel<true, false, S, false, L, V>);
            return g.outflow ? run(batch_pair_kernel<false, true, S, false, L, V>)
                             : run(batch_pair_kernel<false, false, S, false, L, V>);
        };
        auto pick = [&](auto v) {
            constexpr bool V = decltype(v)::value;
            if (g.enthalpy) return run(batch_pair_kernel<false, false, StoreF32o, true, D3Q19, V>);
            if (g.qf == 15) return go(StoreF32o{}, D3Q15{}, v);
            if (g.storage == 1) return go(StoreF16o{}, D3Q19{}, v);
            if (g.storage == 2) return go(StoreBF16o{}, D3Q19{}, v);
            return go(StoreF32o{}, D3Q19{}, v);
        };
        return g.vec ? pick(std::true_type{}) : pick(std::false_type{});
    }
    // plane offsets beyond 32 bits: one site per thread
    if (g.enthalpy) return run(batch_step_kernel<false, false, StoreF32, true>);
    if (g.qf == 15) {
        if (g.het) return g.outflow ? run(batch_step_kernel<true, true, StoreF32, false, D3Q15>)
                                    : run(batch_step_kernel<true, false, StoreF32, false, D3Q15>);
        return g.outflow ? run(batch_step_kernel<false, true, StoreF32, false, D3Q15>)
                         : run(batch_step_kernel<false, false, StoreF32, false, D3Q15>);
    }
    return with_storage(g.storage, [&](auto tag) {
        using S = decltype(tag);
        if (g.het) return g.outflow ? run(batch_step_kernel<true, true, S>) : run(batch_step_kernel<true, false, S>);
        return g.outflow ? run(batch_step_kernel<false, true, S>) : run(batch_step_kernel<false, false, S>);
    });
}

cudaError_t launch_batch_aa(const BatchLattice* tab, const unsigned short* blk_lat, int nblocks,
                            int block_threads, int rows, const BatchVariant& g, int flip, bool pdl,
                            cudaStream_t st) {
    if (nblocks <= 0) return cudaSuccess;
    auto run = [&](auto k) {
        return launch_kernel(pdl, k, dim3((unsigned)nblocks), dim3((unsigned)block_threads), 0, st, tab,
                             blk_lat, flip, rows);
    };
    if (g.pair && g.vec) return g.het ? run(batch_aa_pair_kernel<true, true>) : run(batch_aa_pair_kernel<false, true>);
    if (g.pair) return g.het ? run(batch_aa_pair_kernel<true, false>) : run(batch_aa_pair_kernel<false, false>);
    return g.het ? run(batch_aa_kernel<true>) : run(batch_aa_kernel<false>);
}

int batch_layout(const KParams& p, bool pair, int block_threads, int rows, BatchLattice* L) {
    L->w.pairs = FastDiv((unsigned)(p.nx + 1) / 2);
    L->w.ny = FastDiv((unsigned)p.ny);
    L->w.dense = 1;
    if (pair) {
        L->bx = L->gx = L->gy = 0;
        const long long n = (long long)L->w.pairs.d * p.ny * p.nz, per = (long long)block_threads * rows;
        return (int)((n + per - 1) / per);
    }
    L->bx = block_x_of(p.nx, block_threads);
    const int by = block_threads / L->bx;
    L->gx = (p.nx + L->bx - 1) / L->bx;
    L->gy = (p.ny + by - 1) / by;
    return L->gx * L->gy * ((p.nz + rows - 1) / rows);
}

}  // namespace lbm
