// Macroscopic fields and the steady-state residual, two x-adjacent sites per thread: the gather
// and the moments of the step (gather_pair_*, collide_t without the relaxation) over the whole
// lattice, the fields stored, and, for a residual, the sums of (u - u_prev)^2, u^2, (T -
// T_prev)^2, T^2 and the non-finite values taken while they are in registers.  The last block to
// finish adds up the blocks' partial sums in a fixed order and writes the totals where the host
// reads them, so a residual is one launch and no copy.
//
// What bounds it: reading the 26 populations, and in a residual the FP64 sums (a GB300 SM adds
// two FP64 values per clock).  Measured (GB300, us for the call with its synchronisation, lattice
// alone; one site per thread with predicated loads, then a second and a third kernel and a copy
// for the sums -> here): fields BF16 128^3 157 -> 50, FP16 256x64x64 56 -> 28, FP32 39 -> 34;
// residual 32^3 53 -> 27, 63x61x59 60 -> 39, BF16 128^3 296 -> 128, FP32 256^3 1231 -> 753
// (814 with the conversions and differences in FP64).
#define LBM_DEVICE_ONLY
#include "lbm_kernels.cu"

namespace lbm {
namespace {

constexpr int kFThreads = 128;  // 608 blocks of 128 threads are resident at once (152 SMs)

// Sums of the block's NV values per thread, in out[0 .. NV) of thread 0's choice.
template <int NV>
__device__ __forceinline__ void block_sums(double (&v)[NV], double* out) {
    __shared__ double sh[NV][kFThreads / 32];
#pragma unroll
    for (int k = 0; k < NV; ++k) {
        double x = v[k];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
        if ((threadIdx.x & 31) == 0) sh[k][threadIdx.x >> 5] = x;
    }
    __syncthreads();
    if (threadIdx.x < NV) {
        double x = 0.0;
#pragma unroll
        for (int w = 0; w < kFThreads / 32; ++w) x += sh[threadIdx.x][w];
        out[threadIdx.x] = x;
    }
}

// An FP32 value as FP64 by integer operations (exact): the conversion instruction shares the FP64
// pipe.  Subnormal values take the instruction; a non-finite one gives a finite value here (it is
// counted as non-finite, and the sums are then not used).
__device__ __forceinline__ double widen(float x) {
    const unsigned u = __float_as_uint(x), a = u & 0x7fffffffu;
    if (a != 0u && a < 0x00800000u) return (double)x;
    const unsigned hi = a ? (u & 0x80000000u) | ((a >> 3) + 0x38000000u) : 0u;
    return __hiloint2double((int)hi, (int)(u << 29));
}
// a - b in FP64.  Between two residuals the fields change little and the FP32 difference is exact
// (the error term of the two-sum is 0): it is widened instead of both operands.
__device__ __forceinline__ double diff(float a, float b, double aw) {
    const float s = __fsub_rn(a, b), bb = __fsub_rn(s, a);
    const float e = __fsub_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fadd_rn(b, bb));
    return e == 0.0f ? widen(s) : aw - widen(b);
}
// One site's terms of the residual sums (FP64; the finiteness of the FP32 values needs none).
__device__ __forceinline__ void residual_add(double (&v)[5], float x, float y, float z, float xp,
                                             float yp, float zp, float T, float Tp) {
    const float c[3] = {x, y, z}, cp[3] = {xp, yp, zp};
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const double q = widen(c[a]), d = diff(c[a], cp[a], q);
        v[0] += d * d;
        v[1] += q * q;
        if (!isfinite(c[a])) v[4] += 1.0;
    }
    const double t = widen(T), dt = diff(T, Tp, t);
    v[2] += dt * dt;
    v[3] += t * t;
    if (!isfinite(T)) v[4] += 1.0;
}

// What a launch reads and writes: rho, u (3 planes), T may be null; sums: the residual against pu,
// pT (null: the fields themselves).  vst: the field pointers take aligned 2-element accesses.
struct Fields {
    float* rho;
    float* u;
    float* T;
    const float* pu;
    const float* pT;
    bool sums, vst;
};

// Blocks j of nr (both uniform over the block): pairs j * kFThreads + thread, then every
// nr * kFThreads further, so that a lattice's sums do not depend on what else the grid holds.
template <bool HET, bool OUTF, class S, bool ENTH, class L, bool VEC>
__device__ __forceinline__ void fields_block(const KParams& p, const Planes& pl, const PairGrid& w,
                                             const Fields& o, int j, int nr, double (&v)[5]) {
    const unsigned n = w.pairs.d * (unsigned)(p.ny * p.nz), stride = (unsigned)nr * kFThreads;
    for (unsigned k = (unsigned)j * kFThreads; k < n; k += stride) {
        const unsigned t = k + threadIdx.x;
        const unsigned row = w.pairs.div(t);
        const int z = (int)w.ny.div(row), y = (int)row - z * p.ny;
        const int xa = 2 * (int)(t - row * w.pairs.d);
        const bool valid = t < n;
        const int mode = warp_pair_mode(p, xa, y, z, valid);
        if (!valid) continue;
        const bool vb = VEC || xa + 1 < p.nx;
        const int sa = xa + p.nx * (y + p.ny * z);
        L2 f[L::kQ], g[kQT];
        if (mode == kGatherInterior) gather_pair_interior<S, L, VEC>(pl, p, xa, y, z, sa, f, g);
        else if (mode == kGatherX) gather_pair_sel<OUTF, S, L, VEC, false>(pl, p, xa, y, z, sa, vb, f, g);
        else gather_pair_sel<OUTF, S, L, VEC, true>(pl, p, xa, y, z, sa, vb, f, g);
        const MediumT<L2> md = medium_pair<HET>(p, sa, vb ? 1 : 0);
        MacroT<L2> m;
        if constexpr (L::kQ == 15) m = collide15_t<L2, false>(p, md, f, g);
        else m = collide_t<L2, false, ENTH>(p, md, f, g);
        const long long ns = p.ns;
        auto put = [&](float* a, L2 x) {
            if (!a) return;
            a += sa;
            if (VEC && o.vst) {
                *reinterpret_cast<float2*>(a) = x.v;
            } else {
                a[0] = x.v.x;
                if (vb) a[1] = x.v.y;
            }
        };
        put(o.rho, m.rho);
        put(o.u, m.ux);
        put(o.u ? o.u + ns : nullptr, m.uy);
        put(o.u ? o.u + 2 * ns : nullptr, m.uz);
        put(o.T, m.T);
        if (!o.sums) continue;
        L2 px = m.ux, py = m.uy, pz = m.uz, pT = m.T;
        if (o.pu) {
            auto get = [&](const float* a) {
                a += sa;
                if constexpr (VEC) return L2{*reinterpret_cast<const float2*>(a)};
                else return pair(a[0], vb ? a[1] : 0.0f);
            };
            px = get(o.pu);
            py = get(o.pu + ns);
            pz = get(o.pu + 2 * ns);
            pT = get(o.pT);
        }
        residual_add(v, m.ux.v.x, m.uy.v.x, m.uz.v.x, px.v.x, py.v.x, pz.v.x, m.T.v.x, pT.v.x);
        if (vb)
            residual_add(v, m.ux.v.y, m.uy.v.y, m.uz.v.y, px.v.y, py.v.y, pz.v.y, m.T.v.y, pT.v.y);
    }
}

// After a block's sums are in partials[5 j]: whether this block is the last of nr to arrive; it
// then holds the totals in out (5 doubles, any memory the GPU writes) and the counter is 0 again.
__device__ __forceinline__ void residual_finish(double (&v)[5], double* partials, int j, int nr,
                                                unsigned* arrived, double* out) {
    __shared__ bool last;
    block_sums<5>(v, partials + 5 * j);
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(arrived, 1u) == (unsigned)nr - 1u;
    __syncthreads();
    if (!last) return;
    __threadfence();
#pragma unroll
    for (int k = 0; k < 5; ++k) v[k] = 0.0;
    for (int b = threadIdx.x; b < nr; b += kFThreads)
#pragma unroll
        for (int k = 0; k < 5; ++k) v[k] += __ldcg(partials + 5 * b + k);
    block_sums<5>(v, out);
    if (threadIdx.x == 0) {
        *arrived = 0u;
        __threadfence_system();
    }
}

template <bool HET, bool OUTF, class S, bool ENTH, class L, bool VEC>
__global__ void __launch_bounds__(kFThreads, 4)
    fields_kernel(const __grid_constant__ KParams p, const __grid_constant__ Planes pl,
                  const __grid_constant__ PairGrid w, const __grid_constant__ Fields o,
                  double* __restrict__ partials, unsigned* arrived, double* out) {
    double v[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
    fields_block<HET, OUTF, S, ENTH, L, VEC>(p, pl, w, o, (int)blockIdx.x, (int)gridDim.x, v);
    if (o.sums) residual_finish(v, partials, (int)blockIdx.x, (int)gridDim.x, arrived, out);
}

// The residuals of many lattices: block b takes lattice blk[b].x as its block blk[b].y, with the
// sums of fields_kernel over the same number of blocks, bit for bit.
template <bool HET, bool OUTF, class S, bool ENTH, bool VEC>
__global__ void __launch_bounds__(kFThreads, 4)
    batch_residual_kernel(ResLattice* __restrict__ tab, const int2* __restrict__ blk) {
    const int2 lb = blk[blockIdx.x];
    ResLattice& R = tab[lb.x];
    double v[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
    const Fields o{nullptr, R.cu, R.cT, R.pu, R.pT, true, true};
    fields_block<HET, OUTF, S, ENTH, D3Q19, VEC>(R.p, R.pl, R.w, o, lb.y, R.nr, v);
    residual_finish(v, R.partials, lb.y, R.nr, &R.arrived, R.out);
}

PairGrid pair_grid(const KParams& p) {
    PairGrid w;
    w.pairs = FastDiv((unsigned)(p.nx + 1) / 2);
    w.ny = FastDiv((unsigned)p.ny);
    w.dense = 1;
    return w;
}

}  // namespace

// Blocks of a lattice's fields: one per kFThreads pairs, in whole passes over at most
// reduction_blocks() blocks.
int fields_blocks(const KParams& p) {
    const long long pairs = (long long)((p.nx + 1) / 2) * p.ny * p.nz;
    const long long nb = (pairs + kFThreads - 1) / kFThreads, most = reduction_blocks();
    const long long passes = (nb + most - 1) / most;
    return (int)((nb + passes - 1) / passes);
}

cudaError_t launch_fields(const KParams& p, bool outflow, const Planes& pl, float* rho, float* u,
                          float* T, const float* pu, const float* pT, double* partials,
                          unsigned* arrived, double* out, cudaStream_t st) {
    const PairGrid w = pair_grid(p);
    auto even = [](const void* a) { return (reinterpret_cast<uintptr_t>(a) & 7u) == 0u; };
    const Fields o{rho, u, T, pu, pT, out != nullptr, even(rho) && even(u) && even(T)};
    const int blocks = fields_blocks(p);
    const bool het = p.phi_field != nullptr, vec = p.nx % 2 == 0;
    auto run = [&](auto k) {
        k<<<blocks, kFThreads, 0, st>>>(p, pl, w, o, partials, arrived, out);
        return cudaGetLastError();
    };
    auto go = [&](auto tag, auto lat, auto v) {
        using S = decltype(tag);
        using L = decltype(lat);
        constexpr bool V = decltype(v)::value;
        if (het) return outflow ? run(fields_kernel<true, true, S, false, L, V>)
                                : run(fields_kernel<true, false, S, false, L, V>);
        return outflow ? run(fields_kernel<false, true, S, false, L, V>)
                       : run(fields_kernel<false, false, S, false, L, V>);
    };
    auto pick = [&](auto v) {
        constexpr bool V = decltype(v)::value;
        if (p.enthalpy) return run(fields_kernel<false, false, StoreF32o, true, D3Q19, V>);
        if (p.qf == 15) return go(StoreF32o{}, D3Q15{}, v);
        if (p.storage == 1) return go(StoreF16o{}, D3Q19{}, v);
        if (p.storage == 2) return go(StoreBF16o{}, D3Q19{}, v);
        return go(StoreF32o{}, D3Q19{}, v);
    };
    return vec ? pick(std::true_type{}) : pick(std::false_type{});
}

void residual_grid(ResLattice* R) { R->w = pair_grid(R->p); }

cudaError_t launch_batch_residual(ResLattice* tab, const int2* blk, int nblocks, bool het, bool outflow,
                                  int storage, bool enthalpy, bool vec, cudaStream_t st) {
    if (nblocks < 1) return cudaSuccess;
    auto run = [&](auto k) {
        k<<<nblocks, kFThreads, 0, st>>>(tab, blk);
        return cudaGetLastError();
    };
    auto go = [&](auto tag, auto v) {
        using S = decltype(tag);
        constexpr bool V = decltype(v)::value;
        if (het) return outflow ? run(batch_residual_kernel<true, true, S, false, V>)
                                : run(batch_residual_kernel<true, false, S, false, V>);
        return outflow ? run(batch_residual_kernel<false, true, S, false, V>)
                       : run(batch_residual_kernel<false, false, S, false, V>);
    };
    auto pick = [&](auto v) {
        constexpr bool V = decltype(v)::value;
        if (enthalpy) return run(batch_residual_kernel<false, false, StoreF32o, true, V>);
        if (storage == 1) return go(StoreF16o{}, v);
        if (storage == 2) return go(StoreBF16o{}, v);
        return go(StoreF32o{}, v);
    };
    return vec ? pick(std::true_type{}) : pick(std::false_type{});
}

}  // namespace lbm
