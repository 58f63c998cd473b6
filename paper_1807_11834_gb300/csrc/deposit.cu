// deposit.cu -- (a1) porosity and (a3) reaction deposition onto the bulk
// grid, the bulk pack feeding the drag gather, and the FP64 conservation
// sums.
//
// Porosity (Table 1 of arXiv 1807.11834: porosity field from the particle
// volumes of a cell; Sec. 2.4, beside Eq. DragLaw: porosity = fluid volume / cell volume):
// phi_B = sum_{p in B} V_p / V_B, eps_B = 1 - phi_B.
// Reaction (Eq. UFP: F_fpi is the fluid-side reaction to F_drag):
// S_B = -(1/V_B) sum_{p in B} F_p.
//
// The porosity is a sum of whole numbers per cell (volume_add_row, exact in
// any order); the reaction a segmented sum over the stable bin order with
// compensated carries, so its result depends only on the particle set of the
// cell, never on the launch shape.
#include <algorithm>

#include "cg_internal.cuh"
#include "batch.cuh"

namespace cg {


template <typename T>
__device__ __forceinline__ void fill_body(T* __restrict__ a, long long m, T v, Blk b) {
    for (long long i = b.id * blockDim.x + threadIdx.x; i < m; i += b.n * blockDim.x) a[i] = v;
}

// ----------------------------------------------------------------------
// Porosity: the spheres of the binned order to their cells' accumulators,
// then one pass over the cells (an incremental binning does both itself).
// Rows of 32 consecutive slots per warp, four rows loaded ahead; GATHER: the
// diameters from the caller's records through the permutation, else in
// sorted order already.  About 60 instructions per row, where the segmented
// compensated sums took 110 to 140 (4M packed 25 -> 15 us, FP64 1M 82 -> 15.5).
// ----------------------------------------------------------------------
template <typename T, bool GATHER>
__device__ __forceinline__ void volume_rows_body(const T* __restrict__ d, long long n, const int32_t* __restrict__ perm,
                                                 const int32_t* __restrict__ key_sorted, const GridDev& g,
                                                 const EpsOut<T>& o, Blk b) {
    constexpr int B = 4;
    const int lane = threadIdx.x & 31;
    const long long span = (long long)blockDim.x * B, step = b.n * span;
    for (long long r0 = b.id * span + (threadIdx.x >> 5) * (32 * B); r0 < n; r0 += step) {
        int key[B];
        T v[B];
#pragma unroll
        for (int j = 0; j < B; ++j) {
            const long long i = r0 + 32 * j + lane;
            key[j] = -1;
            v[j] = T(0);
            if (i < n) {
                key[j] = __ldg(key_sorted + i);
                v[j] = GATHER ? __ldg(d + 4 * (long long)__ldg(perm + i) + 3) : __ldg(d + i);
            }
        }
#pragma unroll
        for (int j = 0; j < B; ++j) {
            if (r0 + 32 * j >= n) break;   // warp-uniform
            volume_add_row_wide(key[j] >= 0, key[j], v[j], g, o.acc);
        }
    }
}

template <typename T, bool GATHER>
__global__ void __launch_bounds__(256)
k_volume_rows(const T* __restrict__ d, long long n, const int32_t* __restrict__ perm,
              const int32_t* __restrict__ key_sorted, GridDev g, EpsOut<T> o) {
    pdl_wait();
    volume_rows_body<T, GATHER>(d, n, perm, key_sorted, g, o, launch_blk());
}

template <typename T, bool SUMS>
__global__ void __launch_bounds__(256) k_eps_finish(GridDev g, int items, EpsOut<T> o, T* __restrict__ part) {
    pdl_wait();
    // the cells of a block as in the incremental binning's pass over them, so
    // that the sums come out the same
    CSum<T> tot[1];
    for (int j = 0; j < items; ++j) {
        const long long c = ((long long)blockIdx.x * items + j) * 256 + threadIdx.x;
        if (c < g.nbulk) eps_finish<T, SUMS>(c, g, o, tot[0]);
    }
    if (SUMS) block_sums<T, 1>(tot, part, gridDim.x, blockIdx.x);
}

// Reaction from the forces the drag wrote in sorted order (T4 per slot).
template <typename T>
__device__ __forceinline__ void deposit_sorted_force_body(const T* __restrict__ Fs, long long n,
                                                          const int32_t* __restrict__ key_sorted,
                                                          const int32_t* __restrict__ cs, const GridDev& g,
                                                          T* __restrict__ S, Blk b) {
    const long long wg = b.id * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const long long nw = b.n * (blockDim.x >> 5);
    for (long long base = wg * seg_chunk(n); base < n; base += nw * seg_chunk(n)) {
        long long s, t;
        seg_chunk_range(base, n, key_sorted, cs, s, t);
        seg_rounds<T, 3>(
            s, t, key_sorted,
            [&](long long i, T (&v)[3]) {
                const V4<T> f = ld4(Fs, i);
                v[0] = f.x;
                v[1] = f.y;
                v[2] = f.z;
            },
            [&](int key, int k, T sum) { reaction_emit<T>(g, S, key, k, sum); });
    }
}

// Semi-implicit coefficients (Eq. UFP): per cell A = (1/V_B) sum beta and
// b = (1/V_B) sum beta u_p from the drag's sorted (beta, beta u) records,
// with the reaction's segmented sums.
template <typename T>
__device__ __forceinline__ void deposit_implicit_body(const T* __restrict__ Bs, long long n,
                                                      const int32_t* __restrict__ key_sorted,
                                                      const int32_t* __restrict__ cs, const GridDev& g,
                                                      T* __restrict__ coef, Blk b) {
    const long long wg = b.id * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const long long nw = b.n * (blockDim.x >> 5);
    for (long long base = wg * seg_chunk(n); base < n; base += nw * seg_chunk(n)) {
        long long s, t;
        seg_chunk_range(base, n, key_sorted, cs, s, t);
        seg_rounds<T, 4>(
            s, t, key_sorted,
            [&](long long i, T (&v)[4]) {
                const V4<T> r = ld4(Bs, i);
                v[0] = r.x;
                v[1] = r.y;
                v[2] = r.z;
                v[3] = r.w;
            },
            [&](int key, int k, T sum) {
                coef[k * g.nbulk + key] = sum * (sizeof(T) == 4 ? (T)g.invVBf : (T)g.invVB);
            });
    }
}

template <typename T>
__global__ void __launch_bounds__(256, 4)
k_deposit_implicit(const T* __restrict__ Bs, long long n, const int32_t* __restrict__ key_sorted,
                   const int32_t* __restrict__ cs, GridDev g, T* __restrict__ coef) {
    pdl_wait();
    deposit_implicit_body<T>(Bs, n, key_sorted, cs, g, coef, launch_blk());
}

template <typename T>
__global__ void __launch_bounds__(256, sizeof(T) == 4 ? 5 : 4)
k_deposit_sorted_force(const T* __restrict__ Fs, long long n, const int32_t* __restrict__ key_sorted,
                       const int32_t* __restrict__ cs, GridDev g, T* __restrict__ S) {
    pdl_wait();
    deposit_sorted_force_body(Fs, n, key_sorted, cs, g, S, launch_blk());
}

// ----------------------------------------------------------------------
// Reaction source from caller-order SoA forces, over the sorted order as
// above (inside the coupling step the reaction is fused into the drag).
// S_B must be zero beforehand for cells without particles.
// ----------------------------------------------------------------------
template <typename T>
__global__ void __launch_bounds__(256)
k_deposit_momentum(const T* __restrict__ F, long long n, const int32_t* __restrict__ perm,
                   const int32_t* __restrict__ key_sorted, const int32_t* __restrict__ cs, GridDev g,
                   T* __restrict__ S) {
    pdl_wait();
    const long long wg = (long long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const long long nw = (long long)gridDim.x * (blockDim.x >> 5);
    for (long long base = wg * seg_chunk(n); base < n; base += nw * seg_chunk(n)) {
        long long s, t;
        seg_chunk_range(base, n, key_sorted, cs, s, t);
        seg_rounds<T, 3>(
            s, t, key_sorted,
            [&](long long i, T (&v)[3]) {
                const long long p = __ldg(perm + i);
#pragma unroll
                for (int k = 0; k < 3; ++k) v[k] = __ldg(F + k * n + p);
            },
            [&](int key, int k, T sum) { reaction_emit<T>(g, S, key, k, sum); });
    }
}

// ----------------------------------------------------------------------
// Pack the bulk fields read by the drag gather: (eps, u_x, u_y, u_z) per
// cell in the path precision.  Interpolating eps itself (not 1 - eps) keeps
// the porosity at the particle accurate to a few roundings of eps also in
// near-packed cells, where the drag is most sensitive to it.
// ----------------------------------------------------------------------
template <typename T>
__device__ __forceinline__ void pack_body(const double* __restrict__ eps, const T* __restrict__ u, const GridDev& g,
                                          T* __restrict__ bulk4, T* __restrict__ eps_t, Blk b) {
    for (long long c = b.id * blockDim.x + threadIdx.x; c < g.nbulk; c += b.n * blockDim.x) {
        const double e = __ldg(eps + c);
        st4(bulk4, c, (T)e, __ldg(u + c), __ldg(u + g.nbulk + c), __ldg(u + 2 * g.nbulk + c));
        if (eps_t) eps_t[c] = (T)e;
    }
}

template <typename T>
__global__ void __launch_bounds__(256)
k_pack(const double* __restrict__ eps, const T* __restrict__ u, GridDev g, T* __restrict__ bulk4,
       T* __restrict__ eps_t) {
    pdl_wait();
    pack_body(eps, u, g, bulk4, eps_t, launch_blk());
}

// ----------------------------------------------------------------------
// Final FP64 reduction of the block partials (one block, fixed order)
// ----------------------------------------------------------------------

// One block per sum: merge the compensated pairs in a fixed order (strided
// per thread, then a fixed tree), convert the final pair to double.
template <typename T>
__device__ __forceinline__ void sums_body(const T* __restrict__ part, const SumsMap& map, double* __restrict__ sums,
                                          Blk b) {
    __shared__ T sh_s[8], sh_c[8];
    const int nw = blockDim.x >> 5;
    const int k = (int)b.id;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    CSum<T> a;
    if (map.off[k] >= 0)
        for (long long i = threadIdx.x; i < map.cnt[k]; i += blockDim.x) {
            CSum<T> o;
            o.s = part[2 * (map.off[k] + i)];
            o.c = part[2 * (map.off[k] + i) + 1];
            a.merge(o);
        }
    a = warp_reduce(a);
    if (lane == 0) {
        sh_s[warp] = a.s;
        sh_c[warp] = a.c;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        CSum<T> t;
        t.s = sh_s[0];
        t.c = sh_c[0];
        for (int w = 1; w < nw; ++w) {
            CSum<T> o;
            o.s = sh_s[w];
            o.c = sh_c[w];
            t.merge(o);
        }
        sums[k] = map.off[k] >= 0 ? (double)t.s + (double)t.c : __longlong_as_double(0x7ff8000000000000LL);
    }
}

template <typename T>
__global__ void __launch_bounds__(256) k_sums(const T* __restrict__ part, SumsMap map, double* __restrict__ sums) {
    pdl_wait();
    sums_body(part, map, sums, launch_blk());
}

// ----------------------------------------------------------------------
// Batched phases (FP32 instances): zeroing, porosity, pack, reaction, sums
// ----------------------------------------------------------------------
// Cell counts to 0.
__global__ void __launch_bounds__(256) kb_zero(BLaunch L) {
    batch_loop(L, [&](const BInst& I, Blk b) { fill_body<int32_t>(I.count, I.gd.nbulk + 1, 0, b); });
}

__global__ void __launch_bounds__(256) kb_deposit_volume(BLaunch L) {
    batch_loop(L, [&](const BInst& I, Blk b) {
        volume_rows_body<float, false>(I.vol_sorted, I.n, nullptr, I.key_sorted, I.gd, I.eps_out, b);
    });
}

// The porosity from the accumulators, and the drag's record with the mean velocity.
__global__ void __launch_bounds__(256) kb_pack(BLaunch L) {
    batch_loop(L, [&](const BInst& I, Blk b) {
        CSum<float> tot[1];
        const GridDev& g = I.gd;
        for (long long c = b.id * blockDim.x + threadIdx.x; c < g.nbulk; c += b.n * blockDim.x) {
            eps_finish<float, true>(c, g, I.eps_out, tot[0]);
#pragma unroll
            for (int k = 0; k < 3; ++k) I.bulk4[4 * c + 1 + k] = __ldg(I.u_bulk + k * g.nbulk + c);
        }
        if (I.sums) block_sums<float, 1>(tot, I.part + 2 * I.part_off[PS_VOL], I.part_blocks[PS_VOL], b.id);
    });
}

__global__ void __launch_bounds__(256) kb_deposit_momentum(BLaunch L) {
    batch_loop(L, [&](const BInst& I, Blk b) {
        deposit_sorted_force_body<float>(I.Fs, I.n, I.key_sorted, I.count, I.gd, I.S_bulk, b);
    });
}

__global__ void __launch_bounds__(256) kb_sums(BLaunch L) {
    batch_loop(L, [&](const BInst& I, Blk b) { sums_body<float>(I.part, I.smap, I.sums, b); });
}

cg_status launch_batch_deposit(int phase, const BLaunch& L, unsigned grid, cudaStream_t s) {
    if (L.total == 0 || grid == 0) return CG_OK;
    switch (phase) {
        case BP_ZERO: kb_zero<<<grid, 256, 0, s>>>(L); break;
        case BP_DEPV: kb_deposit_volume<<<grid, 256, 0, s>>>(L); break;
        case BP_PACK: kb_pack<<<grid, 256, 0, s>>>(L); break;
        case BP_DEPM: kb_deposit_momentum<<<grid, 256, 0, s>>>(L); break;
        case BP_SUMS: kb_sums<<<grid, 256, 0, s>>>(L); break;
        default: return CG_ERR_INVALID_ARG;
    }
    CG_CUDA(cudaGetLastError());
    return CG_OK;
}

int batch_deposit_occupancy(int phase) {
    int occ = 0;
    cudaError_t e = cudaSuccess;
    switch (phase) {
        case BP_ZERO: e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kb_zero, 256, 0); break;
        case BP_DEPV: e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kb_deposit_volume, 256, 0); break;
        case BP_PACK: e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kb_pack, 256, 0); break;
        case BP_DEPM: e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kb_deposit_momentum, 256, 0); break;
        default: e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kb_sums, 256, 0); break;
    }
    if (e != cudaSuccess) {
        cudaGetLastError();
        return 1;
    }
    return occ > 0 ? occ : 1;
}

// ----------------------------------------------------------------------
// Launchers
// ----------------------------------------------------------------------
static inline unsigned blocks_for(long long n, int per) { return (unsigned)((n + per - 1) / per); }

// Grid of the segmented deposits: at most one chunk per warp, and no more
// CTAs than are resident at once (the reaction's 48 registers allow five per
// SM, 64 four), so the grid-stride loop runs without a second, partial wave.
static unsigned seg_blocks(cg_grids* g, long long n, int per_sm = 4) {
    const long long chunks = (n + seg_chunk(n) - 1) / seg_chunk(n), per = seg_threads(g, n) / 32;
    return (unsigned)std::max(1LL, std::min((chunks + per - 1) / per, (long long)g->num_sms * per_sm * 8 / per));
}

template <typename T>
static cg_status deposit_volume_launches(cg_grids* g, long long n, const T* pos_d, StepEps* e) {
    const EpsOut<T> o = eps_out<T>(g, e);
    if (n > 0) {
        const unsigned nblk = (unsigned)std::min<long long>((n + 1023) / 1024, (long long)g->num_sms * 8);
        if (pos_d)
            CG_LAUNCH(g, "deposit_volume", (k_volume_rows<T, true>), nblk, 256, 0, pos_d, n, (const int32_t*)g->perm,
                      (const int32_t*)g->key_sorted, g->gd, o);
        else
            CG_LAUNCH(g, "deposit_volume", (k_volume_rows<T, false>), nblk, 256, 0, (const T*)g->vol_sorted, n,
                      (const int32_t*)g->perm, (const int32_t*)g->key_sorted, g->gd, o);
    }
    const unsigned fblk = (unsigned)cell_blocks(g->gd.nbulk, sizeof(T) == 8);
    const int items = cell_items(g->gd.nbulk, sizeof(T) == 8);
    T* part = (T*)part_ptr(g, PS_VOL);
    g->part_blocks[PS_VOL] = e->sums ? (long long)fblk : -1;
    if (e->sums) CG_LAUNCH(g, "deposit_volume", (k_eps_finish<T, true>), fblk, 256, 0, g->gd, items, o, part);
    else CG_LAUNCH(g, "deposit_volume", (k_eps_finish<T, false>), fblk, 256, 0, g->gd, items, o, part);
    e->formed = true;
    if (e->ready) CG_CUDA(cudaEventRecord(e->ready, g->stream));
    return CG_OK;
}

cg_status launch_deposit_volume(cg_grids* g, long long n, const void* pos_d, StepEps* e) {
    const cg_status st = g->fp64 ? deposit_volume_launches<double>(g, n, (const double*)pos_d, e)
                                 : deposit_volume_launches<float>(g, n, (const float*)pos_d, e);
    if (st != CG_OK) {
        clear_volumes(g, g->stream);
        cudaGetLastError();
    }
    return st;
}

cg_status launch_deposit_sorted_force(cg_grids* g, long long n, void* S_bulk, bool cleared) {
    if (!cleared) CG_CUDA(cudaMemsetAsync(S_bulk, 0, 3 * g->tsize * (size_t)g->gd.nbulk, g->stream));
    if (n == 0) return CG_OK;
    const unsigned nblk = seg_blocks(g, n, 5);
    if (g->fp64)
        CG_LAUNCH(g, "deposit_momentum", k_deposit_sorted_force<double>, nblk, seg_threads(g, n), 0, (const double*)g->Fs, n,
                  g->key_sorted, g->cell_start, g->gd, (double*)S_bulk);
    else
        CG_LAUNCH(g, "deposit_momentum", k_deposit_sorted_force<float>, nblk, seg_threads(g, n), 0, (const float*)g->Fs, n,
                  g->key_sorted, g->cell_start, g->gd, (float*)S_bulk);
    return CG_OK;
}

cg_status launch_deposit_implicit(cg_grids* g, long long n, void* coef_bulk) {
    CG_CUDA(cudaMemsetAsync(coef_bulk, 0, 4 * g->tsize * (size_t)g->gd.nbulk, g->stream));
    if (n == 0) return CG_OK;
    const unsigned nblk = seg_blocks(g, n);
    if (g->fp64)
        CG_LAUNCH(g, "deposit_implicit", k_deposit_implicit<double>, nblk, seg_threads(g, n), 0, (const double*)g->Bs.p, n,
                  g->key_sorted, g->cell_start, g->gd, (double*)coef_bulk);
    else
        CG_LAUNCH(g, "deposit_implicit", k_deposit_implicit<float>, nblk, seg_threads(g, n), 0, (const float*)g->Bs.p, n,
                  g->key_sorted, g->cell_start, g->gd, (float*)coef_bulk);
    return CG_OK;
}

cg_status launch_deposit_momentum(cg_grids* g, long long n, const void* force_soa, void* S_bulk) {
    CG_CUDA(cudaMemsetAsync(S_bulk, 0, 3 * g->tsize * (size_t)g->gd.nbulk, g->stream));
    if (n == 0) return CG_OK;
    const unsigned nblk = seg_blocks(g, n);
    if (g->fp64)
        CG_LAUNCH(g, "deposit_momentum", k_deposit_momentum<double>, nblk, seg_threads(g, n), 0, (const double*)force_soa, n,
                  g->perm, g->key_sorted, g->cell_start, g->gd, (double*)S_bulk);
    else
        CG_LAUNCH(g, "deposit_momentum", k_deposit_momentum<float>, nblk, seg_threads(g, n), 0, (const float*)force_soa, n,
                  g->perm, g->key_sorted, g->cell_start, g->gd, (float*)S_bulk);
    return CG_OK;
}

cg_status launch_pack(cg_grids* g, const double* eps, const void* u_bulk, bool want_eps_t) {
    const unsigned nblk = blocks_for(g->gd.nbulk, 256);
    if (g->fp64)
        CG_LAUNCH(g, "pack", k_pack<double>, nblk, 256, 0, eps, (const double*)u_bulk, g->gd,
                  (double*)g->bulk4, want_eps_t ? (double*)g->eps_t : nullptr);
    else
        CG_LAUNCH(g, "pack", k_pack<float>, nblk, 256, 0, eps, (const float*)u_bulk, g->gd, (float*)g->bulk4,
                  want_eps_t ? (float*)g->eps_t : nullptr);
    return CG_OK;
}

SumsMap sums_map(const long long* part_off, const long long* part_blocks) {
    SumsMap m;
    for (int k = 0; k < CG_NSUMS; ++k) {
        m.off[k] = -1;
        m.cnt[k] = 0;
    }
    auto col = [&](int dst, int region, int k) {
        if (part_blocks[region] >= 0) {
            m.off[dst] = part_off[region] + (long long)k * part_blocks[region];
            m.cnt[dst] = part_blocks[region];
        }
    };
    col(0, PS_DRAG, 0);
    col(1, PS_VOL, 0);
    for (int a = 0; a < 3; ++a) {
        col(2 + a, PS_DRAG, 1 + a);
        col(5 + a, PS_PROJ, 3 + a);   // S_B V_B: formed by the projection from the S_B it reads
        col(8 + a, PS_PROJ, a);
        col(12 + a, PS_DRAG, 5 + a);
    }
    col(11, PS_DRAG, 4);
    col(15, PS_DRAG, 8);
    return m;
}

cg_status launch_sums(cg_grids* g, double* sums) {
    const SumsMap m = sums_map(g->part_off, g->part_blocks);
    // FP64: two warps for the few partials of a small grid, whose time is the
    // warps' trees (10,000 particles, 512 cells: 7 -> 5 us)
    long long most = 0;
    for (int k = 0; k < CG_NSUMS; ++k) most = std::max(most, m.cnt[k]);
    if (g->fp64)
        CG_LAUNCH(g, "sums", k_sums<double>, CG_NSUMS, most <= 2048 ? 64 : 256, 0, (const double*)g->partials, m, sums);
    else
        CG_LAUNCH(g, "sums", k_sums<float>, CG_NSUMS, 256, 0, (const float*)g->partials, m, sums);
    return CG_OK;
}

}  // namespace cg
