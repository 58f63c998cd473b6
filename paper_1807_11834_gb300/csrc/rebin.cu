// rebin.cu -- incremental rebinning: the per-step particle-to-cell
// connectivity rebuild of Sec. 2.2 of arXiv 1807.11834, started from the
// binning of the previous step.
//
// From one coupling step to the next a particle moves a small fraction of a
// bulk cell, so most particles keep their cell.  The handle's last binning
// of the same particle count (perm_old, key_sorted_old, cell_start_old: the
// stable order, ids ascending within each cell) is therefore nearly the
// new one.  Call a particle whose cell is unchanged a stayer and one whose
// cell changed a mover.  Stayers keep their relative order (their old order
// is sorted by (cell, id) and their cells did not change), so with
//   D(s)   = movers at old slots before s (departures),
//   A(c)   = movers arriving in cells before c,
//   a_c(i) = movers arriving in c with an id below i,
// the new slot of the stayer at old slot s, of cell c and id i, is
//   s - D(s) + A(c) + a_c(i),
// and the new slot of a mover i arriving in c is
//   start_new(c) + (stayers of c with an id below i) + a_c(i),
// where start_new is the exclusive scan of the new counts
// count_old(c) - departures(c) + arrivals(c).  This holds for any new
// positions and any valid binning of the same count: the old order only
// decides how many particles are movers, never the result, which is the
// stable order of the new cells exactly as a full sort gives it.
//
// Old slot s holds particle perm_old[s] when the caller kept its particle
// order, or particle s when the particles are the sorted output of the last
// step (cg_step_sorted; the identity hint).  The movers of a cell are a linked
// list (its few entries are walked, in any order, to count the ids below
// one).  In a cell that receives more than kRebinMaxArrivals movers, a crowded
// one, the walks would grow with the square of the arrivals: the slots kernel
// puts its stayers, in order, and then its movers into a second array, and the
// last kernel sorts the movers and merges the two.  The scan makes the list of
// the crowded cells on the device, so a captured CUDA graph takes the right path
// on every replay.  When no particle changed its cell the device leaves the scans
// out and keeps the bins.
//
// In a coupling step the kernels also form the porosity: the first one, which
// has every particle's position and diameter in nearly sorted order, adds the
// spheres to their cells' accumulators (volume_add_row), and the second one,
// which goes over the cells, turns them into the porosity.
#include <algorithm>

#include "cg_internal.cuh"

namespace cg {

namespace {

struct RebinPtrs {
    int32_t* cnt;       // [n_b + 1] new counts, then (scanned in place) new starts
    int32_t* blk;       // [nblk + 1] departures per block of old slots, then their starts
    int2* arr;          // [n_b + 1] arrivals per cell, then their starts; first mover of the cell's list + 1 (0: none)
    int32_t* dep;       // [n_b] departures per cell
    int32_t* ctr;       // [kRebinCounters]
    int32_t* part;      // block totals of the scans
    size_t zero_bytes;  // arr .. part: zero before the first kernel
};

RebinPtrs rebin_ptrs(cg_grids* g) {
    const long long nb1 = rebin_pad(g->gd.nbulk + 1);
    RebinPtrs r;
    r.cnt = g->rb_small;
    r.blk = r.cnt + nb1;
    r.arr = (int2*)(r.blk + rebin_pad(g->rb_nblk + 1));
    r.dep = (int32_t*)(r.arr + nb1);
    r.ctr = r.dep + nb1;
    r.part = r.ctr + rebin_pad(kRebinCounters);
    r.zero_bytes = sizeof(int32_t) * (3 * nb1 + rebin_pad(kRebinCounters) + 2 * rebin_tiles(g->gd.nbulk + 1) +
                                      rebin_tiles(g->rb_nblk + 1));
    return r;
}

__device__ __forceinline__ void add_status_counts(unsigned long long* st, int outside, int nonfin) {
    if (outside) {
        atomicAdd(&st[ST_OUTSIDE], (unsigned long long)outside);
        atomicOr(&st[ST_FLAGS], (unsigned long long)CG_FLAG_OUTSIDE);
    }
    if (nonfin) {
        atomicAdd(&st[ST_NONFINITE], (unsigned long long)nonfin);
        atomicOr(&st[ST_FLAGS], (unsigned long long)CG_FLAG_NONFINITE);
    }
}

}  // namespace

// Mark the movers, over the old slots (slot base + k * threads + t of
// thread t): the new cell of every old slot, complemented for a mover (rkn),
// and the old id (rid, only when the particles kept the caller's order, whose
// records are gathered through the old permutation: neighbours of a cell, so
// the cells come out nearly sorted in either case); per mover one departure
// from its old cell, one arrival (with its rank) in its new cell, and an entry
// at the head of that cell's list, in the block's own part of the mover array
// (no atomic decides a position).  VOL: the spheres are added to their new
// cells' volumes.  IDENT: old slot s holds particle s.
//
// Bound by HBM in the sorted step (20 bytes read, 4 written per particle) and
// by instruction issue with VOL (about 190 warp instructions per 32 slots);
// 32M particles 209 us, where marking and the porosity as kernels of their
// own took 201 + 148.  In the caller's order it replaces a key kernel over the
// particles as well: 4M packed 31 + 19 + 25 -> 54 us.
template <typename T, bool IDENT, bool VOL>
__global__ void __launch_bounds__(kRebinThreads, sizeof(T) == 4 ? (IDENT ? 5 : 4) : 3)
k_rebin_mark(const T* __restrict__ pos, int n, GridDev g, const int32_t* __restrict__ perm_old,
             const int32_t* __restrict__ ks_old, int32_t* __restrict__ rid, int32_t* __restrict__ rkn,
             int2* __restrict__ arr, int32_t* __restrict__ dep, int4* __restrict__ mov, int32_t* __restrict__ blk_dep, int32_t* __restrict__ ctr,
             unsigned long long* __restrict__ status, unsigned long long* __restrict__ acc) {
    pdl_wait();
    constexpr int W = kRebinThreads / 32;
    __shared__ int s_cnt[W];
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int nblk = (n + kRebinTile - 1) / kRebinTile;   // n < 2^30
    int n_out = 0, n_nf = 0;
    int idk[kRebinItems], cok[kRebinItems];
    auto fetch = [&](int b) {   // ids and old cells of a block of old slots
#pragma unroll
        for (int k = 0; k < kRebinItems; ++k) {
            const int s = b * kRebinTile + k * kRebinThreads + threadIdx.x;
            const bool valid = b < nblk && s < n;
            idk[k] = IDENT ? s : valid ? __ldg(perm_old + s) : 0;
            cok[k] = valid ? __ldg(ks_old + s) : 0;
        }
    };
    fetch(blockIdx.x);
    for (int b = blockIdx.x; b < nblk; b += gridDim.x) {
        const int base = b * kRebinTile;
        int id[kRebinItems], co[kRebinItems], cn[kRebinItems];
        V4<T> pv[kRebinItems];
        // every load of the thread first, so that they are in flight together
#pragma unroll
        for (int k = 0; k < kRebinItems; ++k) {
            const int s = base + k * kRebinThreads + threadIdx.x;
            id[k] = idk[k];
            co[k] = cok[k];
            pv[k] = {T(0), T(0), T(0), T(0)};
            if (s < n) pv[k] = ld4(pos, id[k]);
        }
        if (!IDENT) fetch(b + gridDim.x);
        unsigned mb[kRebinItems];
        int wc = 0;
#pragma unroll
        for (int k = 0; k < kRebinItems; ++k) {
            const int s = base + k * kRebinThreads + threadIdx.x;
            const bool valid = s < n;
            cn[k] = 0;
            if (valid) {
                cn[k] = cell_of(pv[k], g, n_out, n_nf);
            }
            const bool moved = valid && cn[k] != co[k];
            mb[k] = __ballot_sync(full, moved);
            wc += __popc(mb[k]);
            if (valid) {
                rkn[s] = moved ? ~cn[k] : cn[k];
                if (!IDENT) rid[s] = id[k];
            }
            if (VOL) {
                if (IDENT) volume_add_row(valid, cn[k], pv[k].w, g, acc);
                else volume_add_row_wide(valid, cn[k], pv[k].w, g, acc);
            }
        }
        if (lane == 0) s_cnt[warp] = wc;
        __syncthreads();
        // each warp its own prefix over the warps' counts
        int before = 0, total = 0;
#pragma unroll
        for (int w = 0; w < W; ++w) {
            const int c = s_cnt[w];
            if (w < warp) before += c;
            total += c;
        }
        if (threadIdx.x == 0) {
            blk_dep[b] = total;
            if (total) atomicAdd(&ctr[RB_MOVERS], total);
        }
        if (wc) {
            int idx = base + before;
#pragma unroll
            for (int k = 0; k < kRebinItems; ++k) {
                if (mb[k] >> lane & 1u) {
                    const int j = idx + __popc(mb[k] & lanemask_lt());
                    atomicAdd(&dep[co[k]], 1);
                    const int r = atomicAdd(&arr[cn[k]].x, 1);
                    const int next = atomicExch(&arr[cn[k]].y, j + 1);
                    mov[j] = make_int4(id[k], cn[k], next, r);
                }
                idx += __popc(mb[k]);
            }
        }
        if (IDENT) break;   // one block of old slots per CTA
        __syncthreads();
    }
    n_out = __reduce_add_sync(full, n_out);
    n_nf = __reduce_add_sync(full, n_nf);
    if (lane == 0 && (n_out | n_nf)) add_status_counts(status, n_out, n_nf);
}

// Over the cells: the new count of every cell, the tile totals of the scans
// (of the counts, the arrivals, and the departures per block of old slots),
// and the porosity of every cell.  When no particle changed its cell the new
// starts are the old ones, written in their scanned form, and the scans are
// left out.  A cell per thread (cell_items): the chain of one cell's loads and of its few
// FP64 operations bounds small grids (16,384 cells, four per thread 9.3 -> 4.9
// us; 1M cells 25 -> 21).  FP32: five CTAs per SM (48 registers; at 56, four: 27
// -> 31 us in the step of 32M particles).
template <typename T, bool EPS, bool SUMS>
__global__ void __launch_bounds__(256, sizeof(T) == 4 ? 5 : 4)
k_rebin_cells(const int32_t* __restrict__ cs_old, GridDev g, const int32_t* __restrict__ dep,
              const int2* __restrict__ arr, int32_t* __restrict__ cnt, const int32_t* __restrict__ blk, long long nblk,
              const int32_t* __restrict__ ctr, int32_t* __restrict__ part, long long tiles, long long cblk,
              int items, EpsOut<T> eps, T* __restrict__ vpart) {
    pdl_wait();
    const int per = kRebinScan / 256 / items;   // blocks over cells per tile of a scan
    __shared__ int sh[2][8];
    const bool moved = ctr[RB_MOVERS] != 0;
    const long long nbulk = g.nbulk, b = blockIdx.x;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int s0 = 0, s1 = 0;
    if (b < cblk) {
        CSum<T> tot[1];
        for (int j = 0; j < items; ++j) {
            const long long c = (b * items + j) * 256 + threadIdx.x;
            if (c < nbulk) {
                const int start = __ldg(cs_old + c);
                if (moved) {
                    const int a = __ldg(&arr[c].x), v = __ldg(cs_old + c + 1) - start - __ldg(dep + c) + a;
                    cnt[c] = v;
                    s0 += v;
                    s1 += a;
                } else {
                    cnt[c] = start;
                }
                if (EPS) eps_finish<T, SUMS>(c, g, eps, tot[0]);
            } else if (c == nbulk) {
                cnt[c] = moved ? 0 : __ldg(cs_old + c);
            }
        }
        if (SUMS) block_sums<T, 1>(tot, vpart, cblk, b);
    } else if (moved) {
        const long long i = (b - cblk) * 256 + threadIdx.x;
        if (i < nblk) s0 = __ldg(blk + i);
    }
    if (!moved) return;
    s0 = __reduce_add_sync(0xffffffffu, s0);
    s1 = __reduce_add_sync(0xffffffffu, s1);
    if (lane == 0) {
        sh[0][warp] = s0;
        sh[1][warp] = s1;
    }
    __syncthreads();
    if (threadIdx.x < 2) {
        int t = 0;
        for (int w = 0; w < 8; ++w) t += sh[threadIdx.x][w];
        // counts, then (after the arrivals) the blocks' departures
        int32_t* p = threadIdx.x ? part + tiles + b / per : part + (b < cblk ? b / per : 2 * tiles + (b - cblk) / (kRebinScan / 256));
        if (t) atomicAdd(p, t);
    }
}

// Exclusive scan of one tile of 1024 elements, four consecutive ones per
// thread; `before` is the sum of the tiles before it.
__device__ __forceinline__ void scan4(int (&v)[4], int before, int* sh) {
    int total;
    int e = before + block_exclusive_scan(v[0] + v[1] + v[2] + v[3], sh, total);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const int x = v[j];
        v[j] = e;
        e += x;
    }
}
__device__ __forceinline__ void scan_tile(int32_t* __restrict__ a, long long first, long long m, int before, int* sh,
                                          int (&raw)[4]) {
    const long long i = first + 4 * threadIdx.x;
    int v[4] = {0, 0, 0, 0};
    const bool whole = i + 4 <= m;
    if (whole) {
        const int4 q = *reinterpret_cast<const int4*>(a + i);
        v[0] = q.x;
        v[1] = q.y;
        v[2] = q.z;
        v[3] = q.w;
    } else {
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if (i + j < m) v[j] = a[i + j];
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) raw[j] = v[j];
    scan4(v, before, sh);
    if (whole) {
        *reinterpret_cast<int4*>(a + i) = make_int4(v[0], v[1], v[2], v[3]);
    } else {
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if (i + j < m) a[i + j] = v[j];
    }
}
__device__ __forceinline__ void scan_tile_x(int2* __restrict__ a, long long first, long long m, int before, int* sh,
                                            int (&raw)[4]) {
    const long long i = first + 4 * threadIdx.x;
    int2 q[4];
    int v[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        q[j] = i + j < m ? a[i + j] : make_int2(0, 0);
        raw[j] = v[j] = q[j].x;
    }
    scan4(v, before, sh);
#pragma unroll
    for (int j = 0; j < 4; ++j)
        if (i + j < m) a[i + j] = make_int2(v[j], q[j].y);
}

// Starts from the counts and the block totals: the cells' counts and
// arrivals, and the departures per block of old slots.  The cells of many
// arrivals go on the list of the crowded ones, (cell, arrivals, part, parts),
// an entry per part of kCrowdPart ids where the last kernel merges by parts; fewer
// than n / 4 in all, which the list's place, an int per particle, holds.
__global__ void __launch_bounds__(256)
k_rebin_scan(int32_t* __restrict__ cnt, int2* __restrict__ arr, long long ncell, int32_t* __restrict__ blk,
             long long nblk, const int32_t* __restrict__ part, long long tiles, int32_t* ctr, int4* __restrict__ crowd) {
    pdl_wait();
    __shared__ int sh[32];
    if (ctr[RB_MOVERS] == 0) return;
    const bool cells = blockIdx.x < tiles;
    const long long b = cells ? blockIdx.x : blockIdx.x - tiles;
    const int32_t* p0 = cells ? part : part + 2 * tiles;
    int a0 = 0, a1 = 0;
    for (long long i = threadIdx.x; i < b; i += blockDim.x) {
        a0 += __ldg(p0 + i);
        if (cells) a1 += __ldg(part + tiles + i);
    }
    int t0, t1 = 0;
    block_exclusive_scan(a0, sh, t0);
    if (cells) {
        block_exclusive_scan(a1, sh, t1);
        int count[4], in[4];
        scan_tile(cnt, b * kRebinScan, ncell, t0, sh, count);
        scan_tile_x(arr, b * kRebinScan, ncell, t1, sh, in);
        int parts[4], mine = 0;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            parts[j] = in[j] <= kRebinMaxArrivals ? 0 : in[j] <= kSegWarpMax ? (count[j] + kCrowdPart - 1) / kCrowdPart : 1;
            mine += parts[j];
        }
        if (__any_sync(0xffffffffu, mine != 0)) {   // one atomic per warp
            const int lane = threadIdx.x & 31;
            int at = mine;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const int o = __shfl_up_sync(0xffffffffu, at, off);
                if (lane >= off) at += o;
            }
            int base = 0;
            if (lane == 31) base = atomicAdd(ctr + RB_CROWD, at);
            at += __shfl_sync(0xffffffffu, base, 31) - mine;
#pragma unroll
            for (int j = 0; j < 4; ++j)
                for (int p = 0; p < parts[j]; ++p)
                    crowd[at++] = make_int4((int)(b * kRebinScan) + 4 * (int)threadIdx.x + j, in[j], p, parts[j]);
        }
    } else {
        int count[4];
        scan_tile(blk, b * kRebinScan, nblk + 1, t0, sh, count);
    }
}

// Movers of the list starting at h with an id below i.
__device__ __forceinline__ int movers_below(const int4* __restrict__ mov, int h, int i) {
    int a = 0;
    while (h) {
        const int4 m = __ldg(mov + ((unsigned)h - 1u));
        a += m.x < i;
        h = m.z;
    }
    return a;
}

// New slots of the stayers, in the layout of the mark kernel (coalesced
// rows), one block of old slots at a time; the records of the next one are
// loaded while this one's gathers (the arrivals before its cell and its cell's
// list) are under way.  Departures before a slot: the block's start (scan of
// the block totals), the rows and warps before it in the block (a table of
// warp counts), and the lanes before it (ballot).
template <bool IDENT>
__device__ __forceinline__ void rebin_stay_body(const int32_t* __restrict__ rid, const int32_t* __restrict__ rkn,
                                                int n, const int32_t* __restrict__ blk_start,
                                                const int2* __restrict__ arr, const int4* __restrict__ mov,
                                                int32_t* __restrict__ perm, int32_t* __restrict__ key_sorted,
                                                int32_t* __restrict__ inv_perm, int32_t* __restrict__ place,
                                                int nblk, int bid, int nb) {
    constexpr int W = kRebinThreads / 32;
    __shared__ int s_tab[2][kRebinItems * W];
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int kn[kRebinItems], id[kRebinItems];
    auto fetch = [&](int b) {
#pragma unroll
        for (int k = 0; k < kRebinItems; ++k) {
            const int s = b * kRebinTile + k * kRebinThreads + threadIdx.x;
            const bool valid = b < nblk && s < n;
            kn[k] = valid ? __ldg(rkn + s) : -1;
            id[k] = IDENT ? s : (valid ? __ldg(rid + s) : 0);
        }
    };
    fetch(bid);
    int turn = 0;
    for (int b = bid; b < nblk; b += nb, turn ^= 1) {
        const int base = b * kRebinTile;
        int2 ah[kRebinItems];
        int c[kRebinItems], i[kRebinItems];
        unsigned db[kRebinItems];
        int* tab = s_tab[turn];
#pragma unroll
        for (int k = 0; k < kRebinItems; ++k) {
            const int s = base + k * kRebinThreads + threadIdx.x;
            c[k] = kn[k];
            i[k] = id[k];
            ah[k] = make_int2(0, 0);
            if (c[k] >= 0) ah[k] = __ldg(arr + c[k]);
            db[k] = __ballot_sync(full, s < n && c[k] < 0);
            if (lane == 0) tab[k * W + warp] = __popc(db[k]);
        }
        fetch(b + nb);
        __syncthreads();
        static_assert(kRebinItems * W == 32, "one lane per (row, warp) entry");
        // exclusive prefix over (row, warp) in slot order: every warp its own shuffle scan
        const int mine = tab[lane];
        int incl = mine;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const int o = __shfl_up_sync(full, incl, off);
            if (lane >= off) incl += o;
        }
        incl += __ldg(blk_start + b) - mine;
#pragma unroll
        for (int k = 0; k < kRebinItems; ++k) {
            const int s = base + k * kRebinThreads + threadIdx.x;
            const int D = __shfl_sync(full, incl, k * W + warp) + __popc(db[k] & lanemask_lt());
            if (c[k] < 0) continue;
            int ns = s - D + ah[k].x;
            const bool crowded = place && ah[k].y && __ldg(&arr[c[k] + 1].x) - ah[k].x > kRebinMaxArrivals;
            if (ah[k].y && !crowded) ns += movers_below(mov, ah[k].y, i[k]);
            if ((unsigned)ns >= (unsigned)n) continue;   // never for a valid binning
            if (crowded) {
                place[ns] = i[k];
                continue;
            }
            perm[ns] = i[k];
            key_sorted[ns] = c[k];
            if (!IDENT) inv_perm[i[k]] = ns;
        }
    }
}

// Movers, `warps` warps (1, 2, 4 or 8) per block of old slots: the stayers of the new cell with
// an id below the mover's (a binary search over the old segment, whose ids
// ascend, then a count of the stayers before that point) and the movers of
// its list with an id below it.
template <bool IDENT>
__device__ __forceinline__ void rebin_movers_body(const int32_t* __restrict__ rid, const int32_t* __restrict__ rkn,
                                                  long long n, const int32_t* __restrict__ blk_start,
                                                  const int32_t* __restrict__ cs_old,
                                                  const int32_t* __restrict__ cs_new,
                                                  const int2* __restrict__ arr, const int4* __restrict__ mov,
                                                  int32_t* __restrict__ perm, int32_t* __restrict__ key_sorted,
                                                  int32_t* __restrict__ inv_perm, int32_t* __restrict__ place,
                                                  long long nblk, long long bid, long long nb, int warps) {
    const int W = (blockDim.x >> 5) / warps, w = threadIdx.x >> 5;
    for (long long b = bid * W + w / warps; b < nblk; b += nb * W) {
        const int cntb = __ldg(blk_start + b + 1) - __ldg(blk_start + b);
        for (int j = threadIdx.x % (32 * warps); j < cntb; j += 32 * warps) {
            const int4 m = __ldg(mov + b * kRebinTile + j);
            const int i = m.x, c = m.y;
            long long ns;
            const int in = place ? __ldg(&arr[c + 1].x) - __ldg(&arr[c].x) : 0;
            const bool crowded = in > kRebinMaxArrivals;
            if (crowded) {
                // after the cell's stayers, in the order of arrival
                ns = (long long)__ldg(cs_new + c + 1) - in + m.w;
            } else {
                const int o0 = __ldg(cs_old + c), o1 = __ldg(cs_old + c + 1);
                int lo = o0, hi = o1;
                if (IDENT) {
                    lo = i < o0 ? o0 : (i > o1 ? o1 : i);   // the old ids of the segment are its slots
                } else {
                    while (lo < hi) {
                        const int mid = lo + ((hi - lo) >> 1);
                        if (__ldg(rid + mid) < i) lo = mid + 1;
                        else hi = mid;
                    }
                }
                int stay = 0;
                for (int p = o0; p < lo; ++p) stay += __ldg(rkn + p) >= 0;
                ns = (long long)__ldg(cs_new + c) + stay + movers_below(mov, __ldg(&arr[c].y), i);
            }
            if ((unsigned long long)ns >= (unsigned long long)n) continue;   // never for a valid binning
            if (crowded) {
                place[ns] = i;
                continue;
            }
            perm[ns] = i;
            key_sorted[ns] = c;
            if (!IDENT) inv_perm[i] = (int)ns;
        }
    }
}

// Every particle's new slot in one launch: blocks [0, mgrid) place the
// movers (first, so that their searches run beside the stayers), the other
// blocks the stayers.  The ids of crowded cells go to `place` instead, the
// stayers in their order, then the movers in any.  Bound by HBM and by the latency of the
// gather behind each record: 32M particles 105 us, against 207 for one
// block of old slots per CTA with the diameters and the inverse carried along.
template <bool IDENT>
__global__ void __launch_bounds__(kRebinThreads, 6)
k_rebin_slots(const int32_t* __restrict__ rid, const int32_t* __restrict__ rkn, long long n,
              const int32_t* __restrict__ blk_start, const int32_t* __restrict__ cs_old,
              const int32_t* __restrict__ cs_new, const int2* __restrict__ arr, const int4* __restrict__ mov,
              int32_t* __restrict__ perm, int32_t* __restrict__ key_sorted, int32_t* __restrict__ inv_perm,
              int32_t* __restrict__ place, const int32_t* __restrict__ ctr, long long nblk, long long mgrid, int mwarps) {
    pdl_wait();
    int32_t* const where = ctr[RB_CROWD] ? place : nullptr;
    if (ctr[RB_MOVERS] == 0) {
        // slot s keeps its particle and cell; with the identity hint the
        // particles are renumbered to their slots, without it the inverse is
        // made where the steps before left it out
        const bool stale = !IDENT && ctr[RB_INV_STALE];
        if (IDENT || stale)
            for (long long s = (long long)blockIdx.x * blockDim.x + threadIdx.x; s < n; s += (long long)gridDim.x * blockDim.x) {
                if (IDENT) perm[s] = (int)s;
                else inv_perm[__ldg(perm + s)] = (int)s;
            }
        return;
    }
    if ((long long)blockIdx.x < mgrid)
        rebin_movers_body<IDENT>(rid, rkn, n, blk_start, cs_old, cs_new, arr, mov, perm, key_sorted, inv_perm, where,
                                 nblk, blockIdx.x, mgrid, mwarps);
    else
        rebin_stay_body<IDENT>(rid, rkn, (int)n, blk_start, arr, mov, perm, key_sorted, inv_perm, where, (int)nblk,
                               (int)(blockIdx.x - mgrid), (int)(gridDim.x - mgrid));
}

template <typename T>
static cg_status rebin_launches(cg_grids* g, long long n, const T* pos, bool ident, StepEps* eps) {
    const long long nbulk = g->gd.nbulk;
    const RebinPtrs R = rebin_ptrs(g);
    const long long nblk = (n + kRebinTile - 1) / kRebinTile;
    const EpsOut<T> eo = eps_out<T>(g, eps);
    // the caller's order: resident CTAs that walk the blocks of old slots, the
    // next block's ids and cells loaded ahead of the gather they lead to
    const long long walk = (long long)g->num_sms * (sizeof(T) == 4 ? 4 : 3);
#define CG_REBIN_MARK(ID, VOL)                                                                                     \
    CG_LAUNCH(g, "rebin_mark", (k_rebin_mark<T, ID, VOL>), (unsigned)(ID ? nblk : std::min(nblk, walk)), kRebinThreads, 0, pos, (int)n, g->gd,    \
              (const int32_t*)g->perm, (const int32_t*)g->key_sorted, g->rb_rid, g->rb_rkn, R.arr, R.dep,           \
              g->rb_mov, R.blk, R.ctr, g->status, eo.acc)
    if (ident) {
        if (eps) CG_REBIN_MARK(true, true);
        else CG_REBIN_MARK(true, false);
    } else {
        if (eps) CG_REBIN_MARK(false, true);
        else CG_REBIN_MARK(false, false);
    }
#undef CG_REBIN_MARK
    const long long tiles = rebin_tiles(nbulk + 1), btiles = rebin_tiles(nblk + 1);
    const int items = cell_items(nbulk, sizeof(T) == 8);
    const long long cblk = cell_blocks(nbulk, sizeof(T) == 8);
    T* vpart = (T*)part_ptr(g, PS_VOL);
#define CG_REBIN_CELLS(EPS, SUMS)                                                                                  \
    CG_LAUNCH(g, "rebin_cells", (k_rebin_cells<T, EPS, SUMS>), (unsigned)(cblk + (nblk + 255) / 256), 256, 0,       \
              (const int32_t*)g->cell_start, g->gd, (const int32_t*)R.dep, (const int2*)R.arr, R.cnt,               \
              (const int32_t*)R.blk, nblk, (const int32_t*)R.ctr, R.part, tiles, cblk, items, eo, vpart)
    if (eps && eps->sums) CG_REBIN_CELLS(true, true);
    else if (eps) CG_REBIN_CELLS(true, false);
    else CG_REBIN_CELLS(false, false);
#undef CG_REBIN_CELLS
    if (eps) {
        g->part_blocks[PS_VOL] = eps->sums ? cblk : -1;
        eps->formed = true;
        if (eps->ready) CG_CUDA(cudaEventRecord(eps->ready, g->stream));
    }
    CG_LAUNCH(g, "rebin_scan", k_rebin_scan, (unsigned)(tiles + btiles), 256, 0, R.cnt, R.arr, nbulk + 1, R.blk, nblk,
              (const int32_t*)R.part, tiles, R.ctr, (int4*)g->key);
    // few blocks of old slots: several warps for the movers of each, since a bed of
    // which every particle has moved is a chain of 32 rounds for one (500,000
    // particles in another order: the step 180 -> 140 us)
    const long long mgrid = std::max((nblk + 7) / 8, std::min<long long>(nblk, (long long)g->num_sms * 3));
    const int mwarps = nblk <= mgrid ? 8 : nblk <= 2 * mgrid ? 4 : nblk <= 4 * mgrid ? 2 : 1;
    // resident blocks that walk the old slots (the sorted step), or, where the
    // scattered stores of a caller's random order dominate, a block per 1024
    // slots (4M particles: 42 us against 50)
    const long long sgrid = ident ? std::min<long long>(nblk, (long long)g->num_sms * 6) : nblk;
#define CG_REBIN_SLOTS(ID)                                                                                        \
    CG_LAUNCH(g, "rebin_slots", (k_rebin_slots<ID>), (unsigned)(mgrid + sgrid), kRebinThreads, 0,                   \
              (const int32_t*)g->rb_rid, (const int32_t*)g->rb_rkn, n, (const int32_t*)R.blk,                      \
              (const int32_t*)g->cell_start, (const int32_t*)R.cnt, (const int2*)R.arr, (const int4*)g->rb_mov,      \
              g->perm, g->key_sorted, g->inv_perm, g->val1, (const int32_t*)R.ctr, nblk, mgrid, mwarps)
    if (ident) CG_REBIN_SLOTS(true);
    else CG_REBIN_SLOTS(false);
#undef CG_REBIN_SLOTS
    const long long nb1 = rebin_pad(nbulk + 1);
    CG_TRY(launch_rebin_finish(g, R.cnt, R.ctr, (const int4*)g->key, g->cell_start, ident ? nullptr : g->inv_perm,
                               {(int4*)R.arr, 3 * nb1 / 4, R.part, 2 * tiles + btiles}));
    return CG_OK;
}

// The last kernel clears what the next rebinning counts in (a clear of its own
// at the head of the chain costs 2 to 3 us); a launch that fails before it leaves
// that to this, with the volumes that no pass over the cells has taken.
template <typename T>
static cg_status rebin_impl(cg_grids* g, long long n, const T* pos, bool ident, StepEps* eps) {
    if ((n + kRebinTile - 1) / kRebinTile > g->rb_nblk) return CG_ERR_OUT_OF_RANGE;
    const cg_status st = rebin_launches<T>(g, n, pos, ident, eps);
    if (st == CG_OK) return CG_OK;
    const RebinPtrs R = rebin_ptrs(g);
    cudaMemsetAsync(R.arr, 0, R.zero_bytes, g->stream);
    cudaMemsetAsync(R.ctr + RB_INV_STALE, 0xff, sizeof(int32_t), g->stream);
    if (eps) clear_volumes(g, g->stream);
    cudaGetLastError();
    return st;
}

// Caller-order cells of the binning's slots.
__global__ void __launch_bounds__(256)
k_scatter_cells(const int32_t* __restrict__ perm, const int32_t* __restrict__ key_sorted, long long n,
                int32_t* __restrict__ out) {
    pdl_wait();
    for (long long s = (long long)blockIdx.x * blockDim.x + threadIdx.x; s < n; s += (long long)gridDim.x * blockDim.x)
        out[__ldg(perm + s)] = __ldg(key_sorted + s);
}

// The inverse of perm, where it is out of date; the block that finishes last
// marks it valid, when every block has read the mark.
__global__ void __launch_bounds__(256)
k_inverse(const int32_t* __restrict__ perm, long long n, int32_t* __restrict__ inv_perm, int32_t* ctr) {
    pdl_wait();
    if (ctr[RB_INV_STALE] == 0) return;
    for (long long s = (long long)blockIdx.x * blockDim.x + threadIdx.x; s < n; s += (long long)gridDim.x * blockDim.x)
        inv_perm[__ldg(perm + s)] = (int)s;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        if (atomicAdd(ctr + RB_INV_DONE, 1) == (int)gridDim.x - 1) ctr[RB_INV_STALE] = ctr[RB_INV_DONE] = 0;
    }
}

cg_status copy_cells(cg_grids* g, long long n, int32_t* cell_out) {
    if (n <= 0) return CG_OK;
    if (g->key_valid) {
        CG_CUDA(cudaMemcpyAsync(cell_out, g->key, sizeof(int32_t) * n, cudaMemcpyDeviceToDevice, g->stream));
        return CG_OK;
    }
    const unsigned grid = (unsigned)std::min<long long>((n + 255) / 256, (long long)g->num_sms * 8);
    CG_LAUNCH(g, "bin_cells", k_scatter_cells, grid, 256, 0, (const int32_t*)g->perm, (const int32_t*)g->key_sorted, n,
              cell_out);
    return CG_OK;
}

cg_status ensure_inverse(cg_grids* g, long long n) {
    if (!g->ident_seen || n <= 0) return CG_OK;
    const unsigned grid = (unsigned)std::min<long long>((n + 255) / 256, (long long)g->num_sms * 8);
    CG_LAUNCH(g, "bin_inverse", k_inverse, grid, 256, 0, (const int32_t*)g->perm, n, g->inv_perm, rebin_ptrs(g).ctr);
    return CG_OK;
}

cg_status launch_rebin(cg_grids* g, long long n, const void* pos_d, bool ident, StepEps* eps) {
    return g->fp64 ? rebin_impl<double>(g, n, (const double*)pos_d, ident, eps)
                   : rebin_impl<float>(g, n, (const float*)pos_d, ident, eps);
}

}  // namespace cg
