// drag.cu -- (a3) drag on every particle, Eq. (DragLaw) of arXiv 1807.11834:
// F = beta (u_f - u_p), with the porosity and the fluid velocity taken at the
// particle from the bulk grid (the cell value or a local interpolant,
// Sec. 1), and beta from a correlation of slip, densities, diameter,
// viscosity and porosity.  Optionally (a5) the semi-implicit Euler advance
// of Eq. (DEM_EQUATIONS) without contacts.
//
// One thread per particle in the caller's order: the particle record is
// read once (two 16-byte loads) and the force written once (three
// coalesced stores).  The bulk fields are gathered from a packed array of
// (eps, u_x, u_y, u_z) per cell, eight 16-byte loads that stay in L2.  For
// the fused reaction deposit the force is also written, as a 16-byte
// record, to its slot in bin order, so the following segmented sum reads
// it contiguously.
//
// FP32 path: the lattice coordinate (x - x0)/H - 1/2 is formed in
// float-float (FMA TwoProduct and one TwoSum), so the interpolation weights
// carry only the final float rounding even at |xi| ~ 100; the correlations
// run in float with explicitly rounded operations, their powers, logarithm,
// roots and reciprocals on the special-function unit (drag_law.cuh).
// The sorted step's kernel (k_drag_sorted) takes the particles in cell order,
// stages the bulk records around a run of cells in shared memory and sums the
// reaction itself.
#include <algorithm>

#include "cg_internal.cuh"
#include "drag_law.cuh"
#include "batch.cuh"

namespace cg {

template <typename T>
__device__ __forceinline__ V4<T> ld4_plain(const T* p, long long i) {
    if (sizeof(T) == 4) {
        float4 v = reinterpret_cast<const float4*>(p)[i];
        return {(T)v.x, (T)v.y, (T)v.z, (T)v.w};
    } else {
        const double2* q = reinterpret_cast<const double2*>(p) + 2 * i;
        double2 a = q[0], b = q[1];
        return {(T)a.x, (T)a.y, (T)b.x, (T)b.y};
    }
}

// ----------------------------------------------------------------------
// One particle: the porosity and fluid velocity gathered at x, the drag
// force, and with EULER the advanced state (else x and u unchanged).
// ----------------------------------------------------------------------
template <typename T>
struct DragOne {
    T f[3], beta, smag, vp, m, x[3], u[3];
    int cl;
};

// Whether x may lie outside [lo, hi]; exact in FP32.  FP64 compares the upper words
// as integers (their order for equal signs, reversed for negative ones), off the FP64
// pipe; x within 2^-20 of a bound counts as outside, which the caller then
// decides exactly.
__device__ __forceinline__ bool outside_of(float x, float lo, float hi) { return x < lo || x > hi; }
__device__ __forceinline__ int ordered_hi(double x) {
    const int h = __double2hiint(x);
    return h ^ ((h >> 31) & 0x7fffffff);
}
__device__ __forceinline__ bool outside_of(double x, double lo, double hi) {
    const int h = ordered_hi(x);
    return h <= ordered_hi(lo) || h >= ordered_hi(hi);
}

template <typename T, bool EULER>
__device__ __forceinline__ DragOne<T> drag_from(const V4<T>& x, const V4<T>& v, const V4<T>& b, const GridDev& g,
                                                const Phys<T>& P, T dt) {
    using X = M<T>;
    DragOne<T> r;
    T eps = b.x;
    T phi = X::sub(T(1), eps);
    r.cl = 0;
    if (eps < P.eps_min) {
        eps = P.eps_min;
        phi = X::sub(T(1), P.eps_min);
        r.cl = 1;
    }
    const T sx = X::sub(b.y, v.x), sy = X::sub(b.z, v.y), sz = X::sub(b.w, v.z);
    r.smag = X::sqrt_(X::fma_(sx, sx, X::fma_(sy, sy, X::mul(sz, sz))));
    const T d = x.w;
    r.beta = drag_beta(g.law, eps, phi, d, r.smag, P);
    r.f[0] = X::mul(r.beta, sx);
    r.f[1] = X::mul(r.beta, sy);
    r.f[2] = X::mul(r.beta, sz);
    r.vp = X::mul(X::mul(X::mul(M<T>::pi6(), d), d), d);
    r.m = X::mul(P.rho_p, r.vp);
    r.x[0] = x.x;
    r.x[1] = x.y;
    r.x[2] = x.z;
    r.u[0] = v.x;
    r.u[1] = v.y;
    r.u[2] = v.z;
    if (EULER) {
        const T inv_m = X::rcp_(r.m);   // one reciprocal for the three components
        bool out = false;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            r.u[a] = X::fma_(dt, X::fma_(r.f[a], inv_m, P.g[a]), r.u[a]);
            r.x[a] = X::fma_(dt, r.u[a], r.x[a]);
            // the FP32 path reads the bounds' float copies (no conversion in the loop)
            const T lo = sizeof(T) == 4 ? (T)g.x0f[a] : (T)g.x0[a];
            const T hi = sizeof(T) == 4 ? (T)g.xhif[a] : (T)g.xhi[a];
            out = out || outside_of(r.x[a], lo, hi);
        }
        if (out)   // specular walls: rare, so one branch for the three axes
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                const T lo = sizeof(T) == 4 ? (T)g.x0f[a] : (T)g.x0[a];
                const T hi = sizeof(T) == 4 ? (T)g.xhif[a] : (T)g.xhi[a];
                if (r.x[a] < lo) { r.x[a] = X::sub(X::mul(T(2), lo), r.x[a]); r.u[a] = -r.u[a]; }
                else if (r.x[a] > hi) { r.x[a] = X::sub(X::mul(T(2), hi), r.x[a]); r.u[a] = -r.u[a]; }
            }
    }
    return r;
}

template <typename T, bool EULER>
__device__ __forceinline__ DragOne<T> drag_one(const V4<T>& x, const V4<T>& v, const GridDev& g, const Phys<T>& P,
                                               const T* __restrict__ bulk4, T dt) {
    return drag_from<T, EULER>(x, v, gather(bulk4, x.x, x.y, x.z, g), g, P, dt);
}

// Per-lane diagnostics: V_p, F (3), |F|, m u (3) after the advance.
template <typename T>
__device__ __forceinline__ void drag_lane_sums(T (&ls)[kDragLaneSums], const DragOne<T>& r) {
    using X = M<T>;
    ls[0] = X::add(ls[0], r.vp);
    ls[1] = X::add(ls[1], r.f[0]);
    ls[2] = X::add(ls[2], r.f[1]);
    ls[3] = X::add(ls[3], r.f[2]);
    ls[4] = X::fma_(r.beta, r.smag, ls[4]);
    ls[5] = X::fma_(r.m, r.u[0], ls[5]);
    ls[6] = X::fma_(r.m, r.u[1], ls[6]);
    ls[7] = X::fma_(r.m, r.u[2], ls[7]);
}

// The end of a drag kernel: the block's clamped particles to the status, its
// diagnostics to the partials.
template <typename T>
__device__ __forceinline__ void drag_totals(int clamped, const T (&lane_sums)[kDragLaneSums], T* __restrict__ part,
                                            long long pstride, int do_sums, unsigned long long* __restrict__ status,
                                            long long bid) {
    clamped = __reduce_add_sync(0xffffffffu, clamped);
    if ((threadIdx.x & 31) == 0 && clamped) {
        atomicAdd(&status[ST_CLAMPED], (unsigned long long)clamped);
        atomicOr(&status[ST_FLAGS], (unsigned long long)CG_FLAG_EPS_CLAMPED);
    }
    if (do_sums) {
        CSum<T> acc[kDragLaneSums];
#pragma unroll
        for (int k = 0; k < kDragLaneSums; ++k) acc[k].s = lane_sums[k];
        block_sums<T, kDragLaneSums>(acc, part, pstride, bid);
        block_count<T>(clamped, part + 2 * (kDragLaneSums * pstride + bid));
    }
}

// ----------------------------------------------------------------------
// Drag kernel.  Partial sums (per block): V_p, F (3), |F|, m u (3), clamped.
// With EULER the particle is advanced in place after its force is known:
// u += dt (F/m + g), x += dt u, specular reflection at the domain faces.
// ----------------------------------------------------------------------
// Bs (nullable): the semi-implicit record (beta, beta u_p) of each particle,
// written to its sorted slot beside the force record.
template <typename T, bool EULER, bool PREFETCH = true>
__device__ __forceinline__ void drag_body(T* pos, T* vel, long long n, const GridDev& g, const Phys<T>& P,
                                          const T* __restrict__ bulk4, T* __restrict__ F, T* __restrict__ Fs,
                                          const int32_t* __restrict__ inv_perm, T dt, T* __restrict__ part,
                                          long long pstride, int do_sums, unsigned long long* __restrict__ status,
                                          Blk b, T* __restrict__ Bs = nullptr) {
    T lane_sums[kDragLaneSums];
#pragma unroll
    for (int k = 0; k < kDragLaneSums; ++k) lane_sums[k] = T(0);
    int clamped_total = 0;
    const long long stride = b.n * blockDim.x;
    // PREFETCH: the next particle's record is loaded while this one's
    // stencil is gathered and its force computed (its DRAM latency overlaps
    // them); the batched kernel, short of registers, loads it in turn
    V4<T> xn, vn;
    int slot_n = 0;
    long long p = b.id * blockDim.x + threadIdx.x;
    if (p < n) {
        xn = EULER ? ld4_plain(pos, p) : ld4((const T*)pos, p);
        vn = EULER ? ld4_plain(vel, p) : ld4((const T*)vel, p);
        if (Fs) slot_n = __ldg(inv_perm + p);
    }
    for (; p < n; p += stride) {
        if (!PREFETCH && p != b.id * blockDim.x + threadIdx.x) {
            xn = EULER ? ld4_plain(pos, p) : ld4((const T*)pos, p);
            vn = EULER ? ld4_plain(vel, p) : ld4((const T*)vel, p);
            if (Fs) slot_n = __ldg(inv_perm + p);
        }
        const V4<T> x = xn, v = vn;
        const int slot = slot_n;
        if (PREFETCH && p + stride < n) {
            xn = EULER ? ld4_plain(pos, p + stride) : ld4((const T*)pos, p + stride);
            vn = EULER ? ld4_plain(vel, p + stride) : ld4((const T*)vel, p + stride);
            if (Fs) slot_n = __ldg(inv_perm + p + stride);
        }
        const DragOne<T> r = drag_one<T, EULER>(x, v, g, P, bulk4, dt);
        clamped_total += r.cl;
        F[p] = r.f[0];
        F[n + p] = r.f[1];
        F[2 * n + p] = r.f[2];
        if (Fs) st4(Fs, slot, r.f[0], r.f[1], r.f[2], T(0));
        if (Bs) st4(Bs, slot, r.beta, r.beta * v.x, r.beta * v.y, r.beta * v.z);
        if (EULER) {
            st4(pos, p, r.x[0], r.x[1], r.x[2], x.w);
            st4(vel, p, r.u[0], r.u[1], r.u[2], v.w);
        }
        if (do_sums) drag_lane_sums(lane_sums, r);
    }
    drag_totals<T>(clamped_total, lane_sums, part, pstride, do_sums, status, b.id);
}

template <typename T, bool EULER>
__global__ void __launch_bounds__(256, sizeof(T) == 4 ? 4 : 2)
k_drag(T* pos, T* vel, long long n, GridDev g, Phys<T> P, const T* __restrict__ bulk4,
       T* __restrict__ F, T* __restrict__ Fs, const int32_t* __restrict__ inv_perm, T dt,
       T* __restrict__ part, long long pstride, int do_sums, unsigned long long* __restrict__ status,
       T* __restrict__ Bs) {
    pdl_wait();
    drag_body<T, EULER>(pos, vel, n, g, P, bulk4, F, Fs, inv_perm, dt, part, pstride, do_sums, status,
                        launch_blk(), Bs);
}

// Window of bulk records in a warp's shared memory (FP32): the stencils of
// the particles of up to kWinCells consecutive cells of one x row reach from
// the cell before to the cell after, in three rows of three layers.  The
// strides are 2 and 4 modulo 8 records (of 16 bytes; eight cover the 32
// banks), so that the eight stencils of one cell's octants lie in eight
// different bank groups.
constexpr int kWinX = 16, kWinCells = kWinX - 2, kWinRow = 18, kWinLayer = 60;
constexpr int kWinRecs = 2 * kWinLayer + 2 * kWinRow + kWinX;
struct Window {
    int begin = 0, end = -1;   // cells covered (linear; none at first)
    int I, J, K;               // position of the first one
};
// Make the window cover the cells [first, last]; false when they are not in
// one row or too many.  Called by the whole warp with uniform arguments.
__device__ __forceinline__ bool window_cover(Window& w, int first, int last, const V4<float>* __restrict__ rec,
                                             const GridDev& g, V4<float>* __restrict__ win) {
    if (first >= w.begin && last <= w.end) return true;
    const int nbx = g.nb[0], nby = g.nb[1], nbz = g.nb[2];
    const int row = (int)((unsigned)first / (unsigned)nbx);
    const int end = min(first + kWinCells, (row + 1) * nbx) - 1;
    if (last > end) return false;
    w.begin = first;
    w.end = end;
    w.K = (int)((unsigned)row / (unsigned)nby);
    w.J = row - w.K * nby;
    w.I = first - row * nbx;
    const int lane = threadIdx.x & 31, x = lane & (kWinX - 1);
    const int cx = min(max(w.I - 1 + x, 0), nbx - 1);
    __syncwarp();   // every lane has read the window before
#pragma unroll
    for (int p = 0; p < 5; ++p) {
        const int q = 2 * p + (lane >> 4);   // row of the window, three per layer
        const int z = (q * 11) >> 5, y = q - 3 * z;
        if (q < 9) {
            const int cy = min(max(w.J - 1 + y, 0), nby - 1), cz = min(max(w.K - 1 + z, 0), nbz - 1);
            const V4<float> v = ldv4(rec + cx + nbx * (cy + nby * cz));
            *reinterpret_cast<float4*>(win + x + kWinRow * y + kWinLayer * z) = make_float4(v.x, v.y, v.z, v.w);
        }
    }
    __syncwarp();
    return true;
}
__device__ __forceinline__ Pair2 ld_win(const V4<float>* q) {
    const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(q);
    return {v.x, v.y};
}
// (eps, u) at a point of a covered cell.
__device__ __forceinline__ V4<float> window_gather(const Window& w, const V4<float>* __restrict__ win,
                                                   const float* __restrict__ bulk4, const V4<float>& x,
                                                   const GridDev& g) {
    int i, j, k;
    float tx, ty, tz;
    axis_weight(x.x, g, 0, i, tx);
    axis_weight(x.y, g, 1, j, ty);
    axis_weight(x.z, g, 2, k, tz);
    const int lx = i - w.I + 1, ly = j - w.J + 1, lz = k - w.K + 1;
    // a stencil begins at its cell or at the one before it
    if ((unsigned)lx <= (unsigned)(kWinX - 2) && (unsigned)ly <= 1u && (unsigned)lz <= 1u)
    {
        // interp8 in pairs
        const V4<float>* c = win + lx + kWinRow * ly + kWinLayer * lz;
        const unsigned long long t = f2_pack(tx, tx), u = f2_pack(ty, ty), w2 = f2_pack(tz, tz);
        const Pair2 a00 = lerp_pairs(ld_win(c), ld_win(c + 1), t);
        const Pair2 a10 = lerp_pairs(ld_win(c + kWinRow), ld_win(c + kWinRow + 1), t);
        const Pair2 a01 = lerp_pairs(ld_win(c + kWinLayer), ld_win(c + kWinLayer + 1), t);
        const Pair2 a11 = lerp_pairs(ld_win(c + kWinLayer + kWinRow), ld_win(c + kWinLayer + kWinRow + 1), t);
        const Pair2 r = lerp_pairs(lerp_pairs(a00, a10, u), lerp_pairs(a01, a11, u), w2);
        V4<float> o;
        f2_unpack(r.a, o.x, o.y);
        f2_unpack(r.b, o.z, o.w);
        return o;
    }
    return gather(bulk4, x.x, x.y, x.z, g);
}

// The drag of the sorted step, in the order of the binning: lane l of a warp
// takes slot r + l, the particle perm[r + l] (nearly r + l, since the particles
// come in the last step's cell order), and its record, advanced when EULER,
// leaves at that slot.  The force goes to the particle's own index, and its
// reaction is summed right here, in the rounds of the segmented sum (seg_round)
// over the chunks that k_deposit_sorted_force would take: the same additions
// in the same order, without the 16-byte force record per particle written and
// read back.  A block's warps take neighbouring chunks (they share the bulk
// records in L1); a warp walks the rounds of its chunks as one sequence, with
// the ids loaded two rounds ahead and the records one.
//
// 84 bytes per particle instead of 96 and another 20 for the reaction; 32M
// particles 710 us, against 607 + 172 + 50 for the drag in the particles'
// order, the reaction as a kernel of its own and the inverse permutation it
// needs.  Bound by instruction issue (about 530 a round, 60 to 70% of the
// slots) and the load / store unit (40 to 48%; 69% with the eight gathers of a
// stencil from L1 in place of the window, 725 us).  Three CTAs per SM: two 795,
// four (spilling) 789.  Neighbouring chunks per block rather than a run of
// chunks per warp: 714 against 855 (L1 misses).
template <typename T, bool EULER, bool WIN>
__global__ void __launch_bounds__(256, sizeof(T) == 4 ? 3 : 2)
k_drag_sorted(const T* __restrict__ pos, const T* __restrict__ vel, long long n, GridDev g, Phys<T> P,
              const T* __restrict__ bulk4, T* __restrict__ F, const int32_t* __restrict__ perm,
              const int32_t* __restrict__ key_sorted, const int32_t* __restrict__ cs, T* __restrict__ S, T dt,
              T* __restrict__ part, long long pstride, int do_sums, unsigned long long* __restrict__ status,
              T* __restrict__ Bs, T* __restrict__ pos_out, T* __restrict__ vel_out, int32_t* __restrict__ perm_out,
              T* __restrict__ Fs) {
    extern __shared__ __align__(16) V4<float> s_win[];   // WIN: kWinRecs per warp
    pdl_wait();
    const unsigned full = 0xffffffffu;
    const unsigned lane = threadIdx.x & 31;
    V4<float>* win = s_win + (threadIdx.x >> 5) * kWinRecs;
    Window wd;
    T lane_sums[kDragLaneSums];
#pragma unroll
    for (int k = 0; k < kDragLaneSums; ++k) lane_sums[k] = T(0);
    int clamped_total = 0;
    // slots as 32-bit unsigned (n < 2^31); tt = 0 after the last round
    const unsigned un = (unsigned)n;
    const unsigned long long step = (unsigned long long)gridDim.x * (blockDim.x >> 5) * seg_chunk(n);
    unsigned long long base = ((unsigned long long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)) * seg_chunk(n);
    auto chunk = [&](unsigned& rr, unsigned& tt) {   // the first round from the chunk at `base` on
        for (; base < un; base += step) {
            long long s, e;
            seg_chunk_range((long long)base, n, key_sorted, cs, s, e);
            if (s < e) {
                rr = (unsigned)s;
                tt = (unsigned)e;
                base += step;
                return;
            }
        }
        tt = 0u;
    };
    unsigned r = 0, t = 0;
    chunk(r, t);
    if (t) {
        int id = 0, key = -1, id1 = 0, key1 = -1;
        V4<T> x = {T(0), T(0), T(0), T(0)}, v = x;
        auto ids = [&](unsigned rr, unsigned tt, int& i, int& k) {
            k = -1;
            if (rr + lane < tt) {
                i = __ldg(perm + rr + lane);
                k = __ldg(key_sorted + rr + lane);
            }
        };
        auto advance = [&](unsigned& rr, unsigned& tt) {
            rr += 32;
            if (rr >= tt) chunk(rr, tt);
        };
        ids(r, t, id, key);
        if (key >= 0) {
            x = ld4(pos, id);
            v = ld4(vel, id);
        }
        unsigned r1 = r, t1 = t;
        advance(r1, t1);
        ids(r1, t1, id1, key1);
        SegCarry<T, 3> carry;
        for (;;) {
            V4<T> x1 = {T(0), T(0), T(0), T(0)}, v1 = x1;
            if (key1 >= 0) {
                x1 = ld4(pos, id1);
                v1 = ld4(vel, id1);
            }
            unsigned r2 = r1, t2 = t1;
            int id2 = 0, key2 = -1;
            if (t1) {
                advance(r2, t2);
                ids(r2, t2, id2, key2);
            }
            bool in_win = false;
            if constexpr (WIN) {
                const unsigned left = t - r;   // slots of this round: min(left, 32), at least one
                const int c0 = __shfl_sync(full, key, 0), c1 = __shfl_sync(full, key, left < 32u ? left - 1u : 31u);
                in_win = window_cover(wd, c0, c1, reinterpret_cast<const V4<float>*>(bulk4), g, win);
            }
            T f[3] = {T(0), T(0), T(0)};
            if (key >= 0) {
                V4<T> b;
                if constexpr (WIN) b = in_win ? window_gather(wd, win, bulk4, x, g) : gather(bulk4, x.x, x.y, x.z, g);
                else b = gather(bulk4, x.x, x.y, x.z, g);
                const DragOne<T> d = drag_from<T, EULER>(x, v, b, g, P, dt);
                clamped_total += d.cl;
                const unsigned slot = r + lane;
#pragma unroll
                for (int k = 0; k < 3; ++k) f[k] = d.f[k];
                if (Fs) st4(Fs, slot, f[0], f[1], f[2], T(0));
                else
#pragma unroll
                    for (int k = 0; k < 3; ++k) F[k * n + id] = f[k];
                if (Bs) st4(Bs, slot, d.beta, d.beta * v.x, d.beta * v.y, d.beta * v.z);
                st4(pos_out, slot, d.x[0], d.x[1], d.x[2], x.w);
                st4(vel_out, slot, d.u[0], d.u[1], d.u[2], v.w);
                if (perm_out) perm_out[slot] = id;
                if (do_sums) drag_lane_sums(lane_sums, d);
            }
            const int next31 = __shfl_sync(full, key1, 0);
            seg_round<T, 3>(f, key, r + 32 >= t ? -1 : next31, carry,
                            [&](int c, int k, T sum) { reaction_emit<T>(g, S, c, k, sum); });
            if (!t1) break;
            r = r1;
            t = t1;
            id = id1;
            key = key1;
            x = x1;
            v = v1;
            r1 = r2;
            t1 = t2;
            id1 = id2;
            key1 = key2;
        }
    }
    drag_totals<T>(clamped_total, lane_sums, part, pstride, do_sums, status, blockIdx.x);
}

// The forces from the binned order into the particles' own.
template <typename T>
__global__ void __launch_bounds__(256)
k_unsort_force(const T* __restrict__ Fs, const int32_t* __restrict__ inv_perm, long long n, T* __restrict__ F) {
    pdl_wait();
    for (long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x; p < n; p += (long long)gridDim.x * blockDim.x) {
        const V4<T> f = ld4(Fs, __ldg(inv_perm + p));
        F[p] = f.x;
        F[n + p] = f.y;
        F[2 * n + p] = f.z;
    }
}

template <typename T>
static cg_status launch_drag_sorted(cg_grids* g, long long n, const T* pos, const T* vel, T* force, T* S, bool sums,
                                    double dt, T* Bs, T* pos_out, T* vel_out, int32_t* perm_out) {
    // Particles that come in any order (the binning was not the identity-hint
    // one): their forces leave in the order of the binning and are gathered from
    // there, instead of three scattered 4-byte stores each (32M in random order,
    // the first step: 4390 -> 2480 us)
    T* Fs = g->bin_ident ? nullptr : (T*)g->Fs;
    // at most the resident CTAs
    const long long chunks = (n + seg_chunk(n) - 1) / seg_chunk(n);
    const int bs = (int)seg_threads(g, n), warps = bs / 32;
    const long long nblk = std::min((chunks + warps - 1) / warps, (long long)g->num_sms * (sizeof(T) == 4 ? 24 : 16) / warps);
    T* part = (T*)part_ptr(g, PS_DRAG);
    g->part_blocks[PS_DRAG] = sums ? nblk : -1;
#define CG_DRAGS(E, W)                                                                                          \
    CG_LAUNCH(g, "drag", (k_drag_sorted<T, E, W>), (unsigned)nblk, bs, W ? warps * kWinRecs * sizeof(V4<float>) : 0, pos,  \
              vel, n, g->gd, phys_of<T>(g->gd),                                                                 \
              (const T*)g->bulk4, force, (const int32_t*)g->perm, (const int32_t*)g->key_sorted,                  \
              (const int32_t*)g->cell_start, S, (T)dt, part, nblk, (int)sums, g->status, Bs, pos_out, vel_out,      \
              perm_out, Fs)
    const bool win = sizeof(T) == 4 && g->gd.interp != CG_INTERP_CELL;
    if constexpr (sizeof(T) == 4) {
        if (win && dt > 0.0) CG_DRAGS(true, true);
        else if (win) CG_DRAGS(false, true);
    }
    if (!win && dt > 0.0) CG_DRAGS(true, false);
    else if (!win) CG_DRAGS(false, false);
#undef CG_DRAGS
    if (Fs)
        CG_LAUNCH(g, "unsort_force", k_unsort_force<T>, (unsigned)std::min((n + 255) / 256, (long long)g->num_sms * 16), 256, 0,
                  (const T*)Fs, (const int32_t*)g->inv_perm, n, force);
    return CG_OK;
}

// Batched drag with the fused sorted-order force record (FP32 instances).
template <bool EULER>
__global__ void __launch_bounds__(256) kb_drag(BLaunch L, float dt) {
    batch_loop(L, [&](const BInst& I, Blk b) {
        drag_body<float, EULER, false>(I.pos, I.vel, I.n, I.gd, I.P, I.bulk4, I.force, I.Fs, I.inv_perm, dt,
                                I.part + 2 * I.part_off[PS_DRAG], I.part_blocks[PS_DRAG], I.sums != nullptr, I.status, b);
    });
}

cg_status launch_batch_drag(const BLaunch& L, unsigned grid, float dt, cudaStream_t s) {
    if (L.total == 0 || grid == 0) return CG_OK;
    if (dt > 0.f) kb_drag<true><<<grid, 256, 0, s>>>(L, dt);
    else kb_drag<false><<<grid, 256, 0, s>>>(L, 0.f);
    CG_CUDA(cudaGetLastError());
    return CG_OK;
}

int batch_drag_occupancy() {
    int occ = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kb_drag<true>, 256, 0) != cudaSuccess) {
        cudaGetLastError();
        return 1;
    }
    return occ > 0 ? occ : 1;
}

cg_status launch_drag(cg_grids* g, long long n, const void* pos_d, const void* vel, void* force, void* S_bulk,
                      bool sums, double dt, bool S_cleared, void* coef_bulk, void* pos_out, void* vel_out,
                      int32_t* perm_out) {
    const bool euler = dt > 0.0;
    void* part = part_ptr(g, PS_DRAG);
    // exactly the resident CTAs (the launch bounds' minimum per SM): a grid-stride
    // loop with no second, partial wave of blocks
    // (of 256 threads); small counts take smaller blocks, so that they reach every SM
    const long long per_sm = g->fp64 ? 2 : 4;
    int bs = 32;
    while (bs < 256 && n > 8LL * g->num_sms * bs) bs *= 2;
    const unsigned nblk = (unsigned)std::max(1LL, std::min((n + bs - 1) / bs, (long long)g->num_sms * per_sm * 256 / bs));
    g->part_blocks[PS_DRAG] = sums ? (long long)nblk : -1;
    void* Bs = nullptr;
    if (coef_bulk && n > 0) {
        // sized by the step before its first launch
        if (g->Bs.bytes < 4 * g->tsize * (size_t)n) return CG_ERR_INVALID_ARG;
        Bs = g->Bs.p;
    }
    if (pos_out && !S_bulk) return CG_ERR_INVALID_ARG;   // the sorted slots come with the fused reaction
    if (pos_out && n > 0) {
        if (!S_cleared) CG_CUDA(cudaMemsetAsync(S_bulk, 0, 3 * g->tsize * (size_t)g->gd.nbulk, g->stream));
        if (g->fp64)
            CG_TRY(launch_drag_sorted<double>(g, n, (const double*)pos_d, (const double*)vel, (double*)force,
                                              (double*)S_bulk, sums, dt, (double*)Bs, (double*)pos_out,
                                              (double*)vel_out, perm_out));
        else
            CG_TRY(launch_drag_sorted<float>(g, n, (const float*)pos_d, (const float*)vel, (float*)force, (float*)S_bulk,
                                             sums, dt, (float*)Bs, (float*)pos_out, (float*)vel_out, perm_out));
        if (coef_bulk) CG_TRY(launch_deposit_implicit(g, n, coef_bulk));
        return CG_OK;
    }
    if (perm_out && n > 0)
        CG_CUDA(cudaMemcpyAsync(perm_out, g->perm, sizeof(int32_t) * n, cudaMemcpyDeviceToDevice, g->stream));
    void* Fs = S_bulk ? g->Fs : nullptr;
    if (n > 0 || sums) {
#define CG_DRAGP(T, E)                                                                                      \
    CG_LAUNCH(g, "drag", (k_drag<T, E>), nblk, bs, 0, (T*)pos_d, (T*)vel, n, g->gd, phys_of<T>(g->gd),          \
              (const T*)g->bulk4, (T*)force, (T*)Fs, g->inv_perm, (T)dt, (T*)part, (long long)nblk, (int)sums,   \
              g->status, (T*)Bs)
        if (g->fp64) {
            if (euler) CG_DRAGP(double, true);
            else CG_DRAGP(double, false);
        } else {
            if (euler) CG_DRAGP(float, true);
            else CG_DRAGP(float, false);
        }
#undef CG_DRAGP
    }
    if (S_bulk) CG_TRY(launch_deposit_sorted_force(g, n, S_bulk, S_cleared));
    if (coef_bulk) CG_TRY(launch_deposit_implicit(g, n, coef_bulk));
    return CG_OK;
}

}  // namespace cg
