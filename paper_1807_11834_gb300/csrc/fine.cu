// fine.cu -- the two fine-grid sweeps of the coupling step (Fig. 1 of
// arXiv 1807.11834): (a2) the fluid solution goes fine -> bulk, (a4) the
// particle-related fields go bulk -> fine.
//
// Average: the r^2 rows of a bulk cell's r^3 fine cells go to several lanes
// of a warp (average_lanes), consecutive bulk cells beside each other; a row
// is one 16-byte vector per component for r = 4 (8 bytes for r = 2, two
// vectors for r = 8), and the lanes' sums merge by shuffles.  Projection: one thread per fine column of a bulk
// row, walking along z.  Every fine value is read or written exactly once
// and full lines at a time.  These two sweeps carry most of the bytes of a
// step, so they are written to stream at HBM speed.
#include <algorithm>

#include "cg_internal.cuh"
#include "batch.cuh"

namespace cg {

template <typename T, int R> struct Row;
template <> struct Row<float, 4> {
    static __device__ __forceinline__ void load(const float* p, float v[4]) {
        float4 q = __ldcs(reinterpret_cast<const float4*>(p));
        v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w;
    }
    static __device__ __forceinline__ void store(float* p, const float v[4]) {
        __stcs(reinterpret_cast<float4*>(p), make_float4(v[0], v[1], v[2], v[3]));
    }
};
template <> struct Row<float, 2> {
    static __device__ __forceinline__ void load(const float* p, float v[2]) {
        float2 q = __ldcs(reinterpret_cast<const float2*>(p));
        v[0] = q.x; v[1] = q.y;
    }
    static __device__ __forceinline__ void store(float* p, const float v[2]) {
        __stcs(reinterpret_cast<float2*>(p), make_float2(v[0], v[1]));
    }
};
template <> struct Row<float, 8> {
    static __device__ __forceinline__ void load(const float* p, float v[8]) {
        float4 a = __ldcs(reinterpret_cast<const float4*>(p)), b = __ldcs(reinterpret_cast<const float4*>(p) + 1);
        v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w; v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
    }
    static __device__ __forceinline__ void store(float* p, const float v[8]) {
        __stcs(reinterpret_cast<float4*>(p), make_float4(v[0], v[1], v[2], v[3]));
        __stcs(reinterpret_cast<float4*>(p) + 1, make_float4(v[4], v[5], v[6], v[7]));
    }
};
template <int R> struct Row<double, R> {
    static __device__ __forceinline__ void load(const double* p, double v[R]) {
#pragma unroll
        for (int i = 0; i < R; i += 2) {
            double2 q = __ldcs(reinterpret_cast<const double2*>(p + i));
            v[i] = q.x;
            v[i + 1] = q.y;
        }
    }
    static __device__ __forceinline__ void store(double* p, const double v[R]) {
#pragma unroll
        for (int i = 0; i < R; i += 2) __stcs(reinterpret_cast<double2*>(p + i), make_double2(v[i], v[i + 1]));
    }
};

__device__ __forceinline__ void bulk_ijk(long long cb, const GridDev& g, int& I, int& J, int& K) {
    I = (int)(cb % g.nb[0]);
    long long t = cb / g.nb[0];
    J = (int)(t % g.nb[1]);
    K = (int)(t / g.nb[1]);
}

// ----------------------------------------------------------------------
// (a2) mean and variance of the r^3 fine cells of a bulk cell, r = 2, 4, 8.
// The values are first shifted by the cell's first value (the subtraction
// is exact for values within a factor two of it), so that nothing below
// carries the mean's magnitude.
//
// FP32: pairwise over the rows of r values: each row gives its sum S and
// squared deviations M = sum (d - S/r)^2, and two sets of k values each
// merge as (S_a + S_b, M_a + M_b + (S_b - S_a)^2 / (2k)) (the pairwise update
// of Chan, Golub & LeVeque), in a fixed binary tree over the r^2 rows, the
// last levels across the cell's lanes; every division is by a power of two.
//
// FP64: GB300 issues FP64 at 1/64 of the FP32 rate, which bounds this path,
// so it takes the form with the fewest operations: the sum over the lanes'
// values (one addition each), then the squared deviations from the cell's
// mean (two each), four operations per value with the shift against the
// pairwise form's 5.5.
//
// Several lanes per cell instead of one thread: that many times the threads,
// which is what small grids lack (FP64, 512 bulk cells: two CTAs
// and 74 us before, 10 now; FP64, 128,000 cells 286 -> 245 us;
// FP32, 16,384 cells 10.5 -> 8.9 us).
// ----------------------------------------------------------------------
template <typename T, int RC>
__device__ __forceinline__ void average_warp(const T* __restrict__ u, const GridDev& g, T* __restrict__ ub,
                                             T* __restrict__ var, long long cell0, T* __restrict__ rec) {
    constexpr int LPC = average_lanes(RC, sizeof(T) == 8);       // lanes per cell
    constexpr int CPW = 32 / LPC;                                // cells per warp
    constexpr int NR = RC * RC / LPC;                            // rows per lane
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31, sub = lane / CPW;
    const long long cb = cell0 + lane % CPW;
    const bool valid = cb < g.nbulk;
    int I, J, K;
    bulk_ijk(valid ? cb : g.nbulk - 1, g, I, J, K);
    const long long nx = g.nf[0], nxy = (long long)g.nf[0] * g.nf[1];
    const int row0 = sub * NR;   // this lane's first row of the cell (y fastest)
    const long long f0 = (long long)I * RC + nx * ((long long)J * RC + row0 % RC) + nxy * ((long long)K * RC + row0 / RC);
    T v[3][NR][RC], ref[3], S[3], M[3];
    auto load = [&](int c) {
#pragma unroll
        for (int r = 0; r < NR; ++r) Row<T, RC>::load(u + c * g.nfine + f0 + nx * (r % RC) + nxy * (r / RC), v[c][r]);
    };
    constexpr bool ahead = NR * RC * sizeof(T) <= 128;   // all components' loads in flight together
    if constexpr (ahead)
#pragma unroll
        for (int c = 0; c < 3; ++c) load(c);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        if constexpr (!ahead) load(c);
        ref[c] = __shfl_sync(full, v[c][0][0], lane % CPW);
        T row[NR], sq[NR];
#pragma unroll
        for (int r = 0; r < NR; ++r) {
            // the row's pairwise sum
            T w[RC];
#pragma unroll
            for (int i = 0; i < RC; ++i) w[i] = v[c][r][i] -= ref[c];
#pragma unroll
            for (int h = RC / 2; h >= 1; h /= 2)
#pragma unroll
                for (int i = 0; i < h; ++i) w[i] = w[2 * i] + w[2 * i + 1];
            row[r] = w[0];
            sq[r] = T(0);
        }
        if constexpr (sizeof(T) == 4) {
#pragma unroll
            for (int r = 0; r < NR; ++r) {
                const T mean = row[r] * (T(1) / T(RC));
#pragma unroll
                for (int i = 0; i < RC; ++i) {
                    const T d = v[c][r][i] - mean;
                    sq[r] = fma(d, d, sq[r]);
                }
            }
            T k = T(RC);
#pragma unroll
            for (int h = NR / 2; h >= 1; h /= 2) {
#pragma unroll
                for (int r = 0; r < h; ++r) {
                    const T d = row[2 * r + 1] - row[2 * r];
                    sq[r] = fma(d * d, T(0.5) / k, sq[2 * r] + sq[2 * r + 1]);
                    row[r] = row[2 * r] + row[2 * r + 1];
                }
                k *= T(2);
            }
            S[c] = row[0];
            M[c] = sq[0];
#pragma unroll
            for (int off = CPW; off < 32; off <<= 1) {
                const T so = __shfl_xor_sync(full, S[c], off), mo = __shfl_xor_sync(full, M[c], off);
                const T d = S[c] - so;
                M[c] = fma(d * d, T(0.5) / k, mo + M[c]);
                S[c] = so + S[c];
                k *= T(2);
            }
        } else {
#pragma unroll
            for (int h = NR / 2; h >= 1; h /= 2)
#pragma unroll
                for (int r = 0; r < h; ++r) row[r] = row[2 * r] + row[2 * r + 1];
            S[c] = row[0];
#pragma unroll
            for (int off = CPW; off < 32; off <<= 1) S[c] += __shfl_xor_sync(full, S[c], off);
            M[c] = T(0);
            if (var) {
                const T mean = S[c] * (T(1) / T(RC * RC * RC));
#pragma unroll
                for (int r = 0; r < NR; ++r)
#pragma unroll
                    for (int i = 0; i < RC; ++i) {
                        const T d = v[c][r][i] - mean;
                        sq[r] = fma(d, d, sq[r]);
                    }
#pragma unroll
                for (int h = NR / 2; h >= 1; h /= 2)
#pragma unroll
                    for (int r = 0; r < h; ++r) sq[r] = sq[2 * r] + sq[2 * r + 1];
                M[c] = sq[0];
#pragma unroll
                for (int off = CPW; off < 32; off <<= 1) M[c] += __shfl_xor_sync(full, M[c], off);
            }
        }
    }
    if (!valid || sub != 0) return;
    constexpr T invn = T(1) / T(RC * RC * RC);
    T m2 = T(0);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const T mean = ref[c] + S[c] * invn;
        ub[c * g.nbulk + cb] = mean;
        if (rec) rec[4 * cb + 1 + c] = mean;
        m2 += M[c];
    }
    if (var) var[cb] = m2 * invn;
}

// sum (u - ref) of n values from their compensated sum: (s - n ref) + c, the
// n ref product split exactly.
template <typename T>
__device__ __forceinline__ T sum_of_shifted(const CSum<T>& s, T n, T ref) {
    const T p = n * ref, pe = fma(n, ref, -p);
    T d, e;
    two_sum(s.s, -p, d, e);
    return d + (e + (s.c - pe));
}

// (a2) r = 3: one thread per bulk cell holds a component's 27 values (their
// loads in flight together), the sum of the values (not of their differences
// to one of them, whose roundings a mean near zero would show) and then the
// squared deviations from the mean, shifted, both compensated.  The any-ratio form
// below reads value by value into one chain (39 us for 128,527 cells, 19 here).
template <typename T>
__device__ __forceinline__ void average_cell3(const T* __restrict__ u, const GridDev& g, T* __restrict__ ub,
                                              T* __restrict__ var, long long cb, T* __restrict__ rec) {
    int I, J, K;
    bulk_ijk(cb, g, I, J, K);
    const long long nx = g.nf[0], nxy = (long long)g.nf[0] * g.nf[1];
    const long long f0 = 3LL * I + nx * (3LL * J) + nxy * (3LL * K);
    CSum<T> m2;
#pragma unroll 1
    for (int c = 0; c < 3; ++c) {
        const T* p = u + c * g.nfine + f0;
        T v[27];
#pragma unroll
        for (int r = 0; r < 9; ++r)
#pragma unroll
            for (int i = 0; i < 3; ++i) v[3 * r + i] = __ldg(p + nx * (r % 3) + nxy * (r / 3) + i);
        const T ref = v[0];
        CSum<T> s;
#pragma unroll
        for (int i = 0; i < 27; ++i) s.add(v[i]);
        const T mean = s.get() / T(27);
        ub[c * g.nbulk + cb] = mean;
        if (rec) rec[4 * cb + 1 + c] = mean;
        if (var) {
            const T dm = sum_of_shifted(s, T(27), ref) / T(27);
#pragma unroll
            for (int i = 0; i < 27; ++i) {
                const T d = (v[i] - ref) - dm;
                m2.add(d * d);
            }
        }
    }
    if (var) var[cb] = m2.get() / T(27);
}

// ----------------------------------------------------------------------
// (a2) mean and variance of the r^3 fine cells of a bulk cell, any r: the ratios
// but 2, 3, 4 and 8, which have no form of their own because no workload here
// uses them in earnest (the projection has one for 5 besides).
// The variance uses a shift by the first fine value of the cell:
// var = (Q - sum_c D_c^2 / n) / n with Q = sum (u - ref)^2 and
// D_c = sum_f u_c - n ref_c, both compensated, which equals the two-pass
// population variance without a second read of the fine data.
// ----------------------------------------------------------------------
// rec (nullable): the drag's packed record (eps, u_x, u_y, u_z) per cell;
// the mean velocity is also written to its u part.
template <typename T>
__device__ __forceinline__ void average_cell(const T* __restrict__ u, const GridDev& g, T* __restrict__ ub,
                                             T* __restrict__ var, long long cb, T* __restrict__ rec);

// Bulk cells a block of nthreads takes per turn.
template <int RC, bool fp64>
__host__ __device__ constexpr int average_cells(int nthreads) {
    return nthreads / average_lanes(RC, fp64);
}

template <typename T, int RC>
__device__ __forceinline__ void average_body(const T* __restrict__ u, const GridDev& g, T* __restrict__ ub,
                                             T* __restrict__ var, Blk b, T* __restrict__ rec = nullptr) {
    const long long per = average_cells<RC, sizeof(T) == 8>(blockDim.x);
    for (long long c0 = b.id * per; c0 < g.nbulk; c0 += b.n * per) {
        if constexpr (RC == 2 || RC == 4 || RC == 8) {
            const long long w0 = c0 + (threadIdx.x >> 5) * (32 / average_lanes(RC, sizeof(T) == 8));
            if (w0 < g.nbulk) average_warp<T, RC>(u, g, ub, var, w0, rec);
        } else {
            const long long cb = c0 + threadIdx.x;
            if (cb < g.nbulk) {
                if constexpr (RC == 3) average_cell3<T>(u, g, ub, var, cb, rec);
                else average_cell<T>(u, g, ub, var, cb, rec);
            }
        }
    }
}

template <typename T, int RC>
__global__ void __launch_bounds__(256, 2)
k_average(const T* __restrict__ u, GridDev g, T* __restrict__ ub, T* __restrict__ var, T* __restrict__ rec) {
    pdl_wait();
    average_body<T, RC>(u, g, ub, var, launch_blk(), rec);
}

template <typename T>
__device__ __forceinline__ void average_cell(const T* __restrict__ u, const GridDev& g, T* __restrict__ ub,
                                             T* __restrict__ var, long long cb, T* __restrict__ rec) {
    int I, J, K;
    bulk_ijk(cb, g, I, J, K);
    const int r = g.r;
    const long long nx = g.nf[0], nxy = (long long)g.nf[0] * g.nf[1];
    const long long f0 = (long long)I * r + nx * ((long long)J * r) + nxy * ((long long)K * r);
    CSum<T> s[3], q;
    T ref[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) ref[c] = __ldg(u + c * g.nfine + f0);
    for (int dk = 0; dk < r; ++dk)
        for (int dj = 0; dj < r; ++dj) {
            const long long f = f0 + nx * dj + nxy * dk;
            for (int i = 0; i < r; ++i)
                for (int c = 0; c < 3; ++c) {
                    T v = __ldg(u + c * g.nfine + f + i);
                    s[c].add(v);
                    T dv = v - ref[c];
                    q.add(dv * dv);
                }
        }
    const T n = (T)r * (T)r * (T)r;
    const T invn = (T)1 / n;
    T corr = 0;
    T mean[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        mean[c] = s[c].get() * invn;
        ub[c * g.nbulk + cb] = mean[c];
        if (var) {
            const T D = sum_of_shifted(s[c], n, ref[c]);
            corr += D * D;
        }
    }
    if (var) {
        T a, e;
        two_sum(q.s, -corr * invn, a, e);
        T v = (a + (e + q.c)) * invn;
        var[cb] = v > T(0) ? v : T(0);
    }
    if (rec)
#pragma unroll
        for (int c = 0; c < 3; ++c) rec[4 * cb + 1 + c] = mean[c];
}

// ----------------------------------------------------------------------
// (a4) interpolate ncomp bulk fields at the fine cell centres of a bulk
// cell.  Along one axis, fine offset a in [0, r) of bulk cell I sits at
// lattice coordinate xi = I + (2a + 1 - r) / (2r): for 2a + 1 < r it lies
// between bulk centres I-1 and I with t = (2a + 1 + r) / (2r), otherwise
// between I and I+1 with t = (2a + 1 - r) / (2r).  At the domain edges the
// neighbour index is clamped to I, which reproduces constant extrapolation
// in the outer half cell exactly because lerp(a, a, t) == a.  The weights
// are exact dyadic rationals for power-of-two r.
// ----------------------------------------------------------------------
template <typename T>
__device__ __forceinline__ T lerp(T a, T b, T t) { return fma(t, b - a, a); }

// Support of fine offset a in a bulk cell along one axis: whether it is the
// lower pair (I-1, I) or the upper one (I, I+1), and the upper weight.
template <typename T>
__host__ __device__ __forceinline__ constexpr T fine_weight(int a, int r) {
    return T(2 * a + 1 < r ? 2 * a + 1 + r : 2 * a + 1 - r) / T(2 * r);
}

// Multiply a compensated sum by V_f, keeping the product's rounding error.
__device__ __forceinline__ void scale_sum(CSum<float>& a, const GridDev& g) {
    float hi = a.s * g.Vfh;
    float lo = fmaf(a.s, g.Vfh, -hi);
    lo = fmaf(a.s, g.Vfl, lo);
    lo = fmaf(a.c, g.Vfh, lo);
    a.s = hi;
    a.c = lo;
}
__device__ __forceinline__ void scale_sum(CSum<double>& a, const GridDev& g) {
    a.s *= g.Vf;
    a.c *= g.Vf;
}

// S_B V_B of one bulk cell into a conservation sum: an exact float-float
// product on the FP32 path (the reaction deposit's S_B = -(1/V_B) sum F,
// so the sums of S_B V_B and of the forces cancel to the compensated sums'
// accuracy).
__device__ __forceinline__ void add_bulk_term(CSum<float>& a, float sb, const GridDev& g) {
    const float hi = sb * g.VBh;
    float lo = fmaf(sb, g.VBh, -hi);
    lo = fmaf(sb, g.VBl, lo);
    a.add(hi);
    a.c += lo;
}
__device__ __forceinline__ void add_bulk_term(CSum<double>& a, double sb, const GridDev& g) { a.add(sb * g.VB); }

// Projection of one component.  A thread takes one fine x position of one
// bulk row (J) and walks over `depth` bulk layers K.  For each layer it loads
// the two x neighbours in the three bulk rows around J of the next layer (a
// bulk value is loaded by the r lanes of its cell at once), interpolates
// them in x and then in y to the r fine rows of J, and keeps three layers of
// such rows in registers; each of the r^2 fine values of the layer is then
// one fused multiply-add between two of them.  Stores are 32 consecutive
// values per warp for any ratio.  Against one thread per bulk cell (27 loads
// and the z, y, x interpolation per cell) an output takes 2.0 instead of 3.5
// operations for r = 4 and 2.8 instead of 9.5 for r = 2, and there are r times
// the threads, which small grids lack.  RC = 0: any ratio, the y
// interpolation repeated for each fine row (no register arrays).
// Measured before -> now, three components: FP64 512 cells (r = 4) 119 -> 12
// us; FP64 128,000 cells (r = 4) 458 -> 227; FP32 524,288 cells (r = 4) 72.3
// -> 70, (r = 2) 38.4 -> 25; FP32 128,527 cells (r = 3) 133 -> 18.
template <typename T>
struct ProjIO {
    const T* in[4];
    T* out[4];
};

// Sum of N values, neighbours first (log2 N roundings deep).
template <typename T, int N>
__device__ __forceinline__ T tree_sum(const T (&v)[N]) {
    T w[N];
#pragma unroll
    for (int i = 0; i < N; ++i) w[i] = v[i];
#pragma unroll
    for (int m = N; m > 1; m = (m + 1) / 2)
#pragma unroll
        for (int i = 0; i < (m + 1) / 2; ++i) w[i] = 2 * i + 1 < m ? w[2 * i] + w[2 * i + 1] : w[2 * i];
    return w[0];
}

template <typename T, int RC, bool SUMS>
__device__ __forceinline__ void project_body(const T* __restrict__ B, T* __restrict__ O, const GridDev& g, int depth,
                                             T* __restrict__ part, long long pstride, int comp, Blk b) {
    const int r = RC ? RC : g.r;
    const unsigned nfx = (unsigned)g.nf[0], nbx = (unsigned)g.nb[0], nby = (unsigned)g.nb[1];
    const int nbz = g.nb[2];
    const long long t = b.id * blockDim.x + threadIdx.x;
    const unsigned nseg = (unsigned)((nbz + depth - 1) / depth);
    CSum<T> acc[2];   // sum S_f, then sum S_B V_B
    T mine_left = T(0);
    if (t < (long long)nfx * nby * nseg) {
        const unsigned row = (unsigned)(t / nfx), fx = (unsigned)(t - (long long)row * nfx);
        const unsigned seg = row / nby;
        const int J = (int)(row - seg * nby);
        const int I = (int)(fx / (unsigned)r), off = (int)fx - I * r;
        const bool cell = g.interp == CG_INTERP_CELL;
        const bool xl = 2 * off + 1 < r;
        const int x0 = cell ? I : xl ? max(I - 1, 0) : I, x1 = cell || xl ? I : min(I + 1, (int)nbx - 1);
        const T tx = fine_weight<T>(off, r);
        const unsigned y0 = nbx * (unsigned)(cell ? J : max(J - 1, 0)), y1 = nbx * (unsigned)J;
        const unsigned y2 = nbx * (unsigned)(cell ? J : min(J + 1, (int)nby - 1));
        const unsigned layer = nbx * nby;
        const int k0 = (int)seg * depth, k1 = min(k0 + depth, nbz);
        constexpr int NY = RC ? RC : 3;   // rows kept per layer: the r fine ones, or the three bulk ones
        T lo[NY], mid[NY], hi[NY], dlo[NY], centre = T(0), centre_n = T(0), mine = T(0);
        int turn = 0;
        auto rows = [&](int K, T (&p)[NY], T& c) {
            const T* q = B + (size_t)layer * (unsigned)K;
            T a[3], e[3], x[3];
            a[0] = __ldg(q + y0 + x0);
            e[0] = __ldg(q + y0 + x1);
            a[1] = __ldg(q + y1 + x0);
            e[1] = __ldg(q + y1 + x1);
            a[2] = __ldg(q + y2 + x0);
            e[2] = __ldg(q + y2 + x1);
            c = xl ? e[1] : a[1];   // this bulk cell's own value
#pragma unroll
            for (int j = 0; j < 3; ++j) x[j] = lerp(a[j], e[j], tx);
            if constexpr (RC > 0) {
#pragma unroll
                for (int ay = 0; ay < RC; ++ay) {
                    constexpr int R = RC;
                    p[ay] = 2 * ay + 1 < R ? lerp(x[0], x[1], fine_weight<T>(ay, R)) : lerp(x[1], x[2], fine_weight<T>(ay, R));
                }
            } else {
#pragma unroll
                for (int j = 0; j < 3; ++j) p[j] = x[j];
            }
        };
        T dummy;
        rows(cell ? k0 : max(k0 - 1, 0), lo, dummy);
        rows(k0, mid, centre);
        if constexpr (RC > 0)
#pragma unroll
            for (int ay = 0; ay < RC; ++ay) dlo[ay] = mid[ay] - lo[ay];
        const size_t nx = nfx, nxy = (size_t)nfx * (unsigned)g.nf[1];
        T* o = O + fx + nx * ((size_t)J * r) + nxy * ((size_t)k0 * r);
        for (int K = k0; K < k1; ++K) {
            rows(min(K + 1, nbz - 1), hi, centre_n);
            if constexpr (RC > 0) {
                T rs[RC];
#pragma unroll
                for (int ay = 0; ay < RC; ++ay) {
                    // cell values: no slope (T(0) * x keeps a NaN or an infinity a NaN, as the difference does)
                    const T flat = T(0) * mid[ay], base = cell ? mid[ay] : lo[ay];
                    const T dl = cell ? flat : dlo[ay], dhi = cell ? flat : hi[ay] - mid[ay];
                    T v[RC];
#pragma unroll
                    for (int az = 0; az < RC; ++az) {
                        v[az] = 2 * az + 1 < RC ? fma(fine_weight<T>(az, RC), dl, base)
                                                : fma(fine_weight<T>(az, RC), dhi, mid[ay]);
                        __stcs(o + nx * ay + nxy * az, v[az]);
                    }
                    dlo[ay] = dhi;
                    if (SUMS) rs[ay] = tree_sum(v);
                }
                if (SUMS) acc[0].add(tree_sum(rs));
            } else {
                for (int ay = 0; ay < r; ++ay) {
                    const bool yl = 2 * ay + 1 < r;
                    const T ty = fine_weight<T>(ay, r);
                    const T m = yl ? lerp(mid[0], mid[1], ty) : lerp(mid[1], mid[2], ty);
                    const T a = cell ? m : yl ? lerp(lo[0], lo[1], ty) : lerp(lo[1], lo[2], ty);
                    const T h = cell ? m : yl ? lerp(hi[0], hi[1], ty) : lerp(hi[1], hi[2], ty);
                    for (int az = 0; az < r; ++az) {
                        const T v = 2 * az + 1 < r ? lerp(a, m, fine_weight<T>(az, r)) : lerp(m, h, fine_weight<T>(az, r));
                        __stcs(o + nx * ay + nxy * az, v);
                        if (SUMS) acc[0].add(v);
                    }
                }
            }
            if (SUMS) {
                // each of the r lanes of a bulk cell takes every r-th layer's S_B, so that all add at once
                if (off == turn) mine = centre;
                if (++turn == r) {
                    add_bulk_term(acc[1], mine, g);
                    mine = T(0);
                    turn = 0;
                }
            }
            o += nxy * r;
            centre = centre_n;
#pragma unroll
            for (int j = 0; j < NY; ++j) {
                lo[j] = mid[j];
                mid[j] = hi[j];
            }
        }
        mine_left = mine;
    }
    if (SUMS) {
        add_bulk_term(acc[1], mine_left, g);
        // sum_f S_f V_f = V_f sum_f S_f; V_f applied as a float-float product
        scale_sum(acc[0], g);
        // columns comp (S_f V_f) and comp + 3 (S_B V_B) of the partials
        block_sums<T, 2>(acc, part + 2 * comp * pstride, 3 * pstride, b.id);
    }
}

// Layers per thread: the two extra layers a thread loads at its ends cost
// 2 / depth of the loads and of the x and y interpolations, so as many as
// leave enough threads: about 200,000 for FP32 (streaming stores; FP32, r = 3,
// 128,527 cells: depth 1 28.7, 2 20.5, 5 16.8 us), 80,000 for FP64, which its
// few FP64 lanes bound (128,000 cells: depth 1 543, 3 328, 7 266 us); at most
// 8 and 16, where the cost of the ends is small already.
int project_depth(const GridDev& g, int ncomp, bool fp64) {
    const long long cols = (long long)g.nf[0] * g.nb[1] * ncomp;
    return (int)std::max(1LL, std::min<long long>(fp64 ? 16 : 8, cols * g.nb[2] / (fp64 ? 80000 : 200000)));
}
long long project_threads(const GridDev& g, int depth) {
    return (long long)g.nf[0] * g.nb[1] * ((g.nb[2] + depth - 1) / depth);
}
// Small grids take small blocks, so that their few warps reach every SM; so
// does FP64, whose time is the busiest SM's share of the arithmetic.
int project_block(const GridDev& g, int ncomp, bool fp64, int num_sms) {
    return project_threads(g, project_depth(g, ncomp, fp64)) * ncomp >= 512LL * num_sms ? (fp64 ? 64 : 256) : 32;
}
long long project_blocks(const GridDev& g, int ncomp, bool fp64, int num_sms) {
    const int bs = project_block(g, ncomp, fp64, num_sms);
    return (project_threads(g, project_depth(g, ncomp, fp64)) + bs - 1) / bs;
}

template <typename T, int RC, bool SUMS>
__global__ void __launch_bounds__(256)
k_project(ProjIO<T> io, GridDev g, int depth, T* __restrict__ part, long long pstride) {
    pdl_wait();
    const int c = blockIdx.y;
    project_body<T, RC, SUMS>(c == 0 ? io.in[0] : c == 1 ? io.in[1] : c == 2 ? io.in[2] : io.in[3],
                              c == 0 ? io.out[0] : c == 1 ? io.out[1] : c == 2 ? io.out[2] : io.out[3], g, depth, part,
                              pstride, c, launch_blk());
}

// ----------------------------------------------------------------------
// Batched fine-grid phases (FP32 instances, ratio 2, 4 or 8)
// ----------------------------------------------------------------------
__global__ void __launch_bounds__(256, 2) kb_average(BLaunch L) {
    batch_loop(L, [&](const BInst& I, Blk b) {
        switch (I.gd.r) {
            case 2: average_body<float, 2>(I.u_fine, I.gd, I.u_bulk, I.var, b); break;
            case 4: average_body<float, 4>(I.u_fine, I.gd, I.u_bulk, I.var, b); break;
            default: average_body<float, 8>(I.u_fine, I.gd, I.u_bulk, I.var, b); break;
        }
    });
}

// eps: project the porosity (one component, no sums) instead of the source
// (three components, a third of the instance's blocks each); SUMS: some
// instance of the batch wants its conservation sums
template <bool EPS, bool SUMS>
__global__ void __launch_bounds__(256) kb_project(BLaunch L) {
    batch_loop(L, [&](const BInst& I, Blk b) {
        const long long nb = I.gd.nbulk, nf = I.gd.nfine;
        const long long per = EPS ? b.n : b.n / 3;
        const int c = (int)(b.id / per);
        const float* in = EPS ? I.eps_t : I.S_bulk + c * nb;
        float* out = EPS ? I.eps_fine : I.S_fine + c * nf;
        float* part = I.part + 2 * I.part_off[PS_PROJ];
        const Blk bb = {b.id - c * per, per};
        const int depth = EPS ? I.depth_eps : I.depth;
        switch (I.gd.r) {
            case 2: project_body<float, 2, SUMS>(in, out, I.gd, depth, part, per, c, bb); break;
            case 4: project_body<float, 4, SUMS>(in, out, I.gd, depth, part, per, c, bb); break;
            default: project_body<float, 8, SUMS>(in, out, I.gd, depth, part, per, c, bb); break;
        }
    });
}

cg_status launch_batch_fine(int phase, const BLaunch& L, unsigned grid, cudaStream_t s) {
    if (L.total == 0 || grid == 0) return CG_OK;
    switch (phase) {
        case BP_AVG: kb_average<<<grid, 256, 0, s>>>(L); break;
        case BP_PROJ:
            if (L.sums) kb_project<false, true><<<grid, 256, 0, s>>>(L);
            else kb_project<false, false><<<grid, 256, 0, s>>>(L);
            break;
        case BP_PROJE: kb_project<true, false><<<grid, 256, 0, s>>>(L); break;
        default: return CG_ERR_INVALID_ARG;
    }
    CG_CUDA(cudaGetLastError());
    return CG_OK;
}

int batch_fine_occupancy(int phase, bool sums) {
    int occ = 0;
    auto of = [&](auto k) { return cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k, 256, 0); };
    const cudaError_t e = phase == BP_AVG     ? of(kb_average)
                          : phase == BP_PROJE ? of(kb_project<true, false>)
                          : sums              ? of(kb_project<false, true>)
                                              : of(kb_project<false, false>);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return 1;
    }
    return occ > 0 ? occ : 1;
}

// The average's grid.  Large grids: grid-stride over two blocks per SM
// (four for r = 2, whose threads hold fewer values), enough loads in flight to stream near HBM speed while leaving warp slots
// to the particle kernels beside it (with one thread per cell, two blocks of
// 256 per SM slowed the step by 12 us).  Small grids take blocks of 64
// threads, so that their warps reach every SM; ratio 3 and the any-ratio form
// take a thread per cell at full occupancy.
template <typename T, int RC>
static cg_status average_launch(cg_grids* g, const void* u_fine, void* u_bulk, void* var_bulk, void* rec) {
    constexpr bool warp = RC == 2 || RC == 4 || RC == 8;
    const int bs = warp && g->gd.nbulk >= 64LL * g->num_sms ? 256 : 64;
    const long long need = (g->gd.nbulk + average_cells<RC, sizeof(T) == 8>(bs) - 1) / average_cells<RC, sizeof(T) == 8>(bs);
    // FP64: a block per group of cells.  The busiest SM's arithmetic is its time, and two
    // resident blocks per SM, placed beside the particle kernels that have
    // started first, fall unevenly on the SMs (1M particles, 128,000 cells: the
    // step 1026 -> 939 us)
    const unsigned nblk =
        (unsigned)std::min(need, (long long)g->num_sms * (bs == 256 && sizeof(T) == 4 ? (RC == 2 ? 4 : 2) : 32));
    CG_LAUNCH(g, "average", (k_average<T, RC>), nblk, bs, 0, (const T*)u_fine, g->gd, (T*)u_bulk, (T*)var_bulk, (T*)rec);
    return CG_OK;
}

cg_status launch_average(cg_grids* g, const void* u_fine, void* u_bulk, void* var_bulk, void* rec) {
#define CG_AVG(T)                                                                          \
    switch (g->gd.r) {                                                                     \
        case 2: return average_launch<T, 2>(g, u_fine, u_bulk, var_bulk, rec);             \
        case 3: return average_launch<T, 3>(g, u_fine, u_bulk, var_bulk, rec);             \
        case 4: return average_launch<T, 4>(g, u_fine, u_bulk, var_bulk, rec);             \
        case 8: return average_launch<T, 8>(g, u_fine, u_bulk, var_bulk, rec);             \
        default: return average_launch<T, 0>(g, u_fine, u_bulk, var_bulk, rec);            \
    }
    if (g->fp64) CG_AVG(double)
    CG_AVG(float)
#undef CG_AVG
}

template <typename T, int RC>
static cg_status project_launch(cg_grids* g, int ncomp, const void* const* in, void* const* out, bool sums) {
    ProjIO<T> io;
    for (int c = 0; c < 4; ++c) {
        io.in[c] = (const T*)in[c];
        io.out[c] = (T*)out[c];
    }
    const bool fp64 = sizeof(T) == 8;
    const int depth = project_depth(g->gd, ncomp, fp64), bs = project_block(g->gd, ncomp, fp64, g->num_sms);
    const long long nblk = project_blocks(g->gd, ncomp, fp64, g->num_sms);
    // only the projection that forms the sums claims their partials (a later
    // projection without sums, of the porosity or the semi-implicit
    // coefficients, leaves them to it)
    if (sums) g->part_blocks[PS_PROJ] = nblk;
    const char* name = ncomp == 1 ? "project_eps" : ncomp == 4 ? "project_implicit" : "project";
    T* part = (T*)part_ptr(g, PS_PROJ);
    const dim3 grid((unsigned)nblk, (unsigned)ncomp);
    if (sums) CG_LAUNCH(g, name, (k_project<T, RC, true>), grid, bs, 0, io, g->gd, depth, part, nblk);
    else CG_LAUNCH(g, name, (k_project<T, RC, false>), grid, bs, 0, io, g->gd, depth, part, nblk);
    return CG_OK;
}

cg_status launch_project(cg_grids* g, int ncomp, const void* const* in, void* const* out, bool sums) {
#define CG_PRJ(T)                                                              \
    switch (g->gd.r) {                                                         \
        case 2: return project_launch<T, 2>(g, ncomp, in, out, sums);          \
        case 3: return project_launch<T, 3>(g, ncomp, in, out, sums);          \
        case 4: return project_launch<T, 4>(g, ncomp, in, out, sums);          \
        case 5: return project_launch<T, 5>(g, ncomp, in, out, sums);          \
        case 8: return project_launch<T, 8>(g, ncomp, in, out, sums);          \
        default: return project_launch<T, 0>(g, ncomp, in, out, sums);         \
    }
    if (g->fp64) CG_PRJ(double)
    CG_PRJ(float)
#undef CG_PRJ
}

}  // namespace cg
