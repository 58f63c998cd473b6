// map.cu -- maps between two uniform grids in any relative position and
// with any spacings: the grid-to-grid transfer of arXiv 1807.11834
// (Fig. 1 arrows; Sec. 2.3: the mapping structure is static and computed
// once per simulation) for grids that are not nested.
//
// With V(B & f) the volume of the intersection of bulk cell B and fine
// cell f:
//   average (fine -> bulk):  u_B = sum_f V(B & f) u_f / sum_f V(B & f)
//   project (bulk -> fine):  S_f = sum_B V(B & f) S_B / V_f   (conserves sum S V
//                            where the fine grid covers the bulk one)
// Both grids are boxes, so V(B & f) is the product of the overlaps of the
// cells' intervals on the three axes.  The static structure is one
// compressed-row table per axis and direction (bulk index -> overlapping
// fine indices and overlap lengths, and fine -> bulk), built once on the
// host in double and kept on the device; the 3-D weight of a pair is the
// product of its three axis entries.  Average: a thread per fine x index of a
// bulk row sums its fine column over y and z, and the block combines the
// columns along x in shared memory.  Projection: when no fine cell overlaps
// more than two bulk cells along an axis (fine cells no larger than bulk
// cells), a thread per fine column along z with the bulk planes collapsed over
// x and y in registers; else one thread per fine cell through the compressed
// rows.
#include <math.h>
#include <string.h>

#include <algorithm>
#include <new>
#include <vector>

#include "cg_internal.cuh"

struct cg_map {
    cg_box_grid bulk, fine;
    int fp64 = 0;
    size_t tsize = 4;
    cudaStream_t stream = nullptr;
    int num_sms = 148;
    long long nbulk = 0, nfine = 0;
    // per axis: [ptr (n+1) int32][idx int32][w T], average (bulk rows) and projection (fine rows)
    void* dev = nullptr;
    long long off_bptr[3], off_bidx[3], off_bw[3], off_fptr[3], off_fidx[3], off_fw[3], off_cov[3];
    // when no fine cell overlaps more than two bulk cells along any axis:
    // per axis and fine index, the first bulk index and the two overlaps
    bool two = false;
    long long off_f2b[3], off_f2w0[3], off_f2w1[3];
    double Vf = 0.0;
    int avg_tile = 0, avg_threads = 0;   // bulk x cells and threads per block of the average; 0: a cell per thread
    int avg_rows = 0;                    // most fine rows (y) under a bulk row
};

namespace cg {
namespace {

// Cell bounds along an axis: x0 + i L / n (the same expression for the upper
// bound of cell i and the lower bound of cell i + 1).
inline double bound(const cg_box_grid& G, int a, long long i) { return G.origin[a] + (double)i * (G.extent[a] / G.n[a]); }

inline double overlap_len(double a0, double a1, double b0, double b1) {
    const double lo = std::max(a0, b0), hi = std::min(a1, b1);
    return hi > lo ? hi - lo : 0.0;
}

// Compressed rows of grid R's cells along axis a: for each row cell, the
// cells of grid C along a that overlap it, and the overlap lengths.
void axis_rows(const cg_box_grid& R, const cg_box_grid& Cg, int a, std::vector<int>& ptr, std::vector<int>& idx,
               std::vector<double>& w) {
    const int nr = R.n[a], nc = Cg.n[a];
    const double hc = Cg.extent[a] / nc;
    ptr.assign(nr + 1, 0);
    idx.clear();
    w.clear();
    for (int i = 0; i < nr; ++i) {
        const double lo = bound(R, a, i), hi = bound(R, a, i + 1);
        long long j0 = (long long)floor((lo - Cg.origin[a]) / hc) - 1, j1 = (long long)floor((hi - Cg.origin[a]) / hc) + 1;
        j0 = std::max(j0, 0LL);
        j1 = std::min(j1, (long long)nc - 1);
        for (long long j = j0; j <= j1; ++j) {
            const double v = overlap_len(lo, hi, bound(Cg, a, j), bound(Cg, a, j + 1));
            if (v > 0.0) {
                idx.push_back((int)j);
                w.push_back(v);
            }
        }
        ptr[i + 1] = (int)idx.size();
    }
}

template <typename T>
struct MapDev {
    const int* bptr[3];
    const int* bidx[3];
    const T* bw[3];
    const int* fptr[3];
    const int* fidx[3];
    const T* fw[3];
    const T* cov[3];   // per bulk index: covered length along the axis
    const int* f2b[3];
    const T* f2w0[3];
    const T* f2w1[3];
    int nb[3], nf[3];
    T inv_Vf;
};

template <typename T>
MapDev<T> dev_view(const cg_map* m) {
    MapDev<T> d;
    const char* base = (const char*)m->dev;
    for (int a = 0; a < 3; ++a) {
        d.bptr[a] = (const int*)(base + m->off_bptr[a]);
        d.bidx[a] = (const int*)(base + m->off_bidx[a]);
        d.bw[a] = (const T*)(base + m->off_bw[a]);
        d.fptr[a] = (const int*)(base + m->off_fptr[a]);
        d.fidx[a] = (const int*)(base + m->off_fidx[a]);
        d.fw[a] = (const T*)(base + m->off_fw[a]);
        d.cov[a] = (const T*)(base + m->off_cov[a]);
        d.f2b[a] = m->two ? (const int*)(base + m->off_f2b[a]) : nullptr;
        d.f2w0[a] = m->two ? (const T*)(base + m->off_f2w0[a]) : nullptr;
        d.f2w1[a] = m->two ? (const T*)(base + m->off_f2w1[a]) : nullptr;
        d.nb[a] = m->bulk.n[a];
        d.nf[a] = m->fine.n[a];
    }
    d.inv_Vf = (T)(1.0 / m->Vf);
    return d;
}

constexpr int kMapMaxComp = 8;

// Average, thread t of a block taking the t-th fine x index under a tile of bulk
// x cells, over the fine rows of bulk row (J, K) for the K of a chunk: the
// column's y terms in plain FMAs (MANY, some bulk row over more than map_plain of
// them: in chains of that length, compensated; as one chain 4096 rows were off by
// 2e-6), its planes (weighted by z) into a compensated sum, then the x terms,
// compensated likewise, from shared memory.
// A plane shared by the cells K and K + 1 is kept.  Every fine value is read
// once from HBM, those of the rows shared by two bulk rows a second time from L2.
// The loads are coalesced along x and copied asynchronously into shared memory
// two planes ahead (in registers they cost half of the occupancy: 117 us).
// Bound by instruction issue and latency (issue 53%).  A thread per bulk cell
// (the form below, kept for a bulk cell over more than 256 fine x indices)
// gathers runs of a few values per lane, four times the L1 wavefronts: 250 x 250
// x 500 fine to 64 x 64 x 128 bulk cells, three components, FP32 127 -> 102 us.
template <typename T>
__device__ __forceinline__ void copy_async(T* dst, const T* src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src),
                 "n"(sizeof(T))
                 : "memory");
}
constexpr int kMapRows = 6, kMapStages = 2;   // rows of a plane in shared memory, planes in flight
// Terms of a plain chain; more go chain by chain into a compensated sum.
__host__ __device__ constexpr int map_plain(size_t tsize) { return tsize == 4 ? 8 : 16; }
template <typename T, int NC, bool MANY>
__global__ void __launch_bounds__(256) k_map_average_rows(MapDev<T> d, int tile, int ntiles, int depth,
                                                          const T* __restrict__ in, T* __restrict__ out) {
    pdl_wait();
    constexpr int G = sizeof(T) == 4 ? kMapRows : kMapRows / 2, P = map_plain(sizeof(T));
    __shared__ T sh[2][NC][256];
    __shared__ T ring[kMapStages][G][NC][256];   // a thread copies and reads its own column only
    const int nbx = d.nb[0], nby = d.nb[1], nbz = d.nb[2];
    const size_t nbk = (size_t)nbx * nby * nbz;
    const size_t nfx = d.nf[0], plane = nfx * d.nf[1], nfn = plane * d.nf[2];
    in += blockIdx.y * (NC * nfn);
    out += blockIdx.y * (NC * nbk);
    unsigned b = blockIdx.x;
    const int t = (int)(b % (unsigned)ntiles);
    b /= (unsigned)ntiles;
    const int J = (int)(b % (unsigned)nby);
    const int K0 = (int)(b / (unsigned)nby) * depth, K1 = min(K0 + depth, nbz);
    const int I0 = t * tile, I1 = min(I0 + tile, nbx);
    const int p0 = __ldg(d.bptr[0] + I0), p1 = __ldg(d.bptr[0] + I1);
    const int f0 = p1 > p0 ? __ldg(d.bidx[0] + p0) : 0;
    const int span = p1 > p0 ? __ldg(d.bidx[0] + p1 - 1) - f0 + 1 : 0;
    const int y0 = __ldg(d.bptr[1] + J), ny = __ldg(d.bptr[1] + J + 1) - y0;
    const int zp0 = __ldg(d.bptr[2] + K0), zp1 = __ldg(d.bptr[2] + K1);
    const bool on = (int)threadIdx.x < span && ny > 0 && zp1 > zp0;
    // the overlapping indices of a row are consecutive
    const T* wy = d.bw[1] + y0;
    T w[G];
#pragma unroll
    for (int y = 0; y < G; ++y) w[y] = y < ny ? __ldg(wy + y) : T(0);
    int fz = on ? __ldg(d.bidx[2] + zp0) : 0;   // the next plane to be added; ahead: to be copied
    const int zlast = on ? __ldg(d.bidx[2] + zp1 - 1) : -1;
    const T* ahead = in + (f0 + (int)threadIdx.x) + (on ? nfx * __ldg(d.bidx[1] + y0) : 0) + plane * fz;
    int za = fz;
    auto copy_plane = [&](int stage) {
        if (za <= zlast) {
            const T* q = ahead;
#pragma unroll
            for (int y = 0; y < G; ++y, q += nfx)
                if (y < ny)
#pragma unroll
                    for (int c = 0; c < NC; ++c) copy_async(&ring[stage][y][c][threadIdx.x], q + c * nfn);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
        ahead += plane;
        ++za;
    };
    int stage = 0;
    if (on)
#pragma unroll
        for (int i = 0; i < kMapStages; ++i) copy_plane(i);
    T rs[NC];
    int have = -1;   // the plane that rs holds
    for (int K = K0; K < K1; ++K) {
        if (on) {
            CSum<T> acc[NC];
            const int z1 = __ldg(d.bptr[2] + K + 1);
            for (int kz = __ldg(d.bptr[2] + K); kz < z1; ++kz) {
                const int f = __ldg(d.bidx[2] + kz);
                const T wz = __ldg(d.bw[2] + kz);
                if (f != have) {   // then f is the next plane
                    have = f;
                    asm volatile("cp.async.wait_group %0;" ::"n"(kMapStages - 1) : "memory");
#pragma unroll
                    for (int c = 0; c < NC; ++c) rs[c] = T(0);
#pragma unroll
                    for (int y = 0; y < G; ++y)
                        if (y < ny)
#pragma unroll
                            for (int c = 0; c < NC; ++c) rs[c] = fma(w[y], ring[stage][y][c][threadIdx.x], rs[c]);
                    if (ny > G) {
                        const T* q = ahead - kMapStages * plane + nfx * G;
                        CSum<T> sum[NC];   // MANY: of these terms and then P by P
                        for (int y = G; y < ny;) {
                            if (MANY)
#pragma unroll
                                for (int c = 0; c < NC; ++c) {
                                    sum[c].add(rs[c]);
                                    rs[c] = T(0);
                                }
                            for (const int end = MANY ? min(y + P, ny) : ny; y < end; ++y, q += nfx)
#pragma unroll
                                for (int c = 0; c < NC; ++c) rs[c] = fma(__ldg(wy + y), __ldg(q + c * nfn), rs[c]);
                        }
                        if (MANY)
#pragma unroll
                            for (int c = 0; c < NC; ++c) {
                                sum[c].add(rs[c]);
                                rs[c] = sum[c].get();
                            }
                    }
                    copy_plane(stage);
                    stage = stage + 1 == kMapStages ? 0 : stage + 1;
                }
#pragma unroll
                for (int c = 0; c < NC; ++c) acc[c].add(wz * rs[c]);
            }
#pragma unroll
            for (int c = 0; c < NC; ++c) sh[K & 1][c][threadIdx.x] = acc[c].get();
        }
        __syncthreads();   // one per K: the next one writes the other half
        const T wJK = __ldg(d.cov[1] + J) * __ldg(d.cov[2] + K);
        const int m = I1 - I0;
        for (int o = threadIdx.x; o < m * NC; o += blockDim.x) {
            const int c = o / m, I = I0 + o - c * m;
            const T W = __ldg(d.cov[0] + I) * wJK;
            CSum<T> a;
            if (W > T(0)) {
                const int x0 = __ldg(d.bptr[0] + I), x1 = __ldg(d.bptr[0] + I + 1);
                const T* v = sh[K & 1][c] + (__ldg(d.bidx[0] + x0) - f0 - x0);
                for (int kx = x0; kx < x1; ++kx) a.add(__ldg(d.bw[0] + kx) * v[kx]);
            }
            out[c * nbk + I + (size_t)nbx * (J + (size_t)nby * K)] = W > T(0) ? a.get() / W : T(0);
        }
    }
}

// The kernels over cells take them in x-fastest order with 32-bit index
// arithmetic (grids hold fewer than 2^31 cells): one division per cell splits
// the index into the x index and the row (y, z), whose two axis ranges are
// looked up once per cell.
template <typename T, int NC>
__global__ void __launch_bounds__(256) k_map_average(MapDev<T> d, const T* __restrict__ in, T* __restrict__ out) {
    pdl_wait();
    const unsigned nbx = (unsigned)d.nb[0], nby = (unsigned)d.nb[1];
    const unsigned nbk = nbx * nby * (unsigned)d.nb[2];
    const unsigned nfx = (unsigned)d.nf[0], nfy = (unsigned)d.nf[1];
    const size_t nfn = (size_t)nfx * nfy * (unsigned)d.nf[2];
    for (unsigned cb = blockIdx.x * blockDim.x + threadIdx.x; cb < nbk; cb += gridDim.x * blockDim.x) {
        const unsigned row = cb / nbx;
        const unsigned I = cb - row * nbx;
        const unsigned J = row % nby, K = row / nby;
        const int x0 = __ldg(d.bptr[0] + I), x1 = __ldg(d.bptr[0] + I + 1);
        const int y0 = __ldg(d.bptr[1] + J), y1 = __ldg(d.bptr[1] + J + 1);
        const int z0 = __ldg(d.bptr[2] + K), z1 = __ldg(d.bptr[2] + K + 1);
        // each fine row's x terms in plain FMAs (FP32: of up to 16), these sums (weighted
        // by y and z) into compensated sums
        const int chain = sizeof(T) == 4 ? 16 : max(x1 - x0, 1);
        CSum<T> acc[NC];
        for (int kz = z0; kz < z1; ++kz) {
            const unsigned fz = (unsigned)__ldg(d.bidx[2] + kz);
            const T wz = __ldg(d.bw[2] + kz);
            for (int ky = y0; ky < y1; ++ky) {
                const unsigned fy = (unsigned)__ldg(d.bidx[1] + ky);
                const T wyz = __ldg(d.bw[1] + ky) * wz;
                const T* rowp = in + (size_t)nfx * (fy + nfy * fz);
                for (int k0 = x0; k0 < x1; k0 += chain) {
                    T rs[NC];
#pragma unroll
                    for (int c = 0; c < NC; ++c) rs[c] = T(0);
                    for (int kx = k0; kx < min(k0 + chain, x1); ++kx) {
                        const unsigned fx = (unsigned)__ldg(d.bidx[0] + kx);
                        const T wx = __ldg(d.bw[0] + kx);
#pragma unroll
                        for (int c = 0; c < NC; ++c) rs[c] = fma(wx, __ldg(rowp + c * nfn + fx), rs[c]);
                    }
#pragma unroll
                    for (int c = 0; c < NC; ++c) acc[c].add(wyz * rs[c]);
                }
            }
        }
        const T W = __ldg(d.cov[0] + I) * __ldg(d.cov[1] + J) * __ldg(d.cov[2] + K);
#pragma unroll
        for (int c = 0; c < NC; ++c) out[(size_t)c * nbk + cb] = W > T(0) ? acc[c].get() / W : T(0);
    }
}

template <typename T, int NC>
__global__ void __launch_bounds__(256) k_map_project(MapDev<T> d, const T* __restrict__ in, T* __restrict__ out) {
    pdl_wait();
    const unsigned nbx = (unsigned)d.nb[0], nby = (unsigned)d.nb[1];
    const size_t nbk = (size_t)nbx * nby * (unsigned)d.nb[2];
    const unsigned nfx = (unsigned)d.nf[0], nfy = (unsigned)d.nf[1];
    const unsigned nfn = nfx * nfy * (unsigned)d.nf[2];
    for (unsigned cf = blockIdx.x * blockDim.x + threadIdx.x; cf < nfn; cf += gridDim.x * blockDim.x) {
        const unsigned row = cf / nfx;
        const unsigned i = cf - row * nfx;
        const unsigned j = row % nfy, k = row / nfy;
        const int x0 = __ldg(d.fptr[0] + i), x1 = __ldg(d.fptr[0] + i + 1);
        const int y0 = __ldg(d.fptr[1] + j), y1 = __ldg(d.fptr[1] + j + 1);
        const int z0 = __ldg(d.fptr[2] + k), z1 = __ldg(d.fptr[2] + k + 1);
        T acc[NC];
#pragma unroll
        for (int c = 0; c < NC; ++c) acc[c] = T(0);
        for (int kz = z0; kz < z1; ++kz) {
            const unsigned bz = (unsigned)__ldg(d.fidx[2] + kz);
            const T wz = __ldg(d.fw[2] + kz);
            for (int ky = y0; ky < y1; ++ky) {
                const unsigned by = (unsigned)__ldg(d.fidx[1] + ky);
                const T wyz = __ldg(d.fw[1] + ky) * wz;
                const size_t brow = (size_t)nbx * (by + nby * bz);
                for (int kx = x0; kx < x1; ++kx) {
                    const size_t b = brow + (unsigned)__ldg(d.fidx[0] + kx);
                    const T w = __ldg(d.fw[0] + kx) * wyz;
#pragma unroll
                    for (int c = 0; c < NC; ++c) acc[c] = fma(w, __ldg(in + c * nbk + b), acc[c]);
                }
            }
        }
#pragma unroll
        for (int c = 0; c < NC; ++c) out[(size_t)c * nfn + cf] = acc[c] * d.inv_Vf;
    }
}

// Projection when every fine cell overlaps at most two bulk cells per axis (the
// second weight 0 where there is one): a thread per fine column walks `depth`
// fine planes along z with the two bulk planes around it, collapsed over x and
// y, in registers, so that a plane costs one load of its z weights and two
// operations and a store per component.  Bound by the HBM stores: 64 x 64 x 128
// bulk to 250 x 250 x 500 fine cells, three components, FP32 78 us, against
// 169 for a block per fine row with the bulk rows collapsed in shared memory.
template <typename T, int NC>
__global__ void __launch_bounds__(256) k_map_project2(MapDev<T> d, unsigned colblk, int depth,
                                                      const T* __restrict__ in, T* __restrict__ out) {
    pdl_wait();
    const unsigned nbx = (unsigned)d.nb[0], nby = (unsigned)d.nb[1], nbz = (unsigned)d.nb[2];
    const size_t bplane = (size_t)nbx * nby, nbk = bplane * nbz;
    const unsigned nfx = (unsigned)d.nf[0], plane = nfx * (unsigned)d.nf[1];
    const size_t nfn = (size_t)plane * (unsigned)d.nf[2];
    const unsigned chunk = blockIdx.x / colblk;
    const unsigned q = (blockIdx.x - chunk * colblk) * blockDim.x + threadIdx.x;
    if (q >= plane) return;
    const unsigned j = q / nfx, i = q - j * nfx;
    const unsigned bx = (unsigned)__ldg(d.f2b[0] + i), by = (unsigned)__ldg(d.f2b[1] + j);
    const T wx0 = __ldg(d.f2w0[0] + i), wx1 = __ldg(d.f2w1[0] + i);
    const T wy0 = __ldg(d.f2w0[1] + j), wy1 = __ldg(d.f2w1[1] + j);
    // the second neighbour stays inside the grid (its weight is 0 at the edge)
    const unsigned dx = bx + 1 < nbx ? 1u : 0u, dy = by + 1 < nby ? nbx : 0u;
    const T* s0 = in + bx + (size_t)nbx * by;
    T lo[NC], hi[NC];
    auto collapse = [&](unsigned bz, T (&v)[NC]) {
        const T* s = s0 + bplane * bz;
#pragma unroll
        for (int c = 0; c < NC; ++c, s += nbk)
            v[c] = wy0 * fma(wx1, __ldg(s + dx), wx0 * __ldg(s)) + wy1 * fma(wx1, __ldg(s + dy + dx), wx0 * __ldg(s + dy));
    };
    const unsigned k0 = chunk * (unsigned)depth, k1 = min(k0 + (unsigned)depth, (unsigned)d.nf[2]);
    unsigned have = ~0u;   // the bulk plane that lo holds
    T* o = out + q + (size_t)plane * k0;
    for (unsigned k = k0; k < k1; ++k, o += plane) {
        const unsigned bz = (unsigned)__ldg(d.f2b[2] + k);
        if (bz != have) {
            if (have + 1 == bz && have != ~0u)
#pragma unroll
                for (int c = 0; c < NC; ++c) lo[c] = hi[c];
            else
                collapse(bz, lo);
            collapse(bz + 1 < nbz ? bz + 1 : bz, hi);
            have = bz;
        }
        const T wz0 = __ldg(d.f2w0[2] + k), wz1 = __ldg(d.f2w1[2] + k);
#pragma unroll
        for (int c = 0; c < NC; ++c) o[c * nfn] = fma(wz1, hi[c], wz0 * lo[c]) * d.inv_Vf;
    }
}

bool finite3(const double* v) { return isfinite(v[0]) && isfinite(v[1]) && isfinite(v[2]); }

bool valid_box(const cg_box_grid& G) {
    if (!finite3(G.origin) || !finite3(G.extent)) return false;
    for (int a = 0; a < 3; ++a)
        if (!(G.extent[a] > 0.0) || G.n[a] < 1) return false;
    const long long n = (long long)G.n[0] * G.n[1] * G.n[2];
    return n <= 2147483647LL && (G.prec == CG_FP32 || G.prec == CG_FP64);
}

unsigned grid_for(long long m) { return (unsigned)std::max(1LL, std::min((m + 255) / 256, 1LL << 16)); }

}  // namespace
}  // namespace cg

using namespace cg;

extern "C" cg_status cg_map_create(const cg_box_grid* bulk, const cg_box_grid* fine, void* cuda_stream,
                                   cg_map** out) {
    if (!out) return CG_ERR_INVALID_ARG;
    *out = nullptr;
    if (!bulk || !fine || !valid_box(*bulk) || !valid_box(*fine) || bulk->prec != fine->prec) return CG_ERR_INVALID_ARG;
    cg_map* m = new (std::nothrow) cg_map();
    if (!m) return CG_ERR_OOM;
    m->bulk = *bulk;
    m->fine = *fine;
    m->fp64 = bulk->prec == CG_FP64;
    m->tsize = m->fp64 ? 8 : 4;
    m->stream = (cudaStream_t)cuda_stream;
    int dev = 0;
    if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&m->num_sms, cudaDevAttrMultiProcessorCount, dev);
    m->nbulk = (long long)bulk->n[0] * bulk->n[1] * bulk->n[2];
    m->nfine = (long long)fine->n[0] * fine->n[1] * fine->n[2];
    m->Vf = (fine->extent[0] / fine->n[0]) * (fine->extent[1] / fine->n[1]) * (fine->extent[2] / fine->n[2]);
    // host tables, then one device block: per axis, bulk rows, fine rows, covered lengths
    std::vector<int> bp[3], bi[3], fp[3], fi[3];
    std::vector<double> bw[3], fw[3], cov[3];
    for (int a = 0; a < 3; ++a) {
        axis_rows(*bulk, *fine, a, bp[a], bi[a], bw[a]);
        axis_rows(*fine, *bulk, a, fp[a], fi[a], fw[a]);
        cov[a].assign(bulk->n[a], 0.0);
        for (int i = 0; i < bulk->n[a]; ++i)
            for (int k = bp[a][i]; k < bp[a][i + 1]; ++k) cov[a][i] += bw[a][k];
    }
    std::vector<unsigned char> host;
    auto put = [&](const void* p, size_t bytes) {
        const long long off = (long long)((host.size() + 255) & ~(size_t)255);
        host.resize((size_t)off + bytes);
        if (bytes) memcpy(host.data() + off, p, bytes);
        return off;
    };
    auto put_t = [&](const std::vector<double>& v) {
        if (m->fp64) return put(v.data(), v.size() * sizeof(double));
        std::vector<float> f(v.begin(), v.end());
        return put(f.data(), f.size() * sizeof(float));
    };
    m->two = true;
    for (int a = 0; a < 3; ++a)
        for (int i = 0; i < fine->n[a]; ++i) m->two = m->two && fp[a][i + 1] - fp[a][i] <= 2;
    for (int a = 0; a < 3 && m->two; ++a) {
        std::vector<int> b0(fine->n[a], 0);
        std::vector<double> w0(fine->n[a], 0.0), w1(fine->n[a], 0.0);
        for (int i = 0; i < fine->n[a]; ++i) {
            const int k0 = fp[a][i], k1 = fp[a][i + 1];
            if (k1 > k0) {
                b0[i] = fi[a][k0];
                w0[i] = fw[a][k0];
                if (k1 - k0 == 2) w1[i] = fw[a][k0 + 1];
            }
        }
        m->off_f2b[a] = put(b0.data(), b0.size() * sizeof(int));
        m->off_f2w0[a] = put_t(w0);
        m->off_f2w1[a] = put_t(w1);
    }
    for (int a = 0; a < 3; ++a) {
        m->off_bptr[a] = put(bp[a].data(), bp[a].size() * sizeof(int));
        m->off_bidx[a] = put(bi[a].data(), bi[a].size() * sizeof(int));
        m->off_bw[a] = put_t(bw[a]);
        m->off_fptr[a] = put(fp[a].data(), fp[a].size() * sizeof(int));
        m->off_fidx[a] = put(fi[a].data(), fi[a].size() * sizeof(int));
        m->off_fw[a] = put_t(fw[a]);
        m->off_cov[a] = put_t(cov[a]);
    }
    // the widest tile of bulk x cells whose fine indices fit a block's 256 threads
    auto span = [&](int tile) {
        int most = 0;
        for (int i = 0; i < bulk->n[0]; i += tile) {
            const int p0 = bp[0][i], p1 = bp[0][std::min(i + tile, bulk->n[0])];
            if (p1 > p0) most = std::max(most, bi[0][p1 - 1] - bi[0][p0] + 1);
        }
        return most;
    };
    // (for rows that are runs of consecutive indices, one after the other, which
    // rounding could break only for cells below the resolution of their coordinates)
    bool runs = true;
    for (int a = 0; a < 3; ++a)
        for (size_t k = 1; k < bi[a].size(); ++k) {
            const int step = bi[a][k] - bi[a][k - 1];
            runs = runs && (step == 0 || step == 1);
        }
    for (int j = 0; j < bulk->n[1]; ++j) m->avg_rows = std::max(m->avg_rows, (int)(bp[1][j + 1] - bp[1][j]));
    for (int parts = 1; parts <= bulk->n[0] && runs && !m->avg_tile; ++parts) {
        const int tile = (bulk->n[0] + parts - 1) / parts, w = span(tile);
        if (w > 256) continue;
        m->avg_tile = tile;
        m->avg_threads = std::max(32, (w + 31) / 32 * 32);
    }
    if (cudaMalloc(&m->dev, std::max<size_t>(host.size(), 16)) != cudaSuccess) {
        cudaGetLastError();
        delete m;
        return CG_ERR_OOM;
    }
    if (cudaMemcpy(m->dev, host.data(), host.size(), cudaMemcpyHostToDevice) != cudaSuccess) {
        cudaGetLastError();
        cudaFree(m->dev);
        delete m;
        return CG_ERR_CUDA;
    }
    *out = m;
    return CG_OK;
}

extern "C" cg_status cg_map_destroy(cg_map* m) {
    if (!m) return CG_OK;
    if (m->stream) cudaStreamSynchronize(m->stream);
    else cudaDeviceSynchronize();
    cudaFree(m->dev);
    delete m;
    return CG_OK;
}

// The map's launches go through CG_LAUNCH's counterpart without a handle:
// a programmatic dependent launch on the map's stream.
template <typename K, typename... Args>
static cg_status map_launch(cg_map* m, K kernel, dim3 grid, int block, Args... args) {
    cudaLaunchAttribute a[1];
    a[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    a[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t c = {};
    c.gridDim = grid;
    c.blockDim = dim3((unsigned)block);
    c.stream = m->stream;
    c.attrs = a;
    c.numAttrs = 1;
    cudaError_t e = cudaLaunchKernelEx(&c, kernel, args...);
    if (e == cudaSuccess) e = cudaGetLastError();
    return e == cudaSuccess ? CG_OK : CG_ERR_CUDA;
}

// z planes per thread: as many as leave `fill` threads for each of the chip's
// (2048 per SM), since the start of a walk is work of its own; at most 64.
// Average: fill 1 102, 2 104, 4 106 us at the size above; projection: 81, 87, 78.
static int map_depth(const cg_map* m, long long columns, long long nz, int fill) {
    const long long chunks = (fill * 2048LL * m->num_sms + columns - 1) / columns;
    return (int)std::max(1LL, std::min((nz + chunks - 1) / chunks, 64LL));
}

template <typename T, int NC>
static cg_status map_apply(cg_map* m, bool avg, const void* in, void* out) {
    const MapDev<T> d = dev_view<T>(m);
    if (avg) {
        if (m->avg_tile) {
            // components per block: what shared memory holds
            constexpr int NB = NC % 3 == 0 ? 3 : NC % 2 == 0 ? 2 : 1;
            const long long tiles = (m->bulk.n[0] + m->avg_tile - 1) / m->avg_tile, rows = tiles * m->bulk.n[1];
            const int depth = map_depth(m, rows * m->avg_threads * (NC / NB), m->bulk.n[2], 1);
            const auto kernel = m->avg_rows > map_plain(sizeof(T)) ? k_map_average_rows<T, NB, true> : k_map_average_rows<T, NB, false>;
            return map_launch(m, kernel,
                              dim3((unsigned)(rows * ((m->bulk.n[2] + depth - 1) / depth)), NC / NB), m->avg_threads, d,
                              m->avg_tile, (int)tiles, depth, (const T*)in, (T*)out);
        }
        return map_launch(m, k_map_average<T, NC>, grid_for(m->nbulk), 256, d, (const T*)in, (T*)out);
    }
    if (m->two) {
        const long long columns = (long long)m->fine.n[0] * m->fine.n[1], colblk = (columns + 255) / 256;
        const int depth = map_depth(m, columns, m->fine.n[2], 4);
        return map_launch(m, k_map_project2<T, NC>, dim3((unsigned)(colblk * ((m->fine.n[2] + depth - 1) / depth))), 256, d, (unsigned)colblk,
                          depth, (const T*)in, (T*)out);
    }
    return map_launch(m, k_map_project<T, NC>, grid_for(m->nfine), 256, d, (const T*)in, (T*)out);
}

template <typename T>
static cg_status map_dispatch(cg_map* m, bool avg, int ncomp, const void* in, void* out) {
    switch (ncomp) {
        case 1: return map_apply<T, 1>(m, avg, in, out);
        case 2: return map_apply<T, 2>(m, avg, in, out);
        case 3: return map_apply<T, 3>(m, avg, in, out);
        case 4: return map_apply<T, 4>(m, avg, in, out);
        case 5: return map_apply<T, 5>(m, avg, in, out);
        case 6: return map_apply<T, 6>(m, avg, in, out);
        case 7: return map_apply<T, 7>(m, avg, in, out);
        case 8: return map_apply<T, 8>(m, avg, in, out);
    }
    return CG_ERR_INVALID_ARG;
}

static bool aligned_for(const cg_map* m, const void* p) { return ((uintptr_t)p & (m->tsize - 1)) == 0; }

extern "C" cg_status cg_map_average(cg_map* m, int32_t ncomp, const void* fine_in, void* bulk_out) {
    if (!m || ncomp < 1 || ncomp > kMapMaxComp || !fine_in || !bulk_out) return CG_ERR_INVALID_ARG;
    if (!aligned_for(m, fine_in) || !aligned_for(m, bulk_out)) return CG_ERR_INVALID_ARG;
    return m->fp64 ? map_dispatch<double>(m, true, ncomp, fine_in, bulk_out)
                   : map_dispatch<float>(m, true, ncomp, fine_in, bulk_out);
}

extern "C" cg_status cg_map_project(cg_map* m, int32_t ncomp, const void* bulk_in, void* fine_out) {
    if (!m || ncomp < 1 || ncomp > kMapMaxComp || !bulk_in || !fine_out) return CG_ERR_INVALID_ARG;
    if (!aligned_for(m, bulk_in) || !aligned_for(m, fine_out)) return CG_ERR_INVALID_ARG;
    return m->fp64 ? map_dispatch<double>(m, false, ncomp, bulk_in, fine_out)
                   : map_dispatch<float>(m, false, ncomp, bulk_in, fine_out);
}
