// pfc_surface.cu -- cells of the curvature diagram (Sec. 4.1, eq.
// curva_diagram): the surface {u = level} triangulated by marching
// tetrahedra, each triangle giving (area, kappa1, kappa2) with the diffuse
// curvatures (eqs. kepsa/kepsb, k_curvatures) interpolated trilinearly at
// its barycenter.
//
// Every voxel (x, y, z) owns the cube spanning to (x+1, y+1, z+1) (periodic)
// and splits it into the six tetrahedra of the Freudenthal triangulation
// (from corner 000 to corner 111 along the axes in each of the six orders,
// so neighbouring cubes agree on their shared faces).  In a tetrahedron
// with one corner on its own side of the level the surface is a triangle
// around that corner; with two on each side it is a quadrilateral, split
// into two triangles along a fixed diagonal.  Edge points interpolate
// u - level linearly.
//
// Records come out in cube order (z, y, x), then tetrahedron order, then
// triangle order, which makes the output deterministic: pass 1 counts the
// triangles of every chunk of cubes, a one-block scan turns the counts into
// offsets, pass 2 lists the chunk's triangles in shared memory and gives one
// thread to each.  A call that only asks for their number stops after pass 1.
//
// Both passes are bound by L1 and latency (22 loads per triangle), not HBM.
// The triangles of a cube come from a table over its corner mask: the
// tetrahedra worked out per thread kept two index lists in local memory and
// left most lanes of a warp idle.  4.4 million cells of a 200^3 field: count
// 87 -> 18 us (four cubes per thread from 16-byte loads), scan 31 -> 8 us,
// emit 685 -> 111 us (it took 490 us when only the number was asked for).
#include "pfc_device.cuh"

namespace pfc {

namespace {

constexpr int kSurfThreads = 256;
constexpr int kScanThreads = 1024;
constexpr int kChunk = 4 * kSurfThreads;   // cubes per chunk, four consecutive ones per thread

// The triangles of a cube by its corner mask (bit c: corner c = i + 2j + 4k is
// above the level), in tetrahedron then triangle order: three edges of 6 bits,
// each from a corner above (low 3 bits) to one below.
struct SurfTable {
    unsigned char n[256];
    unsigned tri[256][12];
};
constexpr SurfTable make_surf_table()
{
    SurfTable S{};
    const int axes[6][3] = { { 0, 1, 2 }, { 0, 2, 1 }, { 1, 0, 2 }, { 1, 2, 0 }, { 2, 0, 1 }, { 2, 1, 0 } };
    for (int m = 0; m < 256; ++m) {
        int n = 0;
        for (int t = 0; t < 6; ++t) {
            const int w[4] = { 0, 1 << axes[t][0], (1 << axes[t][0]) | (1 << axes[t][1]), 7 };
            int pos[4] = {}, neg[4] = {}, np = 0, nn = 0;
            for (int k = 0; k < 4; ++k) {
                if ((m >> w[k]) & 1) pos[np++] = w[k];
                else neg[nn++] = w[k];
            }
            auto edge = [](int a, int b) { return (unsigned)(a | (b << 3)); };
            auto add = [&](unsigned A, unsigned B, unsigned C) { S.tri[m][n++] = A | (B << 6) | (C << 12); };
            if (np == 1) add(edge(pos[0], neg[0]), edge(pos[0], neg[1]), edge(pos[0], neg[2]));
            if (np == 3) add(edge(pos[0], neg[0]), edge(pos[1], neg[0]), edge(pos[2], neg[0]));
            if (np == 2) {
                const unsigned A = edge(pos[0], neg[0]), B = edge(pos[0], neg[1]), C = edge(pos[1], neg[1]),
                               D = edge(pos[1], neg[0]);
                add(A, B, C);
                add(A, C, D);
            }
        }
        S.n[m] = (unsigned char)n;
    }
    return S;
}
__device__ const SurfTable d_surf = make_surf_table();

// A grid holds at most 2e9 voxels, so cube indices are 32-bit.  The cube of
// voxel i: corner c lies at i + (c & 1 ? dx : 0) + (c & 2 ? dy : 0) + (c & 4 ?
// dz : 0), periodic.
struct Cube {
    int i, dx, dy, dz;
    __device__ __forceinline__ Cube(int idx, int nx, int ny, int nz) : i(idx)
    {
        const int row = i / nx, z = row / ny, x = i - row * nx, y = row - z * ny, pls = nx * ny;
        dx = x + 1 == nx ? -x : 1;
        dy = y + 1 == ny ? -y * nx : nx;
        dz = z + 1 == nz ? -z * pls : pls;
    }
    __device__ __forceinline__ int at(int c) const
    {
        return i + ((c & 1) ? dx : 0) + ((c & 2) ? dy : 0) + ((c & 4) ? dz : 0);
    }
};

template <typename T>
__device__ __forceinline__ unsigned above_mask(const T* __restrict__ u, const Cube& q, T level)
{
    unsigned m = 0;
#pragma unroll
    for (int c = 0; c < 8; ++c) m |= (__ldg(u + q.at(c)) > level ? 1u : 0u) << c;
    return m;
}

// The corner masks of the cubes i0 .. i0 + 3 as four bytes (0, which has no
// triangles, past the grid's end).  VEC (nx % 4 == 0, u 16-byte aligned): the
// four share a row, whose values above the level give 5 bits for each of the
// cubes' four edges along x.
template <typename T, bool VEC>
__device__ __forceinline__ unsigned masks4(const T* __restrict__ u, long long i0, int n, int nx, int ny, int nz, T level)
{
    unsigned m = 0;
    if (i0 >= n) return 0;
    if constexpr (VEC) {
        const Cube q((int)i0, nx, ny, nz);
        const int row = q.i / nx, x = q.i - row * nx, xn = x + 4 == nx ? -x : 4;
        unsigned b[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const T* p = u + q.i + ((e & 1) ? q.dy : 0) + ((e & 2) ? q.dz : 0);
            const float4 v = *reinterpret_cast<const float4*>(p);
            b[e] = (v.x > level ? 1u : 0u) | (v.y > level ? 2u : 0u) | (v.z > level ? 4u : 0u) |
                   (v.w > level ? 8u : 0u) | (__ldg(p + xn) > level ? 16u : 0u);
        }
#pragma unroll
        for (int j = 0; j < 4; ++j)
            m |= (((b[0] >> j) & 3u) | (((b[1] >> j) & 3u) << 2) | (((b[2] >> j) & 3u) << 4) | (((b[3] >> j) & 3u) << 6)) << (8 * j);
    } else {
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if (i0 + j < n) m |= above_mask(u, Cube((int)i0 + j, nx, ny, nz), level) << (8 * j);
    }
    return m;
}
__device__ __forceinline__ unsigned count4(unsigned m)
{
    return d_surf.n[m & 255] + d_surf.n[(m >> 8) & 255] + d_surf.n[(m >> 16) & 255] + d_surf.n[m >> 24];
}

// Corner masks (4 bytes per thread, for the emit pass) and counts per chunk,
// or, with counts null, the total alone.
template <typename T, bool VEC>
__global__ void __launch_bounds__(kSurfThreads) k_surf_count(const T* __restrict__ u, int nx, int ny, int nz,
                                                             T level, int nchunks, unsigned* __restrict__ masks,
                                                             unsigned* __restrict__ counts,
                                                             unsigned long long* __restrict__ total)
{
    __shared__ unsigned sh[2][kSurfThreads / 32];
    const int n = nx * ny * nz;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    unsigned long long mine = 0;
    int par = 0;
    for (int ch = blockIdx.x; ch < nchunks; ch += gridDim.x, par ^= 1) {
        const long long quad = (long long)ch * kSurfThreads + threadIdx.x;
        const unsigned m = masks4<T, VEC>(u, 4 * quad, n, nx, ny, nz, level);
        unsigned cnt = count4(m);
        if (!counts) {
            mine += cnt;
            continue;
        }
        masks[quad] = m;
        cnt = __reduce_add_sync(0xffffffffu, cnt);
        if (lane == 0) sh[par][wid] = cnt;
        __syncthreads();
        if (threadIdx.x == 0) {
            unsigned t = 0;
#pragma unroll
            for (int w = 0; w < kSurfThreads / 32; ++w) t += sh[par][w];
            counts[ch] = t;
        }
    }
    if (counts) return;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mine += __shfl_xor_sync(0xffffffffu, mine, o);
    if (lane == 0 && mine) atomicAdd(total, mine);
}

// Exclusive scan of nb counts into offsets (one block); total at offsets[nb].
__global__ void __launch_bounds__(kScanThreads) k_surf_scan(const unsigned* __restrict__ counts, int nb,
                                                            long long* __restrict__ offsets)
{
    constexpr int V = 8;                                 // consecutive counts per thread
    __shared__ long long part[2][kScanThreads / 32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    long long base = 0;
    int par = 0;
    for (int b0 = 0; b0 < nb; b0 += V * kScanThreads, par ^= 1) {
        const int b = b0 + V * threadIdx.x;
        long long c[V], v = 0;
#pragma unroll
        for (int j = 0; j < V; ++j) {
            c[j] = v;                                    // before count j of this thread
            v += b + j < nb ? (long long)counts[b + j] : 0;
        }
        long long s = v;                                 // inclusive scan of the warp
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const long long w = __shfl_up_sync(0xffffffffu, s, o);
            if (lane >= o) s += w;
        }
        if (lane == 31) part[par][wid] = s;
        __syncthreads();
        const long long p = part[par][lane];             // 32 warps
        long long q = p;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const long long w = __shfl_up_sync(0xffffffffu, q, o);
            if (lane >= o) q += w;
        }
        const long long pre = base + __shfl_sync(0xffffffffu, q - p, wid) + s - v;
#pragma unroll
        for (int j = 0; j < V; ++j)
            if (b + j < nb) offsets[b + j] = pre + c[j];
        base += __shfl_sync(0xffffffffu, q, 31);
    }
    if (threadIdx.x == 0) offsets[nb] = base;
}

template <typename T>
__device__ __forceinline__ void edge_point(T fa, T fb, int a, int b, T q[3])
{
    const T t = fa / (fa - fb);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const T qa = (T)((a >> k) & 1), qb = (T)((b >> k) & 1);
        q[k] = qa + t * (qb - qa);
    }
}

template <typename T>
__device__ __forceinline__ void write_cell(const T P0[3], const T P1[3], const T P2[3], const T k1c[8],
                                           const T k2c[8], T h2, T* __restrict__ cell)
{
    T a[3], b[3], bc[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        a[k] = P1[k] - P0[k];
        b[k] = P2[k] - P0[k];
        bc[k] = (P0[k] + P1[k] + P2[k]) / T(3);
    }
    const T cx = a[1] * b[2] - a[2] * b[1], cy = a[2] * b[0] - a[0] * b[2], cz = a[0] * b[1] - a[1] * b[0];
    const T area = T(0.5) * sqrt_(cx * cx + cy * cy + cz * cz) * h2;
    T s1 = 0, s2 = 0;
#pragma unroll
    for (int c = 0; c < 8; ++c) {
        const T wx = (c & 1) ? bc[0] : T(1) - bc[0];
        const T wy = ((c >> 1) & 1) ? bc[1] : T(1) - bc[1];
        const T wz = ((c >> 2) & 1) ? bc[2] : T(1) - bc[2];
        const T w = wx * wy * wz;
        s1 += w * k1c[c];
        s2 += w * k2c[c];
    }
    cell[0] = area;
    cell[1] = s1;
    cell[2] = s2;
}

template <typename T>
__global__ void __launch_bounds__(kSurfThreads) k_surf_emit(const T* __restrict__ u, const T* __restrict__ k1,
                                                            const T* __restrict__ k2, int nx, int ny, int nz, T level,
                                                            T h2, int nchunks, const unsigned* __restrict__ masks,
                                                            const long long* __restrict__ offsets, long long cap,
                                                            T* __restrict__ cells)
{
    // the chunk's triangles: cube in the chunk (10 bits), triangle of the cube (4 bits)
    __shared__ unsigned short list[kChunk * 12];
    __shared__ unsigned mask[kSurfThreads];
    __shared__ unsigned sh[kSurfThreads / 32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    for (int ch = blockIdx.x; ch < nchunks; ch += gridDim.x) {
        const unsigned m = masks[(size_t)ch * kSurfThreads + threadIdx.x];
        mask[threadIdx.x] = m;
        const unsigned cnt = count4(m);
        unsigned s = cnt;                                // inclusive scan of the warp, then of the warps
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned w = __shfl_up_sync(0xffffffffu, s, o);
            if (lane >= o) s += w;
        }
        if (lane == 31) sh[wid] = s;
        __syncthreads();
        unsigned pos = s - cnt, total = 0;
#pragma unroll
        for (int w = 0; w < kSurfThreads / 32; ++w) {
            const unsigned v = sh[w];
            pos += w < wid ? v : 0;
            total += v;
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const unsigned c = d_surf.n[(m >> (8 * j)) & 255];
            for (unsigned t = 0; t < c; ++t) list[pos++] = (unsigned short)((4 * threadIdx.x + j) | (t << 10));
        }
        __syncthreads();
        const long long base = offsets[ch];
        for (unsigned q = threadIdx.x; q < total; q += kSurfThreads) {
            const long long slot = base + q;
            if (slot >= cap) break;
            const unsigned id = list[q], l = id & (kChunk - 1);
            const unsigned tri = d_surf.tri[(mask[l >> 2] >> (8 * (l & 3))) & 255][id >> 10];
            const Cube cube(ch * kChunk + (int)l, nx, ny, nz);
            T P[3][3];
#pragma unroll
            for (int e = 0; e < 3; ++e) {
                const int a = (tri >> (6 * e)) & 7, b = (tri >> (6 * e + 3)) & 7;
                edge_point(__ldg(u + cube.at(a)) - level, __ldg(u + cube.at(b)) - level, a, b, P[e]);
            }
            T k1c[8], k2c[8];
#pragma unroll
            for (int c = 0; c < 8; ++c) {
                const int o = cube.at(c);
                k1c[c] = __ldg(k1 + o);
                k2c[c] = __ldg(k2 + o);
            }
            write_cell(P[0], P[1], P[2], k1c, k2c, h2, cells + 3 * slot);
        }
        __syncthreads();                                 // the list is reused by the next chunk
    }
}

// The histogram bin of x along one axis, floor((x - lo) * inv_w) in FP64
// clamped to [0, nbins).  FP64 runs at 1/64 of the FP32 rate here, so FP32
// values are binned in FP32 first: its result stands unless the quotient is
// closer to a whole number than its rounding error (or is not finite).
__device__ __forceinline__ int hist_bin64(double x, double lo, double inv_w, int nbins)
{
    const int b = (int)floor((x - lo) * inv_w);
    return b < 0 ? 0 : (b >= nbins ? nbins - 1 : b);
}
__device__ __forceinline__ int hist_bin(double x, double lo, double inv_w, float, float, int nbins)
{
    return hist_bin64(x, lo, inv_w, nbins);
}
__device__ __forceinline__ int hist_bin(float x, double lo, double inv_w, float lof, float iwf, int nbins)
{
    const float q = (x - lof) * iwf, f = floorf(q);
    // lo, inv_w, the difference and the product are each rounded once: |error of
    // q| <= 4 * 2^-24 * (|x| + |lo|) * inv_w; 2^-20 is four times that
    const float err = 9.5367432e-07f * (fabsf(x) + fabsf(lof)) * iwf;
    if (q - f > err && f + 1.0f - q > err && fabsf(q) < 1e9f) {
        const int b = (int)f;
        return b < 0 ? 0 : (b >= nbins ? nbins - 1 : b);
    }
    return hist_bin64((double)x, lo, inv_w, nbins);
}

// Area-weighted 2-D histogram of (kappa1, kappa2) over [lo, hi)^2, values
// outside clamped into the edge bins; hist[b1 * nbins + b2] (FP64 atomics).
// Curvatures crowd into few bins, and atomics on one address queue in L2 (790
// us for 4.4 million cells in one table), so with many cells the blocks spread
// over `copies` tables (44 us), which k_hist_sum adds up (8 us).
template <typename T>
__global__ void k_curv_hist(const T* __restrict__ cells, long long n, int nbins, double lo, double inv_w, int copies,
                            double* __restrict__ hist)
{
    const float lof = (float)lo, iwf = (float)inv_w;
    double* mine = hist + (size_t)(blockIdx.x % copies) * nbins * nbins;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const T a = cells[3 * i], c1 = cells[3 * i + 1], c2 = cells[3 * i + 2];
        const int b1 = hist_bin(c1, lo, inv_w, lof, iwf, nbins), b2 = hist_bin(c2, lo, inv_w, lof, iwf, nbins);
        atomicAdd(mine + (size_t)b1 * nbins + b2, (double)a);
    }
}

// 32 bins per block, eight threads each over the copies
__global__ void __launch_bounds__(256) k_hist_sum(const double* __restrict__ part, int copies, long bins,
                                                  double* __restrict__ hist)
{
    __shared__ double sh[8][32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const long b = blockIdx.x * 32L + lane;
    double s = 0;
    if (b < bins)
        for (int c = w; c < copies; c += 8) s += part[(size_t)c * bins + b];
    sh[w][lane] = s;
    __syncthreads();
    if (w == 0 && b < bins) {
        for (int j = 1; j < 8; ++j) s += sh[j][lane];
        hist[b] = s;
    }
}

}  // namespace

long surface_blocks(long n) { return (n + kChunk - 1) / kChunk; }
long surface_work(long n) { return surface_blocks(n) * (1 + kSurfThreads); }

template <typename T>
static void surface_count(const T* u, int nx, int ny, int nz, double level, unsigned* masks, unsigned* counts,
                          long long* total, cudaStream_t s)
{
    const long nb = surface_blocks((long)nx * ny * nz);
    const unsigned grid = (unsigned)(nb < 8L * device_sms() ? nb : 8L * device_sms());
    if constexpr (sizeof(T) == 4) {
        if (nx % 4 == 0 && ((uintptr_t)u) % 16 == 0) {
            k_surf_count<T, true><<<grid, kSurfThreads, 0, s>>>(u, nx, ny, nz, (T)level, (int)nb, masks, counts,
                                                                (unsigned long long*)total);
            return;
        }
    }
    k_surf_count<T, false><<<grid, kSurfThreads, 0, s>>>(u, nx, ny, nz, (T)level, (int)nb, masks, counts,
                                                         (unsigned long long*)total);
}

template <typename T>
cudaError_t launch_surface_count(const T* u, int nx, int ny, int nz, double level, long long* total, cudaStream_t s)
{
    cudaError_t e = cudaMemsetAsync(total, 0, sizeof(long long), s);
    if (e != cudaSuccess) return e;
    surface_count<T>(u, nx, ny, nz, level, nullptr, nullptr, total, s);
    return cudaGetLastError();
}
template cudaError_t launch_surface_count<float>(const float*, int, int, int, double, long long*, cudaStream_t);
template cudaError_t launch_surface_count<double>(const double*, int, int, int, double, long long*, cudaStream_t);

template <typename T>
cudaError_t launch_surface_cells(const T* u, const T* k1, const T* k2, int nx, int ny, int nz, double h, double level,
                                 unsigned* work, long long* offsets, T* cells, long long cap, cudaStream_t s)
{
    const long nb = surface_blocks((long)nx * ny * nz);
    unsigned *counts = work, *masks = work + nb;
    const unsigned grid = (unsigned)(nb < 8L * device_sms() ? nb : 8L * device_sms());
    surface_count<T>(u, nx, ny, nz, level, masks, counts, nullptr, s);
    k_surf_scan<<<1, kScanThreads, 0, s>>>(counts, (int)nb, offsets);
    k_surf_emit<T><<<grid, kSurfThreads, 0, s>>>(u, k1, k2, nx, ny, nz, (T)level, (T)(h * h), (int)nb, masks, offsets,
                                                 cap, cells);
    return cudaGetLastError();
}
template cudaError_t launch_surface_cells<float>(const float*, const float*, const float*, int, int, int, double,
                                                 double, unsigned*, long long*, float*, long long, cudaStream_t);
template cudaError_t launch_surface_cells<double>(const double*, const double*, const double*, int, int, int, double,
                                                  double, unsigned*, long long*, double*, long long, cudaStream_t);

// Tables of the histogram: one per SM while they take no more than HIST_BYTES.  Few
// cells for the bins add into one: its atomics take about 10 ns times n / nbins
// (20 to 700 bins of smooth surfaces; noise a little less above 100 bins), and
// the tables' clearing and sum make a call 24 us instead of 16.
// 100 bins: 110 000 cells 18 us (24 in tables), 240 000 29 (25), 7.2 million 725 (69).
int histogram_copies(long long n, int nbins)
{
    if (n < 1600LL * nbins) return 1;
    const double bytes = 8.0 * nbins * nbins;
    const double c = HIST_BYTES / bytes;
    return c < 2.0 ? 1 : (c < device_sms() ? (int)c : device_sms());
}

template <typename T>
cudaError_t launch_curvature_histogram(const T* cells, long long n, int nbins, double lo, double hi, double* part,
                                       double* hist, cudaStream_t s)
{
    const long bins = (long)nbins * nbins;
    const int copies = part ? histogram_copies(n, nbins) : 1;
    double* to = copies > 1 ? part : hist;
    cudaError_t e = cudaMemsetAsync(to, 0, sizeof(double) * (size_t)bins * copies, s);
    if (e != cudaSuccess) return e;
    if (n > 0) {
        long long b = (n + 255) / 256;
        if (b > 8LL * device_sms()) b = 8LL * device_sms();
        k_curv_hist<T><<<(unsigned)b, 256, 0, s>>>(cells, n, nbins, lo, nbins / (hi - lo), copies, to);
    }
    if (copies > 1) {
        k_hist_sum<<<(unsigned)((bins + 31) / 32), 256, 0, s>>>(part, copies, bins, hist);
    }
    return cudaGetLastError();
}
template cudaError_t launch_curvature_histogram<float>(const float*, long long, int, double, double, double*,
                                                       double*, cudaStream_t);
template cudaError_t launch_curvature_histogram<double>(const double*, long long, int, double, double, double*,
                                                        double*, cudaStream_t);

}  // namespace pfc
