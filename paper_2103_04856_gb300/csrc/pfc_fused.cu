// pfc_fused.cu -- launches of the fused forward + adjoint stencil sweep
// (pfc_fused_kernel.cuh) and the small kernels around it.
#include <atomic>
#include <cstring>

#include "pfc_fused_kernel.cuh"

namespace pfc {

// ------------------------------------------------------------ small kernels

template <typename T>
__global__ void k_add_offset(T* __restrict__ out, const T* __restrict__ in, long n, const double* c)
{
    const T off = (T)(*c);
    for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x)
        out[i] = in[i] + off;
}

// Batched form: blockIdx.y selects the problem; out[i] += its offset.
struct OffsetLaunch {
    int n;
    float* out[BATCH_MAX];
    const double* c[BATCH_MAX];
    long len[BATCH_MAX];
    int vec[BATCH_MAX];      // 1: out is 16-byte aligned (float4 accesses, scalar tail)
};
__global__ void k_add_offset_batch(const __grid_constant__ OffsetLaunch L)
{
    const int k = blockIdx.y;
    const float off = (float)(*L.c[k]);
    float* out = L.out[k];
    const long n = L.len[k];
    const long t0 = blockIdx.x * (long)blockDim.x + threadIdx.x, stride = (long)gridDim.x * blockDim.x;
    long done = 0;
    if (L.vec[k]) {
        float4* o4 = reinterpret_cast<float4*>(out);
        const long n4 = n >> 2;
        for (long i = t0; i < n4; i += stride) {
            float4 v = o4[i];
            v.x += off; v.y += off; v.z += off; v.w += off;
            o4[i] = v;
        }
        done = n4 << 2;
    }
    for (long i = done + t0; i < n; i += stride) out[i] += off;
}

// The scalars of a z-slab step from every slab's FP64 sums, combined by one
// thread in rank order (so every slab given the same rows computes the same
// offset c, bit for bit).
__global__ void k_slab_finish(const double* __restrict__ rows, int nslabs, double inv_N, int mode, double* scal,
                              unsigned* ints, double* out5)
{
    if (threadIdx.x != 0 || blockIdx.x != 0) return;
    double s[NPART];
    for (int i = 0; i < NPART; ++i) s[i] = 0.0;
    for (int r = 0; r < nslabs; ++r)
        for (int i = 0; i < NPART; ++i) {
            const double x = rows[(size_t)r * SLAB_NSUMS + i];
            s[i] = i == P_GMAX ? fmax(s[i], x) : s[i] + x;
        }
    set_scalars(s, inv_N, mode, scal, ints, nullptr, 0);
    if (out5) {
        out5[0] = scal[S_E];
        out5[1] = scal[S_MASS];
        out5[2] = scal[S_LAMBDA];
        out5[3] = scal[S_GMAX];
        out5[4] = scal[S_GMEAN];
    }
}

cudaError_t launch_slab_finish(const double* rows, int nslabs, double inv_N, int mode, double* scal, unsigned* ints,
                               double* out5, cudaStream_t s)
{
    k_slab_finish<<<1, 32, 0, s>>>(rows, nslabs, inv_N, mode, scal, ints, out5);
    return cudaGetLastError();
}

// Diffuse principal curvatures (Sec. 3.1, eqs. kepsa/kepsb) of a voxel;
// at(dx, dy, dz): u at that offset.
template <typename T, class At>
__device__ __forceinline__ void voxel_curvatures(const At& at, const Coef<T>& C, T eps, T* k1, T* k2)
{
    const T u0 = at(0, 0, 0);
    const T dx = at(1, 0, 0) - at(-1, 0, 0), dy = at(0, 1, 0) - at(0, -1, 0), dz = at(0, 0, 1) - at(0, 0, -1);
    const T hxx = at(1, 0, 0) + at(-1, 0, 0) - T(2) * u0;
    const T hyy = at(0, 1, 0) + at(0, -1, 0) - T(2) * u0;
    const T hzz = at(0, 0, 1) + at(0, 0, -1) - T(2) * u0;
    const T hxy = at(1, 1, 0) - at(1, -1, 0) - at(-1, 1, 0) + at(-1, -1, 0);
    const T hxz = at(1, 0, 1) - at(1, 0, -1) - at(-1, 0, 1) + at(-1, 0, -1);
    const T hyz = at(0, 1, 1) - at(0, 1, -1) - at(0, -1, 1) + at(0, -1, -1);
    const T Gx = dx * C.sg, Gy = dy * C.sg, Gz = dz * C.sg;
    const T rho = Gx * Gx + Gy * Gy + Gz * Gz + C.xi2;
    T Mxx, Myy, Mzz, Mxy, Mxz, Myz;
    if (C.proj) {   // M = P K P, K = -eps Hess u, P = I - G G^T / rho
        const T Kxx = C.kd * hxx, Kyy = C.kd * hyy, Kzz = C.kd * hzz;
        const T Kxy = C.ko * hxy, Kxz = C.ko * hxz, Kyz = C.ko * hyz;
        const T kx = Kxx * Gx + Kxy * Gy + Kxz * Gz, ky = Kxy * Gx + Kyy * Gy + Kyz * Gz;
        const T kz = Kxz * Gx + Kyz * Gy + Kzz * Gz;
        const T s = Gx * kx + Gy * ky + Gz * kz;
        const T ir = T(1) / rho, s2 = s * ir * ir;
        Mxx = Kxx - T(2) * ir * Gx * kx + s2 * Gx * Gx;
        Myy = Kyy - T(2) * ir * Gy * ky + s2 * Gy * Gy;
        Mzz = Kzz - T(2) * ir * Gz * kz + s2 * Gz * Gz;
        Mxy = Kxy - ir * (Gx * ky + kx * Gy) + s2 * Gx * Gy;
        Mxz = Kxz - ir * (Gx * kz + kx * Gz) + s2 * Gx * Gz;
        Myz = Kyz - ir * (Gy * kz + ky * Gz) + s2 * Gy * Gz;
    } else {
        const T wp = C.well == 0 ? T(2) * u0 * (T(1) - u0) * (T(1) - T(2) * u0) : u0 * u0 * u0 - u0;
        const T wr = wp * C.inv_eps / rho;
        Mxx = C.kd * hxx + wr * Gx * Gx; Myy = C.kd * hyy + wr * Gy * Gy; Mzz = C.kd * hzz + wr * Gz * Gz;
        Mxy = C.ko * hxy + wr * Gx * Gy; Mxz = C.ko * hxz + wr * Gx * Gz; Myz = C.ko * hyz + wr * Gy * Gz;
    }
    const T Tr = Mxx + Myy + Mzz;
    const T S = Mxx * Mxx + Myy * Myy + Mzz * Mzz + T(2) * (Mxy * Mxy + Mxz * Mxz + Myz * Myz);
    const T D = T(2) * S - Tr * Tr;
    const T root = sqrt_(D > T(0) ? D : T(0));
    const T den = T(2) * eps * sqrt_(rho);
    *k1 = (Tr + root) / den;
    *k2 = (Tr - root) / den;
}

// FP32: a block of 32 x 8 columns marches up a chunk of zc planes; a thread
// keeps the 3 x 3 neighbourhood of its column on the planes z - 1, z, z + 1 in
// registers and loads that of the next plane (9 loads a voxel, from L1 but for
// its own).
// 4 B read and 8 B written a voxel; a voxel at a time in a grid-stride loop,
// with two 64-bit divisions and 19 wrapped neighbours, it took 148 us at 200^3
// (0.65 TB/s); now 71 us, bound by instruction issue (240 a voxel, a quarter of
// them the correctly rounded roots and quotients: 2-ulp ones, 61 us, move cells
// across the histogram's bin edges).  Not kept: three planes per loop trip
// without register moves (78 us) and loads one plane further ahead (103 us, 91
// registers): fewer resident warps cost more than either saves.
constexpr int kCurvX = 32, kCurvY = 8;
template <typename T>
__global__ void __launch_bounds__(kCurvX* kCurvY) k_curvatures(const T* __restrict__ u, T* __restrict__ k1,
                                                               T* __restrict__ k2, int nx, int ny, int nz,
                                                               int tiles_x, int chunks, int zc, Coef<T> C, T eps)
{
    const int t = blockIdx.x / chunks;            // block = (tile, chunk), the chunks of a tile in order
    const int x = (t % tiles_x) * kCurvX + threadIdx.x, y = (t / tiles_x) * kCurvY + threadIdx.y;
    const int z0 = (blockIdx.x - t * chunks) * zc, z1 = min(nz, z0 + zc);
    if (x >= nx || y >= ny) return;
    const size_t pls = (size_t)nx * ny;
    unsigned off[9];                              // of the 3 x 3 columns in a plane
    {
        const int xs[3] = { wrapi(x - 1, nx), x, wrapi(x + 1, nx) };
        const int ys[3] = { wrapi(y - 1, ny) * nx, y * nx, wrapi(y + 1, ny) * nx };
#pragma unroll
        for (int j = 0; j < 9; ++j) off[j] = (unsigned)(ys[j / 3] + xs[j % 3]);
    }
    T a[9], b[9], c[9];                           // planes z - 1, z, z + 1: [3 (dy + 1) + dx + 1]
    auto load = [&](int z, T w[9]) {
        const T* p = u + (size_t)z * pls;
#pragma unroll
        for (int j = 0; j < 9; ++j) w[j] = __ldg(p + off[j]);
    };
    load(wrapi(z0 - 1, nz), a);
    load(z0, b);
    T* o1 = k1 + (size_t)z0 * pls + off[4];
    T* o2 = k2 + (size_t)z0 * pls + off[4];
#pragma unroll 1
    for (int z = z0; z < z1; ++z) {
        load(z + 1 == nz ? 0 : z + 1, c);
        auto at = [&](int ddx, int ddy, int ddz) {
            const int j = 3 * (ddy + 1) + ddx + 1;
            return ddz < 0 ? a[j] : ddz > 0 ? c[j] : b[j];
        };
        voxel_curvatures<T>(at, C, eps, o1, o2);
        o1 += pls;
        o2 += pls;
#pragma unroll
        for (int j = 0; j < 9; ++j) { a[j] = b[j]; b[j] = c[j]; }
    }
}

// FP64: a voxel at a time.  Bound by the FP64 roots and quotients, so what
// counts is that every lane has a voxel and the last wave is full; the march's
// padded rows, longer blocks and chunks of eight planes made 200^3 1.54 -> 1.90
// ms, 100^3 0.20 -> 0.31 ms and 16^3 18 -> 69 us.
__global__ void __launch_bounds__(256) k_curvatures_each(const double* __restrict__ u, double* __restrict__ k1,
                                                         double* __restrict__ k2, int nx, int ny, int nz,
                                                         Coef<double> C, double eps)
{
    const long n = (long)nx * ny * nz;
    for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x) {
        const int x = (int)(i % nx), y = (int)((i / nx) % ny), z = (int)(i / ((long)nx * ny));
        auto at = [&](int dx, int dy, int dz) {
            return __ldg(u + ((long)wrapi(z + dz, nz) * ny + wrapi(y + dy, ny)) * nx + wrapi(x + dx, nx));
        };
        voxel_curvatures<double>(at, C, eps, k1 + i, k2 + i);
    }
}

// ------------------------------------------------------------ host side

template <typename T>
Coef<T> make_coef(const double a[6], double h, double eps, double xi, int well, double mu, const double* theta,
                  int proj, int refine)
{
    const double h3 = h * h * h;
    Coef<T> C;
    memset(&C, 0, sizeof C);
    C.c1 = (T)((a[0] + a[2] - a[1]) / (2.0 * eps) * h3);
    C.c2 = (T)(a[1] / (2.0 * eps) * h3);
    C.c3 = (T)((a[0] - a[2]) / (2.0 * eps) * h3);
    C.c4 = (T)((a[3] + a[4]) / 2.0 * h3);
    C.c5 = (T)((a[3] - a[4]) / 2.0 * h3);
    C.c6 = (T)(a[5] * eps * h3);
    C.c1x2 = T(2) * C.c1;
    C.c2x2 = T(2) * C.c2;
    C.c6x2 = T(2) * C.c6;
    C.kd = (T)(-eps / (h * h));
    C.ko = (T)(-eps / (4.0 * h * h));
    C.ko2 = T(2) * C.ko;
    C.sg = (T)(1.0 / (2.0 * h));
    C.inv_eps = (T)(1.0 / eps);
    C.xi = (T)xi;
    C.xi2 = (T)(xi * xi);
    C.inv_xi = (T)(1.0 / xi);
    C.well = well;
    C.R.kd = -eps / (h * h);
    C.R.ko = -eps / (4.0 * h * h);
    C.R.sg = 1.0 / (2.0 * h);
    C.R.inv_eps = 1.0 / eps;
    C.R.xi2 = xi * xi;
    auto split = [](double v, float& hi, float& lo) {
        hi = (float)v;
        lo = (float)(v - (double)hi);
    };
    split(C.R.kd, C.R.kd_h, C.R.kd_l);
    split(C.R.ko, C.R.ko_h, C.R.ko_l);
    split(C.R.sg, C.R.sg_h, C.R.sg_l);
    split(C.R.inv_eps, C.R.ie_h, C.R.ie_l);
    split(C.R.xi2, C.R.xi2_h, C.R.xi2_l);
    C.c7 = (T)(eps * mu * h3);
    C.th0 = (T)(theta ? theta[0] : 0.0);
    C.th1 = (T)(theta ? theta[1] : 0.0);
    C.th2 = (T)(theta ? theta[2] : 0.0);
    C.proj = proj ? 1 : 0;
    C.sym = (C.c3 == T(0) && C.c5 == T(0)) ? 1 : 0;
    // the refinement test is scale > rthr max(|D|, xi): 2^16 = 2^22 / 2^6, or never
    C.rthr = refine ? T(65536) : T(INFINITY);
    const double kd = C.R.kd, sg = C.R.sg, K = 1.0 / (eps * kd);
    C.wA = (T)(well == 0 ? -12.0 * K : 3.0 * K);
    C.wB = (T)(well == 0 ? 2.0 * K : -K);
    const double n[5] = { (double)C.c1 * kd * kd, (double)C.c2 * kd * kd, 0.5 * C.c4 * sg * kd, (double)C.c6 * sg * sg,
                          xi * xi / (sg * sg) };
    C.n1 = (T)n[0]; C.n2 = (T)n[1]; C.n4 = (T)n[2]; C.n6 = (T)n[3]; C.nx2 = (T)n[4];
    auto fits = [](double v) { return v == 0.0 || (fabs(v) > 1e-30 && fabs(v) < 1e30); };
    C.nform = C.sym && n[4] > 1e-30;
    for (double v : n) C.nform = C.nform && fits(v);
    // eval_sym's N is up to |K| W', its square is summed, and w up to |K| W' / nx2
    // on a flat voxel: below 1e30 for W' of order 1, with room for larger u
    C.nform = C.nform && fits(K) && fabs(K) < 1e15 && fabs(K) < 1e30 * n[4];
    return C;
}
template Coef<float> make_coef<float>(const double*, double, double, double, int, double, const double*, int, int);
template Coef<double> make_coef<double>(const double*, double, double, double, int, double, const double*, int, int);

// c(x) from a(x): the coefficients of eq. Feps (times h^3) per voxel, in FP64
// then rounded to the arithmetic type, exactly as make_coef does for a constant a.
template <typename T>
__global__ void k_coef_field(const T* __restrict__ a, T* __restrict__ c, long n, double h3, double eps)
{
    for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x) {
        const double a20 = a[i], a11 = a[n + i], a02 = a[2 * n + i];
        const double a10 = a[3 * n + i], a01 = a[4 * n + i], a00 = a[5 * n + i];
        c[i] = (T)((a20 + a02 - a11) / (2.0 * eps) * h3);
        c[n + i] = (T)(a11 / (2.0 * eps) * h3);
        c[2 * n + i] = (T)((a20 - a02) / (2.0 * eps) * h3);
        c[3 * n + i] = (T)((a10 + a01) / 2.0 * h3);
        c[4 * n + i] = (T)((a10 - a01) / 2.0 * h3);
        c[5 * n + i] = (T)(a00 * eps * h3);
    }
}

template <typename T>
cudaError_t launch_coef_field(const T* a_field, T* c_field, long n, double h, double eps, cudaStream_t s)
{
    const long b = (n + 255) / 256;
    k_coef_field<T><<<(unsigned)(b < 4096 ? b : 4096), 256, 0, s>>>(a_field, c_field, n, h * h * h, eps);
    return cudaGetLastError();
}
template cudaError_t launch_coef_field<float>(const float*, float*, long, double, double, cudaStream_t);
template cudaError_t launch_coef_field<double>(const double*, double*, long, double, double, cudaStream_t);

size_t fused_smem_bytes(int elem_size, int tile_y)
{
    const int plane = tile_y == 8 ? Tile<8>::PLANE : tile_y == 13 ? Tile<13>::PLANE : Tile<16>::PLANE;
    const int next = tile_y == 8 ? Tile<8>::NEXT : tile_y == 13 ? Tile<13>::NEXT : Tile<16>::NEXT;
    const int nt = tile_y == 8 ? Tile<8>::NT : tile_y == 13 ? Tile<13>::NT : Tile<16>::NT;
    return (size_t)elem_size * ((size_t)NBUF * plane + 2 * 5 * (size_t)next) + sizeof(float) * NPART * (size_t)nt;
}

int device_sms()
{
    static std::atomic<int> cache[64];   // 0: not queried yet
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) {
        (void)cudaGetLastError();
        dev = -1;
    }
    if (dev >= 0 && dev < 64) {
        const int c = cache[dev].load(std::memory_order_relaxed);
        if (c > 0) return c;
    }
    int n = 0;
    if (dev < 0 || cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0) {
        (void)cudaGetLastError();
        return 1;   // no device to ask: the launch that follows reports the error
    }
    if (dev < 64) cache[dev].store(n, std::memory_order_relaxed);
    return n;
}

long long fused_grid(long long units, int max_run)
{
    long long G = device_sms();                   // one CTA per SM
    if (max_run > 0 && (units + max_run - 1) / max_run > G) G = (units + max_run - 1) / max_run;
    return G < units ? G : units;
}

long long fused_units(int nx, int ny, int nz)
{
    return (long long)((nx + TX - 1) / TX) * ((ny + 7) / 8) * nz;
}

template <typename T, int TY, int EXT = 0>
static cudaError_t launch_mode(const Inst<T>& in, int mode, int max_run, cudaStream_t s)
{
    Launch<T, 1> L;
    L.n = 1;
    L.inst[0] = in;
    plan(L, TY, max_run);
    switch (mode) {
    case MODE_ENERGY: return launch_kernel<T, TY, MODE_ENERGY, EXT>(L, L.grid, s);
    case MODE_GRAD: return launch_kernel<T, TY, MODE_GRAD, EXT>(L, L.grid, s);
    case MODE_STEP: return launch_kernel<T, TY, MODE_STEP, EXT>(L, L.grid, s);
    default: return cudaErrorInvalidValue;
    }
}

template <typename T>
cudaError_t launch_fused(const Inst<T>& in, int mode, int tile_y, int max_run, cudaStream_t s)
{
    if (in.halo) return launch_fused_halo<T>(in, mode, tile_y, max_run, s);
    if (in.C.proj) return launch_mode<T, EXT_TILE_Y, 2>(in, mode, max_run, s);
    if constexpr (std::is_same<T, float>::value) {
        Launch<float, 1> L;
        L.n = 1;
        L.inst[0] = in;
        if (needs_ext(in)) return launch_pair_ext(L, mode, max_run, s);
        return in.C.nform ? launch_pair_sym<1>(L, mode, tile_y, max_run, s) : launch_pair<1>(L, mode, tile_y, max_run, s);
    } else {
        if (needs_ext(in)) return launch_mode<T, EXT_TILE_Y, 1>(in, mode, max_run, s);
        if (in.work) return launch_split(in, mode, s);
        if (tile_y == 8) return launch_mode<T, 8>(in, mode, max_run, s);
        if (tile_y == 13) return launch_mode<T, 13>(in, mode, max_run, s);
        return launch_mode<T, 16>(in, mode, max_run, s);
    }
}
template cudaError_t launch_fused<float>(const Inst<float>&, int, int, int, cudaStream_t);
template cudaError_t launch_fused<double>(const Inst<double>&, int, int, int, cudaStream_t);

// Batches of up to BATCH_MAX problems go in one launch (their descriptors
// travel as kernel parameters); larger batches take one launch per group.
// MODE_STEP (descent steps) or MODE_GRAD (energies and gradients).
cudaError_t launch_fused_batch(const Inst<float>* insts, int n_inst, int tile_y, int max_run, cudaStream_t s,
                               int mode)
{
    if (mode != MODE_STEP && mode != MODE_GRAD) return cudaErrorInvalidValue;
    thread_local Launch<float, BATCH_MAX> L;   // host staging (per thread); the launch copies it
    for (int g0 = 0; g0 < n_inst; g0 += BATCH_MAX) {
        const int cnt = n_inst - g0 < BATCH_MAX ? n_inst - g0 : BATCH_MAX;
        L.n = cnt;
        bool sym = true;
        for (int k = 0; k < cnt; ++k) {
            L.inst[k] = insts[g0 + k];
            sym = sym && L.inst[k].C.nform;
        }
        cudaError_t e = sym ? launch_pair_sym<BATCH_MAX>(L, mode, tile_y, max_run, s)
                            : launch_pair<BATCH_MAX>(L, mode, tile_y, max_run, s);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

template <typename T>
cudaError_t launch_add_offset(T* out, const T* in, long n, const double* c, cudaStream_t s)
{
    if (n <= 0) return cudaSuccess;
    long blocks = (n + 255) / 256;
    if (blocks > 16L * device_sms()) blocks = 16L * device_sms();
    k_add_offset<T><<<(int)blocks, 256, 0, s>>>(out, in, n, c);
    return cudaGetLastError();
}
template cudaError_t launch_add_offset<float>(float*, const float*, long, const double*, cudaStream_t);
template cudaError_t launch_add_offset<double>(double*, const double*, long, const double*, cudaStream_t);

cudaError_t launch_add_offset_batch(const Inst<float>* insts, int n_inst, cudaStream_t s)
{
    thread_local OffsetLaunch L;   // host staging (per thread)
    for (int g0 = 0; g0 < n_inst; g0 += BATCH_MAX) {
        const int cnt = n_inst - g0 < BATCH_MAX ? n_inst - g0 : BATCH_MAX;
        L.n = cnt;
        for (int k = 0; k < cnt; ++k) {
            const Inst<float>& in = insts[g0 + k];
            L.out[k] = in.out;
            L.c[k] = in.scal + S_C;
            L.len[k] = (long)in.nx * in.ny * in.nz;
            L.vec[k] = ((uintptr_t)in.out & 15) == 0;
        }
        int bx = (8 * device_sms() + cnt - 1) / cnt;
        if (bx < 8) bx = 8;
        k_add_offset_batch<<<dim3(bx, cnt), 256, 0, s>>>(L);
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

template <typename T>
cudaError_t launch_curvatures(const T* u, T* k1, T* k2, int nx, int ny, int nz, const Coef<T>& C, double eps,
                              cudaStream_t s)
{
    if constexpr (sizeof(T) == 8) {
        const long n = (long)nx * ny * nz, b = (n + 255) / 256, most = 16L * device_sms();
        k_curvatures_each<<<(unsigned)(b < most ? b : most), 256, 0, s>>>(u, k1, k2, nx, ny, nz, C, eps);
    } else {
        const long tiles_x = (nx + kCurvX - 1) / kCurvX, tiles = tiles_x * ((ny + kCurvY - 1) / kCurvY);
        // chunks of planes so that about 16 blocks per SM share the work, no shorter than 8 planes
        // (a chunk loads two planes more than it writes)
        int zc = nz;
        while (zc > 8 && tiles * ((nz + zc - 1) / zc) < 16L * device_sms()) zc = (zc + 1) / 2;
        const int chunks = (nz + zc - 1) / zc;
        k_curvatures<T><<<(unsigned)(tiles * chunks), dim3(kCurvX, kCurvY), 0, s>>>(u, k1, k2, nx, ny, nz, (int)tiles_x,
                                                                                   chunks, zc, C, (T)eps);
    }
    return cudaGetLastError();
}
template cudaError_t launch_curvatures<float>(const float*, float*, float*, int, int, int, const Coef<float>&,
                                              double, cudaStream_t);
template cudaError_t launch_curvatures<double>(const double*, double*, double*, int, int, int,
                                               const Coef<double>&, double, cudaStream_t);

}  // namespace pfc
