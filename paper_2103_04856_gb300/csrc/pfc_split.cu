// pfc_split.cu -- the FP64 energy, gradient and descent step of eq. Feps as two
// kernels: k_cot evaluates every voxel once (density, and the pieces of its
// transposed stencils, ten doubles a voxel, to memory), k_adj gathers the
// exact gradient from them and writes g or u - tau g.
//
// FP64 runs at 1/64 of the FP32 rate here (two lanes per SM and clock), so a
// step costs its FP64 operations, not its bytes: about 180 a voxel against 250
// bytes, which grids of up to 10^6 voxels or so find in L2 (80 bytes a voxel of
// it at a time); above, they come from HBM, and the operations still take
// longer.  The fused sweep (k_fused)
// evaluates the halo of its tiles again, and two planes more per run, which
// on a 32^3 grid (runs of one plane, 11 warps for 8 rows) is every voxel four
// times, and always takes the softplus's exp and log1p (about 150 operations),
// also where its weight is zero.  Here symmetric polynomials leave them out
// and every voxel is evaluated once: a 32^3 step 79 -> 22 us, 20.5 with the
// next kernel's blocks waiting on the SMs (pfc_chain.cuh).
#include "pfc_chain.cuh"
#include "pfc_pair.cuh"

namespace pfc {

namespace {

constexpr int kThreads = 128;     // a warp per scheduler: its FP64 pipes see equal shares
enum { F_C = 0, F_X1, F_X2, F_Y1, F_Y2, F_Z1, F_Z2, F_XY, F_XZ, F_YZ, NFIELD };

// Voxel i of planes of nx * ny values: its column in the plane, its plane, and
// the offsets of its periodic x and y neighbours.
struct Nbrs {
    int col, z, xm, xp, ym, yp;
    __device__ __forceinline__ Nbrs(int i, int nx, int ny)
    {
        const int row = i / nx, x = i - row * nx, pls = nx * ny;
        z = row / ny;
        const int y = row - z * ny;
        col = i - z * pls;
        xm = x == 0 ? nx - 1 : -1;
        xp = x == nx - 1 ? 1 - nx : 1;
        ym = y == 0 ? pls - nx : -nx;
        yp = y == ny - 1 ? nx - pls : nx;
    }
};

// Sums of four values over the warp: two steps halve the values a lane holds
// until one is left, which the last three add across lanes: six additions
// where four butterflies take twenty.  Lane l ends with the total of value l >> 3.
__device__ __forceinline__ double warp_sum4(const double v[4], int lane)
{
    const bool h = lane & 16;
    const double a0 = h ? v[2] : v[0], a1 = h ? v[3] : v[1];
    const double b0 = h ? v[0] : v[2], b1 = h ? v[1] : v[3];
    const double c0 = a0 + __shfl_xor_sync(0xffffffffu, b0, 16);
    const double c1 = a1 + __shfl_xor_sync(0xffffffffu, b1, 16);
    const bool q = lane & 8;
    double s = (q ? c1 : c0) + __shfl_xor_sync(0xffffffffu, q ? c0 : c1, 8);
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    return s;
}
// max of non-negative numbers by their bits, without an FP64 operation
__device__ __forceinline__ double max_pos(double a, double b)
{
    return __longlong_as_double(max(__double_as_longlong(a), __double_as_longlong(b)));
}
__device__ __forceinline__ double warp_max_pos(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = max_pos(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}
// Block totals of NPART values of one thread each (all sums but P_GMAX) into
// tot[NPART].
__device__ __forceinline__ void block_parts(const double v[NPART], double* tot)
{
    __shared__ double sh[kThreads / 32][NPART];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const double four[4] = { v[P_U], v[P_G], v[P_AG], v[P_OUT] };
    const double s = warp_sum4(four, lane);
    const double e = warp_sum(v[P_E]);
    const double m = warp_max_pos(v[P_GMAX]);
    if ((lane & 7) == 0)
        sh[wid][(lane >> 3) == 0 ? P_U : (lane >> 3) == 1 ? P_G : (lane >> 3) == 2 ? P_AG : P_OUT] = s;
    if (lane == 0) { sh[wid][P_E] = e; sh[wid][P_GMAX] = m; }
    __syncthreads();
    if (threadIdx.x < NPART) {
        double t = sh[0][threadIdx.x];
        for (int w = 1; w < kThreads / 32; ++w) {
            const double x = sh[w][threadIdx.x];
            t = threadIdx.x == P_GMAX ? max_pos(t, x) : t + x;
        }
        tot[threadIdx.x] = t;
    }
    __syncthreads();
}

// The last block of the launch to arrive (ticket) combines every block's
// partials with all its threads, in a fixed order, and sets the scalars.
__device__ __forceinline__ void finish_split(const Inst<double>& in, int mode, double* part, const double* tot)
{
    __shared__ int am_last;
    if (threadIdx.x == 0) {
#pragma unroll
        for (int i = 0; i < NPART; ++i) part[(size_t)blockIdx.x * NPART + i] = tot[i];
        __threadfence();
        am_last = atomicAdd(&in.ints[I_TICKET], 1u) == gridDim.x - 1u;
    }
    __syncthreads();
    if (!am_last) return;
    __threadfence();
    double v[NPART] = { 0, 0, 0, 0, 0, 0 };
    for (int b = threadIdx.x; b < (int)gridDim.x; b += kThreads)
#pragma unroll
        for (int i = 0; i < NPART; ++i) {
            const double x = __ldcg(part + (size_t)b * NPART + i);
            v[i] = i == P_GMAX ? max_pos(v[i], x) : v[i] + x;
        }
    __shared__ double all[NPART];
    block_parts(v, all);
    if (threadIdx.x != 0) return;
    double s[NPART];
    for (int i = 0; i < NPART; ++i) s[i] = all[i];
    if (in.sums_out) {
        for (int i = 0; i < NPART; ++i) in.sums_out[i] = s[i];
    } else {
        set_scalars(s, in.inv_N, mode, in.scal, in.ints, in.trace, in.trace_cap);
        if (in.e_host) *in.e_host = s[P_E];
    }
    __threadfence();
    in.ints[I_TICKET] = 0;
}

// The block sums of the two kernels: rows of NPART doubles after the fields.
__device__ __forceinline__ double* split_part(double* F, int n) { return F + (long)NFIELD * n; }

// Density of every voxel and, if GRAD, the pieces of its transposed stencils
// (with half the gradient's scale for SYM); block sums of the density.
// HALO (a z-slab): the n voxels are those of its planes and of one more on
// either side, whose u comes from in.halo and whose density is not counted.
template <bool SYM, bool GRAD, bool HALO>
__global__ void __launch_bounds__(kThreads) k_cot(const __grid_constant__ Inst<double> in, int n, int mode, double* __restrict__ F_)
{
    chain_wait();
    const double* __restrict__ u = after_wait(in.u);
    double* __restrict__ F = after_wait(F_);
    const double c = mode == MODE_STEP ? in.scal[S_C] : 0.0;
    const Coef<double>& C = in.C;
    const int nz = in.nz;
    const long pls = (long)in.nx * in.ny;
    double* part = split_part(F, GRAD ? n : 0);
    double se = 0;
    for (long i0 = blockIdx.x * (long)kThreads + threadIdx.x; i0 < n; i0 += (long)gridDim.x * kThreads) {
        const Nbrs b((int)i0, in.nx, in.ny);
        const int z = HALO ? b.z - 1 : b.z;
        auto at = [&](int k) {   // the voxel's place in plane k
            if (HALO) return (k < 0 ? in.halo + (k + 2) * pls : k >= nz ? in.halo + (k - nz + 2) * pls : u + k * pls) + b.col;
            return u + (k < 0 ? k + nz : k >= nz ? k - nz : k) * pls + b.col;
        };
        const double *p = at(z), *pm = at(z - 1), *pp = at(z + 1);
        const double uc = p[0], u0 = uc + c;
        const double xp = p[b.xp], xm = p[b.xm], yp = p[b.yp], ym = p[b.ym], zp = pp[0], zm = pm[0];
        const double dx = xp - xm, dy = yp - ym, dz = zp - zm;
        const double hxx = fma_(-2.0, uc, xp + xm), hyy = fma_(-2.0, uc, yp + ym), hzz = fma_(-2.0, uc, zp + zm);
        const double hxy = (p[b.xp + b.yp] - p[b.xm + b.yp]) - (p[b.xp + b.ym] - p[b.xm + b.ym]);
        const double hxz = (pp[b.xp] - pp[b.xm]) - (pm[b.xp] - pm[b.xm]);
        const double hyz = (pp[b.yp] - pp[b.ym]) - (pm[b.yp] - pm[b.ym]);
        const bool own = !HALO || (z >= 0 && z < nz);
        double e;
        CotH<double> t;
        if constexpr (SYM) {
            e = eval_sym<GRAD>(C, u0, dx, dy, dz, hxx, hyy, hzz, hxy, hxz, hyz, t);
        } else {
            Cot<double> f;
            e = voxel_eval<double, GRAD>(C, u0, dx, dy, dz, hxx, hyy, hzz, hxy, hxz, hyz, f);
            t = { f.u, f.dx, f.dy, f.dz, f.hxx, f.hyy, f.hzz, f.hxy, f.hxz, f.hyz };
        }
        if (own) se += e;
        if constexpr (GRAD) {
            double* o = F + i0;
            const size_t N = (size_t)n;
            o[F_C * N] = fma_(-2.0, t.hxx + t.hyy + t.hzz, t.u);
            o[F_X1 * N] = t.hxx + t.dx; o[F_X2 * N] = t.hxx - t.dx;
            o[F_Y1 * N] = t.hyy + t.dy; o[F_Y2 * N] = t.hyy - t.dy;
            o[F_Z1 * N] = t.hzz + t.dz; o[F_Z2 * N] = t.hzz - t.dz;
            o[F_XY * N] = t.hxy; o[F_XZ * N] = t.hxz; o[F_YZ * N] = t.hyz;
        }
    }
    __shared__ double tot[NPART];
    if (GRAD) {   // the energy's block sum alone; k_adj does the rest
        const double e = warp_sum(se);
        if ((threadIdx.x & 31) == 0) tot[threadIdx.x >> 5] = e;
        __syncthreads();
        if (threadIdx.x == 0) {
            double t = tot[0];
            for (int w = 1; w < kThreads / 32; ++w) t += tot[w];
            part[(size_t)blockIdx.x * NPART + P_E] = t;
        }
        return;
    }
    const double v[NPART] = { se, 0, 0, 0, 0, 0 };
    block_parts(v, tot);
    finish_split(in, mode, part, tot);
}

template <bool SYM, int MODE, bool HALO>
__global__ void __launch_bounds__(kThreads) k_adj(const __grid_constant__ Inst<double> in, int n, double* __restrict__ F_)
{
    chain_wait();
    double* __restrict__ F = after_wait(F_);
    const double c = MODE == MODE_STEP ? in.scal[S_C] : 0.0;
    double* part = split_part(F, n);
    double v[NPART] = { 0, 0, 0, 0, 0, 0 };
    const size_t N = (size_t)n;
    const int pls = in.nx * in.ny, own = HALO ? n - 2 * pls : n;
    for (long i0 = blockIdx.x * (long)kThreads + threadIdx.x; i0 < own; i0 += (long)gridDim.x * kThreads) {
        const Nbrs b((int)i0, in.nx, in.ny);
        const double* p = F + i0 + (HALO ? pls : 0);
        const long zm = !HALO && b.z == 0 ? (long)(in.nz - 1) * pls : -(long)pls;
        const long zp = !HALO && b.z == in.nz - 1 ? -(long)(in.nz - 1) * pls : (long)pls;
        const double s = p[F_C * N] + p[F_X1 * N + b.xm] + p[F_X2 * N + b.xp] + p[F_Y1 * N + b.ym] + p[F_Y2 * N + b.yp] +
                    (p + F_Z1 * N)[zm] + (p + F_Z2 * N)[zp];
        // a mixed difference is its own transpose
        auto mixed = [&](int f, long ap, long am, long bp, long bm) {
            const double* q = p + f * N;
            return (q[ap + bp] - q[ap + bm]) - (q[am + bp] - q[am + bm]);
        };
        const double mx = mixed(F_XY, b.xp, b.xm, b.yp, b.ym) + mixed(F_XZ, b.xp, b.xm, zp, zm) +
                     mixed(F_YZ, b.yp, b.ym, zp, zm);
        const double g = SYM ? fma_(2.0, s, mx) : s + mx;
        const double ag = fabs(g);
        v[P_G] += g;
        v[P_AG] += ag;
        v[P_GMAX] = max_pos(v[P_GMAX], ag);
        if (MODE == MODE_GRAD) {
            in.out[i0] = g;
        } else {
            const double u0 = in.u[i0] + c, w = fma_(-in.tau, g, u0);
            in.out[i0] = w;
            v[P_U] += u0;
            v[P_OUT] += w;
        }
    }
    __shared__ double tot[NPART];
    block_parts(v, tot);
    if (threadIdx.x == 0) tot[P_E] = part[(size_t)blockIdx.x * NPART + P_E];   // k_cot's block sum (the same grid)
    finish_split(in, MODE, part, tot);
}

int split_blocks(long n)
{
    const long b = (n + kThreads - 1) / kThreads, cap = 8L * device_sms();
    return (int)(b < cap ? b : cap);
}

}  // namespace

// An explicit tile height or run length asks for the fused sweep.
bool split_fits(int nx, int ny, int nz, int tile_y, int tile_z, double mu, int proj)
{
    return (double)nx * ny * nz <= (double)SPLIT_MAX && tile_y == 0 && tile_z == 0 && mu == 0.0 && !proj;
}

size_t split_work(long n) { return sizeof(double) * (size_t)(NFIELD * n + (long)NPART * split_blocks(n)); }

template <bool SYM, bool HALO>
static void split(const Inst<double>& in, int mode, cudaStream_t s)
{
    const long n = (long)in.nx * in.ny * (in.nz + (HALO ? 2 : 0));
    const int nb = split_blocks(n);
#if PFC_DEBUG
    cudaMemsetAsync(in.work, 0xff, split_work(n), s);   // NaN
    const bool chained = false;
#else
    const bool chained = in.chained != 0;
#endif
    if (mode == MODE_ENERGY) {
        launch_chained(chained, k_cot<SYM, false, HALO>, nb, kThreads, 0, s, in, (int)n, mode, in.work);
        return;
    }
    launch_chained(chained, k_cot<SYM, true, HALO>, nb, kThreads, 0, s, in, (int)n, mode, in.work);
    if (mode == MODE_GRAD) launch_chained(true, k_adj<SYM, MODE_GRAD, HALO>, nb, kThreads, 0, s, in, (int)n, in.work);
    else launch_chained(true, k_adj<SYM, MODE_STEP, HALO>, nb, kThreads, 0, s, in, (int)n, in.work);
}

cudaError_t launch_split(const Inst<double>& in, int mode, cudaStream_t s)
{
    if (in.halo) {
        if (in.C.nform) split<true, true>(in, mode, s);
        else split<false, true>(in, mode, s);
    } else {
        if (in.C.nform) split<true, false>(in, mode, s);
        else split<false, false>(in, mode, s);
    }
    return cudaGetLastError();
}

}  // namespace pfc
