// pfc_pair_kernel.cuh -- the FP32 fused forward + adjoint sweep, two voxels
// per thread (pfc_pair.cuh).
//
// One CTA owns an output tile of 32 x TY columns and marches up a run of z
// planes.  Warp j holds the row pair (2j - 1, 2j) of the tile, lane = x: the
// TY/2 + 1 row warps cover the tile and the halo rows -1 and TY exactly, one
// more warp holds the pairs of both halo columns.  Per plane m a thread
//   1. evaluates eq. Feps and its reverse mode for its two voxels from a ring
//      of u planes in shared memory (rows interleaved in pairs, so one 64-bit
//      load serves both voxels; the stencil values of the two planes below
//      come up the march in registers, and the y neighbour inside the pair is
//      a register too);
//   2. keeps the z parts of the transposed stencil in registers and publishes
//      four pairs of x/y pieces per plane in shared memory;
//   3. one plane later gathers the transposed stencil (the exact gradient of
//      the discrete sum) and writes g or u - tau g.
// The u planes come by 4-byte cp.async three planes ahead (each warp copies
// two of the 2 (TY/2 + 2) rows), so rows of any length and alignment take
// one path.  Warps whose rows lie past a ragged tile's halo row only copy.
//
// What bounds it: register operands and latency, not HBM (8 bytes a voxel).
// The register file gives a scheduler about two 32-bit operands per lane and
// clock, so a multiply-add of three registers takes 1.5 clocks, packed or not
// (measured 1.55 and 2.95); what packing saves is the slots and operands of
// the loads, addresses, selects and barriers, which two voxels share, and an
// evaluated halo of 24 rows for 20 instead of 20 for 16.  Twelve warps of two
// voxels (168 registers) hide less latency than twenty of one, so the square
// root's softplus is branch-free (root_softplus) and the run bookkeeping lives
// in shared memory (the general form spilled 240 bytes per thread with it in
// registers; without, a single problem's 16 to 24, a batch's 92 and the a(x)
// sweep's 104).  Tiles of 20 rows (28 for symmetric polynomials, see sym_tall): 12 and 8 rows ran 1.17 and 1.6 times longer
// on a 512^3 field.  A phase per plane on an mbarrier, waited for two planes
// later, instead of a barrier per plane was 19 % slower.
// Against the one-voxel sweep before it (32 x 16 and 32 x 13 tiles): four
// symmetric 128^3 problems 92 -> 80 us a launch, a 512^3 general step 1.82 ->
// 1.64 ms, a 256^3 general step at xi = 1e-2 0.251 -> 0.211 ms, 24 mixed
// problems 0.413 -> 0.341 ms a step, the energy of 201 x 150 x 133 voxels 112
// -> 51 us, a 150-odd^3 step with rows of no multiple of four 264 -> 163 us.
#pragma once

#include <type_traits>

#include "pfc_fused_kernel.cuh"
#include "pfc_pair.cuh"

namespace pfc {

constexpr int CBUF = 4;     // ring of coefficient planes (EXT = 2)
constexpr int CP = 44;      // pitch of their rows: columns x0-4 .. x0+35

template <int TY>
struct PairTile {
    static constexpr int NPR = TY / 2 + 1;        // pair rows
    static constexpr int NW = NPR + 1;            // warps: the pair rows, then the halo columns
    static constexpr int NT = NW * 32;
    static constexpr int UPR = NPR + 2;           // u pair rows: y0-3 .. y0+TY+2 (the first and last half empty)
    static constexpr int UP = 37;                 // pitch of a u pair row (36 columns x0-2 .. x0+33): a column of lanes
                                                  // meets distinct banks
    static constexpr int PLANE = UPR * UP;
    static constexpr int FP = 35;                 // pitch of a field pair row (34 columns and a guard column)
    static constexpr int FPL = (NPR + 2) * FP;    // one field plane, a guard row before and after
    static constexpr size_t SMEM = sizeof(F2) * ((size_t)NBUF * PLANE + 2 * 4 * FPL) + sizeof(float) * NPART * NT;
    static constexpr int CR = TY + 2;             // rows of a coefficient plane: y0-1 .. y0+TY
    static constexpr size_t CSMEM = sizeof(float) * (size_t)CBUF * NCF * CR * CP;   // EXT = 2
    static_assert(TY % 2 == 0 && 2 * NPR <= 32, "the halo columns' pairs fit one warp");
};

__device__ __forceinline__ void copy4(unsigned shared, const float* global)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(shared), "l"(global) : "memory");
}

__device__ __forceinline__ void copy16(unsigned shared, const float* global)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(shared), "l"(global) : "memory");
}

// The coefficients of one pair from its planes in shared memory (EXT = 2),
// `plane` values each; c: the pair's first voxel.
__device__ __forceinline__ void field_coefs(const float* c, int plane, Coef2& C)
{
    F2* const to[NCF] = { &C.c1, &C.c2, &C.c3, &C.c4, &C.c5, &C.c6 };
#pragma unroll
    for (int q = 0; q < NCF; ++q) *to[q] = pk(c[q * plane], c[q * plane + CP]);
    C.c6x2 = C.c6 + C.c6;
}

// Copies of a run's coefficient planes (EXT = 2): rows yc .. yc + CR - 1,
// columns x0 - 4 .. x0 + 35, periodic.  Rows of a multiple of four values go
// in 16-byte pieces, one column of pieces for all six planes per thread;
// others value by value, with the rows and columns of the u copies (rows r0
// and r0 + 1 counted from yc, columns x0 - 2 .. x0 + 33).
template <int CR>
struct FieldCopy {
    int off = -1;           // 16-byte path: this thread's piece in a plane, or -1
    unsigned dst = 0;
    __device__ __forceinline__ void init(int tid, int nx, int ny, int x0, int yc)
    {
        off = -1;
        if (nx % 4 == 0 && tid < CR * 10) {
            const int r = tid / 10, c = tid - r * 10;
            off = wrapi(yc + r, ny) * nx + wrapi(x0 - 4 + 4 * c, nx);
            dst = (unsigned)(r * CP + 4 * c) * 4;
        }
    }
    __device__ __forceinline__ void issue(unsigned cs, const float* src, size_t stride, int nx, int lane, int r0, int offa,
                                          int offb, int offc) const
    {
        if (nx % 4 == 0) {
            if (off >= 0)
#pragma unroll
                for (int q = 0; q < NCF; ++q, src += stride) copy16(cs + dst + q * (CR * CP * 4), src + off);
            return;
        }
        const bool a = r0 >= 0 && r0 < CR, b = r0 + 1 >= 0 && r0 + 1 < CR;
        const unsigned d = cs + (unsigned)(r0 * CP + 2 + lane) * 4, e = cs + (unsigned)(r0 * CP + 34 + (lane & 3)) * 4;
        for (int q = 0; q < NCF; ++q, src += stride) {
            const unsigned o = (unsigned)q * (CR * CP * 4);
            if (a) copy4(d + o, src + offa);
            if (b) copy4(d + o + CP * 4, src + offb);
            if (lane < 8 && ((lane & 4) ? b : a)) copy4(e + o + ((lane & 4) ? CP * 4 : 0), src + offc);
        }
    }
};

// A warp-uniform value, for the compiler to see as one (it then keeps what
// depends on it in uniform registers: 8 to 12 fewer per thread).
__device__ __forceinline__ int uni(int x) { return __shfl_sync(0xffffffffu, x, 0); }

// The unit whose weight range holds w (0 <= w < L.units), and its problem;
// all units for w = L.units.
template <int MAXI>
__device__ __forceinline__ long long unit_at(const Launch<float, MAXI>& L, long long w, int& k)
{
    k = 0;
    if (MAXI > 1) {
        int hi = L.n - 1;
        while (k < hi) {
            const int mid = (k + hi + 1) >> 1;
            if (L.inst[mid].wbase <= w) k = mid; else hi = mid - 1;
        }
    }
    const Inst<float>& in = L.inst[k];
    const long long rel = w - in.wbase, nfull = (long long)in.tiles_full * in.nz, wf = nfull * in.w_full;
    const bool full = rel < wf;
    const int one = full ? in.w_full : in.w_last;
    const long long r = full ? rel : rel - wf;
    return in.unit_base + (full ? 0 : nfull) + (one == 1 ? r : r / one);
}

// EXT: 1 = the orientation term of Sec. 5.2 (its weight c7 may be zero); 2 =
// the same with coefficients read per voxel from a field c(x), whose six
// planes travel through shared memory beside u's (24 more bytes a voxel-step):
// held one plane ahead in registers they would not fit.
template <int TY, int MODE, int MAXI, bool SYM, bool HALO, int EXT = 0>
__global__ void __launch_bounds__(PairTile<TY>::NT, 1) k_pair(const __grid_constant__ Launch<float, MAXI> L)
{
    using TL = PairTile<TY>;
    constexpr int NPR = TL::NPR, NT = TL::NT, UP = TL::UP, PLANE = TL::PLANE, FP = TL::FP, FPL = TL::FPL;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    F2* us = reinterpret_cast<F2*>(smem_raw);                   // [NBUF][UPR][UP]
    F2* fs = us + NBUF * PLANE;                                 // [2][4][NPR + 2][FP]
    float* scr = reinterpret_cast<float*>(fs + 2 * 4 * FPL);    // [NPART][NT]
    float* cs = scr + NPART * NT;                               // EXT = 2: [CBUF][NCF][CR][CP]
    __shared__ double tot[NPART];
    __shared__ long long st[3];                   // the CTA's next unit, the end of its units, the next problem

    const int tid = threadIdx.x;
    const int warp = tid >> 5, lane = tid & 31;
    int pj, ex;                                   // pair row and extended column of this thread
    bool active = true;
    if (warp < NPR) { pj = warp; ex = lane + 1; }
    else {   // both halo columns; lanes past them duplicate the last pair and never publish
        ex = lane < NPR ? 0 : TX + 1;
        pj = lane < NPR ? lane : (lane < 2 * NPR ? lane - NPR : NPR - 1);
        active = lane < 2 * NPR;
    }
    const int uc = (pj + 1) * UP + ex + 1;        // this pair in a u plane
    const int fc = (pj + 1) * FP + ex;            // this pair in a field plane
    // the guard rows and column of the field planes are read into values that are not output
    for (int i = tid; i < 2 * 4 * FPL; i += NT) fs[i].b = 0;

    F2 se{ 0 }, su{ 0 }, sg{ 0 }, sout{ 0 };
    float sag = 0, gmax = 0;
    auto flush = [&](const Inst<float>& pin) {
        constexpr float HS = SYM ? 2.0f : 1.0f;   // the symmetric form's sums are of half the gradient
        const float v[NPART] = { lo(se) + hi(se), lo(su) + hi(su), HS * (lo(sg) + hi(sg)), HS * sag, HS * gmax,
                                 lo(sout) + hi(sout) };
        block_sums<NT>(v, scr, tot);
        finish_problem(pin, (int)blockIdx.x - pin.first_block, MODE, tot, MAXI > 1);
        se.b = su.b = sg.b = sout.b = 0;
        sag = gmax = 0;
    };

    // both ends at once, each a chain of divisions (0.3 us of a small launch: a symmetric 16^3
    // gradient 8.96 us with one thread and a 64-bit division per weight, 8.64 so, 8.82 before tiles had weights)
    if (lane == 0 && warp < 2) {
        int k;
        st[warp] = unit_at<MAXI>(L, ((long long)blockIdx.x + warp) * L.units / L.grid, k);
        if (warp == 0) st[2] = k;
    }
    __syncthreads();
    while (st[0] < st[1]) {
    const Inst<float>& in = L.inst[MAXI > 1 ? uni((int)st[2]) : 0];
    while (st[0] < min(st[1], in.unit_base + (long long)in.tiles_x * in.tiles_y * in.nz)) {
        // ---- the run: one column tile of one problem, a contiguous z range
        const int nx = in.nx, ny = in.ny, nz = in.nz;
        int ct, z0, zend;
        {
            const long long U = st[0], rel = U - in.unit_base;
            ct = uni((int)((unsigned)rel / (unsigned)nz));   // a problem has fewer than 2^31 units
            z0 = uni((int)(rel - (long long)ct * nz));
            const long long run_end = min(st[1], in.unit_base + (long long)(ct + 1) * nz);
            zend = uni(z0 + (int)(run_end - U));   // exclusive
            __syncthreads();
            if (tid == 0) st[0] = run_end;
        }
        const int x0 = (ct % in.tiles_x) * TX, y0 = (ct / in.tiles_x) * TY;
        const int rows = min(TY, ny - y0);
        const int plast = zend + 1;                    // last u plane needed
        const size_t plane_g = (size_t)nx * ny;
        const int gx = x0 + ex - 1, gy = y0 + 2 * pj - 1;   // the pair's voxels (gx, gy) and (gx, gy + 1)
        const bool row = warp < NPR;
        const bool in0 = row && gx < nx && pj > 0 && 2 * pj - 1 < rows;
        const bool in1 = row && gx < nx && 2 * pj < rows;
        float* optr = in.out + (size_t)z0 * plane_g + (long long)gy * nx + gx;
        // batch steps: a retired instance (see k_fused) writes NaN and adds nothing
        if constexpr (MAXI > 1 && MODE == MODE_STEP) {
            if (__ldcg(&in.ints[I_NONFINITE])) {
                for (int z = z0; z < zend; ++z, optr += plane_g) {
                    if (in0) optr[0] = NAN;
                    if (in1) optr[nx] = NAN;
                }
                __syncthreads();               // st[0] is written
                continue;
            }
        }

        // ---- loads: rows y0 - 2 + 2 warp and the next, columns x0 - 2 .. x0 + 33, periodic
        int offa, offb, offc;
        {
            const int ra = wrapi(y0 - 2 + 2 * warp, ny), rb = wrapi(y0 - 1 + 2 * warp, ny);
            const int xa = wrapi(x0 - 2 + lane, nx), xc = wrapi(x0 + 30 + (lane & 3), nx);
            offa = ra * nx + xa;
            offb = rb * nx + xa;
            offc = ((lane & 4) ? rb : ra) * nx + xc;
        }
        // row 2 warp of the tile's u rows is the second half of pair row `warp`, the next the first half of the one above
        const unsigned dsta = (unsigned)__cvta_generic_to_shared(us) + (warp * UP + lane) * 8 + 4;
        const unsigned dstc = (unsigned)__cvta_generic_to_shared(us) + (warp * UP + 32 + (lane & 3)) * 8 +
                              ((lane & 4) ? UP * 8 : 4);
        int pz = wrapi(z0 - 2, nz);                    // planes are issued in increasing order
        int pc = wrapi(z0 - 3, nz);                    // the plane before
        const unsigned cso = (unsigned)__cvta_generic_to_shared(cs);
        FieldCopy<TL::CR> fcopy;
        if constexpr (EXT == 2) fcopy.init(tid, nx, ny, x0, y0 - 1);
        auto issue = [&](int p) {
            if (p <= plast) {
                const unsigned o = (unsigned)(p & (NBUF - 1)) * (PLANE * 8);
                const float* src = (HALO && (p < 0 || p >= nz)) ? in.halo + (size_t)(p < 0 ? p + 2 : p - nz + 2) * plane_g
                                                                : in.u + (size_t)pz * plane_g;
                copy4(dsta + o, src + offa);
                copy4(dsta + o + (UP * 8 - 4), src + offb);
                if (lane < 8)
                    copy4(dstc + o, src + offc);
            }
            if constexpr (EXT == 2) {   // the coefficients of plane p - 1
                if (p >= z0 && p <= zend + 1)
                    fcopy.issue(cso + (unsigned)((p - 1) & (CBUF - 1)) * (NCF * TL::CR * CP * 4),
                                in.cf + (size_t)pc * plane_g, plane_g * nz, nx, lane, 2 * warp - 1, offa, offb, offc);
                pc = pz;
            }
            cp_async_commit();   // one group per plane slot, empty past the run
            pz = pz + 1 == nz ? 0 : pz + 1;
        };

#if PFC_DEBUG
        if constexpr (EXT == 2)
            for (int i = tid; i < CBUF * NCF * TL::CR * CP; i += NT) cs[i] = NAN;
        for (int i = tid; i < NBUF * PLANE + 2 * 4 * FPL; i += NT) {
            const int f = i - NBUF * PLANE, r = f < 0 ? 1 : (f % FPL) / FP;
            if (r > 0 && r <= NPR) us[i] = dup(NAN);
        }
        __syncthreads();
#endif
        using Y = std::true_type;
        using N = std::false_type;
        for (int p = z0 - 2; p <= z0 + PD - 1; ++p) issue(p);
        // warps past the halo row of a ragged tile take part in the copies and barriers only
        if (row && 2 * pj - 1 > rows) {
            for (int m = z0 - 1; m <= zend; ++m) {
                cp_async_wait<PD - 1>();
                bar_cta();
                issue(m + 1 + PD);
            }
            bar_cta();
            cp_async_wait<0>();
            bar_cta();
            continue;
        }
        const double cind = (MODE == MODE_STEP) ? in.scal[S_C] : 0.0;
        const F2 cin = dup((float)cind);
        const Coef<float>& C = in.C;
        const Coef2 C2 = coef2(in.C);
        const F2 ntau = dup(SYM ? -2.0f * in.tau : -in.tau);
        {
            const F2 wI = pk(in0 ? 1.0f : 0.0f, in1 ? 1.0f : 0.0f);
            const F2 zero{ 0 };
            F2 accC = zero, zdn = zero, hxz2 = zero, hyz2 = zero, hxz1 = zero, hyz1 = zero;
            F2 fx1 = zero, fx2 = zero, fy1 = zero, fy2 = zero, fxy = zero, cpend = zero;
            float f2a = 0, f3b = 0;      // the y pieces the pair's voxels give each other
            F2 um_ = zero, dxm_ = zero, dym_ = zero, u0_ = zero, dx0_ = zero, dy0_ = zero, sx0_ = zero, sy0_ = zero;
            F2 umm_ = zero;

            auto gather = [&](int par) {   // from field buffer par
                const F2* F = fs + par * 4 * FPL + fc;
                const F2 x4m = F[3 * FPL - 1], x4p = F[3 * FPL + 1];
                const float* Fl = reinterpret_cast<const float*>(F);
                constexpr int DN = -2 * FP + 1, UPW = 2 * FP;       // the row below (second half), the row above (first half)
                const F2 y2 = pk(Fl[2 * 2 * FPL + DN], f2a);
                const F2 y3 = pk(f3b, Fl[2 * 2 * FPL + UPW]);
                const float* X = Fl + 3 * 2 * FPL;
                const F2 xm = pk(X[-2 + DN] - hi(x4m), lo(x4m) - X[-2 + UPW]);
                const F2 xp = pk(X[2 + DN] - hi(x4p), lo(x4p) - X[2 + UPW]);
                const F2 g5 = cpend + F[-1] + F[FPL + 1] + y2 + y3;
                const F2 g = SYM ? fma_(dup(0.5f), xm - xp, g5) : (g5 + xm) - xp;
                const float g0 = in0 ? lo(g) : 0.0f, g1 = in1 ? hi(g) : 0.0f;
                sg = sg + pk(g0, g1);
                sag += fabsf(g0) + fabsf(g1);   // a term per plane: a term per row rounds twice as often
                gmax = fmaxf(gmax, fabsf(g0));
                gmax = fmaxf(gmax, fabsf(g1));
                if (MODE == MODE_GRAD) {
                    if (in0) optr[0] = SYM ? g0 + g0 : g0;
                    if (in1) optr[nx] = SYM ? g1 + g1 : g1;
                } else {
                    const F2 u0 = umm_ + cin;
                    const F2 v = fma_(ntau, pk(g0, g1), u0);
                    if (in0) optr[0] = lo(v);
                    if (in1) optr[nx] = hi(v);
                    su = fma_(wI, u0, su);
                    sout = fma_(wI, v, sout);
                }
                optr += plane_g;
            };

            // One plane m of the march.  GATHER: write plane m-2; PUBLISH: plane
            // m-1 is complete, publish its pieces in field buffer par ((m - 1 -
            // z0) & 1); OWN: plane m is in the run (its energy counts).
            auto plane = [&](int m, int par, auto GATHER, auto PUBLISH, auto OWN, auto FIRST) {
                constexpr bool kGather = decltype(GATHER)::value, kPublish = decltype(PUBLISH)::value;
                constexpr bool kOwn = decltype(OWN)::value, kFirst = decltype(FIRST)::value;
                cp_async_wait<PD - 1>();
                bar_cta();
                if constexpr (kGather) gather(par ^ 1);
                issue(m + 1 + PD);
                const F2* p0 = us + (m & (NBUF - 1)) * PLANE + uc;
                const F2* pp = us + ((m + 1) & (NBUF - 1)) * PLANE + uc;
                constexpr int DN = -2 * UP + 1, UPW = 2 * UP;
                auto f = [](const F2* p) { return reinterpret_cast<const float*>(p); };
                auto ydiff = [&](const F2* p, F2 c, F2& d, F2& s) {
                    const float a = f(p)[DN], b = f(p)[UPW];
                    d = pk(hi(c) - a, b - lo(c));
                    s = pk(hi(c) + a, b + lo(c));
                };
                if constexpr (kFirst) {
                    const F2* q = us + ((m - 1) & (NBUF - 1)) * PLANE + uc;
                    F2 dummy;
                    um_ = q[0]; dxm_ = q[1] - q[-1];
                    ydiff(q, um_, dym_, dummy);
                    u0_ = p0[0]; dx0_ = p0[1] - p0[-1]; sx0_ = p0[1] + p0[-1];
                    ydiff(p0, u0_, dy0_, sy0_);
                }
                const F2 mtwo = dup(-2.0f);
                const F2 up = pp[0], xr = pp[1], xl = pp[-1];
                const F2 dxp = xr - xl, sxp = xr + xl;
                F2 dyp, syp;
                ydiff(pp, up, dyp, syp);
                const F2 u0 = u0_, dx = dx0_, dy = dy0_;
                const F2 dz = up - um_;
                const F2 hxx = fma_(mtwo, u0, sx0_), hyy = fma_(mtwo, u0, sy0_), hzz = fma_(mtwo, u0, up + um_);
                // x differences of the rows beside the pair
                const float dxd = f(p0)[DN + 2] - f(p0)[DN - 2], dxu = f(p0)[UPW + 2] - f(p0)[UPW - 2];
                const F2 hxy = pk(hi(dx) - dxd, dxu - lo(dx));
                const F2 hxz = dxp - dxm_, hyz = dyp - dym_;
                umm_ = um_; um_ = u0_; dxm_ = dx0_; dym_ = dy0_;
                u0_ = up; dx0_ = dxp; dy0_ = dyp; sx0_ = sxp; sy0_ = syp;
                auto refine = [&](int h) -> float {
                    const int yu = h == 0 ? 1 : 2 * UP - 1, yd = h == 0 ? -2 * UP + 1 : -1;
                    const float* pm = f(us + ((m - 1) & (NBUF - 1)) * PLANE + uc);
                    return discriminant_df_at<float>(in.C.R, C.well, pm + h, f(p0) + h, f(pp) + h, 2, yu, yd, cind);
                };
                Cot2 t;
                F2 e;
                if constexpr (SYM) e = eval_sym<true>(C, u0 + cin, dx, dy, dz, hxx, hyy, hzz, hxy, hxz, hyz, t);
                else {
                    Coef2 Cv = C2;
                    if constexpr (EXT == 2) field_coefs(cs + (m & (CBUF - 1)) * (NCF * TL::CR * CP) + 2 * pj * CP + ex + 3, TL::CR * CP, Cv);
                    e = pair_eval<true, EXT != 0>(Cv, u0 + cin, dx, dy, dz, hxx, hyy, hzz, hxy, hxz, hyz, t, refine);
                }
                if constexpr (kOwn) se = fma_(wI, e, se);
                // transposed-stencil pieces of the pair (see the gather)
                F2 X1, X2, Y1, Y2, zd, zu;
                if constexpr (SYM) {
                    X1 = t.dx + t.hxx; X2 = t.hxx - t.dx; Y1 = t.dy + t.hyy; Y2 = t.hyy - t.dy;
                    zd = t.dz + t.hzz; zu = t.hzz - t.dz;
                } else {
                    X1 = fma_(C2.sg, t.dx, t.hxx); X2 = fma_(C2.nsg, t.dx, t.hxx);
                    Y1 = fma_(C2.sg, t.dy, t.hyy); Y2 = fma_(C2.nsg, t.dy, t.hyy);
                    zd = fma_(C2.sg, t.dz, t.hzz); zu = fma_(C2.nsg, t.dz, t.hzz);
                }
                const F2 cpart = fma_(mtwo, t.hxx + t.hyy + t.hzz, t.u);
                if constexpr (kPublish) {   // plane m-1 is complete
                    cpend = accC + zu;
                    const F2 dxz = hxz2 - t.hxz, dyz = hyz2 - t.hyz;
                    F2* F = fs + par * 4 * FPL + fc;
                    const F2 half = dup(0.5f), mhalf = dup(-0.5f);
                    const F2 a2 = SYM ? fma_(half, dyz, fy1) : fy1 + dyz, a3 = SYM ? fma_(mhalf, dyz, fy2) : fy2 - dyz;
                    f2a = lo(a2);
                    f3b = hi(a3);
                    if (active) {
                        F[0] = SYM ? fma_(half, dxz, fx1) : fx1 + dxz;
                        F[FPL] = SYM ? fma_(mhalf, dxz, fx2) : fx2 - dxz;
                        F[2 * FPL] = pk(lo(a3), hi(a2));
                        F[3 * FPL] = fxy;
                    }
                }
                accC = cpart + zdn;
                zdn = zd;
                hxz2 = hxz1; hyz2 = hyz1;
                hxz1 = t.hxz; hyz1 = t.hyz;
                fx1 = X1; fx2 = X2; fy1 = Y1; fy2 = Y2; fxy = t.hxy;
            };
            plane(z0 - 1, 0, N{}, N{}, N{}, Y{});
            plane(z0, 1, N{}, N{}, Y{}, N{});
            if (zend - z0 == 1) {
                plane(z0 + 1, 0, N{}, Y{}, N{}, N{});
            } else {
                plane(z0 + 1, 0, N{}, Y{}, Y{}, N{});
                int m = z0 + 2;
#pragma unroll 1
                for (; m + 1 < zend; m += 2) { plane(m, 1, Y{}, Y{}, Y{}, N{}); plane(m + 1, 0, Y{}, Y{}, Y{}, N{}); }
                if (m < zend) {
                    plane(m, 1, Y{}, Y{}, Y{}, N{});
                    plane(zend, 0, Y{}, Y{}, N{}, N{});
                } else {
                    plane(zend, 1, Y{}, Y{}, N{}, N{});
                }
            }
            bar_cta();
            gather((zend - 1 - z0) & 1);
            cp_async_wait<0>();
            bar_cta();   // the ring and the field planes are reused by the next run
        }
    }
    if (tid == 0) ++st[2];
    flush(in);
    }
}

// The energy alone: no halo cotangents, no gather.  Warp j holds the rows
// 2j, 2j + 1 of a 32 x TY tile, lane = x; one more warp only copies.  General
// polynomials take 30 rows (16 warps of 128 registers; 24 rows: 300^3 170 ->
// 161 us, 133 x 150 x 201 50 -> 48), symmetric ones 24, which measure the same
// within 4 % either way.
template <bool SYM>
struct PairEnergyTile {
    static constexpr int TY = SYM ? 24 : 30;
    static constexpr int NPR = TY / 2, NW = NPR + 1, NT = NW * 32, UP = 37, PLANE = (NPR + 2) * UP;
    static constexpr size_t SMEM = sizeof(F2) * (size_t)NBUF * PLANE + sizeof(float) * NPART * NT;
    static constexpr int CR = TY;
    static constexpr size_t CSMEM = sizeof(float) * (size_t)CBUF * NCF * CR * CP;
};

template <bool SYM, bool HALO, int EXT = 0>
__global__ void __launch_bounds__(PairEnergyTile<SYM>::NT, 1) k_pair_energy(const __grid_constant__ Launch<float, 1> L)
{
    using TL = PairEnergyTile<SYM>;
    constexpr int PE_TY = TL::TY, NPR = TL::NPR, NT = TL::NT, UP = TL::UP, PLANE = TL::PLANE;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    F2* us = reinterpret_cast<F2*>(smem_raw);
    float* scr = reinterpret_cast<float*>(us + NBUF * PLANE);
    float* cs = scr + NPART * NT;
    __shared__ double tot[NPART];
    const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
    const Inst<float>& in = L.inst[0];
    const int nx = in.nx, ny = in.ny, nz = in.nz;
    const size_t plane_g = (size_t)nx * ny;
    const Coef<float>& C = in.C;
    const Coef2 C2 = coef2(in.C);
    F2 se{ 0 };
    const long long W = L.units;
    int k;
    long long U = unit_at<1>(L, (long long)blockIdx.x * W / L.grid, k);
    const long long Uend = unit_at<1>(L, ((long long)blockIdx.x + 1) * W / L.grid, k);
    while (U < Uend) {
        const int ct = (int)((unsigned)U / (unsigned)nz);
        const int z0 = (int)(U - (long long)ct * nz);
        const long long run_end = min(Uend, (long long)(ct + 1) * nz);
        const int zend = z0 + (int)(run_end - U);
        U = run_end;
        const int x0 = (ct % in.tiles_x) * TX, y0 = (ct / in.tiles_x) * PE_TY;
        const int rows = min(PE_TY, ny - y0);
        int offa, offb, offc;
        {
            const int ra = wrapi(y0 - 1 + 2 * warp, ny), rb = wrapi(y0 + 2 * warp, ny);
            const int xa = wrapi(x0 - 2 + lane, nx), xc = wrapi(x0 + 30 + (lane & 3), nx);
            offa = ra * nx + xa;
            offb = rb * nx + xa;
            offc = ((lane & 4) ? rb : ra) * nx + xc;
        }
        const unsigned dsta = (unsigned)__cvta_generic_to_shared(us) + (warp * UP + lane) * 8 + 4;
        const unsigned dstc = (unsigned)__cvta_generic_to_shared(us) + (warp * UP + 32 + (lane & 3)) * 8 +
                              ((lane & 4) ? UP * 8 : 4);
        int pz = wrapi(z0 - 1, nz), pc = wrapi(z0 - 2, nz);
        const unsigned cso = (unsigned)__cvta_generic_to_shared(cs);
        FieldCopy<TL::CR> fcopy;
        if constexpr (EXT == 2) fcopy.init(threadIdx.x, nx, ny, x0, y0);
        auto issue = [&](int p) {
            if (p <= zend) {
                const unsigned o = (unsigned)(p & (NBUF - 1)) * (PLANE * 8);
                const float* src = (HALO && (p < 0 || p >= nz)) ? in.halo + (size_t)(p < 0 ? p + 2 : p - nz + 2) * plane_g
                                                                : in.u + (size_t)pz * plane_g;
                copy4(dsta + o, src + offa);
                copy4(dsta + o + (UP * 8 - 4), src + offb);
                if (lane < 8)
                    copy4(dstc + o, src + offc);
            }
            if constexpr (EXT == 2) {   // the coefficients of plane p - 1
                if (p > z0 && p <= zend)
                    fcopy.issue(cso + (unsigned)((p - 1) & (CBUF - 1)) * (NCF * TL::CR * CP * 4),
                                in.cf + (size_t)pc * plane_g, plane_g * nz, nx, lane, 2 * warp - 1, offa, offb, offc);
                pc = pz;
            }
            cp_async_commit();
            pz = pz + 1 == nz ? 0 : pz + 1;
        };
#if PFC_DEBUG
        if constexpr (EXT == 2)
            for (int i = threadIdx.x; i < CBUF * NCF * TL::CR * CP; i += NT) cs[i] = NAN;
        for (int i = threadIdx.x; i < NBUF * PLANE; i += NT) us[i] = dup(NAN);
        __syncthreads();
#endif
        for (int p = z0 - 1; p <= z0 + PD; ++p) issue(p);
        const int uc = (warp + 1) * UP + lane + 2;
        const bool live = warp < NPR && 2 * warp < rows;
        const bool inx = x0 + lane < nx;
        const F2 wI = pk(inx ? 1.0f : 0.0f, inx && 2 * warp + 1 < rows ? 1.0f : 0.0f);
        F2 um_{ 0 }, dxm_{ 0 }, dym_{ 0 }, u0_{ 0 }, dx0_{ 0 }, dy0_{ 0 }, sx0_{ 0 }, sy0_{ 0 };
        constexpr int DN = -2 * UP + 1, UPW = 2 * UP;
        auto f = [](const F2* p) { return reinterpret_cast<const float*>(p); };
        auto ydiff = [&](const F2* p, F2 c, F2& d, F2& s) {
            const float a = f(p)[DN], b = f(p)[UPW];
            d = pk(hi(c) - a, b - lo(c));
            s = pk(hi(c) + a, b + lo(c));
        };
        auto plane = [&](int m, auto FIRST) {
            constexpr bool kFirst = decltype(FIRST)::value;
            cp_async_wait<PD - 1>();
            __syncthreads();
            issue(m + 1 + PD);
            if (!live) return;
            const F2* p0 = us + (m & (NBUF - 1)) * PLANE + uc;
            const F2* pp = us + ((m + 1) & (NBUF - 1)) * PLANE + uc;
            if constexpr (kFirst) {
                const F2* q = us + ((m - 1) & (NBUF - 1)) * PLANE + uc;
                F2 dummy;
                um_ = q[0]; dxm_ = q[1] - q[-1];
                ydiff(q, um_, dym_, dummy);
                u0_ = p0[0]; dx0_ = p0[1] - p0[-1]; sx0_ = p0[1] + p0[-1];
                ydiff(p0, u0_, dy0_, sy0_);
            }
            const F2 mtwo = dup(-2.0f);
            const F2 up = pp[0], xr = pp[1], xl = pp[-1];
            const F2 dxp = xr - xl, sxp = xr + xl;
            F2 dyp, syp;
            ydiff(pp, up, dyp, syp);
            const F2 u0 = u0_, dx = dx0_, dy = dy0_, dz = up - um_;
            const F2 hxx = fma_(mtwo, u0, sx0_), hyy = fma_(mtwo, u0, sy0_), hzz = fma_(mtwo, u0, up + um_);
            const float dxd = f(p0)[DN + 2] - f(p0)[DN - 2], dxu = f(p0)[UPW + 2] - f(p0)[UPW - 2];
            const F2 hxy = pk(hi(dx) - dxd, dxu - lo(dx));
            const F2 hxz = dxp - dxm_, hyz = dyp - dym_;
            um_ = u0_; dxm_ = dx0_; dym_ = dy0_;
            u0_ = up; dx0_ = dxp; dy0_ = dyp; sx0_ = sxp; sy0_ = syp;
            auto refine = [&](int h) -> float {
                const int yu = h == 0 ? 1 : 2 * UP - 1, yd = h == 0 ? -2 * UP + 1 : -1;
                const float* pm = f(us + ((m - 1) & (NBUF - 1)) * PLANE + uc);
                return discriminant_df_at<float>(in.C.R, C.well, pm + h, f(p0) + h, f(pp) + h, 2, yu, yd, 0.0);
            };
            Cot2 t;
            F2 e;
            if constexpr (SYM) e = eval_sym<false>(C, u0, dx, dy, dz, hxx, hyy, hzz, hxy, hxz, hyz, t);
            else {
                Coef2 Cv = C2;
                if constexpr (EXT == 2)
                    field_coefs(cs + (m & (CBUF - 1)) * (NCF * TL::CR * CP) + 2 * warp * CP + lane + 4, TL::CR * CP, Cv);
                e = pair_eval<false, EXT != 0>(Cv, u0, dx, dy, dz, hxx, hyy, hzz, hxy, hxz, hyz, t, refine);
            }
            se = fma_(wI, e, se);
        };
        plane(z0, std::true_type{});
        for (int m = z0 + 1; m < zend; ++m) plane(m, std::false_type{});
        cp_async_wait<0>();
        __syncthreads();
    }
    const float v[NPART] = { lo(se) + hi(se), 0.0f, 0.0f, 0.0f, 0.0f, 0.0f };
    block_sums<NT>(v, scr, tot);
    finish_problem(in, (int)blockIdx.x - in.first_block, MODE_ENERGY, tot);
}

// ------------------------------------------------------------ launches

// Split the launch's work over G CTAs by weight and record, per problem, the
// first CTA that holds a partial of it and how many do.  In a ragged last row
// of tiles the warps past its halo row do not evaluate; a plane of it weighs
// 16 (the barrier, the copies and the latencies, which it shares with a full
// one) + the warps that do, against 16 + 12 (measured on planes of 12, 20 and
// 24 rows: eight live warps of twelve take 0.86 of the time, six 0.75; weights
// in proportion to the warps made the CTAs that hold ragged planes finish
// last, a 512^3 step 27 % slower).  With few planes per CTA, or a cap on them,
// every plane weighs the same.
static inline int plane_cost(int rows, bool energy)
{
    const int r = (rows + 1) / 2;
    return 16 + (energy ? r : r + 2 - rows % 2);
}

// work units of the launch's problems in tiles of TY rows
template <int MAXI>
static long long pair_units(const Launch<float, MAXI>& L, int TY)
{
    long long units = 0;
    for (int k = 0; k < L.n; ++k) {
        const Inst<float>& in = L.inst[k];
        units += (long long)((in.nx + TX - 1) / TX) * ((in.ny + TY - 1) / TY) * in.nz;
    }
    return units;
}

template <int MAXI>
static void plan_pair(Launch<float, MAXI>& L, int TY, bool energy, int max_run)
{
    long long units = 0;
    for (int k = 0; k < L.n; ++k) {
        Inst<float>& in = L.inst[k];
        in.tiles_x = (in.nx + TX - 1) / TX;
        in.tiles_y = (in.ny + TY - 1) / TY;
        in.unit_base = units;
        units += (long long)in.tiles_x * in.tiles_y * in.nz;
    }
    const bool weigh = max_run <= 0 && units > 4LL * device_sms();
    auto cost = [&](int rows) { return plane_cost(rows, energy); };
    long long W = 0;
    for (int k = 0; k < L.n; ++k) {
        Inst<float>& in = L.inst[k];
        const int last = in.ny - (in.tiles_y - 1) * TY;
        in.w_full = weigh ? cost(TY) : 1;
        in.w_last = weigh ? cost(last) : 1;
        in.tiles_full = in.w_last == in.w_full ? in.tiles_x * in.tiles_y : in.tiles_x * (in.tiles_y - 1);
        in.wbase = W;
        W += ((long long)in.tiles_full * in.w_full + (long long)(in.tiles_x * in.tiles_y - in.tiles_full) * in.w_last) * in.nz;
    }
    const long long G = fused_grid(units, max_run);
    L.units = W;
    L.grid = (int)G;
    for (int k = 0; k < L.n; ++k) {
        Inst<float>& in = L.inst[k];
        const long long end = k + 1 < L.n ? L.inst[k + 1].wbase : W;
        // CTA b holds the unit with the weights [x, x + w) iff floor(b W / G) < x + w <= floor((b + 1) W / G)
        const int w0 = in.tiles_full ? in.w_full : in.w_last;
        in.first_block = (int)(((in.wbase + w0) * G - 1) / W);
        in.nblocks = (int)((end * G - 1) / W) - in.first_block + 1;
    }
}

// Symmetric polynomials fit 128 registers, so 16 warps and tiles of 28 rows (24
// ran 5 % slower than 20: 14 warps share four schedulers unevenly).  A plane of
// 28 rows takes 1.15 to 1.25 times what plan_pair's weights say of it against
// one of 20 (measured on eleven grids of 64 to 333 rows), a few percent less a
// row; which height is faster is then a matter of the ragged last row of tiles,
// so the weights' sums are compared.  Gradients: 128 x 112 x 128 28.6 -> 27.0 us,
// 150 x 333 x 129 79.5 -> 73.8, four 128^3 problems a step 93.8 -> 89.9; where 20
// rows fit (100, 160, 200) 28 ones took 3 to 9 % longer.
template <int MAXI>
static bool sym_tall(const Launch<float, MAXI>& L)
{
    auto column = [](int ny, int TY) {
        const int full = (ny - 1) / TY, last = ny - full * TY;
        return full * plane_cost(TY, false) + plane_cost(last, false);
    };
    double w20 = 0, w28 = 0;
    for (int k = 0; k < L.n; ++k) {
        const Inst<float>& in = L.inst[k];
        const double planes = (double)((in.nx + TX - 1) / TX) * in.nz;
        w20 += planes * column(in.ny, 20);
        w28 += planes * 1.21 * column(in.ny, 28);
    }
    return w28 < w20;
}

template <int TY, int MODE, int MAXI, bool SYM, bool HALO, int EXT = 0>
static cudaError_t launch_pair_one(Launch<float, MAXI>& L, int max_run, cudaStream_t s)
{
    plan_pair(L, TY, false, max_run);
    const size_t smem = PairTile<TY>::SMEM + (EXT == 2 ? PairTile<TY>::CSMEM : 0);
    static OncePerDevice once;
    const cudaError_t e = allow_smem(once, k_pair<TY, MODE, MAXI, SYM, HALO, EXT>, smem);
    if (e != cudaSuccess) return e;
    k_pair<TY, MODE, MAXI, SYM, HALO, EXT><<<L.grid, PairTile<TY>::NT, smem, s>>>(L);
    return cudaGetLastError();
}

template <bool SYM, bool HALO, int EXT = 0>
static cudaError_t launch_pair_energy(Launch<float, 1>& L, int max_run, cudaStream_t s)
{
    using TL = PairEnergyTile<SYM>;
    plan_pair(L, TL::TY, true, max_run);
    const size_t smem = TL::SMEM + (EXT == 2 ? TL::CSMEM : 0);
    static OncePerDevice once;
    const cudaError_t e = allow_smem(once, k_pair_energy<SYM, HALO, EXT>, smem);
    if (e != cudaSuccess) return e;
    k_pair_energy<SYM, HALO, EXT><<<L.grid, TL::NT, smem, s>>>(L);
    return cudaGetLastError();
}

// Tile rows for the height hint tile_y (pfc_problem.tile_y: 8, 13 or 16): 8 or
// 12 while there are at most four planes of 20 rows per SM, where the smaller
// tiles' shorter shares can pay (a 48^3 gradient 17.2 us in 20 rows, 14.7 in
// 12; 64^3 17.1, 17.5 and, in 8, 18.9), or where they take no more tiles and
// leave fewer warps idle (512 x 8 x 512: 54.3 us in 20 rows, 49.7 in 12).  Else they
// never did (100^3: 28.6, 31.3, 37.6 us; a symmetric 512^3: 958, 1277, 1680 us,
// where the one-voxel sweep's tiles of 13 and 8 rows had taken 1162 and 1364),
// so the hint is not followed.
template <int MAXI>
static int pair_rows(const Launch<float, MAXI>& L, int tile_y)
{
    const int rows = tile_y == 8 ? 8 : tile_y == 13 ? 12 : 20;
    const long long units = pair_units(L, 20);
    return units <= 4LL * device_sms() || units == pair_units(L, rows) ? rows : 20;
}

template <int MAXI, bool SYM, bool HALO>
static cudaError_t launch_pair_mode(Launch<float, MAXI>& L, int mode, int tile_y, int max_run, cudaStream_t s)
{
    if constexpr (MAXI == 1) {
        if (mode == MODE_ENERGY) return launch_pair_energy<SYM, HALO>(L, max_run, s);
    }
    const int rows = pair_rows(L, tile_y);
    if constexpr (SYM) {
        if (rows == 20 && sym_tall(L))
            return mode == MODE_GRAD   ? launch_pair_one<28, MODE_GRAD, MAXI, SYM, HALO>(L, max_run, s)
                   : mode == MODE_STEP ? launch_pair_one<28, MODE_STEP, MAXI, SYM, HALO>(L, max_run, s)
                                       : cudaErrorInvalidValue;
    }
    if (mode == MODE_GRAD)
        return rows == 8    ? launch_pair_one<8, MODE_GRAD, MAXI, SYM, HALO>(L, max_run, s)
               : rows == 12 ? launch_pair_one<12, MODE_GRAD, MAXI, SYM, HALO>(L, max_run, s)
                            : launch_pair_one<20, MODE_GRAD, MAXI, SYM, HALO>(L, max_run, s);
    if (mode == MODE_STEP)
        return rows == 8    ? launch_pair_one<8, MODE_STEP, MAXI, SYM, HALO>(L, max_run, s)
               : rows == 12 ? launch_pair_one<12, MODE_STEP, MAXI, SYM, HALO>(L, max_run, s)
                            : launch_pair_one<20, MODE_STEP, MAXI, SYM, HALO>(L, max_run, s);
    return cudaErrorInvalidValue;
}

// The orientation term (EXT = 1) or a coefficient field (2): 20-row tiles.
template <bool HALO, int EXT>
static cudaError_t launch_pair_ext_mode(Launch<float, 1>& L, int mode, int max_run, cudaStream_t s)
{
    switch (mode) {
    case MODE_ENERGY: return launch_pair_energy<false, HALO, EXT>(L, max_run, s);
    case MODE_GRAD: return launch_pair_one<20, MODE_GRAD, 1, false, HALO, EXT>(L, max_run, s);
    case MODE_STEP: return launch_pair_one<20, MODE_STEP, 1, false, HALO, EXT>(L, max_run, s);
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace pfc
