// Wilson dslash on FP64 and double-float fields: one warp per hop, the colour multiply in block fixed
// point on the integer pipes (dslash_fix.cuh).
//
// A block of eight warps takes 32 sites of one right-hand side at a time: warp w forms hop w (+x, -x,
// +y, ... -t) of the 32 sites, one site per lane, and leaves its 6 complex results per site in shared
// memory; then the warps share the 12 complex components of the output, sum the eight hops and store.
// Against one thread per site this has an eighth of the registers' live state and of the serial chain
// (a site's hops are loaded at once, small lattices spread over eight times the SMs), and one copy of
// the multiply in the instruction cache instead of eight (the straight-line double-float kernel was
// 14 000 instructions and stalled on instruction fetch for three quarters of its time).
//
// us per launch at 24^3 x 64 / 12 right-hand sides at 8^3 x 16 / one at 4^4: FP64 423 / 54 / 5.9 (one thread
// per site and FP64 multiply-adds: 1583 / 190 / 33), double-float 592 / 70 / 6.0 (973 / 209 / 28).  The integer
// multiply pipe is 57 %, the integer and FP64 pipes 42 % busy (FP64); half of the issue slots are used, the
// rest waits on dependent operations and the block's barriers.
//
// A block walks over bx / 32 groups of sites and `by` right-hand sides (the innermost, so that a site
// group's links are re-read from L1).  Sites that the fixed-point format does not hold send their
// block through the same steps again in the field's own arithmetic.
#include "dslash_common.cuh"

namespace ov {

namespace {

constexpr int SPLIT_THREADS = 256;

template <int SP>
struct Wide;

template <>
struct Wide<P_F64> {
    using Real = double;
    static constexpr int ESHIFT = 20;
    __device__ static __forceinline__ uint32_t range(const double h[12]) { return fix_range(h); }
    __device__ static __forceinline__ Fix fix(double x, uint32_t e) { return to_fix(x, e); }
    __device__ static __forceinline__ double real(long long v, int e) { return fix_to_f64(v, e); }
    __device__ static __forceinline__ double coef(double c, float2) { return c; }
    __device__ static __forceinline__ double flip(double c, bool neg)
    {
        return __hiloint2double(__double2hiint(c) ^ (neg ? (int)0x80000000 : 0), __double2loint(c));
    }
    __device__ static __forceinline__ void get(int4 t, double& re, double& im)
    {
        re = __hiloint2double(t.y, t.x);
        im = __hiloint2double(t.w, t.z);
    }
    __device__ static __forceinline__ int4 put(double re, double im)
    {
        return make_int4(__double2loint(re), __double2hiint(re), __double2loint(im), __double2hiint(im));
    }
};

template <>
struct Wide<P_DF64> {
    using Real = df64;
    static constexpr int ESHIFT = 23;
    __device__ static __forceinline__ uint32_t range(const df64 h[12])
    {
        float a[12], b[12];
#pragma unroll
        for (int i = 0; i < 12; ++i) {
            a[i] = h[i].hi;
            b[i] = h[i].lo;
        }
        return fixd_range(a, b);
    }
    __device__ static __forceinline__ Fix fix(df64 x, uint32_t e) { return fixd_to_fix(x.hi, x.lo, e); }
    __device__ static __forceinline__ df64 real(long long v, int e)
    {
        df64 r;
        fixd_from_fix(v, e, r.hi, r.lo);
        return r;
    }
    __device__ static __forceinline__ df64 coef(double, float2 c) { return df64(c.x, c.y); }
    __device__ static __forceinline__ df64 flip(df64 c, bool neg) { return neg ? -c : c; }
    __device__ static __forceinline__ void get(int4 t, df64& re, df64& im)
    {
        re = df64(__int_as_float(t.x), __int_as_float(t.y));
        im = df64(__int_as_float(t.z), __int_as_float(t.w));
    }
    __device__ static __forceinline__ int4 put(df64 re, df64 im)
    {
        return make_int4(__float_as_int(re.hi), __float_as_int(re.lo), __float_as_int(im.hi), __float_as_int(im.lo));
    }
};

// the projected neighbour spinor of hop w (warp-uniform) with its boundary phase
template <int SP>
__device__ __forceinline__ void load_half(const DslashArgs& A, const char* in_q, int w, int sn, bool cross,
                                          real_t<SP> h[12])
{
    using Real = real_t<SP>;
    Real v[24];
    load_spinor<SP, Real, false>(in_q, nullptr, A.g.Vh, sn, v);
    project_hop<Real>(w, v, h);
    if (cross && A.g.bc[w >> 1] != 1.0) {
        const Real f = (Real)A.g.bc[w >> 1];
#pragma unroll
        for (int i = 0; i < 12; ++i) h[i] *= f;
    }
}

// U h (forward) or U^dag h in fixed point: out[(3 a + i) * 32] = spin a, colour i.  One code for both
// directions and both spins (a quarter of the instructions to fetch, half the live registers: the link is
// read again for the second spin, from L1): the backward hop reads the link's transpose and negates its
// imaginary parts.  h is overwritten.
template <int SP>
__device__ __forceinline__ void colour_fix(const int4* lb, int Vh, bool fwd, real_t<SP> h[12], uint32_t emax, int4* out)
{
    const int m = fwd ? 0 : -1;
    const size_t si = (size_t)(fwd ? 3 : 1) * Vh, sj = (size_t)(fwd ? 1 : 3) * Vh;
#pragma unroll 1
    for (int a = 0; a < 2; ++a) {
        Fix f[6], n[3];  // n = -Im h
#pragma unroll
        for (int i = 0; i < 6; ++i) f[i] = Wide<SP>::fix(h[i], emax);
#pragma unroll
        for (int i = 0; i < 3; ++i) n[i] = fix_neg(f[2 * i + 1]);
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            FixProd re = {}, im = {};
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                const int4 t = __ldg(lb + i * si + j * sj);
                const Fix ur{t.x, t.y}, ui = fix_sign(Fix{t.z, t.w}, m);
                fix_mac(re, ur, f[2 * j]);
                fix_mac(re, ui, n[j]);
                fix_mac(im, ur, f[2 * j + 1]);
                fix_mac(im, ui, f[2 * j]);
            }
            const long long x = fix_sum(re), y = fix_sum(im);
            out[i * 32] = make_int4((int)x, (int)(x >> 32), (int)y, (int)(y >> 32));
        }
        out += 3 * 32;
#pragma unroll
        for (int i = 0; i < 6; ++i) h[i] = h[i + 6];
    }
}

// hop w of one site in the field's own arithmetic (its own call: its registers stay out of the main path)
template <int SP>
__device__ __noinline__ void hop_real(const DslashArgs& A, const char* in_q, const char* lb, int w, int sn, int ls,
                                      bool cross, int4* out)
{
    using Real = real_t<SP>;
    Real h[12], u[18], chi[12];
    load_half<SP>(A, in_q, w, sn, cross, h);
    load_link<SP, Real>(lb, A.g.Vh, ls, u);
    if ((w & 1) == 0)
        link_mul<+1, Real>(u, h, chi);
    else
        link_mul<-1, Real>(u, h, chi);
#pragma unroll
    for (int k = 0; k < 6; ++k) out[k * 32] = Wide<SP>::put(chi[2 * k], chi[2 * k + 1]);
}

template <int SP, int NY, int MINB>
__global__ void __launch_bounds__(SPLIT_THREADS, MINB) dslash_split_kernel(const __grid_constant__ DslashArgs A, int ngrp, int nby)
{
    using Real = real_t<SP>;
    using W = Wide<SP>;
    __shared__ int4 sh[8][6][32];
    __shared__ uint32_t she[8][32];
    pdl_begin();
    const Geom& g = A.g;
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const BlockWork bw = block_work((A.nrhs + nby - 1) / nby);
    const int p = bw.p, q = 1 - p;
    const size_t par_bytes = (size_t)192 * g.Vh;
    const int r1 = min(A.nrhs, (bw.grp + 1) * nby);
    for (int gi = 0; gi < ngrp; ++gi) {
        const int s_raw = (bw.sb * ngrp + gi) * 32 + lane;
        if (s_raw - lane >= g.Vh) break;
        const bool live = s_raw < g.Vh;
        const int s = live ? s_raw : g.Vh - 1;
        int c[4], sn;
        bool cross;
        cb_coords(g, s, p, c);
        hop_neighbour(g, w, s, c, sn, cross);
        const bool fwd = (w & 1) == 0;
        const int ls = fwd ? s : sn;
        const char* lb = A.gauge + (size_t)((fwd ? p : q) * 4 + (w >> 1)) * g.Vh * 144;
        pdl_wait();
        for (int r = bw.grp * nby; r < r1; ++r) {
            const char* in_q = A.in + ((size_t)r * 2 + q) * par_bytes;
            {
                Real h[12];
                load_half<SP>(A, in_q, w, sn, cross, h);
                const uint32_t e = W::range(h);
                she[w][lane] = e;
                const int4* lf = reinterpret_cast<const int4*>(lb) + ls;
                colour_fix<SP>(lf, g.Vh, fwd, h, e, &sh[w][0][lane]);
            }
            __syncthreads();
            uint32_t emax = 0, emin = FIX_BAD;
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const uint32_t e = she[k][lane];
                emax = max(emax, e);
                emin = min(emin, e - 1u);  // a vanishing hop wraps to the top
            }
            const bool bad = emax == FIX_BAD || (emax != 0 && emax - emin > ((uint32_t)FIX_HOPS << W::ESHIFT) + 1u);
            const bool redo = __syncthreads_or(bad);
            if (redo) {
                hop_real<SP>(A, in_q, lb, w, sn, ls, cross, &sh[w][0][lane]);
                __syncthreads();
            }
            // 12 complex components over 8 warps
            int d[8];  // right shift of each hop to the common unit (at most FIX_HOPS unless the block redoes)
            if (!redo) {
#pragma unroll
                for (int k = 0; k < 8; ++k) d[k] = (int)((emax - she[k][lane]) >> W::ESHIFT) & 31;
            }
            for (int k = w; k < 12; k += 8) {
                const int sp = k / 3, col = k - 3 * sp;
                Real re, im;
                if (redo) {
                    sum_hops<Real>(sp, [&](int hop, int a, Real& x, Real& y) { W::get(sh[hop][3 * a + col][lane], x, y); },
                                   re, im);
                } else {
                    long long vr, vi;
                    sum_hops<long long>(sp,
                                        [&](int hop, int a, long long& x, long long& y) {
                                            const int4 t = sh[hop][3 * a + col][lane];
                                            x = fix_sar(t.y, t.x, d[hop]);
                                            y = fix_sar(t.w, t.z, d[hop]);
                                        },
                                        vr, vi);
                    const int e = (int)(emax >> W::ESHIFT);
                    re = W::real(vr, e);
                    im = W::real(vi, e);
                }
                if (!live) continue;
                const size_t off = ((size_t)r * 2 + p) * par_bytes + ((size_t)k * g.Vh + s) * 16;
                // gamma5 on spins 2, 3: its signs on the coefficients
                const bool low = sp >= 2;
                const Real a = W::flip(W::coef(A.a, A.da), low && (A.g5_core ^ A.g5_out));
                const Real b = W::flip(W::coef(A.b, A.db), low && (A.g5_core ^ A.g5_out));
                Real xr, xi;
                W::get(ld_field<false>(reinterpret_cast<const int4*>(A.in + off)), xr, xi);
                Real o0 = a * xr + b * re, o1 = a * xi + b * im;
#pragma unroll
                for (int j = 0; j < NY; ++j) {
                    const Real sj = W::flip(W::coef(A.sy[j], A.dsy[j]), low && A.g5_out);
                    W::get(ld_field<false>(reinterpret_cast<const int4*>(A.y[j] + off)), xr, xi);
                    o0 += sj * xr;
                    o1 += sj * xi;
                }
                *reinterpret_cast<int4*>(A.out + off) = W::put(o0, o1);
            }
            __syncthreads();  // shared memory is rewritten by the next right-hand side
        }
    }
}

template <int SP, int MINB>
cudaError_t launch_ny(const DslashArgs& A, int ny, int ngrp, int by, cudaStream_t st)
{
    const dim3 grid = block_grid(A.g.Vh, 32 * ngrp, (A.nrhs + by - 1) / by);
    switch (ny) {
    case 0: return launch_kernel(dslash_split_kernel<SP, 0, MINB>, grid, dim3(SPLIT_THREADS), st, A.pdl, A, ngrp, by);
    case 1: return launch_kernel(dslash_split_kernel<SP, 1, MINB>, grid, dim3(SPLIT_THREADS), st, A.pdl, A, ngrp, by);
    case 2: return launch_kernel(dslash_split_kernel<SP, 2, MINB>, grid, dim3(SPLIT_THREADS), st, A.pdl, A, ngrp, by);
    case 3: return launch_kernel(dslash_split_kernel<SP, 3, MINB>, grid, dim3(SPLIT_THREADS), st, A.pdl, A, ngrp, by);
    }
    return cudaErrorInvalidValue;
}

template <int SP>
cudaError_t launch_var(const DslashArgs& A, int ny, int var, int ngrp, int by, cudaStream_t st)
{
    switch (var) {
    case 0: return launch_ny<SP, 2>(A, ny, ngrp, by, st);
    case 1: return launch_ny<SP, 3>(A, ny, ngrp, by, st);
    case 2: return launch_ny<SP, 4>(A, ny, ngrp, by, st);
    }
    return cudaErrorInvalidValue;
}

}  // namespace

cudaError_t launch_dslash_split(const DslashArgs& A, int sp, int gp, int ny, int var, int bx, int by, cudaStream_t st)
{
    const int ngrp = (bx + 31) / 32;
    if (sp == P_F64 && gp == P_F64) return launch_var<P_F64>(A, ny, var, ngrp, by, st);
    if (sp == P_DF64 && gp == P_DF64) return launch_var<P_DF64>(A, ny, var, ngrp, by, st);
    return cudaErrorInvalidValue;
}

}  // namespace ov
