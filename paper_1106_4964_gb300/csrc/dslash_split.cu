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
// us per launch at 24^3 x 64 / 12 right-hand sides at 8^3 x 16 / one at 4^4: FP64 436 / 54 / 5.8 (one thread
// per site and FP64 multiply-adds: 1583 / 190 / 33), double-float 600 / 71 / 5.8 (973 / 209 / 28).  12 right-hand
// sides at 8^3 x 16: FP64 51 % of the integer multiply pipe, 45 % of the FP64 and 37 % of the integer pipe;
// double-float 58 % of the integer pipe; half of the issue slots are used, the rest waits on dependent
// operations and the block's barriers.
//
// A block walks over bx / 32 groups of sites and `by` right-hand sides (the innermost, so that a site
// group's links are re-read from L1).  A component far below the site's scale is formed again from its own
// products (small_components); sites that the fixed-point format does not hold send their block through the
// same steps again in the field's own arithmetic (hop_real).
#include "dslash_common.cuh"

namespace ov {

namespace {

constexpr int SPLIT_THREADS = 256;

template <int SP>
struct Wide;

template <>
struct Wide<P_F64> {
    using Real = double;
    static constexpr int ESHIFT = 20, KEEP = FIX_KEEP;
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
    __device__ static __forceinline__ bool zero(int4 t) { return (((t.y | t.w) << 1) | t.x | t.z) == 0; }
    __device__ static __forceinline__ int4 put(double re, double im)
    {
        return make_int4(__double2loint(re), __double2hiint(re), __double2loint(im), __double2hiint(im));
    }
};

template <>
struct Wide<P_DF64> {
    using Real = df64;
    static constexpr int ESHIFT = 23, KEEP = FIXD_KEEP;
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
    __device__ static __forceinline__ bool zero(int4 t) { return (t.x | t.y | t.z | t.w) << 1 == 0; }
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
__device__ __noinline__ void hop_real(const DslashArgs& A, const char* in_q, int lp, int w, int sn, int ls, bool cross,
                                      int4* out)
{
    using Real = real_t<SP>;
    Real h[12], u[18], chi[12];
    load_half<SP>(A, in_q, w, sn, cross, h);
    load_link<SP, Real>(A.gauge_r + (size_t)(lp * 4 + (w >> 1)) * A.g.Vh * 144, A.g.Vh, ls, u);
    if ((w & 1) == 0)
        link_mul<+1, Real>(u, h, chi);
    else
        link_mul<-1, Real>(u, h, chi);
#pragma unroll
    for (int k = 0; k < 6; ++k) out[k * 32] = Wide<SP>::put(chi[2 * k], chi[2 * k + 1]);
}

template <int SP>
struct Cplx {
    real_t<SP> re, im;
};

// What hop w and colour j add to complex component k of the hop sum at a site of parity p, in the field's own
// arithmetic with the FP64 links.  The link entry and the spinor's two numbers are loaded first (the loads of
// several terms together), then multiplied; nothing is done when the link's entry or the spinor vanishes (finite
// fields only).  Tests are on the bits: comparisons of doubles run on the FP64 pipe
template <int SP>
struct Term {
    int sp, mu, a;  // output spin, direction, spin of the hop's result
    bool fwd, cross;
    int4 u, up, dn;

    // s: the site, sn: its neighbour along hop w
    __device__ __forceinline__ void load(const DslashArgs& A, const char* in_q, int p, int s, int sn, bool crossing, int k,
                                         int w, int j)
    {
        const int Vh = A.g.Vh;
        sp = k / 3;
        const int col = k - 3 * sp, b = sp & 1;
        mu = w >> 1;
        fwd = (w & 1) == 0;
        cross = crossing;
        a = sp < 2 || mu >= 2 ? b : 1 - b;              // (sum_hops)
        const int ad = 2 + (mu < 2 ? 1 - a : a);        // lower spin in its half spinor (project)
        const int4* lb = reinterpret_cast<const int4*>(A.gauge_r) + (size_t)((fwd ? p : 1 - p) * 4 + mu) * Vh * 9;
        const int4* v = reinterpret_cast<const int4*>(in_q) + sn;
        u = __ldg(lb + (size_t)(fwd ? 3 * col + j : 3 * j + col) * Vh + (fwd ? s : sn));
        up = ld_field<false>(v + (size_t)(3 * a + j) * Vh);
        dn = ld_field<false>(v + (size_t)(3 * ad + j) * Vh);
    }
    // t += the term
    __device__ __forceinline__ void add_to(const DslashArgs& A, Cplx<SP>& t) const
    {
        using Real = real_t<SP>;
        using W = Wide<SP>;
        if (Wide<P_F64>::zero(u) || (W::zero(up) && W::zero(dn))) return;
        const bool turn = mu == 0 || mu == 2;
        Real hr, hi, dr, di;
        double ux, uy;
        W::get(up, hr, hi);
        W::get(dn, dr, di);
        Wide<P_F64>::get(u, ux, uy);
        // (A_mu d)_a: -i d1, -i d0 | -d1, d0 | -i d0, i d1 | d0, d1; h = up - S (A_mu d)_a
        const bool add = ((mu == 1 && a == 0) || (mu == 2 && a == 1)) == fwd;
        hr += W::flip(turn ? di : dr, !add);
        hi += W::flip(turn ? -dr : di, !add);
        if (cross && A.g.bc[mu] != 1.0) {
            const Real f = (Real)A.g.bc[mu];
            hr *= f;
            hi *= f;
        }
        if (sp >= 2) {  // -S A_mu^dag chi (sum_hops): chi, or i chi, with a sign
            const bool neg = fwd != ((mu == 1 || mu == 2) && (sp & 1));
            const Real x = turn ? -hi : hr, y = turn ? hr : hi;
            hr = W::flip(x, neg);
            hi = W::flip(y, neg);
        }
        const Real ur = (Real)ux, ui = (Real)(fwd ? uy : -uy);
        t.re = fmac<Real>(ur, hr, t.re);
        t.im = fmac<Real>(ur, hi, t.im);
        t.re = fmac<Real>(-ui, hi, t.re);
        t.im = fmac<Real>(ui, hr, t.im);
    }
};

// The component as the sum of its 24 terms by one lane
template <int SP>
__device__ __forceinline__ Cplx<SP> component_lane(const DslashArgs& A, const char* in_q, int p, int s, int k)
{
    int c[4];
    cb_coords(A.g, s, p, c);
    Cplx<SP> sum{real_t<SP>(0), real_t<SP>(0)};
#pragma unroll 1
    for (int w = 0; w < 8; ++w) {
        int sn;
        bool cross;
        hop_neighbour(A.g, w, s, c, sn, cross);
        Term<SP> x[3];
#pragma unroll
        for (int j = 0; j < 3; ++j) x[j].load(A, in_q, p, s, sn, cross, k, w, j);
#pragma unroll
        for (int j = 0; j < 3; ++j) x[j].add_to(A, sum);
    }
    return sum;
}

template <int SP>
__device__ __forceinline__ real_t<SP> shfl_xor(real_t<SP> x, int m)
{
    if constexpr (SP == P_DF64)
        return df64(__shfl_xor_sync(~0u, x.hi, m), __shfl_xor_sync(~0u, x.lo, m));
    else
        return __shfl_xor_sync(~0u, x, m);
}

// component k (hop sum re, im) of site s: epilogue and store
template <int SP, int NY>
__device__ __forceinline__ void store_component(const DslashArgs& A, int r, int p, int s, int k, real_t<SP> re,
                                                real_t<SP> im)
{
    using Real = real_t<SP>;
    using W = Wide<SP>;
    const size_t off = ((size_t)r * 2 + p) * 192 * A.g.Vh + ((size_t)k * A.g.Vh + s) * 16;
    // gamma5 on spins 2, 3: its signs on the coefficients
    const bool low = k >= 6;
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

// Components w and w + 8 of the lanes of need0 and need1, which the main path has not stored (its own call: its
// registers stay out of the main path).  Where many lanes need it, each takes its own site; else four sites at a
// time, eight lanes each, a lane the three terms of one hop.  us per FP64 launch for 12 sources at 8^4, Gaussian fields
// (no such component) / a propagator's columns (one in a few hundred): 30.9 / 36.6; a term per lane and one site at a
// time 30.4 / 40.6.  24^3 x 64, unit links, one filled colour: 1037, without the lanes' own form 2283.
template <int SP, int NY>
__device__ __noinline__ void small_components(const DslashArgs& A, const char* in_q, int r, int p, int s, int w,
                                              unsigned need0, unsigned need1)
{
    const int lane = threadIdx.x & 31, hop = lane & 7;
    for (int k = w; k < 12; k += 8) {
        unsigned need = k < 8 ? need0 : need1;
        if (__popc(need) > 8) {
            if (need >> lane & 1) {
                const Cplx<SP> t = component_lane<SP>(A, in_q, p, s, k);
                store_component<SP, NY>(A, r, p, s, k, t.re, t.im);
            }
            continue;
        }
        while (need) {
            unsigned mine = need;  // the lowest set lane that is left to these eight lanes
            for (int i = lane >> 3; i; --i) mine &= mine - 1;
            const int sm = __shfl_sync(~0u, s, mine ? __ffs((int)mine) - 1 : 0);
            Cplx<SP> t{real_t<SP>(0), real_t<SP>(0)};
            if (mine) {
                int c[4], sn;
                bool cross;
                cb_coords(A.g, sm, p, c);
                hop_neighbour(A.g, hop, sm, c, sn, cross);
                Term<SP> x[3];
#pragma unroll
                for (int j = 0; j < 3; ++j) x[j].load(A, in_q, p, sm, sn, cross, k, hop, j);
#pragma unroll
                for (int j = 0; j < 3; ++j) x[j].add_to(A, t);
            }
#pragma unroll
            for (int m = 4; m; m >>= 1) {
                t.re += shfl_xor<SP>(t.re, m);
                t.im += shfl_xor<SP>(t.im, m);
            }
            if (mine && hop == 0) store_component<SP, NY>(A, r, p, sm, k, t.re, t.im);
#pragma unroll
            for (int i = 0; i < 4; ++i) need &= need - 1;
        }
    }
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
            uint32_t emax = 0;
#pragma unroll
            for (int k = 0; k < 8; ++k) emax = max(emax, she[k][lane]);
            const bool redo = __syncthreads_or(emax == FIX_BAD);
            if (redo) {
                hop_real<SP>(A, in_q, fwd ? p : q, w, sn, ls, cross, &sh[w][0][lane]);
                __syncthreads();
            }
            // 12 complex components over 8 warps
            uint32_t d[8];  // right shift of each hop to the common unit
#pragma unroll
            for (int k = 0; k < 8; ++k) d[k] = (emax - she[k][lane]) >> W::ESHIFT;
            unsigned need0 = 0, need1 = 0;  // lanes whose component w, w + 8 has to be formed again
            for (int k = w; k < 12; k += 8) {
                const int sp = k / 3, col = k - 3 * sp;
                Real re, im;
                bool store = live;
                if (redo) {
                    sum_hops<Real>(sp, [&](int hop, int a, Real& x, Real& y) { W::get(sh[hop][3 * a + col][lane], x, y); },
                                   re, im);
                } else {
                    long long vr, vi;
                    sum_hops<long long>(sp,
                                        [&](int hop, int a, long long& x, long long& y) {
                                            const int4 t = sh[hop][3 * a + col][lane];
                                            x = fix_sar(((long long)t.y << 32) | (uint32_t)t.x, d[hop]);
                                            y = fix_sar(((long long)t.w << 32) | (uint32_t)t.z, d[hop]);
                                        },
                                        vr, vi);
                    const int e = (int)(emax >> W::ESHIFT);
                    re = W::real(vr, e);
                    im = W::real(vi, e);
                    bool small = fix_small(vr, vi, W::KEEP) && emax != 0 && live;
                    if (small) {  // unless by cancellation between the hops, which floating point rounds as well
#pragma unroll 1
                        for (int hop = 0; hop < 8 && small; ++hop) {
                            const int4 t = sh[hop][3 * (sp < 2 || hop >= 4 ? sp & 1 : 1 - (sp & 1)) + col][lane];
                            const uint32_t n = (emax - she[hop][lane]) >> W::ESHIFT;
                            small = fix_small(fix_sar((long long)t.y << 32, n), fix_sar((long long)t.w << 32, n), W::KEEP);
                        }
                    }
                    const unsigned need = __ballot_sync(~0u, small);
                    if (k < 8)
                        need0 = need;
                    else
                        need1 = need;
                    store = live && !small;
                }
                if (store) store_component<SP, NY>(A, r, p, s, k, re, im);
            }
            if (need0 | need1) small_components<SP, NY>(A, in_q, r, p, s, w, need0, need1);
            __syncthreads();  // shared memory is rewritten by the next right-hand side
        }
    }
}

template <int SP, int MINB>
cudaError_t launch_ny(const DslashArgs& A, int ny, int ngrp, int by, cudaStream_t st)
{
    const dim3 grid = block_grid(A.g.Vh, 32 * ngrp, (A.nrhs + by - 1) / by);
    switch (ny) {
    case 0: return launch_kernel(dslash_split_kernel<SP, 0, MINB>, grid, dim3(SPLIT_THREADS), st, A.pdl, PDL_SPLIT, A, ngrp, by);
    case 1: return launch_kernel(dslash_split_kernel<SP, 1, MINB>, grid, dim3(SPLIT_THREADS), st, A.pdl, PDL_SPLIT, A, ngrp, by);
    case 2: return launch_kernel(dslash_split_kernel<SP, 2, MINB>, grid, dim3(SPLIT_THREADS), st, A.pdl, PDL_SPLIT, A, ngrp, by);
    case 3: return launch_kernel(dslash_split_kernel<SP, 3, MINB>, grid, dim3(SPLIT_THREADS), st, A.pdl, PDL_SPLIT, A, ngrp, by);
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
