// Learned gauge-covariant preconditioner (no counterpart in the paper).
//
// Layer (channels cin -> cout):
//   y_c(n) = sum_{c'} sum_{p=0..8} W[p][c][c'] (T_p x_{c'})(n)
// with T_0 = 1, T_{1+2mu} x(n) = U_mu(n) x(n+mu), T_{2+2mu} x(n) = U_mu(n-mu)^dag x(n-mu)
// (boundary phases applied) and W[p][c][c'] a complex 4x4 spin matrix.  The
// map is linear and commutes with gauge transformations.  The network is
// M = L2 . L1 with 1 -> 16 -> 1 channels, applied to batches of right-hand sides in FP32 (internal
// even/odd layout; the activations of a batch of nb are a field of 16 nb right-hand sides).
//
// Backward pass: the adjoint of T_p is T_{pbar} (forward <-> backward hop),
// so the input gradient is the forward kernel with weights
// W'[q][c'][c] = W[qbar][c][c']^dag; the weight gradient
// gW[p][c][c'] = sum_n gy_c(n) (T_p x_{c'}(n))^dag (summed over colour) is a
// product over sites and colours with block partials summed in fixed order.
// Training: loss sum_k |M(r_k) - e_k|^2 / |e_k|^2 over (residual, error)
// pairs recorded at the FP64 true-residual points of the library's own
// deflated CG solves, Adam on the device.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "ctx.h"

namespace ov {

constexpr int NET_C = 16;              // hidden channels
constexpr int NET_W = 9 * NET_C * 16;  // complex weights per layer (9 paths x 16 ch x 4x4 spin)
constexpr int NET_PARAMS = 2 * NET_W;  // complex parameters of the network
constexpr int NET_MAXPAIRS = 256;

struct NetState {
    int trained = 0;
    float2* W = nullptr;     // layer 1 [9][16][1][16] then layer 2 [9][1][16][16]
    float2* Wadj = nullptr;  // adjoint weights, same layout per layer with channels swapped
    float2* G = nullptr;     // gradient
    float* adam = nullptr;   // first moments [2*NET_PARAMS] then second moments
    float2* partials = nullptr;
    size_t partials_n = 0;
    int adam_t = 0;
    int adj_valid = 0;  // Wadj matches W
    int batch = 0;      // fields the work fields hold
    int batch_max = 16; // fields the device had room for
    // recorded training pairs: residuals and iterates (then errors), f32 single-rhs fields
    int recording = 0;
    FieldDesc pr{}, px{};
    int npairs = 0, cap = 0;
    std::vector<double> history;  // mean loss per pair before each Adam step of the last training
};

namespace {

// t = (T_path x)(site s of parity p, coordinates c); x: one FP32 field, both parities
__device__ __forceinline__ void transport(const Geom& g, const char* gauge, const char* x, int p, int s, const int c[4],
                                          int path, float t[24])
{
    const size_t par = (size_t)6 * 16 * g.Vh;
    if (path == 0) {
        load_spinor<P_F32, float>(x + p * par, nullptr, g.Vh, s, t);
        return;
    }
    int sn;
    float ph = 1.f;
    switch (path) {
    case 1: sn = cb_neighbour<0>(g, s, c); if (c[0] + 1 == g.L[0]) ph = g.fbc[0]; break;
    case 2: sn = cb_neighbour<1>(g, s, c); if (c[0] == 0) ph = g.fbc[0]; break;
    case 3: sn = cb_neighbour<2>(g, s, c); if (c[1] + 1 == g.L[1]) ph = g.fbc[1]; break;
    case 4: sn = cb_neighbour<3>(g, s, c); if (c[1] == 0) ph = g.fbc[1]; break;
    case 5: sn = cb_neighbour<4>(g, s, c); if (c[2] + 1 == g.L[2]) ph = g.fbc[2]; break;
    case 6: sn = cb_neighbour<5>(g, s, c); if (c[2] == 0) ph = g.fbc[2]; break;
    case 7: sn = cb_neighbour<6>(g, s, c); if (c[3] + 1 == g.L[3]) ph = g.fbc[3]; break;
    default: sn = cb_neighbour<7>(g, s, c); if (c[3] == 0) ph = g.fbc[3]; break;
    }
    const int mu = (path - 1) >> 1;
    const bool fwd = (path & 1) != 0;
    float v[24], u[18];
    load_spinor<P_F32, float>(x + (1 - p) * par, nullptr, g.Vh, sn, v);
    load_link<P_F32, float>(gauge + ((size_t)((fwd ? p : 1 - p) * 4 + mu) * g.Vh) * 48, g.Vh, fwd ? s : sn, u);
    if (!fwd) {  // U^dag
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            u[2 * (4 * i) + 1] = -u[2 * (4 * i) + 1];
#pragma unroll
            for (int j = i + 1; j < 3; ++j) {
                const float ar = u[2 * (3 * i + j)], ai = u[2 * (3 * i + j) + 1];
                u[2 * (3 * i + j)] = u[2 * (3 * j + i)];
                u[2 * (3 * i + j) + 1] = -u[2 * (3 * j + i) + 1];
                u[2 * (3 * j + i)] = ar;
                u[2 * (3 * j + i) + 1] = -ai;
            }
        }
    }
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            float re = 0, im = 0;
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                const float ur = u[2 * (3 * i + j)], ui = u[2 * (3 * i + j) + 1];
                const float xr = v[2 * (3 * q + j)], xi = v[2 * (3 * q + j) + 1];
                re = fmaf(ur, xr, re);
                im = fmaf(ur, xi, im);
                re = fmaf(-ui, xi, re);
                im = fmaf(ui, xr, im);
            }
            t[2 * (3 * q + i)] = ph * re;
            t[2 * (3 * q + i) + 1] = ph * im;
        }
}

// acc += w t: a complex 4 x 4 spin matrix (two weights per float4) on a spinor
__device__ __forceinline__ void spin_mix(const float4 w[8], const float t[24], float acc[24])
{
#pragma unroll
    for (int sa = 0; sa < 4; ++sa)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const float4 w2 = w[2 * sa + h];
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                const float wr = q ? w2.z : w2.x, wi = q ? w2.w : w2.y;
                const int sb = 2 * h + q;
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    const float tr = t[2 * (3 * sb + a)], ti = t[2 * (3 * sb + a) + 1];
                    float& re = acc[2 * (3 * sa + a)];
                    float& im = acc[2 * (3 * sa + a) + 1];
                    re = fmaf(wr, tr, re);
                    im = fmaf(wr, ti, im);
                    re = fmaf(-wi, ti, re);
                    im = fmaf(wi, tr, im);
                }
            }
        }
}

// All kernels take a batch of fields (training pairs, right-hand sides): blockIdx.z, or the site index of
// the weight gradients, runs over it.  One launch per pair left the 8^3 x 16 lattice with 7 warps per SM:
// a gradient over 8 pairs took 3.77 ms in 90 launches, of which the one-block sums of the weight
// gradients' partials were 1.6 ms; batched, with one spinor transported per path, 0.75 ms.  The FP32
// multiply-adds (150 000 per site and pair) are 0.27 ms of that.
constexpr int NET_CG = 4;  // output channels per thread of the 1 -> 16 layer

// 1 -> 16 layer: thread per (site, 4 output channels); each transported spinor feeds 4 x 192 multiply-adds
__global__ void __launch_bounds__(128, 3) net_many_kernel(Geom g, const char* gauge, const char* x, char* y,
                                                       const float2* __restrict__ Wg)
{
    __shared__ float4 W[9][NET_CG][8];  // two complex weights each
    const int grp = blockIdx.y;
    for (int k = threadIdx.x; k < 9 * NET_CG * 16; k += blockDim.x) {
        const int path = k / (NET_CG * 16), e = k % (NET_CG * 16);
        reinterpret_cast<float2*>(W)[k] = Wg[(path * NET_C + grp * NET_CG) * 16 + e];
    }
    __syncthreads();
    const int idx = blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= 2 * g.Vh) return;
    const int p = idx >= g.Vh, s = idx - p * g.Vh;
    int c[4];
    cb_coords(g, s, p, c);
    const size_t par = (size_t)6 * 16 * g.Vh, chan = 2 * par;  // bytes of one parity and of one FP32 field
    x += blockIdx.z * chan;
    float acc[NET_CG][24];
#pragma unroll
    for (int j = 0; j < NET_CG; ++j)
#pragma unroll
        for (int k = 0; k < 24; ++k) acc[j][k] = 0.f;
    for (int path = 0; path < 9; ++path) {
        float t[24];
        transport(g, gauge, x, p, s, c, path, t);
#pragma unroll
        for (int j = 0; j < NET_CG; ++j) spin_mix(W[path][j], t, acc[j]);
    }
#pragma unroll
    for (int j = 0; j < NET_CG; ++j)
        store_spinor<P_F32, float>(y + ((size_t)blockIdx.z * NET_C + grp * NET_CG + j) * chan + p * par, nullptr, g.Vh, s,
                                   acc[j]);
}

// 16 -> 1 layer, first half: the spin matrices commute with the transport, so the 16 channels are mixed
// where they lie, z_p(n) = sum_c W[p][c] x_c(n) (thread per site and three paths), and one spinor per path
// is transported instead of 16 (net_gather_kernel)
__global__ void __launch_bounds__(128, 4) net_mix_kernel(Geom g, const char* x, char* z, const float2* __restrict__ Wg)
{
    __shared__ float4 W[3][NET_C][8];
    const int p0 = blockIdx.y * 3;
    for (int k = threadIdx.x; k < 3 * NET_C * 16; k += blockDim.x)
        reinterpret_cast<float2*>(W)[k] = Wg[p0 * NET_C * 16 + k];
    __syncthreads();
    const int idx = blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= 2 * g.Vh) return;
    const int p = idx >= g.Vh, s = idx - p * g.Vh;
    const size_t par = (size_t)6 * 16 * g.Vh, chan = 2 * par;
    x += (size_t)blockIdx.z * NET_C * chan + p * par;
    float acc[3][24];
#pragma unroll
    for (int j = 0; j < 3; ++j)
#pragma unroll
        for (int k = 0; k < 24; ++k) acc[j][k] = 0.f;
    for (int ci = 0; ci < NET_C; ++ci) {
        float v[24];
        load_spinor<P_F32, float>(x + ci * chan, nullptr, g.Vh, s, v);
#pragma unroll
        for (int j = 0; j < 3; ++j) spin_mix(W[j][ci], v, acc[j]);
    }
#pragma unroll
    for (int j = 0; j < 3; ++j)
        store_spinor<P_F32, float>(z + ((size_t)blockIdx.z * 9 + p0 + j) * chan + p * par, nullptr, g.Vh, s, acc[j]);
}

// second half: y(n) = sum_p (T_p z_p)(n)
__global__ void __launch_bounds__(128) net_gather_kernel(Geom g, const char* gauge, const char* z, char* y)
{
    const int idx = blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= 2 * g.Vh) return;
    const int p = idx >= g.Vh, s = idx - p * g.Vh;
    int c[4];
    cb_coords(g, s, p, c);
    const size_t par = (size_t)6 * 16 * g.Vh, chan = 2 * par;
    float acc[24];
#pragma unroll
    for (int k = 0; k < 24; ++k) acc[k] = 0.f;
    for (int path = 0; path < 9; ++path) {
        float t[24];
        transport(g, gauge, z + ((size_t)blockIdx.z * 9 + path) * chan, p, s, c, path, t);
#pragma unroll
        for (int k = 0; k < 24; ++k) acc[k] += t[k];
    }
    store_spinor<P_F32, float>(y + blockIdx.z * chan + p * par, nullptr, g.Vh, s, acc);
}

// Weight gradients of both layers as one product over sites and colours,
//   X[(c, s)][(p, s')] = sum_n sum_colour a_c(n)_s conj((T_p b)(n)_s'),
// a: 16 channels at the site itself, b: one spinor, transported along each path.  Layer 1 has a = the
// hidden gradient, b = the input; in layer 2 sum_n gy(n) (T_p h_c(n))^dag = sum_m (T_pbar gy)(m) h_c(m)^dag,
// so a = the hidden field, b = gy and the result is conjugated (net_wgrad_reduce): one spinor is
// transported instead of 16.  A block stages OUT_NS sites and keeps the whole 64 x 36 product in the
// registers of its 192 threads (4 x 3 each); per-chunk FP32 sums are added to (hi, lo) pairs.
constexpr int OUT_NS = 16;
constexpr int OUT_THREADS = 192;
constexpr int OUT_AS = 194, OUT_TS = 110;  // complex numbers per staged site (192 and 108, padded)
constexpr int NET_X = 4 * NET_C * 36;

__global__ void __launch_bounds__(OUT_THREADS, 3) net_outer_kernel(Geom g, const char* gauge, const char* a, const char* b,
                                                                int nbatch, float2* partials)
{
    __shared__ __align__(16) float2 sa[OUT_NS * OUT_AS];
    __shared__ __align__(16) float2 st[OUT_NS * OUT_TS];
    const size_t par = (size_t)6 * 16 * g.Vh, chan = 2 * par;
    const int N = 2 * g.Vh;  // a multiple of 16: a chunk lies in one field
    const long total = (long)N * nbatch;
    const int i = threadIdx.x & 15, jj = threadIdx.x >> 4;
    float hr[4][3], hi[4][3], lr[4][3], li[4][3];
#pragma unroll
    for (int x = 0; x < 4; ++x)
#pragma unroll
        for (int y = 0; y < 3; ++y) hr[x][y] = hi[x][y] = lr[x][y] = li[x][y] = 0.f;
    for (long base = (long)blockIdx.x * OUT_NS; base < total; base += (long)gridDim.x * OUT_NS) {
        const int fb = (int)(base / N), n0 = (int)(base - (long)fb * N);
        __syncthreads();
        for (int k = threadIdx.x; k < OUT_NS * (NET_C + 9); k += OUT_THREADS) {
            const int j = k % OUT_NS, ch = k / OUT_NS;
            const int idx = n0 + j;
            const int p = idx >= g.Vh, s = idx - p * g.Vh;
            float v[24];
            float2* dst;
            int stride;
            if (ch < NET_C) {
                load_spinor<P_F32, float>(a + ((size_t)fb * NET_C + ch) * chan + p * par, nullptr, g.Vh, s, v);
                dst = sa + j * OUT_AS + 4 * ch;
                stride = 64;
            } else {
                int c[4];
                cb_coords(g, s, p, c);
                transport(g, gauge, b + fb * chan, p, s, c, ch - NET_C, v);
                dst = st + j * OUT_TS + 4 * (ch - NET_C);
                stride = 36;
            }
#pragma unroll
            for (int sp = 0; sp < 4; ++sp)
#pragma unroll
                for (int q = 0; q < 3; ++q)
                    dst[q * stride + sp] = make_float2(v[2 * (3 * sp + q)], v[2 * (3 * sp + q) + 1]);
        }
        __syncthreads();
        float cr[4][3], ci[4][3];
#pragma unroll
        for (int x = 0; x < 4; ++x)
#pragma unroll
            for (int y = 0; y < 3; ++y) cr[x][y] = ci[x][y] = 0.f;
        for (int j = 0; j < OUT_NS; ++j) {
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                const float4* pa = reinterpret_cast<const float4*>(sa + j * OUT_AS + q * 64 + 4 * i);
                const float4 a0 = pa[0], a1 = pa[1];
                const float2* pt = st + j * OUT_TS + q * 36 + 3 * jj;
                const float ar[4] = {a0.x, a0.z, a1.x, a1.z}, ai[4] = {a0.y, a0.w, a1.y, a1.w};
#pragma unroll
                for (int y = 0; y < 3; ++y) {
                    const float2 t = pt[y];
#pragma unroll
                    for (int x = 0; x < 4; ++x) {
                        cr[x][y] = fmaf(ar[x], t.x, cr[x][y]);
                        ci[x][y] = fmaf(ai[x], t.x, ci[x][y]);
                        cr[x][y] = fmaf(ai[x], t.y, cr[x][y]);
                        ci[x][y] = fmaf(-ar[x], t.y, ci[x][y]);
                    }
                }
            }
        }
        // (hi, lo) += the chunk's sum, the low word collecting the exact rounding error of each addition
#pragma unroll
        for (int x = 0; x < 4; ++x)
#pragma unroll
            for (int y = 0; y < 3; ++y) {
                float t = hr[x][y] + cr[x][y], v = t - hr[x][y];
                lr[x][y] += (hr[x][y] - (t - v)) + (cr[x][y] - v);
                hr[x][y] = t;
                t = hi[x][y] + ci[x][y];
                v = t - hi[x][y];
                li[x][y] += (hi[x][y] - (t - v)) + (ci[x][y] - v);
                hi[x][y] = t;
            }
    }
    float2* out = partials + (size_t)blockIdx.x * NET_X;
#pragma unroll
    for (int x = 0; x < 4; ++x)
#pragma unroll
        for (int y = 0; y < 3; ++y)
            out[(4 * i + x) * 36 + 3 * jj + y] = make_float2(hr[x][y] + lr[x][y], hi[x][y] + li[x][y]);
}

// gW (+)= the sum of X over the blocks, in FP64 and a fixed order: 32 entries per block, 32 threads
// per entry (each a share of the blocks).  bar: layer 2 (conjugate, spins exchanged, path reversed)
__global__ void __launch_bounds__(1024) net_wgrad_reduce(const float2* partials, int nblk, float2* gW, int bar)
{
    __shared__ double2 sh[32][32];
    const int lane = threadIdx.x & 31, part = threadIdx.x >> 5;
    const int k = blockIdx.x * 32 + lane;
    double r = 0, im = 0;
    const int b1 = (int)((long)nblk * (part + 1) / 32);
    for (int b = (int)((long)nblk * part / 32); b < b1; ++b) {
        const float2 v = partials[(size_t)b * NET_X + k];
        r += v.x;
        im += v.y;
    }
    sh[part][lane] = make_double2(r, im);
    __syncthreads();
    if (part) return;
#pragma unroll
    for (int q = 1; q < 32; ++q) {
        r += sh[q][lane].x;
        im += sh[q][lane].y;
    }
    const int row = k / 36, col = k - row * 36;
    const int ch = row >> 2, s = row & 3, path = col >> 2, s2 = col & 3;
    int o;
    if (bar) {
        const int pb = path == 0 ? 0 : (((path - 1) & 1) ? path - 1 : path + 1);
        o = (pb * NET_C + ch) * 16 + 4 * s2 + s;
        im = -im;
    } else {
        o = (path * NET_C + ch) * 16 + 4 * s + s2;
    }
    gW[o].x += (float)r;
    gW[o].y += (float)im;
}

// coefficients of gy_k = 2 (y_k - e_k) / |e_k|^2 (|e_k|^2 = 1 where e_k vanishes)
__global__ void net_loss_coef(const double2* en, int n, double2* co)
{
    const int k = threadIdx.x + blockIdx.x * blockDim.x;
    if (k >= n) return;
    const double v = 2.0 / (en[k].x > 0 ? en[k].x : 1.0);
    co[k] = make_double2(v, 0);
    co[n + k] = make_double2(-v, 0);
}

// W'[q][c'][c] = W[qbar][c][c']^dag for a layer W[9][cout][cin][16]
__global__ void net_adjoint_weights(const float2* W, float2* Wa, int cin, int cout)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= 9 * cout * cin * 16) return;
    const int q = k / (cin * cout * 16);
    int rem = k % (cin * cout * 16);
    const int cp = rem / (cout * 16);  // adjoint output channel = W input channel
    rem %= cout * 16;
    const int cc = rem / 16;           // adjoint input channel = W output channel
    const int e = rem % 16, sa = e / 4, sb = e % 4;
    const int qbar = q == 0 ? 0 : (((q - 1) & 1) ? q - 1 : q + 1);
    const float2 w = W[((qbar * cout + cc) * cin + cp) * 16 + 4 * sb + sa];
    Wa[k] = make_float2(w.x, -w.y);
}

__global__ void adam_kernel(float2* W, const float2* G, float* m, float* v, int n, float lr, float b1, float b2,
                            float eps, float c1, float c2, float gscale)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= 2 * n) return;
    float* w = reinterpret_cast<float*>(W);
    const float gk = reinterpret_cast<const float*>(G)[k] * gscale;
    m[k] = b1 * m[k] + (1 - b1) * gk;
    v[k] = b2 * v[k] + (1 - b2) * gk * gk;
    w[k] -= lr * (m[k] / c1) / (sqrtf(v[k] / c2) + eps);
}

FieldDesc some(const FieldDesc& f, int i, int n)
{
    FieldDesc s = f;
    s.nrhs = n;
    s.data = f.data + (size_t)i * f.rhs_bytes();
    s.norm = f.norm ? f.norm + (size_t)i * 2 * f.Vh : nullptr;
    return s;
}

FieldDesc one(const FieldDesc& f, int i) { return some(f, i, 1); }

int net_init(ov_ctx* c)
{
    if (c->net) return OV_OK;
    NetState* n = new NetState();
    c->net = n;
    void* p = nullptr;
    OV_TRY(dev_alloc(c, &p, sizeof(float2) * NET_PARAMS));
    n->W = (float2*)p;
    OV_TRY(dev_alloc(c, &p, sizeof(float2) * NET_PARAMS));
    n->Wadj = (float2*)p;
    OV_TRY(dev_alloc(c, &p, sizeof(float2) * NET_PARAMS));
    n->G = (float2*)p;
    OV_TRY(dev_alloc(c, &p, sizeof(float) * 4 * NET_PARAMS));
    n->adam = (float*)p;
    OV_CUDA(c, cudaMemset(n->adam, 0, sizeof(float) * 4 * NET_PARAMS));
    OV_CUDA(c, cudaMemset(n->W, 0, sizeof(float2) * NET_PARAMS));
    return OV_OK;
}

// fields of a batch: the number asked for, such that the work fields stay below about 2 GB
int net_batch(const ov_ctx* c, int want)
{
    const double per = (2.0 * NET_C + 2) * 192.0 * c->g.Vh;
    const int cap = (int)std::min(16.0, std::max(1.0, 2e9 / per));
    return std::min(want, cap);
}

struct NetWork {
    FieldDesc h, gh, z, y, gy, a, b, d;
};

// Work fields of a batch of *nb: h and gh (16 channels each), y, gy, and those that the preconditioner asks for
// (a, b: FP32 copies of its input and output, d: the adjoint's result).  z, the 9 paths' fields of the 16 -> 1
// layer, lies in gh, which is written after z's last use.  They are kept, and grown when a larger batch is asked
// for; where the device has no room for it the batch is halved (*nb) and stays there.
int net_work(ov_ctx* c, int* nb, bool a, bool b, bool d, NetWork* w)
{
    NetState* n = c->net;
    const int slots[] = {WS_NET_H, WS_NET_GH, WS_NET_Y, WS_NET_G, WS_NET_A, WS_NET_B, WS_NET_S};
    for (int want = std::max(std::min(*nb, n->batch_max), n->batch);; want /= 2) {
        if (n->batch < want) {
            cudaDeviceSynchronize();  // queued kernels may still use the smaller fields
            for (int slot : slots) ws_release(c, slot);
        }
        n->batch = want;
        int s = ws_field(c, WS_NET_H, P_F32, NET_C * want, &w->h);
        if (s == OV_OK) s = ws_field(c, WS_NET_GH, P_F32, NET_C * want, &w->gh);
        if (s == OV_OK) s = ws_field(c, WS_NET_Y, P_F32, want, &w->y);
        if (s == OV_OK) s = ws_field(c, WS_NET_G, P_F32, want, &w->gy);
        if (s == OV_OK && a) s = ws_field(c, WS_NET_A, P_F32, want, &w->a);
        if (s == OV_OK && b) s = ws_field(c, WS_NET_B, P_F32, want, &w->b);
        if (s == OV_OK && d) s = ws_field(c, WS_NET_S, P_F32, want, &w->d);
        if (s == OV_OK) {
            w->z = w->gh;
            *nb = std::min(*nb, want);
            return OV_OK;
        }
        cudaDeviceSynchronize();
        for (int slot : slots) ws_release(c, slot);
        n->batch = 0;
        if (s != OV_ENOMEM || want == 1) return s;
        n->batch_max = want / 2;
    }
}

// layer (or its adjoint) on nb fields; z: work field of the 16 -> 1 form
int layer_fwd(ov_ctx* c, int layer, bool adj, const FieldDesc& x, const FieldDesc& y, const FieldDesc& z, int nb,
              cudaStream_t st)
{
    NetState* n = c->net;
    const float2* W = (adj ? n->Wadj : n->W) + (size_t)layer * NET_W;
    const Geom& g = c->g;
    const char* gauge = (const char*)c->gauge[P_F32];
    const unsigned sites = (unsigned)((2 * g.Vh + 127) / 128);
    // layer 0: 1 -> 16 (adjoint 16 -> 1); layer 1: 16 -> 1 (adjoint 1 -> 16)
    if ((layer == 0) != adj) {
        net_many_kernel<<<dim3(sites, NET_C / NET_CG, nb), 128, 0, st>>>(g, gauge, x.data, y.data, W);
    } else {
        net_mix_kernel<<<dim3(sites, 3, nb), 128, 0, st>>>(g, x.data, z.data, W);
        net_gather_kernel<<<dim3(sites, 1, nb), 128, 0, st>>>(g, gauge, z.data, y.data);
    }
    OV_CUDA(c, cudaGetLastError());
    return OV_OK;
}

int refresh_adjoint(ov_ctx* c, cudaStream_t st)
{
    NetState* n = c->net;
    net_adjoint_weights<<<(NET_W + 255) / 256, 256, 0, st>>>(n->W, n->Wadj, 1, NET_C);
    net_adjoint_weights<<<(NET_W + 255) / 256, 256, 0, st>>>(n->W + NET_W, n->Wadj + NET_W, NET_C, 1);
    OV_CUDA(c, cudaGetLastError());
    return OV_OK;
}

// loss over pairs k0..k1 of (pr, pe) and its gradient into n->G
int loss_grad(ov_ctx* c, const FieldDesc& pr, const FieldDesc& pe, int k0, int k1, double* loss, cudaStream_t st)
{
    NetState* n = c->net;
    const Geom& g = c->g;
    const int np = k1 - k0;
    int B = net_batch(c, np);
    NetWork w;
    OV_TRY(net_work(c, &B, false, false, false, &w));
    const int nblk_max = 4 * 152;
    const size_t need = (size_t)nblk_max * NET_X;
    if (n->partials_n < need) {
        if (n->partials) {
            cudaDeviceSynchronize();
            dev_free(c, n->partials, sizeof(float2) * n->partials_n);
            n->partials = nullptr;
            n->partials_n = 0;
        }
        void* p = nullptr;
        OV_TRY(dev_alloc(c, &p, sizeof(float2) * need));
        n->partials = (float2*)p;
        n->partials_n = need;
    }
    OV_CUDA(c, cudaMemsetAsync(n->G, 0, sizeof(float2) * NET_PARAMS, st));
    OV_TRY(refresh_adjoint(c, st));
    std::vector<double2> en(np);
    std::vector<double> gn(np);
    double2* dn = (double2*)(c->dscal + DSCAL_DOT);
    double2* dco = (double2*)(c->dscal + DSCAL_CGCO);
    double* dg = c->dscal + DSCAL_NORM;
    const char* gauge = (const char*)c->gauge[P_F32];
    OV_TRY(norm2(c, some(pe, k0, np), (double*)dn, st));
    for (int k = k0; k < k1; k += B) {
        const int nb = std::min(B, k1 - k);
        FieldDesc r = some(pr, k, nb), e = some(pe, k, nb), y = some(w.y, 0, nb), gy = some(w.gy, 0, nb);
        OV_TRY(layer_fwd(c, 0, false, r, w.h, w.z, nb, st));
        OV_TRY(layer_fwd(c, 1, false, w.h, y, w.z, nb, st));
        // gy = 2 (y - e) / |e|^2, with |gy|^2 recorded for the loss
        net_loss_coef<<<1, 32, 0, st>>>(dn + (k - k0), nb, dco);
        FieldDesc xs[2] = {y, e};
        OV_TRY(lincomb(c, gy, 2, xs, nullptr, dco, 0, dg + (k - k0), st));
        const int nblk = (int)std::min<long>(nblk_max, (2L * g.Vh * nb) / OUT_NS);
        net_outer_kernel<<<nblk, OUT_THREADS, 0, st>>>(g, gauge, w.h.data, gy.data, nb, n->partials);
        net_wgrad_reduce<<<NET_X / 32, 1024, 0, st>>>(n->partials, nblk, n->G + NET_W, 1);
        OV_TRY(layer_fwd(c, 1, true, gy, w.gh, w.z, nb, st));  // gh = L2^dag gy
        net_outer_kernel<<<nblk, OUT_THREADS, 0, st>>>(g, gauge, w.gh.data, r.data, nb, n->partials);
        net_wgrad_reduce<<<NET_X / 32, 1024, 0, st>>>(n->partials, nblk, n->G, 0);
        OV_CUDA(c, cudaGetLastError());
    }
    OV_CUDA(c, cudaMemcpyAsync(en.data(), dn, sizeof(double2) * np, cudaMemcpyDeviceToHost, st));
    OV_CUDA(c, cudaMemcpyAsync(gn.data(), dg, sizeof(double) * np, cudaMemcpyDeviceToHost, st));
    OV_CUDA(c, cudaStreamSynchronize(st));
    double total = 0;
    for (int k = 0; k < np; ++k) total += gn[k] * (en[k].x > 0 ? en[k].x : 1.0) / 4.0;  // |y-e|^2/|e|^2 = |gy|^2 |e|^2 / 4
    *loss = total;
    return OV_OK;
}

}  // namespace

bool net_ready(const ov_ctx* c) { return c->net && c->net->trained; }

void net_free(ov_ctx* c)
{
    NetState* n = c->net;
    if (!n) return;
    cudaDeviceSynchronize();
    if (n->W) dev_free(c, n->W, sizeof(float2) * NET_PARAMS);
    if (n->Wadj) dev_free(c, n->Wadj, sizeof(float2) * NET_PARAMS);
    if (n->G) dev_free(c, n->G, sizeof(float2) * NET_PARAMS);
    if (n->adam) dev_free(c, n->adam, sizeof(float) * 4 * NET_PARAMS);
    if (n->partials) dev_free(c, n->partials, sizeof(float2) * n->partials_n);
    field_free(c, &n->pr);
    field_free(c, &n->px);
    delete n;
    c->net = nullptr;
}

// z = M r for every rhs of r (any precision; computed in FP32)
int net_apply_precond(ov_ctx* c, const FieldDesc& r, const FieldDesc& z, cudaStream_t st)
{
    if (!c->net) return set_err(c, OV_ESTATE, "learned preconditioner has no weights");
    NetState* n = c->net;
    const bool sym = c->net_sym != 0;
    if (sym && !n->adj_valid) {
        OV_TRY(refresh_adjoint(c, st));
        n->adj_valid = 1;
    }
    const int R = r.nrhs;
    int B = net_batch(c, R);
    NetWork w;
    const bool f32in = r.prec == P_F32, f32out = z.prec == P_F32;
    OV_TRY(net_work(c, &B, !f32in, !f32out, sym, &w));
    const FieldDesc &a = w.a, &b = w.b, &d = w.d;
    for (int q = 0; q < R; q += B) {
        const int nb = std::min(B, R - q);
        FieldDesc rq = some(r, q, nb), zq = some(z, q, nb);
        if (!f32in) OV_TRY(convert(c, rq, some(a, 0, nb), st));
        const FieldDesc x = f32in ? rq : some(a, 0, nb), out = f32out ? zq : some(b, 0, nb);
        const FieldDesc y = sym ? some(w.y, 0, nb) : out;
        OV_TRY(layer_fwd(c, 0, false, x, w.h, w.z, nb, st));
        OV_TRY(layer_fwd(c, 1, false, w.h, y, w.z, nb, st));
        if (sym) {
            // z = (M + M^dag) r / 2, M^dag = L1^dag L2^dag: Hermitian, as CG expects of a preconditioner
            OV_TRY(layer_fwd(c, 1, true, x, w.h, w.z, nb, st));
            OV_TRY(layer_fwd(c, 0, true, w.h, some(d, 0, nb), w.z, nb, st));
            FieldDesc v[2] = {y, some(d, 0, nb)};
            double2 hc[2] = {make_double2(0.5, 0), make_double2(0.5, 0)};
            OV_TRY(lincomb(c, out, 2, v, hc, nullptr, 0, nullptr, st));
        }
        if (!f32out) OV_TRY(convert(c, out, zq, st));
    }
    return OV_OK;
}

// called by the CG at each FP64 true-residual point while recording
int net_record_pair(ov_ctx* c, const FieldDesc& r64, const FieldDesc& x64, cudaStream_t st)
{
    NetState* n = c->net;
    if (!n || !n->recording) return OV_OK;
    for (int q = 0; q < r64.nrhs && n->npairs < n->cap; ++q, ++n->npairs) {
        OV_TRY(convert(c, one(r64, q), one(n->pr, n->npairs), st));
        OV_TRY(convert(c, one(x64, q), one(n->px, n->npairs), st));
    }
    return OV_OK;
}

}  // namespace ov

using namespace ov;

extern "C" {

int ov_net_set_weights(ov_ctx* c, const double* w, int n)
{
    if (!c) return OV_EINVAL;
    if (!w || n != 2 * NET_PARAMS) return set_err(c, OV_EINVAL, "weights: expected %d doubles", 2 * NET_PARAMS);
    CallScope call(c, (cudaStream_t)0);
    OV_TRY(call.begin());
    OV_TRY(net_init(c));
    std::vector<float2> h(NET_PARAMS);
    for (int i = 0; i < NET_PARAMS; ++i) h[i] = make_float2((float)w[2 * i], (float)w[2 * i + 1]);
    OV_CUDA(c, cudaMemcpy(c->net->W, h.data(), sizeof(float2) * NET_PARAMS, cudaMemcpyHostToDevice));
    c->net->trained = 1;
    c->net->adj_valid = 0;
    return OV_OK;
}

int ov_net_get_weights(ov_ctx* c, double* w, int n)
{
    if (!c) return OV_EINVAL;
    if (!w || n != 2 * NET_PARAMS) return set_err(c, OV_EINVAL, "weights: expected %d doubles", 2 * NET_PARAMS);
    if (!c->net) return set_err(c, OV_ESTATE, "no network weights");
    CallScope call(c, (cudaStream_t)0);
    OV_TRY(call.begin());
    std::vector<float2> h(NET_PARAMS);
    OV_CUDA(c, cudaMemcpy(h.data(), c->net->W, sizeof(float2) * NET_PARAMS, cudaMemcpyDeviceToHost));
    for (int i = 0; i < NET_PARAMS; ++i) {
        w[2 * i] = h[i].x;
        w[2 * i + 1] = h[i].y;
    }
    return OV_OK;
}

int ov_net_apply(ov_ctx* c, const void* in, void* out, int nrhs, void* stream)
{
    if (!c) return OV_EINVAL;
    if (!in || !out || in == out) return set_err(c, OV_EINVAL, "bad buffers");
    if (nrhs < 1 || nrhs > 16) return set_err(c, OV_EINVAL, "nrhs out of range");
    if (!c->have_gauge) return set_err(c, OV_ESTATE, "no gauge field");
    if (!c->net) return set_err(c, OV_ESTATE, "no network weights");
    cudaStream_t st = (cudaStream_t)stream;
    CallScope call(c, st);
    OV_TRY(call.begin());
    const size_t bytes = (size_t)nrhs * 2 * c->g.Vh * 12 * 16;
    const double* din = nullptr;
    double* dout = nullptr;
    OV_TRY(stage_in(c, 0, in, bytes, st, &din));
    OV_TRY(stage_out_buffer(c, 1, out, bytes, &dout));
    FieldDesc fi, fo;
    OV_TRY(ws_field(c, WS_IN, P_F32, nrhs, &fi));
    OV_TRY(ws_field(c, WS_OUT, P_F32, nrhs, &fo));
    OV_CUDA(c, launch_pack(c->g, din, fi, st));
    OV_TRY(net_apply_precond(c, fi, fo, st));
    OV_CUDA(c, launch_unpack(c->g, fo, dout, st));
    return call.finish(stage_out_finish(c, out, dout, bytes, st));
}

int ov_net_loss_grad(ov_ctx* c, const void* r, const void* e, int npairs, double* loss, double* grad, void* stream)
{
    if (!c) return OV_EINVAL;
    if (!r || !e || !loss || npairs < 1 || npairs > 16) return set_err(c, OV_EINVAL, "bad arguments");
    if (!c->have_gauge) return set_err(c, OV_ESTATE, "no gauge field");
    if (!c->net) return set_err(c, OV_ESTATE, "no network weights");
    cudaStream_t st = (cudaStream_t)stream;
    CallScope call(c, st);
    OV_TRY(call.begin());
    const size_t bytes = (size_t)npairs * 2 * c->g.Vh * 12 * 16;
    const double *dr = nullptr, *de = nullptr;
    FieldDesc fr, fe;
    OV_TRY(ws_field(c, WS_CG_R, P_F32, npairs, &fr));
    OV_TRY(ws_field(c, WS_CG_T, P_F32, npairs, &fe));
    OV_TRY(stage_in(c, 0, r, bytes, st, &dr));
    OV_CUDA(c, launch_pack(c->g, dr, fr, st));
    OV_TRY(stage_in(c, 1, e, bytes, st, &de));
    OV_CUDA(c, launch_pack(c->g, de, fe, st));
    OV_TRY(loss_grad(c, fr, fe, 0, npairs, loss, st));
    if (grad) {
        std::vector<float2> h(NET_PARAMS);
        OV_CUDA(c, cudaMemcpyAsync(h.data(), c->net->G, sizeof(float2) * NET_PARAMS, cudaMemcpyDeviceToHost, st));
        OV_CUDA(c, cudaStreamSynchronize(st));
        for (int i = 0; i < NET_PARAMS; ++i) {
            grad[2 * i] = h[i].x;
            grad[2 * i + 1] = h[i].y;
        }
    }
    return OV_OK;
}

int ov_net_train(ov_ctx* c, int nsolves, int steps, double lr, double mass, double* final_loss, void* stream)
{
    if (!c) return OV_EINVAL;
    if (nsolves < 1 || nsolves > 64 || steps < 0 || !(lr > 0)) return set_err(c, OV_EINVAL, "bad training arguments");
    if (!c->have_gauge || !c->have_poly) return set_err(c, OV_ESTATE, "training needs gauge field and sign polynomial");
    cudaStream_t st = (cudaStream_t)stream;
    CallScope call(c, st);
    OV_TRY(call.begin());
    OV_TRY(net_init(c));
    NetState* n = c->net;
    // ---- record (residual, iterate) pairs from deflated mixed-precision CG solves of random sources
    if (!n->pr.data) {
        n->cap = NET_MAXPAIRS;
        OV_TRY(field_alloc(c, P_F32, n->cap, &n->pr));
        OV_TRY(field_alloc(c, P_F32, n->cap, &n->px));
    }
    n->npairs = 0;
    FieldDesc b, xs32;
    OV_TRY(ws_field(c, WS_AUX1, P_F64, 1, &b));
    OV_TRY(ws_field(c, WS_AUX1, P_F32, 1, &xs32));
    const int was_trained = n->trained;
    n->trained = 0;
    for (int s = 0; s < nsolves && n->npairs < n->cap; ++s) {
        OV_CUDA(c, launch_fill_random(c->g, b, 9001ull + s, st));
        if (c->chiral) {  // chiral-sector solves need sources of definite chirality: alternate the sectors
            const double chi = (s & 1) ? -1.0 : 1.0;
            FieldDesc v2[2] = {b, b};
            double2 h2[2] = {make_double2(0.5, 0), make_double2(0.5 * chi, 0)};
            OV_TRY(lincomb(c, b, 2, v2, h2, nullptr, 2, nullptr, st));
        }
        const int first = n->npairs;
        n->recording = 1;
        FieldDesc bb, xx;
        OV_TRY(ws_field(c, WS_CG_B, P_F64, 1, &bb));
        OV_TRY(copy_field(c, b, bb, st));
        OV_TRY(ws_field(c, WS_CG_X, P_F64, 1, &xx));
        int r = cg_impl(c, bb, xx, mass, 1e-8, 400, 0, P_F32, nullptr, st);
        n->recording = 0;
        if (r != OV_OK && r != OV_ENOTCONV) return r;
        // e_k = x* - x_k (in place over the recorded iterates)
        OV_TRY(convert(c, xx, xs32, st));
        for (int k = first; k < n->npairs; ++k) {
            FieldDesc v[2] = {xs32, one(n->px, k)};
            double2 h[2] = {make_double2(1, 0), make_double2(-1, 0)};
            OV_TRY(lincomb(c, one(n->px, k), 2, v, h, nullptr, 0, nullptr, st));
        }
        // drop the last pair of the solve (converged: e ~ 0)
        if (n->npairs > first + 1) --n->npairs;
    }
    if (n->npairs < 2) return set_err(c, OV_ESTATE, "training: only %d pairs recorded", n->npairs);
    // ---- initialise: M = alpha * identity path (least-squares alpha), small deterministic noise elsewhere
    if (!was_trained) {
        std::vector<float2> w0(NET_PARAMS);
        unsigned long long z = 0x12345678ull;
        auto rnd = [&]() {
            z = z * 6364136223846793005ull + 1442695040888963407ull;
            return (float)((double)(z >> 11) / 9007199254740992.0 - 0.5);
        };
        for (auto& v : w0) v = make_float2(0.02f * rnd(), 0.02f * rnd());
        double num = 0, den = 0;
        for (int k = 0; k < n->npairs; ++k) {
            double* d = c->dscal + DSCAL_DOT;
            OV_TRY(dot(c, one(n->pr, k), one(n->px, k), (double2*)d, st));
            double2 re;
            OV_CUDA(c, cudaMemcpyAsync(&re, d, sizeof re, cudaMemcpyDeviceToHost, st));
            OV_TRY(norm2(c, one(n->pr, k), d, st));
            double2 rr;
            OV_CUDA(c, cudaMemcpyAsync(&rr, d, sizeof rr, cudaMemcpyDeviceToHost, st));
            OV_CUDA(c, cudaStreamSynchronize(st));
            double e2;
            OV_TRY(norm2(c, one(n->px, k), d, st));
            double2 ee;
            OV_CUDA(c, cudaMemcpyAsync(&ee, d, sizeof ee, cudaMemcpyDeviceToHost, st));
            OV_CUDA(c, cudaStreamSynchronize(st));
            e2 = ee.x > 0 ? ee.x : 1.0;
            num += re.x / e2;
            den += rr.x / e2;
        }
        const float alpha = (float)(den > 0 ? num / den : 1.0);
        for (int sa = 0; sa < 4; ++sa) {
            w0[(0 * NET_C + 0) * 16 + 5 * sa] = make_float2(1.f, 0.f);                   // layer 1, path 0, c=0
            w0[NET_W + (0 * 1 + 0) * NET_C * 16 + 5 * sa] = make_float2(alpha, 0.f);      // layer 2, path 0, c'=0
        }
        OV_CUDA(c, cudaMemcpyAsync(n->W, w0.data(), sizeof(float2) * NET_PARAMS, cudaMemcpyHostToDevice, st));
        OV_CUDA(c, cudaMemsetAsync(n->adam, 0, sizeof(float) * 4 * NET_PARAMS, st));
        n->adam_t = 0;
    }
    // ---- Adam over all recorded pairs
    double loss = 0;
    const float b1 = 0.9f, b2 = 0.999f;
    n->history.clear();
    for (int it = 0; it < steps; ++it) {
        OV_TRY(loss_grad(c, n->pr, n->px, 0, n->npairs, &loss, st));
        n->history.push_back(loss / n->npairs);
        ++n->adam_t;
        const float c1 = 1.f - powf(b1, (float)n->adam_t), c2 = 1.f - powf(b2, (float)n->adam_t);
        const float lr_t = (float)(lr * (it < steps / 2 ? 1.0 : 0.3));
        adam_kernel<<<(2 * NET_PARAMS + 255) / 256, 256, 0, st>>>(n->W, n->G, n->adam, n->adam + 2 * NET_PARAMS,
                                                                   NET_PARAMS, lr_t, b1, b2, 1e-8f, c1, c2,
                                                                   1.0f / (float)n->npairs);
        OV_CUDA(c, cudaGetLastError());
    }
    OV_TRY(loss_grad(c, n->pr, n->px, 0, n->npairs, &loss, st));  // also refreshes the adjoint weights
    if (final_loss) *final_loss = loss / n->npairs;
    n->history.push_back(loss / n->npairs);
    n->trained = 1;
    n->adj_valid = 1;
    return OV_OK;
}

int ov_net_pairs(const ov_ctx* c) { return c && c->net ? c->net->npairs : 0; }

int ov_net_loss_history(const ov_ctx* c, double* out, int cap)
{
    if (!c || cap < 0 || (cap > 0 && !out)) return -OV_EINVAL;
    if (!c->net) return 0;
    const auto& h = c->net->history;
    for (int i = 0; i < cap && i < (int)h.size(); ++i) out[i] = h[i];
    return (int)h.size();
}

}  // extern "C"
