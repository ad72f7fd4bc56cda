// Wilson dslash in FP32 arithmetic, launch variant 12: one warp per hop, for lattices that leave most of
// the chip idle with one site per thread.
//
// A block of eight warps takes 32 sites of one right-hand side: warp w forms hop w, the 6 complex results
// per site go through shared memory (12 KB), and six warps sum four output reals per site each.  One
// site's loads are all in flight at once and its serial chain is an eighth as long (4^4: 2.2 us per launch
// in a graph, 2.8 with one site per thread; 8^4: 2.3 / 3.0).  Above about 10^4 sites and right-hand sides
// the shared-memory exchange (18 clocks of L1 bandwidth per site beside 10 of loads) costs more than the
// latency it saves: default_shape draws the line.
#include "dslash_common.cuh"

namespace ov {

namespace {

constexpr int HOP_THREADS = 256;

template <int SP, int GP, int NY>
__global__ void __launch_bounds__(HOP_THREADS) dslash_hop_kernel(const __grid_constant__ DslashArgs A)
{
    constexpr bool H16 = SP == P_F16 || SP == P_BF16;
    __shared__ float4 sh[8][3][32];           // hop results: reals 4 k .. 4 k + 3 of the half spinor
    __shared__ float4 so[H16 ? 6 : 1][32];    // 16-bit: the output reals before scaling
    pdl_begin();
    const Geom& g = A.g;
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const BlockWork bw = block_work(A.nrhs);
    const int p = bw.p, q = 1 - p, r = bw.grp;
    const int s_raw = bw.sb * 32 + lane;
    const bool live = s_raw < g.Vh;
    const int s = live ? s_raw : g.Vh - 1;
    constexpr size_t CH = nchunk_dev<SP>() * 16;
    const size_t par_bytes = CH * g.Vh;
    const size_t off = ((size_t)r * 2 + p) * par_bytes, noff = ((size_t)r * 2 + p) * g.Vh;
    int c[4], sn;
    bool cross;
    cb_coords(g, s, p, c);
    hop_neighbour(g, w, s, c, sn, cross);
    pdl_wait();
    {
        const char* in_q = A.in + ((size_t)r * 2 + q) * par_bytes;
        const float* inn_q = A.in_n ? A.in_n + ((size_t)r * 2 + q) * g.Vh : nullptr;
        float v[24], h[12], u[18], chi[12];
        float ph = cross ? A.g.fbc[w >> 1] : 1.f;
        if constexpr (H16)
            ph *= load_spinor_unscaled<SP, false>(in_q, inn_q, g.Vh, sn, v);
        else
            load_spinor<SP, float, false>(in_q, inn_q, g.Vh, sn, v);
        const bool fwd = (w & 1) == 0;
        load_link<GP, float>(A.gauge + (size_t)((fwd ? p : q) * 4 + (w >> 1)) * g.Vh * gauge_link_bytes_dev<GP>(), g.Vh,
                             fwd ? s : sn, u);
        project_hop<float>(w, v, h);
#pragma unroll
        for (int i = 0; i < 12; ++i) h[i] *= ph;
        if (fwd)
            link_mul<+1, float>(u, h, chi);
        else
            link_mul<-1, float>(u, h, chi);
#pragma unroll
        for (int k = 0; k < 3; ++k)
            sh[w][k][lane] = make_float4(chi[4 * k], chi[4 * k + 1], chi[4 * k + 2], chi[4 * k + 3]);
    }
    __syncthreads();
    float o[4];
    if (w < 6) {
        // output reals 4 w .. 4 w + 3: complex components 2 w and 2 w + 1 (spin, colour = component / 3, % 3)
#pragma unroll
        for (int m = 0; m < 2; ++m) {
            const int k = 2 * w + m, sp = k / 3, col = k - 3 * sp;
            float re, im;
            sum_hops<float>(sp,
                            [&](int hop, int a, float& x, float& y) {
                                const float2 t = reinterpret_cast<const float2*>(
                                    &sh[hop][(3 * a + col) >> 1][lane])[(3 * a + col) & 1];
                                x = t.x;
                                y = t.y;
                            },
                            re, im);
            o[2 * m] = re;
            o[2 * m + 1] = im;
        }
        auto field4 = [&](const char* base, const float* nrm, float x[4]) {
            if constexpr (H16) {
                const uint2 t = ld_field<false>(reinterpret_cast<const uint2*>(base + off) + 2 * ((size_t)(w >> 1) * g.Vh + s) + (w & 1));
                const float n = ld_field<false>(nrm + noff + s);
                const float2 a = Half<SP>::to2(t.x), b = Half<SP>::to2(t.y);
                x[0] = a.x * n;
                x[1] = a.y * n;
                x[2] = b.x * n;
                x[3] = b.y * n;
            } else {
                const float4 t = ld_field<false>(reinterpret_cast<const float4*>(base + off) + (size_t)w * g.Vh + s);
                x[0] = t.x;
                x[1] = t.y;
                x[2] = t.z;
                x[3] = t.w;
            }
        };
        const bool low = w >= 3;  // spins 2, 3
        float x[4];
        field4(A.in, A.in_n, x);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            o[i] = A.fa * x[i] + A.fb * o[i];
            if (A.g5_core && low) o[i] = -o[i];
        }
#pragma unroll
        for (int j = 0; j < NY; ++j) {
            field4(A.y[j], A.y_n[j], x);
#pragma unroll
            for (int i = 0; i < 4; ++i) o[i] += A.fsy[j] * x[i];
        }
#pragma unroll
        for (int i = 0; i < 4; ++i)
            if (A.g5_out && low) o[i] = -o[i];
        if constexpr (H16)
            so[w][lane] = make_float4(o[0], o[1], o[2], o[3]);
        else if (live)
            reinterpret_cast<float4*>(A.out + off)[(size_t)w * g.Vh + s] = make_float4(o[0], o[1], o[2], o[3]);
    }
    if constexpr (H16) {
        __syncthreads();
        if (w < 3 && live) {
            float v[24];
#pragma unroll
            for (int k = 0; k < 6; ++k) {
                const float4 t = so[k][lane];
                v[4 * k] = t.x;
                v[4 * k + 1] = t.y;
                v[4 * k + 2] = t.z;
                v[4 * k + 3] = t.w;
            }
            store_spinor_chunk<SP>(A.out + off, A.out_n + noff, g.Vh, s, v, w);
        }
    }
}

struct Hop32 {
    template <int SP, int GP>
    static cudaError_t run(const DslashArgs& A, int ny, int, dim3, dim3, cudaStream_t st)
    {
        const dim3 grid = block_grid(A.g.Vh, 32, A.nrhs), block(HOP_THREADS);
        switch (ny) {
        case 0: return launch_kernel(dslash_hop_kernel<SP, GP, 0>, grid, block, st, A.pdl, PDL_HOP32, A);
        case 1: return launch_kernel(dslash_hop_kernel<SP, GP, 1>, grid, block, st, A.pdl, PDL_HOP32, A);
        case 2: return launch_kernel(dslash_hop_kernel<SP, GP, 2>, grid, block, st, A.pdl, PDL_HOP32, A);
        case 3: return launch_kernel(dslash_hop_kernel<SP, GP, 3>, grid, block, st, A.pdl, PDL_HOP32, A);
        }
        return cudaErrorInvalidValue;
    }
};

}  // namespace

cudaError_t launch_dslash_hop32(const DslashArgs& A, int sp, int gp, int ny, int var, dim3 grid, dim3 block, cudaStream_t st)
{
    return dispatch_prec<Hop32>(A, sp, gp, ny, var, grid, block, st);
}

}  // namespace ov
