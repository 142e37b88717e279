// Backward of the cone-beam projection proj = exp(-sum_g tau_g) (Eq. 21 with diverging rays).
//
// dL/dtau = -proj dL/dproj for every Gaussian on a pixel's ray, whatever the order, so nothing is
// replayed: a warp takes a (view, Gaussian) item, walks the item's own footprint rectangle and writes
// its 13 moment sums (render_bwd.cu) once, without atomics.  With w = -dL/dproj proj |d_c| per pixel
// (written by the forward) dL/dln(kappa) at a pixel is G = w K exp(-m^2 / 2) / |d'|.  A lane owns a pixel
// column of a strip and two rows at a time: dx is constant along a column, so per pixel only the sums
// over dy (1, dy, dy^2) of 2 dL/da and 2 dL/dq are formed, packed over the two rows, and dx enters once per
// column.  The lanes stand 4 to 32 side by side, whichever covers the rectangle in the fewest steps.
// Bound by issue (about 45 slots per 64 pixels).  20,000 Gaussians, 12 views of 256 x 256: 1.28 -> 0.38 ms
// against the blend's backward, which replays per (tile, Gaussian) and reduces 16 sums for each (2 / 4 CTAs
// per SM 0.44 / 0.41 ms).
#include <algorithm>

#include "blend.cuh"

namespace vg {

constexpr int kConeWarps = 8;
// Items of a warp, at most.  1 / 4 / 8 / 16 / 32: 20,000 Gaussians and 12 views of 256 x 256 429 / 374 / 370 / 381 / 379 us,
// 50,000 and 16 views of 320 x 320 2.04 / 1.74 / 1.66 / 1.65 / 1.66 ms.
constexpr int kConeItems = 16;

__global__ void __launch_bounds__(32 * kConeWarps, 3)
k_cone_bwd(const ViewInfo *__restrict__ views, long long n_items, int per_warp, int n_per_view,
           const float4 *__restrict__ rec, const short4 *__restrict__ prect, const float *__restrict__ weights,
           float *__restrict__ acc) {
    pdl_entry();
    const int lane = threadIdx.x & 31;
    // a CTA takes a run of items, dealt to its warps in turn
    const long long at0 = (long long)blockIdx.x * kConeWarps * per_warp + (threadIdx.x >> 5);
    const long long mine = at0 + (long long)lane * kConeWarps;
    short4 my_rect = make_short4(-1, -1, -1, -1);
    if (lane < per_warp && mine < n_items) my_rect = prect[mine];
    for (unsigned todo = __ballot_sync(0xffffffffu, my_rect.x >= 0); todo; todo &= todo - 1) {
        const int from = __ffs(todo) - 1;
        const long long it = at0 + (long long)from * kConeWarps;
        const int xr = __shfl_sync(0xffffffffu, (int)my_rect.x | (int)my_rect.z << 16, from);
        const int yr = __shfl_sync(0xffffffffu, (int)my_rect.y | (int)my_rect.w << 16, from);
        const int rx0 = xr & 0xffff, rx1 = xr >> 16, ry0 = yr & 0xffff, ry1 = yr >> 16;
        RecPairs r;
        {
            const float4 *src = rec + it * kRecF4;
            const float4 q0 = __ldg(src), q1 = __ldg(src + 1), q2 = __ldg(src + 2), q3 = __ldg(src + 3), q4 = __ldg(src + 4);
            r.ac0[0] = f2_pack(q0.x, q0.y), r.ac0[1] = f2_pack(q0.z, q0.w), r.ac0[2] = f2_pack(q1.x, q1.y);
            r.ac1[0] = f2_pack(q1.z, q1.w), r.ac1[1] = f2_pack(q2.x, q2.y), r.ac1[2] = f2_pack(q2.z, q2.w);
            r.ac2[0] = f2_pack(q3.x, q3.y), r.ac2[1] = f2_pack(q3.z, q3.w), r.ac2[2] = f2_pack(q4.x, q4.y);
            r.px0 = q4.z, r.py0 = q4.w;
            r.q5 = __ldg(src + 5);
        }
        const ViewInfo &V = views[it / n_per_view];
        const int W = V.W, w = rx1 - rx0 + 1, h = ry1 - ry0 + 1;
        int lxb = 2, best = 1 << 30;   // log2 of the lanes side by side
#pragma unroll
        for (int b = 2; b <= 5; ++b) {
            const int cost = ((w + (1 << b) - 1) >> b) * (((h + (64 >> b) - 1) >> (6 - b)) * 3 + 2);   // a strip costs 2/3 of a step (0 to 4 of them: within 1%)
            if (cost <= best) best = cost, lxb = b;
        }
        const int lx = lane & ((1 << lxb) - 1), ly = lane >> lxb, row_step = 64 >> lxb;
        const float *img = weights + V.pix_base;
        float m[16];
#pragma unroll
        for (int k = 0; k < 16; ++k) m[k] = 0.0f;
        for (int x = rx0 + lx; x <= rx1; x += 1 << lxb) {
            ColBase col;
            col_base(r, (float)x, col);
            F2 g0 = f2_dup(0.0f), a0 = g0, a1 = g0, a2 = g0, q0 = g0, q1 = g0, q2 = g0;
            for (int y = ry0 + 2 * ly; y <= ry1; y += row_step) {
                const bool two = y < ry1;   // else the pair's second row repeats the first with weight 0
                const float *p = img + (long long)y * W + x;
                const F2 wt = f2_pack(__ldg(p), two ? __ldg(p + W) : 0.0f);
                const F2 dy = f2_add(f2_pack((float)y, (float)(two ? y + 1 : y)), f2_dup(-r.py0));
                float dy0, dy1, sa[2], sq[2], w2[2], e[2];
                f2_unpack(dy, dy0, dy1);
                f2_unpack(pair_squares(r, col, dy0), sa[0], sq[0]);
                f2_unpack(pair_squares(r, col, dy1), sa[1], sq[1]);
                const F2 rs = f2_pack(rsqrt_approx(sa[0]), rsqrt_approx(sa[1])), rs2 = f2_mul(rs, rs);
                f2_unpack(rs2, w2[0], w2[1]);
                const F2 m2 = f2_pack(sq[0] * w2[0], sq[1] * w2[1]);
                f2_unpack(f2_fma(m2, f2_dup(-kHalfLog2e), f2_dup(r.q5.x)), e[0], e[1]);
                const F2 G = f2_mul(f2_mul(f2_pack(ex2_approx(e[0]), ex2_approx(e[1])), rs), wt);
                const F2 gq = f2_mul(G, rs2), ga = f2_mul(gq, f2_add(m2, f2_dup(-1.0f)));   // -2 dL/dq, 2 dL/da
                const F2 tq = f2_mul(gq, dy), ta = f2_mul(ga, dy);
                g0 = f2_add(g0, G);
                a0 = f2_add(a0, ga);
                a1 = f2_add(a1, ta);
                a2 = f2_fma(ta, dy, a2);
                q0 = f2_add(q0, gq);
                q1 = f2_add(q1, tq);
                q2 = f2_fma(tq, dy, q2);
            }
            const float A0 = f2_sum(a0), A1 = f2_sum(a1), Q0 = -f2_sum(q0), Q1 = -f2_sum(q1), dx = col.dx, xx = dx * dx;
            m[0] = fmaf(xx, A0, m[0]), m[1] = fmaf(xx, Q0, m[1]);
            m[2] = fmaf(dx, A1, m[2]), m[3] = fmaf(dx, Q1, m[3]);
            m[4] = fmaf(dx, A0, m[4]), m[5] = fmaf(dx, Q0, m[5]);
            m[6] += f2_sum(a2), m[7] -= f2_sum(q2);
            m[8] += A1, m[9] += Q1;
            m[10] += A0, m[11] += Q0;
            m[12] += f2_sum(g0);
        }
        const int k = warp_reduce_scatter_part<16, 4>(m, lane);
        m[0] += __shfl_xor_sync(0xffffffffu, m[0], 1);
        if ((lane & 1) == 0) acc[it * kGradN + k] = m[0];
    }
}

cudaError_t launch_cone_bwd(const ViewInfo *views_d, long long n_items, int n_per_view, const float4 *rec,
                            const short4 *prect, const float *weights, float *acc, cudaStream_t st, long long *launches) {
    if (n_items <= 0) return cudaSuccess;
    // several items a warp while that leaves four CTAs for every resident one
    const long long resident = 152LL * 3 * kConeWarps;
    const int per = (int)std::max<long long>(1, std::min<long long>(kConeItems, n_items / (4 * resident)));
    const long long b = (n_items + (long long)kConeWarps * per - 1) / ((long long)kConeWarps * per);
    pdl_launch(k_cone_bwd, (unsigned)b, 32 * kConeWarps, 0, st, views_d, n_items, per, n_per_view, rec, prect, weights, acc);
    *launches += 1;
    return cudaGetLastError();
}

}  // namespace vg
