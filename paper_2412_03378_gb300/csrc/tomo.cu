// Tomography mode (Sec. 6.2, Eq. 21): parallel-beam projection proj = exp(-sum_g tau_g) of the
// same closed-form line integrals (Eq. 19), and its backward.
//
// For a parallel beam the ray direction d is fixed per angle, so per (angle, Gaussian) the
// line integral over the detector is an exact 2D Gaussian.  With W = S^-1 Rq^T the whitening,
// d' = W d and w_u = W e_u, w_v = W e_v, the whitened offset of the ray through detector pixel
// (i, j) from the centre is y = ((i - i_mu) pu (w_u x d') + (j - j_mu) pv (w_v x d')) / |d'|,
// a vector in the plane orthogonal to d'.  In the orthonormal basis (e1, e2) of that plane with e1
// along w_u x d' it is triangular, y = (l00 dx + l10 dy, l11 dy), and
//     tau = kappa sqrt(2 pi) / |d'| * exp(-|y|^2 / 2):
// the second component is constant along a detector row, and a pixel costs two packed FP32
// operations and one ex2.  Records hold l00, l10, l11 times sqrt(log2(e) / 2), so that
// log2 tau = log2 A - y0^2 - y1^2.
#include <algorithm>

#include "blend.cuh"
#include "geometry.cuh"

namespace vg {

// per-item accumulator: sum G, G y0, G y1, G y0^2, G y0 y1, G y1^2 (G = dL / dln tau, y scaled as in the
// record), 2 unused
constexpr int kTomoGradN = 8;
constexpr float kYScale = 0.84932180028801907f;   // sqrt(log2(e) / 2)

// Per-item tomography geometry (shared by the preprocess and the chain kernels).
struct TomoGeom {
    float W[9];          // row-major whitening S^-1 Rq^T
    float dp[3], wu[3], wv[3];
    float C0[3], C1[3];  // pu (w_u x d'), pv (w_v x d')
    float n;             // |d'|
    float e1[3], e2[3];  // C0 / |C0| and d' x C0 / (|d'| |C0|)
    float l00, l10, l11; // C0 / n = l00 e1, C1 / n = l10 e1 + l11 e2
    float imu, jmu;
};

__device__ __forceinline__ void tomo_geom(const float mu[3], const float s[3], const float Rq[9], float ct, float st,
                                          float pu, float pv, float u0, float v0, TomoGeom &G) {
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        const float is = 1.0f / s[i];
#pragma unroll
        for (int j = 0; j < 3; ++j) G.W[3 * i + j] = Rq[3 * j + i] * is;
        G.dp[i] = G.W[3 * i] * ct + G.W[3 * i + 1] * st;
        G.wu[i] = -G.W[3 * i] * st + G.W[3 * i + 1] * ct;
        G.wv[i] = G.W[3 * i + 2];
    }
    G.n = sqrtf(G.dp[0] * G.dp[0] + G.dp[1] * G.dp[1] + G.dp[2] * G.dp[2]);
    const float in = 1.0f / G.n;
    const float nn[3] = {G.dp[0] * in, G.dp[1] * in, G.dp[2] * in};
    float c0[3], c1[3];
    cross3(G.wu, nn, c0);
    cross3(G.wv, nn, c1);
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        c0[i] *= pu;
        c1[i] *= pv;
        G.C0[i] = c0[i] * G.n;
        G.C1[i] = c1[i] * G.n;
    }
    G.l00 = sqrtf(c0[0] * c0[0] + c0[1] * c0[1] + c0[2] * c0[2]);
    const float il = 1.0f / G.l00;
#pragma unroll
    for (int i = 0; i < 3; ++i) G.e1[i] = c0[i] * il;
    cross3(nn, G.e1, G.e2);
    G.l10 = c1[0] * G.e1[0] + c1[1] * G.e1[1] + c1[2] * G.e1[2];
    // C0 x C1 = pu pv det(W) d' with det(W) = 1 / (s0 s1 s2): the remaining factor without cancellation
    G.l11 = (pu / s[0]) * in * ((pv / s[1]) / (s[2] * G.l00));
    const float um = -st * mu[0] + ct * mu[1];
    G.imu = (um - u0) / pu - 0.5f;
    G.jmu = (mu[2] - v0) / pv - 0.5f;
}

__device__ __forceinline__ bool same_bits(const float4 &a, const float4 &b) {
    return __float_as_uint(a.x) == __float_as_uint(b.x) && __float_as_uint(a.y) == __float_as_uint(b.y) &&
           __float_as_uint(a.z) == __float_as_uint(b.z) && __float_as_uint(a.w) == __float_as_uint(b.w);
}

// ---------------------------------------------------------------------------- preprocess
// changed (may be NULL): set where a record or a count differs from what the buffers hold
template <typename RT>
__global__ void __launch_bounds__(256)
k_tomo_preprocess(GaussIn g, const float *__restrict__ cs, int n_angles, int det_w, int det_h, float pu, float pv,
                  float u0, float v0, float tau_cut, float4 *__restrict__ rec, uint32_t *__restrict__ count,
                  short4 *__restrict__ rect, uint32_t *__restrict__ changed) {
    pdl_entry();
    const long long n_items = (long long)g.n * n_angles;
    for (long long it = (long long)blockIdx.x * blockDim.x + threadIdx.x; it < n_items;
         it += (long long)gridDim.x * blockDim.x) {
        const int a = (int)(it / g.n);
        const long long gi = it - (long long)a * g.n;
        const float ct = cs[2 * a], st = cs[2 * a + 1];
        float mu[3], s[3], q[4], kin, Sig[9], Rq[9], qn[4], smax, k2;
        load_gauss<RT>(g, gi, mu, s, q, kin);
        const Density dn = density_of(g, kin, s);
        const float kap = dn.kap;
        short4 rc = make_short4(-1, -1, -1, -1);
        uint32_t cnt = 0;
        if (key_cov(mu, s, q, dn.kap_key, Sig, Rq, qn, smax) && key_k2(dn.kap_key, smax, tau_cut, k2)) {
            // key function: orthographic bounding box of the Mahalanobis-k ellipsoid (FP32, fixed order)
            const float um = VG_ADD(VG_MUL(-st, mu[0]), VG_MUL(ct, mu[1]));
            const float vm = mu[2];
            float suu = VG_ADD(VG_SUB(VG_MUL(VG_MUL(st, st), Sig[0]), VG_MUL(2.0f, VG_MUL(VG_MUL(st, ct), Sig[1]))),
                               VG_MUL(VG_MUL(ct, ct), Sig[4]));
            if (!(suu > 0.0f)) suu = 0.0f;
            const float svv = Sig[8];
            const float hu = VG_SQRT(VG_MUL(k2, suu)), hv = VG_SQRT(VG_MUL(k2, svv));
            const float xlo = VG_SUB(VG_DIV(VG_SUB(VG_SUB(um, hu), u0), pu), 0.5f);
            const float xhi = VG_SUB(VG_DIV(VG_SUB(VG_ADD(um, hu), u0), pu), 0.5f);
            const float ylo = VG_SUB(VG_DIV(VG_SUB(VG_SUB(vm, hv), v0), pv), 0.5f);
            const float yhi = VG_SUB(VG_DIV(VG_SUB(VG_ADD(vm, hv), v0), pv), 0.5f);
            int ix0, ix1, iy0, iy1;
            pixel_span(xlo, xhi, det_w, ix0, ix1);
            pixel_span(ylo, yhi, det_h, iy0, iy1);
            if (ix0 <= ix1 && iy0 <= iy1) {
                rc = make_short4((short)(ix0 / kTile), (short)(iy0 / kTile), (short)(ix1 / kTile), (short)(iy1 / kTile));
                cnt = (uint32_t)(rc.z - rc.x + 1) * (uint32_t)(rc.w - rc.y + 1);
                TomoGeom G;
                tomo_geom(mu, s, Rq, ct, st, pu, pv, u0, v0, G);
                const float lnA2 = log2f(kap) + kLog2Sqrt2Pi - log2f(G.n);
                // the pixel rectangle (< 65536 on both axes) rides in the record's last two words
                const float4 q0 = make_float4(G.imu, G.jmu, G.l00 * kYScale, G.l10 * kYScale);
                const float4 q1 = make_float4(G.l11 * kYScale, lnA2, __uint_as_float((unsigned)ix0 | (unsigned)ix1 << 16),
                                              __uint_as_float((unsigned)iy0 | (unsigned)iy1 << 16));
                if (changed && !(same_bits(rec[2 * it], q0) && same_bits(rec[2 * it + 1], q1))) *changed = 1u;
                rec[2 * it] = q0;
                rec[2 * it + 1] = q1;
            }
        }
        if (changed && count[it] != cnt) *changed = 1u;
        count[it] = cnt;
        if (rect) rect[it] = rc;
    }
}

cudaError_t launch_tomo_preprocess(const GaussIn &g, const float *cs_d, int n_angles, int det_w, int det_h,
                                   float pitch_u, float pitch_v, float u0, float v0, float tau_cut, float4 *rec,
                                   uint32_t *count, short4 *rect, uint32_t *changed, cudaStream_t st,
                                   long long *launches) {
    const long long n_items = (long long)g.n * n_angles;
    long long b = (n_items + 255) / 256;
    if (b > 152 * 32) b = 152 * 32;
    if (b < 1) b = 1;
    *launches += 1;
    if (g.rec_dtype == VG_BF16)
        pdl_launch(k_tomo_preprocess<__nv_bfloat16>, (unsigned)b, 256, 0, st, g, cs_d, n_angles, det_w, det_h, pitch_u, pitch_v,
                                                                      u0, v0, tau_cut, rec, count, rect, changed);
    else if (g.rec_dtype == VG_F16)
        pdl_launch(k_tomo_preprocess<__half>, (unsigned)b, 256, 0, st, g, cs_d, n_angles, det_w, det_h, pitch_u, pitch_v, u0,
                                                               v0, tau_cut, rec, count, rect, changed);
    else
        pdl_launch(k_tomo_preprocess<float>, (unsigned)b, 256, 0, st, g, cs_d, n_angles, det_w, det_h, pitch_u, pitch_v, u0,
                                                              v0, tau_cut, rec, count, rect, changed);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------- projector
// One warp per detector tile (four independent warps per CTA): lane l owns the 2 x 4 pixels from
// (2 (l % 8), 4 (l / 8)) of the tile and sums them over the tile's list, 32 records staged at a time in
// the warp's part of shared memory.  Bound by issue slots and the ex2 unit (8 ex2 = 32 cycles of a
// sub-partition's 8 lanes per visit): pairs are packed over two rows, whose shared terms (l10 dy, y1^2 -
// log2 A) are formed once for the lane's two columns, and the coefficients a pair needs twice are
// staged twice, so that no instruction duplicates them.  Every listed record touches the tile; a tile
// that is not entirely inside the record's pixel rectangle puts the pixels outside at y0 = kFar,
// where tau is exactly 0.  200,000 Gaussians, 64 angles, 512 x 512 detectors (264 M visits): 17.7 ms
// against 30.3 ms for 2 x 2 pixels per lane, two warps per tile and scalar operations.  1 or 2 warps per
// CTA 17.4 / 17.9 ms there, but 4% slower on 8,000 Gaussians; 40 warps per SM (51 registers) 19.1 ms.
constexpr int kProjWarps = 4;
constexpr float kFar = 1e15f;   // y^2 stays finite

struct __align__(16) TomoRec {   // a staged record
    float imu, l00;
    unsigned in, pad;         // the tile's columns (bits 0..15) and rows (16..31) inside the pixel rectangle
    F2 njmu, l10, l11, nlnA;  // -j_mu, l10, l11, -log2 A, twice each
};

// bits max(first, 0) .. min(last, 15)
__device__ __forceinline__ unsigned span_bits(int first, int last) {
    const int a = max(first, 0), b = min(last, kTile - 1);
    return b < a ? 0u : ((2u << b) - 1u) & ~((1u << a) - 1u);
}

__device__ __forceinline__ TomoRec tomo_stage(const float4 &r0, const float4 &r1, int tx0, int ty0) {
    TomoRec t;
    t.imu = r0.x;
    t.l00 = r0.z;
    const unsigned rx = __float_as_uint(r1.z), ry = __float_as_uint(r1.w);
    t.in = span_bits((int)(rx & 0xffffu) - tx0, (int)(rx >> 16) - tx0) |
           span_bits((int)(ry & 0xffffu) - ty0, (int)(ry >> 16) - ty0) << 16;
    t.pad = 0u;
    t.njmu = f2_dup(-r0.y);
    t.l10 = f2_dup(r0.w);
    t.l11 = f2_dup(r1.x);
    t.nlnA = f2_dup(-r1.y);
    return t;
}

__global__ void __launch_bounds__(32 * kProjWarps, 8)
k_tomo_fwd(const uint2 *__restrict__ ranges, long long n_tiles, int tiles_x, int tiles_per_view, int det_w, int det_h,
           const uint32_t *__restrict__ sorted_item, const float4 *__restrict__ rec, float *__restrict__ proj) {
    pdl_entry();
    __shared__ TomoRec stage[kProjWarps][32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const long long tile = (long long)blockIdx.x * kProjWarps + w;
    if (tile >= n_tiles) return;
    const int view = (int)(tile / tiles_per_view), local = (int)(tile - (long long)view * tiles_per_view);
    const int ty = local / tiles_x, tx = local - ty * tiles_x;
    const int x0 = tx * kTile + 2 * (lane & 7), y0 = ty * kTile + 4 * (lane >> 3);
    const float xf = (float)x0, yf = (float)y0;
    const F2 ya = f2_pack(yf, yf + 1.0f), yb = f2_pack(yf + 2.0f, yf + 3.0f);
    const unsigned cbit = 1u << (2 * (lane & 7)), rbit = 1u << (16 + 4 * (lane >> 3));
    const uint2 rg = ranges[tile];
    F2 sum[2][2];   // [column][row pair]
#pragma unroll
    for (int k = 0; k < 4; ++k) sum[k >> 1][k & 1] = f2_dup(0.0f);
    float4 p0 = make_float4(0.0f, 0.0f, 0.0f, 0.0f), p1 = p0;   // the next chunk's record of this lane
    if (rg.x + lane < rg.y) {
        const float4 *src = rec + 2 * (size_t)sorted_item[rg.x + lane];
        p0 = __ldg(src);
        p1 = __ldg(src + 1);
    }
    for (uint32_t base = rg.x; base < rg.y; base += 32) {
        const int n = (int)min(32u, rg.y - base);
        __syncwarp();
        stage[w][lane] = tomo_stage(p0, p1, tx * kTile, ty * kTile);
        if (base + 32 + lane < rg.y) {
            const float4 *src = rec + 2 * (size_t)sorted_item[base + 32 + lane];
            p0 = __ldg(src);
            p1 = __ldg(src + 1);
        }
        __syncwarp();
#pragma unroll 2
        for (int j = 0; j < n; ++j) {
            const TomoRec r = stage[w][j];
            const float dx = xf - r.imu;
            float b[2] = {r.l00 * dx, fmaf(r.l00, dx, r.l00)};
            F2 Lc[2], wc[2];   // y1^2 - log2 A and l10 dy of the two row pairs
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const F2 dy = f2_add(h ? yb : ya, r.njmu);
                const F2 v = f2_mul(r.l11, dy);
                wc[h] = f2_mul(r.l10, dy);
                Lc[h] = f2_fma(v, v, r.nlnA);
            }
            if (r.in != 0xffffffffu) {   // not the whole tile
                if (!(r.in & cbit)) b[0] = kFar;
                if (!(r.in & (cbit << 1))) b[1] = kFar;
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    float l0, l1;
                    f2_unpack(Lc[h], l0, l1);
                    if (!(r.in & (rbit << (2 * h)))) l0 = kFar;
                    if (!(r.in & (rbit << (2 * h + 1)))) l1 = kFar;
                    Lc[h] = f2_pack(l0, l1);
                }
            }
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                const F2 bc = f2_dup(b[c]);
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const F2 y = f2_add(bc, wc[h]);
                    float a0, a1;
                    f2_unpack(f2_fma(y, y, Lc[h]), a0, a1);
                    sum[c][h] = f2_add(sum[c][h], f2_pack(ex2_approx(-a0), ex2_approx(-a1)));
                }
            }
        }
    }
#pragma unroll
    for (int c = 0; c < 2; ++c)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            float s[2];
            f2_unpack(sum[c][h], s[0], s[1]);
            const int x = x0 + c;
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                const int y = y0 + 2 * h + k;
                if (x < det_w && y < det_h) proj[((long long)view * det_h + y) * det_w + x] = ex2_approx(-kLog2eF * s[k]);
            }
        }
}

cudaError_t launch_tomo_fwd(const uint2 *ranges, long long n_tiles, int tiles_x, int tiles_per_view, int det_w,
                            int det_h, const uint32_t *sorted_item, const float4 *rec, float *proj, cudaStream_t st,
                            long long *launches) {
    if (n_tiles <= 0) return cudaSuccess;
    pdl_launch(k_tomo_fwd, (unsigned)((n_tiles + kProjWarps - 1) / kProjWarps), 32 * kProjWarps, 0, st, ranges, n_tiles,
               tiles_x, tiles_per_view, det_w, det_h, sorted_item, rec, proj);
    *launches += 1;
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------- backward
// proj = exp(-sum tau)  =>  dL/dtau = -proj dL/dproj for every Gaussian on the ray, whatever the
// order: the weights of the pixels, written once as an image of 16-byte aligned rows.
__global__ void __launch_bounds__(256)
k_tomo_weights(const float *__restrict__ proj, const float *__restrict__ dL, const float *__restrict__ target,
               float scale, float *__restrict__ loss, long long rows, int det_w, int pitch, float *__restrict__ out) {
    pdl_entry();
    float acc = 0.0f;
    for (long long y = blockIdx.x; y < rows; y += gridDim.x) {
        const float *p = proj + y * det_w, *d = (dL ? dL : target) + y * det_w;
        for (int x = threadIdx.x; x < pitch; x += blockDim.x) {
            float g = 0.0f;
            if (x < det_w) {
                if (dL) {
                    g = -p[x] * d[x];
                } else {
                    const float e = p[x] - d[x];
                    g = -p[x] * (2.0f * scale * e);
                    acc = fmaf(e, e, acc);
                }
            }
            if (out) out[y * pitch + x] = g;
        }
    }
    if (dL) return;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    __shared__ float ws[8];
    if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        float t = 0.0f;
        for (int k = 0; k < 8; ++k) t += ws[k];
        atomicAdd(loss, t * scale);
    }
}

cudaError_t launch_tomo_weights(const float *proj, const float *dL, const float *target, float scale, float *loss,
                                int n_views, int det_w, int det_h, float *weights, cudaStream_t st,
                                long long *launches) {
    const long long rows = (long long)n_views * det_h;
    const long long b = rows < 152 * 16 ? rows : 152 * 16;
    if (b < 1) return cudaSuccess;
    pdl_launch(k_tomo_weights, (unsigned)b, 256, 0, st, proj, dL, target, scale, loss, rows, det_w, tomo_pitch(det_w), weights);
    *launches += 1;
    return cudaGetLastError();
}

// Where the image of weights cannot be had (a fixed-capacity workspace whose buffer is smaller, no memory) a weight is
// formed where it is used, by the same operations: one value of proj and one of dL (or target) per pixel and item, unaligned.
struct TomoDirect {
    const float *proj, *dL, *target;   // dL NULL: the L2 loss against target
    float scale;
    __device__ float operator()(long long i) const {
        if (dL) return -proj[i] * dL[i];
        const float e = proj[i] - target[i];
        return -proj[i] * (2.0f * scale * e);
    }
};

// One warp per (angle, Gaussian) item: the sum over its pixels needs neither the tile lists nor their
// order, so a warp walks the item's own pixel rectangle and writes its six sums once -- no
// reduction per (tile, Gaussian), no atomics, and no pixels of half-covered tiles.  With G = dL/dln tau =
// weight tau the partials of ln tau = ln A - |y|^2 / 2 follow from sum G, G y and G y y^T in the
// whitened coordinates, where they are well conditioned for any elongation.  A lane owns eight pixel
// columns (two 16-byte loads per row, requested a row ahead; columns left or right of the rectangle sit
// at y0 = kFar, where tau is 0; only an item whose sums come out not finite is summed again with their weights masked,
// which costs 1.6% here against 7% for masking every row) and every LY-th row, so that a row's shared terms and sums serve
// eight pixels; 1, 2 or 4 lanes stand side by side, as the rectangle is wide.  The loop is bound by the
// FMA pipe (a packed instruction holds it for two cycles): about 65 cycles per row of eight pixels.
// A warp's items are requested together (one per lane) before the first is summed.  On the workload above 23.7 ms (chain
// included) against 62.4 ms for one reduction per (tile, Gaussian) in tile order; at 1 / 2 / 4 / 8 / 32 items a warp 30.8 /
// 27.3 / 25.3 / 24.2 / 23.7 ms, at 2 or 4 CTAs per SM 25-29 ms.  Taking the items by the place of their footprints, so
// that a CTA's warps share rows of the weights, is worth nothing at 16 items a warp: 23.7 ms there, and with its sort
// 3% slower at 256 x 256 (1.19 -> 1.22 ms, 50,000 Gaussians), 17% at 200 x 200 (133 -> 156 us, 8,000).
constexpr int kTomoBwdWarps = 8, kTomoBwdCtas = 3;   // warps per CTA, CTAs per SM
constexpr int kTomoBwdItems = 16;                    // items of a warp, at most

template <bool DIRECT>   // pitch: floats from row to row of the weights, or of proj and dL
__global__ void __launch_bounds__(32 * kTomoBwdWarps, kTomoBwdCtas)
k_tomo_bwd(long long n_items, int per_warp, int n_per_view, int det_h, int pitch, const uint32_t *__restrict__ count,
           const float4 *__restrict__ rec, const float *__restrict__ weights, TomoDirect direct,
           float *__restrict__ acc) {
    pdl_entry();
    const int lane = threadIdx.x & 31;
    const long long at0 = (long long)blockIdx.x * kTomoBwdWarps * per_warp + (threadIdx.x >> 5);
    long long my_it = -1;
    float4 my0 = make_float4(0.0f, 0.0f, 0.0f, 0.0f), my1 = my0;
    unsigned my_count = 0;
    if (lane < per_warp && at0 + lane * kTomoBwdWarps < n_items) {
        my_it = at0 + lane * kTomoBwdWarps;
        my_count = count[my_it];
        if (my_count) {
            my0 = __ldg(rec + 2 * my_it);
            my1 = __ldg(rec + 2 * my_it + 1);
        } else {
            float4 *dst = reinterpret_cast<float4 *>(acc + my_it * kTomoGradN);
            dst[0] = dst[1] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        }
    }
    for (unsigned todo = __ballot_sync(0xffffffffu, my_count != 0); todo; todo &= todo - 1) {
        const int from = __ffs(todo) - 1;
        const long long it = __shfl_sync(0xffffffffu, my_it, from);
        const float4 r0 = make_float4(__shfl_sync(0xffffffffu, my0.x, from), __shfl_sync(0xffffffffu, my0.y, from),
                                      __shfl_sync(0xffffffffu, my0.z, from), __shfl_sync(0xffffffffu, my0.w, from));
        const float2 r1 = make_float2(__shfl_sync(0xffffffffu, my1.x, from), __shfl_sync(0xffffffffu, my1.y, from));
        const unsigned rx = __float_as_uint(__shfl_sync(0xffffffffu, my1.z, from));
        const unsigned ry = __float_as_uint(__shfl_sync(0xffffffffu, my1.w, from));
        const int rx0 = (int)(rx & 0xffffu), rx1 = (int)(rx >> 16), ry0 = (int)(ry & 0xffffu), ry1 = (int)(ry >> 16);
        const long long img0 = (it / n_per_view) * (long long)det_h * pitch;
        const float *img = weights + img0;
        const int o0 = rx0 >> 3, o1 = rx1 >> 3;
        const int lxb = min(o1 - o0, 2);   // log2 of the lanes side by side
        const int lx = lane & ((1 << lxb) - 1), ly = lane >> lxb, LY = 32 >> lxb;
        const float LYf = (float)LY;
        float m0, n0, n1, m01, m11;
        F2 m00;
        auto sum_up = [&](auto mask_columns) {
            m0 = n0 = n1 = m01 = m11 = 0.0f;
            m00 = f2_dup(0.0f);
            for (int o = o0 + lx; o <= o1; o += 1 << lxb) {
                F2 b[4];
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    const int x = 8 * o + 2 * c;
                    b[c] = f2_pack((x < rx0 || x > rx1) ? kFar : r0.z * ((float)x - r0.x),
                                   (x + 1 < rx0 || x + 1 > rx1) ? kFar : r0.z * ((float)(x + 1) - r0.x));
                }
                const float4 *src = reinterpret_cast<const float4 *>(img + (long long)(ry0 + ly) * pitch + 8 * o);
                float yf = (float)(ry0 + ly);
                float4 na = make_float4(0.0f, 0.0f, 0.0f, 0.0f), nb = na;
                if (!DIRECT && ry0 + ly <= ry1) {
                    na = __ldg(src);
                    nb = __ldg(src + 1);
                }
                for (int y = ry0 + ly; y <= ry1; y += LY) {
                    F2 g[4] = {f2_pack(na.x, na.y), f2_pack(na.z, na.w), f2_pack(nb.x, nb.y), f2_pack(nb.z, nb.w)};
                    if constexpr (DIRECT || mask_columns) {
#pragma unroll
                        for (int c = 0; c < 4; ++c) {
                            const int x = 8 * o + 2 * c;
                            const bool in0 = x >= rx0 && x <= rx1, in1 = x + 1 >= rx0 && x + 1 <= rx1;
                            float w0, w1;
                            f2_unpack(g[c], w0, w1);
                            if constexpr (DIRECT) {
                                const long long i = img0 + (long long)y * pitch + x;
                                w0 = in0 ? direct(i) : 0.0f;
                                w1 = in1 ? direct(i + 1) : 0.0f;
                            }
                            g[c] = f2_pack(in0 ? w0 : 0.0f, in1 ? w1 : 0.0f);
                        }
                    }
                    src += (size_t)(LY * (pitch >> 2));
                    if (!DIRECT && y + LY <= ry1) {
                        na = __ldg(src);
                        nb = __ldg(src + 1);
                    }
                    const float dy = yf - r0.y;
                    yf += LYf;
                    const float v = r1.x * dy;
                    const F2 wd = f2_dup(r0.w * dy), Ld = f2_dup(fmaf(v, v, -r1.y));
                    F2 G[4], u[4];
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        const F2 yc = f2_add(b[c], wd);
                        float a0, a1;
                        f2_unpack(f2_fma(yc, yc, Ld), a0, a1);
                        G[c] = f2_mul(g[c], f2_pack(ex2_approx(-a0), ex2_approx(-a1)));
                        u[c] = f2_mul(G[c], yc);
                        m00 = f2_fma(u[c], yc, m00);
                    }
                    const float Gs = f2_sum(f2_add(f2_add(G[0], G[1]), f2_add(G[2], G[3])));
                    const float us = f2_sum(f2_add(f2_add(u[0], u[1]), f2_add(u[2], u[3])));
                    const float tv = v * Gs;
                    m0 += Gs;
                    n0 += us;
                    n1 += tv;
                    m01 = fmaf(v, us, m01);
                    m11 = fmaf(v, tv, m11);
                }
            }
        };
        sum_up(std::false_type());
        // a weight that is not finite makes 0 x weight of a column outside the rectangle NaN: sum again without them
        if (!DIRECT && __any_sync(0xffffffffu, !isfinite(m0))) sum_up(std::true_type());
        float v[kTomoGradN] = {m0, n0, n1, f2_sum(m00), m01, m11, 0.0f, 0.0f};
        const int k = warp_reduce_scatter_part<kTomoGradN, 3>(v, lane);
        v[0] += __shfl_xor_sync(0xffffffffu, v[0], 2);
        v[0] += __shfl_xor_sync(0xffffffffu, v[0], 1);
        if ((lane & 3) == 0) acc[it * kTomoGradN + k] = v[0];
    }
}

cudaError_t launch_tomo_bwd(long long n_items, int n_per_view, int det_w, int det_h, const uint32_t *count,
                            const float4 *rec, const float *weights, const float *proj, const float *dL,
                            const float *target, float scale, float *acc, cudaStream_t st,
                            long long *launches) {
    if (n_items <= 0) return cudaSuccess;
    // several items a warp while that leaves four CTAs for every resident one
    const long long resident = 152 * kTomoBwdCtas * kTomoBwdWarps;
    const int per = (int)std::max<long long>(1, std::min<long long>(kTomoBwdItems, n_items / (4 * resident)));
    const long long b = (n_items + (long long)kTomoBwdWarps * per - 1) / ((long long)kTomoBwdWarps * per);
    const TomoDirect direct{proj, dL, target, scale};
    if (weights)
        pdl_launch(k_tomo_bwd<false>, (unsigned)b, 32 * kTomoBwdWarps, 0, st, n_items, per, n_per_view, det_h, tomo_pitch(det_w),
                   count, rec, weights, direct, acc);
    else
        pdl_launch(k_tomo_bwd<true>, (unsigned)b, 32 * kTomoBwdWarps, 0, st, n_items, per, n_per_view, det_h, det_w, count, rec,
                   weights, direct, acc);
    *launches += 1;
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------- chain
template <typename RT>
__global__ void __launch_bounds__(128)
k_tomo_chain(GaussIn g, const float *__restrict__ cs, int n_angles, long long item0, long long n_items, float pu,
             float pv, float u0, float v0, const float *__restrict__ grad_acc, float *__restrict__ dmu,
             float *__restrict__ dscale, float *__restrict__ dquat, float *__restrict__ dkappa) {
    pdl_entry();
    (void)n_angles;
    for (long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x; k < n_items;
         k += (long long)gridDim.x * blockDim.x) {
        const float4 a4 = *(const float4 *)(grad_acc + k * kTomoGradN);
        const float4 b4 = *(const float4 *)(grad_acc + k * kTomoGradN + 4);
        if (a4.x == 0.0f && a4.y == 0.0f && a4.z == 0.0f && a4.w == 0.0f && b4.x == 0.0f && b4.y == 0.0f) continue;
        const long long it = item0 + k;
        const int a = (int)(it / g.n);
        const long long gi = it - (long long)a * g.n;
        const float ct = cs[2 * a], st = cs[2 * a + 1];
        float mu[3], s[3], q[4], kin, Sig[9], Rq[9], qn[4], smax;
        load_gauss<RT>(g, gi, mu, s, q, kin);
        const Density dns = density_of(g, kin, s);
        const float kap = dns.kap;
        if (!key_cov(mu, s, q, dns.kap_key, Sig, Rq, qn, smax)) continue;
        TomoGeom G;
        tomo_geom(mu, s, Rq, ct, st, pu, pv, u0, v0, G);
        // the sums in unscaled y: dL/dc_k = -sum G y d_k with dx = (y0 - (l10 / l11) y1) / l00, dy = y1 / l11
        constexpr float kS1 = 1.0f / kYScale, kS2 = 1.0f / (kYScale * kYScale);
        const float S00 = a4.w * kS2, S01 = b4.x * kS2, S11 = b4.y * kS2;
        const float i0 = 1.0f / G.l00, i1 = 1.0f / G.l11, lr = G.l10 * i1;
        const float dc0[2] = {-(S00 - lr * S01) * i0, -(S01 - lr * S11) * i0}, dc1[2] = {-S01 * i1, -S11 * i1};
        const float dys[2] = {-a4.y * kS1, -a4.z * kS1};
        const float dlnA = a4.x;
        // c_k = (C_k . e) / n (2D, in the plane orthogonal to d'); lnA = ln(kappa sqrt(2pi)) - ln n
        const float in = 1.0f / G.n;
        float gC0[3], gC1[3];
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            gC0[i] = (dc0[0] * G.e1[i] + dc0[1] * G.e2[i]) * in;
            gC1[i] = (dc1[0] * G.e1[i] + dc1[1] * G.e2[i]) * in;
        }
        const float dn = -(gC0[0] * G.C0[0] + gC0[1] * G.C0[1] + gC0[2] * G.C0[2] + gC1[0] * G.C1[0] +
                           gC1[1] * G.C1[1] + gC1[2] * G.C1[2]) * in - dlnA * in;
        float gdp[3], gwu[3], gwv[3];
#pragma unroll
        for (int i = 0; i < 3; ++i) gdp[i] = dn * G.dp[i] * in;
        // C0 = pu (w_u x d'), C1 = pv (w_v x d')
        float t[3];
        cross3(gC0, G.wu, t);
#pragma unroll
        for (int i = 0; i < 3; ++i) gdp[i] += pu * t[i];
        cross3(gC1, G.wv, t);
#pragma unroll
        for (int i = 0; i < 3; ++i) gdp[i] += pv * t[i];
        cross3(G.dp, gC0, gwu);
        cross3(G.dp, gC1, gwv);
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            gwu[i] *= pu;
            gwv[i] *= pv;
        }
        // d' = W d, w_u = W e_u, w_v = W e_v with d = (ct, st, 0), e_u = (-st, ct, 0), e_v = (0, 0, 1)
        float dW[9];
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            dW[3 * i + 0] = gdp[i] * ct - gwu[i] * st;
            dW[3 * i + 1] = gdp[i] * st + gwu[i] * ct;
            dW[3 * i + 2] = gwv[i];
        }
        // W[i][j] = Rq[j][i] / s_i
        float dsc[3], dR[9];
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            const float is = 1.0f / s[i];
            dsc[i] = -(dW[3 * i] * G.W[3 * i] + dW[3 * i + 1] * G.W[3 * i + 1] + dW[3 * i + 2] * G.W[3 * i + 2]) * is;
#pragma unroll
            for (int j = 0; j < 3; ++j) dR[3 * j + i] = dW[3 * i + j] * is;
        }
        const float w = qn[0], x = qn[1], y = qn[2], z = qn[3];
        float dqn[4];
        dqn[0] = 2.0f * (-z * dR[1] + y * dR[2] + z * dR[3] - x * dR[5] - y * dR[6] + x * dR[7]);
        dqn[1] = 2.0f * (y * dR[1] + z * dR[2] + y * dR[3] - 2.0f * x * dR[4] - w * dR[5] + z * dR[6] + w * dR[7] -
                         2.0f * x * dR[8]);
        dqn[2] = 2.0f * (-2.0f * y * dR[0] + x * dR[1] + w * dR[2] + x * dR[3] + z * dR[5] - w * dR[6] + z * dR[7] -
                         2.0f * y * dR[8]);
        dqn[3] = 2.0f * (-2.0f * z * dR[0] - w * dR[1] + x * dR[2] + w * dR[3] - 2.0f * z * dR[4] + y * dR[5] +
                         x * dR[6] + y * dR[7]);
        const float qnorm = sqrtf(q[0] * q[0] + q[1] * q[1] + q[2] * q[2] + q[3] * q[3]);
        const float dot = qn[0] * dqn[0] + qn[1] * dqn[1] + qn[2] * dqn[2] + qn[3] * dqn[3];
        // i_mu = (e_u . mu - u0)/pu - 1/2, j_mu = (mu_z - v0)/pv - 1/2; dL/di_mu = -c0 . sum dL/dy
        const float gi_mu = -(G.l00 * dys[0]);
        const float gj_mu = -(G.l10 * dys[0] + G.l11 * dys[1]);
        const float dm[3] = {-st * gi_mu / pu, ct * gi_mu / pu, gj_mu / pv};
        float dk = dlnA / kap;   // dL/dkappa; with Eq. 20 it becomes dL/dtheta plus a share of dL/ds
        if (g.density_theta) {
#pragma unroll
            for (int c = 0; c < 3; ++c) dsc[c] -= dk * dns.lnv / (3.0f * s[c] * s[c]);
            dk = dk * 0.99f / (1.0f - 0.99f * kin) * dns.m;
        }
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            atomicAdd(&dmu[3 * gi + c], dm[c]);
            atomicAdd(&dscale[3 * gi + c], dsc[c]);
        }
#pragma unroll
        for (int c = 0; c < 4; ++c) atomicAdd(&dquat[4 * gi + c], (dqn[c] - qn[c] * dot) / qnorm);
        atomicAdd(&dkappa[gi], dk);
    }
}

cudaError_t launch_tomo_chain(const GaussIn &g, const float *cs_d, int n_angles, long long item0, long long n_items,
                              float pitch_u, float pitch_v, float u0, float v0, const float *grad_acc, float *dmu,
                              float *dscale, float *dquat, float *dkappa, cudaStream_t st, long long *launches) {
    long long b = (n_items + 127) / 128;
    if (b > 152 * 32) b = 152 * 32;
    if (b < 1) b = 1;
    *launches += 1;
    if (g.rec_dtype == VG_BF16)
        pdl_launch(k_tomo_chain<__nv_bfloat16>, (unsigned)b, 128, 0, st, g, cs_d, n_angles, item0, n_items, pitch_u, pitch_v, u0,
                                                                 v0, grad_acc, dmu, dscale, dquat, dkappa);
    else if (g.rec_dtype == VG_F16)
        pdl_launch(k_tomo_chain<__half>, (unsigned)b, 128, 0, st, g, cs_d, n_angles, item0, n_items, pitch_u, pitch_v, u0, v0,
                                                          grad_acc, dmu, dscale, dquat, dkappa);
    else
        pdl_launch(k_tomo_chain<float>, (unsigned)b, 128, 0, st, g, cs_d, n_angles, item0, n_items, pitch_u, pitch_v, u0, v0,
                                                         grad_acc, dmu, dscale, dquat, dkappa);
    return cudaGetLastError();
}

}  // namespace vg
