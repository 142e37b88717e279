// Ray-marching reference of the volume rendering equation (Eq. 1) with the fields of Supp. A,
// sigma(x) = sum kappa_i G_i(x) and c(x) = sum c_i kappa_i G_i(x) / sigma(x), for measuring the
// blend's no-overlap approximation (Sec. 4.1) on the GPU: per pixel, NeRF's quadrature on
// midpoint samples t_k = t_near + (k + 1/2) delta of the unit ray from the camera centre,
//   C = sum_k T_k (1 - exp(-sigma_k delta)) c(x_k) + T bg,  T_k = exp(-delta sum_{j<k} sigma_j).
//
// Along a pixel's ray each Gaussian is a 1D Gaussian in t (Supp. B): with the record's
// d' = A u and o' x d' = C u (u = (dx, dy, 1)) and E = (o'.A0, o'.A1, o'.A2),
//   kappa G(o + t d) = kappa exp(-m^2/2) exp(-(t - gamma)^2 / (2 beta^2)),
//   m^2 = |C u|^2 / |A u|^2,  gamma = -(E . u) |d_c| / |A u|^2,  beta^2 = |d_c|^2 / |A u|^2,
// so a sample costs one FMA chain and one ex2 per (pixel, Gaussian).  The Gaussians near a pixel
// are those of its tile list whose footprint rectangle holds the pixel (every other one adds less
// than tau_cut to the ray's optical depth); the march needs no order.
//
// Samples are processed 16 at a time in registers (two per packed FP32 operation), each pass
// walking the tile's list (records staged in shared memory) and skipping Gaussians whose 1D
// Gaussian is below 2^-50 on the pass's samples: first per warp, by the footprint rectangle and by
// a range of t no ray can exceed, |t - |mu - o|| <= smax sqrt(2 ln(2^50 kappa)), then per pixel.
//
// What bounds it: issue, and before that the longest list.  One CTA per tile, one pixel per thread,
// walks its list once per pass; at 320 x 208 pixels (260 tiles) and 256 samples the passes of the
// longest list in sequence were the whole 2.80 ms.  With no early stop (T_stop = 0) the passes of a
// pixel are independent up to their transmittance, so they are spread over groups of CTAs, each
// leaving its colour and transmittance per pixel, which k_march_combine strings together.  A frame
// of that size and its march: 2.83 -> 0.39 ms (the march 2.80 -> 0.31 ms).
#include "blend.cuh"
#include "geometry.cuh"

namespace vg {

constexpr int kMarchS = 16;        // samples per pass
constexpr int kMarchChunk = 128;   // records per shared-memory chunk

// E = (o'.A0, o'.A1, o'.A2) of every visible item; w: the two ends, as FP16 rounded outwards, of the range of t
// outside of which no pixel's ray sees the Gaussian above 2^-50.
template <typename RT>
__global__ void __launch_bounds__(256)
k_march_prep(GaussIn g, const ViewInfo *__restrict__ views, long long n_items, const uint32_t *__restrict__ count,
             float4 *__restrict__ E) {
    pdl_entry();
    for (long long it = (long long)blockIdx.x * blockDim.x + threadIdx.x; it < n_items;
         it += (long long)gridDim.x * blockDim.x) {
        float4 e = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        if (count[it] != 0) {
            const int v = (int)(it / g.n);
            const long long gi = it - (long long)v * g.n;
            float mu[3], s[3], q[4], kin, Sig[9], Rq[9], qn[4], smax;
            load_gauss<RT>(g, gi, mu, s, q, kin);
            const Density dn = density_of(g, kin, s);
            if (key_cov(mu, s, q, dn.kap_key, Sig, Rq, qn, smax)) {
                ItemGeom G;
                item_geom(views[v], mu, s, Rq, G);
                e.x = G.op[0] * G.A[0] + G.op[1] * G.A[1] + G.op[2] * G.A[2];
                e.y = G.op[0] * G.A[3] + G.op[1] * G.A[4] + G.op[2] * G.A[5];
                e.z = G.op[0] * G.A[6] + G.op[1] * G.A[7] + G.op[2] * G.A[8];
                // |x - mu| <= smax m and |x - mu| >= |t - |mu - o|| for x = o + t d (1% and 1e-4 of slack)
                const float ox = mu[0] - views[v].of[0], oy = mu[1] - views[v].of[1], oz = mu[2] - views[v].of[2];
                const float dist = sqrtf(fmaf(ox, ox, fmaf(oy, oy, oz * oz)));
                const float smx = fmaxf(s[0], fmaxf(s[1], s[2]));
                const float room = log2f(dn.kap) + 50.01f;
                const float half = room > 0.0f ? fmaf(1.01f * smx, sqrtf(1.3862944f * room), 1e-4f * dist) : -INFINITY;
                e.w = __uint_as_float((uint32_t)__half_as_ushort(__float2half_rd(dist - half)) |
                                      ((uint32_t)__half_as_ushort(__float2half_ru(dist + half)) << 16));
            }
        }
        E[it] = e;
    }
}

struct MarchOut {
    const float *raster;     // image the error map compares with (NULL: none)
    float *rgb, *T, *err;    // each optional
    float bg0, bg1, bg2;
};

__device__ __forceinline__ void march_store(const MarchOut &o, long long pix, float T, float C0, float C1, float C2) {
    const float c0 = fmaf(T, o.bg0, C0), c1 = fmaf(T, o.bg1, C1), c2 = fmaf(T, o.bg2, C2);
    if (o.rgb) {
        o.rgb[3 * pix] = c0;
        o.rgb[3 * pix + 1] = c1;
        o.rgb[3 * pix + 2] = c2;
    }
    if (o.T) o.T[pix] = T;
    if (o.err && o.raster)
        o.err[pix] = fmaxf(fabsf(c0 - o.raster[3 * pix]),
                           fmaxf(fabsf(c1 - o.raster[3 * pix + 1]), fabsf(c2 - o.raster[3 * pix + 2])));
}

// One CTA per tile (longest list first) and group of consecutive passes; groups > 1 only with T_stop = 0, each group
// then starting from T = 1 and leaving (C, T) in part[group][pixel].
__global__ void __launch_bounds__(kMaxTilePix)
k_ray_march(const ViewInfo *__restrict__ views, const int *__restrict__ tile_view, const int *__restrict__ tile_order,
            const uint2 *__restrict__ ranges, const uint32_t *__restrict__ sorted_item, const float4 *__restrict__ rec,
            const float4 *__restrict__ E, const short4 *__restrict__ prect, float t_near, float delta, int n_samples,
            float T_stop, int groups, long long n_pixels, float4 *__restrict__ part, MarchOut out) {
    pdl_entry();
    __shared__ float4 srec[kMarchChunk * (kRecF4 + 1)];
    __shared__ short4 srect[kMarchChunk];
    __shared__ uint32_t srange[kMarchChunk];
    const int tile = tile_order[blockIdx.x / groups], group = (int)(blockIdx.x % groups);
    const ViewInfo &V = views[tile_view[tile]];
    const int local = tile - V.tile_base;
    const int tyi = local / V.tiles_x, txi = local - tyi * V.tiles_x;
    int ix, iy;
    PixLayout<1>::origin(threadIdx.x, V.tw, ix, iy);
    const int x = txi * V.tw + ix, y = tyi * V.th + iy, lane = threadIdx.x & 31;
    const WarpBox wb = warp_box<1>(x, y);
    const bool inside = x < V.W && y < V.H;
    const float xf = (float)x, yf = (float)y;
    const float pu = ((float)x + 0.5f - V.cx) / V.fx, pv = ((float)y + 0.5f - V.cy) / V.fy;
    const float dcn2 = fmaf(pu, pu, fmaf(pv, pv, 1.0f)), dcn = sqrtf(dcn2), hscale = kHalfLog2e / dcn2;
    const uint2 rg = ranges[tile];
    const int passes = (n_samples + kMarchS - 1) / kMarchS;
    const int pass0 = (int)((long long)passes * group / groups), pass1 = (int)((long long)passes * (group + 1) / groups);
    float T = 1.0f, C0 = 0.0f, C1 = 0.0f, C2 = 0.0f;
    bool live = inside;
    for (int k0 = pass0 * kMarchS; k0 < pass1 * kMarchS; k0 += kMarchS) {
        if (!__syncthreads_or(live)) break;
        F2 sg[kMarchS / 2], a0[kMarchS / 2], a1[kMarchS / 2], a2[kMarchS / 2];
#pragma unroll
        for (int s = 0; s < kMarchS / 2; ++s) sg[s] = a0[s] = a1[s] = a2[s] = f2_dup(0.0f);
        const float tk0 = fmaf((float)k0 + 0.5f, delta, t_near), tk1 = fmaf((float)(kMarchS - 1), delta, tk0);
        for (uint32_t base = rg.x; base < rg.y; base += kMarchChunk) {
            const int n = (int)min((uint32_t)kMarchChunk, rg.y - base);
            __syncthreads();
            for (int r = threadIdx.x; r < n; r += blockDim.x) {
                const uint32_t item = sorted_item[base + r];
#pragma unroll
                for (int c = 0; c < kRecF4; ++c) srec[r * (kRecF4 + 1) + c] = __ldg(rec + (size_t)item * kRecF4 + c);
                const float4 e = __ldg(E + item);
                srec[r * (kRecF4 + 1) + kRecF4] = e;
                srect[r] = prect[item];
                srange[r] = __float_as_uint(e.w);
            }
            __syncthreads();
            for (int w0 = 0; w0 < n; w0 += 32) {
                const int jl = w0 + lane;
                bool need = jl < n && !box_misses(wb, srect[jl]);
                if (need) {
                    const uint32_t w = srange[jl];
                    need = !(__half2float(__ushort_as_half((unsigned short)(w & 0xFFFFu))) > tk1 ||
                             __half2float(__ushort_as_half((unsigned short)(w >> 16))) < tk0);
                }
                unsigned m = __ballot_sync(0xffffffffu, need);
                while (m) {
                    const int j = w0 + __ffs(m) - 1;
                    m &= m - 1;
                    if (!live || pixel_outside(x, y, srect[j])) continue;
                    const float4 *rr = &srec[j * (kRecF4 + 1)];
                    RecPairs R;
                    load_rec(rr, R);
                    const float4 r5 = R.q5, e4 = rr[6];
                    ColBase col;
                    col_base(R, xf, col);
                    const float dx = col.dx, dy = yf - R.py0;
                    float a, qq;
                    f2_unpack(pair_squares(R, col, dy), a, qq);
                    const float bq = fmaf(e4.x, dx, fmaf(e4.y, dy, e4.z));
                    float ia = rcp_approx(a);   // and one Newton step, in place of the rounded division's dozen instructions
                    ia = fmaf(ia, fmaf(-a, ia, 1.0f), ia);
                    const float lp = fmaf(-qq * ia, kHalfLog2e, r5.x - kLog2Sqrt2Pi);   // log2(kappa exp(-m^2/2))
                    const float gam = -bq * dcn * ia;
                    const float h = hscale * a;                                          // log2(e) / (2 beta^2)
                    // largest value on [tk0, tk1]: 2^(lp - h off^2); the pass counts from 2^-50 on
                    const float off = fmaxf(fmaxf(tk0 - gam, gam - tk1), 0.0f);
                    if (!(fmaf(-off * off, h, lp) > -50.0f)) continue;
                    const F2 h2 = f2_dup(-h), lp2 = f2_dup(lp), d2v = f2_pack(2.0f * delta, 2.0f * delta);
                    const F2 tg = f2_pack(tk0 - gam, (tk0 - gam) + delta);
                    const F2 cr = f2_dup(r5.y), cg = f2_dup(r5.z), cb = f2_dup(r5.w);
#pragma unroll
                    for (int s = 0; s < kMarchS / 2; ++s) {
                        const F2 dt = f2_fma(f2_dup((float)s), d2v, tg);
                        const F2 ex = f2_fma(f2_mul(dt, dt), h2, lp2);
                        float e0, e1;
                        f2_unpack(ex, e0, e1);
                        const F2 v = f2_pack(ex2_approx(e0), ex2_approx(e1));
                        sg[s] = f2_add(sg[s], v);
                        a0[s] = f2_fma(cr, v, a0[s]);
                        a1[s] = f2_fma(cg, v, a1[s]);
                        a2[s] = f2_fma(cb, v, a2[s]);
                    }
                }
            }
        }
        if (live) {
#pragma unroll
            for (int s = 0; s < kMarchS; ++s) {
                if (k0 + s >= n_samples || !live) continue;
                float lo, hi, p0, p1, p2, t;
                f2_unpack(sg[s / 2], lo, hi);
                const float sig = s & 1 ? hi : lo;
                if (sig > 0.0f) {
                    f2_unpack(a0[s / 2], lo, hi), p0 = s & 1 ? hi : lo;
                    f2_unpack(a1[s / 2], lo, hi), p1 = s & 1 ? hi : lo;
                    f2_unpack(a2[s / 2], lo, hi), p2 = s & 1 ? hi : lo;
                    const float xs = sig * delta;
                    const float w = T * (-expm1f(-xs) / sig);   // T (1 - e^{-sigma delta}) / sigma
                    C0 = fmaf(w, p0, C0);
                    C1 = fmaf(w, p1, C1);
                    C2 = fmaf(w, p2, C2);
                    t = expf(-xs);
                    T *= t;
                }
                if (T < T_stop) live = false;
            }
        }
    }
    if (!inside) return;
    const long long pix = V.pix_base + (long long)y * V.W + x;
    if (groups > 1)
        part[(size_t)group * n_pixels + pix] = make_float4(C0, C1, C2, T);
    else
        march_store(out, pix, T, C0, C1, C2);
}

// C = sum_g T_1 .. T_(g-1) C_g, T = prod T_g over the groups of passes.
__global__ void __launch_bounds__(256)
k_march_combine(const float4 *__restrict__ part, int groups, long long n_pixels, MarchOut out) {
    pdl_entry();
    for (long long pix = (long long)blockIdx.x * blockDim.x + threadIdx.x; pix < n_pixels;
         pix += (long long)gridDim.x * blockDim.x) {
        float T = 1.0f, C0 = 0.0f, C1 = 0.0f, C2 = 0.0f;
        for (int g = 0; g < groups; ++g) {
            const float4 p = part[(size_t)g * n_pixels + pix];
            C0 = fmaf(T, p.x, C0);
            C1 = fmaf(T, p.y, C1);
            C2 = fmaf(T, p.z, C2);
            T *= p.w;
        }
        march_store(out, pix, T, C0, C1, C2);
    }
}

cudaError_t launch_ray_march(const GaussIn &g, const ViewInfo *views_d, const int *tile_view, const int *tile_order,
                             long long n_tiles, int tile_px, long long n_items, long long n_pixels,
                             const uint2 *ranges, const uint32_t *sorted_item, const float4 *rec,
                             const uint32_t *count, const short4 *prect, float4 *E, float t_near, float t_far,
                             int n_samples, float T_stop, int groups, float4 *part, const float bg[3],
                             const float *raster, float *rgb, float *T_out, float *err, cudaStream_t st,
                             long long *launches) {
    if (n_items > 0) {
        long long b = (n_items + 255) / 256;
        if (b > 152 * 32) b = 152 * 32;
        if (g.rec_dtype == VG_BF16)
            pdl_launch(k_march_prep<__nv_bfloat16>, (unsigned)b, 256, 0, st, g, views_d, n_items, count, E);
        else if (g.rec_dtype == VG_F16)
            pdl_launch(k_march_prep<__half>, (unsigned)b, 256, 0, st, g, views_d, n_items, count, E);
        else
            pdl_launch(k_march_prep<float>, (unsigned)b, 256, 0, st, g, views_d, n_items, count, E);
        *launches += 1;
    }
    if (n_tiles > 0) {
        const float delta = (t_far - t_near) / (float)n_samples;
        const int passes = (n_samples + kMarchS - 1) / kMarchS;
        if (groups > passes) groups = passes;
        const MarchOut out{raster, rgb, T_out, err, bg[0], bg[1], bg[2]};
        pdl_launch(k_ray_march, (unsigned)(n_tiles * groups), (unsigned)tile_px, 0, st, views_d, tile_view, tile_order,
                   ranges, sorted_item, rec, E, prect, t_near, delta, n_samples, T_stop, groups, n_pixels, part, out);
        *launches += 1;
        if (groups > 1) {
            long long b = (n_pixels + 255) / 256;
            if (b > 152 * 32) b = 152 * 32;
            pdl_launch(k_march_combine, (unsigned)b, 256, 0, st, part, groups, n_pixels, out);
            *launches += 1;
        }
    }
    return cudaGetLastError();
}

}  // namespace vg
