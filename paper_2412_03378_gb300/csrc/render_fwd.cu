// Front-to-back blend of the depth-sorted per-tile lists (Eq. 14 with the Eq. 19 alpha).
//
// One CTA per tile (16 x 16, 32 x 16 or 16 x 8 pixels), tiles taken longest list first; each of
// the tw th / P threads owns P pixels (P = 1, 2, 4).  Records of the tile's Gaussians are staged through shared memory in
// depth-ordered chunks (one record per thread); every record is read once per thread and
// serves its P pixels, which share the record's per-column inner terms (col_base: the pixels
// of a thread lie in one or two columns).  The closed form is evaluated in FP32 (FMA pipe + 3 MUFU ops per pair); the CTA
// leaves once all of its pixels have reached T < T_stop.  The per-pixel update is branch-free: a
// pixel that does not blend the visited Gaussian (finished, outside the image or the footprint,
// or below the skip threshold) takes tau = 0 (alpha = 0), which leaves its colour, T and S
// unchanged bit for bit (0.247 ms against 0.270 ms with per-pixel branches).  Issue slots bound it, so
// the operations are packed two to an instruction: d' with o' x d' (RecPairs) and, with two rows per
// thread, the pixels' own chains (1M Gaussians, 1280 x 832: 0.255 -> 0.235 ms).  SPLAT selects the 3DGS comparison
// mode's alpha (Eq. 6) in the same loop, on records of half the size.  No tensor cores: the work is not a
// dense contraction.
#include "blend.cuh"

namespace vg {

// Records evaluated together with one pixel per thread, the form for few tiles, whose time is the longest list's chain of
// dependent instructions.  1,040 tiles (100,000 Gaussians) at 1 / 2 / 3 / 4: 116.8 / 99.7 / 98.1 / 95.9 us.  With two
// pixels per thread one record at a time, and two where every footprint pixel counts (3,584 tiles, no skip: 926 / 812 us;
// with the skip's shorter visits 229 / 235 us on the 1M-Gaussian 1280 x 832 workload).
constexpr int kIlp = 4;
// volumetric blend, the 3DGS comparison mode, cone-beam projection (rgb NULL, nothing skipped, clamped or stopped)
constexpr int kModeBlend = 0, kModeSplat = 1, kModeCone = 2;

// One CTA of tw th / P threads per tile (with P = 1, `split` CTAs of as many threads in all, see
// tile_split).  The register cap is that of 3 / 7 / 12 CTAs of a 16 x 16 tile per SM for P = 1 / 2 / 4 (the occupancy measured fastest), whatever the tile shape.
template <int P, bool COUNT, bool PIXTEST, int MODE, int CH>
__global__ void __maxnreg__(PixLayout<P>::kFwdRegs)
k_render_fwd(const ViewInfo *__restrict__ views, const int *__restrict__ tile_view, const int *__restrict__ tile_order,
             const uint2 *__restrict__ ranges, const uint32_t *__restrict__ sorted_item, const float4 *__restrict__ rec,
             const short4 *__restrict__ prect, BlendParams bp, float *__restrict__ rgb, float *__restrict__ T_user, float *__restrict__ T_ws,
             float *__restrict__ S_out, uint32_t *__restrict__ nlast_out, uint32_t *__restrict__ tile_replay,
             unsigned long long *__restrict__ pair_count, L2Fused l2, int split) {
    pdl_entry();
    using L = PixLayout<P>;
    constexpr bool SPLAT = MODE == kModeSplat, CONE = MODE == kModeCone;
    constexpr int kChunk = CH;   // records per barrier
    constexpr int kRF4 = RecOf<SPLAT>::kF4, kCF4 = kCullF4<SPLAT>;
    __shared__ float4 srec[kChunk * kRF4];
    // footprints; where every pixel is tested, as (first x, first y, width - 1, height - 1) in 32 bits: a subtraction and an
    // unsigned comparison per axis, nothing to unpack
    using Rect = std::conditional_t<PIXTEST, int4, short4>;
    __shared__ Rect srect[kChunk];
    __shared__ float4 scull[PIXTEST ? 1 : kChunk * kCF4];   // Gram matrices for the opacity test
    // per record, contiguous for the opacity test: (px0, py0, log2 K, |A0|) and |A1|
    __shared__ float4 sref[PIXTEST ? 1 : kChunk];
    __shared__ float ssq1[PIXTEST ? 1 : kChunk];
    int rank = (int)blockIdx.x, tid = (int)threadIdx.x;
    if constexpr (P == 1) {
        rank = (int)blockIdx.x / split;
        tid += ((int)blockIdx.x - rank * split) * (int)blockDim.x;
    }
    const int tile = tile_order ? tile_order[rank] : rank;
    const ViewInfo &V = views[tile_view[tile]];
    const int local = tile - V.tile_base;
    const int tyi = local / V.tiles_x, txi = local - tyi * V.tiles_x;
    int ix, iy;
    L::origin(tid, V.tw, ix, iy);
    const int x0 = txi * V.tw + ix, y0 = tyi * V.th + iy;
    float Lp[P], T[P], S[P], c0[P], c1[P], c2[P];
    uint32_t last[P];
    const uint2 rg = ranges[tile];
    unsigned live = 0;   // bit k: pixel k is inside the image and not finished
#pragma unroll
    for (int k = 0; k < P; ++k) {
        const int x = x0 + L::ox(k), y = y0 + L::oy(k);
        Lp[k] = SPLAT ? 0.0f : pixel_ray(V, x, y).Lp;
        T[k] = 1.0f;
        S[k] = c0[k] = c1[k] = c2[k] = 0.0f;
        last[k] = rg.x;
        if (x < V.W && y < V.H) live |= 1u << k;
    }
    const float xf = (float)x0, yf = (float)y0;
    const WarpBox wb = warp_box<P>(x0, y0);
    const BoxCull bc = SPLAT ? box_cull_splat(wb, bp.alpha_min) : box_cull(V, wb, bp.tau_skip);
    const int lane = threadIdx.x & 31;
    unsigned long long pairs = 0, blended = 0;   // evaluated / blended pairs (COUNT only)
    for (uint32_t base = rg.x; base < rg.y; base += kChunk) {
        const uint32_t n = min((uint32_t)kChunk, rg.y - base);
        for (uint32_t r = threadIdx.x; r < n; r += blockDim.x) {
            const uint32_t item = sorted_item[base + r];
            const float4 *src = rec + (size_t)item * kRecF4;
            float4 q[kRF4];
#pragma unroll
            for (int k = 0; k < kRF4; ++k) {
                q[k] = __ldg(src + k);
                srec[r * kRF4 + k] = q[k];
            }
            put_rect(srect[r], prect[item]);
            if (!PIXTEST) {
                float4 c[kCF4];
                cull_row<SPLAT>(q, c, sref[r], ssq1[r]);
#pragma unroll
                for (int k = 0; k < kCF4; ++k) scull[r * kCF4 + k] = c[k];
            }
        }
        __syncthreads();
        // the warp ballots the records whose footprint touches its pixels (and, when pairs below
        // tau_skip are skipped, whose opacity can reach tau_skip there) and visits only those
        for (int w0 = 0; w0 < (int)n; w0 += 32) {
            if (!__any_sync(0xffffffffu, live != 0)) break;
            const int jl = w0 + lane;
            bool need = jl < (int)n && !box_misses(wb, srect[jl]);
            if (!PIXTEST && need)   // skip records whose opacity stays below tau_skip on this warp
                need = rec_may_blend<SPLAT>([&](int k) { return scull[jl * kCF4 + k]; }, sref[jl], ssq1[jl], bc);
            unsigned m = __ballot_sync(0xffffffffu, need);
            if constexpr (P == 1) {
                // kIlp records at a time: what does not depend on the pixel's state (opacity, its exponential)
                // is formed for all of them before the first is blended, so that their chains overlap
                while (m) {
                    int js[kIlp];
                    float t[kIlp], e2[kIlp], al[kIlp];
                    bool in[kIlp], v[kIlp];
#pragma unroll
                    for (int i = 0; i < kIlp; ++i) {
                        in[i] = m != 0;
                        js[i] = w0 + (m ? __ffs(m) - 1 : 0);
                        m &= m - 1;
                    }
#pragma unroll
                    for (int i = 0; i < kIlp; ++i) {
                        typename RecOf<SPLAT>::type r;
                        load_rec(&srec[js[i] * kRF4], r);
                        if constexpr (PIXTEST) in[i] = in[i] & pixel_in(x0, y0, srect[js[i]]);
                        if constexpr (SPLAT) {   // Eq. 6: alpha = min(o G'(p), alpha_max)
                            SplatCol sc;
                            splat_col(r, xf, sc);
                            float dx, dy, q;
                            const float a_c = fminf(splat_at(r, sc, yf, dx, dy, q), bp.alpha_max);
                            v[i] = in[i] & (a_c >= bp.alpha_min);
                            al[i] = v[i] ? a_c : 0.0f;
                            e2[i] = __fsub_rn(1.0f, al[i]);
                            t[i] = -log1pf(-al[i]);
                        } else {
                            ColBase cb;
                            col_base(r, xf, cb);
                            PairEval e;
                            pair_eval_col(r, cb, yf, Lp[0], e);
                            const float t_c = fminf(e.tau, bp.tau_max);
                            v[i] = in[i] & (t_c >= bp.tau_skip);
                            t[i] = v[i] ? t_c : 0.0f;
                            e2[i] = ex2_approx(__fmul_rn(-kLog2eF, t[i]));
                            al[i] = __fsub_rn(1.0f, e2[i]);
                        }
                    }
#pragma unroll
                    for (int i = 0; i < kIlp; ++i) {
                        const float4 q5 = srec[js[i] * kRF4 + kRF4 - 1];
                        if (COUNT) {
                            pairs += live && in[i];
                            blended += live && v[i];
                        }
                        if constexpr (CONE) {   // the sum of tau is all the projection needs
                            S[0] = __fadd_rn(S[0], live ? t[i] : 0.0f);
                            if (live && v[i]) last[0] = base + js[i] + 1;
                            continue;
                        }
                        const float w = __fmul_rn(live ? al[i] : 0.0f, T[0]);
                        c0[0] = fmaf(q5.y, w, c0[0]);
                        c1[0] = fmaf(q5.z, w, c1[0]);
                        c2[0] = fmaf(q5.w, w, c2[0]);
                        T[0] = __fmul_rn(T[0], live ? e2[i] : 1.0f);
                        S[0] = __fadd_rn(S[0], live ? t[i] : 0.0f);
                        if (live && v[i]) last[0] = base + js[i] + 1;
                        if (T[0] < bp.T_stop) live = 0;
                    }
                }
            }
            while (P > 1 && SPLAT && m) {
                const int j = w0 + __ffs(m) - 1;
                m &= m - 1;
                if constexpr (P > 1 && SPLAT) {
                    SplatRec r;
                    load_rec(&srec[j * kRF4], r);
                    const Rect pr = srect[j];
                    SplatCol sc[P / 2];   // pixel columns of the thread
#pragma unroll
                    for (int c = 0; c < P / 2; ++c) splat_col(r, c ? xf + 1.0f : xf, sc[c]);
#pragma unroll
                    for (int k = 0; k < P; ++k) {   // Eq. 6: alpha = min(o G'(p), alpha_max)
                        bool valid = (live >> k) & 1u;
                        if constexpr (PIXTEST) valid = valid & pixel_in(x0 + L::ox(k), y0 + L::oy(k), pr);
                        float dx, dy, q;
                        const float a_c =
                            fminf(splat_at(r, sc[L::ox(k)], L::oy(k) ? yf + (float)L::oy(k) : yf, dx, dy, q), bp.alpha_max);
                        if (COUNT) pairs += valid;
                        valid = valid && a_c >= bp.alpha_min;
                        if (COUNT) blended += valid;
                        const float alpha = valid ? a_c : 0.0f, e2 = __fsub_rn(1.0f, alpha), tau = -log1pf(-alpha);
                        const float w = __fmul_rn(alpha, T[k]);
                        c0[k] = fmaf(r.q5.y, w, c0[k]);
                        c1[k] = fmaf(r.q5.z, w, c1[k]);
                        c2[k] = fmaf(r.q5.w, w, c2[k]);
                        T[k] = __fmul_rn(T[k], e2);
                        S[k] = __fadd_rn(S[k], tau);
                        if (valid) last[k] = base + j + 1;
                        if (T[k] < bp.T_stop) live &= ~(1u << k);
                    }
                }
            }
            while (P > 1 && !SPLAT && m) {   // the same operations, packed over the two rows of a column
                if constexpr (P > 1 && !SPLAT) {
                    constexpr int kN = P == 2 && PIXTEST && !CONE ? 2 : 1, kRow = P / 2;   // pixel k = c + row kRow
                    int js[kN];
                    bool in[kN];
                    float t[kN][P / 2][2];
                    F2 e2[kN][P / 2];
                    bool v[kN][P / 2][2];
#pragma unroll
                    for (int i = 0; i < kN; ++i) {
                        in[i] = m != 0;
                        js[i] = w0 + (m ? __ffs(m) - 1 : 0);
                        m &= m - 1;
                    }
#pragma unroll
                    for (int i = 0; i < kN; ++i) {
                        RecPairs r;
                        load_rec(&srec[js[i] * kRF4], r);
                        const Rect pr = srect[js[i]];
#pragma unroll
                        for (int c = 0; c < P / 2; ++c) {
                            ColBase cb;
                            col_base(r, c ? xf + 1.0f : xf, cb);
                            float e[2];
                            pair_tau2(r, cb, f2_pack(yf, yf + 1.0f), f2_pack(Lp[c], Lp[c + kRow]), t[i][c]);
#pragma unroll
                            for (int h = 0; h < 2; ++h) {
                                // (no pixel of the projection finishes, and footprints end at the image's edge)
                                bool ok = CONE ? true : (kN == 1 ? ((live >> (c + h * kRow)) & 1u) != 0 : in[i]);
                                if constexpr (PIXTEST) ok = ok & pixel_in(x0 + c, y0 + h, pr);
                                if (COUNT && kN == 1) pairs += ok & ((live >> (c + h * kRow)) & 1u);
                                const float t_c = fminf(t[i][c][h], bp.tau_max);
                                v[i][c][h] = CONE ? ok : ok & (t_c >= bp.tau_skip);   // tau_skip = 0, and t_c is no NaN
                                t[i][c][h] = v[i][c][h] ? t_c : 0.0f;
                            }
                            if (!CONE) {
                                f2_unpack(f2_mul(f2_dup(-kLog2eF), f2_pack(t[i][c][0], t[i][c][1])), e[0], e[1]);
                                e2[i][c] = f2_pack(ex2_approx(e[0]), ex2_approx(e[1]));
                            }
                        }
                    }
#pragma unroll
                    for (int i = 0; i < kN; ++i) {
                        const float4 q5 = srec[js[i] * kRF4 + kRF4 - 1];
#pragma unroll
                        for (int c = 0; c < P / 2; ++c) {
                            if constexpr (COUNT && kN > 1) {   // (with the pixels that earlier records of the batch finished)
                                const Rect pr = srect[js[i]];
#pragma unroll
                                for (int h = 0; h < 2; ++h)
                                    pairs += in[i] & pixel_in(x0 + c, y0 + h, pr) & ((live >> (c + h * kRow)) & 1u);
                            }
                            if (kN > 1 && !CONE) {   // a pixel finished by an earlier record of the batch
                                float e[2];
                                f2_unpack(e2[i][c], e[0], e[1]);
#pragma unroll
                                for (int h = 0; h < 2; ++h)
                                    if (!((live >> (c + h * kRow)) & 1u)) e[h] = 1.0f, t[i][c][h] = 0.0f, v[i][c][h] = false;
                                e2[i][c] = f2_pack(e[0], e[1]);
                            }
#pragma unroll
                            for (int h = 0; h < 2; ++h) {
                                if (COUNT) blended += v[i][c][h];
                                if (v[i][c][h]) last[c + h * kRow] = base + js[i] + 1;
                            }
                            f2_unpack(f2_add(f2_pack(S[c], S[c + kRow]), f2_pack(t[i][c][0], t[i][c][1])), S[c], S[c + kRow]);
                            if constexpr (!CONE) {   // (the projection needs the sum of tau alone)
                                const F2 Tk = f2_pack(T[c], T[c + kRow]);
                                const F2 w = f2_mul(f2_fma(e2[i][c], f2_dup(-1.0f), f2_dup(1.0f)), Tk);   // (1 - e2) T
                                f2_unpack(f2_fma(f2_dup(q5.y), w, f2_pack(c0[c], c0[c + kRow])), c0[c], c0[c + kRow]);
                                f2_unpack(f2_fma(f2_dup(q5.z), w, f2_pack(c1[c], c1[c + kRow])), c1[c], c1[c + kRow]);
                                f2_unpack(f2_fma(f2_dup(q5.w), w, f2_pack(c2[c], c2[c + kRow])), c2[c], c2[c + kRow]);
                                f2_unpack(f2_mul(Tk, e2[i][c]), T[c], T[c + kRow]);
#pragma unroll
                                for (int h = 0; h < 2; ++h)
                                    if (T[c + h * kRow] < bp.T_stop) live &= ~(1u << (c + h * kRow));
                            }
                        }
                    }
                }
            }
        }
        if (__syncthreads_count(live != 0) == 0) break;
    }
    float l2acc = 0.0f;   // this thread's share of sum (rgb - target)^2 (fused loss only)
#pragma unroll
    for (int k = 0; k < P; ++k) {
        const int x = x0 + L::ox(k), y = y0 + L::oy(k);
        if (x >= V.W || y >= V.H) continue;
        const long long pix = V.pix_base + (long long)y * V.W + x;
        if constexpr (CONE) T[k] = ex2_approx(__fmul_rn(-kLog2eF, S[k]));
        if (CONE && l2.weights) l2.weights[pix] = -l2.dproj[pix] * T[k] * exp2f(Lp[k]);
        if (rgb) {   // absent for the cone-beam projection, which needs T alone
            const float o[3] = {fmaf(T[k], bp.bg[0], c0[k]), fmaf(T[k], bp.bg[1], c1[k]), fmaf(T[k], bp.bg[2], c2[k])};
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                rgb[3 * pix + c] = o[c];
                if (l2.target) {   // the operations of k_l2_loss: the same gradient bits
                    const float d = o[c] - l2.target[3 * pix + c];
                    l2.grad[3 * pix + c] = 2.0f * l2.scale * d;
                    l2acc = fmaf(d, d, l2acc);
                }
            }
        }
        T_ws[pix] = T[k];
        if (T_user) T_user[pix] = T[k];
        S_out[pix] = S[k];
        nlast_out[pix] = last[k];
    }
    if (l2.target) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) l2acc += __shfl_xor_sync(0xffffffffu, l2acc, o);
        if (lane == 0 && l2acc != 0.0f) atomicAdd(l2.loss, l2acc * l2.scale);
    }
    if (tile_replay) {   // the backward's replay length of this tile: its largest last blended position
        uint32_t m = rg.x;
#pragma unroll
        for (int k = 0; k < P; ++k) m = max(m, last[k]);
        m = __reduce_max_sync(0xffffffffu, m);
        if (lane == 0 && m > rg.x) atomicMax(tile_replay + tile, m - rg.x);
    }
    if (COUNT) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            pairs += __shfl_xor_sync(0xffffffffu, pairs, o);
            blended += __shfl_xor_sync(0xffffffffu, blended, o);
        }
        if (lane == 0 && pairs) atomicAdd(pair_count, pairs);
        if (lane == 0 && blended) atomicAdd(pair_count + 1, blended);
    }
}

template <int P, bool PIXTEST, int MODE, int CH>
static void launch_fwd_ptsc(const ViewInfo *views_d, const int *tile_view, const int *tile_order, long long n_tiles,
                            const uint2 *ranges, const uint32_t *sorted_item, const float4 *rec, const short4 *prect,
                            const BlendParams &bp, float *rgb, float *T_user, float *T_ws, float *S_out,
                            uint32_t *nlast_out, uint32_t *tile_replay, unsigned long long *pair_count,
                            const L2Fused &l2, cudaStream_t st) {
    const int split = P == 1 ? tile_split(n_tiles, bp.tile_px / P) : 1;
    const unsigned threads = (unsigned)(bp.tile_px / P / split);
    n_tiles *= split;
    if (pair_count)
        pdl_launch(k_render_fwd<P, true, PIXTEST, MODE, CH>, (unsigned)n_tiles, threads, 0, st,
            views_d, tile_view, tile_order, ranges, sorted_item, rec, prect, bp, rgb, T_user, T_ws, S_out, nlast_out, tile_replay,
            pair_count, l2, split);
    else
        pdl_launch(k_render_fwd<P, false, PIXTEST, MODE, CH>, (unsigned)n_tiles, threads, 0, st,
            views_d, tile_view, tile_order, ranges, sorted_item, rec, prect, bp, rgb, T_user, T_ws, S_out, nlast_out, tile_replay,
            nullptr, l2, split);
}

template <int P, bool PIXTEST, int MODE>
static void launch_fwd_pts(const ViewInfo *views_d, const int *tile_view, const int *tile_order, long long n_tiles,
                           const uint2 *ranges, const uint32_t *sorted_item, const float4 *rec, const short4 *prect,
                           const BlendParams &bp, float *rgb, float *T_user, float *T_ws, float *S_out,
                           uint32_t *nlast_out, uint32_t *tile_replay, unsigned long long *pair_count,
                           const L2Fused &l2, cudaStream_t st) {
    if (bp.chunk_fwd == 64)
        launch_fwd_ptsc<P, PIXTEST, MODE, 64>(views_d, tile_view, tile_order, n_tiles, ranges, sorted_item, rec, prect,
                                               bp, rgb, T_user, T_ws, S_out, nlast_out, tile_replay, pair_count, l2, st);
    else
        launch_fwd_ptsc<P, PIXTEST, MODE, 128>(views_d, tile_view, tile_order, n_tiles, ranges, sorted_item, rec, prect,
                                                bp, rgb, T_user, T_ws, S_out, nlast_out, tile_replay, pair_count, l2, st);
}

template <int P, bool PIXTEST>
static void launch_fwd_pt(const ViewInfo *views_d, const int *tile_view, const int *tile_order, long long n_tiles,
                          const uint2 *ranges, const uint32_t *sorted_item, const float4 *rec, const short4 *prect,
                          const BlendParams &bp, float *rgb, float *T_user, float *T_ws, float *S_out,
                          uint32_t *nlast_out, uint32_t *tile_replay, unsigned long long *pair_count,
                          const L2Fused &l2, cudaStream_t st) {
    if constexpr (PIXTEST) {   // the projection's tau_skip is 0, below any tau_cut
        if (!rgb) {
            launch_fwd_pts<P, PIXTEST, kModeCone>(views_d, tile_view, tile_order, n_tiles, ranges, sorted_item, rec, prect,
                                                  bp, rgb, T_user, T_ws, S_out, nlast_out, tile_replay, pair_count, l2, st);
            return;
        }
    }
    if (bp.splat)
        launch_fwd_pts<P, PIXTEST, kModeSplat>(views_d, tile_view, tile_order, n_tiles, ranges, sorted_item, rec, prect, bp,
                                               rgb, T_user, T_ws, S_out, nlast_out, tile_replay, pair_count, l2, st);
    else
        launch_fwd_pts<P, PIXTEST, kModeBlend>(views_d, tile_view, tile_order, n_tiles, ranges, sorted_item, rec, prect, bp,
                                               rgb, T_user, T_ws, S_out, nlast_out, tile_replay, pair_count, l2, st);
}

template <int P>
static void launch_fwd_p(const ViewInfo *views_d, const int *tile_view, const int *tile_order, long long n_tiles,
                         const uint2 *ranges, const uint32_t *sorted_item, const float4 *rec, const short4 *prect,
                         const BlendParams &bp, float *rgb, float *T_user, float *T_ws, float *S_out,
                         uint32_t *nlast_out, uint32_t *tile_replay, unsigned long long *pair_count,
                         const L2Fused &l2, cudaStream_t st) {
    if (bp.pixel_test)
        launch_fwd_pt<P, true>(views_d, tile_view, tile_order, n_tiles, ranges, sorted_item, rec, prect, bp, rgb,
                               T_user, T_ws, S_out, nlast_out, tile_replay, pair_count, l2, st);
    else
        launch_fwd_pt<P, false>(views_d, tile_view, tile_order, n_tiles, ranges, sorted_item, rec, prect, bp, rgb,
                                T_user, T_ws, S_out, nlast_out, tile_replay, pair_count, l2, st);
}

cudaError_t launch_render_fwd(const ViewInfo *views_d, const int *tile_view, const int *tile_order, long long n_tiles,
                              const uint2 *ranges, const uint32_t *sorted_item, const float4 *rec, const short4 *prect,
                              const BlendParams &bp, int ppt, float *rgb, float *T_user, float *T_ws, float *S_out,
                              uint32_t *nlast_out, uint32_t *tile_replay, unsigned long long *pair_count,
                              const L2Fused &l2, cudaStream_t st, long long *launches) {
    if (n_tiles <= 0) return cudaSuccess;
    if (ppt == 1)
        launch_fwd_p<1>(views_d, tile_view, tile_order, n_tiles, ranges, sorted_item, rec, prect, bp, rgb, T_user, T_ws, S_out,
                        nlast_out, tile_replay, pair_count, l2, st);
    else if (ppt == 4)
        launch_fwd_p<4>(views_d, tile_view, tile_order, n_tiles, ranges, sorted_item, rec, prect, bp, rgb, T_user, T_ws, S_out,
                        nlast_out, tile_replay, pair_count, l2, st);
    else
        launch_fwd_p<2>(views_d, tile_view, tile_order, n_tiles, ranges, sorted_item, rec, prect, bp, rgb, T_user, T_ws, S_out,
                        nlast_out, tile_replay, pair_count, l2, st);
    *launches += 1;
    return cudaGetLastError();
}

}  // namespace vg
