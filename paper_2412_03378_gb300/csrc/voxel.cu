// Voxel density query: sigma(x) = sum_g kappa_g exp(-(x - mu)' P (x - mu) / 2) (Eq. 3-4) at the
// centres of a regular grid, for volumetric comparisons of a reconstruction.
//
// Each Gaussian is truncated to the voxel box of its ellipsoid (x - mu)' P (x - mu) <= k^2,
// k^2 = 2 ln 2 e with kappa / sigma_cut = m 2^e, computed in FP32 with a fixed operation order
// (the same rule as the key function).  Gaussians are binned into bricks of 8^3 voxels with the
// scan / radix sort / range kernels of the tile binning; one warp per brick sums its list at its
// voxels (two columns of eight per lane), so no atomics are needed and the sum is deterministic.
#include "geometry.cuh"

namespace vg {

constexpr int kBrick = 8;
constexpr int kVoxWarps = 4;                  // bricks per CTA, a warp each
constexpr int kVoxRecF4 = 3;                  // (mu, log2 kappa), (Q00 Q01 Q02 Q11), (Q12 Q22 - -), Q = -log2(e) P / 2
constexpr int kVoxStageF4 = 4;                // a staged record: (mu_x mu_y Q00 2Q01) (Q11 2Q02 2Q12 mu_z) (u[8])

// Truncation box, record and brick count of every Gaussian.
template <typename RT>
__global__ void __launch_bounds__(256)
k_voxel_pre(GaussIn g, VoxelGrid grid, float sigma_cut, float4 *__restrict__ rec, short4 *__restrict__ box,
            uint32_t *__restrict__ count) {
    pdl_entry();
    for (long long gi = (long long)blockIdx.x * blockDim.x + threadIdx.x; gi < g.n;
         gi += (long long)gridDim.x * blockDim.x) {
        float mu[3], s[3], q[4], kin, Sig[9], Rq[9], qn[4], smax;
        load_gauss<RT>(g, gi, mu, s, q, kin);
        const Density dn = density_of(g, kin, s);
        short4 b0 = make_short4(-1, -1, -1, -1), b1 = make_short4(-1, -1, 0, 0);
        uint32_t cnt = 0;
        if (key_cov(mu, s, q, dn.kap_key, Sig, Rq, qn, smax)) {
            const float xr = VG_DIV(dn.kap_key, sigma_cut);
            if (xr > 1.0f) {
                const int e = (xr > FLT_MAX) ? 128 : (int)((__float_as_uint(xr) >> 23) & 0xFFu) - 126;
                const float k2 = VG_MUL((float)e, 1.3862944f);
                const float o[3] = {grid.ox, grid.oy, grid.oz}, v[3] = {grid.vx, grid.vy, grid.vz};
                const int n[3] = {grid.nx, grid.ny, grid.nz};
                int lo[3], hi[3];
                bool ok = true;
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    const float h = VG_SQRT(VG_MUL(k2, Sig[4 * a]));
                    const float c = VG_SUB(mu[a], o[a]);
                    const float flo = VG_SUB(VG_DIV(VG_SUB(c, h), v[a]), 0.5f);
                    const float fhi = VG_SUB(VG_DIV(VG_ADD(c, h), v[a]), 0.5f);
                    pixel_span(flo, fhi, n[a], lo[a], hi[a]);
                    ok = ok && lo[a] <= hi[a];
                }
                if (ok) {
                    b0 = make_short4((short)lo[0], (short)lo[1], (short)lo[2], (short)hi[0]);
                    b1 = make_short4((short)hi[1], (short)hi[2], 0, 0);
                    cnt = (uint32_t)(hi[0] / kBrick - lo[0] / kBrick + 1) * (uint32_t)(hi[1] / kBrick - lo[1] / kBrick + 1) *
                          (uint32_t)(hi[2] / kBrick - lo[2] / kBrick + 1);
                    // Q = -log2(e) / 2 times the precision Rq diag(1/s^2) Rq^T (columns of Rq are the principal axes).
                    // 1/s^2 is kept where (x - mu)' P (x - mu) stays finite over a brick: at that limit anything
                    // but a voxel centre on mu itself is at 2^-inf already.
                    float P[6];
                    const float ext = fmaf(v[0], v[0], fmaf(v[1], v[1], v[2] * v[2])) * (float)(kBrick * kBrick);
                    const float wmax = fminf(1e36f / ext, 1e37f);
                    const float w0 = -0.72134752f * fminf(1.0f / (s[0] * s[0]), wmax),
                                w1 = -0.72134752f * fminf(1.0f / (s[1] * s[1]), wmax),
                                w2 = -0.72134752f * fminf(1.0f / (s[2] * s[2]), wmax);
                    const int ij[6][2] = {{0, 0}, {0, 1}, {0, 2}, {1, 1}, {1, 2}, {2, 2}};
#pragma unroll
                    for (int k = 0; k < 6; ++k) {
                        const int i = ij[k][0], j = ij[k][1];
                        P[k] = Rq[3 * i] * Rq[3 * j] * w0 + Rq[3 * i + 1] * Rq[3 * j + 1] * w1 +
                               Rq[3 * i + 2] * Rq[3 * j + 2] * w2;
                    }
                    float4 *r = rec + gi * kVoxRecF4;
                    r[0] = make_float4(mu[0], mu[1], mu[2], log2f(dn.kap));
                    r[1] = make_float4(P[0], P[1], P[2], P[3]);
                    r[2] = make_float4(P[4], P[5], 0.0f, 0.0f);
                }
            }
        }
        box[2 * gi] = b0;
        box[2 * gi + 1] = b1;
        count[gi] = cnt;
    }
}

// (brick, Gaussian) instances in Gaussian order; brick id = (bz * bricks_y + by) * bricks_x + bx.  A
// warp takes 32 consecutive Gaussians, whose instances fill one contiguous output range that the lanes
// write together (as k_duplicate does): 24 M instances of 200,000 Gaussians 0.385 -> 0.123 ms against one
// thread per Gaussian, whose stores lie apart.
constexpr int kVoxDupWarps = 8;

__global__ void __launch_bounds__(32 * kVoxDupWarps)
k_voxel_dup(const uint32_t *__restrict__ offsets, const short4 *__restrict__ box, VoxelGrid grid, long long n,
            uint32_t *__restrict__ inst_key, uint32_t *__restrict__ inst_val, long long capacity) {
    pdl_entry();
    __shared__ uint32_t s_off[kVoxDupWarps][32];
    __shared__ uint32_t s_first[kVoxDupWarps][32], s_nx[kVoxDupWarps][32], s_nxy[kVoxDupWarps][32];
    const int lane = threadIdx.x & 31, wi = threadIdx.x >> 5;
    const long long stride = (long long)gridDim.x * kVoxDupWarps * 32;
    for (long long w0 = ((long long)blockIdx.x * kVoxDupWarps + wi) * 32; w0 < n; w0 += stride) {
        const long long i = w0 + lane;
        uint32_t off = 0, end = 0, first = 0, nx = 1, nxy = 1;
        if (i < n) {
            off = offsets[i];
            end = offsets[i + 1];
            if (end > off) {
                const short4 b0 = box[2 * i], b1 = box[2 * i + 1];
                const int x0 = b0.x / kBrick, y0 = b0.y / kBrick, z0 = b0.z / kBrick;
                first = (uint32_t)((z0 * grid.by + y0) * grid.bx + x0);
                nx = (uint32_t)(b0.w / kBrick - x0 + 1);
                nxy = nx * (uint32_t)(b1.x / kBrick - y0 + 1);
            }
        }
        const int last = (int)min(31LL, n - 1 - w0);
        const uint32_t r0 = __shfl_sync(0xffffffffu, off, 0), r1 = __shfl_sync(0xffffffffu, end, last);
        s_off[wi][lane] = i < n ? off : r1;   // lanes past the end own nothing
        s_first[wi][lane] = first;
        s_nx[wi][lane] = nx;
        s_nxy[wi][lane] = nxy;
        __syncwarp();
        for (uint32_t o = r0 + lane; o < r1; o += 32) {
            int l = 0;   // the last Gaussian whose first instance is at or before o
#pragma unroll
            for (int step = 16; step > 0; step >>= 1)
                if (s_off[wi][l + step] <= o) l += step;
            const uint32_t r = o - s_off[wi][l], z = r / s_nxy[wi][l], q = r - z * s_nxy[wi][l];
            const uint32_t y = q / s_nx[wi][l], x = q - y * s_nx[wi][l];
            if ((long long)o < capacity) {
                inst_key[o] = s_first[wi][l] + (z * (uint32_t)grid.by + y) * (uint32_t)grid.bx + x;
                inst_val[o] = (uint32_t)(w0 + l);
            }
        }
        __syncwarp();   // the staged values are reused by the warp's next 32
    }
}

// One warp per brick (four independent warps per CTA): lane l owns the two columns (l % 8, l / 8) and
// (l % 8, l / 8 + 4) of the brick, eight voxels along z each.  With dz_c the offset of the brick's c-th layer,
// log2 of a record's value at a voxel is
//   (Q00 dx^2 + 2 Q01 dx dy + Q11 dy^2) + dz_c (2 Q02 dx + 2 Q12 dy) + u_c,   u_c = log2 kappa + Q22 dz_c^2:
// u_c is the same for the whole brick, so the lane that stages the record forms it once (-inf for a
// layer outside the record's box, which masks it), a column adds its two terms in x and y (-inf
// outside the box), and two voxels cost two packed operations, two ex2 and one packed sum.  Bound by
// the FMA pipe (28 packed operations of two cycles and 16 others per brick and sub-partition), the ex2
// unit (64 cycles) and the shared-memory reads of the staged record, of which a warp-wide 16-byte
// broadcast takes 4 cycles of the SM's.  The list comes 32 records at a time, one per lane, the next
// ones requested before the present ones are summed; each carries the rows of the brick inside its
// box as a word of bits (x 0..7, y 8..15, z 16..23).
// 256^3 grid, 200,000 Gaussians (24 M instances): 8.58 -> 2.28 ms against two voxels per thread and
// eight warps per brick.  Skipping quarters of the brick outside a box 2.39 ms (the branches keep two records'
// chains from overlapping), 28 or 32 warps per SM instead of 16 2.34 / 2.53 ms, one column per lane 2.67 ms.
__global__ void __launch_bounds__(32 * kVoxWarps, 4)
k_voxel_eval(const uint2 *__restrict__ ranges, const uint32_t *__restrict__ sorted, const float4 *__restrict__ rec,
             const short4 *__restrict__ box, VoxelGrid grid, int n_bricks, float *__restrict__ out) {
    pdl_entry();
    __shared__ float4 s_rec[kVoxWarps][32 * kVoxStageF4];
    __shared__ uint32_t s_bits[kVoxWarps][32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, brick = (int)blockIdx.x * kVoxWarps + w;
    if (brick >= n_bricks) return;
    float4 *srec = s_rec[w];
    uint32_t *sbits = s_bits[w];
    const int bxi = brick % grid.bx, byi = (brick / grid.bx) % grid.by, bzi = brick / (grid.bx * grid.by);
    const int vx0 = bxi * kBrick, vy0 = byi * kBrick, vz0 = bzi * kBrick;
    const int i = vx0 + (lane & 7), j = vy0 + (lane >> 3);
    const uint32_t mine = 1u << (lane & 7) | 1u << (8 + (lane >> 3)), mine4 = 1u << (lane & 7) | 1u << (12 + (lane >> 3));
    const float x = VG_ADD(grid.ox, VG_MUL((float)i + 0.5f, grid.vx));
    const float y[2] = {VG_ADD(grid.oy, VG_MUL((float)j + 0.5f, grid.vy)), VG_ADD(grid.oy, VG_MUL((float)j + 4.5f, grid.vy))};
    float zl[kBrick];
    F2 sum[2][4];
#pragma unroll
    for (int c = 0; c < kBrick; ++c) {
        zl[c] = VG_ADD(grid.oz, VG_MUL((float)(vz0 + c) + 0.5f, grid.vz));
        sum[c >> 2][c & 3] = f2_dup(0.0f);
    }
    auto span = [](int first, int last) {   // bits max(first, 0) .. min(last, 7)
        const int a = max(first, 0), b = min(last, kBrick - 1);
        return b < a ? 0u : ((2u << b) - 1u) & ~((1u << a) - 1u);
    };
    const uint2 rg = ranges[brick];
    float4 p0 = make_float4(0.0f, 0.0f, 0.0f, 0.0f), p1 = p0, p2 = p0;
    uint32_t pb = 0;
    auto fetch = [&](uint32_t at) {
        if (at >= rg.y) return;
        const uint32_t gi = sorted[at];
        const float4 *src = rec + (size_t)gi * kVoxRecF4;
        p0 = __ldg(src), p1 = __ldg(src + 1), p2 = __ldg(src + 2);
        const short4 a = box[2 * gi], b = box[2 * gi + 1];
        pb = span(a.x - vx0, a.w - vx0) | span(a.y - vy0, b.x - vy0) << 8 | span(a.z - vz0, b.y - vz0) << 16;
    };
    fetch(rg.x + lane);
    for (uint32_t base = rg.x; base < rg.y; base += 32) {
        const int n = (int)min(32u, rg.y - base);
        __syncwarp();
        {
            float4 *st = srec + lane * kVoxStageF4;
            float u[kBrick];
#pragma unroll
            for (int c = 0; c < kBrick; ++c) {
                const float dz = zl[c] - p0.z;
                u[c] = pb & (0x10000u << c) ? fmaf(p2.y * dz, dz, p0.w) : -INFINITY;
            }
            st[0] = make_float4(p0.x, p0.y, p1.x, 2.0f * p1.y);
            st[1] = make_float4(p1.w, 2.0f * p1.z, 2.0f * p2.x, p0.z);
            st[2] = make_float4(u[0], u[1], u[2], u[3]);
            st[3] = make_float4(u[4], u[5], u[6], u[7]);
            sbits[lane] = pb;
        }
        fetch(base + 32 + lane);
        __syncwarp();
#pragma unroll 2
        for (int jj = 0; jj < n; ++jj) {
            const uint32_t bits = sbits[jj];
            const float4 *st = srec + jj * kVoxStageF4;
            const float4 r0 = st[0], r1 = st[1];
            const float dx = x - r0.x, qx = r0.z * dx;
            const F2 nz = f2_dup(-r1.w);
            F2 q[2], b[2];
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                const uint32_t in = k ? mine4 : mine;
                const float dy = y[k] - r0.y;
                const float qxy = fmaf(qx, dx, fmaf(r0.w * dx, dy, r1.x * dy * dy));
                q[k] = f2_dup((bits & in) == in ? qxy : -INFINITY);
                b[k] = f2_dup(fmaf(r1.y, dx, r1.z * dy));
            }
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const ulonglong2 uu = *reinterpret_cast<const ulonglong2 *>(st + 2 + h);
                F2 dz[2], u[2];
                u[0].v = uu.x, u[1].v = uu.y;
#pragma unroll
                for (int c = 0; c < 2; ++c) dz[c] = f2_add(f2_pack(zl[4 * h + 2 * c], zl[4 * h + 2 * c + 1]), nz);
#pragma unroll
                for (int k = 0; k < 2; ++k) {
#pragma unroll
                    for (int c = 0; c < 2; ++c) {
                        float e0, e1;
                        f2_unpack(f2_fma(dz[c], b[k], f2_add(u[c], q[k])), e0, e1);
                        sum[k][2 * h + c] = f2_add(sum[k][2 * h + c], f2_pack(ex2_approx(e0), ex2_approx(e1)));
                    }
                }
            }
        }
    }
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        if (i >= grid.nx || j + 4 * k >= grid.ny) continue;
#pragma unroll
        for (int c = 0; c < kBrick; ++c) {
            float s[2];
            f2_unpack(sum[k][c >> 1], s[0], s[1]);
            if (vz0 + c < grid.nz) out[((size_t)(vz0 + c) * grid.ny + j + 4 * k) * grid.nx + i] = s[c & 1];
        }
    }
}

cudaError_t launch_voxel_pre(const GaussIn &g, const VoxelGrid &grid, float sigma_cut, float4 *rec, short4 *box,
                             uint32_t *count, cudaStream_t st, long long *launches) {
    if (g.n <= 0) return cudaSuccess;
    long long b = (g.n + 255) / 256;
    if (b > 152 * 16) b = 152 * 16;
    if (g.rec_dtype == VG_BF16)
        pdl_launch(k_voxel_pre<__nv_bfloat16>, (unsigned)b, 256, 0, st, g, grid, sigma_cut, rec, box, count);
    else if (g.rec_dtype == VG_F16)
        pdl_launch(k_voxel_pre<__half>, (unsigned)b, 256, 0, st, g, grid, sigma_cut, rec, box, count);
    else
        pdl_launch(k_voxel_pre<float>, (unsigned)b, 256, 0, st, g, grid, sigma_cut, rec, box, count);
    *launches += 1;
    return cudaGetLastError();
}

cudaError_t launch_voxel_dup(const uint32_t *offsets, const short4 *box, const VoxelGrid &grid, long long n,
                             uint32_t *inst_key, uint32_t *inst_val, long long capacity, cudaStream_t st,
                             long long *launches) {
    if (n <= 0) return cudaSuccess;
    long long b = (n + 32 * kVoxDupWarps - 1) / (32 * kVoxDupWarps);
    if (b > 152 * 32) b = 152 * 32;
    pdl_launch(k_voxel_dup, (unsigned)b, 32 * kVoxDupWarps, 0, st, offsets, box, grid, n, inst_key, inst_val, capacity);
    *launches += 1;
    return cudaGetLastError();
}

cudaError_t launch_voxel_eval(const uint2 *ranges, const uint32_t *sorted, const float4 *rec, const short4 *box,
                              const VoxelGrid &grid, float *out, cudaStream_t st, long long *launches) {
    const long long bricks = (long long)grid.bx * grid.by * grid.bz;
    if (bricks <= 0) return cudaSuccess;
    pdl_launch(k_voxel_eval, (unsigned)((bricks + kVoxWarps - 1) / kVoxWarps), 32 * kVoxWarps, 0, st, ranges, sorted, rec,
               box, grid, (int)bricks, out);
    *launches += 1;
    return cudaGetLastError();
}

}  // namespace vg
