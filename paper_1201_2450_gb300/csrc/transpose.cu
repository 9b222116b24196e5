// The exact transpose P^T of the cone-beam projector (Eq. 5's gradient
// step), voxel-driven: each thread owns a short z-run of one voxel column
// and gathers, for every view of its phase, the pixels whose rays cross each
// voxel, weighted by the exact chord length.  k_backproject tests every
// cell; k_colscan + k_backproject_bands split each chord at the z
// boundaries it crosses and sum the rows between them by prefix sums.
//
// The ray parameter is measured in units of the source->pixel vector D
// (chord = delta_parameter * |D|) and anchored at the voxel column so that
// FP32 positions keep ~1e-5 voxel resolution.
#include "ray_common.cuh"

namespace tnlm {
namespace {

constexpr int kBpBX = 32, kBpBY = 4, kBpCH = 8;  // exact transpose block: 32 x 4 columns, 8 voxels in z each

template <bool SCALED, class T>
__global__ void __launch_bounds__(kBpBX *kBpBY)
    k_backproject(KGeom G, const ViewGeom *__restrict__ views, const int *__restrict__ view_off,
                  const float *__restrict__ proj, const T *vin, T *vout, float alpha, float beta,
                  int nchunks)
{
    constexpr int NT = kBpBX * kBpBY;
    extern __shared__ float4 sm4[];
    float4 *s_row = sm4;                                // per detector row: (v, 1/v or 0, v^2, 0)
    float *s_acc = reinterpret_cast<float *>(sm4 + G.nv);  // [kBpCH][NT] per-thread accumulators
    const int tid = threadIdx.y * kBpBX + threadIdx.x;
    for (int t = tid; t < G.nv; t += NT) {
        const float v = ((float)t - G.vc) * G.dv + G.v_off;
        s_row[t] = make_float4(v, v != 0.f ? 1.0f / v : 0.f, v * v, 0.f);
    }
#pragma unroll
    for (int k = 0; k < kBpCH; ++k) s_acc[k * NT + tid] = 0.f;
    __syncthreads();
    const int ix = blockIdx.x * kBpBX + threadIdx.x;
    const int iy = blockIdx.y * kBpBY + threadIdx.y;
    const int phase = blockIdx.z / nchunks;
    const int iz0 = (blockIdx.z % nchunks) * kBpCH;
    if (ix >= G.nx || iy >= G.ny) return;
    const int nzc = min(kBpCH, G.nz - iz0);
    const float xc = G.b0x + ((float)ix + 0.5f) * G.dx;
    const float yc = G.b0y + ((float)iy + 0.5f) * G.dy;
    const float fvscale = G.inv_dv, fvoff = G.vc - G.v_off * G.inv_dv;  // row coordinate of v: v*fvscale + fvoff

    const int v_end = view_off[phase + 1];
    for (int vg = view_off[phase]; vg < v_end; ++vg) {
        const float c = views[vg].c, s = views[vg].s;
        const float a = xc * c + yc * s;   // view-frame coordinate toward the source
        const float b = -xc * s + yc * c;  // view-frame coordinate along u
        const float ac = (G.sad - a) * G.inv_sdd;  // ray parameter at the column centre's depth
        // u footprint of the column: perspective images of its four xy corners
        float umin = FLT_MAX, umax = -FLT_MAX;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const float ex = (q & 1) ? G.hx : -G.hx, ey = (q & 2) ? G.hy : -G.hy;
            const float ak = a + ex * c + ey * s;
            const float bk = b - ex * s + ey * c;
            const float uk = bk * G.sdd / (G.sad - ak);
            umin = fminf(umin, uk);
            umax = fmaxf(umax, uk);
        }
        const float fu_lo = fmaxf((umin - G.u_off) * G.inv_du + G.uc - 1e-3f, -1.f);
        const float fu_hi = fminf((umax - G.u_off) * G.inv_du + G.uc + 1e-3f, (float)G.nu);
        const int iu_lo = max(0, (int)ceilf(fu_lo));
        const int iu_hi = min(G.nu - 1, (int)floorf(fu_hi));
        const float *__restrict__ pv = proj + (long long)vg * G.npix;
        for (int iu = iu_lo; iu <= iu_hi; ++iu) {
            const float u = ((float)iu - G.uc) * G.du + G.u_off;
            const float w = ac * u - b;          // lateral offset of the ray at the column depth (view frame)
            const float qx = -w * s, qy = w * c;  // the same offset on the world axes
            const float gx = -G.sdd * c - u * s;  // world xy direction per unit ray parameter
            const float gy = -G.sdd * s + u * c;
            float glo = -ac, ghi = 1.f - ac;     // segment source .. pixel
            bool ok = true;
            slab_local(qx, gx, G.hx, glo, ghi, ok);
            slab_local(qy, gy, G.hy, glo, ghi, ok);
            if (!ok || !(glo < ghi)) continue;
            const float ialo = 1.0f / (ac + glo), iahi = 1.0f / (ac + ghi);
            const float dg = ghi - glo;  // xy chord of this pixel column (ray-parameter units)
            const float len_u2 = G.sdd * G.sdd + u * u;
            const float *__restrict__ pc = pv + iu;
            // Row coordinate of the image of a z boundary seen at the near / far end of the xy chord:
            // row = z * (1/alpha) / dv + (vc - v_off/dv).  Adjacent cells share a boundary, so each
            // boundary is mapped once and carried to the next cell.
            const float sra = ialo * fvscale, srb = iahi * fvscale;
            float zb = fmaf((float)iz0, G.dz, G.b0z);
            float pa = fmaf(zb, sra, fvoff), pb = fmaf(zb, srb, fvoff);
            float rlo = fminf(pa, pb), rhi = fmaxf(pa, pb);
            for (int k = 0; k < nzc; ++k) {
                const float zc = fmaf((float)(iz0 + k) + 0.5f, G.dz, G.b0z);
                const float zlo = zc - G.hz, zhi = zc + G.hz;
                zb = fmaf((float)(iz0 + k + 1), G.dz, G.b0z);
                pa = fmaf(zb, sra, fvoff);
                pb = fmaf(zb, srb, fvoff);
                const float rlo2 = fminf(pa, pb), rhi2 = fmaxf(pa, pb);
                // candidate rows meet the cell somewhere; full rows stay inside its z slab over the whole
                // xy chord (both with a 1e-3-row safety margin; the exact test decides the rest)
                const int iv_lo = max(0, __float2int_ru(fmaxf(rlo - 1e-3f, -1.f)));
                const int iv_hi = min(G.nv - 1, __float2int_rd(fminf(rhi2 + 1e-3f, (float)G.nv)));
                int if_lo = max(iv_lo, __float2int_ru(fmaxf(rhi + 1e-3f, -1.f)));
                int if_hi = min(iv_hi, __float2int_rd(fminf(rlo2 - 1e-3f, (float)G.nv)));
                rlo = rlo2;
                rhi = rhi2;
                if (if_lo > if_hi) {  // no full row: every candidate row is partial
                    if_lo = iv_hi + 1;
                    if_hi = iv_hi;
                }
                // full rows: the exact chord is the whole xy chord dg
                float sfull = 0.f;
                for (int iv = if_lo; iv <= if_hi; ++iv) {
                    float r = __ldg(pc + iv * G.nu);
                    if (!SCALED) r *= sqrtf(len_u2 + s_row[iv].z);
                    sfull += r;
                }
                // partial rows (below and above the full range): exact z-slab test
                float spart = 0.f;
                for (int iv = iv_lo; iv <= iv_hi; ++iv) {
                    if (iv == if_lo) {  // skip the full range
                        iv = if_hi;
                        continue;
                    }
                    const float4 rw = s_row[iv];
                    float zl, zh;
                    if (rw.x != 0.f) {
                        const float oz = fmaf(ac, rw.x, -zc);  // z offset of the ray from the cell centre at gamma 0
                        const float t0 = (-G.hz - oz) * rw.y;
                        const float t1 = (G.hz - oz) * rw.y;
                        zl = fminf(t0, t1);
                        zh = fmaxf(t0, t1);
                    } else {  // ray in the plane z = 0: inside iff zlo <= 0 < zhi
                        const bool in = (zlo <= 0.f) && (0.f < zhi);
                        zl = in ? -FLT_MAX : FLT_MAX;
                        zh = in ? FLT_MAX : -FLT_MAX;
                    }
                    const float seg = fminf(ghi, zh) - fmaxf(glo, zl);
                    if (seg > 0.f) {
                        float r = __ldg(pc + iv * G.nu);
                        if (!SCALED) r *= sqrtf(len_u2 + rw.z);
                        spart = fmaf(r, seg, spart);
                    }
                }
                s_acc[k * NT + tid] += fmaf(sfull, dg, spart);
            }
        }
    }
    const long long base = (long long)phase * G.nvox + ((long long)iz0 * G.ny + iy) * G.nx + ix;
    for (int k = 0; k < nzc; ++k) {
        const long long o = base + (long long)k * G.nx * G.ny;
        const float bp = alpha * s_acc[k * NT + tid];
        st_v(vout + o, beta != 0.f ? fmaf(beta, ld_v(vin + o), bp) : bp);
    }
}

// Exclusive prefix sums along each detector column (fixed view and iu) of the
// ray-length-scaled projection, accumulated in double-float arithmetic and
// stored as an (hi, lo) float pair: pref[vg][iv][iu] = sum_{t < iv} r(t) |D(t)|.  A sum over
// a run of rows is then two loads and a difference, exact to FP32 rounding.
// For an unscaled input the scaled values are also written to scaled_out.
template <bool SCALED>
__global__ void __launch_bounds__(256) k_colscan(KGeom G, const float *__restrict__ proj, float2 *__restrict__ pref,
                                                 float *__restrict__ scaled_out)
{
    const int iu = blockIdx.x * blockDim.x + threadIdx.x;
    const int vg = blockIdx.y;
    if (iu >= G.nu) return;
    const float u = ((float)iu - G.uc) * G.du + G.u_off;
    const float len_u2 = G.sdd * G.sdd + u * u;
    const float *__restrict__ pc = proj + (long long)vg * G.npix + iu;
    float *__restrict__ so = SCALED ? nullptr : scaled_out + (long long)vg * G.npix + iu;
    float2 *__restrict__ po = pref + (long long)vg * (G.nv + 1) * G.nu + iu;
    // running sum as an unevaluated pair hi + lo: each addition is split into its
    // rounded result and exact error (Knuth's two-sum), the errors gather in lo;
    // FP64 adds would cost far more issue slots on this GPU
    float hi = 0.f, lo = 0.f;
    po[0] = make_float2(0.f, 0.f);
    for (int iv = 0; iv < G.nv; ++iv) {
        float r = __ldg(pc + (long long)iv * G.nu);
        if (!SCALED) {  // scale by the ray length once, for the band rows too
            const float v = ((float)iv - G.vc) * G.dv + G.v_off;
            r *= sqrtf(len_u2 + v * v);
            so[(long long)iv * G.nu] = r;
        }
        const float t = hi + r;
        const float bv = t - hi;
        lo += (hi - (t - bv)) + (r - bv);
        hi = t;
        po[(long long)(iv + 1) * G.nu] = make_float2(hi, lo);
    }
}

// Transpose for geometries where a ray's chord through one voxel column spans
// at most two z cells.  For each view, pixel column iu and z boundary z_m, let
//   B_m = sum over detector rows of r |D| (length of the row's chord below z_m);
// cell m receives B_{m+1} - B_m.  The rows below L_m, the first row whose chord
// may cross z_m, lie wholly below it, so B_m is the xy chord dg times one prefix
// sum, plus the crossing rows' own shares: an exact clamp per row, 0 for a row
// that turns out to lie above.  The boundary images at the near and far end of
// the chord are less than one or two rows apart on most scanners (band_rows),
// so the rows L_m (and L_m + 1) are the only candidates and a boundary needs no
// loop and no test.
// Equal to the per-cell exact tests of k_backproject up to rounding.
//
// A warp covers 8 x 4 voxel columns: whatever the view angle its lanes read
// detector columns within ~12 voxels of each other (a row of 32 voxels spread
// over 120 pixel columns when the rays run along y).  Rows are rounded up in
// floating point (add a power of two with rounding up: the integer is in the
// low mantissa bits) and addresses formed from those bits directly.
constexpr int kBandWX = 8, kBandWY = 4;  // voxel columns of a warp
constexpr float kRowMagic = 12582912.0f;                // 1.5 * 2^23: one unit per ulp
constexpr long long kRowMagicBits = 0x4B400000LL;

// One view of a thread's column chunk: every pixel column iu of the column's
// footprint, each of its chord's cell boundaries in turn.
// ROWS: candidate rows per boundary, 1 or 2, or 0 for any number (a loop).
template <int CH, int ROWS>
__device__ __forceinline__ void bands_view(const KGeom &G, const float4 *s_row, float c, float s, float xc, float yc,
                                           int iz0, const float *__restrict__ pv, const float2 *__restrict__ ppv,
                                           float (&acc)[CH])
{
    const float fvscale = G.inv_dv;
    const float fvlo = G.vc - G.v_off * G.inv_dv - 1e-3f;  // row coordinate of v: v * fvscale + fvlo, less a margin
    const float a = xc * c + yc * s;   // view-frame coordinate toward the source
    const float b = -xc * s + yc * c;  // view-frame coordinate along u
    const float U = G.sad - a;
    const float ac = U * G.inv_sdd;  // ray parameter at the column centre's depth
    // u footprint: the column's half extent across the ray through its centre, at the nearest depth of its
    // corners (a bound; pixel columns that miss the square drop out by their empty chord)
    const float t = __fdividef(b, U);
    const float ext = G.hx * fabsf(fmaf(t, c, -s)) + G.hy * fabsf(fmaf(t, s, c));
    const float near = U - (G.hx * fabsf(c) + G.hy * fabsf(s));
    const float fu = fmaf(t * G.sdd - G.u_off, G.inv_du, G.uc);
    const float fw = __fdividef(ext * G.sdd, near) * G.inv_du + 2e-3f;
    const int iu_lo = max(0, (int)ceilf(fmaxf(fu - fw, -1.f)));
    const int iu_hi = min(G.nu - 1, (int)floorf(fminf(fu + fw, (float)G.nu)));
    const int strideP = G.nu * (int)sizeof(float2), strideR = G.nu * (int)sizeof(float);
    for (int iu = iu_lo; iu <= iu_hi; ++iu) {
        const float u = ((float)iu - G.uc) * G.du + G.u_off;
        const float w = ac * u - b;
        const float qx = -w * s, qy = w * c;
        const float gx = -G.sdd * c - u * s;
        const float gy = -G.sdd * s + u * c;
        float glo = -ac, ghi = 1.f - ac;
        bool ok = true;
        slab_local_fast(qx, gx, G.hx, glo, ghi, ok);
        slab_local_fast(qy, gy, G.hy, glo, ghi, ok);
        if (!ok || !(glo < ghi)) continue;
        const float dg = ghi - glo;  // xy chord of this pixel column (ray-parameter units)
        const float sra = __fdividef(fvscale, ac + glo), srb = __fdividef(fvscale, ac + ghi);  // row maps (margin)
        const float idg = __fdividef(1.f, dg);
        const float cmid = 0.5f * (glo + ghi) * idg;  // the chord's midpoint in units of dg
        const char *pr = reinterpret_cast<const char *>(pv + iu) - kRowMagicBits * strideR;
        const char *pp = reinterpret_cast<const char *>(ppv + iu) - kRowMagicBits * strideP;
        // share of row iv's chord below z = zm: the ray rises (v > 0) or falls (v < 0) through the crossing
        // gs = (zm - ac v) / v, so the share is sat(sign(v) (gs - gmid) / dg + 1/2); a ray in the plane z = 0
        // (v = 0, 1/|v| = inf) lies below every zm > 0 and above every zm <= 0 (half-open cells): +-inf, or NaN
        // for zm = 0, saturate to 1 and 0; s_row[nv] and s_row[nv + 1] stand for no row: above every zm.  A row
        // with no share adds nothing whatever its value (not read as 0 * inf; row nv is not a row of this view).
        auto add_share = [&](float sum, int row, float zm, float r) {
            const float4 rw = s_row[row];  // (v, 1/|v|, sign of v)
            const float gs = fmaf(-ac, rw.x, zm) * rw.y;  // sign(v) gs
            const float share = __saturatef(fmaf(gs, idg, fmaf(-rw.z, cmid, 0.5f)));
            return share > 0.f ? fmaf(r, share, sum) : sum;
        };
        float hi_m = 0.f, lo_m = 0.f;  // B_m / dg as the prefix sum's high part and the rest
#pragma unroll
        for (int m = 0; m <= CH; ++m) {
            const float zm = fmaf((float)(iz0 + m), G.dz, G.b0z);
            const float pa = fmaf(zm, sra, fvlo), pb = fmaf(zm, srb, fvlo);
            const float lo = fmaxf(fminf(fminf(pa, pb), (float)G.nv), 0.f);
            const int jb = __float_as_int(__fadd_ru(lo, kRowMagic));  // L_m, biased by kRowMagicBits
            const float2 P = __ldg(reinterpret_cast<const float2 *>(at(pp, jb, strideP)));
            const float r = __ldg(reinterpret_cast<const float *>(at(pr, jb, strideR)));
            const int row = jb - (int)kRowMagicBits;
            float rest = add_share(P.y, row, zm, r);
            if (ROWS == 2) rest = add_share(rest, row + 1, zm, __ldg(reinterpret_cast<const float *>(at(pr, jb + 1, strideR))));
            if (ROWS == 0) {  // further rows of a wider band
                const int r1 = min(G.nv - 1, __float2int_rd(fmaxf(pa, pb) + 2e-3f));
                for (int iv = row + 1; iv <= r1; ++iv) rest = add_share(rest, iv, zm, __ldg(pv + iu + (long long)iv * G.nu));
            }
            if (m > 0) acc[m - 1] = fmaf((P.x - hi_m) + (rest - lo_m), dg, acc[m - 1]);
            hi_m = P.x;
            lo_m = rest;
        }
    }
}

// Resident warps per SM that the registers are budgeted for.  The 17 boundaries of 16 cells are one straight run
// of independent gathers, and 128 registers let their loads be issued ahead: on the 10 x 256x256x64 workload 16
// cells took 6.61 ms at 16 warps per SM, 7.5 at 20, 8.7 at 24; 8 cells 7.47 ms at 20 (7.8 at 16, 8.0 at 28), all
// before the addresses were written out (at() in ray_common.cuh), which took the chosen form to 6.39.
constexpr int bands_warps(int ch) { return ch == 16 ? 16 : 20; }

// NW warps of 8 x 4 voxel columns, each thread CH z cells of one column.  A voxel is the sum of ORDER partial sums over
// the views p, p + ORDER, ... of its phase, p = 0, 1, ... added in that order.  SPLIT = 1: the warps lie side by side
// (two along x) and each takes every partial sum in turn (those before in shared memory).  SPLIT = ORDER = NW: the warps
// share one patch of columns and warp p takes partial sum p, for launches too small to fill the GPU otherwise.
// The input is the ray-length-scaled residual (k_colscan writes a scaled copy of an unscaled input).  The chunk's
// boundaries beyond the volume (ragged nz) are computed like the others and their cells not stored.
// Bound by instruction issue (74 % of the slots, 22 instructions per boundary) with the L1's gathers behind it (67 %
// of its wavefront rate); 2.7 times faster per boundary than row tests with min/max bounds on both ends of each band
// and 32 x 1 column warps (k_backproject_bands at 10 x 256x256x64, 360 views x 512x384: 15.4 -> 6.3 ms, with k_colscan 15.5 -> 6.39).
template <int CH, int NW, int SPLIT, int ORDER, int ROWS, class T>
__global__ void __launch_bounds__(32 * NW, bands_warps(CH) / NW)
    k_backproject_bands(KGeom G, const ViewGeom *__restrict__ views, const int *__restrict__ view_off,
                        const float *__restrict__ proj, const float2 *__restrict__ pref, const T *vin,
                        T *vout, float alpha, float beta, int nchunks)
{
    static_assert(SPLIT == 1 || (SPLIT == NW && SPLIT == ORDER), "warps lie side by side or share one patch");
    constexpr int NT = 32 * NW;
    extern __shared__ float4 sm4[];
    float4 *s_row = sm4;  // per detector row: (v, 1/|v| or +inf, sign of v (+1 for v = 0), 0); [nv], [nv + 1]: no row
    const int tid = threadIdx.x;
    for (int t = tid; t < G.nv; t += NT) {
        const float v = ((float)t - G.vc) * G.dv + G.v_off;
        s_row[t] = make_float4(v, v != 0.f ? 1.0f / fabsf(v) : INFINITY, v < 0.f ? -1.f : 1.f, 0.f);
    }
    if (tid < 2) s_row[G.nv + tid] = make_float4(1e30f, 1.f, 1.f, 0.f);
    __syncthreads();
    const int lane = tid & 31, warp = tid >> 5;
    const int px = SPLIT > 1 ? (int)blockIdx.x : (int)blockIdx.x * 2 + (warp & 1);
    const int py = SPLIT > 1 ? (int)blockIdx.y : (int)blockIdx.y * (NW / 2) + (warp >> 1);
    const int ix = px * kBandWX + (lane & (kBandWX - 1)), iy = py * kBandWY + lane / kBandWX;
    const int phase = blockIdx.z / nchunks;
    const int iz0 = (blockIdx.z % nchunks) * CH;
    bool inside = ix < G.nx && iy < G.ny;
    if (SPLIT == 1 && !inside) return;
    float acc[CH];
#pragma unroll
    for (int k = 0; k < CH; ++k) acc[k] = 0.f;
    float *s_acc = reinterpret_cast<float *>(s_row + G.nv + 2);  // partial sums: [NW - 1][CH][32], unsplit [CH][NT]
    if (inside) {
        const float xc = G.b0x + ((float)ix + 0.5f) * G.dx;
        const float yc = G.b0y + ((float)iy + 0.5f) * G.dy;
        const int v0 = view_off[phase], v_end = view_off[phase + 1];
        // one loop over the views of all partial sums: with a loop per sum the 16-cell form took 6 % longer
        int vg = v0 + (SPLIT > 1 ? warp : 0), p = 0;
        while (vg < v_end) {
            bands_view<CH, ROWS>(G, s_row, views[vg].c, views[vg].s, xc, yc, iz0, proj + (long long)vg * G.npix,
                                  pref + (long long)vg * (G.nv + 1) * G.nu, acc);
            vg += ORDER;
            if (SPLIT > 1 || ORDER == 1 || vg < v_end) continue;
            vg = p + 1 < ORDER ? v0 + p + 1 : v_end;
#pragma unroll
            for (int k = 0; k < CH; ++k) {  // a thread reads only what it wrote itself
                if (p > 0) acc[k] = s_acc[k * NT + tid] + acc[k];
                if (vg < v_end) {
                    s_acc[k * NT + tid] = acc[k];
                    acc[k] = 0.f;
                }
            }
            ++p;
        }
    }
    if (SPLIT > 1) {
        if (warp > 0)
#pragma unroll
            for (int k = 0; k < CH; ++k) s_acc[((warp - 1) * CH + k) * 32 + lane] = acc[k];
        __syncthreads();
        inside = inside && warp == 0;
        if (!inside) return;
#pragma unroll
        for (int k = 0; k < CH; ++k)
#pragma unroll
            for (int w = 0; w < NW - 1; ++w) acc[k] += s_acc[(w * CH + k) * 32 + lane];
    }
    const long long base = (long long)phase * G.nvox + ((long long)iz0 * G.ny + iy) * G.nx + ix;
#pragma unroll
    for (int k = 0; k < CH; ++k) {
        if (iz0 + k < G.nz) {
            const long long o = base + (long long)k * G.nx * G.ny;
            const float bp = alpha * acc[k];
            st_v(vout + o, beta != 0.f ? fmaf(beta, ld_v(vin + o), bp) : bp);
        }
    }
}

}  // namespace

bool bands_apply(const KGeom &kg)
{
    // a ray's chord through one voxel column rises by at most |v|max / SDD per mm of horizontal path,
    // over at most the column's xy diagonal: keep it well below one cell height
    const double vmax = 0.5 * (kg.nv - 1) * (double)kg.dv + fabs((double)kg.v_off);
    const double rise = sqrt((double)kg.dx * kg.dx + (double)kg.dy * kg.dy) * vmax / (double)kg.sdd;
    return rise <= 0.9 * (double)kg.dz;
}

// The band transpose may read (and not use) the two rows after a view's last one, so a projection set it reads from is
// allocated two rows longer.
size_t projection_floats(const KGeom &kg, int n_views_total) { return (size_t)n_views_total * kg.npix + 2 * (size_t)kg.nu; }

size_t prefix_floats(const KGeom &kg, int n_views_total)
{
    // (hi, lo) prefix sums plus a ray-length-scaled copy of an unscaled input (projection_floats)
    return (size_t)2 * n_views_total * (kg.nv + 1) * kg.nu + projection_floats(kg, n_views_total);
}

// Detector rows that a z boundary's images at the two ends of a chord through one voxel column may lie apart, as the
// number of candidate rows (1, 2; 0: more), with the margins of bands_view: at depth U a chord of horizontal length
// diag moves the image v of a boundary by at most |v| diag / U.  Images off the detector do not count (no rows there).
static int band_rows(const KGeom &kg)
{
    const double x1 = fabs((double)kg.b0x), x2 = fabs((double)kg.b0x + (double)kg.nx * kg.dx);
    const double y1 = fabs((double)kg.b0y), y2 = fabs((double)kg.b0y + (double)kg.ny * kg.dy);
    const double z1 = fabs((double)kg.b0z), z2 = fabs((double)kg.b0z + (double)kg.nz * kg.dz);
    const double near = (double)kg.sad - hypot(fmax(x1, x2), fmax(y1, y2));  // > 0: the volume lies inside the orbit
    const double vmax = 0.5 * (kg.nv - 1) * (double)kg.dv + fabs((double)kg.v_off) + 2.0 * kg.dv;
    const double v = fmin(fmax(z1, z2) * kg.sdd / near, vmax);
    const double rows = v * hypot((double)kg.dx, (double)kg.dy) / (near * (double)kg.dv);
    return rows <= 0.98 ? 1 : (rows <= 1.98 ? 2 : 0);
}

template <int CH, int NW, int SPLIT, int ORDER, int ROWS, class T>
static tnlm_status launch_bands_m(const KGeom &kg, const ViewGeom *views, const int *view_off, const float *src,
                                  const float2 *pref, const T *vin, T *vout, float alpha, float beta, cudaStream_t st)
{
    const int nchb = (kg.nz + CH - 1) / CH;
    constexpr int TX = SPLIT > 1 ? kBandWX : 2 * kBandWX, TY = SPLIT > 1 ? kBandWY : (NW / 2) * kBandWY;
    dim3 grid((kg.nx + TX - 1) / TX, (kg.ny + TY - 1) / TY, kg.np * nchb);
    const size_t smem = sizeof(float4) * (kg.nv + 2) +
                        sizeof(float) * CH * (SPLIT > 1 ? (NW - 1) * 32 : (ORDER > 1 ? NW * 32 : 0));
    auto kern = k_backproject_bands<CH, NW, SPLIT, ORDER, ROWS, T>;
    if (smem > 48 * 1024)
        TNLM_TRY_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    kern<<<grid, 32 * NW, smem, st>>>(kg, views, view_off, src, pref, vin, vout, alpha, beta, nchb);
    TNLM_TRY_CUDA(cudaGetLastError());
    return TNLM_OK;
}

// Wide bands run in one shape per form (the result does not depend on it): pixels that fine against the voxels are
// rare, and the row loop, not the shape, sets their time.
template <int CH, int NW, int SPLIT, int ORDER, class T>
static tnlm_status launch_bands(const KGeom &kg, const ViewGeom *views, const int *view_off, const float *src,
                                const float2 *pref, const T *vin, T *vout, float alpha, float beta, cudaStream_t st)
{
    switch (band_rows(kg)) {
    case 1: return launch_bands_m<CH, NW, SPLIT, ORDER, 1, T>(kg, views, view_off, src, pref, vin, vout, alpha, beta, st);
    case 2: return launch_bands_m<CH, NW, SPLIT, ORDER, 2, T>(kg, views, view_off, src, pref, vin, vout, alpha, beta, st);
    default: return launch_bands_m<8, 4, SPLIT, ORDER, 0, T>(kg, views, view_off, src, pref, vin, vout, alpha, beta, st);
    }
}

// Blocks of 16 x 8 voxel columns and ch cells that np phases make
static long long band_blocks(const KGeom &kg, int np, int ch)
{
    return (long long)((kg.nx + 15) / 16) * ((kg.ny + 7) / 8) * np * ((kg.nz + ch - 1) / ch);
}

// A launch fills the GPU from about kBandsFill blocks, four resident on each of the 152 SMs; kBandsSplit is where the
// launches that take their partial sums in turn become the faster ones, with kBandsViews views a phase or more.
constexpr long long kBandsFill = 152 * 4, kBandsSplit = 152 * 10;
constexpr int kBandsViews = 10;

// Cells per thread: chunks of 8 where bp_ch asks for them and the volume has more than 4 slices, as the boundaries
// beyond the volume cost what the others do (6 x 192x192x1, 30 views of 256x192: 290 us in chunks of 8, 225 of 4; one
// phase of 256x256x1, 360 views of 512x64: 985 and 665).
static int band_cells(const KGeom &kg) { return kg.nz <= 4 ? 4 : kg.bp_ch; }

// The forms of the order of summation ORDER, by size.  With bp_ch = 8 and bp_by = 4 (the defaults) the chunk is 16 cells
// where the volume has them: a thread's chord set-up serves twice the cells (6.61 against 7.47 ms at 10 x 256x256x64),
// which padding an odd number of 8-cell chunks must not eat up.
template <int ORDER, class T>
static tnlm_status launch_bands_shape(const KGeom &kg, const ViewGeom *views, const int *view_off, const float *src,
                                      const float2 *pref, const T *vin, T *vout, float alpha, float beta,
                                      cudaStream_t st)
{
    const int n8 = (kg.nz + 7) / 8, ch = band_cells(kg);
    if (ch == 8 && kg.bp_by == 4 && band_blocks(kg, kg.np, 16) >= kBandsFill && (n8 % 2 == 0 || n8 > 8))
        return launch_bands<16, 4, 1, ORDER, T>(kg, views, view_off, src, pref, vin, vout, alpha, beta, st);
    if (ch == 8 && kg.bp_by == 4)
        return launch_bands<8, 4, 1, ORDER, T>(kg, views, view_off, src, pref, vin, vout, alpha, beta, st);
    if (ch == 8 && kg.bp_by == 2)
        return launch_bands<8, 2, 1, ORDER, T>(kg, views, view_off, src, pref, vin, vout, alpha, beta, st);
    if (ch == 4 && kg.bp_by == 4)
        return launch_bands<4, 4, 1, ORDER, T>(kg, views, view_off, src, pref, vin, vout, alpha, beta, st);
    return launch_bands<4, 2, 1, ORDER, T>(kg, views, view_off, src, pref, vin, vout, alpha, beta, st);
}

// The form of the band transpose by size.  Volumes of which one phase does not fill the GPU are summed in four partial
// sums, so that the warps of a block can split the views of one patch where the whole launch is small (4 x 32^3, 20
// views: stage 37 -> 25 us; 27 us in chunks of 4).  The order depends on the volume alone, not on how many phases the
// handle holds, so a rank that holds some of a scan's phases gets the bits of a process that holds all.  Partial sums in
// turn / split, 36 views a phase, by the launch's blocks: 768 (6 of 64x64x32) 175 / 142 us, 1024 (4 of 64^3) 197 / 186,
// 1280 (10 of 64x64x32) 241 / 219, 1536 (6 of 64^3) 266 / 265, 2304 (4 of 96x96x64) 339 / 378, 2560 (10 of 64^3) 411 / 446;
// 4 of 64^3 by views: 1 28 / 36, 4 45 / 46, 9 66 / 72, 12 82 / 81, 60 315 / 294.
template <class T>
static tnlm_status launch_bands_by_size(const KGeom &kg, const ViewGeom *views, const int *view_off, const float *src,
                                        const float2 *pref, const T *vin, T *vout, float alpha, float beta,
                                        int n_views_total, cudaStream_t st)
{
    if (band_blocks(kg, 1, 8) >= kBandsFill)
        return launch_bands_shape<1, T>(kg, views, view_off, src, pref, vin, vout, alpha, beta, st);
    if (band_blocks(kg, kg.np, 8) >= (n_views_total >= kBandsViews * kg.np ? kBandsSplit : kBandsFill))
        return launch_bands_shape<4, T>(kg, views, view_off, src, pref, vin, vout, alpha, beta, st);
    if (band_cells(kg) == 8)
        return launch_bands<8, 4, 4, 4, T>(kg, views, view_off, src, pref, vin, vout, alpha, beta, st);
    return launch_bands<4, 4, 4, 4, T>(kg, views, view_off, src, pref, vin, vout, alpha, beta, st);
}

template <class T>
static tnlm_status launch_backproject_t(const KGeom &kg, const ViewGeom *views, const int *view_off, const float *proj,
                                        const T *vin, T *vout, float alpha, float beta, bool scaled, float *pref_ws,
                                        int n_views_total, cudaStream_t st)
{
    const int nchunks = (kg.nz + kBpCH - 1) / kBpCH;
    dim3 block(kBpBX, kBpBY);
    dim3 grid((kg.nx + kBpBX - 1) / kBpBX, (kg.ny + kBpBY - 1) / kBpBY, kg.np * nchunks);
    if (pref_ws && bands_apply(kg)) {
        float2 *pref = reinterpret_cast<float2 *>(pref_ws);
        float *rtil = pref_ws + (size_t)2 * n_views_total * (kg.nv + 1) * kg.nu;  // unscaled input: r |D| copy
        dim3 sg((kg.nu + 255) / 256, n_views_total);
        if (scaled)
            k_colscan<true><<<sg, 256, 0, st>>>(kg, proj, pref, nullptr);
        else
            k_colscan<false><<<sg, 256, 0, st>>>(kg, proj, pref, rtil);
        TNLM_TRY_CUDA(cudaGetLastError());
        const float *src = scaled ? proj : rtil;
        if ((kg.bp_ch != 4 && kg.bp_ch != 8) || (kg.bp_by != 2 && kg.bp_by != 4)) {
            set_error("band transpose shape must be CH in {4, 8} and BY in {2, 4} (got %d, %d)", kg.bp_ch, kg.bp_by);
            return TNLM_ERR_ARG;
        }
        TNLM_TRY(launch_bands_by_size<T>(kg, views, view_off, src, pref, vin, vout, alpha, beta, n_views_total, st));
        return TNLM_OK;
    }
    const size_t smem = sizeof(float4) * kg.nv + sizeof(float) * kBpCH * kBpBX * kBpBY;
    if (smem > 48 * 1024) {
        TNLM_TRY_CUDA(cudaFuncSetAttribute(k_backproject<true, T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        TNLM_TRY_CUDA(cudaFuncSetAttribute(k_backproject<false, T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    }
    if (scaled)
        k_backproject<true, T><<<grid, block, smem, st>>>(kg, views, view_off, proj, vin, vout, alpha, beta, nchunks);
    else
        k_backproject<false, T><<<grid, block, smem, st>>>(kg, views, view_off, proj, vin, vout, alpha, beta, nchunks);
    TNLM_TRY_CUDA(cudaGetLastError());
    return TNLM_OK;
}

tnlm_status launch_backproject(const KGeom &kg, const ViewGeom *views, const int *view_off, const float *proj,
                               const float *vin, float *vout, float alpha, float beta, bool scaled, float *pref_ws,
                               int n_views_total, cudaStream_t st)
{
    return launch_backproject_t<float>(kg, views, view_off, proj, vin, vout, alpha, beta, scaled, pref_ws,
                                       n_views_total, st);
}

tnlm_status launch_backproject(const KGeom &kg, const ViewGeom *views, const int *view_off, const float *proj,
                               const uint16_t *vin, uint16_t *vout, float alpha, float beta, bool scaled,
                               float *pref_ws, int n_views_total, cudaStream_t st)
{
    using B = __nv_bfloat16;
    return launch_backproject_t<B>(kg, views, view_off, proj, reinterpret_cast<const B *>(vin),
                                   reinterpret_cast<B *>(vout), alpha, beta, scaled, pref_ws, n_views_total, st);
}

tnlm_status launch_backproject(const KGeom &kg, const ViewGeom *views, const int *view_off, const float *proj,
                               const __half *vin, __half *vout, float alpha, float beta, bool scaled,
                               float *pref_ws, int n_views_total, cudaStream_t st)
{
    return launch_backproject_t<__half>(kg, views, view_off, proj, vin, vout, alpha, beta, scaled, pref_ws,
                                        n_views_total, st);
}

}  // namespace tnlm
