// Total energy of Eq. 1 (with the J of Eq. 2 over the search window and the
// Eq. 9 weights frozen, computed from weight-source images a) and its
// gradient, for differentiable use:
//   E(f)   = mu/2 sum_i ||P_i f_i - y_i||^2 + 1/2 sum_i J[f_i, f_{i+1}],
//   grad_i(x) = mu (P_i^T (P_i f_i - y_i))(x)
//               + sum_delta w_i(x, delta) (f_i(x) - f_{i+1}(x + delta))
//               + sum_{y = x + delta'} w_{i-1}(y, x - y) (f_i(x) - f_{i-1}(y)),
// with w_i the row-normalised weights of phase i toward i+1 (the second line
// is W_i applied to the differences, the third the transposed term of
// W_{i-1}); each pair adds its own difference, so nothing of size f cancels
// when f is close to its weighted means.  The transposed term needs, at voxel y of phase i,
// the weight that the voxel x = y + delta' of phase i-1 gives to y; it uses
// x's own normaliser, so a first pass stores Lambda(x) = log2 Z(x) - m(x)
// per voxel (k_lognorm) and the gradient pass (k_energy_grad) gathers both
// directions with w = 2^(-t - Lambda), t = D log2(e) / 2h^2.  Patch distances
// are summed in the same order in both passes, so the two see identical t.
#include <cfloat>
#include <cmath>
#include <type_traits>

#include "tnlm_internal.cuh"

namespace tnlm {
namespace {

constexpr int kTX = 8, kTY = 8, kTZ = 4;  // output tile of one CTA
constexpr int kNT = kTX * kTY * kTZ;
constexpr float kRescale = 16.f;

__device__ __forceinline__ float ex2(float x)
{
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

__device__ __forceinline__ int clampi(int a, int n) { return a < 0 ? 0 : (a >= n ? n - 1 : a); }

__device__ __forceinline__ void stage(float *dst, const float *__restrict__ src, int ox, int oy, int oz, int ex,
                                      int ey, int ez, int nx, int ny, int nz, int tid)
{
    const int n = ex * ey * ez;
    for (int t = tid; t < n; t += kNT) {
        const int lx = t % ex, ly = (t / ex) % ey, lz = t / (ex * ey);
        dst[t] = __ldg(src + ((long long)clampi(oz + lz, nz) * ny + clampi(oy + ly, ny)) * nx + clampi(ox + lx, nx));
    }
}

// squared patch distance between the staged patch of phase i at the thread's
// voxel and the staged neighbour patch at window offset (dx, dy, dz)
__device__ __forceinline__ float patch_dist(const float *s_ai, const float *s_aj, int tx, int ty, int tz, int dx,
                                            int dy, int dz, int d, int R)
{
    const int aix = kTX + 2 * d, aiy = kTY + 2 * d;
    const int ajx = kTX + 2 * R, ajy = kTY + 2 * R;
    float D = 0.f;
    for (int oz = -d; oz <= d; ++oz)
        for (int oy = -d; oy <= d; ++oy) {
            const float *pa = s_ai + ((tz + d + oz) * aiy + (ty + d + oy)) * aix + (tx + d);
            const float *pb = s_aj + ((tz + R + dz + oz) * ajy + (ty + R + dy + oy)) * ajx + (tx + R + dx);
            for (int ox = -d; ox <= d; ++ox) {
                const float t = pa[ox] - pb[ox];
                D = fmaf(t, t, D);
            }
        }
    return D;
}

// Lambda_i(x) = log2 sum_delta 2^(m - t) - m over the valid window toward phase i+1
__global__ void __launch_bounds__(kNT) k_lognorm(int nx, int ny, int nz, int np, int ntz, const float *__restrict__ a,
                                                 int d, int M, float c2, float *__restrict__ lam)
{
    extern __shared__ float sm[];
    const int R = M + d;
    float *s_ai = sm;
    float *s_aj = s_ai + (kTX + 2 * d) * (kTY + 2 * d) * (kTZ + 2 * d);
    const int tx = threadIdx.x, ty = threadIdx.y, tz = threadIdx.z, tid = (tz * kTY + ty) * kTX + tx;
    const int i = blockIdx.z / ntz;
    const int X0 = blockIdx.x * kTX, Y0 = blockIdx.y * kTY, Z0 = (blockIdx.z % ntz) * kTZ;
    const long long nvox = (long long)nx * ny * nz;
    const int x = X0 + tx, y = Y0 + ty, z = Z0 + tz;
    const int j = (i + 1) % np;
    stage(s_ai, a + i * nvox, X0 - d, Y0 - d, Z0 - d, kTX + 2 * d, kTY + 2 * d, kTZ + 2 * d, nx, ny, nz, tid);
    stage(s_aj, a + j * nvox, X0 - R, Y0 - R, Z0 - R, kTX + 2 * R, kTY + 2 * R, kTZ + 2 * R, nx, ny, nz, tid);
    __syncthreads();
    float mref = FLT_MAX, Z = 0.f;
    for (int dz = -M; dz <= M; ++dz) {
        if ((unsigned)(z + dz) >= (unsigned)nz) continue;
        for (int dy = -M; dy <= M; ++dy) {
            if ((unsigned)(y + dy) >= (unsigned)ny) continue;
            for (int dx = -M; dx <= M; ++dx) {
                if ((unsigned)(x + dx) >= (unsigned)nx) continue;
                const float t = patch_dist(s_ai, s_aj, tx, ty, tz, dx, dy, dz, d, R) * c2;
                if (t < mref - kRescale) {
                    Z *= ex2(t - mref);
                    mref = t;
                }
                Z += ex2(mref - t);
            }
        }
    }
    if (x < nx && y < ny && z < nz) lam[i * nvox + ((long long)z * ny + y) * nx + x] = log2f(Z) - mref;
}

__global__ void __launch_bounds__(kNT) k_energy_grad(int nx, int ny, int nz, int np, int ntz,
                                                     const float *__restrict__ a, const float *__restrict__ f,
                                                     const float *__restrict__ lam, int d, int M, float c2,
                                                     float *__restrict__ grad, double *__restrict__ jpart)
{
    extern __shared__ float sm[];
    __shared__ double ws[kNT / 32];
    const int R = M + d;
    const int aiN = (kTX + 2 * d) * (kTY + 2 * d) * (kTZ + 2 * d);
    const int ajN = (kTX + 2 * R) * (kTY + 2 * R) * (kTZ + 2 * R);
    const int vjx = kTX + 2 * M, vjy = kTY + 2 * M, vjz = kTZ + 2 * M;
    float *s_ai = sm;
    float *s_aj = s_ai + aiN;
    float *s_fj = s_aj + ajN;            // neighbour values
    float *s_lj = s_fj + vjx * vjy * vjz;  // neighbour normalisers (direction i-1 only)
    const int tx = threadIdx.x, ty = threadIdx.y, tz = threadIdx.z, tid = (tz * kTY + ty) * kTX + tx;
    const int i = blockIdx.z / ntz;
    const int X0 = blockIdx.x * kTX, Y0 = blockIdx.y * kTY, Z0 = (blockIdx.z % ntz) * kTZ;
    const long long nvox = (long long)nx * ny * nz;
    const int x = X0 + tx, y = Y0 + ty, z = Z0 + tz;
    const bool inside = x < nx && y < ny && z < nz;
    const long long o = i * nvox + ((long long)clampi(z, nz) * ny + clampi(y, ny)) * nx + clampi(x, nx);
    const float fi = __ldg(f + o), li = __ldg(lam + o);
    stage(s_ai, a + i * nvox, X0 - d, Y0 - d, Z0 - d, kTX + 2 * d, kTY + 2 * d, kTZ + 2 * d, nx, ny, nz, tid);
    float term1 = 0.f, term2 = 0.f, jy = 0.f;
    for (int dir = 0; dir < 2; ++dir) {
        const int j = dir == 0 ? (i + 1) % np : (i - 1 + np) % np;
        __syncthreads();
        stage(s_aj, a + j * nvox, X0 - R, Y0 - R, Z0 - R, kTX + 2 * R, kTY + 2 * R, kTZ + 2 * R, nx, ny, nz, tid);
        stage(s_fj, f + j * nvox, X0 - M, Y0 - M, Z0 - M, vjx, vjy, vjz, nx, ny, nz, tid);
        if (dir == 1) stage(s_lj, lam + j * nvox, X0 - M, Y0 - M, Z0 - M, vjx, vjy, vjz, nx, ny, nz, tid);
        __syncthreads();
        for (int dz = -M; dz <= M; ++dz) {
            if ((unsigned)(z + dz) >= (unsigned)nz) continue;
            for (int dy = -M; dy <= M; ++dy) {
                if ((unsigned)(y + dy) >= (unsigned)ny) continue;
                for (int dx = -M; dx <= M; ++dx) {
                    if ((unsigned)(x + dx) >= (unsigned)nx) continue;
                    const float t = patch_dist(s_ai, s_aj, tx, ty, tz, dx, dy, dz, d, R) * c2;
                    const int q = ((tz + M + dz) * vjy + (ty + M + dy)) * vjx + (tx + M + dx);
                    const float fj = s_fj[q];
                    const float df = fi - fj;
                    if (dir == 0) {  // this voxel's own weights toward phase i+1
                        const float w = ex2(-t - li);
                        term1 = fmaf(w, df, term1);
                        jy = fmaf(w, df * df, jy);
                    } else {  // weights of the phase i-1 voxel y+delta toward this voxel
                        const float w = ex2(-t - s_lj[q]);
                        term2 = fmaf(w, df, term2);
                    }
                }
            }
        }
    }
    if (inside) grad[o] += term1 + term2;
    // block partial of J (FP64)
    double v = inside ? (double)jy : 0.0;
    for (int off = 16; off > 0; off >>= 1) v += __shfl_down_sync(0xffffffffu, v, off);
    if ((tid & 31) == 0) ws[tid >> 5] = v;
    __syncthreads();
    if (tid == 0) {
        double s = 0.0;
        for (int k = 0; k < kNT / 32; ++k) s += ws[k];
        jpart[((long long)blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x] = s;
    }
}

// ---------------------------------------------------------------------------
// Gradient of 1/2 sum_i J[f_i, f_{i+1}] through the weights, with respect to
// the weight-source images a (f fixed).  With c = 1/(2h^2),
//   G(x,delta) = dJ_x/dD(x,delta) = 1/2 c w(x,delta) (Qbar(x) - q(x,delta)),
//   Qbar(x) = sum_delta w q,  q = (f_i(x) - f_j(x+delta))^2,  j = i+1,
// and D(x,delta) = sum_o s(x+o), s(p) = (a_i(cl(p)) - a_j(cl(p+delta)))^2 on
// the grid padded by d (cl = clamp to the volume).  So, with the box sum
// B(p,delta) = sum_o G(p-o,delta) over the x inside the volume,
//   v(p,delta) = 2 B(p,delta) (a_i(cl(p)) - a_j(cl(p+delta))),
//   grad_i(z) += sum over p with cl(p) = z of sum_delta v(p,delta),
//   grad_j(z) -= sum over (p,delta) with cl(p+delta) = z of v(p,delta).
// Per phase pair: k_wa_G writes G[delta][x] (0 for invalid candidates),
// k_wa_B writes B[delta][p] on the padded grid, k_wa_sides sums both sides
// over delta at every (clamped) position of a grid padded by d + M, and
// k_wa_fold adds the positions that clamp to a voxel (gathers only; no
// atomics, deterministic).

__global__ void __launch_bounds__(kNT) k_wa_G(int nx, int ny, int nz, int ntz, const float *__restrict__ ai,
                                              const float *__restrict__ aj, const float *__restrict__ fi,
                                              const float *__restrict__ fj, int d, int M, float c2, float cg,
                                              float *__restrict__ G)
{
    extern __shared__ float sm[];
    const int R = M + d;
    const int vjx = kTX + 2 * M, vjy = kTY + 2 * M, vjz = kTZ + 2 * M;
    float *s_ai = sm;
    float *s_aj = s_ai + (kTX + 2 * d) * (kTY + 2 * d) * (kTZ + 2 * d);
    float *s_fj = s_aj + (kTX + 2 * R) * (kTY + 2 * R) * (kTZ + 2 * R);
    const int tx = threadIdx.x, ty = threadIdx.y, tz = threadIdx.z, tid = (tz * kTY + ty) * kTX + tx;
    const int X0 = blockIdx.x * kTX, Y0 = blockIdx.y * kTY, Z0 = blockIdx.z * kTZ;
    const long long nvox = (long long)nx * ny * nz;
    const int x = X0 + tx, y = Y0 + ty, z = Z0 + tz;
    const bool inside = x < nx && y < ny && z < nz;
    const long long o = ((long long)clampi(z, nz) * ny + clampi(y, ny)) * nx + clampi(x, nx);
    const float f0 = __ldg(fi + o);
    stage(s_ai, ai, X0 - d, Y0 - d, Z0 - d, kTX + 2 * d, kTY + 2 * d, kTZ + 2 * d, nx, ny, nz, tid);
    stage(s_aj, aj, X0 - R, Y0 - R, Z0 - R, kTX + 2 * R, kTY + 2 * R, kTZ + 2 * R, nx, ny, nz, tid);
    stage(s_fj, fj, X0 - M, Y0 - M, Z0 - M, vjx, vjy, vjz, nx, ny, nz, tid);
    __syncthreads();
    (void)ntz;
    // pass 1: normaliser and weighted mean of q (online reference as in the sweep)
    float mref = FLT_MAX, Z = 0.f, S = 0.f;
    for (int dz = -M; dz <= M; ++dz) {
        if ((unsigned)(z + dz) >= (unsigned)nz) continue;
        for (int dy = -M; dy <= M; ++dy) {
            if ((unsigned)(y + dy) >= (unsigned)ny) continue;
            for (int dx = -M; dx <= M; ++dx) {
                if ((unsigned)(x + dx) >= (unsigned)nx) continue;
                const float t = patch_dist(s_ai, s_aj, tx, ty, tz, dx, dy, dz, d, R) * c2;
                const float df = f0 - s_fj[((tz + M + dz) * vjy + (ty + M + dy)) * vjx + (tx + M + dx)];
                if (t < mref - kRescale) {
                    const float sc = ex2(t - mref);
                    Z *= sc;
                    S *= sc;
                    mref = t;
                }
                const float e = ex2(mref - t);
                Z += e;
                S = fmaf(e, df * df, S);
            }
        }
    }
    const float lam = log2f(Z) - mref, qbar = S / Z;
    // pass 2: G for every window offset (0 where the candidate is outside the volume)
    int k = 0;
    for (int dz = -M; dz <= M; ++dz)
        for (int dy = -M; dy <= M; ++dy)
            for (int dx = -M; dx <= M; ++dx, ++k) {
                float g = 0.f;
                if ((unsigned)(z + dz) < (unsigned)nz && (unsigned)(y + dy) < (unsigned)ny &&
                    (unsigned)(x + dx) < (unsigned)nx) {
                    const float t = patch_dist(s_ai, s_aj, tx, ty, tz, dx, dy, dz, d, R) * c2;
                    const float df = f0 - s_fj[((tz + M + dz) * vjy + (ty + M + dy)) * vjx + (tx + M + dx)];
                    g = cg * ex2(-t - lam) * (qbar - df * df);
                }
                if (inside) G[(long long)k * nvox + ((long long)z * ny + y) * nx + x] = g;
            }
}

// B[k][p] = sum over o in [-d,d]^3 with x = p - o inside the volume of G[k][x];
// p on the padded grid [-d, n+d)^3, stored at (p + d).  A warp takes 32 - 2d
// positions of one row and one offset through every z (CUT: nch runs of len): 2d + 1
// coalesced loads a slice, the x sum by shuffles, the z sum from a ring of slice
// sums (27 loads a position otherwise: 1.17 -> 0.38 ms per phase pair of 95 x 90
// x 71, M = 2).
template <int D, bool CUT>
__global__ void __launch_bounds__(256) k_wa_B(int nx, int ny, int nz, int nch, int len, const float *__restrict__ G,
                                              float *__restrict__ B)
{
    const int px_n = nx + 2 * D, py_n = ny + 2 * D, pz_n = nz + 2 * D;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int tx = blockIdx.x * (32 - 2 * D) + lane - D;  // position in the padded row
    const int ty = blockIdx.y * 8 + warp;
    if (ty >= py_n) return;
    const int gx = tx - D, gy = ty - D;
    const int k = CUT ? blockIdx.z / nch : blockIdx.z, z0 = CUT ? (blockIdx.z % nch) * len : 0;
    const int z1 = CUT ? min(z0 + len, pz_n) : pz_n;
    const float *__restrict__ Gk = G + (long long)k * nx * ny * nz;
    float *__restrict__ Bk = B + (long long)k * px_n * py_n * pz_n + (long long)ty * px_n + tx;
    const bool in_x = gx >= 0 && gx < nx, out = lane >= D && lane < 32 - D && tx < px_n;
    const int y0 = max(gy - D, 0), y1 = min(gy + D, ny - 1);
    float ring[2 * D + 1];
#pragma unroll
    for (int i = 0; i <= 2 * D; ++i) ring[i] = 0.f;
    for (int z = CUT ? z0 - 2 * D : 0; z < z1; ++z) {
        float s = 0.f;
        if (in_x && (!CUT || z >= 0) && z < nz) {
            const float *__restrict__ row = Gk + (long long)z * ny * nx + gx;
            for (int y = y0; y <= y1; ++y) s += __ldg(row + (long long)y * nx);
        }
        float c = s;
#pragma unroll
        for (int o = 1; o <= D; ++o) c += __shfl_up_sync(0xffffffffu, s, o) + __shfl_down_sync(0xffffffffu, s, o);
#pragma unroll
        for (int i = 0; i < 2 * D; ++i) ring[i] = ring[i + 1];
        ring[2 * D] = c;
        float b = ring[0];
#pragma unroll
        for (int i = 1; i <= 2 * D; ++i) b += ring[i];
        if (out && (!CUT || z >= z0)) Bk[(long long)z * py_n * px_n] = b;
    }
}

// At every position r of the grid padded by d + M: side j, the sum over (p, delta) with p + delta = r of v; and
// inside the padding d, side i, the sum over delta of v(r, delta).  Clamping to voxels is left to k_wa_fold, so that
// the sums are the same straight run of loads everywhere (a range of positions per voxel at the faces otherwise).
template <int M>
__global__ void __launch_bounds__(256) k_wa_sides(int nx, int ny, int nz, int d, const float *__restrict__ ai,
                                                  const float *__restrict__ aj, const float *__restrict__ B,
                                                  float *__restrict__ side_i, float *__restrict__ side_j)
{
    const int R = d + M, ex_n = nx + 2 * R, ey_n = ny + 2 * R, ez_n = nz + 2 * R;
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= (long long)ex_n * ey_n * ez_n) return;
    const int x = (int)(t % ex_n) - R, y = (int)((t / ex_n) % ey_n) - R, z = (int)(t / ((long long)ex_n * ey_n)) - R;
    const int px_n = nx + 2 * d, py_n = ny + 2 * d, pz_n = nz + 2 * d;
    const int pn_yx = px_n * py_n;
    const long long pn = (long long)pn_yx * pz_n;
    const long long c = ((long long)clampi(z, nz) * ny + clampi(y, ny)) * nx + clampi(x, nx);
    const float air = __ldg(ai + c), ajr = __ldg(aj + c);
    auto in_pad = [&](int v, int n) { return v >= -d && v < n + d; };
    const bool own = in_pad(x, nx) && in_pad(y, ny) && in_pad(z, nz);
    const long long pos = (long long)(z + d) * pn_yx + (long long)(y + d) * px_n + (x + d);  // of r in B
    int cx[2 * M + 1];
    bool okx[2 * M + 1];
#pragma unroll
    for (int e = 0; e <= 2 * M; ++e) {
        cx[e] = clampi(x + e - M, nx);
        okx[e] = in_pad(x - (e - M), nx);
    }
    float si = 0.f, sj = 0.f;
    const float *__restrict__ Bk = B;
    for (int dz = -M; dz <= M; ++dz)
        for (int dy = -M; dy <= M; ++dy) {
            const bool oky = in_pad(z - dz, nz) && in_pad(y - dy, ny);
            const float *__restrict__ aj_row = aj + ((long long)clampi(z + dz, nz) * ny + clampi(y + dy, ny)) * nx;
            const float *__restrict__ ai_row = ai + ((long long)clampi(z - dz, nz) * ny + clampi(y - dy, ny)) * nx;
            const long long back = pos - (long long)dz * pn_yx - (long long)dy * px_n;
#pragma unroll
            for (int e = 0; e <= 2 * M; ++e, Bk += pn) {
                if (own) si = fmaf(2.f * __ldg(Bk + pos), air - __ldg(aj_row + cx[e]), si);
                if (oky && okx[e]) sj = fmaf(2.f * __ldg(Bk + back - (e - M)), __ldg(ai_row + cx[2 * M - e]) - ajr, sj);
            }
        }
    if (own) side_i[pos] = si;
    side_j[t] = sj;
}

// grad_i(z) += side i over the positions of the grid padded by d that clamp to z, grad_j(z) -= side j over those of
// the grid padded by d + M
__global__ void __launch_bounds__(256) k_wa_fold(int nx, int ny, int nz, int d, int R, const float *__restrict__ side_i,
                                                 const float *__restrict__ side_j, float *__restrict__ gi,
                                                 float *__restrict__ gj)
{
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= (long long)nx * ny * nz) return;
    const int x = (int)(t % nx), y = (int)((t / nx) % ny), z = (int)(t / ((long long)nx * ny));
    auto fold = [&](const float *__restrict__ s, int r) {
        float sum = 0.f;
        for (int a = z == 0 ? -r : z; a <= (z == nz - 1 ? nz - 1 + r : z); ++a)
            for (int b = y == 0 ? -r : y; b <= (y == ny - 1 ? ny - 1 + r : y); ++b)
                for (int c = x == 0 ? -r : x; c <= (x == nx - 1 ? nx - 1 + r : x); ++c)
                    sum += __ldg(s + ((long long)(a + r) * (ny + 2 * r) + (b + r)) * (nx + 2 * r) + (c + r));
        return sum;
    };
    gi[t] += fold(side_i, d);
    gj[t] -= fold(side_j, R);
}

}  // namespace

size_t energy_weights_grad_floats(int nx, int ny, int nz, int np, int d, int M)
{
    const size_t W = (size_t)(2 * M + 1) * (2 * M + 1) * (2 * M + 1);
    const size_t nvox = (size_t)nx * ny * nz;
    const size_t pn = (size_t)(nx + 2 * d) * (ny + 2 * d) * (nz + 2 * d);
    const int R = 2 * (d + M);
    // G and its box sum B, the box path's normalisers and weighted means of q (all phases), the two sides of a pair
    return W * (nvox + pn) + 2 * (size_t)np * nvox + pn + (size_t)(nx + R) * (ny + R) * (nz + R);
}

tnlm_status launch_wa_box_gather(int nx, int ny, int nz, int np, int i, int d, int M, const float *a, const float *G,
                                 float *B, float *grad_a, cudaStream_t st)
{
    const long long nvox = (long long)nx * ny * nz;
    const int S = 2 * M + 1, W = S * S * S;
    const long long pn = (long long)(nx + 2 * d) * (ny + 2 * d) * (nz + 2 * d);
    const int j = (i + 1) % np;
    const float *ai = a + (long long)i * nvox, *aj = a + (long long)j * nvox;
    const int R = d + M;
    float *side_i = B + (size_t)W * pn + 2 * (size_t)np * nvox, *side_j = side_i + pn;
    // z is cut into runs of 8 or more where whole marches are too few blocks (four on each of the 152 SMs), as with a window
    // of one candidate (4 x 64^3, d = 1, M = 0: call 304 -> 178 us); the sums do not depend on the cuts
    const int gx = (nx + 2 * d + 31 - 2 * d) / (32 - 2 * d), gy = (ny + 2 * d + 7) / 8, pz = nz + 2 * d;
    const long long blocks = (long long)gx * gy * W;
    const int cuts = (int)(blocks < 608 ? 608 / blocks : 1), runs = cuts < (pz + 7) / 8 ? cuts : (pz + 7) / 8;
    const int len = (pz + runs - 1) / runs, nch = (pz + len - 1) / len;
    const dim3 grid(gx, gy, W * nch);
    auto box = [&](auto cut_tag) {
        constexpr bool CUT = decltype(cut_tag)::value;
        switch (d) {
        case 0: k_wa_B<0, CUT><<<grid, 256, 0, st>>>(nx, ny, nz, nch, len, G, B); break;
        case 1: k_wa_B<1, CUT><<<grid, 256, 0, st>>>(nx, ny, nz, nch, len, G, B); break;
        case 2: k_wa_B<2, CUT><<<grid, 256, 0, st>>>(nx, ny, nz, nch, len, G, B); break;
        default: k_wa_B<3, CUT><<<grid, 256, 0, st>>>(nx, ny, nz, nch, len, G, B); break;  // check_sweep_args: d <= 3
        }
    };
    if (nch > 1)
        box(std::true_type{});
    else
        box(std::false_type{});
    TNLM_TRY_CUDA(cudaGetLastError());
    const long long en = (long long)(nx + 2 * R) * (ny + 2 * R) * (nz + 2 * R);
    const unsigned eb = (unsigned)((en + 255) / 256);
    switch (M) {
    case 0: k_wa_sides<0><<<eb, 256, 0, st>>>(nx, ny, nz, d, ai, aj, B, side_i, side_j); break;
    case 1: k_wa_sides<1><<<eb, 256, 0, st>>>(nx, ny, nz, d, ai, aj, B, side_i, side_j); break;
    case 2: k_wa_sides<2><<<eb, 256, 0, st>>>(nx, ny, nz, d, ai, aj, B, side_i, side_j); break;
    case 3: k_wa_sides<3><<<eb, 256, 0, st>>>(nx, ny, nz, d, ai, aj, B, side_i, side_j); break;
    default: k_wa_sides<4><<<eb, 256, 0, st>>>(nx, ny, nz, d, ai, aj, B, side_i, side_j); break;  // M <= 4
    }
    TNLM_TRY_CUDA(cudaGetLastError());
    k_wa_fold<<<(unsigned)((nvox + 255) / 256), 256, 0, st>>>(nx, ny, nz, d, R, side_i, side_j, grad_a + (long long)i * nvox,
                                                              grad_a + (long long)j * nvox);
    TNLM_TRY_CUDA(cudaGetLastError());
    return TNLM_OK;
}

tnlm_status launch_energy_weights_grad(int nx, int ny, int nz, int np, const float *f, const float *a, int d, int M,
                                       float h, float *grad_a, float *ws, cudaStream_t st)
{
    const long long nvox = (long long)nx * ny * nz;
    const int S = 2 * M + 1, W = S * S * S, R = M + d;
    float *G = ws, *B = ws + (size_t)W * nvox;
    const long long pn = (long long)(nx + 2 * d) * (ny + 2 * d) * (nz + 2 * d);
    // the box-sum form of the normalisers and of G where it is compiled, the direct tiled form otherwise
    float *lam = B + (size_t)W * pn, *qbar = lam + (size_t)np * nvox;
    tnlm_status status = TNLM_OK;
    if (launch_energy_weights_grad_box(d, M, nx, ny, nz, np, f, a, h, grad_a, ws, lam, qbar, st, &status))
        return status;
    const float c2 = (float)(1.4426950408889634 / (2.0 * (double)h * (double)h));
    const float cg = (float)(0.5 / (2.0 * (double)h * (double)h));
    const size_t smem = sizeof(float) * ((size_t)(kTX + 2 * d) * (kTY + 2 * d) * (kTZ + 2 * d) +
                                         (size_t)(kTX + 2 * R) * (kTY + 2 * R) * (kTZ + 2 * R) +
                                         (size_t)(kTX + 2 * M) * (kTY + 2 * M) * (kTZ + 2 * M));
    if (smem > 48 * 1024) TNLM_TRY_CUDA(cudaFuncSetAttribute(k_wa_G, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    TNLM_TRY_CUDA(cudaMemsetAsync(grad_a, 0, sizeof(float) * (size_t)np * nvox, st));
    const int ntz = (nz + kTZ - 1) / kTZ;
    dim3 block(kTX, kTY, kTZ), grid((nx + kTX - 1) / kTX, (ny + kTY - 1) / kTY, ntz);
    for (int i = 0; i < np; ++i) {
        const int j = (i + 1) % np;
        const float *ai = a + (long long)i * nvox, *aj = a + (long long)j * nvox;
        k_wa_G<<<grid, block, smem, st>>>(nx, ny, nz, ntz, ai, aj, f + (long long)i * nvox, f + (long long)j * nvox, d, M,
                                          c2, cg, G);
        TNLM_TRY_CUDA(cudaGetLastError());
        TNLM_TRY(launch_wa_box_gather(nx, ny, nz, np, i, d, M, a, G, B, grad_a, st));
    }
    (void)pn;
    return TNLM_OK;
}

long long energy_blocks(int nx, int ny, int nz, int np)
{
    return (long long)((nx + kTX - 1) / kTX) * ((ny + kTY - 1) / kTY) * (((nz + kTZ - 1) / kTZ) * np);
}

tnlm_status launch_energy_tnlm(int nx, int ny, int nz, int np, const float *a, const float *f, int d, int M, float h,
                               float *lam, float *t1, float *grad, double *jpart, long long *nblk, cudaStream_t st)
{
    // the box-sum form for the (d, M) it is compiled for, the direct tiled form otherwise
    cudaError_t err = cudaSuccess;
    if (launch_energy_box(d, M, nx, ny, nz, np, a, f, h, lam, t1, grad, jpart, nblk, st, &err)) {
        TNLM_TRY_CUDA(err);
        return TNLM_OK;
    }
    const int ntz = (nz + kTZ - 1) / kTZ;
    dim3 block(kTX, kTY, kTZ), grid((nx + kTX - 1) / kTX, (ny + kTY - 1) / kTY, np * ntz);
    const float c2 = (float)(1.4426950408889634 / (2.0 * (double)h * (double)h));
    const int R = M + d;
    const size_t s1 = sizeof(float) * ((size_t)(kTX + 2 * d) * (kTY + 2 * d) * (kTZ + 2 * d) +
                                       (size_t)(kTX + 2 * R) * (kTY + 2 * R) * (kTZ + 2 * R));
    const size_t s2 = s1 + sizeof(float) * 2 * (kTX + 2 * M) * (kTY + 2 * M) * (kTZ + 2 * M);
    if (s1 > 48 * 1024) TNLM_TRY_CUDA(cudaFuncSetAttribute(k_lognorm, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)s1));
    if (s2 > 48 * 1024)
        TNLM_TRY_CUDA(cudaFuncSetAttribute(k_energy_grad, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)s2));
    k_lognorm<<<grid, block, s1, st>>>(nx, ny, nz, np, ntz, a, d, M, c2, lam);
    TNLM_TRY_CUDA(cudaGetLastError());
    k_energy_grad<<<grid, block, s2, st>>>(nx, ny, nz, np, ntz, a, f, lam, d, M, c2, grad, jpart);
    TNLM_TRY_CUDA(cudaGetLastError());
    *nblk = energy_blocks(nx, ny, nz, np);
    return TNLM_OK;
}

}  // namespace tnlm
