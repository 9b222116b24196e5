// FDK (Feldkamp, Davis and Kress, the paper's ref. 16): the initial value of
// TNLM-R and the input of TNLM-E (Sec. 2.2-2.3).  Each phase is reconstructed
// from its own views, assumed to cover a full rotation evenly:
//   k_fdk_filter : cosine weight SDD / sqrt(SDD^2 + u^2 + v^2), then the
//                  discrete ramp (Ram-Lak) filter along each detector row,
//                  F(u_n) = du sum_k h[n-k] R'(u_k), h[0] = 1/(4 du^2),
//                  h[odd m] = -1/(m^2 pi^2 du^2), h[even] = 0;
//   k_fdk_bp     : voxel-driven backprojection, bilinear in (u, v), weight
//                  (d_theta / 2) SAD SDD / U^2, U = SAD - (x cos t + y sin t).
#include <cfloat>
#include <cmath>

#include "tnlm_internal.cuh"

namespace tnlm {
namespace {

// The ramp's even taps vanish apart from h[0], so the outputs of one parity are a dense convolution of the samples of
// the other:  F(u_{2j+p}) = du (h[0] R'_{2j+p} + sum_k h[2(j - k) + 2p - 1] R'_{2k+1-p}).
// A block takes 64 detector rows and 256 outputs of one parity: per sample k a thread multiplies 8 rows (one 32-byte
// broadcast) by 8 consecutive outputs' taps, which slide through registers (two 16-byte loads per four samples).  138 k
// rows of 512: 5.7 -> 1.33 ms against one output per thread with three shared loads to two taps, 36 % of the FMA peak by
// operations; the chunks' loads and barriers are not overlapped with the products.  Short rows and few rows take a tile of
// 16 x 64 (filter_small), which sums every output in the same order, to the same bits.
// The ramp nearly cancels on smooth rows (h[0] against the taps next to it), so the order of the sum decides its
// rounding: the taps beyond kNear, whose sum is small, go through the tiles, and the near ones are summed outward from
// h[0] on their own and added last.
constexpr int kFiltThreads = 256, kFiltK = 64;  // samples per chunk
constexpr int kNear = 15;                       // odd
// RT rows x OT outputs of one parity per thread; a block's 8 warps lie along the rows, their lanes along the outputs
template <int RT, int OT>
struct FiltTile {
    static constexpr int Rows = 8 * RT, Out = 32 * OT, Pitch = Rows + 4;
    static constexpr int Strip = 2 * Out + 2 * kNear + 2;  // samples around a block's outputs in one row
};

// N consecutive floats of shared memory, 4 N (N < 4) or 16 bytes at a time
template <int N>
__device__ __forceinline__ void load_floats(const float *p, float *out)
{
    if constexpr (N == 2) {
        const float2 t = *reinterpret_cast<const float2 *>(p);
        out[0] = t.x, out[1] = t.y;
    } else {
#pragma unroll
        for (int i = 0; i < N; i += 4) {
            const float4 t = *reinterpret_cast<const float4 *>(p + i);
            out[i] = t.x, out[i + 1] = t.y, out[i + 2] = t.z, out[i + 3] = t.w;
        }
    }
}

// The far taps of output n of one row, in the tiles' order, where the tiles' sum is not finite: their zeros for the near
// taps make NaN of an infinite sample (0 * inf) that only the near sum holds.  q: SDD^2 + v^2 of the row.
__device__ __noinline__ float far_taps(const KGeom &G, const float *__restrict__ row, float q, float hs, int n)
{
    float sum = 0.f;
    for (int i = (n + 1) & 1; i < G.nu; i += 2) {
        const float u = ((float)i - G.uc) * G.du + G.u_off, m = (float)(n - i);
        if (abs(n - i) > kNear) sum = fmaf(__ldg(row + i) * G.sdd * rsqrtf(q + u * u), hs / (m * m), sum);
    }
    return sum;
}

template <int RT, int OT>
__global__ void __launch_bounds__(kFiltThreads, RT == 8 ? 2 : 4)
    k_fdk_filter(KGeom G, long long rows, const float *__restrict__ proj, float *__restrict__ filt)
{
    using C = FiltTile<RT, OT>;
    constexpr int V = OT < 4 ? OT : 4;              // taps of one load
    constexpr int kWork = 8 * (C::Out + C::Strip);  // the last step's strips, per warp
    __shared__ __align__(16) float s_x[kFiltK * C::Pitch > kWork ? kFiltK * C::Pitch : kWork];  // [sample][row]
    __shared__ float s_q[C::Rows];  // SDD^2 + v^2
    __shared__ __align__(16) float s_h[C::Out + kFiltK];    // taps of the chunk: s_h[i] = tap of j - k = j0 - k0 - K + i
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int p = blockIdx.y & 1, j0 = (blockIdx.y >> 1) * C::Out;
    const long long row0 = (long long)blockIdx.x * C::Rows;
    const float hs = -1.0f / (float)(M_PI * M_PI) * G.inv_du * G.inv_du;
    if (tid < C::Rows) {
        const float v = ((float)((unsigned)(row0 + tid) % (unsigned)G.nv) - G.vc) * G.dv + G.v_off;
        s_q[tid] = G.sdd * G.sdd + v * v;
    }
    __syncthreads();
    const float *__restrict__ pr = proj + row0 * G.nu;
    auto weighted = [&](int r, int i) {  // R' at sample i of the block's row r
        const float u = ((float)i - G.uc) * G.du + G.u_off;
        return __ldg(pr + (long long)r * G.nu + i) * G.sdd * rsqrtf(s_q[r] + u * u);
    };
    // near taps; the big tile has no registers to keep them
    constexpr int kTaps = RT == 8 ? 1 : (kNear + 1) / 2;
    float hn[kTaps];
#pragma unroll
    for (int i = 0; i < kTaps; ++i) hn[i] = hs / (float)((2 * i + 1) * (2 * i + 1));
    float acc[RT][OT];  // [row][output]
#pragma unroll
    for (int r = 0; r < RT; ++r)
#pragma unroll
        for (int o = 0; o < OT; ++o) acc[r][o] = 0.f;
    const int nk = (G.nu + p) / 2;  // samples of the other parity, 2k + 1 - p < nu
    for (int k0 = 0; k0 < nk; k0 += kFiltK) {
        // of this chunk; the big tile takes it whole (a bound that is not constant costs it 5 %)
        const int kend = RT == 8 ? kFiltK : min(kFiltK, (nk - k0 + 15) & ~15);
        __syncthreads();
        for (int t = tid; t < C::Rows * kFiltK; t += kFiltThreads) {
            const int k = k0 + t % kFiltK, r = t / kFiltK;
            if (t % kFiltK < kend)
                s_x[(t % kFiltK) * C::Pitch + r] = (k < nk && row0 + r < rows) ? weighted(r, 2 * k + 1 - p) : 0.f;
        }
        for (int t = tid; t < C::Out + kFiltK; t += kFiltThreads) {
            const float m = (float)(2 * (j0 - k0 - kFiltK + t) + 2 * p - 1);  // odd
            s_h[t] = fabsf(m) <= (float)kNear ? 0.f : hs / (m * m);
        }
        __syncthreads();
        // output o of the thread at sample k (in the chunk): tap index OT lane + o + K - k
        const float *hp = s_h + OT * lane;
        float h[OT + 4];
        load_floats<OT>(hp + kFiltK, h + 4);
        for (int kb = 0; kb < kend; kb += 16)
#pragma unroll
            for (int k = kb; k < kb + 16; k += 4) {  // h[4 + i] = tap index OT lane + K - k + i
#pragma unroll
                for (int i = 0; i < 4; i += V) load_floats<V>(hp + kFiltK - k - 4 + i, h + i);
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    float x[RT];
                    load_floats<RT>(s_x + (k + q) * C::Pitch + RT * warp, x);
#pragma unroll
                    for (int r = 0; r < RT; ++r)
#pragma unroll
                        for (int o = 0; o < OT; ++o) acc[r][o] = fmaf(x[r], h[4 + o - q], acc[r][o]);
                }
#pragma unroll
                for (int i = OT + 3; i >= 4; --i) h[i] = h[i - 4];
            }
    }
    // a row at a time through shared memory: the near taps from the row's samples around the block's outputs, and
    // stores of neighbouring outputs by neighbouring lanes
    __syncthreads();
    const float h0 = 0.25f * G.inv_du * G.inv_du;
    float *s_o = s_x + warp * (C::Out + C::Strip), *s_r = s_o + C::Out;
    const int first = 2 * j0 + p - kNear;  // sample of s_r[0]
#pragma unroll
    for (int r = 0; r < RT; ++r) {
        __syncwarp();
        if constexpr (OT == 2) {
            *reinterpret_cast<float2 *>(s_o + OT * lane) = make_float2(acc[r][0], acc[r][1]);
        } else {
#pragma unroll
            for (int o = 0; o < OT; o += 4)
                *reinterpret_cast<float4 *>(s_o + OT * lane + o) = make_float4(acc[r][o], acc[r][o + 1], acc[r][o + 2], acc[r][o + 3]);
        }
        const long long row = row0 + RT * warp + r;
        if (row < rows)
            for (int t = lane; t < C::Strip; t += 32)
                s_r[t] = (first + t >= 0 && first + t < G.nu) ? weighted(RT * warp + r, first + t) : 0.f;
        __syncwarp();
        if (row >= rows) continue;
        for (int o = lane; o < C::Out; o += 32) {
            const int n = 2 * (j0 + o) + p;
            const float *c = s_r + 2 * o + kNear;
            float near = h0 * c[0];
#pragma unroll
            for (int m = 1; m <= kNear; m += 2) near = fmaf(RT == 8 ? hs / (float)(m * m) : hn[m / 2 % kTaps], c[-m] + c[m], near);
            float far = s_o[o];
            if (!(fabsf(far) <= FLT_MAX)) far = far_taps(G, proj + row * G.nu, s_q[RT * warp + r], hs, n);
            if (n < G.nu) filt[row * G.nu + n] = G.du * (near + far);
        }
    }
}

// Voxel-driven: a thread owns CH voxels of one (x, y) column, so a view's u, its interpolation weights and its
// distance weight (which do not depend on z) serve all of them; a warp covers 8 x 4 columns, whose pixels lie close
// together whatever the view angle.  Per voxel and view the four gathers remain (10 x 256x256x64, 360 views: 4.4 ->
// 1.49 ms against a thread per voxel and warps of 32 x 1).  A view of 8 voxels is a chain of gathers behind branches, so
// small volumes take one voxel per thread (bp_small).
template <int CH>
__global__ void __launch_bounds__(128) k_fdk_bp(KGeom G, const ViewGeom *__restrict__ views,
                                                const int *__restrict__ view_off, const float *__restrict__ filt,
                                                float *__restrict__ vol, int nchunks)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int ix = (blockIdx.x * 2 + (warp & 1)) * 8 + (lane & 7), iy = (blockIdx.y * 2 + (warp >> 1)) * 4 + (lane >> 3);
    const int iz0 = (blockIdx.z % nchunks) * CH, phase = blockIdx.z / nchunks;
    if (ix >= G.nx || iy >= G.ny) return;
    const float x = G.b0x + ((float)ix + 0.5f) * G.dx;
    const float y = G.b0y + ((float)iy + 0.5f) * G.dy;
    const int v0 = view_off[phase], v1 = view_off[phase + 1];
    const float wscale = 0.5f * (float)(2.0 * M_PI) / (float)(v1 - v0) * G.sad * G.sdd;
    float acc[CH];
#pragma unroll
    for (int k = 0; k < CH; ++k) acc[k] = 0.f;
    for (int vg = v0; vg < v1; ++vg) {
        const float c = views[vg].c, s = views[vg].s;
        const float U = G.sad - (x * c + y * s);
        const float iU = 1.0f / U;
        const float u = G.sdd * (-x * s + y * c) * iU;
        const float fu = (u - G.u_off) * G.inv_du + G.uc;
        const float fu0 = floorf(fu);
        if (!(fu > -1.f && fu < (float)G.nu)) continue;  // both columns off the detector
        const int iu0 = (int)fu0;
        const float au = fu - fu0, wv = wscale * iU * iU;
        // a column off the detector reads its neighbour, at half that one's weight each (with weight 0 an infinite
        // neighbour would make NaN; a select per gather took the call at 10 x 256x256x64 from 2.89 to 3.80 ms)
        const bool in_a = iu0 >= 0, in_b = iu0 + 1 < G.nu;
        const float wa = in_a ? (in_b ? 1.f : 0.5f) * (1.f - au) : 0.5f * au;
        const float wb = in_a && in_b ? au : wa;
        const int ca = max(iu0, 0), cb = min(iu0 + 1, G.nu - 1);
        const float *__restrict__ F = filt + (long long)vg * G.npix;
        const float *__restrict__ Fa = F + ca, *__restrict__ Fb = F + cb;
#pragma unroll
        for (int k = 0; k < CH; ++k) {
            const float z = G.b0z + ((float)(iz0 + k) + 0.5f) * G.dz;
            const float v = G.sdd * z * iU;
            const float fv = (v - G.v_off) * G.inv_dv + G.vc;
            const float fv0 = floorf(fminf(fmaxf(fv, -2.f), (float)G.nv));
            const int iv0 = (int)fv0;
            const float av = fv - fv0;
            float val = 0.f;
            if (iv0 >= 0 && iv0 < G.nv) {
                const int o = iv0 * G.nu;
                val = (1.f - av) * fmaf(wa, __ldg(Fa + o), wb * __ldg(Fb + o));
            }
            if (iv0 + 1 >= 0 && iv0 + 1 < G.nv) {
                const int o = (iv0 + 1) * G.nu;
                val = fmaf(av, fmaf(wa, __ldg(Fa + o), wb * __ldg(Fb + o)), val);
            }
            acc[k] = fmaf(wv, val, acc[k]);
        }
    }
    const long long base = (long long)phase * G.nvox + ((long long)iz0 * G.ny + iy) * G.nx + ix;
#pragma unroll
    for (int k = 0; k < CH; ++k)
        if (iz0 + k < G.nz) vol[base + (long long)k * G.nx * G.ny] = acc[k];
}

}  // namespace

template <int RT, int OT>
static void launch_filter(const KGeom &kg, long long rows, const float *proj, float *filt, cudaStream_t st)
{
    using C = FiltTile<RT, OT>;
    const int halves = ((kg.nu + 1) / 2 + C::Out - 1) / C::Out;  // tiles of the outputs of one parity
    k_fdk_filter<RT, OT><<<dim3((unsigned)((rows + C::Rows - 1) / C::Rows), 2 * halves), kFiltThreads, 0, st>>>(kg, rows, proj,
                                                                                                                filt);
}

template <int CH>
static void launch_bp(const KGeom &kg, const ViewGeom *views, const int *view_off, const float *filt, float *vol,
                      cudaStream_t st)
{
    const int nchunks = (kg.nz + CH - 1) / CH;
    k_fdk_bp<CH><<<dim3((kg.nx + 15) / 16, (kg.ny + 7) / 8, nchunks * kg.np), 128, 0, st>>>(kg, views, view_off, filt, vol,
                                                                                         nchunks);
}

// One voxel per thread where runs of 8 are too few threads, or mostly padding.  8 / 1 voxels per thread, 30 views a phase:
// 4 x 32^3 112 / 24 us, 96x96x48 80 / 48, 4 x 48^3 101 / 50, 96^3 82 / 87, 4 x 64^3 94 / 102, 10 x 64^3 165 / 245;
// 4 x 512x512x1 225 / 72, 4 x 256x256x3 114 / 76, 4 x 256x256x5 116 / 122.
static bool bp_small(const KGeom &kg) { return kg.np * kg.nvox < 900000 || kg.nz < 4; }

// The small tile where its estimated time is the shorter: 1e7 products a microsecond, against 16.5 us for each chunk of 64
// samples and wave of big tiles (two on each of the 152 SMs).  Big / small, us: 120 k rows of 64 410 / 144, of 256 688 / 560,
// of 384 919 / 1141; 11520 of 512 172 / 147, 40 k of 512 415 / 572; 1024 of 1024 100 / 59, 3840 of 1024 140 / 167.
static bool filter_small(int nu, long long rows)
{
    const double small = 0.5 * rows * nu * nu / 1e7;
    const double big = 16.5 * ceil(nu / 128.0) * ceil((rows + 63) / 64 * 2 * ((nu + 511) / 512) / 304.0);
    return small < big;
}

tnlm_status launch_fdk(const KGeom &kg, const ViewGeom *views, const int *view_off, int n_views_total,
                       const float *proj, float *filt, float *vol, cudaStream_t st)
{
    const long long rows = (long long)n_views_total * kg.nv;
    if (filter_small(kg.nu, rows))
        launch_filter<2, 2>(kg, rows, proj, filt, st);
    else
        launch_filter<8, 8>(kg, rows, proj, filt, st);
    TNLM_TRY_CUDA(cudaGetLastError());
    if (bp_small(kg))
        launch_bp<1>(kg, views, view_off, filt, vol, st);
    else
        launch_bp<8>(kg, views, view_off, filt, vol, st);
    TNLM_TRY_CUDA(cudaGetLastError());
    return TNLM_OK;
}

}  // namespace tnlm
