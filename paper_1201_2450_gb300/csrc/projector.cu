// Cone-beam projector of the (P1) data-fidelity step (Eq. 1, Eq. 5): the
// exact radiological path of each detector pixel's ray (Siddon model, the
// paper's ref. 40 as used in Sec. 2.5), one thread per pixel, optionally
// fused with the residual r = P f - y and FP64 block partials of ||r||^2.
// Two walkers compute it: k_forward finds all of a ray's crossings itself,
// k_forward_tab reads the xy crossings its detector column shares from
// tables built once per geometry.  The transpose is in transpose.cu.
//
// The ray parameter is measured in units of the source->pixel vector D
// (chord = delta_parameter * |D|) and anchored at the isocentre plane so
// that FP32 positions keep ~1e-5 voxel resolution.
#include <type_traits>

#include "ray_common.cuh"

namespace tnlm {
namespace {

constexpr int kFwdBX = 32;                       // projector block: 32 u x BY v pixels (BY in {2, 4, 8})

template <int MODE, int BY, class T>
__global__ void __launch_bounds__(kFwdBX *BY)
    k_forward(KGeom G, const ViewGeom *__restrict__ views, const T *__restrict__ vol,
              const T *__restrict__ y, float *__restrict__ out, double *__restrict__ partials)
{
    __shared__ double ws[BY];
    const int iu = blockIdx.x * kFwdBX + threadIdx.x;
    const int iv = blockIdx.y * BY + threadIdx.y;
    const int vg = blockIdx.z;
    const ViewGeom V = views[vg];
    double r2 = 0.0;
    if (iu < G.nu && iv < G.nv) {
        const float u = ((float)iu - G.uc) * G.du + G.u_off;
        const float v = ((float)iv - G.vc) * G.dv + G.v_off;
        // source->pixel vector (mm): the view-frame vector (-SDD, u, v) rotated by the view angle
        const float Dx = -G.sdd * V.c - u * V.s;
        const float Dy = -G.sdd * V.s + u * V.c;
        const float Dz = v;
        const float len = sqrtf(Dx * Dx + Dy * Dy + Dz * Dz);
        // anchor Q: the ray's point in the isocentre plane (parameter alpha0 = SAD/SDD)
        const float au = G.alpha0 * u;
        const float Ex = (-au * V.s - G.b0x) * G.inv_dx;
        const float Ey = (au * V.c - G.b0y) * G.inv_dy;
        const float Ez = (G.alpha0 * v - G.b0z) * G.inv_dz;
        const float Gx = Dx * G.inv_dx, Gy = Dy * G.inv_dy, Gz = Dz * G.inv_dz;
        // beta = alpha - alpha0 spans the segment source (alpha 0) .. pixel (alpha 1)
        float blo = -G.alpha0, bhi = 1.f - G.alpha0;
        bool ok = true;
        slab_grid(Ex, Gx, G.nx, blo, bhi, ok);
        slab_grid(Ey, Gy, G.ny, blo, bhi, ok);
        slab_grid(Ez, Gz, G.nz, blo, bhi, ok);
        float acc = 0.f;
        if (ok && blo < bhi) {
            // Axis roles: a = the dominant of x, y (z if steeper than both), b = the other in-plane
            // axis, c = the remaining one (z for every ray of a practical cone).  A slab between two
            // a-planes holds at most one b crossing (|Gb| <= |Ga|), taken without branching; c
            // crossings depend only on the detector row, so the lanes of a warp (one row, adjacent
            // columns) cross c planes together and the branch for them stays coherent.
            const float ax = fabsf(Gx), ay = fabsf(Gy), az = fabsf(Gz);
            const bool zdom = az > ax && az > ay;
            const bool xa = !zdom && ax >= ay;  // x dominant: (a,b,c) = (x,y,z); y dominant: (y,x,z)
            const int sxy = G.nx * G.ny;
            const float Ea = zdom ? Ez : (xa ? Ex : Ey), Eb = xa ? Ey : Ex, Ec = zdom ? Ey : Ez;
            const float Ga = zdom ? Gz : (xa ? Gx : Gy), Gb = xa ? Gy : Gx, Gc = zdom ? Gy : Gz;
            const int na = zdom ? G.nz : (xa ? G.nx : G.ny), nb = xa ? G.ny : G.nx, nc = zdom ? G.ny : G.nz;
            const int ta = zdom ? sxy : (xa ? 1 : G.nx), tb = xa ? G.nx : 1, tc = zdom ? G.nx : sxy;
            const int sa = Ga > 0.f ? 1 : -1, sb = Gb > 0.f ? 1 : -1, sc = Gc > 0.f ? 1 : -1;
            const int pa = Ga > 0.f, pb = Gb > 0.f, pc = Gc > 0.f;
            const float iva = 1.0f / Ga;
            const float ivb = Gb != 0.f ? 1.0f / Gb : 0.f;
            const float ivc = Gc != 0.f ? 1.0f / Gc : 0.f;
            int ia = clamp_floor(fmaf(blo, Ga, Ea), na);
            int ib = clamp_floor(fmaf(blo, Gb, Eb), nb);
            int ic = clamp_floor(fmaf(blo, Gc, Ec), nc);
            // next plane crossing on each axis, one FMA per step: beta = f * iv - E * iv, with the
            // plane coordinates f kept as exact float shadows of the integer indices (small
            // integers), so no conversion and no drift per step.  An exit plane may then differ
            // from bhi by an ulp: slabs are counted separately, and a crossing an ulp past the
            // exit only steps to an index whose load is guarded.
            float fa = (float)(ia + pa), fb = (float)(ib + pb), fc = (float)(ic + pc);
            const float saf = (float)sa, sbf = (float)sb, scf = (float)sc;
            const float oa = -Ea * iva, ob = -Eb * ivb, oc = -Ec * ivc;
            float ba = fmaf(fa, iva, oa);
            float bb = Gb != 0.f ? fmaf(fb, ivb, ob) : FLT_MAX;
            float bc = Gc != 0.f ? fmaf(fc, ivc, oc) : FLT_MAX;
            // a-slabs visited: from the entry cell to the cell holding the exit point (a slab of zero
            // length at either end is harmless; every index stays inside the volume)
            const int ia_last = clamp_floor(fmaf(bhi, Ga, Ea), na);
            const int n_slabs = max(1, sa > 0 ? ia_last - ia + 1 : ia - ia_last + 1);
            const T *__restrict__ fp = vol + (long long)V.phase * G.nvox;
            int idx = ia * ta + ib * tb + ic * tc;
            float fcur = ldg_v(fp + idx);
            float bcur = blo;
            // one a-slab: its c and b crossings; true when the ray left the volume through c
            auto slab = [&]() -> bool {
                const float bend = fminf(ba, bhi);  // end of this a-slab inside the volume
                if (bc < bend) {                    // c crossings (coherent across the warp, rare)
                    for (int rc = 0; rc < 4 && bc < bend; ++rc) {
                        if (bb < bc) {
                            acc = fmaf(fcur, bb - bcur, acc);
                            bcur = bb;
                            ib += sb;
                            idx += sb * tb;
                            fcur = (unsigned)ib < (unsigned)nb ? ldg_v(fp + idx) : 0.f;
                            fb += sbf;
                            bb = fmaf(fb, ivb, ob);
                        }
                        acc = fmaf(fcur, bc - bcur, acc);
                        bcur = bc;
                        ic += sc;
                        if ((unsigned)ic >= (unsigned)nc || (unsigned)ib >= (unsigned)nb) return true;
                        idx += sc * tc;
                        fcur = ldg_v(fp + idx);
                        fc += scf;
                        bc = fmaf(fc, ivc, oc);
                    }
                }
                // at most one b crossing in the rest of the slab
                const bool hit = bb < bend;
                const float e1 = hit ? bb : bend;
                acc = fmaf(fcur, e1 - bcur, acc);
                if (hit) {
                    ib += sb;
                    idx += sb * tb;
                    fcur = (unsigned)ib < (unsigned)nb ? ldg_v(fp + idx) : 0.f;
                    fb += sbf;
                    bb = fmaf(fb, ivb, ob);
                }
                acc = fmaf(fcur, bend - e1, acc);
                bcur = bend;
                return false;
            };
            // every slab but the last ends on an a-plane: step into the next one unconditionally
            bool left = false;
#pragma unroll 2
            for (int k = 1; k < n_slabs; ++k) {
                if (slab()) {
                    left = true;
                    break;
                }
                idx += sa * ta;
                fcur = (unsigned)ib < (unsigned)nb ? ldg_v(fp + idx) : 0.f;
                fa += saf;
                ba = fmaf(fa, iva, oa);
            }
            if (!left) slab();
            acc *= len;
        }
        const long long o = ((long long)vg * G.nv + iv) * G.nu + iu;
        if (MODE == 0) {
            out[o] = acc;
        } else {
            const float r = acc - ldg_v(y + o);
            out[o] = r * len;  // scaled residual consumed by the transpose
            r2 = (double)r * (double)r;
        }
    }
    if (MODE == 1) {
        const double s = block_sum_warps<BY>(r2, ws);
        if (threadIdx.x == 0 && threadIdx.y == 0)
            partials[((long long)blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x] = s;
    }
}

// ---------------------------------------------------------------------------
// The table walker.  The rays of one detector column lie in one vertical
// plane (their x and y coordinates along the ray parameter do not depend on
// the detector row), so every row of the column crosses the same xy cells at
// the same ray parameters.  k_coltab lays out that sequence once per
// geometry handle -- entry k of (view, column): the ray parameter where the
// ray leaves its k-th xy cell, and the offset of that cell in a copy of the
// volume that each projection writes first.  Two walks, one of them per
// handle (walk_by_columns):
//   k_forward_tab walks the rows of a column through its entries together: a
//   warp is 32 adjacent rows of one column, so an entry is one value for the
//   whole warp and the rows' voxels are neighbours in z.  Its copy is stored
//   z-fastest (k_zfirst): 32 rows span a few voxels of one z run, one or two
//   sectors per gather where a row of 32 columns touched three cache lines.
//   k_forward_cols walks 32 adjacent columns of one row, each lane through its
//   own column's entries (tables interleaved by column), with the row's z
//   crossings in place.  Its copy holds the z slices in 4 x 8 (x, y) bricks of
//   32 voxels (k_brick).  It costs more per voxel, but nothing for rows that
//   miss the volume or do not exist, and less per z plane.
// ---------------------------------------------------------------------------

constexpr int kColtabHead = 4;  // float2 before a column's entries: what the walk needs of the column, and its start
constexpr int kColtabPad = 1;   // room after the last entry, so that entries can be read in pairs
constexpr int kColtabAhead = 16;  // room after the last column: the walk reads up to two batches of entries ahead

// Column iu of view vg: kmax consecutive float2 (kmax even: pairs are 16-byte aligned).  The head is
//   [0] (ga, ha), [1] (gb, hb): planes of the two in-plane axes crossed before beta: floor(beta ga + ha), ...
//   [2] (entries, as bits; their end), [3] (their start, unused)
// and entry k stands at [kColtabHead + k].
__host__ __device__ __forceinline__ long long coltab_base(int vg, int iu, int kmax, int nu)
{
    return ((long long)vg * nu + iu) * kmax;
}

// The column walk's tables: entries in pairs, pair j of column iu of view vg holds entries 2j, 2j+1 as one float4 at
// float4 index (vg * kmax / 2 + j) * nu + iu (kmax even), so a warp's lanes read adjacent pairs.  No head.
constexpr int kPairPad = 3;  // exit entry repeated after the last so reads ahead need no test

__host__ __device__ __forceinline__ long long pair_slot(int vg, int e, int iu, int kmax, int nu)
{
    return (((long long)vg * (kmax >> 1) + (e >> 1)) * nu + iu) * 2 + (e & 1);
}

// The in-plane part of the ray of detector column iu of view V (the same
// expressions as k_forward).
struct ColumnRay {
    float Dx, Dy, Ex, Ey, Gx, Gy, blo, bhi;
    bool ok;
    // a = the dominant in-plane axis (at most one b crossing per a-slab), b = the other
    bool xa;
    float Ea, Eb, Ga, Gb, iva, ivb, oa, ob, fa0, fb0, saf, sbf;
    int na, nb, sa, sb, ia0, ib0, ia1, ib1, n_a, n_b;

    __device__ __forceinline__ void init(const KGeom &G, const ViewGeom &V, int iu)
    {
        const float u = ((float)iu - G.uc) * G.du + G.u_off;
        Dx = -G.sdd * V.c - u * V.s;
        Dy = -G.sdd * V.s + u * V.c;
        const float au = G.alpha0 * u;
        Ex = (-au * V.s - G.b0x) * G.inv_dx;
        Ey = (au * V.c - G.b0y) * G.inv_dy;
        Gx = Dx * G.inv_dx;
        Gy = Dy * G.inv_dy;
        blo = -G.alpha0;
        bhi = 1.f - G.alpha0;
        ok = true;
        slab_grid(Ex, Gx, G.nx, blo, bhi, ok);
        slab_grid(Ey, Gy, G.ny, blo, bhi, ok);
        ok = ok && blo < bhi;
        n_a = n_b = 0;
        if (!ok) return;
        xa = fabsf(Gx) >= fabsf(Gy);
        Ea = xa ? Ex : Ey;
        Eb = xa ? Ey : Ex;
        Ga = xa ? Gx : Gy;
        Gb = xa ? Gy : Gx;
        na = xa ? G.nx : G.ny;
        nb = xa ? G.ny : G.nx;
        sa = Ga > 0.f ? 1 : -1;
        sb = Gb > 0.f ? 1 : -1;
        iva = 1.0f / Ga;
        ivb = Gb != 0.f ? 1.0f / Gb : 0.f;
        oa = -Ea * iva;
        ob = -Eb * ivb;
        ia0 = clamp_floor(fmaf(blo, Ga, Ea), na);
        ib0 = clamp_floor(fmaf(blo, Gb, Eb), nb);
        ia1 = clamp_floor(fmaf(bhi, Ga, Ea), na);
        ib1 = clamp_floor(fmaf(bhi, Gb, Eb), nb);
        // interior planes crossed between the entry and exit cells, in walking order:
        // a-plane m at fmaf(fa0 + sa m, iva, oa), b-plane k at fmaf(fb0 + sb k, ivb, ob)
        n_a = abs(ia1 - ia0);
        n_b = Gb != 0.f ? abs(ib1 - ib0) : 0;
        fa0 = (float)(ia0 + (Ga > 0.f));
        fb0 = (float)(ib0 + (Gb > 0.f));
        saf = (float)sa;
        sbf = (float)sb;
    }
    __device__ __forceinline__ float beta_a(int m) const { return fmaf(fmaf((float)m, saf, fa0), iva, oa); }
    __device__ __forceinline__ float beta_b(int k) const { return fmaf(fmaf((float)k, sbf, fb0), ivb, ob); }
    // offset of cell (a, b)'s z run in a phase of the z-fastest volume
    __device__ __forceinline__ int cell(const KGeom &G, int ia, int ib) const
    {
        return ((xa ? ib : ia) * G.nx + (xa ? ia : ib)) * G.nz;
    }
    // offset of cell (a, b) in a bricked z slice
    __device__ __forceinline__ int brick_cell(const KGeom &G, int ia, int ib) const
    {
        const int x = xa ? ia : ib, y = xa ? ib : ia;
        return (((y >> 3) * ((G.nx + 3) >> 2) + (x >> 2)) << 5) + ((y & 7) << 2) + (x & 3);
    }
    // entries of the column: one per interior plane crossed, and the exit
    __device__ __forceinline__ int entries() const { return ok ? n_a + n_b + 1 : 0; }
};

// Entries of every (view, column): thread t of (view vg, column iu) places the
// t-th plane crossing (a-planes first, then b-planes) at its rank in the merged
// order, found by binary search over the other axis (ties: the a-plane first);
// the thread with t == n_a + n_b writes the exit, thread 0 the head.
// kmax = kColtabHead + nx + ny - 1 + kColtabPad rounded up to an even count, or nx + ny - 1 + kPairPad (COLS: the
// column walk's tables).
template <bool COLS>
__global__ void __launch_bounds__(128) k_coltab(KGeom G, const ViewGeom *__restrict__ views, float2 *__restrict__ tab,
                                                int kmax)
{
    const int iu = blockIdx.y, vg = blockIdx.z;
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    ColumnRay R;
    R.init(G, views[vg], iu);
    float2 *col = tab + coltab_base(vg, iu, kmax, G.nu);
    if (!COLS && t == 0) {
        col[0] = make_float2(R.ok ? fabsf(R.Ga) : 0.f, R.ok ? (R.sa > 0 ? R.Ea - (float)R.ia0 : (float)(R.ia0 + 1) - R.Ea) : 0.f);
        col[1] = make_float2(R.ok ? fabsf(R.Gb) : 0.f, R.ok ? (R.sb > 0 ? R.Eb - (float)R.ib0 : (float)(R.ib0 + 1) - R.Eb) : 0.f);
        col[2] = make_float2(__int_as_float(R.entries()), R.bhi);
        col[3] = make_float2(R.blo, 0.f);
    }
    if (!R.ok || t > R.n_a + R.n_b) return;
    float beta;
    int e, ca, cb;
    if (t == R.n_a + R.n_b) {
        beta = R.bhi;
        e = t;
        ca = R.ia1;
        cb = R.ib1;
    } else if (t < R.n_a) {
        // a-plane m: preceded by the b-planes crossed strictly before it
        const int m = t;
        beta = R.beta_a(m);
        int lo = 0, hi = R.n_b;
        while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if (R.beta_b(mid) < beta) lo = mid + 1;
            else hi = mid;
        }
        e = m + lo;
        ca = R.ia0 + R.sa * m;
        cb = R.ib0 + R.sb * lo;
    } else {
        // b-plane k: preceded by the a-planes crossed at or before it
        const int k = t - R.n_a;
        beta = R.beta_b(k);
        int lo = 0, hi = R.n_a;
        while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if (R.beta_a(mid) <= beta) lo = mid + 1;
            else hi = mid;
        }
        e = k + lo;
        ca = R.ia0 + R.sa * lo;
        cb = R.ib0 + R.sb * k;
    }
    // the cell before this crossing; the crossing clamped to the column's extent
    const float end = fminf(fmaxf(beta, R.blo), R.bhi);
    if (!COLS) {
        col[kColtabHead + e] = make_float2(end, __int_as_float(R.cell(G, ca, cb)));
    } else {
        const float2 ent = make_float2(end, __int_as_float(R.brick_cell(G, ca, cb)));
        tab[pair_slot(vg, e, iu, kmax, G.nu)] = ent;
        if (t == R.n_a + R.n_b)
            for (int q = 1; q <= kPairPad; ++q) tab[pair_slot(vg, e + q, iu, kmax, G.nu)] = ent;
    }
}

constexpr float kCellMagic = 12582912.0f;  // 1.5 * 2^23: one unit per ulp, so z + kCellMagic rounded down holds floor(z)
constexpr int kCellMagicBits = 0x4B400000;

// The entry of a column that holds beta, to rounding (h0: the first two of the column's head)
__device__ __forceinline__ int entry_near(const float4 &h0, int K, float beta)
{
    const int na = __float_as_int(__fadd_rd(fmaf(beta, h0.x, h0.y), kCellMagic));
    const int nb = __float_as_int(__fadd_rd(fmaf(beta, h0.z, h0.w), kCellMagic));
    return min(max((na - kCellMagicBits) + (nb - kCellMagicBits), 0), K - 1);
}

// sum plus the parts that the walk of one row (z = ez + beta gz) took wrongly, one per z plane crossed between the
// column's two ends; two planes at a time, so that their loads overlap.
__device__ __forceinline__ float add_planes(const float4 *__restrict__ head, const float4 &h1,
                                            const float *__restrict__ fp, int nz, float ez, float gz, float sum)
{
    const float2 *__restrict__ tc = reinterpret_cast<const float2 *>(head) + kColtabHead;
    const int K = __float_as_int(h1.x);
    const float blo = h1.z, bhi = h1.y, fnz = (float)nz;
    const float za = fmaf(blo, gz, ez), zb = fmaf(bhi, gz, ez);
    const int ia = (int)floorf(fminf(fmaxf(za, -1.f), fnz)), ib = (int)floorf(fminf(fmaxf(zb, -1.f), fnz));
    const int n = abs(ib - ia);
    if (n == 0) return sum;  // gz != 0 from here
    const float4 h0 = __ldg(head);
    const bool up = gz > 0.f;
    const float iv = 1.0f / gz, ov = -ez * iv, stepf = up ? 1.f : -1.f;
    const float p0 = (float)(up ? ia + 1 : ia);
    for (int q = 0; q < n; q += 2) {
        float pf[2], bp[2], e0[2];
        float2 t[2];
        int k[2];
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            pf[i] = fmaf((float)(q + i), stepf, p0);
            bp[i] = fminf(fmaxf(fmaf(pf[i], iv, ov), blo), bhi);
            k[i] = entry_near(h0, K, bp[i]);
            t[i] = __ldg(tc + k[i]);
            e0[i] = __ldg(tc + k[i] - 1).x;
        }
        float diff[2];  // (voxel before plane p) - (voxel after)
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            auto past = [&](float e) { return (fmaf(e, gz, ez) >= pf[i]) == up; };
            while (k[i] > 0 && past(e0[i])) {
                t[i] = __ldg(tc + --k[i]);
                e0[i] = __ldg(tc + k[i] - 1).x;
            }
            while (k[i] < K - 1 && !past(t[i].x)) {
                e0[i] = t[i].x;
                t[i] = __ldg(tc + ++k[i]);
            }
            const int p = (int)pf[i];
            const float *cp = fp + (__float_as_int(t[i].y) + p);  // the voxel above plane p
            const float above = q + i < n && p < nz ? __ldg(cp) : 0.f, below = q + i < n && p > 0 ? __ldg(cp - 1) : 0.f;
            diff[i] = up ? below - above : above - below;
        }
#pragma unroll
        for (int i = 0; i < 2; ++i)
            sum = q + i < n ? fmaf(diff[i], fminf(fmaxf(bp[i], e0[i]), t[i].x) - e0[i], sum) : sum;
    }
    return sum;
}

// The walk of one row with every entry split at its z planes in turn, for a row whose sum is not finite: the differences
// of add_planes make NaN of an infinite voxel next to a plane (inf - inf).  A voxel that the row has no part in is not
// read.
__device__ __noinline__ float walk_row(const float4 *__restrict__ head, const float4 &h1, const float *__restrict__ fp,
                                       int nz, float ez, float gz)
{
    const float2 *__restrict__ tc = reinterpret_cast<const float2 *>(head) + kColtabHead;
    const int K = __float_as_int(h1.x), step = gz > 0.f ? 1 : -1;
    const float iv = gz != 0.f ? 1.0f / gz : 0.f, ov = -ez * iv, fnz = (float)nz;
    auto cell = [&](float e) { return (int)floorf(fminf(fmaxf(fmaf(e, gz, ez), -1.f), fnz)); };
    float sum = 0.f, cur = h1.z;
    int i = cell(cur);
    for (int k = 0; k < K; ++k) {
        const float2 t = __ldg(tc + k);
        const int last = cell(t.x);
        for (int n = max((last - i) * step, 0); n >= 0; --n, i += step) {  // n planes left in the entry
            const float plane = (float)(i + (step > 0 ? 1 : 0));
            const float end = n > 0 ? fminf(fmaxf(fmaf(plane, iv, ov), cur), t.x) : t.x;
            if (end > cur && i >= 0 && i < nz) sum = fmaf(__ldg(fp + (__float_as_int(t.y) + i)), end - cur, sum);
            cur = end;
        }
        i = last;
    }
    return sum;
}

// A warp walks 32 R rows of one detector column (block: NC adjacent columns), R per lane, 32 apart; R = 0: 2^lr2
// rows, 4 to 16, of as many adjacent columns as fill the warp (NC times as many in the block).
// Along an entry's segment e_{k-1} .. e_k a row stays in one voxel unless it crosses a z plane there, once in ~25
// entries.  The walk takes every entry whole, with the voxel at its end:
//   acc += (e_k - e_{k-1}) f(c_k, floor z(e_k)),   z(beta) = Ez + beta Gz, 0 outside the volume,
// five operations per row and no test where all the warp's rows are inside, and add_planes then adds for every z
// plane p of the row the part that this took wrongly:
//   acc += (beta_p - e_{k-1}) (f(c_k, before p) - f(c_k, after p)),
// k the first entry whose end lies past p, found from the planes crossed at beta_p (they number the entries) and
// settled on the same z(e_k) that the walk used, so the two agree whatever the rounding.  The entry's voxels are
// then split at beta_p exactly, any number of planes in one entry included, and a row that enters or leaves through
// the top or bottom of the volume does so at plane 0 or nz.
// vol: the z-fastest FP32 copy (widened from 16-bit storage by k_zfirst); y: the stored measurements.
// Bound by the L1 (80 % of its data cycles: per entry one for each row's gather, and four for the 16 bytes of two
// entries that every lane receives) with issue at 64 %: 17.1 G crossed voxels of 10 x 256x256x64, 360 views x
// 512x384, in 8.3 ms, where a walk of 32 columns x 1 row that tested each entry for its plane took 10.8; 10 x 128^3,
// 400 x 256x192 2.83 -> 1.47 ms.  Two rows per lane: each entry read serves both (1 row: 1.85 ms on the latter; 4
// rows spill or leave too few warps).  32 warps per SM: the loads of two batches in flight want 64 registers (40
// warps: 9.7 ms).
template <int MODE, int NC, int R, class T>
__global__ void __launch_bounds__(32 * NC, 32 / NC)
    k_forward_tab(KGeom G, int lr2, const ViewGeom *__restrict__ views, const float *__restrict__ vol,
                  const T *__restrict__ y, float *__restrict__ out, double *__restrict__ partials)
{
    constexpr bool FEW = R == 0;
    constexpr int RL = FEW ? 1 : R;
    const int rows = FEW ? 1 << lr2 : 32;
    const int nc2 = (NC == 4 ? 2 : (NC == 8 ? 3 : 4)) + (FEW ? 5 - lr2 : 0), ncols = 1 << nc2;  // columns of the block
    __shared__ float s_acc[32 * RL * (NC + 1)];  // [row][ncols + 1]
    __shared__ double ws[NC];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int row0 = blockIdx.y * rows * RL, vg = blockIdx.z;
    const int lane_row = FEW ? lane & (rows - 1) : lane, col = FEW ? (w << (5 - lr2)) + (lane >> lr2) : w;
    const ViewGeom V = views[vg];
    float acc[RL];
#pragma unroll
    for (int j = 0; j < RL; ++j) acc[j] = 0.f;
    const int iu_w = blockIdx.x * ncols + col;
    const float4 *__restrict__ head = reinterpret_cast<const float4 *>(
        G.coltab + coltab_base(vg, iu_w < G.nu ? iu_w : 0, G.coltab_kmax, G.nu));
    const float4 h0 = __ldg(head), h1 = __ldg(head + 1);
    const int K = iu_w < G.nu ? __float_as_int(h1.x) : 0;
    if (FEW ? __any_sync(0xffffffffu, K > 0) : K > 0) {  // the same for the whole warp
        const float2 *__restrict__ tc = reinterpret_cast<const float2 *>(head) + kColtabHead;  // tc[-1].x: the start
        const float *__restrict__ fp = vol + (long long)V.phase * G.nvox;
        const float fnz = (float)G.nz;
        const float blo = h1.z, bhi = h1.y;
        // where in beta any of the warp's rows is inside the volume (lo, hi), and where all are, by more than rounding
        // could move a voxel (clo, chi)
        float Ez[RL], Gz[RL];
        float lo = FLT_MAX, hi = -FLT_MAX, clo = blo, chi = bhi;
#pragma unroll
        for (int j = 0; j < RL; ++j) {
            const float v = ((float)min(row0 + 32 * j + lane_row, G.nv - 1) - G.vc) * G.dv + G.v_off;
            Ez[j] = (G.alpha0 * v - G.b0z) * G.inv_dz;
            Gz[j] = v * G.inv_dz;
            const float za = fmaf(blo, Gz[j], Ez[j]), zb = fmaf(bhi, Gz[j], Ez[j]);
            // at the top face z is known to half an ulp of nz, more than the 1e-3 beyond 2^14 slices
            const float margin = fmaf(fabsf(Gz[j]), 1e-6f, fmaxf(1e-3f, fnz * 0x1p-22f));
            if (fminf(za, zb) >= margin && fmaxf(za, zb) <= fnz - margin) {
                lo = blo;
                hi = bhi;
            } else if (Gz[j] != 0.f) {
                const float iv = 1.0f / Gz[j], m = margin * fabsf(iv);
                const float t0 = -Ez[j] * iv, t1 = (fnz - Ez[j]) * iv;
                const float jlo = fmaxf(blo, fminf(t0, t1)), jhi = fminf(bhi, fmaxf(t0, t1));
                if (jlo < jhi) {
                    lo = fminf(lo, jlo);
                    hi = fmaxf(hi, jhi);
                }
                clo = fmaxf(clo, fminf(t0, t1) + m);
                chi = fminf(chi, fmaxf(t0, t1) - m);
            } else if (Ez[j] >= 0.f && Ez[j] < fnz) {  // in the plane of a face at most: tested voxel by voxel
                lo = blo;
                hi = bhi;
                chi = -FLT_MAX;
            } else {
                chi = -FLT_MAX;
            }
        }
        int k0 = 0, k1 = K, c0 = 0, c1 = K;  // entries to walk, and of them those that need no test
        if (!__all_sync(0xffffffffu, clo == blo && chi == bhi)) {
            for (int o = rows / 2; o > 0; o >>= 1) {
                lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, o));
                hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, o));
                clo = fmaxf(clo, __shfl_xor_sync(0xffffffffu, clo, o));
                chi = fminf(chi, __shfl_xor_sync(0xffffffffu, chi, o));
            }
            // two entries either side for the rounding of entry_near
            k0 = lo < hi ? max(entry_near(h0, K, lo) - 2, 0) : 0;
            k1 = lo < hi ? min(entry_near(h0, K, hi) + 3, K) : 0;
            c0 = clo > blo ? max(entry_near(h0, K, clo) + 3, k0) : k0;
            c1 = chi < bhi ? min(entry_near(h0, K, chi) - 2, k1) : k1;
            if (!(clo < chi) || c0 >= c1) c0 = c1 = k1;
        }
        if (FEW && K == 0) k0 = k1 = c0 = c1 = 0;
        // entries k .. end - 1 of the rows; CHECKED: a voxel outside the volume counts 0
        auto walk = [&](int k, int end, auto checked_tag) {
            constexpr bool CHECKED = decltype(checked_tag)::value;
            float prev = __ldg(tc + k - 1).x;
            auto voxel = [&](float e, float c, int j) {
                const int cell = __float_as_int(__fadd_rd(fmaf(e, Gz[j], Ez[j]), kCellMagic));
                const float *q = fp + (unsigned)(__float_as_int(c) + cell - kCellMagicBits);
                if (!CHECKED) return __ldg(q);
                return (unsigned)(cell - kCellMagicBits) < (unsigned)G.nz ? __ldg(q) : 0.f;
            };
            auto single = [&](int k) {
                const float2 t = __ldg(tc + k);
#pragma unroll
                for (int j = 0; j < RL; ++j) acc[j] = fmaf(voxel(t.x, t.y, j), t.x - prev, acc[j]);
                prev = t.x;
            };
            if ((k & 1) && k < end) single(k++);
            int nb = (end - k) >> 2;  // batches of 4 entries
            if (nb > 0) {
                // the voxels of a batch are requested one batch, its table entries two batches ahead
                const float4 *__restrict__ tp = reinterpret_cast<const float4 *>(tc + k);
                k += 4 * nb;
                float4 ta = __ldg(tp), tb = __ldg(tp + 1);
                float f[4][RL], seg[4];
                auto request = [&] {
                    const float e[4] = {ta.x, ta.z, tb.x, tb.z}, c[4] = {ta.y, ta.w, tb.y, tb.w};
#pragma unroll
                    for (int i = 0; i < 4; ++i)
#pragma unroll
                        for (int j = 0; j < RL; ++j) f[i][j] = voxel(e[i], c[i], j);
                    seg[0] = e[0] - prev;
                    seg[1] = e[1] - e[0];
                    seg[2] = e[2] - e[1];
                    seg[3] = e[3] - e[2];
                    prev = e[3];
                    tp += 2;
                    ta = __ldg(tp);
                    tb = __ldg(tp + 1);
                };
                request();
#pragma unroll 2
                for (; nb > 1; --nb) {
                    float f0[4][RL], seg0[4];
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        seg0[i] = seg[i];
#pragma unroll
                        for (int j = 0; j < RL; ++j) f0[i][j] = f[i][j];
                    }
                    request();
#pragma unroll
                    for (int i = 0; i < 4; ++i)
#pragma unroll
                        for (int j = 0; j < RL; ++j) acc[j] = fmaf(f0[i][j], seg0[i], acc[j]);
                }
#pragma unroll
                for (int i = 0; i < 4; ++i)
#pragma unroll
                    for (int j = 0; j < RL; ++j) acc[j] = fmaf(f[i][j], seg[i], acc[j]);
            }
            for (; k < end; ++k) single(k);
        };
        if (k0 < c0) walk(k0, c0, std::true_type{});
        if (c0 < c1) walk(c0, c1, std::false_type{});
        if (c1 < k1) walk(c1, k1, std::true_type{});
    }
#pragma unroll
    for (int j = 0; j < RL; ++j) s_acc[(32 * j + lane_row) * (ncols + 1) + col] = acc[j];
    __syncthreads();
    // Thread by (row, column) now, ncols adjacent columns of a row together: the outputs are written so, and a plane is
    // crossed by adjacent columns in neighbouring cells, by adjacent rows far apart (the gathers of the planes touch
    // ~12 cache lines instead of 32).
    double r2 = 0.0;
#pragma unroll
    for (int q = 0; q < RL; ++q) {
        const int t = threadIdx.x + 32 * NC * q;
        const int iv = row0 + (t >> nc2), iu = blockIdx.x * ncols + (t & (ncols - 1));
        if (iv >= G.nv || iu >= G.nu) continue;
        const float u = ((float)iu - G.uc) * G.du + G.u_off;
        const float v = ((float)iv - G.vc) * G.dv + G.v_off;
        float sum = s_acc[(t >> nc2) * (ncols + 1) + (t & (ncols - 1))];
        const float4 *__restrict__ head =
            reinterpret_cast<const float4 *>(G.coltab + coltab_base(vg, iu, G.coltab_kmax, G.nu));
        const float4 h1 = __ldg(head + 1);
        if (__float_as_int(h1.x) > 0) {
            const float *__restrict__ fp = vol + (long long)V.phase * G.nvox;
            const float ez = (G.alpha0 * v - G.b0z) * G.inv_dz, gz = v * G.inv_dz;
            sum = add_planes(head, h1, fp, G.nz, ez, gz, sum);
            if (!(fabsf(sum) <= FLT_MAX)) sum = walk_row(head, h1, fp, G.nz, ez, gz);
        }
        const float Dx = -G.sdd * V.c - u * V.s, Dy = -G.sdd * V.s + u * V.c;
        const float len = sqrtf(Dx * Dx + Dy * Dy + v * v);
        const float pf = sum * len;
        const long long o = ((long long)vg * G.nv + iv) * G.nu + iu;
        if (MODE == 0) {
            out[o] = pf;
        } else {
            const float r = pf - ldg_v(y + o);
            out[o] = r * len;  // scaled residual consumed by the transpose
            r2 += (double)r * (double)r;
        }
    }
    if (MODE == 1) {
        const double s = block_sum_warps<NC>(r2, ws);
        if (threadIdx.x == 0)
            partials[((long long)blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x] = s;
    }
}

// The column walk.  One ray per thread (block: 32 adjacent columns x BY rows of one view), walked
// through its column's table two entries per step, the next two entries in
// flight while the current pair is summed; a z crossing splits an entry's
// segment (the loop takes any number of them, so no geometry condition
// applies).
// Launch bounds: 64 warps per SM (the walk is latency-bound on its voxel gathers, and full occupancy at 32
// registers, with a few bytes spilled, beats 48 warps at 40 registers by 5 %).
// vol: the bricked FP32 copy (widened from 16-bit storage by k_brick); y: the stored measurements.
template <int MODE, int BY, class T>
__global__ void __launch_bounds__(kFwdBX *BY, 64 / BY)
    k_forward_cols(KGeom G, const ViewGeom *__restrict__ views, const float *__restrict__ vol,
                  const T *__restrict__ y, float *__restrict__ out, double *__restrict__ partials)
{
    __shared__ double ws[BY];
    const int iu = blockIdx.x * kFwdBX + threadIdx.x;
    const int iv = blockIdx.y * BY + threadIdx.y;
    const int vg = blockIdx.z;
    double r2 = 0.0;
    if (iu < G.nu && iv < G.nv) {
        const ViewGeom V = views[vg];
        ColumnRay R;
        R.init(G, V, iu);
        const float v = ((float)iv - G.vc) * G.dv + G.v_off;
        const float Dz = v;
        const float len = sqrtf(R.Dx * R.Dx + R.Dy * R.Dy + Dz * Dz);
        const float Ez = (G.alpha0 * v - G.b0z) * G.inv_dz;
        const float Gz = Dz * G.inv_dz;
        float blo = R.blo, bhi = R.bhi;
        bool ok = R.ok;
        slab_grid(Ez, Gz, G.nz, blo, bhi, ok);
        float acc = 0.f;
        if (ok && blo < bhi) {
            const int sc = Gz > 0.f ? 1 : -1;
            const float ivc = Gz != 0.f ? 1.0f / Gz : 0.f, oc = -Ez * ivc, scf = (float)sc;
            const int ic0 = clamp_floor(fmaf(blo, Gz, Ez), G.nz), ic1 = clamp_floor(fmaf(bhi, Gz, Ez), G.nz);
            int nzc = Gz != 0.f ? abs(ic1 - ic0) : 0;  // z planes crossed inside the volume
            float fc = (float)(ic0 + (Gz > 0.f));
            float bc = nzc > 0 ? fmaf(fc, ivc, oc) : FLT_MAX;
            const long long zstep = sc * G.brick_slice;  // vol: the bricked copy
            const float *__restrict__ fp = vol + ((long long)V.phase * G.nz + ic0) * G.brick_slice;
            const long long st = G.nu;  // pair stride in the interleaved tables
            const float2 *__restrict__ tc = G.coltab + pair_slot(vg, 0, iu, G.coltab_kmax, G.nu);
            auto entry_x = [&](int e) { return __ldg(tc + (long long)(e >> 1) * 2 * st + (e & 1)).x; };
            const int K = R.entries();
            // this row's entries: the first that ends after blo .. the first that ends at or after bhi
            // (rows inside the volume's z range enter and leave through its sides: all entries)
            int k0 = 0, k1 = K - 1;
            if (blo > R.blo) {
                int lo = 0, hi = K - 1;
                while (lo < hi) {
                    const int mid = (lo + hi) >> 1;
                    if (entry_x(mid) > blo) hi = mid;
                    else lo = mid + 1;
                }
                k0 = lo;
            }
            if (bhi < R.bhi) {
                int lo = k0, hi = K - 1;
                while (lo < hi) {
                    const int mid = (lo + hi) >> 1;
                    if (entry_x(mid) >= bhi) hi = mid;
                    else lo = mid + 1;
                }
                k1 = lo;
            }
            float bcur = blo;
            // one table entry (end e, cell offset c): its z crossings, then the rest of its segment
            auto segment = [&](float e, float c) {
                float f = ldg_v(fp + __float_as_int(c));
                while (bc < e) {
                    acc = fmaf(f, bc - bcur, acc);
                    bcur = bc;
                    fp += zstep;
                    f = ldg_v(fp + __float_as_int(c));
                    fc += scf;
                    bc = --nzc > 0 ? fmaf(fc, ivc, oc) : FLT_MAX;
                }
                acc = fmaf(f, e - bcur, acc);
                bcur = e;
            };
            // entries before k1 end before bhi (the tables ascend), so only the last entry is clamped to
            // the row's exit
            const float4 *__restrict__ tp = reinterpret_cast<const float4 *>(tc) + (long long)(k0 >> 1) * st;
            float4 t = __ldg(tp);
            int k = k0;
            if ((k & 1) && k < k1) {  // the first entry is the second of its pair
                segment(t.z, t.w);
                ++k;
                tp += st;
                t = __ldg(tp);
            }
            for (; k + 1 < k1; k += 2) {  // pairs of entries strictly before k1, the next pair in flight
                tp += st;
                const float4 n = __ldg(tp);
                float f0 = ldg_v(fp + __float_as_int(t.y));
                float f1 = ldg_v(fp + __float_as_int(t.w));
                float e = t.x;
                if (bc < e) {
                    do {  // z crossings inside entry k's segment
                        acc = fmaf(f0, bc - bcur, acc);
                        bcur = bc;
                        fp += zstep;
                        f0 = ldg_v(fp + __float_as_int(t.y));
                        fc += scf;
                        bc = --nzc > 0 ? fmaf(fc, ivc, oc) : FLT_MAX;
                    } while (bc < e);
                    f1 = ldg_v(fp + __float_as_int(t.w));
                }
                acc = fmaf(f0, e - bcur, acc);
                bcur = e;
                e = t.z;
                while (bc < e) {  // z crossings inside entry k+1's segment
                    acc = fmaf(f1, bc - bcur, acc);
                    bcur = bc;
                    fp += zstep;
                    f1 = ldg_v(fp + __float_as_int(t.w));
                    fc += scf;
                    bc = --nzc > 0 ? fmaf(fc, ivc, oc) : FLT_MAX;
                }
                acc = fmaf(f1, e - bcur, acc);
                bcur = e;
                t = n;
            }
            // the last one or two entries: k1 alone (k odd), or k (even) and then k1 if k < k1
            if (k & 1) {
                segment(fminf(t.z, bhi), t.w);
            } else {
                segment(fminf(t.x, bhi), t.y);
                if (k < k1) segment(fminf(t.z, bhi), t.w);
            }
        }
        const float pf = acc * len;
        const long long o = ((long long)vg * G.nv + iv) * G.nu + iu;
        if (MODE == 0) {
            out[o] = pf;
        } else {
            const float r = pf - ldg_v(y + o);
            out[o] = r * len;  // scaled residual consumed by the transpose
            r2 = (double)r * (double)r;
        }
    }
    if (MODE == 1) {
        const double s = block_sum_warps<BY>(r2, ws);
        if (threadIdx.x == 0 && threadIdx.y == 0)
            partials[((long long)blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x] = s;
    }
}

// The bricked copy of the volume: thread t of z slice (phase, z) takes the
// 4 x 2 voxels x = 4 bx .. 4 bx + 3, y = 2 py, 2 py + 1 and writes them as the
// 8 consecutive elements they occupy in brick (bx, py / 4) (rows 2 py and
// 2 py + 1 of a brick are adjacent), in FP32 whatever the stored type (16-bit
// values are widened once here rather than at every gather of the walk).
// Elements outside the volume are written as 0 and never read.
template <class T>
__global__ void __launch_bounds__(256) k_brick(KGeom G, const T *__restrict__ vol, float *__restrict__ volb)
{
    const int nxb = (G.nx + 3) >> 2, nyh = (G.ny + 1) >> 1;
    const long long per_slice = (long long)nxb * nyh;
    const long long n = per_slice * G.nz * G.np;
    for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < n;
         t += (long long)gridDim.x * blockDim.x) {
        const long long sl = t / per_slice;  // phase * nz + z
        const int r = (int)(t - sl * per_slice);
        const int bx = r % nxb, py = r / nxb;
        const T *src = vol + sl * G.nx * G.ny;
        float v[8];
#pragma unroll
        for (int j = 0; j < 2; ++j)
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int x = 4 * bx + i, y = 2 * py + j;
                v[4 * j + i] = (x < G.nx && y < G.ny) ? ld_v(src + (long long)y * G.nx + x) : 0.f;
            }
        float *dst = volb + sl * G.brick_slice + ((((long long)(py >> 2) * nxb + bx) << 5) + ((py & 3) << 3));
        reinterpret_cast<float4 *>(dst)[0] = make_float4(v[0], v[1], v[2], v[3]);
        reinterpret_cast<float4 *>(dst)[1] = make_float4(v[4], v[5], v[6], v[7]);
    }
}

// The z-fastest copy of the volume, [phase][y][x][z] in FP32 whatever the stored type (16-bit values are widened
// once here rather than at every gather of the walk): tiles of 32 x by 32 z of one (phase, y) through shared memory.
template <class T>
__global__ void __launch_bounds__(256) k_zfirst(int nx, int ny, int nz, int ntx, int ntz, const T *__restrict__ vol,
                                                float *__restrict__ volz)
{
    __shared__ float s[32][33];
    long long b = blockIdx.x;
    const int x0 = (int)(b % ntx) * 32;
    b /= ntx;
    const int z0 = (int)(b % ntz) * 32;
    b /= ntz;
    const int iy = (int)(b % ny);
    const long long phase = b / ny, nvox = (long long)nx * ny * nz;
    const int i = threadIdx.x & 31, r = threadIdx.x >> 5;
    const T *src = vol + phase * nvox + (long long)iy * nx;
#pragma unroll
    for (int k = r; k < 32; k += 8)
        if (x0 + i < nx && z0 + k < nz) s[k][i] = ld_v(src + (long long)(z0 + k) * ny * nx + x0 + i);
    __syncthreads();
    float *dst = volz + phase * nvox + (long long)iy * nx * nz;
#pragma unroll
    for (int k = r; k < 32; k += 8)
        if (x0 + k < nx && z0 + i < nz) dst[(long long)(x0 + k) * nz + z0 + i] = s[i][k];
}

}  // namespace

long long brick_slice(int nx, int ny) { return (long long)((nx + 3) / 4) * ((ny + 7) / 8) * 32; }

size_t copy_bytes(const KGeom &kg)
{
    return (size_t)kg.np * (kg.by_columns ? (size_t)kg.nz * kg.brick_slice : (size_t)kg.nvox) * sizeof(float);
}

// Projector launch shape code: 2, 4 or 8 = the slab walker k_forward with blocks of 32 x that
// many rows; 102, 104 or 108 = the table walker, once the handle's column tables exist (else the
// slab walker with 4 rows), with blocks of 4, 8 or 16 warps (k_forward_tab) or of 32 x 2, 4 or 8
// pixels (k_forward_cols).
bool forward_shape_valid(int code)
{
    return code == 2 || code == 4 || code == 8 || code == 102 || code == 104 || code == 108;
}

int forward_shape_in_use(const KGeom &kg)
{
    return (kg.fwd_by > 100 && !(kg.coltab && kg.copy)) ? 4 : kg.fwd_by;
}

// Depth within the circle around the volume: all of it (circle_span), and where any ray of the detector rows a .. b is at
// the volume's height (rows_span)
struct DepthSpan {
    double lo, hi;
    double length() const { return fmax(0.0, hi - lo); }
};

static DepthSpan circle_span(const KGeom &kg)
{
    const double x = fmax(fabs((double)kg.b0x), fabs((double)kg.b0x + (double)kg.nx * kg.dx));
    const double y = fmax(fabs((double)kg.b0y), fabs((double)kg.b0y + (double)kg.ny * kg.dy));
    return DepthSpan{kg.sad - hypot(x, y), kg.sad + hypot(x, y)};
}

static DepthSpan rows_span(const KGeom &kg, int a, int b)
{
    DepthSpan d = circle_span(kg);
    const double z1 = (double)kg.b0z * kg.sdd, z2 = z1 + (double)kg.nz * kg.dz * kg.sdd;  // v times depth at the two faces
    const double va = ((double)a - kg.vc) * kg.dv + kg.v_off, vb = ((double)b - kg.vc) * kg.dv + kg.v_off;
    if (vb > 0) d.lo = fmax(d.lo, z1 / vb);  // some ray above the lower face
    else if (vb < 0) d.hi = fmin(d.hi, z1 / vb);
    else if (z1 > 0) d.hi = -1;
    if (va > 0) d.hi = fmin(d.hi, z2 / va);  // and some below the upper one
    else if (va < 0) d.lo = fmax(d.lo, z2 / va);
    else if (z2 < 0) d.hi = -1;
    return d;
}

// Rows of a warp of the table walker.  64 (two per lane; 32 where the detector has no more) cost least per row, but a warp
// walks all its rows through every entry that any of them has in the volume, with a test where not all have, so few detector
// rows and volumes that few rows see take fewer rows of several columns.  kCost: a tile of so many rows, relative; with the
// other constants fitted to the times of all five on 170 scans.  Fewer rows are taken where they are estimated at 0.8 of the
// time or less (they are never more than 1 % slower there) and the launch is more than one wave (32 warps on each of the 152
// SMs; below that 32 rows have the shorter chain, 12.2 against 13.3 us at 32^3 with 40 views of 64 x 8).  The bits do not
// depend on the choice.  64 rows (32 up to 32 detector rows) / the choice, us; before, 32 columns of one row per warp:
//   128x128x64, 160 views of 256 x 2 pixels 113 / 61 (62), x 4 113 / 61 (68), x 8 114 / 65 (95), x 12 119 / 84 (116);
//   128x128xnz, 160 views of 256x192, nz = 1 228 / 154 (117), 4 230 / 147 (137), 8 232 / 187 (173);
//   256x256xnz, 72 views of 512x384, nz = 1 750 / 300 (242), 4 750 / 363 (341), 8 752 / 438 (478), 12 760 / 540 (611).
int walk_rows(const KGeom &kg, int n_views)
{
    constexpr int kRows[] = {64, 32, 16, 8, 4};
    constexpr double kCost[] = {178, 140, 98, 57, 49};
    const DepthSpan whole = circle_span(kg);
    const int usual = kg.nv <= 32 ? 32 : 64;
    if ((long long)kg.nu * n_views * ((kg.nv + usual - 1) / usual) <= 152 * 32) return usual;
    double limit = DBL_MAX;  // the estimate to fall below
    int rows = usual;
    for (int c = 0; c < 5; ++c) {
        const int n = kRows[c];
        if (n > usual) continue;
        double cost = 0.0;
        for (int a = 0; a < kg.nv; a += n) {
            const int b = a + n < kg.nv ? a + n : kg.nv;
            const DepthSpan top = rows_span(kg, a, a), bottom = rows_span(kg, b - 1, b - 1);
            const double any = rows_span(kg, a, b - 1).length();
            const double all = DepthSpan{fmax(top.lo, bottom.lo), fmin(top.hi, bottom.hi)}.length();
            if (any > 0.0) cost += kCost[c] * (0.8 + 0.2 * (b - a) / n) * (any + 1.05 * (any - all) + 0.06 * whole.length());
        }
        if (n == usual) {
            limit = 0.8 * cost;
        } else if (cost < limit) {
            limit = cost;
            rows = n;
        }
    }
    return rows;
}

// The column walk where rays cross more than 0.4 z planes per xy cell on average: settling a plane takes the row walk
// about twice the column walk's time.  Row / column walk by that ratio, us: 2 x 128x128xnz, 40 views of 256x160 with a
// half cone of 16 degrees 0.22 258 / 293, 0.33 324 / 313, 0.44 391 / 332, 0.88 650 / 445; 2 x 64x64xnz, of 6 degrees 0.22 95 /
// 113, 0.44 145 / 132, 1.8 454 / 307.  And beyond 2^20 slices, where the row walk's cells leave a float's low bits.
bool walk_by_columns(const KGeom &kg)
{
    double sum = 0.0;
    int n = 0;
    for (int iv = 0; iv < kg.nv; ++iv)
        if (rows_span(kg, iv, iv).length() > 0.0) {
            sum += fabs(((double)iv - kg.vc) * kg.dv + kg.v_off);
            ++n;
        }
    const double planes = n ? sum / n / ((double)kg.sdd * kg.dz) : 0.0;          // crossed per mm along the ray's xy path
    const double cells = 2.0 / M_PI * (1.0 / (double)kg.dx + 1.0 / (double)kg.dy);  // averaged over the directions
    return kg.nz > (1 << 20) || planes > 0.4 * cells;
}

static dim3 forward_grid(const KGeom &kg, int code, int n_views)
{
    if (code < 100 || kg.by_columns) {
        const int rows = code % 100;
        return dim3((kg.nu + kFwdBX - 1) / kFwdBX, (kg.nv + rows - 1) / rows, n_views);
    }
    const int rows = kg.walk_rows, nc = 2 * (code - 100) * (rows < 32 ? 32 / rows : 1);
    return dim3((kg.nu + nc - 1) / nc, (kg.nv + rows - 1) / rows, n_views);
}

static long long blocks_of(dim3 g) { return (long long)g.x * g.y * g.z; }

long long forward_blocks(const KGeom &kg, int n_views_total)
{
    return blocks_of(forward_grid(kg, forward_shape_in_use(kg), n_views_total));
}

long long forward_blocks_max(const KGeom &kg, int n_views_total)
{
    const long long a = blocks_of(forward_grid(kg, 2, n_views_total)), b = blocks_of(forward_grid(kg, 102, n_views_total));
    return a > b ? a : b;
}

int coltab_kmax(const KGeom &kg)
{
    return (kg.nx + kg.ny - 1 + (kg.by_columns ? kPairPad : kColtabHead + kColtabPad) + 1) & ~1;
}

size_t coltab_entries(const KGeom &kg, int n_views_total)
{
    return (size_t)n_views_total * (size_t)coltab_kmax(kg) * (size_t)kg.nu + kColtabAhead;
}

tnlm_status build_coltab(const KGeom &kg, const ViewGeom *views, int n_views_total, float2 *tab, cudaStream_t st)
{
    const int kmax = coltab_kmax(kg);
    if (kg.nu > 65535) {
        set_error("column tables need nu <= 65535 (got %d)", kg.nu);
        return TNLM_ERR_ARG;
    }
    dim3 grid((kg.nx + kg.ny + 127) / 128, kg.nu, n_views_total);
    if (kg.by_columns)
        k_coltab<true><<<grid, 128, 0, st>>>(kg, views, tab, kmax);
    else
        k_coltab<false><<<grid, 128, 0, st>>>(kg, views, tab, kmax);
    TNLM_TRY_CUDA(cudaGetLastError());
    return TNLM_OK;
}

template <int MODE, int BY, class T>
static void launch_forward_by(const KGeom &kg, const ViewGeom *views, int n_views, const T *vol, const T *y,
                              float *out, double *partials, cudaStream_t st)
{
    k_forward<MODE, BY, T><<<forward_grid(kg, BY, n_views), dim3(kFwdBX, BY), 0, st>>>(kg, views, vol, y, out, partials);
}

// phases ph .. ph + np - 1 of vol into the walk's copy
template <class T>
static void launch_copy(const KGeom &kg, int ph, int np, const T *vol, cudaStream_t st)
{
    const T *src = vol + (long long)ph * kg.nvox;
    float *dst = static_cast<float *>(kg.copy);
    if (kg.by_columns) {
        KGeom kb = kg;
        kb.np = np;
        const long long n = (long long)((kg.nx + 3) / 4) * ((kg.ny + 1) / 2) * kg.nz * np;
        const long long nb = (n + 255) / 256;
        k_brick<T><<<(unsigned)(nb < 152 * 64 ? nb : 152 * 64), 256, 0, st>>>(
            kb, src, dst + (long long)ph * kg.nz * kg.brick_slice);
    } else {
        const int ntx = (kg.nx + 31) / 32, ntz = (kg.nz + 31) / 32;
        k_zfirst<T><<<(unsigned)((long long)ntx * ntz * kg.ny * np), 256, 0, st>>>(kg.nx, kg.ny, kg.nz, ntx, ntz, src,
                                                                                  dst + (long long)ph * kg.nvox);
    }
}

// BY = 2, 4, 8: rows of a block of the column walk, half the warps of one of the row walk
template <int MODE, int BY, class T>
static void launch_walk(const KGeom &kg, const ViewGeom *views, int n_views, const T *y, float *out, double *partials,
                        cudaStream_t st)
{
    constexpr int NC = 2 * BY;
    const dim3 grid = forward_grid(kg, 100 + BY, n_views);
    const int lr2 = kg.walk_rows == 4 ? 2 : (kg.walk_rows == 8 ? 3 : 4);
    const float *copy = static_cast<const float *>(kg.copy);
    if (kg.by_columns)
        k_forward_cols<MODE, BY, T><<<grid, dim3(kFwdBX, BY), 0, st>>>(kg, views, copy, y, out, partials);
    else if (kg.walk_rows == 64)
        k_forward_tab<MODE, NC, 2, T><<<grid, 32 * NC, 0, st>>>(kg, lr2, views, copy, y, out, partials);
    else if (kg.walk_rows == 32)
        k_forward_tab<MODE, NC, 1, T><<<grid, 32 * NC, 0, st>>>(kg, lr2, views, copy, y, out, partials);
    else
        k_forward_tab<MODE, NC, 0, T><<<grid, 32 * NC, 0, st>>>(kg, lr2, views, copy, y, out, partials);
}

template <int MODE, int BY, class T>
static void launch_forward_tab(const KGeom &kg, const ViewGeom *views, int n_views, const T *vol, const T *y,
                               float *out, double *partials, cudaStream_t st)
{
    launch_copy<T>(kg, 0, kg.np, vol, st);
    launch_walk<MODE, BY, T>(kg, views, n_views, y, out, partials, st);
}

template <int MODE, class T>
static void launch_forward_mode(const KGeom &kg, const ViewGeom *views, int n_views_total, const T *vol, const T *y,
                                float *out, double *partials, cudaStream_t st)
{
    switch (forward_shape_in_use(kg)) {
    case 2: launch_forward_by<MODE, 2, T>(kg, views, n_views_total, vol, y, out, partials, st); break;
    case 8: launch_forward_by<MODE, 8, T>(kg, views, n_views_total, vol, y, out, partials, st); break;
    case 102: launch_forward_tab<MODE, 2, T>(kg, views, n_views_total, vol, y, out, partials, st); break;
    case 104: launch_forward_tab<MODE, 4, T>(kg, views, n_views_total, vol, y, out, partials, st); break;
    case 108: launch_forward_tab<MODE, 8, T>(kg, views, n_views_total, vol, y, out, partials, st); break;
    default: launch_forward_by<MODE, 4, T>(kg, views, n_views_total, vol, y, out, partials, st); break;
    }
}

template <class T>
static tnlm_status launch_forward_t(const KGeom &kg, const ViewGeom *views, int n_views_total, const T *vol,
                                    const T *y, float *out, double *partials, int mode, cudaStream_t st)
{
    if (!forward_shape_valid(kg.fwd_by)) {
        set_error("projector launch shape must be 2, 4, 8 (slab walker) or 102, 104, 108 (table walker) (got %d)",
                  kg.fwd_by);
        return TNLM_ERR_ARG;
    }
    if (mode == 0) launch_forward_mode<0, T>(kg, views, n_views_total, vol, nullptr, out, nullptr, st);
    else launch_forward_mode<1, T>(kg, views, n_views_total, vol, y, out, partials, st);
    TNLM_TRY_CUDA(cudaGetLastError());
    return TNLM_OK;
}

tnlm_status launch_forward(const KGeom &kg, const ViewGeom *views, int n_views_total, const float *vol,
                           const float *y, float *out, double *partials, int mode, cudaStream_t st)
{
    return launch_forward_t<float>(kg, views, n_views_total, vol, y, out, partials, mode, st);
}

// One phase's share of a mode-1 projection: phase ph of vol is copied for the table walker and views
// [view_lo, view_hi) projected, writing the same rows of out and the same block partials as the
// whole-volume launch does; the phases of a volume may so be projected as they arrive.
tnlm_status launch_forward_phase(const KGeom &kg, const ViewGeom *views, int ph, int view_lo, int view_hi,
                                 const float *vol, const float *y, float *out, double *partials, cudaStream_t st)
{
    if (!forward_shape_valid(kg.fwd_by)) {
        set_error("projector launch shape must be 2, 4, 8 (slab walker) or 102, 104, 108 (table walker) (got %d)",
                  kg.fwd_by);
        return TNLM_ERR_ARG;
    }
    if (view_hi <= view_lo) return TNLM_OK;
    const int code = forward_shape_in_use(kg), n = view_hi - view_lo;
    const long long off = (long long)view_lo * kg.npix;
    const ViewGeom *vw = views + view_lo;
    double *part = partials + blocks_of(forward_grid(kg, code, view_lo));
    KGeom kt = kg;
    if (code > 100) {
        launch_copy<float>(kg, ph, 1, vol, st);
        kt.coltab = kg.coltab + (long long)view_lo * kg.coltab_kmax * kg.nu;
    }
    switch (code) {
    case 2: launch_forward_by<1, 2, float>(kg, vw, n, vol, y + off, out + off, part, st); break;
    case 8: launch_forward_by<1, 8, float>(kg, vw, n, vol, y + off, out + off, part, st); break;
    case 102: launch_walk<1, 2, float>(kt, vw, n, y + off, out + off, part, st); break;
    case 104: launch_walk<1, 4, float>(kt, vw, n, y + off, out + off, part, st); break;
    case 108: launch_walk<1, 8, float>(kt, vw, n, y + off, out + off, part, st); break;
    default: launch_forward_by<1, 4, float>(kg, vw, n, vol, y + off, out + off, part, st); break;
    }
    TNLM_TRY_CUDA(cudaGetLastError());
    return TNLM_OK;
}

tnlm_status launch_forward(const KGeom &kg, const ViewGeom *views, int n_views_total, const uint16_t *vol,
                           const uint16_t *y, float *out, double *partials, int mode, cudaStream_t st)
{
    using B = __nv_bfloat16;
    return launch_forward_t<B>(kg, views, n_views_total, reinterpret_cast<const B *>(vol),
                               reinterpret_cast<const B *>(y), out, partials, mode, st);
}

tnlm_status launch_forward(const KGeom &kg, const ViewGeom *views, int n_views_total, const __half *vol,
                           const __half *y, float *out, double *partials, int mode, cudaStream_t st)
{
    return launch_forward_t<__half>(kg, views, n_views_total, vol, y, out, partials, mode, st);
}

}  // namespace tnlm
