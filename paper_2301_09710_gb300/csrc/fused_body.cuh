// fused_body.cuh -- device bodies of the fused projector kernels (rotation,
// separable blur + depth sum, blur adjoint + attenuation), their helpers and
// their host-side dimensioning, shared by the per-plan launches (fused.cu) and
// the grouped launches over many plans (grouped.cu).  The kernels themselves
// are thin wrappers that pass their block coordinates to these bodies, so a
// block computes the same values whichever launch runs it.
#pragma once

#include <cstdlib>
#include <type_traits>

#include "spect_internal.cuh"

namespace spect {

namespace {

__device__ __forceinline__ int clampi(int v, int lo, int hi) { return v < lo ? lo : (v > hi ? hi : v); }

// Rotation table entry of rotated-frame pixel (i, j): base voxel index
// (i0c + nx*j0c, clamped so all four reads are in bounds) and the four weights
// of slots (0,0), (1,0), (0,1), (1,1) relative to it; neighbours outside the
// slice (zero padding) get weight 0.
__device__ __forceinline__ void rot_table_entry(int i, int j, const ViewRot r, const Geometry& g, float4& w, int& base)
{
    const Sample s = rot_sample(i, j, r, g.cint, g.cfrac);
    const int bi = clampi(s.i0, 0, g.nx - 2), bj = clampi(s.j0, 0, g.ny - 2);
    float ww[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int dj = 0; dj < 2; ++dj)
#pragma unroll
        for (int di = 0; di < 2; ++di) {
            const int qi = s.i0 + di, qj = s.j0 + dj;
            if (qi >= 0 && qi < g.nx && qj >= 0 && qj < g.ny) ww[(qi - bi) + 2 * (qj - bj)] = bilinear_w(s, di, dj);
        }
    w = make_float4(ww[0], ww[1], ww[2], ww[3]);
    base = bi + g.nx * bj;
}

}  // namespace

// out[c][r] = in[r][c] for the 32x32 tile (bx, by) of an R x C matrix with row
// pitches ip and op (tiled through shared memory; blocks of 32 x 8 threads).
__device__ __forceinline__ void transpose_body(const float* __restrict__ in, float* __restrict__ out, int R, int C,
                                               int ip, int op, int bx, int by)
{
    __shared__ float tile[32][33];
    const int c0 = bx * 32, r0 = by * 32;
    for (int dy = threadIdx.y; dy < 32; dy += blockDim.y) {
        const int r = r0 + dy, c = c0 + threadIdx.x;
        if (r < R && c < C) tile[dy][threadIdx.x] = in[(size_t)r * ip + c];
    }
    __syncthreads();
    for (int dy = threadIdx.y; dy < 32; dy += blockDim.y) {
        const int c = c0 + dy, r = r0 + threadIdx.x;
        if (r < R && c < C) out[(size_t)c * op + r] = tile[threadIdx.x][dy];
    }
}

// ============================================================================
// Fused forward, separable PSF, padded tap count P (odd).
//
// The forward runs as two kernels: k_rot_fwd rotates and attenuates every
// (view, depth) plane into a plane image [i][k] of the work slab;
// k_fwd_sep_fused (one block per view, depth group and column tile) streams
// tiles of those images in by TMA and blurs them.  Its shared memory:
//   W   one or two tile buffers, as runs of 32 k: W[k / 32][C + i][k % 32], zero
//       outside the plane (the tensor copy's fill); the i-pass windows (lanes over
//       k) are conflict-free loads at immediate offsets.
//   U   nx rows x kpu: i-pass output, U[i][ZH + k], with zero halo columns;
//       kpu/4 is odd so the k-pass float4 windows (lanes over i) are
//       bank-conflict free.
//   Replicate padding enters both passes as folded edge taps on top of the
//   zero-padded FIR: output k adds U(0) sum_{b>k+C} fz(b) + U(nz-1) sum_{b<k+C-nz+1} fz(b),
//   and likewise along i.
//   taps and folded edge taps of every plane of the group, staged once.
// The depth sums stay in registers.
// Per plane there are two block barriers: after the i-pass (which also agrees
// on the bounded TMA wait) and after the k-pass.
// ============================================================================
template <int P>
struct Sep {
    static constexpr int C = (P - 1) / 2;    // tap centre
    static constexpr int CX = 16;            // i outputs per thread (i-pass)
    static constexpr int CZ = 16;            // k outputs per thread (k-pass)
    static constexpr int ZH = (C + 3) & ~3;  // k halo columns, 16-byte aligned
    static constexpr int WZ = CZ + 2 * ZH;   // k-pass window (multiple of 4)
    static constexpr int PT = (P + 3) & ~3;  // tap array length
};

constexpr int kFusedThreads = 640;

// Largest block of the forward blur and the resident blocks its registers are bounded
// for.  Short FIRs (P <= 11) wait more on shared memory and barriers than on FMAs, so
// they get at most 72 registers (two blocks of 448, seven of 128) instead of about 80.
template <int P>
struct FwdBlock {
    static constexpr int T = P <= 11 ? 448 : kFusedThreads;
    static constexpr int B = P <= 11 ? 2 : 1;
    static constexpr int regs = P <= 11 ? 72 : 80;
};

// Bounds of the geometries and launch shapes that the fused kernels take (the kernels
// need less): a plane cut into nT column tiles of TI detector columns (TI a multiple
// of CX), each with C halo columns on each side, two tile buffers, U, accumulators,
// taps and folds in shared memory.
struct FusedDims {
    int wp;     // W row pitch of one tile image (pitch4odd(TI + 2*C))
    int warea;  // floats of one tile image, nz x wp (multiple of 4, keeps U 16-byte aligned)
    int kpu;    // U row pitch (>= nkb*CZ + 2*ZH, multiple of 4, pitch/4 odd)
    int nib, nkb;
    int TI, nT; // tile width in columns (multiple of CX), tiles per plane
    int farea;  // floats of a whole plane with halo columns (bound of the shapes taken, rot_smem_bound)
    int urows;  // rows of U / ACC / MB per tile: min(TI, nx)
    int vrows;  // detector rows a tile's k-adjoint needs: min(nx, TI + 2*C)
    int marea;  // floats of an attenuation tile, urows*kp
    int J, G;   // depth planes per block, depth groups
    int ps;     // plane stride of the attenuation cache / slab (nx*kp)
    int ts;     // rotation table block per (view, row): 5*nx rounded up to 4
    int apc;    // accumulator row pitch (>= nkb*CZ, multiple of 4, pitch/4 odd)
};

template <int P>
__device__ __forceinline__ void load_window_f4(const float* base, float (&win)[Sep<P>::WZ])
{
    const float4* row = reinterpret_cast<const float4*>(base);
#pragma unroll
    for (int m4 = 0; m4 < Sep<P>::WZ / 4; ++m4) {
        const float4 t = row[m4];
        win[4 * m4] = t.x;
        win[4 * m4 + 1] = t.y;
        win[4 * m4 + 2] = t.z;
        win[4 * m4 + 3] = t.w;
    }
}

// A sliding window along a plane-image row (16-byte aligned, pitch4odd pitch):
// N floats (a multiple of 4) as float4 loads; the FIRs read its first CX + P - 1.
template <int N>
__device__ __forceinline__ void load_row_f4(const float* row, float (&win)[N])
{
    static_assert(N % 4 == 0, "window length must be a multiple of 4");
#pragma unroll
    for (int m4 = 0; m4 < N / 4; ++m4) {
        const float4 t = reinterpret_cast<const float4*>(row)[m4];
        win[4 * m4] = t.x;
        win[4 * m4 + 1] = t.y;
        win[4 * m4 + 2] = t.z;
        win[4 * m4 + 3] = t.w;
    }
}

// o[c] = sum_b taps[b] win[c + SIGN*b + OFF]   (SIGN = -1: convolution, +1: correlation)
template <int P, int N, int SIGN, int OFF, int WN>
__device__ __forceinline__ void fir(const float* taps, const float (&win)[WN], float (&o)[N])
{
    constexpr int PT = Sep<P>::PT;
#pragma unroll
    for (int c = 0; c < N; ++c) o[c] = 0.f;
#pragma unroll
    for (int b4 = 0; b4 < PT / 4; ++b4) {
        const float4 f4 = reinterpret_cast<const float4*>(taps)[b4];
        const float fv[4] = {f4.x, f4.y, f4.z, f4.w};
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int b = 4 * b4 + u;
            if (b < P) {
#pragma unroll
                for (int c = 0; c < N; ++c) o[c] = fmaf(fv[u], win[c + SIGN * b + OFF], o[c]);
            }
        }
    }
}

// o[c] += u * f[c] (f 16-byte aligned)
template <int N>
__device__ __forceinline__ void fold_taps(float u, const float* f, float (&o)[N])
{
#pragma unroll
    for (int c4 = 0; c4 < N / 4; ++c4) {
        const float4 t = reinterpret_cast<const float4*>(f)[c4];
        o[4 * c4] = fmaf(u, t.x, o[4 * c4]);
        o[4 * c4 + 1] = fmaf(u, t.y, o[4 * c4 + 1]);
        o[4 * c4 + 2] = fmaf(u, t.z, o[4 * c4 + 2]);
        o[4 * c4 + 3] = fmaf(u, t.w, o[4 * c4 + 3]);
    }
}

// The same for any u: a fold is 0 for the outputs of a run that the padding does not reach,
// and those are left out where u is not finite (0 * inf).  EM updates with u untested and
// tested: 64x32 (two) 144.0 and 144.7 us, 99x53 326.9 and 328.5, 128x80 1453 and 1458;
// testing every fold, or limiting a run to its outputs, costs 1 to 2 %.
template <int N>
__device__ __forceinline__ void fold_taps_any(float u, const float* f, float (&o)[N])
{
    if (fabsf(u) <= FLT_MAX) {
        fold_taps(u, f, o);
    } else {
#pragma unroll
        for (int c = 0; c < N; ++c)
            if (f[c] != 0.f) o[c] = fmaf(u, f[c], o[c]);
    }
}

// Record a timed-out bounded wait in the plan's error word.
__device__ __forceinline__ void flag_timeout(int* err)
{
    if (err) atomicExch(err, (int)SPECT_ETIMEOUT);
}

// ----------------------------------------------------------------------------
// Forward rotation and attenuation into plane images [j][i][k], the layout of x_t, of
// the attenuation factors and of the adjoint's t planes, so nothing is transposed:
// a thread takes four consecutive k of a column i (16-byte corner loads, attenuation
// read and store, coalesced over the lanes at any nz) through JP planes of a view;
// neighbouring planes share source columns in L1, and the next plane's table entry is
// loaded while this one is gathered.  No shared memory and no barriers.
//   Bound by DRAM: 8 bytes per voxel-view, attenuation in and image out (128x128x80,
// 128 views: 238 us, 5.6 TB/s; 160x160x96, 120 views: 418 us; 192x192x128, 128 views:
// 863 us, all of 6.7 TB/s copy rate at most).  Assembling whole [k][i] planes in shared
// memory took 392, 1274 and 3063 us (one block per SM from 160x96 on), 32-column tiles
// transposed through shared memory 418, 642 and 1246 (a barrier per plane before
// each round of gathers).
//   TAPS = 4: bilinear, table block (l, j) = nx float4 weights, then nx base voxels;
//   TAPS = 8: three-pass rotation, nx x 8 weights, then nx x 8 element offsets.
// ----------------------------------------------------------------------------
constexpr int kRotThreads = 256;

struct RotDims {
    int ps, ts;  // plane stride of images and attenuation factors; table block of a (view, plane)
    int nb, JP;  // blocks per plane; planes per block
};

__device__ __forceinline__ float4 ld_stream4(const float* p)
{
    float4 v;
    asm volatile("ld.global.nc.L1::no_allocate.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
                 : "l"(p));
    return v;
}

template <int TAPS>
__device__ __forceinline__ void rot_body(const Geometry& g, const RotDims& d, const float* __restrict__ tabs,
                                         const float* __restrict__ xt, const float* __restrict__ mubar,
                                         float* __restrict__ wsl, int l0, const int bx, const int v)
{
    const int nx = g.nx, kp = g.kp, k4 = kp >> 2;
    const int jb = bx / d.nb, e = (bx - jb * d.nb) * kRotThreads + (int)threadIdx.x;
    if (e >= nx * k4) return;
    const int i = e / k4, l = l0 + v;
    const int j0 = jb * d.JP, j_end = min(g.ny, j0 + d.JP);
    const int pln = nx * kp;
    const float* x = xt + 4 * (e - i * k4);
    constexpr int NO = TAPS == 4 ? 1 : TAPS;  // bilinear: the base column, its neighbours follow from it
    float w[TAPS], wn[TAPS] = {};
    int o[NO], on[NO] = {};
    auto table = [&](int j, float (&tw)[TAPS], int (&to)[NO]) {
        const float* tab = tabs + ((size_t)l * g.ny + j) * d.ts;
        if (TAPS == 4) {
            const float4 t = __ldg(reinterpret_cast<const float4*>(tab) + i);
            tw[0] = t.x, tw[1] = t.y, tw[2] = t.z, tw[3] = t.w;
            to[0] = __ldg(reinterpret_cast<const int*>(tab + 4 * nx) + i) * kp;
        } else {
#pragma unroll
            for (int h = 0; h < NO / 4; ++h) {
                const float4 t = __ldg(reinterpret_cast<const float4*>(tab) + (TAPS / 4) * i + h);
                const int4 b = __ldg(reinterpret_cast<const int4*>(tab + TAPS * nx) + (TAPS / 4) * i + h);
                tw[4 * h] = t.x, tw[4 * h + 1] = t.y, tw[4 * h + 2] = t.z, tw[4 * h + 3] = t.w;
                to[4 * h] = b.x, to[4 * h + 1] = b.y, to[4 * h + 2] = b.z, to[4 * h + 3] = b.w;
            }
        }
    };
    table(j0, w, o);
    const float* mb = mubar + ((size_t)l * g.ny + j0) * d.ps + 4 * (size_t)e;
    float* out = wsl + ((size_t)v * g.ny + j0) * d.ps + 4 * (size_t)e;
#pragma unroll 1
    for (int j = j0; j < j_end; ++j, mb += d.ps, out += d.ps) {
        const float4 m = ld_stream4(mb);
        float4 c[TAPS];
#pragma unroll
        for (int t = 0; t < TAPS; ++t)
            c[t] = __ldg(reinterpret_cast<const float4*>(
                x + (TAPS == 4 ? o[0] + (t & 1) * kp + (t >> 1) * pln : o[t < NO ? t : 0])));
        if (j + 1 < j_end) table(j + 1, wn, on);
        float4 a = make_float4(w[0] * c[0].x, w[0] * c[0].y, w[0] * c[0].z, w[0] * c[0].w);
#pragma unroll
        for (int t = 1; t < TAPS; ++t) {
            a.x = fmaf(w[t], c[t].x, a.x);
            a.y = fmaf(w[t], c[t].y, a.y);
            a.z = fmaf(w[t], c[t].z, a.z);
            a.w = fmaf(w[t], c[t].w, a.w);
        }
        *reinterpret_cast<float4*>(out) = make_float4(a.x * m.x, a.y * m.y, a.z * m.z, a.w * m.w);
#pragma unroll
        for (int t = 0; t < TAPS; ++t) w[t] = wn[t];
#pragma unroll
        for (int t = 0; t < NO; ++t) o[t] = on[t];
    }
}

inline RotDims rot_dims(const Geometry& g, int ps, int ts, int nv, int sms)
{
    RotDims d;
    d.ps = ps;
    d.ts = ts;
    d.nb = (g.nx * (g.kp / 4) + kRotThreads - 1) / kRotThreads;
    // eight planes per block, fewer where that would leave SMs without eight blocks
    d.JP = 8;
    while (d.JP > 1 && (long long)d.nb * ((g.ny + d.JP - 1) / d.JP) * nv < 8ll * sms) d.JP /= 2;
    return d;
}

// Launch shape of the forward blur: one block per depth group of J planes, view
// and column tile of TI detector columns.  A tile is nbox TMA boxes (32 k x wr
// columns) of the rotated plane image, C halo columns on each side included, so
// every tile is blurred independently from one image.
constexpr int kWK = 32;  // k of a box

struct FwdDims {
    int TI, nT;        // tile width in columns (multiple of CX), tiles per plane
    int wr, nbox;      // columns of a box: TI + 2C (at most 256); boxes per plane: ceil(nz / 32)
    int warea;         // floats of a tile buffer: nbox * wr * 32
    int nbuf;          // tile buffers (1 or 2): planes in flight per block
    int kpu, nkb, nib; // U row pitch; k runs; column runs of the whole plane
    int urows;         // rows of U: min(TI, nx)
    int J, G;          // depth planes per block, depth groups
    int T;             // threads per block
    int racc;          // depth sums in registers (every k-pass item has its own thread)
    int apc;           // row pitch of the shared accumulators (racc == 0)
};

// Tap record of one PSF plane (view, depth) for the forward blur, built at plan
// time (k_fwd_records): FX and FZ zero-padded to P and centred (PT floats each),
// then the folded edge taps of replicate padding: along k lo and hi (nkb * 16
// floats each; output k adds U(0) lo(k) + U(nz-1) hi(k), lo(k) = sum_{b > k+C} fz(b),
// hi(k) = sum_{b < k+C-nz+1} fz(b)), along i likewise, lo for the columns
// [0, kFoldLo) and hi for the kFoldHi columns from fold_hi0(nx).  A group's records
// are contiguous, so a block fetches them with one bulk copy instead of building them.
constexpr int kFoldLo = 32;  // runs of 16 columns that start before C <= 18
constexpr int kFoldHi = 48;  // the same at the other end: C + 15 + 15 columns at most
__host__ __device__ inline int fold_hi0(int nx, int C) { return nx > C ? (nx - C) & ~15 : 0; }
__host__ __device__ inline int fwd_rec_floats(int PT, int nkb) { return 2 * PT + 2 * 16 * nkb + kFoldLo + kFoldHi; }

__host__ __device__ inline size_t fwd_smem_floats(const FwdDims& d, int PT)
{
    // W x nbuf | U | tap records of J planes | ACC (racc == 0) | 3 mbarriers
    return (size_t)d.nbuf * d.warea + (size_t)d.urows * d.kpu + (size_t)d.J * fwd_rec_floats(PT, d.nkb) +
           (d.racc ? 0 : (size_t)d.urows * d.apc) + 8;
}

// The compensated sum over depth groups of partials p[q * stride] (comp: their compensation
// terms, or NULL).  One that is not finite is the plain sum's infinity or NaN (an overflow
// leaves NaN in the compensation).
__device__ __forceinline__ float group_sum(const float* __restrict__ p, const float* __restrict__ comp, int G, size_t stride)
{
    KSum acc;
    if (comp)
        for (int q = 0; q < G; ++q) acc.merge(p[(size_t)q * stride], comp[(size_t)q * stride]);
    else
        for (int q = 0; q < G; ++q) acc.add(p[(size_t)q * stride]);
    float s = acc.value();
    if (!(fabsf(s) <= FLT_MAX)) {
        s = 0.f;
        for (int q = 0; q < G; ++q) s += p[(size_t)q * stride];
    }
    return s;
}

// A depth sum: plain, or compensated (KS).  store() leaves a group's sum at p, a
// compensated one's compensation term at p + half, for the reduce to carry on with.
template <bool KS>
struct DepthSum {
    float s = 0.f;
    __device__ __forceinline__ void add(float x) { s += x; }
    __device__ __forceinline__ void store(float* p, size_t) const { *p = s; }
};
template <>
struct DepthSum<true> : KSum {
    __device__ __forceinline__ void store(float* p, size_t half) const { p[0] = s, p[half] = c; }
};

// KS: low-memory plans, whose depth sums are compensated over all depths, as the general
// kernels' are.  Relative error of A, with the groups' terms carried on and with each
// group rounded: 64x32, 11 taps 3.24e-8 and 3.50e-8, 16x600, 3 taps 3.60e-8 and 4.19e-8
// (general kernels 3.04e-8 and 3.60e-8); 96x96x64, 60 views: 508 and 511 us an EM update.
// Compensated sums for every plan cost 5 to 14 % of the forward blur.
// RACC: a thread keeps the depth sums of its one k-pass item (16 k of a column)
// in registers over all planes of the group, so the k-pass touches shared memory
// only to read U; otherwise (planes of more than 640 items) they are in ACC.
template <int P, bool RACC, bool KS>
__device__ __forceinline__ void fwd_sep_body(const Geometry& g, const FwdDims& d, const CUtensorMap* tmap,
                                             const float* __restrict__ rec, float* __restrict__ part, int l0, int nv,
                                             int* err, const int grp, const int v, const int tile)
{
    using S = Sep<P>;
    constexpr int C = S::C, CX = S::CX, CZ = S::CZ, ZH = S::ZH, WZ = S::WZ, PT = S::PT;
    extern __shared__ __align__(128) float smf[];
    const int nx = g.nx, ny = g.ny, nz = g.nz;
    float* WB = smf;                                   // [nbuf][warea]
    float* U = WB + (size_t)d.nbuf * d.warea;
    float* TAP = U + (size_t)d.urows * d.kpu;          // the records of every plane of the group
    const int rf = fwd_rec_floats(PT, d.nkb);
    float* ACC = TAP + (size_t)d.J * rf;               // urows x apc, [i - i0][k] (!RACC)
    uint64_t* bar = reinterpret_cast<uint64_t*>(ACC + (RACC ? 0 : (size_t)d.urows * d.apc));  // buffers, records
    const int tid = threadIdx.x, T = blockDim.x;
    const int l = l0 + v;
    const int i0 = tile * d.TI, ti = min(d.TI, nx - i0), nibt = (ti + CX - 1) / CX;
    const int lp = g.nvp == 1 ? 0 : l;
    const int j_begin = grp * d.J, nj = min(ny - j_begin, d.J);
    const int pln = nx * nz;

    // tensor copies want 128-byte aligned shared memory: refuse (error word) rather than fault
    if ((smem_u32(smf) & 127u) != 0) {
        if (tid == 0 && err) atomicExch(err, (int)SPECT_ECUDA);
        return;
    }
    auto request = [&](int n) {  // plane j_begin + n into its buffer
        const int b = d.nbuf == 1 ? 0 : n & 1;
        float* dst = WB + (size_t)b * d.warea;
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar + b)),
                     "r"((unsigned)d.warea * 4u)
                     : "memory");
        for (int q = 0; q < d.nbox; ++q)
            tma_load_3d(dst + q * d.wr * kWK, tmap, q * kWK, i0 - C, v * ny + j_begin + n, bar + b);
    };
    // the first planes are requested before anything else, so their loads overlap the set-up below
    if (tid == 0) {
        mbar_init(bar, 1);
        mbar_init(bar + 1, 1);
        mbar_init(bar + 2, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        tma_load_1d(TAP, rec + ((size_t)lp * ny + j_begin) * rf, (unsigned)(nj * rf) * 4u, bar + 2);
        for (int n = 0; n < d.nbuf && n < nj; ++n) request(n);
    }
    if (!RACC)
        for (int e = tid; e < d.urows * d.apc; e += T) ACC[e] = 0.f;
    // zero k-halo columns of U (never written again): [0, ZH) and [ZH + nz, kpu) of each row
    for (int r = tid; r < d.urows; r += T) {
        float* ur = U + r * d.kpu;
#pragma unroll
        for (int c = 0; c < ZH; c += 4) *reinterpret_cast<float4*>(ur + c) = make_float4(0.f, 0.f, 0.f, 0.f);
        int c = ZH + nz;
        for (; c & 3; ++c) ur[c] = 0.f;
        for (; c < d.kpu; c += 4) *reinterpret_cast<float4*>(ur + c) = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    __syncthreads();  // the barriers are initialised and U's halos are zero
    bool ok = mbar_wait_bounded(bar + 2, 0u);

    const int hi0 = fold_hi0(nx, C);
    // the thread's first work item of each pass and the step to its next one
    // (the same for every plane: the divisions stay out of the plane loop)
    const int ip_ib = tid / nz, ip_k = tid - ip_ib * nz;    // i-pass: (column run, k)
    const int kp_kb = tid / ti, kp_i = tid - kp_kb * ti;    // k-pass: (k run, column)
    const int ip_dib = T / nz, ip_dk = T - ip_dib * nz;
    const int kp_dkb = T / ti, kp_di = T - kp_dkb * ti;
    DepthSum<KS> acc[CZ];  // RACC: the depth sums of item (kp_kb, kp_i)

    for (int n = 0; n < nj; ++n) {
        const int b = d.nbuf == 1 ? 0 : n & 1;
        const unsigned parity = (unsigned)(d.nbuf == 1 ? n : n >> 1) & 1u;
        const float* FX = TAP + n * rf;
        const float* FZ = FX + PT;
        const float* xlo = FZ + PT + 2 * d.nkb * CZ;
        const float* xhi = xlo + kFoldLo;
        const float* W = WB + (size_t)b * d.warea;
        ok = mbar_wait_bounded(bar + b, parity) && ok;

        // i-pass: U(i,k) = sum_a fx(a) w(clamp(i-a+cx), k); lanes over k
        if (ok) {
            int ib = ip_ib, k = ip_k;
            for (int it = tid; it < nz * nibt; it += T) {
                const int li = ib * CX;  // first column of this run, relative to the tile
                const float* wr = W + (k / kWK) * (d.wr * kWK) + k % kWK;
                float win[CX + P - 1];
#pragma unroll
                for (int m = 0; m < CX + P - 1; ++m) win[m] = wr[(li + m) * kWK];
                float o[CX];
                fir<P, CX, -1, P - 1>(FX, win, o);
                // folded taps of the plane's first and last columns (zero elsewhere)
                if (i0 + li < C) fold_taps_any(wr[(C - i0) * kWK], xlo + i0 + li, o);
                if (i0 + li >= hi0) fold_taps_any(wr[(C + nx - 1 - i0) * kWK], xhi + i0 + li - hi0, o);
                float* ur = U + li * d.kpu + ZH + k;
                if (li + CX <= ti) {
#pragma unroll
                    for (int c = 0; c < CX; ++c) ur[c * d.kpu] = o[c];
                } else {
#pragma unroll
                    for (int c = 0; c < CX; ++c)
                        if (li + c < ti) ur[c * d.kpu] = o[c];
                }
                ib += ip_dib;  // next item: it + T
                k += ip_dk;
                if (k >= nz) k -= nz, ++ib;
            }
        }
        if (__syncthreads_or(!ok)) {
            if (tid == 0) {  // a last chance for the copies in flight to land
                flag_timeout(err);
                mbar_wait_bounded(bar + 2, 0u);
                for (int m = n; m < n + d.nbuf && m < nj; ++m)
                    mbar_wait_bounded(bar + (d.nbuf == 1 ? 0 : m & 1), (unsigned)(d.nbuf == 1 ? m : m >> 1) & 1u);
            }
            return;
        }
        // buffer b has been read: request its next plane (from the last warp, which has the fewest halo rows below)
        if (tid == T - 32 && n + d.nbuf < nj) {
            fence_proxy_async_smem();
            request(n + d.nbuf);
        }

        // k-pass into the depth sums: lanes over i; zero-padded FIR plus the
        // folded replicate-padding terms on the edge rows
        const float* fold_lo = FZ + PT;  // zero outside the first (lo) and last (hi) C rows
        const float* fold_hi = fold_lo + d.nkb * CZ;
        auto kpass = [&](int kb, int i, float (&o)[CZ]) {
            const float* ur = U + i * d.kpu;
            float win[WZ];
            load_window_f4<P>(ur + kb * CZ, win);
            fir<P, CZ, -1, C + ZH>(FZ, win, o);
            const int k0 = kb * CZ;
            // folded taps are zero outside the first and last C rows
            if (k0 + CZ > nz - C) fold_taps(ur[ZH + nz - 1], fold_hi + k0, o);
            if (k0 < C) fold_taps(ur[ZH], fold_lo + k0, o);
        };
        if (RACC) {
            if (tid < ti * d.nkb) {
                float o[CZ];
                kpass(kp_kb, kp_i, o);
#pragma unroll
                for (int c = 0; c < CZ; ++c) acc[c].add(o[c]);
            }
        } else {
            int kb = kp_kb, i = kp_i;  // i relative to the tile
            for (int it = tid; it < ti * d.nkb; it += T) {
                float o[CZ];
                kpass(kb, i, o);
                float4* acc4 = reinterpret_cast<float4*>(ACC + i * d.apc + kb * CZ);
#pragma unroll
                for (int c4 = 0; c4 < CZ / 4; ++c4) {
                    float4 a = acc4[c4];
                    a.x += o[4 * c4];
                    a.y += o[4 * c4 + 1];
                    a.z += o[4 * c4 + 2];
                    a.w += o[4 * c4 + 3];
                    acc4[c4] = a;
                }
                kb += kp_dkb;  // next item: it + T
                i += kp_di;
                if (i >= ti) i -= ti, ++kb;
            }
        }
        __syncthreads();
    }

    // partial depth sums of this group: part[grp][v][k][i] (v of the nv views of the pass), this tile's columns
    float* pout = part + ((size_t)grp * nv + v) * pln + i0;
    const size_t half = (size_t)d.G * nv * pln;
    if (RACC) {
        if (tid < ti * d.nkb) {
#pragma unroll
            for (int c = 0; c < CZ; ++c) {
                const int k = kp_kb * CZ + c;
                if (k < nz) acc[c].store(pout + (size_t)k * nx + kp_i, half);
            }
        }
    } else {
        for (int e = tid; e < nz * ti; e += T) {
            const int k = e / ti, i = e - k * ti;
            pout[(size_t)k * nx + i] = ACC[i * d.apc + k];
        }
    }
}

// ============================================================================
// Fused transpose of the blur + attenuation, separable PSF: the forward blur's tiles
// and passes in the same order (the i and k transposes commute), so no detector
// column is blurred for two tiles.  Per plane of the group:
//   i-adjoint  U(i,k) = sum_a fx~(a) v(i+a-cx, k), lanes over k, windows along the
//     rows of V (nz x vp, V[k][ZH + i - i0]), staged once per block as tensor boxes of
//     the detector plane (zero fill outside);
//   k-adjoint  wbar(i,k) = sum_b fz~(b) U(i, k+b-cz), lanes over i, 16 k per thread,
//     times mubar in MB, in place: t.
// MB is one or two buffers of nkb boxes (16 k x TI columns) that arrive from the
// attenuation factors and leave for the t slab by TMA, 64-byte swizzled: the 16-byte
// chunk q of column i sits at q ^ (i / 2 % 4), so the float4 accesses of eight lanes
// over i are conflict-free.  The first and last detector row and column, where
// replicate padding folds taps together, take their edge-class taps.
// ============================================================================
struct AdjDims {
    int TI, nT;        // tile width in columns (multiple of CX), tiles per plane
    int vp, kpu;       // row pitches of V (pitch4odd(TI + 2ZH) <= 252, a tensor box's width) and U (multiples of 4, /4 odd)
    int vbox, vrows;   // tensor boxes of V and detector rows per box
    int varea;         // floats of V, rounded up to 128 bytes
    int nkb, urows;    // k runs; rows of U: min(TI, nx)
    int marea, nmb;    // floats of an attenuation buffer (nkb * TI * 16); buffers
    int J, G, T;       // depth planes per block, depth groups, threads
};

// Tap record of one PSF plane for the blur adjoint (k_adj_records): FX and FZ of the
// interior class (PT floats each, zero-padded to P and centred), then the taps of the
// first and last column and of the first and last row that are not zero (C + 1 each,
// EC floats): first takes v(0 .. C), last v(n-1-C .. n-1).
template <int P>
struct AdjRec {
    static constexpr int EC = (Sep<P>::C + 4) & ~3;
    static constexpr int N = 2 * Sep<P>::PT + 4 * EC;
};

__host__ __device__ inline size_t adj_smem_floats(const AdjDims& d, int rec)
{
    // MB x nmb | V | U | tap records of J planes | 3 mbarriers
    return (size_t)d.nmb * d.marea + (size_t)d.varea + (size_t)d.urows * d.kpu + (size_t)d.J * rec + 8;
}

// sum_m taps[m] row[s + m], m = 0..N-1 (taps 16-byte aligned): the samples come in as
// float4 loads from the aligned position s & ~3, the shift s & 3 selects a compile-
// time offset.  May read up to 3 floats past row[s + N - 1], which are not used.
template <int N>
__device__ __forceinline__ float edge_dot(const float* taps, const float* row, int s)
{
    float w[4 * ((N + 3 + 3) / 4)], f[(N + 3) & ~3];
    load_row_f4(row + (s & ~3), w);
    load_row_f4(taps, f);
    float acc = 0.f;
    switch (s & 3) {
        case 0:
#pragma unroll
            for (int m = 0; m < N; ++m) acc = fmaf(f[m], w[m], acc);
            break;
        case 1:
#pragma unroll
            for (int m = 0; m < N; ++m) acc = fmaf(f[m], w[m + 1], acc);
            break;
        case 2:
#pragma unroll
            for (int m = 0; m < N; ++m) acc = fmaf(f[m], w[m + 2], acc);
            break;
        default:
#pragma unroll
            for (int m = 0; m < N; ++m) acc = fmaf(f[m], w[m + 3], acc);
    }
    return acc;
}

// sum_m taps[m] w[m + OFF], m = 0..N-1
template <int N, int OFF, int WN>
__device__ __forceinline__ float edge_dot_reg(const float* taps, const float (&w)[WN])
{
    static_assert(N - 1 + OFF < WN, "window too short");
    float f[(N + 3) & ~3], acc = 0.f;
    load_row_f4(taps, f);
#pragma unroll
    for (int m = 0; m < N; ++m) acc = fmaf(f[m], w[m + OFF], acc);
    return acc;
}

template <int P>
__device__ __forceinline__ void adj_sep_body(const Geometry& g, const AdjDims& d, const CUtensorMap* mu_map,
                                             const CUtensorMap* t_map, const CUtensorMap* v_map,
                                             const float* __restrict__ rec, int l0, int mu_l0, int* err,
                                             const int grp, const int v, const int tile)
{
    using S = Sep<P>;
    constexpr int C = S::C, CX = S::CX, CZ = S::CZ, ZH = S::ZH, WZ = S::WZ, PT = S::PT;
    constexpr int EC = AdjRec<P>::EC, RN = AdjRec<P>::N;
    extern __shared__ __align__(1024) float sma[];
    const int nx = g.nx, ny = g.ny, nz = g.nz;
    float* MB = sma;                                       // [nmb][nkb][TI][16]
    float* V = MB + (size_t)d.nmb * d.marea;               // [nz][vp]
    float* U = V + (size_t)d.varea;                        // [urows][kpu]
    float* TAP = U + (size_t)d.urows * d.kpu;              // the records of every plane of the group
    uint64_t* bar = reinterpret_cast<uint64_t*>(TAP + (size_t)d.J * RN);  // buffers, records
    const int tid = threadIdx.x, T = blockDim.x;
    const int l = l0 + v;
    const int i0 = tile * d.TI, ti = min(d.TI, nx - i0), nibt = (ti + CX - 1) / CX;
    const int lp = g.nvp == 1 ? 0 : l;
    const int j_begin = grp * d.J, nj = min(ny - j_begin, d.J);

    // swizzled tensor copies want 512-byte aligned shared memory: refuse (error word) rather than fault
    if ((smem_u32(sma) & 511u) != 0) {
        if (tid == 0 && err) atomicExch(err, (int)SPECT_ECUDA);
        return;
    }
    auto request = [&](int n) {  // attenuation factors of plane j_begin + n into their buffer
        const int b = d.nmb == 1 ? 0 : n & 1;
        float* dst = MB + (size_t)b * d.marea;
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar + b)),
                     "r"((unsigned)d.marea * 4u)
                     : "memory");
        for (int q = 0; q < d.nkb; ++q)
            tma_load_3d(dst + q * d.TI * 16, mu_map, q * 16, i0, (l - mu_l0) * ny + j_begin + n, bar + b);
    };
    if (tid == 0) {
        mbar_init(bar, 1);
        mbar_init(bar + 1, 1);
        mbar_init(bar + 2, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar + 2)),
                     "r"((unsigned)(nj * RN + d.vbox * d.vrows * d.vp) * 4u)
                     : "memory");
        tma_copy_1d(TAP, rec + ((size_t)lp * ny + j_begin) * RN, (unsigned)(nj * RN) * 4u, bar + 2);
        for (int q = 0; q < d.vbox; ++q)
            tma_load_3d(V + q * d.vrows * d.vp, v_map, i0 - ZH, q * d.vrows, l, bar + 2);
        request(0);
    }
    // zero k-halo columns of U (never written again): [0, ZH) and [ZH + nz, kpu) of each row
    for (int r = tid; r < d.urows; r += T) {
        float* ur = U + r * d.kpu;
#pragma unroll
        for (int c = 0; c < ZH; c += 4) *reinterpret_cast<float4*>(ur + c) = make_float4(0.f, 0.f, 0.f, 0.f);
        int c = ZH + nz;
        for (; c & 3; ++c) ur[c] = 0.f;
        for (; c < d.kpu; c += 4) *reinterpret_cast<float4*>(ur + c) = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    __syncthreads();  // the barriers are initialised and U's halos are zero
    bool ok = mbar_wait_bounded(bar + 2, 0u);

    // the thread's first work item of each pass and the step to its next one
    // (the same for every plane: the divisions stay out of the plane loop)
    const int ia_ib = tid / nz, ia_k = tid - ia_ib * nz;    // i-adjoint: (column run, k)
    const int ka_kb = tid / ti, ka_i = tid - ka_kb * ti;    // k-adjoint: (k run, column)
    const int ia_dib = T / nz, ia_dk = T - ia_dib * nz;
    const int ka_dkb = T / ti, ka_di = T - ka_dkb * ti;
    const int last_col = nx - 1 - i0;  // tile-relative position of column nx-1
    for (int n = 0; n < nj; ++n) {
        const int b = d.nmb == 1 ? 0 : n & 1;
        const float* FX = TAP + n * RN;
        const float* FZ = FX + PT;
        const float* FE = FZ + PT;  // edge taps: first column, last column, first row, last row
        if (ok) {
            int ib = ia_ib, k = ia_k;
            for (int it = tid; it < nz * nibt; it += T) {
                const int li = ib * CX;  // first column of this run, relative to the tile
                const float* vr = V + k * d.vp;
                float win[WZ];
                load_window_f4<P>(vr + li, win);
                float o[CX];
                fir<P, CX, 1, ZH - C>(FX, win, o);
                if (i0 + li == 0) o[0] = edge_dot_reg<C + 1, ZH>(FE, win);
                const int cl = last_col - li;  // position of column nx-1 in this run
                float* ur = U + li * d.kpu + ZH + k;
                if (cl >= CX) {
#pragma unroll
                    for (int c = 0; c < CX; ++c) ur[c * d.kpu] = o[c];
                } else {
                    const float e_last = edge_dot<C + 1>(FE + EC, vr, li + cl + ZH - C);
#pragma unroll
                    for (int c = 0; c < CX; ++c)
                        if (c <= cl) ur[c * d.kpu] = c == cl ? e_last : o[c];
                }
                ib += ia_dib;  // next item: it + T
                k += ia_dk;
                if (k >= nz) k -= nz, ++ib;
            }
        }
        __syncthreads();
        // the other buffer: the previous plane's store has had the whole i-adjoint to
        // read it; it now receives the next plane's attenuation
        if (d.nmb == 2 && tid == 0 && n + 1 < nj) {
            tma_store_wait_read<0>();
            request(n + 1);
        }
        float* mb = MB + (size_t)b * d.marea;
        ok = mbar_wait_bounded(bar + b, (unsigned)(d.nmb == 1 ? n : n >> 1) & 1u) && ok;
        if (ok) {
            int kb = ka_kb, i = ka_i;  // i relative to the tile
            for (int it = tid; it < ti * d.nkb; it += T) {
                const float* ur = U + i * d.kpu;
                const int k0 = kb * CZ;
                float win[WZ];
                load_window_f4<P>(ur + k0, win);
                float o[CZ];
                fir<P, CZ, 1, ZH - C>(FZ, win, o);
                if (nz > 1 && k0 == 0) o[0] = edge_dot_reg<C + 1, ZH>(FE + 2 * EC, win);
                const int cl = nz - 1 - k0;  // position of row nz-1 in this run
                if (nz > 1 && cl < CZ) {
                    const float e_last = edge_dot<C + 1>(FE + 3 * EC, ur, ZH + nz - 1 - C);
#pragma unroll
                    for (int c = 0; c < CZ; ++c)
                        if (c == cl) o[c] = e_last;
                }
                float4* m4 = reinterpret_cast<float4*>(mb + ((size_t)kb * d.TI + i) * 16);
                const int sw = (i >> 1) & 3;
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    float4 m = m4[q ^ sw];
                    m.x *= o[4 * q];
                    m.y *= o[4 * q + 1];
                    m.z *= o[4 * q + 2];
                    m.w *= o[4 * q + 3];
                    m4[q ^ sw] = m;
                }
                kb += ka_dkb;  // next item: it + T
                i += ka_di;
                if (i >= ti) i -= ti, ++kb;
            }
        }
        if (__syncthreads_or(!ok)) {
            if (tid == 0) {  // a last chance for the copies in flight
                flag_timeout(err);
                mbar_wait_bounded(bar + 2, 0u);
                for (int m = n; m < n + d.nmb && m < nj; ++m)
                    mbar_wait_bounded(bar + (d.nmb == 1 ? 0 : m & 1), (unsigned)(d.nmb == 1 ? m : m >> 1) & 1u);
                tma_store_wait_all();
            }
            return;
        }
        // t tile -> slab[v][j]
        if (tid == 0) {
            fence_proxy_async_smem();
            for (int q = 0; q < d.nkb; ++q)
                tma_store_3d(t_map, q * 16, i0, v * ny + j_begin + n, mb + q * d.TI * 16);
            tma_store_commit();
            if (d.nmb == 1 && n + 1 < nj) {  // the one buffer: the next plane's factors once the store has read it
                tma_store_wait_read<0>();
                request(n + 1);
            }
        }
    }
    if (tid == 0) tma_store_wait_read<0>();  // the writes complete with the grid
}

cudaError_t encode_v_map(const Geometry& g, const AdjDims& d, const float* v, CUtensorMap* map);

// ---------------------------------------------------------------- host-side dimensioning
namespace {
constexpr int kBuckets[] = {3, 5, 7, 9, 11, 13, 15, 17, 21, 25, 29, 33, 37};

template <int P>
FusedDims dims_for(const Geometry& g, int J, int tiles)
{
    using S = Sep<P>;
    FusedDims d;
    d.ps = g.nx * g.kp;
    d.ts = (5 * g.nx + 3) & ~3;
    d.nib = (g.nx + S::CX - 1) / S::CX;
    d.nkb = (g.nz + S::CZ - 1) / S::CZ;
    tiles = tiles < 1 ? 1 : (tiles > d.nib ? d.nib : tiles);
    d.TI = ((d.nib + tiles - 1) / tiles) * S::CX;
    d.nT = (g.nx + d.TI - 1) / d.TI;
    d.urows = d.TI < g.nx ? d.TI : g.nx;
    d.vrows = d.TI + 2 * S::C < g.nx ? d.TI + 2 * S::C : g.nx;
    d.marea = d.urows * g.kp;
    d.wp = pitch4odd(d.TI + 2 * S::C);
    d.warea = (g.nz * d.wp + 3) & ~3;
    d.farea = (g.nz * pitch4odd(d.nib * S::CX + 2 * S::C) + 3) & ~3;
    int kpu = d.nkb * S::CZ + 2 * S::ZH;
    kpu = (kpu + 3) & ~3;
    if (((kpu / 4) & 1) == 0) kpu += 4;
    d.kpu = kpu;
    int apc = d.nkb * S::CZ;
    if (((apc / 4) & 1) == 0) apc += 4;
    d.apc = apc;
    d.J = J;
    d.G = (g.ny + J - 1) / J;
    return d;
}

// Part of the bound of the geometries taken: a plane with its halos and a rotation table in shared memory.
inline size_t rot_smem_bound(const FusedDims& d) { return ((size_t)d.farea + d.ts) * sizeof(float); }

// Launch shape of the forward blur for `tiles` column tiles (the nearest count
// whose box fits the tensor map's 256 columns) and J planes per block.
//   threads: one per work item where the tile has at most 640 (the depth sums
//     then live in registers), so small planes run as small blocks, several
//     per SM, instead of one block of mostly idle warps;
//   tile buffers: two, or one when that lets more blocks run on an SM (the other
//     blocks then cover the load) or is all that fits.
constexpr size_t kSmSharedBytes = 233472;  // shared memory of an SM (1 KB of it per resident block)

inline int blocks_per_sm(size_t smem_bytes, int T, int regs)
{
    const int by_smem = (int)(kSmSharedBytes / (smem_bytes + 1024));
    const int by_regs = 65536 / (((T + 31) / 32) * 32 * regs);
    const int by_thr = 2048 / T;
    const int b = by_smem < by_regs ? by_smem : by_regs;
    return b < by_thr ? b : by_thr;
}

template <int P>
FwdDims fwd_dims(const Geometry& g, int J, int tiles, size_t smem_limit)
{
    using S = Sep<P>;
    FwdDims d;
    d.nib = (g.nx + S::CX - 1) / S::CX;
    d.nkb = (g.nz + S::CZ - 1) / S::CZ;
    tiles = tiles < 1 ? 1 : (tiles > d.nib ? d.nib : tiles);
    d.TI = ((d.nib + tiles - 1) / tiles) * S::CX;
    while (d.TI + 2 * S::C > 256) d.TI -= S::CX;
    d.nT = (g.nx + d.TI - 1) / d.TI;
    d.wr = d.TI + 2 * S::C;
    d.nbox = (g.nz + kWK - 1) / kWK;
    d.warea = d.nbox * d.wr * kWK;  // every box is a multiple of 128 bytes
    d.urows = d.TI < g.nx ? d.TI : g.nx;
    d.kpu = pitch4odd(d.nkb * S::CZ + 2 * S::ZH);
    d.apc = pitch4odd(d.nkb * S::CZ);
    d.J = J;
    d.G = (g.ny + J - 1) / J;
    const int kitems = d.urows * d.nkb, iitems = g.nz * ((d.urows + S::CX - 1) / S::CX);
    constexpr int kT = FwdBlock<P>::T;
    d.racc = kitems <= kT;
    const int want = kitems > iitems ? kitems : iitems;
    d.T = d.racc && want <= kT ? (want + 31) & ~31 : kT;
    d.nbuf = 2;
    const size_t two = fwd_smem_floats(d, S::PT) * sizeof(float);
    d.nbuf = 1;
    const size_t one = fwd_smem_floats(d, S::PT) * sizeof(float);
    const int b1 = blocks_per_sm(one, d.T, FwdBlock<P>::regs), b2 = blocks_per_sm(two, d.T, FwdBlock<P>::regs);
    if (two <= smem_limit && b2 >= 1 && (b1 <= b2 || b2 * d.T >= 768)) d.nbuf = 2;
    return d;
}

template <int P>
size_t smem_fwd(const FwdDims& d)
{
    return fwd_smem_floats(d, Sep<P>::PT) * sizeof(float);
}

// Launch shape of the blur adjoint for `tiles` column tiles (more where a tile would not
// fit) and J planes per block; threads as the forward blur.  Two attenuation
// buffers unless one lets more blocks run on an SM.
template <int P>
struct AdjBlock {
    static constexpr int T = FwdBlock<P>::T, B = FwdBlock<P>::B, regs = FwdBlock<P>::regs;
};

template <int P>
AdjDims adj_dims(const Geometry& g, int J, int tiles, size_t smem_limit)
{
    using S = Sep<P>;
    constexpr int kT = AdjBlock<P>::T, RN = AdjRec<P>::N;
    AdjDims d;
    const int nib = (g.nx + S::CX - 1) / S::CX;
    d.nkb = (g.nz + S::CZ - 1) / S::CZ;
    tiles = tiles < 1 ? 1 : (tiles > nib ? nib : tiles);
    d.TI = ((nib + tiles - 1) / tiles) * S::CX;
    while (pitch4odd(d.TI + 2 * S::ZH) > 252) d.TI -= S::CX;
    d.J = J;
    d.G = (g.ny + J - 1) / J;
    d.kpu = pitch4odd(d.nkb * S::CZ + 2 * S::ZH);
    for (;; d.TI -= S::CX) {
        d.nT = (g.nx + d.TI - 1) / d.TI;
        d.vp = pitch4odd(d.TI + 2 * S::ZH);
        // boxes of at most 256 rows; more than one start on 128 bytes (vp is 4 * odd: 8 rows are a multiple)
        d.vbox = (g.nz + 255) / 256;
        d.vrows = d.vbox == 1 ? g.nz : ((g.nz + d.vbox - 1) / d.vbox + 7) & ~7;
        d.varea = (d.vbox * d.vrows * d.vp + 31) & ~31;
        d.urows = d.TI < g.nx ? d.TI : g.nx;
        d.marea = d.nkb * d.TI * 16;
        const int kitems = d.urows * d.nkb, iitems = g.nz * ((d.urows + S::CX - 1) / S::CX);
        const int want = kitems > iitems ? kitems : iitems;
        d.T = want <= kT ? (want + 31) & ~31 : kT;
        d.nmb = 2;
        const size_t two = adj_smem_floats(d, RN) * sizeof(float);
        d.nmb = 1;
        const size_t one = adj_smem_floats(d, RN) * sizeof(float);
        const int b1 = blocks_per_sm(one, d.T, AdjBlock<P>::regs), b2 = blocks_per_sm(two, d.T, AdjBlock<P>::regs);
        if (two <= smem_limit && b2 >= 1 && (b1 <= b2 || b2 * d.T >= 768)) d.nmb = 2;
        if (one <= smem_limit || d.TI == S::CX) return d;
    }
}

template <int P>
size_t smem_adj(const AdjDims& d)
{
    return adj_smem_floats(d, AdjRec<P>::N) * sizeof(float);
}

// Part of the bound of the shapes taken: Zb, V, two attenuation tiles and the edge-class taps.
template <int P>
size_t smem_adj_bound(const Geometry& g, const FusedDims& d)
{
    return ((size_t)g.nz * d.wp + (size_t)d.vrows * d.kpu + 2 * (((size_t)d.urows * g.nz + 3) & ~(size_t)3) +
            6 * (size_t)Sep<P>::PT * d.J + 8) * sizeof(float);
}

// The geometries and shapes that the fused kernels take: two tile buffers, U,
// accumulators, taps and folds of a block in shared memory.  (The forward kernel needs
// less: its sums are in registers and one buffer may do.)
template <int P>
size_t smem_fwd_bound(const Geometry& g, const FusedDims& d)
{
    return (2 * (size_t)d.warea + (size_t)d.urows * d.kpu + 2 * (size_t)Sep<P>::PT * d.J + (size_t)d.urows * d.apc +
            2 * (size_t)d.J * d.nkb * 16 + 8) * sizeof(float);
}
}  // namespace

}  // namespace spect
