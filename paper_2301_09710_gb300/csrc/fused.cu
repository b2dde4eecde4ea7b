// fused.cu -- the default (fast) path of the projector on sm_103a.
//
// Same operator as the kernels in rotate.cu / conv.cu (Section II-A of
// arXiv 2301.09710, Algorithms 1 and 2), organised for GB300:
//
//  * Internal volumes use a k-fastest layout [j][i][k] ("transposed"): the
//    bilinear rotation weights depend on (i, j, view) only, so each of the four
//    neighbours of a rotated sample is a contiguous run of nz floats and every
//    rotation gather is a coalesced 128-byte access with lanes over k.
//  * The Eq. (1) attenuation factor mubar is computed once per plan for every
//    view, [l][j][i][k] (nview * nx*ny*nz floats; HBM is plentiful), so the hot
//    kernels multiply by a streamed, coalesced value instead of re-rotating mu.
//  * Forward: a rotation kernel rotates and attenuates every (view, depth)
//    plane into a plane image [i][k] of the work slab.  The blur kernel (one block
//    per view, group of J depth planes and 32-column tile) streams the tiles in
//    as tensor boxes, runs the separable PSF blur as two register-blocked
//    sliding-window passes (i, then k; replicate padding folded into edge
//    taps), and keeps the group's depth sum in registers; the groups' partials
//    are added in a fixed order by a small reduce kernel (deterministic, no atomics).
//  * Transpose: one block per (view, depth group, column tile) expands the detector
//    plane into blurred-adjoint planes times mubar (the t slab, [v][j][i][k]); a
//    gather kernel (gather.cu, k_adj_rot_t) then sums sum_l sum_p W_l(p;q) t_l(p,k) per destination voxel
//    q over fixed-length adjacency lists (weights bitwise those of A).
#include <algorithm>
#include <cmath>

#include "fused_body.cuh"

namespace spect {


// ============================================================================
// Plan-time kernels
// ============================================================================

// out[c][r] = in[r][c] for an R x C matrix (tiled through shared memory).
__global__ void k_transpose(const float* __restrict__ in, float* __restrict__ out, int R, int C, int ip, int op)
{
    wait_previous_kernel();
    transpose_body(in, out, R, C, ip, op, blockIdx.x, blockIdx.y);
}

cudaError_t launch_transpose(const float* in, float* out, int R, int C, int ip, int op, cudaStream_t st)
{
    dim3 grid((C + 31) / 32, (R + 31) / 32);
    return launch_chained(k_transpose, grid, dim3(32, 8), 0, st, in, out, R, C, ip, op);
}

// mubar[l][j][i][k] = exp(-dy (mu~(j)/2 + sum_{s>j} mu~(s))), Eq. (1), for every
// view.  A block owns 32 quads of k of a view's columns; its warps take runs of kMuRun
// depths from the detector side: each rotates its run into registers with the forward
// rotation's weights and sums it (compensated, AttenScan), the runs' sums are exchanged
// through shared memory, and each warp walks its run again from the sum of the runs
// before it.  mu_t is mu in the [j][i][k] layout; planes (l, j) are ps floats apart;
// view l lands at position v.
//   Bound by the latency of table entry and gather (four blocks per SM, two depths' loads
// in flight per thread; longer batches at fewer blocks: 96x64, 20 views of a pass 35 us
// against 41).  Against one thread walking a whole column: EM update with the factors
// recomputed, 160x96 in passes of 2 views 8.5 -> 5.3 ms, 128x80 in passes of 43 2.32 ->
// 2.29, 96x64 in passes of 20 0.522 -> 0.510.
constexpr int kMuBatch = 2, kMuWarps = 8;

__global__ void __launch_bounds__(32 * kMuWarps, 4) k_mubar_cache(Geometry g, int ps, int ts,
                                                                  const float* __restrict__ rtab,
                                                                  const float* __restrict__ mu_t,
                                                                  float* __restrict__ mubar, int l0)
{
    __shared__ float4 run[2][kMuWarps][2][32];  // sums, compensation terms
    wait_previous_kernel();
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int v = blockIdx.y, l = l0 + v, n = g.nx * g.kp, k4 = g.kp >> 2;
    const int e4 = min((int)blockIdx.x * 32 + lane, g.nx * k4 - 1), i = e4 / k4, k = 4 * (e4 - i * k4);
    const bool mine = (int)blockIdx.x * 32 + lane < g.nx * k4;
    const float* m = mu_t + k;
    const float* tab = rtab + (size_t)l * g.ny * ts;
    float* out = mubar + (size_t)v * g.ny * ps + 4 * (size_t)e4;
    AttenScan carry[4];
    int buf = 0;
    for (int top = g.ny - 1; top >= 0; top -= nw * kMuRun, buf ^= 1) {
        const int j0 = top - w * kMuRun;  // this warp's run: j0, j0 - 1, ...
        float mv[kMuRun][4] = {};
        AttenScan own[4];
        if (g.has_mu && j0 >= 0) {  // no branch below: a batch's loads go out together
#pragma unroll
            for (int h = 0; h < kMuRun; h += kMuBatch) {
                float4 t[kMuBatch];
                const float* b[kMuBatch];
#pragma unroll
                for (int q = 0; q < kMuBatch; ++q) {
                    const float* tj = tab + (size_t)max(j0 - h - q, 0) * ts;
                    t[q] = __ldg(reinterpret_cast<const float4*>(tj) + i);
                    b[q] = m + (size_t)__ldg(reinterpret_cast<const int*>(tj + 4 * g.nx) + i) * g.kp;
                }
#pragma unroll
                for (int q = 0; q < kMuBatch; ++q) {
                    const float4 c0 = __ldg(reinterpret_cast<const float4*>(b[q]));
                    const float4 c1 = __ldg(reinterpret_cast<const float4*>(b[q] + g.kp));
                    const float4 c2 = __ldg(reinterpret_cast<const float4*>(b[q] + n));
                    const float4 c3 = __ldg(reinterpret_cast<const float4*>(b[q] + n + g.kp));
                    const bool in = j0 - h - q >= 0;
                    mv[h + q][0] = in ? fmaf(t[q].w, c3.x, fmaf(t[q].z, c2.x, fmaf(t[q].y, c1.x, t[q].x * c0.x))) : 0.f;
                    mv[h + q][1] = in ? fmaf(t[q].w, c3.y, fmaf(t[q].z, c2.y, fmaf(t[q].y, c1.y, t[q].x * c0.y))) : 0.f;
                    mv[h + q][2] = in ? fmaf(t[q].w, c3.z, fmaf(t[q].z, c2.z, fmaf(t[q].y, c1.z, t[q].x * c0.z))) : 0.f;
                    mv[h + q][3] = in ? fmaf(t[q].w, c3.w, fmaf(t[q].z, c2.w, fmaf(t[q].y, c1.w, t[q].x * c0.w))) : 0.f;
                }
            }
        }
#pragma unroll
        for (int q = 0; q < kMuRun; ++q)
#pragma unroll
            for (int c = 0; c < 4; ++c) own[c].add(mv[q][c]);
        run[buf][w][0][lane] = make_float4(own[0].S, own[1].S, own[2].S, own[3].S);
        run[buf][w][1][lane] = make_float4(own[0].c, own[1].c, own[2].c, own[3].c);
        __syncthreads();  // the other buffer is rewritten only after the next one
        AttenScan sc[4];
        for (int u = 0; u < nw; ++u) {
            const float4 s4 = run[buf][u][0][lane], r4 = run[buf][u][1][lane];
            const float ss[4] = {s4.x, s4.y, s4.z, s4.w}, rr[4] = {r4.x, r4.y, r4.z, r4.w};
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                if (u == w) sc[c] = carry[c];
                carry[c].merge({ss[c], rr[c]});
            }
        }
        if (mine)
#pragma unroll
            for (int q = 0; q < kMuRun; ++q)
                if (j0 - q >= 0) {
                    float o[4];
#pragma unroll
                    for (int c = 0; c < 4; ++c) o[c] = k + c < g.nz ? sc[c].step(mv[q][c], g.dy) : 0.f;  // 0: padding
                    *reinterpret_cast<float4*>(out + (size_t)(j0 - q) * ps) = make_float4(o[0], o[1], o[2], o[3]);
                }
    }
}

namespace {
cudaError_t mubar_launch(const spect_plan_s& P, const float* mu_t, int l0, int nv, cudaStream_t st)
{
    const int warps = std::min(kMuWarps, (P.g.ny + kMuRun - 1) / kMuRun);
    const dim3 grid((P.g.nx * (P.g.kp / 4) + 31) / 32, nv);
    return launch_chained(k_mubar_cache, grid, 32 * warps, 0, st, P.g, P.ps, P.ts, rtab_for(P, l0), mu_t, P.mubar, l0);
}
}  // namespace

cudaError_t launch_mubar_cache(const spect_plan_s& P, const float* mu_t, cudaStream_t st)
{
    return mubar_launch(P, mu_t, 0, P.g.nview, st);
}

cudaError_t launch_mubar_range(const spect_plan_s& P, int l0, int nv, cudaStream_t st)
{
    if (!P.recompute || !P.mut || nv < 1 || (size_t)nv * P.g.ny * P.ps > P.mubar_cap) return cudaErrorInvalidValue;
    return mubar_launch(P, P.mut, l0, nv, st);
}

// Rotation tables of views l0 .. l0 + nv - 1, read by the rotation (k_rot_fwd,
// k_rot_patch) and the attenuation factors (k_mubar_cache): block (v, j) holds nx
// float4 weights, then nx int bases (ts floats, 16-byte aligned).
__global__ void k_rot_tables(Geometry g, int ts, const ViewRot* __restrict__ rot, int l0, int nv, float* __restrict__ tab)
{
    const size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (size_t)nv * g.ny * g.nx) return;
    const int i = (int)(idx % g.nx);
    const size_t lj = idx / g.nx;
    const int j = (int)(lj % g.ny), v = (int)(lj / g.ny);
    float4 w;
    int base;
    rot_table_entry(i, j, rot[l0 + v], g, w, base);
    float* blk = tab + lj * ts;
    reinterpret_cast<float4*>(blk)[i] = w;
    reinterpret_cast<int*>(blk + 4 * g.nx)[i] = base;
}

cudaError_t launch_rot_tables(const spect_plan_s& P, int l0, int nv, cudaStream_t st)
{
    const size_t n = (size_t)nv * P.g.ny * P.g.nx;
    k_rot_tables<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(P.g, P.ts, P.rot, l0, nv, P.rtab);
    return cudaGetLastError();
}

// Fixed-length adjacency lists for the transposed rotation: for destination
// q and view l, up to `maxe` (source column offset j*ps + i*kp, weight) pairs,
// zero-padded, laid out [q][l][e].  The candidate search and weights are those
// of k_build_adjacency (rotate.cu).
__global__ void k_build_adjacency_fixed(Geometry g, int ps, const ViewRot* __restrict__ rot, int maxe, AdjEntry* adj)
{
    const size_t nxy = (size_t)g.nx * g.ny;
    const size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= nxy * g.nview) return;
    const int l = (int)(idx / nxy);
    const int q = (int)(idx % nxy);
    const int qi = q % g.nx, qj = q / g.nx;
    const ViewRot r = rot[l];
    const float ct = r.ct_hi + r.ct_lo, st = r.st_hi + r.st_lo;
    const float c = (float)g.cint + g.cfrac;
    const float dqi = (float)qi - c, dqj = (float)qj - c;
    const float pi_ = c + ct * dqi - st * dqj;
    const float pj_ = c + st * dqi + ct * dqj;
    const int bi = (int)floorf(pi_) - 1, bj = (int)floorf(pj_) - 1;
    AdjEntry* out = adj + ((size_t)q * g.nview + l) * maxe;
    int cnt = 0;
    for (int cj = 0; cj < 4; ++cj)
        for (int ci = 0; ci < 4; ++ci) {
            const int pi = bi + ci, pj = bj + cj;
            if (pi < 0 || pi >= g.nx || pj < 0 || pj >= g.ny) continue;
            const Sample s = rot_sample(pi, pj, r, g.cint, g.cfrac);
            const int di = qi - s.i0, dj = qj - s.j0;
            if (di < 0 || di > 1 || dj < 0 || dj > 1) continue;
            const float w = bilinear_w(s, di, dj);
            if (w == 0.f || cnt >= maxe) continue;
            AdjEntry e;
            e.p = pj * ps + pi * g.kp;  // offset of the source column in a [j][i][k] slab with plane stride ps
            e.w = w;
            out[cnt++] = e;
        }
    for (; cnt < maxe; ++cnt) {
        AdjEntry e;
        e.p = 0;
        e.w = 0.f;
        out[cnt] = e;
    }
}

cudaError_t launch_build_adjacency_fixed(const spect_plan_s& P, int l0, int nv, cudaStream_t st)
{
    Geometry g = P.g;  // the lists of these views alone
    g.nview = nv;
    const size_t n = (size_t)g.nx * g.ny * nv;
    k_build_adjacency_fixed<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(g, P.ps, P.rot + l0, P.adj_max, P.adjf);
    return cudaGetLastError();
}

// Rotation + attenuation of every (view, plane) into the plane images: bilinear
// (TAPS = 4) or the three-pass rotation's eight-tap products (rot3.cu, TAPS = 8).
template <int TAPS>
__global__ void __launch_bounds__(kRotThreads, TAPS == 4 ? 5 : 3) k_rot_fwd(Geometry g, RotDims d,
                                                                            const float* __restrict__ tabs,
                                                                            const float* __restrict__ xt,
                                                                            const float* __restrict__ mubar,
                                                                            float* __restrict__ wsl, int l0)
{
    wait_previous_kernel();
    rot_body<TAPS>(g, d, tabs, xt, mubar, wsl, l0, blockIdx.x, blockIdx.y);
}

// ----------------------------------------------------------------------------
// Forward blur + depth sum: one block per (column tile, depth group of J planes,
// view), the tiles of a plane adjacent, so their overlapping boxes hit L2.
// ----------------------------------------------------------------------------
template <int P, bool RACC, bool KS>
__global__ void __launch_bounds__(FwdBlock<P>::T, KS ? 1 : FwdBlock<P>::B) k_fwd_sep_fused(const __grid_constant__ CUtensorMap tmap,
                                                                     Geometry g, FwdDims d,
                                                                     const float* __restrict__ rec,
                                                                     float* __restrict__ part, int l0, int* err)
{
    wait_previous_kernel();
    const int grp = blockIdx.x / d.nT;
    fwd_sep_body<P, RACC, KS>(g, d, &tmap, rec, part, l0, gridDim.y, err, grp, blockIdx.y, blockIdx.x - grp * d.nT);
}

// Plan time: the tap records of the forward blur (layout: fwd_rec_floats), one
// block per PSF plane; the folds are summed in FP64 and rounded once.
__global__ void k_fwd_records(Geometry g, int P, int PT, int nkb, const float* __restrict__ fx,
                              const float* __restrict__ fz, float* __restrict__ rec)
{
    const int row = blockIdx.x, C = (P - 1) / 2, ox = (P - g.px) / 2, oz = (P - g.pz) / 2;
    const float* f = fz + (size_t)row * g.pz;
    float* r = rec + (size_t)row * fwd_rec_floats(PT, nkb);
    for (int a = threadIdx.x; a < PT; a += blockDim.x) {
        r[a] = (a >= ox && a < ox + g.px) ? fx[(size_t)row * g.px + a - ox] : 0.f;
        r[PT + a] = (a >= oz && a < oz + g.pz) ? f[a - oz] : 0.f;
    }
    for (int k = threadIdx.x; k < 16 * nkb; k += blockDim.x) {
        double lo = 0.0, hi = 0.0;
        if (k < g.nz)
            for (int b = 0; b < g.pz; ++b) {
                if (b + oz > k + C) lo += f[b];
                if (b + oz < k + C - g.nz + 1) hi += f[b];
            }
        r[2 * PT + k] = (float)lo;
        r[2 * PT + 16 * nkb + k] = (float)hi;
    }
    const float* h = fx + (size_t)row * g.px;
    float* xf = r + 2 * PT + 32 * nkb;
    for (int e = threadIdx.x; e < kFoldLo + kFoldHi; e += blockDim.x) {
        const int i = e < kFoldLo ? e : fold_hi0(g.nx, C) + e - kFoldLo;
        double s = 0.0;
        if (i < g.nx)
            for (int a = 0; a < g.px; ++a)
                if (e < kFoldLo ? a + ox > i + C : a + ox < i + C - g.nx + 1) s += h[a];
        xf[e] = (float)s;
    }
}

// v(i,k,l) = sum over depth groups of the partials (fixed order) of the views of a pass
// (nproj values; comp: the partials' compensation terms, or NULL), optionally turned into
// the EM ratio y / (v + rbar), whose rows are np long.
__global__ void k_fwd_reduce(const float* __restrict__ part, const float* __restrict__ comp, int G, size_t nproj,
                             float* __restrict__ v, int nx, int np, const float* __restrict__ em_y,
                             const float* __restrict__ em_rbar)
{
    wait_previous_kernel();
    const size_t o = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (o >= nproj) return;
    const float s = group_sum(part + o, comp ? comp + o : nullptr, G, nproj);  // up to ny partials (J = 1): compensated
    if (em_y) {
        const float yb = s + (em_rbar ? em_rbar[o] : 0.f);
        v[np == nx ? o : o + o / nx * (np - nx)] = yb > 0.f ? em_y[o] / yb : 0.f;
    } else {
        v[o] = s;
    }
}

// out (rows of np) = v (n rows of nx)
__global__ void k_pad_rows(const float* __restrict__ v, float* __restrict__ out, size_t n, int nx, int np)
{
    wait_previous_kernel();
    const size_t o = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (o < n * nx) out[o + o / nx * (np - nx)] = v[o];
}

cudaError_t launch_pad_rows(const spect_plan_s& P, const float* v, float* out, cudaStream_t st)
{
    const size_t rows = (size_t)P.g.nz * P.g.nview, n = rows * P.g.nx;
    return launch_chained(k_pad_rows, (unsigned)((n + 255) / 256), 256, 0, st, v, out, rows, P.g.nx, P.g.np);
}

// Blur adjoint + attenuation: one block per (column tile, depth group of J planes, view).
template <int P>
__global__ void __launch_bounds__(AdjBlock<P>::T, AdjBlock<P>::B)
    k_adj_sep_fused(const __grid_constant__ CUtensorMap mu_map, const __grid_constant__ CUtensorMap t_map,
                    const __grid_constant__ CUtensorMap v_map, Geometry g, AdjDims d,
                    const float* __restrict__ rec, int l0, int mu_l0, int* err)
{
    wait_previous_kernel();
    const int grp = blockIdx.x / d.nT;
    adj_sep_body<P>(g, d, &mu_map, &t_map, &v_map, rec, l0, mu_l0, err, grp, blockIdx.y, blockIdx.x - grp * d.nT);
}

// Plan time: the tap records of the blur adjoint (layout: AdjRec), one block per PSF plane.
__global__ void k_adj_records(Geometry g, int P, int PT, int EC, int cls_z, const float* __restrict__ fx_adj,
                              const float* __restrict__ fz_adj, float* __restrict__ rec)
{
    const int row = blockIdx.x, nrow = gridDim.x, C = (P - 1) / 2, ox = (P - g.px) / 2, oz = (P - g.pz) / 2;
    float* r = rec + (size_t)row * (2 * PT + 4 * EC);
    auto tap = [&](const float* f, int cls, int p, int off, int a) {  // class cls, padded tap a
        return a >= off && a < off + p ? f[((size_t)cls * nrow + row) * p + a - off] : 0.f;
    };
    for (int a = threadIdx.x; a < PT; a += blockDim.x) {
        r[a] = tap(fx_adj, 0, g.px, ox, a);
        r[PT + a] = tap(fz_adj, 0, g.pz, oz, a);
    }
    for (int m = threadIdx.x; m < EC; m += blockDim.x) {
        float* e = r + 2 * PT + m;
        const bool in = m <= C;
        e[0] = in ? tap(fx_adj, 1, g.px, ox, C + m) : 0.f;
        e[EC] = in ? tap(fx_adj, 2, g.px, ox, m) : 0.f;
        e[2 * EC] = in && cls_z == 3 ? tap(fz_adj, 1, g.pz, oz, C + m) : 0.f;
        e[3 * EC] = in && cls_z == 3 ? tap(fz_adj, 2, g.pz, oz, m) : 0.f;
    }
}

// ============================================================================
// Fused blur for a full (non-separable) PSF p(a, b, j, l), padded tap count P.
// The 2D convolution of a plane is a sum over tap rows b of 1D FIRs along i
// (taps p(:, b)) applied to row k - b + cz: every term of a row runs through
// the register-blocked FIR of the separable kernels, and the rows add up per
// output (a row partial per b, then the sum over b: short FP32 chains).
//   forward: with the roles of the axes exchanged -- FIRs along k (taps p(a, :)) of
//     column i - a + cx, so lanes run over i and the windows are float4s along the
//     images' k.  Column tiles as in the separable path, W[C + i][ZH + k]; replicate
//     padding along i is a clamped column index, along k the blocks at the plane's
//     ends copy its first / last row into their halo; a thread owns 16 k of one
//     column and keeps their depth sums in registers.
//   adjoint: the same tiles and FIRs along k on the detector plane, staged once per
//     block, transposed and zero-padded (V[C + i][ZH + k]); a lane takes the tap rows
//     of its column's edge class, and the first / last detector row is summed apart
//     with the C + 1 taps of its class that are not zero.
// ============================================================================
// Launch shape of the forward full-PSF blur.
struct DirDims {
    int TI, nT;   // columns per tile, tiles per plane
    int KR, nkr;  // k per block (a multiple of 16), k ranges per plane
    int wr, wp;   // box: wr = TI + 2C columns of wp = pitch4odd(KR + 2ZH) <= 252 k
    int warea;    // floats of a tile buffer (rounded up to 128 bytes)
    int nbuf;     // tile buffers, each followed by the taps of its plane
    int J, G, T;  // planes per block, depth groups, threads (one per work item)
};

__host__ __device__ inline size_t dir_fwd_smem_floats(const DirDims& d, int P, int PT)
{
    return (size_t)d.nbuf * (d.warea + (((size_t)P * PT + 31) & ~(size_t)31)) + 8;  // + 2 mbarriers
}

// Launch shape of the full-PSF adjoint (TI, KR, wr, wp as the forward's).
struct DirAdjDims {
    int TI, nT, KR, nkr, wr, wp;
    int varea;    // floats of V (rounded up to 128 bytes)
    int marea;    // floats of the attenuation boxes, KR * TI
    int nslot;    // tap sets a block may need: interior, and first and / or last column
    int J, G, T;
};

// Adjoint tap set of one PSF plane and column class: P rows (a) along k of PT interior
// taps, then P rows of EC taps of the first and of the last detector row (the C + 1 that
// are not zero).
__host__ __device__ inline int dir_set_floats(int P, int PT, int EC) { return P * (PT + 2 * EC); }

__host__ __device__ inline size_t dir_adj_smem_floats(const DirAdjDims& d, int set)
{
    // MB | V | tap sets | 2 mbarriers
    return (size_t)d.marea + d.varea + (size_t)d.nslot * set + 8;
}

// Plan time: the taps of every PSF plane as rows along k, [a][b], zero-padded to
// P x PT and centred.
__global__ void k_dir_records(Geometry g, int P, int PT, const float* __restrict__ psf, float* __restrict__ rec)
{
    const size_t row = blockIdx.x;
    const int ox = (P - g.px) / 2, oz = (P - g.pz) / 2;
    for (int e = threadIdx.x; e < P * PT; e += blockDim.x) {
        const int a = e / PT - ox, b = e % PT - oz;
        rec[row * P * PT + e] =
            (a >= 0 && a < g.px && b >= 0 && b < g.pz) ? psf[row * g.px * g.pz + (size_t)b * g.px + a] : 0.f;
    }
}

// One block per (column tile, k range, depth group of J planes, view).
constexpr int kDirThreads = 384;  // 32 columns x 192 / 16 k runs

template <int P, bool KS>
__global__ void __launch_bounds__(kDirThreads, 1) k_fwd_dir_fused(const __grid_constant__ CUtensorMap tmap,
                                                                     Geometry g, DirDims d,
                                                                     const float* __restrict__ rec,
                                                                     float* __restrict__ part, int l0, int* err)
{
    using S = Sep<P>;
    constexpr int C = S::C, CZ = S::CZ, ZH = S::ZH, WZ = S::WZ, PT = S::PT;
    constexpr int TAPS = (P * PT + 31) & ~31;
    wait_previous_kernel();
    extern __shared__ __align__(128) float smf[];
    const int nx = g.nx, ny = g.ny, nz = g.nz;
    const int tid = threadIdx.x, T = blockDim.x;
    uint64_t* bar = reinterpret_cast<uint64_t*>(smf + (size_t)d.nbuf * (d.warea + TAPS));
    int bx = blockIdx.x;
    const int tile = bx % d.nT;
    bx /= d.nT;
    const int k_lo = (bx % d.nkr) * d.KR, grp = bx / d.nkr;
    const int v = blockIdx.y, l = l0 + v;
    const int i0 = tile * d.TI, ti = min(d.TI, nx - i0), nkb = (min(d.KR, nz - k_lo) + CZ - 1) / CZ;
    const int lp = g.nvp == 1 ? 0 : l;
    const int j_begin = grp * d.J, nj = min(ny - j_begin, d.J);
    const int ox = (P - g.px) / 2;  // tap columns outside [ox, ox + px) are zero
    const int pln = nx * nz;

    // tensor copies want 128-byte aligned shared memory: refuse (error word) rather than fault
    if ((smem_u32(smf) & 127u) != 0) {
        if (tid == 0 && err) atomicExch(err, (int)SPECT_ECUDA);
        return;
    }
    auto request = [&](int n) {  // plane j_begin + n and its taps into their buffer
        const int b = d.nbuf == 1 ? 0 : n & 1;
        float* dst = smf + (size_t)b * (d.warea + TAPS);
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar + b)),
                     "r"((unsigned)(d.wr * d.wp + P * PT) * 4u)
                     : "memory");
        tma_load_3d(dst, &tmap, k_lo - ZH, i0 - C, v * ny + j_begin + n, bar + b);
        tma_copy_1d(dst + d.warea, rec + ((size_t)lp * ny + j_begin + n) * (P * PT), (unsigned)(P * PT) * 4u, bar + b);
    };
    if (tid == 0) {
        mbar_init(bar, 1);
        mbar_init(bar + 1, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        for (int n = 0; n < d.nbuf && n < nj; ++n) request(n);
    }
    __syncthreads();

    const int kb = tid / ti, i = tid - kb * ti;  // the thread's item: 16 k of column i0 + i
    const bool mine = kb < nkb;
    const int kz = nz - 1 - k_lo + ZH;           // position of row nz - 1 in a column of W
    DepthSum<KS> acc[CZ];
    for (int n = 0; n < nj; ++n) {
        const int b = d.nbuf == 1 ? 0 : n & 1;
        float* W = smf + (size_t)b * (d.warea + TAPS);
        const float* TAP = W + d.warea;
        const bool ok = mbar_wait_bounded(bar + b, (unsigned)(d.nbuf == 1 ? n : n >> 1) & 1u);
        if (ok && k_lo < C)  // rows -C .. -1 that this block holds
            for (int r = tid; r < d.wr; r += T)
                for (int c = max(0, ZH - k_lo - C); c < ZH - k_lo; ++c) W[r * d.wp + c] = W[r * d.wp + ZH - k_lo];
        if (ok && kz < ZH + d.KR + C)  // rows nz .. nz + C - 1
            for (int r = tid; r < d.wr; r += T)
                for (int c = kz + 1; c <= min(kz + C, d.wp - 1); ++c) W[r * d.wp + c] = W[r * d.wp + kz];
        if (__syncthreads_or(!ok)) {
            if (tid == 0) {  // a last chance for the copies in flight to land
                flag_timeout(err);
                for (int m = n; m < n + d.nbuf && m < nj; ++m)
                    mbar_wait_bounded(bar + (d.nbuf == 1 ? 0 : m & 1), (unsigned)(d.nbuf == 1 ? m : m >> 1) & 1u);
            }
            return;
        }
        // c_j(i, k) = sum_a FIR_k(taps p(a, :), column clamp(i - a + cx)); lanes over i
        if (mine) {
            float o[CZ];
#pragma unroll
            for (int c = 0; c < CZ; ++c) o[c] = 0.f;
            for (int a = ox; a < ox + g.px; ++a) {
                const int col = clampi(i0 + i - a + C, 0, nx - 1) - i0 + C;
                float win[WZ];
                load_window_f4<P>(W + col * d.wp + kb * CZ, win);
                float ob[CZ];
                fir<P, CZ, -1, C + ZH>(TAP + a * PT, win, ob);
#pragma unroll
                for (int c = 0; c < CZ; ++c) o[c] += ob[c];
            }
#pragma unroll
            for (int c = 0; c < CZ; ++c) acc[c].add(o[c]);
        }
        __syncthreads();  // buffer b and its taps are free
        if (tid == 0 && n + d.nbuf < nj) {
            fence_proxy_async_smem();
            request(n + d.nbuf);
        }
    }
    if (mine) {
        const int k0 = k_lo + kb * CZ;
        float* pout = part + ((size_t)grp * gridDim.y + v) * pln + i0 + i;
        const size_t half = (size_t)d.G * gridDim.y * pln;
#pragma unroll
        for (int c = 0; c < CZ; ++c)
            if (k0 + c < nz) acc[c].store(pout + (size_t)(k0 + c) * nx, half);
    }
}

// Plan time: the adjoint's tap sets, [plane][column class 0..2][set], from the edge-class
// variants psf_adj[column class * cls_z + row class][plane][b][a].
__global__ void k_dir_adj_records(Geometry g, int P, int PT, int EC, int cls_z, const float* __restrict__ psf_adj,
                                  float* __restrict__ rec)
{
    const size_t row = blockIdx.x, nrow = gridDim.x, pp = (size_t)g.px * g.pz;
    const int ci = blockIdx.y, C = (P - 1) / 2, ox = (P - g.px) / 2, oz = (P - g.pz) / 2;
    const int set = dir_set_floats(P, PT, EC);
    float* r = rec + (row * 3 + ci) * set;
    for (int e = threadIdx.x; e < set; e += blockDim.x) {
        int a, b, ck;
        bool in = true;
        if (e < P * PT) {
            ck = 0, a = e / PT, b = e % PT;
        } else {
            const int f = e - P * PT, h = f % (P * EC), m = h % EC;
            ck = f < P * EC ? 1 : 2, a = h / EC;
            b = ck == 1 ? C + m : m;
            in = m <= C && cls_z == 3;
        }
        in = in && a >= ox && a < ox + g.px && b >= oz && b < oz + g.pz;
        r[e] = in ? psf_adj[((size_t)(ci * cls_z + ck) * nrow + row) * pp + (size_t)(b - oz) * g.px + a - ox] : 0.f;
    }
}

// One block per (column tile, k range, depth group of J planes, view).  The attenuation
// boxes and the tap sets have one buffer each: the factors are needed only after the
// plane's FIRs, the taps' wait is covered by the other blocks of the SM.
template <int P>
__global__ void __launch_bounds__(kDirThreads, 1)
    k_adj_dir_fused(const __grid_constant__ CUtensorMap mu_map, const __grid_constant__ CUtensorMap t_map, Geometry g,
                    DirAdjDims d, const float* __restrict__ vin, const float* __restrict__ rec, int l0, int mu_l0,
                    int* err)
{
    using S = Sep<P>;
    constexpr int C = S::C, CZ = S::CZ, ZH = S::ZH, WZ = S::WZ, PT = S::PT, EC = AdjRec<P>::EC;
    constexpr int SET = P * (PT + 2 * EC);
    wait_previous_kernel();
    extern __shared__ __align__(1024) float sma[];
    const int nx = g.nx, ny = g.ny, nz = g.nz;
    float* MB = sma;                                   // [KR / 16][TI][16], 64-byte swizzled
    float* V = MB + d.marea;                           // [wr][wp]
    float* TAP = V + d.varea;                          // [nslot][SET]
    uint64_t* bar = reinterpret_cast<uint64_t*>(TAP + (size_t)d.nslot * SET);  // factors, taps
    const int tid = threadIdx.x, T = blockDim.x;
    int bx = blockIdx.x;
    const int tile = bx % d.nT;
    bx /= d.nT;
    const int k_lo = (bx % d.nkr) * d.KR, grp = bx / d.nkr;
    const int v = blockIdx.y, l = l0 + v;
    const int i0 = tile * d.TI, ti = min(d.TI, nx - i0), nkb = (min(d.KR, nz - k_lo) + CZ - 1) / CZ;
    const int lp = g.nvp == 1 ? 0 : l;
    const int j_begin = grp * d.J, nj = min(ny - j_begin, d.J);
    const int ox = (P - g.px) / 2;  // tap rows outside [ox, ox + px) are zero
    const bool first_tile = tile == 0, last_tile = tile == d.nT - 1;

    // swizzled tensor copies want 512-byte aligned shared memory: refuse (error word) rather than fault
    if ((smem_u32(sma) & 511u) != 0) {
        if (tid == 0 && err) atomicExch(err, (int)SPECT_ECUDA);
        return;
    }
    auto request_mu = [&](int n) {
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)),
                     "r"((unsigned)(nkb * d.TI * 16) * 4u)
                     : "memory");
        for (int q = 0; q < nkb; ++q)
            tma_load_3d(MB + q * d.TI * 16, &mu_map, k_lo + q * 16, i0, (l - mu_l0) * ny + j_begin + n, bar);
    };
    auto request_taps = [&](int n) {  // the interior set, then those of the first / last column this tile holds
        const float* src = rec + ((size_t)lp * ny + j_begin + n) * 3 * SET;
        const int sets = 1 + first_tile + last_tile;
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar + 1)),
                     "r"((unsigned)(sets * SET) * 4u)
                     : "memory");
        tma_copy_1d(TAP, src, (unsigned)SET * 4u, bar + 1);
        if (first_tile) tma_copy_1d(TAP + SET, src + SET, (unsigned)SET * 4u, bar + 1);
        if (last_tile) tma_copy_1d(TAP + (1 + first_tile) * SET, src + 2 * SET, (unsigned)SET * 4u, bar + 1);
    };
    if (tid == 0) {
        mbar_init(bar, 1);
        mbar_init(bar + 1, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        request_taps(0);
        request_mu(0);
    }
    // the detector plane, transposed, zero outside the detector: lanes over columns
    for (int e = tid; e < d.wr * (d.KR + 2 * ZH); e += T) {
        const int r = e / d.wr, c = e - r * d.wr, k = k_lo - ZH + r, col = i0 - C + c;
        const bool in = k >= 0 && k < nz && col >= 0 && col < nx;
        cp_async_4_or_zero(V + c * d.wp + r, in ? vin + ((size_t)l * nz + k) * g.np + col : vin, in);
    }
    cp_async_wait_all();
    __syncthreads();

    const int kb = tid / ti, i = tid - kb * ti;  // the thread's item: 16 k of column i0 + i
    const bool mine = kb < nkb;
    const int k0 = k_lo + kb * CZ, cl = nz - 1 - k0;  // position of row nz - 1 in the item
    const bool top = mine && nz > 1 && k0 == 0, bottom = mine && nz > 1 && cl < CZ;
    const int slot = i0 + i == 0 ? 1 : (i0 + i == nx - 1 ? 1 + first_tile : 0);
    const float* TS = TAP + slot * SET;  // this column's tap set
    const float* TF = TS + P * PT;       // first row, last row
    const float* TL = TF + P * EC;
    for (int n = 0; n < nj; ++n) {
        bool ok = mbar_wait_bounded(bar + 1, (unsigned)n & 1u);
        float o[CZ], e_first = 0.f, e_last = 0.f;
        if (ok && mine) {
#pragma unroll
            for (int c = 0; c < CZ; ++c) o[c] = 0.f;
            for (int a = ox; a < ox + g.px; ++a) {
                const float* vc = V + (i + a) * d.wp;
                float win[WZ];
                load_window_f4<P>(vc + kb * CZ, win);
                float ob[CZ];
                fir<P, CZ, 1, ZH - C>(TS + a * PT, win, ob);
#pragma unroll
                for (int c = 0; c < CZ; ++c) o[c] += ob[c];
                if (top) e_first += edge_dot_reg<C + 1, ZH>(TF + a * EC, win);
                if (bottom) e_last += edge_dot<C + 1>(TL + a * EC, vc, ZH + nz - 1 - k_lo - C);
            }
            if (top) o[0] = e_first;
            if (bottom) {
#pragma unroll
                for (int c = 0; c < CZ; ++c)
                    if (c == cl) o[c] = e_last;
            }
        }
        ok = mbar_wait_bounded(bar, (unsigned)n & 1u) && ok;
        if (ok && mine) {
            float4* m4 = reinterpret_cast<float4*>(MB + ((size_t)kb * d.TI + i) * 16);
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
        }
        if (__syncthreads_or(!ok)) {
            if (tid == 0) {  // a last chance for the copies in flight
                flag_timeout(err);
                mbar_wait_bounded(bar, (unsigned)n & 1u);
                mbar_wait_bounded(bar + 1, (unsigned)n & 1u);
                tma_store_wait_all();
            }
            return;
        }
        if (tid == 0) {
            fence_proxy_async_smem();
            if (n + 1 < nj) request_taps(n + 1);
            for (int q = 0; q < nkb; ++q)
                tma_store_3d(&t_map, k_lo + q * 16, i0, v * ny + j_begin + n, MB + q * d.TI * 16);
            tma_store_commit();
            tma_store_wait_read<0>();
            if (n + 1 < nj) request_mu(n + 1);
        }
    }
}

// x_t(q,k) (+)= sum_{v in chunk} sum_{e < MAXE} w_e t[v][p_e][k]
// with the EM update (em_update) on the last chunk when em.x is set.  The
// lists are laid out [q][l][e] so one destination's entries for all views are
// contiguous; each entry holds the premultiplied offset p*kp of its source
// column in the slab.  A thread owns four consecutive k of one destination (float4
// loads).  Per view the few terms are summed plainly, the views with Kahan compensation.
template <int MAXE>
__global__ void __launch_bounds__(256) k_adj_rot_t(Geometry g, int ps, const AdjEntry* __restrict__ adj,
                                                   const float* __restrict__ slab, int l0, int nv, float* out,
                                                   PassState ps_, int seglen, EmArgs em)
{
    using VT = float4;
    constexpr int VEC = 4;
    wait_previous_kernel();
    const int nxy = g.nx * g.ny;
    const int nzv = g.kp / VEC;
    const int idx = blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= nxy * nzv) return;
    const int qq = idx / nzv;
    const int k = (idx - qq * nzv) * VEC;
    // destinations in strips 4 wide in i running along j: a block covers a
    // compact patch, so the ~4 reads of each source column mostly hit L1
    int q = qq;
    if ((g.nx & 3) == 0) {
        const int strip = qq / (4 * g.ny), r = qq - strip * 4 * g.ny;
        q = (4 * strip + (r & 3)) + g.nx * (r >> 2);
    }
    const AdjEntry* e = adj + ((size_t)q * g.nview + l0) * MAXE;
    const float* t = slab + k;
    const size_t vstride = (size_t)g.ny * ps;
    const size_t o = (size_t)q * g.kp + k;
    KSum acc[VEC];
    if (ps_.resume)  // the sums of the views of earlier launches
#pragma unroll
        for (int u = 0; u < VEC; ++u) acc[u].s = ps_.acc[o + u], acc[u].c = ps_.acc_c[o + u];
    // four views per step: all entry loads, then all slab loads, are issued
    // before any is used, so the chain of dependent loads is 4x shorter
    constexpr int UV = 4;
    KSum tot[VEC];
    for (int v_end = min(nv, seglen), v = 0; v < nv; v_end = min(nv, v_end + seglen)) {
    for (; v + UV <= v_end; v += UV) {
        AdjEntry a[UV][MAXE];
#pragma unroll
        for (int w = 0; w < UV; ++w)
#pragma unroll
            for (int m = 0; m < MAXE; ++m) a[w][m] = e[w * MAXE + m];
        VT tv[UV][MAXE];
#pragma unroll
        for (int w = 0; w < UV; ++w)
#pragma unroll
            for (int m = 0; m < MAXE; ++m) tv[w][m] = *reinterpret_cast<const VT*>(t + w * vstride + a[w][m].p);
#pragma unroll
        for (int w = 0; w < UV; ++w) {
            float sv[VEC];
#pragma unroll
            for (int u = 0; u < VEC; ++u) sv[u] = 0.f;
#pragma unroll
            for (int m = 0; m < MAXE; ++m) {
                const float* tf = reinterpret_cast<const float*>(&tv[w][m]);
#pragma unroll
                for (int u = 0; u < VEC; ++u) sv[u] = fmaf(a[w][m].w, tf[u], sv[u]);
            }
#pragma unroll
            for (int u = 0; u < VEC; ++u) acc[u].add(sv[u]);
        }
        e += UV * MAXE;
        t += UV * vstride;
    }
    for (; v < v_end; ++v) {
        AdjEntry a[MAXE];
#pragma unroll
        for (int m = 0; m < MAXE; ++m) a[m] = e[m];
        VT tv[MAXE];
#pragma unroll
        for (int m = 0; m < MAXE; ++m) tv[m] = *reinterpret_cast<const VT*>(t + a[m].p);
        float sv[VEC];
#pragma unroll
        for (int u = 0; u < VEC; ++u) sv[u] = 0.f;
#pragma unroll
        for (int m = 0; m < MAXE; ++m) {
            const float* tf = reinterpret_cast<const float*>(&tv[m]);
#pragma unroll
            for (int u = 0; u < VEC; ++u) sv[u] = fmaf(a[m].w, tf[u], sv[u]);
        }
#pragma unroll
        for (int u = 0; u < VEC; ++u) acc[u].add(sv[u]);
        e += MAXE;
        t += vstride;
    }
    if (seglen < nv) {  // the segments of the patch gather, added in order
#pragma unroll
        for (int u = 0; u < VEC; ++u) tot[u].merge(acc[u].s, acc[u].c), acc[u] = KSum();
    }
    }
    if (seglen < nv)
#pragma unroll
        for (int u = 0; u < VEC; ++u) acc[u] = tot[u];
#pragma unroll
    for (int u = 0; u < VEC; ++u) {
        if (ps_.merge) {  // add this segment to the ones before it
            KSum t;
            if (ps_.tot_resume) t.s = out[o + u], t.c = ps_.tot_c[o + u];
            t.merge(acc[u].s, acc[u].c);
            acc[u] = t;
        }
        if (ps_.more || (ps_.merge && ps_.tot_more)) {
            (ps_.more ? ps_.acc : out)[o + u] = acc[u].s;
            (ps_.more ? ps_.acc_c : ps_.tot_c)[o + u] = acc[u].c;
            continue;
        }
        const float val = acc[u].value();
        if (em.x) em.x[o + u] = em_update(em.x[o + u], val, em.s[o + u], em.u ? em.u[o + u] : 0.f, em.beta);
        else out[o + u] = val;
    }
}

namespace {
cudaError_t encode_3d(CUtensorMap* map, const float* base, const cuuint64_t (&dims)[3], const cuuint64_t (&strides)[2],
                      cuuint32_t b0, cuuint32_t b1, CUtensorMapSwizzle swizzle)
{
    const cuuint32_t box[3] = {b0, b1, 1};
    const cuuint32_t estr[3] = {1, 1, 1};
    if (!encode_fn() ||
        encode_fn()(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, const_cast<float*>(base), dims, strides, box, estr,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
        return cudaErrorInvalidValue;
    return cudaSuccess;
}

}  // namespace

// Projections v (rows of np) as a tensor map, boxed as the blur adjoint stages them.
cudaError_t encode_v_map(const Geometry& g, const AdjDims& d, const float* v, CUtensorMap* map)
{
    const cuuint64_t dims[3] = {(cuuint64_t)g.nx, (cuuint64_t)g.nz, (cuuint64_t)g.nview};
    const cuuint64_t strides[2] = {(cuuint64_t)g.np * 4, (cuuint64_t)g.np * g.nz * 4};
    return encode_3d(map, v, dims, strides, d.vp, d.vrows, CU_TENSOR_MAP_SWIZZLE_NONE);
}

// ============================================================================
// host side: dimensioning and launchers
// ============================================================================
namespace {
// The fewest column tiles with which the bounds of the geometries taken fit `limit`
// bytes of shared memory; 0 when none does.
template <int P>
int tiles_that_fit(const Geometry& g, size_t limit, int min_tiles)
{
    const int nib = (g.nx + Sep<P>::CX - 1) / Sep<P>::CX;
    int last_nt = 0;
    for (int t = min_tiles < 1 ? 1 : min_tiles; t <= nib; ++t) {
        const FusedDims d = dims_for<P>(g, 8, t);
        if (d.nT == last_nt) continue;  // same tile width as a smaller request
        last_nt = d.nT;
        if (smem_fwd_bound<P>(g, d) <= limit && smem_adj_bound<P>(g, d) <= limit && rot_smem_bound(d) <= limit &&
            (size_t)d.marea * 4 < (1u << 20))
            return d.nT;
    }
    return 0;
}

template <int P>
cudaError_t fwd_launch(const spect_plan_s& Pl, int l0, int nv, cudaStream_t st)
{
    const FwdDims d = fwd_dims<P>(Pl.g, Pl.fused_J, Pl.fwd_nT, (size_t)Pl.smem_optin);
    const size_t smem = smem_fwd<P>(d);
    auto kern = !d.racc ? k_fwd_sep_fused<P, false, false>
                        : (Pl.low ? k_fwd_sep_fused<P, true, true> : k_fwd_sep_fused<P, true, false>);
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    return launch_chained(kern, dim3(d.G * d.nT, nv), d.T, smem, st, Pl.fmap, Pl.g, d, Pl.frec, Pl.part, l0, Pl.err);
}

template <int P>
cudaError_t adj_launch(const spect_plan_s& Pl, const float* v, int l0, int nv, cudaStream_t st)
{
    const AdjDims d = adj_dims<P>(Pl.g, Pl.adj_J, Pl.adj_nT, (size_t)Pl.smem_optin);
    const size_t smem = smem_adj<P>(d);
    CUtensorMap vmap{};
    cudaError_t e = encode_v_map(Pl.g, d, v, &vmap);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(k_adj_sep_fused<P>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    // a recomputing plan's factors are those of views l0 .. at chunk-relative positions
    return launch_chained(k_adj_sep_fused<P>, dim3(d.G * d.nT, nv), d.T, smem, st, Pl.amap_mu, Pl.amap_t, vmap, Pl.g, d,
                          Pl.arec, l0, Pl.recompute ? l0 : 0, Pl.err);
}
}  // namespace

namespace {
// The bound of the full-PSF geometries taken, forward: two whole planes with halo
// rows, accumulators and taps; adjoint: one plane, two attenuation planes and the taps
// of every edge class (the kernels' tiles need less).
template <int P>
size_t dir_smem_fwd_bound(const Geometry& g, const FusedDims& d)
{
    const size_t xarea = ((size_t)(g.nz + 2 * Sep<P>::ZH) * d.wp + 3) & ~(size_t)3;
    return (2 * xarea + (size_t)P * Sep<P>::PT + (size_t)d.urows * d.apc + 8) * sizeof(float);
}

template <int P>
size_t dir_smem_adj_bound(const Geometry& g, const FusedDims& d, int cls_z)
{
    const size_t xarea = ((size_t)(g.nz + 2 * Sep<P>::ZH) * d.wp + 3) & ~(size_t)3;
    const size_t marea = ((size_t)d.urows * g.nz + 3) & ~(size_t)3;
    return (xarea + 2 * marea + 3 * (size_t)cls_z * P * Sep<P>::PT + 8) * sizeof(float);
}

// Forward launch shape: 32-column tiles, at most 192 k per block (the tensor map's
// 256 with the halos), a thread per work item, as the separable blur.  Two buffers
// unless one lets more blocks run on an SM.
template <int P>
DirDims dir_fwd_dims(const Geometry& g, int J, size_t smem_limit)
{
    using S = Sep<P>;
    DirDims d;
    d.TI = g.nx > 16 ? 32 : 16;
    d.nT = (g.nx + d.TI - 1) / d.TI;
    d.nkr = (g.nz + 191) / 192;
    d.KR = ((g.nz + d.nkr - 1) / d.nkr + 15) & ~15;
    d.nkr = (g.nz + d.KR - 1) / d.KR;
    d.wr = d.TI + 2 * S::C;
    d.wp = pitch4odd(d.KR + 2 * S::ZH);
    d.warea = (d.wr * d.wp + 31) & ~31;
    d.J = J;
    d.G = (g.ny + J - 1) / J;
    d.T = (std::min(d.TI, g.nx) * (d.KR / 16) + 31) & ~31;
    d.nbuf = 2;
    const size_t two = dir_fwd_smem_floats(d, P, S::PT) * sizeof(float);
    d.nbuf = 1;
    const size_t one = dir_fwd_smem_floats(d, P, S::PT) * sizeof(float);
    if (two <= smem_limit && blocks_per_sm(one, d.T, 96) <= blocks_per_sm(two, d.T, 96)) d.nbuf = 2;
    return d;
}

template <int P>
DirAdjDims dir_adj_dims(const Geometry& g, int J)
{
    const DirDims f = dir_fwd_dims<P>(g, J, 0);  // the forward's tiles
    DirAdjDims d;
    d.TI = f.TI, d.nT = f.nT, d.KR = f.KR, d.nkr = f.nkr, d.wr = f.wr, d.wp = f.wp;
    d.varea = f.warea;
    d.marea = d.KR * d.TI;
    d.nslot = d.nT == 1 ? 3 : 2;
    d.J = J, d.G = f.G, d.T = f.T;
    return d;
}

template <int P>
size_t dir_smem_adj(const DirAdjDims& d)
{
    return dir_adj_smem_floats(d, dir_set_floats(P, Sep<P>::PT, AdjRec<P>::EC)) * sizeof(float);
}

template <int P>
bool dir_fits(const Geometry& g, size_t limit, int J, int adj_J)
{
    const int cls_z = g.nz >= 2 ? 3 : 1;
    const FusedDims df = dims_for<P>(g, J, 1), da = dims_for<P>(g, adj_J, 1);
    return df.nT == 1 && dir_smem_fwd_bound<P>(g, df) <= limit && dir_smem_adj_bound<P>(g, da, cls_z) <= limit &&
           rot_smem_bound(df) <= limit && (size_t)df.ps * 4 < (1u << 20);
}

template <int P>
cudaError_t dir_fwd_launch(const spect_plan_s& Pl, int l0, int nv, cudaStream_t st)
{
    const DirDims d = dir_fwd_dims<P>(Pl.g, Pl.fused_J, (size_t)Pl.smem_optin);
    const size_t smem = dir_fwd_smem_floats(d, P, Sep<P>::PT) * sizeof(float);
    auto kern = Pl.low ? k_fwd_dir_fused<P, true> : k_fwd_dir_fused<P, false>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    return launch_chained(kern, dim3(d.nT * d.nkr * d.G, nv), d.T, smem, st, Pl.fmap, Pl.g, d, Pl.frec, Pl.part, l0,
                          Pl.err);
}

template <int P>
cudaError_t dir_adj_launch(const spect_plan_s& Pl, const float* v, int l0, int nv, cudaStream_t st)
{
    const DirAdjDims d = dir_adj_dims<P>(Pl.g, Pl.adj_J);
    const size_t smem = dir_smem_adj<P>(d);
    cudaError_t e = cudaFuncSetAttribute(k_adj_dir_fused<P>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    return launch_chained(k_adj_dir_fused<P>, dim3(d.nT * d.nkr * d.G, nv), d.T, smem, st, Pl.amap_mu, Pl.amap_t, Pl.g, d,
                          v, Pl.arec, l0, Pl.recompute ? l0 : 0, Pl.err);
}
}  // namespace

// Bucket of the fused full-PSF kernels (untiled planes only), 0 when they do not fit.
int fused_dir_bucket(const Geometry& g, size_t smem_limit)
{
    const int p = g.px > g.pz ? g.px : g.pz;
    for (int b : kBuckets) {
        if (b < p) continue;
        bool ok = false;
        switch (b) {
#define SPECT_DF(B) \
    case B: ok = dir_fits<B>(g, smem_limit, 8, 8); break;
            SPECT_DF(3) SPECT_DF(5) SPECT_DF(7) SPECT_DF(9) SPECT_DF(11) SPECT_DF(13) SPECT_DF(15)
            SPECT_DF(17) SPECT_DF(21) SPECT_DF(25) SPECT_DF(29) SPECT_DF(33) SPECT_DF(37)
#undef SPECT_DF
            default: break;
        }
        return ok ? b : 0;
    }
    return 0;
}

int fused_bucket(const Geometry& g, size_t smem_limit, int* tiles)
{
    const int p = g.px > g.pz ? g.px : g.pz;
    *tiles = 0;
    // SPECT_FUSED_TILES: at least this many column tiles (testing and tuning;
    // results are bitwise those of the untiled kernels)
    const char* env = getenv("SPECT_FUSED_TILES");
    const int min_tiles = env ? atoi(env) : 1;
    for (int b : kBuckets) {
        if (b < p) continue;
        int nt = 0;
        switch (b) {
#define SPECT_FITS(B) \
    case B: nt = tiles_that_fit<B>(g, smem_limit, min_tiles); break;
            SPECT_FITS(3) SPECT_FITS(5) SPECT_FITS(7) SPECT_FITS(9) SPECT_FITS(11) SPECT_FITS(13) SPECT_FITS(15)
            SPECT_FITS(17) SPECT_FITS(21) SPECT_FITS(25) SPECT_FITS(29) SPECT_FITS(33) SPECT_FITS(37)
#undef SPECT_FITS
            default: break;
        }
        *tiles = nt;
        return nt > 0 ? b : 0;
    }
    return 0;
}

// Column-tile count the fused kernels use when asked for `tiles` tiles with
// depth groups of J (forward) and adj_J (adjoint) planes, or 0 when that
// configuration does not fit `smem_limit` bytes of shared memory.
int fused_tiles_fit(const Geometry& g, int bucket, int J, int adj_J, int tiles, size_t smem_limit)
{
    auto check = [&](auto tag) -> int {
        constexpr int B = decltype(tag)::value;
        const FusedDims df = dims_for<B>(g, J, tiles), da = dims_for<B>(g, adj_J, tiles);
        const bool ok = smem_fwd_bound<B>(g, df) <= smem_limit && smem_adj_bound<B>(g, da) <= smem_limit &&
                        rot_smem_bound(df) <= smem_limit && (size_t)df.marea * 4 < (1u << 20);
        return ok ? df.nT : 0;
    };
    switch (bucket) {
#define SPECT_TF(B) \
    case B: return check(std::integral_constant<int, B>());
        SPECT_TF(3) SPECT_TF(5) SPECT_TF(7) SPECT_TF(9) SPECT_TF(11) SPECT_TF(13) SPECT_TF(15)
        SPECT_TF(17) SPECT_TF(21) SPECT_TF(25) SPECT_TF(29) SPECT_TF(33) SPECT_TF(37)
#undef SPECT_TF
        default: return 0;
    }
}

// Whether the fused full-PSF kernels fit with depth groups J / adj_J.
bool fused_dir_fit(const Geometry& g, int bucket, int J, int adj_J, size_t smem_limit)
{
    switch (bucket) {
#define SPECT_DF(B) \
    case B: return dir_fits<B>(g, smem_limit, J, adj_J);
        SPECT_DF(3) SPECT_DF(5) SPECT_DF(7) SPECT_DF(9) SPECT_DF(11) SPECT_DF(13) SPECT_DF(15)
        SPECT_DF(17) SPECT_DF(21) SPECT_DF(25) SPECT_DF(29) SPECT_DF(33) SPECT_DF(37)
#undef SPECT_DF
        default: return false;
    }
}

int fused_groups(const spect_plan_s& P) { return (P.g.ny + P.fused_J - 1) / P.fused_J; }

#define SPECT_DISPATCH(FN, ...)                        \
    switch (P.bucket) {                                \
        case 3: return FN<3>(__VA_ARGS__);             \
        case 5: return FN<5>(__VA_ARGS__);             \
        case 7: return FN<7>(__VA_ARGS__);             \
        case 9: return FN<9>(__VA_ARGS__);             \
        case 11: return FN<11>(__VA_ARGS__);           \
        case 13: return FN<13>(__VA_ARGS__);           \
        case 15: return FN<15>(__VA_ARGS__);           \
        case 17: return FN<17>(__VA_ARGS__);           \
        case 21: return FN<21>(__VA_ARGS__);           \
        case 25: return FN<25>(__VA_ARGS__);           \
        case 29: return FN<29>(__VA_ARGS__);           \
        case 33: return FN<33>(__VA_ARGS__);           \
        case 37: return FN<37>(__VA_ARGS__);           \
        default: return cudaErrorInvalidValue;         \
    }

cudaError_t launch_fused_forward(const spect_plan_s& P, int l0, int nv, cudaStream_t st)
{
    if (!P.separable) {
        SPECT_DISPATCH(dir_fwd_launch, P, l0, nv, st)
    }
    SPECT_DISPATCH(fwd_launch, P, l0, nv, st)
}

cudaError_t launch_fused_rotate(const spect_plan_s& P, const float* xt, int l0, int nv, cudaStream_t st)
{
    // read from the plan's own x_t: the patch-staged rotation (rotpatch.cu)
    if (P.rotpatch && P.rotpatch_on && xt == P.xt) return launch_rot_patch(P, l0, nv, st);
    const RotDims d = rot_dims(P.g, P.ps, P.rot3 ? rot3_ts8(P.g.nx) : P.ts, nv, P.sms);
    const dim3 grid(d.nb * ((P.g.ny + d.JP - 1) / d.JP), nv);
    return launch_chained(P.rot3 ? k_rot_fwd<8> : k_rot_fwd<4>, grid, kRotThreads, 0, st, P.g, d,
                          P.rot3 ? P.r3_tab : rtab_for(P, l0), xt, mubar_for(P, l0), P.slab, l0);
}

namespace {
// The planes of the work slab and of the attenuation factors as tensor maps -- k x column
// (nx) x plane -- with the blur kernels' tiles as boxes.  The images end at k = nz
// (zeros beyond); t and the factors at kp.
template <int P>
cudaError_t encode_maps(spect_plan_s& Pl)
{
    const Geometry& g = Pl.g;
    const cuuint64_t strides[2] = {(cuuint64_t)g.kp * 4, (cuuint64_t)Pl.ps * 4};
    const cuuint64_t planes = (cuuint64_t)Pl.chunk * g.ny;
    const cuuint64_t img[3] = {(cuuint64_t)g.nz, (cuuint64_t)g.nx, planes};
    cuuint32_t f0 = kWK, f1, at;
    if (Pl.separable) {
        f1 = fwd_dims<P>(g, Pl.fused_J, Pl.fwd_nT, (size_t)Pl.smem_optin).wr;
        at = adj_dims<P>(g, Pl.adj_J, Pl.adj_nT, (size_t)Pl.smem_optin).TI;
    } else {
        const DirDims d = dir_fwd_dims<P>(g, Pl.fused_J, (size_t)Pl.smem_optin);
        f0 = d.wp, f1 = d.wr, at = d.TI;
    }
    const cuuint64_t t[3] = {(cuuint64_t)g.kp, (cuuint64_t)g.nx, planes};
    const cuuint64_t mu[3] = {(cuuint64_t)g.kp, (cuuint64_t)g.nx, Pl.recompute ? planes : (cuuint64_t)g.nview * g.ny};
    cudaError_t e = encode_3d(&Pl.fmap, Pl.slab, img, strides, f0, f1, CU_TENSOR_MAP_SWIZZLE_NONE);
    if (e == cudaSuccess) e = encode_3d(&Pl.amap_t, Pl.slab, t, strides, 16, at, CU_TENSOR_MAP_SWIZZLE_64B);
    if (e == cudaSuccess) e = encode_3d(&Pl.amap_mu, Pl.mubar, mu, strides, 16, at, CU_TENSOR_MAP_SWIZZLE_64B);
    return e;
}
}  // namespace

// Floats of the forward blur's tap records of a plan.
size_t fwd_records_floats(const spect_plan_s& P)
{
    const int PT = (P.bucket + 3) & ~3, nkb = (P.g.nz + 15) / 16;
    return (size_t)P.g.nvp * P.g.ny * (P.separable ? fwd_rec_floats(PT, nkb) : P.bucket * PT);
}

namespace {
int rec_edge(int P) { return ((P - 1) / 2 + 4) & ~3; }  // AdjRec::EC
}  // namespace

// Floats of the blur adjoint's tap records of a plan.
size_t adj_records_floats(const spect_plan_s& P)
{
    const int PT = (P.bucket + 3) & ~3, EC = rec_edge(P.bucket);
    return (size_t)P.g.nvp * P.g.ny * (P.separable ? 2 * PT + 4 * EC : 3 * dir_set_floats(P.bucket, PT, EC));
}

cudaError_t launch_records(const spect_plan_s& P, cudaStream_t st)
{
    const int PT = (P.bucket + 3) & ~3, nkb = (P.g.nz + 15) / 16, rows = P.g.nvp * P.g.ny;
    if (P.separable) {
        k_fwd_records<<<rows, 128, 0, st>>>(P.g, P.bucket, PT, nkb, P.fx, P.fz, P.frec);
        k_adj_records<<<rows, 64, 0, st>>>(P.g, P.bucket, PT, rec_edge(P.bucket), P.cls_z, P.fx_adj, P.fz_adj, P.arec);
    } else {
        k_dir_records<<<rows, 256, 0, st>>>(P.g, P.bucket, PT, P.psf, P.frec);
        k_dir_adj_records<<<dim3(rows, 3), 256, 0, st>>>(P.g, P.bucket, PT, rec_edge(P.bucket), P.cls_z, P.psf_adj,
                                                         P.arec);
    }
    return cudaGetLastError();
}

cudaError_t build_maps(spect_plan_s& P)
{
    SPECT_DISPATCH(encode_maps, P)
}

namespace {
// Estimated time (us) of a separable blur launch: `blocks` blocks of J planes and T
// threads, B of them resident per SM.  Resident warps W share the issue slots, with
// about four warps' worth lost to latency, so a plane takes W + 4 warp items of
// 32 P + 100 issue slots; a block's set-up costs about s planes; up to four waves the
// last one counts whole, beyond that half a block on average.  Against the measured
// calls (shapes of 16..64 columns and J = 1..8; 16x8, 20x20, 24x60, 37x100, 48x24, 64x32,
// 64x64, 64x80, 96x64, 96x96, 99x53, 113x20, 128x32, 128x64, 128x80, 150x75, 160x48, 160x96,
// 192x128 with 8 to 128 views and 5 to 37 taps) the shapes it picks are within 5 % of the fastest.
double blur_cost(int P, long long blocks, int J, double s, int T, int B, int sms)
{
    const double per_sm = (double)((blocks + sms - 1) / sms);
    const double res = std::min<double>(B, per_sm);
    const double w = (double)blocks / (res * sms);
    const double waves = w <= 4.0 ? std::max(1.0, std::ceil(w - 1e-9)) : w + 0.5;
    return waves * (J + s) * (res * T / 32.0 + 4.0) * (32.0 * P + 100.0) / 4.0 / 1.92e3;
}

template <int P>
void choose_shape(spect_plan_s& Pl)
{
    const Geometry& g = Pl.g;
    const size_t limit = (size_t)Pl.smem_optin;
    const int nib = (g.nx + 15) / 16, nv = Pl.shape_views;
    // J decides how A's depth sum is grouped: the same whatever the passes (a recomputing
    // plan's results are bitwise the caching plan's), except for low-memory plans
    const int keep_J = nv < g.nview && !Pl.low ? Pl.fused_J : 0;
    double fbest = 1e30, abest = 1e30;
    for (int ti : {32, 48, 64, 16}) {  // 32 columns unless another width is clearly better
        const int tiles = (nib + ti / 16 - 1) / (ti / 16);
        for (int J : {8, 4, 6, 7, 5, 3, 2, 1}) {  // longer plain depth sums would cost accuracy
            if (J > g.ny) continue;
            const FwdDims f = fwd_dims<P>(g, J, std::max(tiles, Pl.min_nT), limit);
            // sums in shared memory are plain: one plane per block where they are to be compensated
            const bool sums = f.racc || (ti == 16 && (!Pl.low || J == 1));
            if (smem_fwd<P>(f) <= limit && sums && (keep_J == 0 || J == keep_J)) {
                const int B = blocks_per_sm(smem_fwd<P>(f), f.T, FwdBlock<P>::regs);
                const int comp = Pl.low && f.racc;
                // + the reduce: G partials (and compensation terms) written and read
                const double c = blur_cost(P, (long long)f.G * f.nT * nv, J, 1.0, f.T, B, Pl.sms) +
                                 (double)f.G * g.nx * g.nz * nv * 8.0 * (1 + comp) / 5e6;
                if (c < 0.98 * fbest) fbest = c, Pl.fused_J = J, Pl.fwd_nT = f.nT, Pl.part_comp = comp;
            }
            const AdjDims a = adj_dims<P>(g, J, std::max(tiles, Pl.min_nT), limit);
            if (smem_adj<P>(a) <= limit) {
                const int B = blocks_per_sm(smem_adj<P>(a), a.T, AdjBlock<P>::regs);
                const double c = blur_cost(P, (long long)a.G * a.nT * nv, J, 1.0, a.T, B, Pl.sms);
                if (c < 0.98 * abest) abest = c, Pl.adj_J = J, Pl.adj_nT = a.nT;
            }
        }
    }
}
}  // namespace

// Default launch shapes of the blur kernels.  A block is one thread per work item of a
// column tile, so that several blocks share an SM and one block's barriers, plane
// loads and set-up are covered by the others' FMAs: forward at 128x80, 128 views, 37
// taps 485 us with 32 columns, 542 with 48 (whole planes in one block of 640 threads:
// 513); adjoint 538, 578 with 48; 192x128, 64 views: adjoint 1013 with 32, 952 with 48.
void default_shape(spect_plan_s& P)
{
    const Geometry& g = P.g;
    if (!P.separable) {  // blocks of the full-PSF forward kernel
        // J = 2, 4, 8, A and A' in us: 3.4 blocks of 8 planes per SM (64x32, 32 views, 9x9 PSF) 33.2 33.4 35.5 and
        // 41.0 41.3 45.2; 14 (96x64, 60 views, 21x21) 565 566 579 and 657 636 643; 25 (128x64, 60 views, 11x11)
        // 419 400 396 and 475 432 422; 54 (128x80, 128 views, 9x9) 964 893 860 and 1038 933 882
        P.part_comp = P.low;
        if (P.shape_views < g.nview && !P.low) return;  // as choose_shape's keep_J
        P.fused_J = P.adj_J = 8;
        const long long blocks = (long long)((g.nx + 31) / 32) * ((g.ny + 7) / 8) * P.shape_views;
        if (blocks < 24ll * P.sms) P.fused_J = blocks >= 4ll * P.sms ? 4 : 2;
        P.adj_J = P.fused_J;
        return;
    }
    switch (P.bucket) {
#define SPECT_CS(B) \
    case B: choose_shape<B>(P); break;
        SPECT_CS(3) SPECT_CS(5) SPECT_CS(7) SPECT_CS(9) SPECT_CS(11) SPECT_CS(13) SPECT_CS(15)
        SPECT_CS(17) SPECT_CS(21) SPECT_CS(25) SPECT_CS(29) SPECT_CS(33) SPECT_CS(37)
#undef SPECT_CS
        default: break;
    }
}

// Column tiles of the blur adjoint at its launch shape (what adj_dims makes of the request).
int adj_tiles(const spect_plan_s& P)
{
    switch (P.bucket) {
#define SPECT_AT(B) \
    case B: return adj_dims<B>(P.g, P.adj_J, P.adj_nT, (size_t)P.smem_optin).nT;
        SPECT_AT(3) SPECT_AT(5) SPECT_AT(7) SPECT_AT(9) SPECT_AT(11) SPECT_AT(13) SPECT_AT(15)
        SPECT_AT(17) SPECT_AT(21) SPECT_AT(25) SPECT_AT(29) SPECT_AT(33) SPECT_AT(37)
#undef SPECT_AT
        default: return P.adj_nT;
    }
}

// Column tiles of the forward blur at its launch shape (what fwd_dims makes of the request).
int fwd_tiles(const spect_plan_s& P)
{
    switch (P.bucket) {
#define SPECT_FT(B) \
    case B: return fwd_dims<B>(P.g, P.fused_J, P.fwd_nT, (size_t)P.smem_optin).nT;
        SPECT_FT(3) SPECT_FT(5) SPECT_FT(7) SPECT_FT(9) SPECT_FT(11) SPECT_FT(13) SPECT_FT(15)
        SPECT_FT(17) SPECT_FT(21) SPECT_FT(25) SPECT_FT(29) SPECT_FT(33) SPECT_FT(37)
#undef SPECT_FT
        default: return 1;
    }
}

// floats per view of the work slab the fused path needs (rotated plane images or t planes)
size_t fused_slab_per_view(const spect_plan_s& P)
{
    return (size_t)P.g.ny * P.g.nx * P.g.kp;
}

cudaError_t launch_fused_adjoint(const spect_plan_s& P, const float* v, int l0, int nv, cudaStream_t st)
{
    if (!P.separable) {
        SPECT_DISPATCH(dir_adj_launch, P, v, l0, nv, st)
    }
    SPECT_DISPATCH(adj_launch, P, v, l0, nv, st)
}
#undef SPECT_DISPATCH

cudaError_t launch_fwd_reduce(const spect_plan_s& P, int l0, int nv, float* v, const float* em_y, const float* em_rbar,
                              cudaStream_t st)
{
    const size_t view = (size_t)P.g.nx * P.g.nz, nproj = view * nv, at = view * l0;
    v += em_y ? (size_t)P.g.np * P.g.nz * l0 : at;
    const float* comp = P.part_comp ? P.part + fused_groups(P) * nproj : nullptr;
    return launch_chained(k_fwd_reduce, (unsigned)((nproj + 255) / 256), 256, 0, st, P.part, comp, fused_groups(P), nproj, v,
                          P.g.nx, P.g.np, em_y ? em_y + at : nullptr, em_rbar ? em_rbar + at : nullptr);
}

cudaError_t launch_adj_rot_t(const spect_plan_s& P, int l0, int nv, int s0, float* out, PassState pass, EmArgs em,
                             cudaStream_t st)
{
    const size_t n = (size_t)P.g.nx * P.g.ny * (P.g.kp / 4);
    const unsigned blocks = (unsigned)((n + 255) / 256);
    const float* src = P.slab + (size_t)s0 * P.g.ny * P.ps;
    const int segs = P.adj_chunk >= P.g.nview ? P.gsegs : 1, seglen = (nv + segs - 1) / segs;  // as the patch gather
    switch (P.adj_max) {
#define SPECT_ADJ(M)                                                                                                 \
    case M: return launch_chained(k_adj_rot_t<M>, blocks, 256, 0, st, P.g, P.ps, P.adjf, src, l0, nv, out, pass, seglen, em);
        SPECT_ADJ(1) SPECT_ADJ(2) SPECT_ADJ(3) SPECT_ADJ(4) SPECT_ADJ(5) SPECT_ADJ(6) SPECT_ADJ(7) SPECT_ADJ(8)
#undef SPECT_ADJ
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace spect
