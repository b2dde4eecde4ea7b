// gather.cu -- adjoint rotation and view sum of A' (Section II-A, Algorithm 2)
// as a patch-staged gather:
//
//   x_t(q, k) = sum_l sum_{(p, w) in adj(l, q)} w * t_l(p, k)
//
// One block owns an 8x8 patch of destination columns q, a run of KC consecutive k and
// one of P.gsegs runs of the views.  For every view, the source pixels its destinations read lie
// in a small box of the rotated frame (at most about 8*sqrt(2) + 2 on a side);
// the box is brought into shared memory by one TMA tensor load (3D tile of the
// t slab: k x i x plane) and the patch's adjacency entries by one bulk copy,
// several views ahead of use, so the gathers read shared memory instead of
// waiting on L2.  The entries hold box-local offsets computed at plan time from
// the fixed-length lists k_build_adjacency_fixed writes (same weights, same
// order), and the per-view sum and the Kahan sums over views are those of
// k_adj_rot_t: the results are bitwise the same.
//   Bound by the box traffic from L2 and the shared-memory reads of five (eight) 16-byte
// values per four outputs and view.  A patch's box is loaded at its own size (up to
// kGatherMaps square sizes, a tensor map each), not at the largest of all angles.
// The views are split over blocks where the patches alone leave the chip short of
// them; the last block of a patch adds the segments in order.  The three-pass lists
// (eight taps) take runs of 32 k: two bytes of entries per output less.
//   Measured: 64x32, 64 views 27.4 -> 21.0 us, 24x60, 32 views 16.0 -> 12.4 (segments);
// three-pass 128x64, 60 views 193 -> 137; 128x80, 128 views 208 (l1tex at 82 % of its peak).
// Bilinear lists with runs of 32 k: 243 at 128x80, so they keep 16.
#include <cuda.h>

#include <algorithm>
#include <climits>
#include <cstdlib>
#include <vector>

#include "spect_internal.cuh"

namespace spect {

namespace {

constexpr int kPatch = 8;     // destinations per patch side
constexpr int kStages = 3;    // views in flight per block (measured best: 3 of 3, 4, 6, 8)

// Box of source pixels read by patch `patch` in view l = l0 + blockIdx.y: (i0, j0, width,
// height).  adjf holds the lists of the gridDim.y views from l0 on.
__global__ void k_patch_boxes(Geometry g, int ps, int maxe, const AdjEntry* __restrict__ adjf, int l0, int npx,
                              int4* boxes)
{
    __shared__ int mn_i, mn_j, mx_i, mx_j;
    const int patch = blockIdx.x, l = l0 + blockIdx.y, t = threadIdx.x;
    if (t == 0) {
        mn_i = mn_j = INT_MAX;
        mx_i = mx_j = INT_MIN;
    }
    __syncthreads();
    const int qi = (patch % npx) * kPatch + (t % kPatch), qj = (patch / npx) * kPatch + (t / kPatch);
    if (qi < g.nx && qj < g.ny) {
        const AdjEntry* e = adjf + ((size_t)(qj * g.nx + qi) * gridDim.y + blockIdx.y) * maxe;
        for (int m = 0; m < maxe; ++m) {
            if (e[m].w == 0.f) continue;
            const int pj = e[m].p / ps, pi = (e[m].p - pj * ps) / g.kp;
            atomicMin(&mn_i, pi);
            atomicMin(&mn_j, pj);
            atomicMax(&mx_i, pi);
            atomicMax(&mx_j, pj);
        }
    }
    __syncthreads();
    if (t == 0) {
        int4 b = make_int4(0, 0, 0, 0);
        if (mx_i >= mn_i) b = make_int4(mn_i, mn_j, mx_i - mn_i + 1, mx_j - mn_j + 1);
        boxes[(size_t)patch * g.nview + l] = b;
    }
}

// Patch entries [patch][l][64][maxe]: (box-local offset (row*size + col)*KC, weight);
// zero entries for padding and for destinations outside the image.  boxes: (i0, j0,
// box size, tensor map).  Views and lists as in k_patch_boxes.
__global__ void k_patch_entries(Geometry g, int ps, int maxe, const AdjEntry* __restrict__ adjf, int l0, int npx,
                                const int4* __restrict__ boxes, int kc, AdjEntry* pent)
{
    const int patch = blockIdx.x, l = l0 + blockIdx.y, t = threadIdx.x;
    const int qi = (patch % npx) * kPatch + (t % kPatch), qj = (patch / npx) * kPatch + (t / kPatch);
    const int4 b = boxes[(size_t)patch * g.nview + l];
    AdjEntry* out = pent + (((size_t)patch * g.nview + l) * (kPatch * kPatch) + t) * maxe;
    const bool inside = qi < g.nx && qj < g.ny;
    const AdjEntry* e = adjf + ((size_t)(qj * g.nx + qi) * gridDim.y + blockIdx.y) * maxe;
    for (int m = 0; m < maxe; ++m) {
        AdjEntry o;  // padding and outside destinations: weight 0 on the box's first element
        o.p = 0;
        o.w = 0.f;
        if (inside && e[m].w != 0.f) {
            const int pj = e[m].p / ps, pi = (e[m].p - pj * ps) / g.kp;
            o.p = ((pj - b.y) * b.z + (pi - b.x)) * kc;
            o.w = e[m].w;
        }
        out[m] = o;
    }
}

struct GatherArgs {
    Geometry g;
    int npx;         // patches along i
    int kc;          // k per block (a box: kc x size x size)
    int box_floats;  // floats of the largest box
    int ent_bytes;   // 64 * maxe * 8
    int stage_floats;
    int l0, nv, s0;  // views [l0, l0 + nv) of the plan; slab view s0 + v holds view l0 + v
    int nkc;         // runs of kc depth rows per patch
    int segs, seglen;  // view segments (blocks) per patch and k run, views of one
    float* seg;        // segs > 1: [segs][2][volume] sums and compensation terms of the segments
    int* count;        // segs > 1: [patch, k run] arrivals (0 between launches)
};

// Consumer threads: 64 destinations x KC / 4 float4 groups of k; one more warp
// produces: it refills a stage as soon as every consumer has released it
// (per-stage "empty" barrier), so consumers never meet at a block barrier
// inside the view loop.
template <int MAXE, int KC>
__device__ __forceinline__ void adj_gather_body(const CUtensorMap* maps, const GatherArgs& a,
                                                const int4* __restrict__ boxes, const AdjEntry* __restrict__ pent,
                                                float* out, const PassState& pass, const EmArgs& em, int* err,
                                                const int patch, const int kcb, const int seg)
{
    constexpr int kGT = 16 * KC, K4 = KC / 4;  // consumer threads; float4 groups of k
    extern __shared__ __align__(128) float sm[];
    const Geometry& g = a.g;
    uint64_t* full = reinterpret_cast<uint64_t*>(sm + (size_t)kStages * a.stage_floats);
    uint64_t* empty = full + kStages;
    volatile int* abort_flag = reinterpret_cast<volatile int*>(empty + kStages);
    const int kc0 = kcb * KC;
    const int v0 = seg * a.seglen, nvs = min(a.nv - v0, a.seglen);  // this block's views
    const int tid = threadIdx.x;
    const bool producer = tid >= kGT;

    // tensor copies want 128-byte aligned shared memory: refuse (error word) rather than fault
    if ((smem_u32(sm) & 127u) != 0) {
        if (tid == 0 && err) atomicExch(err, (int)SPECT_ECUDA);
        return;
    }
    if (tid == kGT) {
        for (int s = 0; s < kStages; ++s) {
            mbar_init(full + s, 1);
            mbar_init(empty + s, kGT);
        }
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();

    if (producer) {
        if (tid != kGT) return;  // one lane issues
        int issued = 0;
        for (int v = 0; v < nvs; ++v) {
            const int s = v % kStages;
            if (*abort_flag) break;
            if (v >= kStages && !mbar_wait_bounded(empty + s, (unsigned)(v / kStages - 1) & 1u)) {
                *abort_flag = 1;
                break;
            }
            if (v >= kStages) fence_proxy_async_smem();
            float* st = sm + (size_t)s * a.stage_floats;
            const int l = a.l0 + v0 + v;
            const int4 b = boxes[(size_t)patch * g.nview + l];
            asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(full + s)),
                         "r"((unsigned)(b.z * b.z * KC * 4 + a.ent_bytes))
                         : "memory");
            tma_load_3d(st, maps + b.w, kc0, b.x, (a.s0 + v0 + v) * g.ny + b.y, full + s);
            tma_copy_1d(st + a.box_floats, pent + ((size_t)patch * g.nview + l) * (kPatch * kPatch) * MAXE,
                        (unsigned)a.ent_bytes, full + s);
            issued = v + 1;
        }
        if (*abort_flag) {  // let every copy in flight land before the block's shared memory is released
            if (err) atomicExch(err, (int)SPECT_ETIMEOUT);
            for (int u = issued - kStages < 0 ? 0 : issued - kStages; u < issued; ++u)
                mbar_wait_bounded(full + (u % kStages), (unsigned)(u / kStages) & 1u);
        }
        return;
    }

    const int ql = tid / K4, k4 = tid % K4;  // destination in the patch, float4 group of k
    const int qi = (patch % a.npx) * kPatch + (ql % kPatch), qj = (patch / a.npx) * kPatch + (ql / kPatch);
    // the EM epilogue's operands, fetched before the view loop so their latency hides behind it
    const int k = kc0 + 4 * k4;
    const bool mine = qi < g.nx && qj < g.ny && k < g.kp;
    const size_t o = mine ? (size_t)(qj * g.nx + qi) * g.kp + k : 0;
    float4 ex = make_float4(0.f, 0.f, 0.f, 0.f), es = ex, eu = ex;
    if (mine && em.x && a.segs == 1) {
        ex = *reinterpret_cast<const float4*>(em.x + o);
        es = *reinterpret_cast<const float4*>(em.s + o);
        if (em.u) eu = *reinterpret_cast<const float4*>(em.u + o);
    }

    KSum acc[4];
    if (mine && pass.resume) {  // the sums of the views of earlier launches
        const float4 s = *reinterpret_cast<const float4*>(pass.acc + o), c = *reinterpret_cast<const float4*>(pass.acc_c + o);
        acc[0].s = s.x, acc[1].s = s.y, acc[2].s = s.z, acc[3].s = s.w;
        acc[0].c = c.x, acc[1].c = c.y, acc[2].c = c.z, acc[3].c = c.w;
    }
    bool failed = false;
    for (int v = 0; v < nvs; ++v) {
        const int s = v % kStages;
        if (!failed) {
            if (mbar_wait_bounded(full + s, (unsigned)(v / kStages) & 1u)) {
                const float* box = sm + (size_t)s * a.stage_floats;
                const AdjEntry* e = reinterpret_cast<const AdjEntry*>(box + a.box_floats) + ql * MAXE;
                AdjEntry en[MAXE];
#pragma unroll
                for (int m = 0; m < MAXE; ++m) en[m] = e[m];
                float4 tv[MAXE];
#pragma unroll
                for (int m = 0; m < MAXE; ++m) tv[m] = *reinterpret_cast<const float4*>(box + en[m].p + 4 * k4);
                float sv[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
                for (int m = 0; m < MAXE; ++m) {
                    sv[0] = fmaf(en[m].w, tv[m].x, sv[0]);
                    sv[1] = fmaf(en[m].w, tv[m].y, sv[1]);
                    sv[2] = fmaf(en[m].w, tv[m].z, sv[2]);
                    sv[3] = fmaf(en[m].w, tv[m].w, sv[3]);
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) acc[u].add(sv[u]);
            } else {
                failed = true;
                *abort_flag = 1;
                if (err) atomicExch(err, (int)SPECT_ETIMEOUT);
            }
        }
        // release the stage (also after a failed wait, so the producer never waits on it)
        asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(empty + s)) : "memory");
    }
    if (a.segs == 1 && (failed || *abort_flag)) return;

    if (a.segs > 1) {
        // leave this segment's sums, and let the last block of the patch and k run add
        // all segments in order (each block publishes its sums before it counts itself)
        const size_t vol = (size_t)g.nx * g.ny * g.kp;
        if (mine) {
            float* p = a.seg + (size_t)seg * 2 * vol + o;
            __stcg(reinterpret_cast<float4*>(p), make_float4(acc[0].s, acc[1].s, acc[2].s, acc[3].s));
            __stcg(reinterpret_cast<float4*>(p + vol), make_float4(acc[0].c, acc[1].c, acc[2].c, acc[3].c));
        }
        __threadfence();
        asm volatile("bar.sync 1, %0;" ::"n"(kGT) : "memory");  // every consumer, also after a failed wait
        volatile int* last = abort_flag + 1;
        if (tid == 0) {  // counted also after a failed wait (the error word is set), so the counter ends at 0
            int* cnt = a.count + (size_t)patch * a.nkc + kcb;
            const int l = atomicAdd(cnt, 1) == a.segs - 1;
            if (l) *cnt = 0;
            *last = l;
        }
        asm volatile("bar.sync 1, %0;" ::"n"(kGT) : "memory");
        if (!*last || !mine) return;
        __threadfence();
#pragma unroll
        for (int u = 0; u < 4; ++u) acc[u] = KSum();
        for (int q = 0; q < a.segs; ++q) {
            const float* p = a.seg + (size_t)q * 2 * vol + o;
            const float4 s4 = __ldcg(reinterpret_cast<const float4*>(p));
            const float4 c4 = __ldcg(reinterpret_cast<const float4*>(p + vol));
            const float ss[4] = {s4.x, s4.y, s4.z, s4.w}, cc[4] = {c4.x, c4.y, c4.z, c4.w};
#pragma unroll
            for (int u = 0; u < 4; ++u) acc[u].merge(ss[u], cc[u]);
        }
        if (em.x) {
            ex = *reinterpret_cast<const float4*>(em.x + o);
            es = *reinterpret_cast<const float4*>(em.s + o);
            if (em.u) eu = *reinterpret_cast<const float4*>(em.u + o);
        }
    }

    if (!mine) return;
    if (pass.merge) {  // add this segment to the ones before it
        KSum tot[4];
        if (pass.tot_resume) {
            const float4 s = *reinterpret_cast<const float4*>(out + o), c = *reinterpret_cast<const float4*>(pass.tot_c + o);
            tot[0].s = s.x, tot[1].s = s.y, tot[2].s = s.z, tot[3].s = s.w;
            tot[0].c = c.x, tot[1].c = c.y, tot[2].c = c.z, tot[3].c = c.w;
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) tot[u].merge(acc[u].s, acc[u].c), acc[u] = tot[u];
    }
    if (pass.more || (pass.merge && pass.tot_more)) {
        float *s = pass.more ? pass.acc : out, *c = pass.more ? pass.acc_c : pass.tot_c;
        *reinterpret_cast<float4*>(s + o) = make_float4(acc[0].s, acc[1].s, acc[2].s, acc[3].s);
        *reinterpret_cast<float4*>(c + o) = make_float4(acc[0].c, acc[1].c, acc[2].c, acc[3].c);
        return;
    }
    const float xv[4] = {ex.x, ex.y, ex.z, ex.w}, sv4[4] = {es.x, es.y, es.z, es.w}, uv[4] = {eu.x, eu.y, eu.z, eu.w};
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const float val = acc[u].value();
        if (em.x) em.x[o + u] = em_update(xv[u], val, sv4[u], uv[u], em.beta);
        else out[o + u] = val;
    }
}

template <int MAXE, int KC>
__global__ void __launch_bounds__(16 * KC + 32) k_adj_gather(const __grid_constant__ GatherMaps maps, GatherArgs a,
                                                         const int4* __restrict__ boxes,
                                                         const AdjEntry* __restrict__ pent, float* out,
                                                         PassState pass, EmArgs em, int* err)
{
    wait_previous_kernel();
    // the k runs of a patch are adjacent blocks, so they run side by side and the
    // patch's entries, which each of them reads, come from DRAM about once
    // (0.246 -> 0.213 ms per 128-view launch against the patch-major order)
    const int patch = (int)blockIdx.x / a.nkc, kcb = (int)blockIdx.x - patch * a.nkc;
    adj_gather_body<MAXE, KC>(maps.m, a, boxes, pent, out, pass, em, err, patch, kcb, blockIdx.y);
}


// floats per pipeline stage: the box, then the entries, rounded up to 128 bytes
int stage_floats(int box_floats, int ent_bytes) { return (box_floats + ent_bytes / 4 + 31) & ~31; }

size_t gather_smem(int box_floats, int ent_bytes)
{
    // stages | full and empty barriers | abort flag
    return (size_t)kStages * stage_floats(box_floats, ent_bytes) * sizeof(float) + 2 * kStages * sizeof(uint64_t) +
           16;
}

// One plan's arguments of the grouped gather (the tensor map in the kernel's
// parameter space, as in the per-plan launch).
struct GroupGather {
    GatherMaps maps;
    GatherArgs a;
    const int4* boxes;
    const AdjEntry* pent;
    float* out;
    EmArgs em;
    int* err;
};
struct GroupGathers {
    GroupGather p[kGroupMax];
    GroupGrid grid;
};

template <int MAXE, int KC>
__global__ void __launch_bounds__(16 * KC + 32) k_adj_gather_grp(const __grid_constant__ GroupGathers gg)
{
    const int4 w = group_item(gg.grid);
    const GroupGather& q = gg.p[w.x];
    adj_gather_body<MAXE, KC>(q.maps.m, q.a, q.boxes, q.pent, q.out, PassState(), q.em, q.err, w.z, w.y, w.w);
}

}  // namespace

EncodeTiled encode_fn()
{
    static EncodeTiled fn = nullptr;
    if (!fn) {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiled>(p);
        cudaGetLastError();
    }
    return fn;
}

namespace {
// k per block.  16 measured best for the bilinear lists (128x80, 128 views: 210 us, 243
// with 32), 32 for the eight entries of the three-pass ones, whose reads bound them
// (128x64, 60 views: 137 us, 193 with 16).
int gather_kc(const spect_plan_s& P)
{
    return P.rot3 && P.g.kp > 16 ? 32 : 16;
}
}  // namespace

// View segments of A': as many as fill one wave of resident blocks, of at least 8 views
// each (64x32, 64 views: 27 us with one, 21 with four; 24x60, 30 views: 16 and 12).  More
// than a wave only adds the segments' sums (96x64, 64 views: 52 and 57).  One launch takes
// all segments; where the views go in several passes the launches end at the segments'
// boundaries (fast_back), so that the order of the sums is the same.
int gather_segments(const spect_plan_s& P)
{
    const Geometry& g = P.g;
    const int kc = gather_kc(P), res = kc == 32 ? 2 : 4;
    const long long blocks = (long long)((g.nx + kPatch - 1) / kPatch) * ((g.ny + kPatch - 1) / kPatch) * ((g.kp + kc - 1) / kc);
    const long long want = (long long)res * P.sms / blocks;
    return (int)std::max<long long>(1, std::min<long long>(std::min<long long>(want, 8), g.nview / 8));
}

// Plan time: boxes, box extents and patch entries.  Leaves P.gather = 0 when
// the geometry does not suit the kernel (boxes too large for the tensor map or
// shared memory, no encoder).
cudaError_t build_gather(spect_plan_s& P, cudaStream_t st)
{
    P.gather = 0;
    const Geometry& g = P.g;
    if (!P.fast || !encode_fn()) return cudaSuccess;
    const char* env = getenv("SPECT_GATHER");  // 0: use the list gather k_adj_rot_t (testing)
    if (env && atoi(env) == 0) return cudaSuccess;
    const int npx = (g.nx + kPatch - 1) / kPatch, npy = (g.ny + kPatch - 1) / kPatch;
    const size_t nb = (size_t)npx * npy * g.nview;
    int4* boxes = nullptr;
    cudaError_t e = P.pooled ? cudaMallocAsync((void**)&boxes, nb * sizeof(int4), st)
                             : cudaMalloc((void**)&boxes, nb * sizeof(int4));
    if (e != cudaSuccess) return e;
    // f(l0, nv) for the ranges of views whose lists adjf holds at once
    auto ranges = [&](auto&& f) {
        const int lv = P.list_views;
        cudaError_t er = cudaSuccess;
        for (int l0 = 0; l0 < g.nview && er == cudaSuccess; l0 += lv) {
            const int nv = std::min(lv, g.nview - l0);
            if (lv < g.nview) er = launch_build_adjacency_fixed(P, l0, nv, st);
            if (er == cudaSuccess) f(l0, nv);
            if (er == cudaSuccess) er = cudaGetLastError();
        }
        return er;
    };
    e = ranges([&](int l0, int nv) {
        k_patch_boxes<<<dim3(npx * npy, nv), kPatch * kPatch, 0, st>>>(g, P.ps, P.adj_max, P.adjf, l0, npx, boxes);
    });
    std::vector<int4> hb(nb);
    if (e == cudaSuccess) e = cudaMemcpyAsync(hb.data(), boxes, nb * sizeof(int4), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) {
        if (P.pooled) cudaFreeAsync(boxes, st);
        else cudaFree(boxes);
        return e;
    }
    // box sizes: every size that occurs, rounded up to odd (neighbouring columns and rows
    // then fall into different halves of the banks), neighbours merged (where that
    // adds the least traffic) down to kGatherMaps.  Against one box of the largest size:
    // 128x80, 128 views 215 -> 208 us, 192x128, 43 views 235 -> 222.
    std::vector<std::pair<int, double>> sizes;  // (size, boxes of it)
    {
        std::vector<double> hist(1);
        for (const int4& b : hb) {
            const size_t z = (size_t)(std::max(b.z, b.w) | 1);
            if (hist.size() <= z) hist.resize(z + 1);
            hist[z] += 1.0;
        }
        for (int z = 1; z < (int)hist.size(); ++z)
            if (hist[z] > 0.0) sizes.emplace_back(z, hist[z]);
        while ((int)sizes.size() > kGatherMaps) {
            size_t at = 0;
            double least = 1e300;
            for (size_t q = 0; q + 1 < sizes.size(); ++q) {
                const double a = sizes[q].first, b = sizes[q + 1].first, add = sizes[q].second * (b * b - a * a);
                if (add < least) least = add, at = q;
            }
            sizes[at + 1].second += sizes[at].second;
            sizes.erase(sizes.begin() + at);
        }
    }
    const int kc = gather_kc(P), top = sizes.back().first;
    const int box_floats = top * top * kc;
    const int ent_bytes = kPatch * kPatch * P.adj_max * (int)sizeof(AdjEntry);
    if (top > 256 || gather_smem(box_floats, ent_bytes) > (size_t)P.smem_optin ||
        (size_t)box_floats * 4 + ent_bytes >= (1u << 20)) {
        if (P.pooled) cudaFreeAsync(boxes, st);
        else cudaFree(boxes);
        return cudaSuccess;
    }
    for (int4& b : hb) {
        const int z = (std::max(b.z, b.w) | 1);
        int q = 0;
        while (sizes[q].first < z) ++q;
        b.z = sizes[q].first;
        b.w = q;
    }
    e = cudaMemcpyAsync(boxes, hb.data(), nb * sizeof(int4), cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);  // hb is the source
    if (e != cudaSuccess) {
        if (P.pooled) cudaFreeAsync(boxes, st);
        else cudaFree(boxes);
        return e;
    }
    const size_t nent = nb * kPatch * kPatch * P.adj_max;
    AdjEntry* pent = nullptr;
    e = P.pooled ? cudaMallocAsync((void**)&pent, nent * sizeof(AdjEntry), st)
                 : cudaMalloc((void**)&pent, nent * sizeof(AdjEntry));
    if (e != cudaSuccess) {
        if (P.pooled) cudaFreeAsync(boxes, st);
        else cudaFree(boxes);
        return e;
    }
    e = ranges([&](int l0, int nv) {
        k_patch_entries<<<dim3(npx * npy, nv), kPatch * kPatch, 0, st>>>(g, P.ps, P.adj_max, P.adjf, l0, npx, boxes, kc,
                                                                         pent);
    });
    const size_t ncount = (size_t)npx * npy * ((g.kp + kc - 1) / kc);
    int* count = nullptr;
    if (e == cudaSuccess)
        e = P.pooled ? cudaMallocAsync((void**)&count, ncount * sizeof(int), st)
                     : cudaMalloc((void**)&count, ncount * sizeof(int));
    if (e == cudaSuccess) e = cudaMemsetAsync(count, 0, ncount * sizeof(int), st);
    P.gcount = count;
    P.gboxes = boxes;
    P.gent = pent;
    P.bytes += nb * sizeof(int4) + nent * sizeof(AdjEntry) + ncount * sizeof(int);
    P.gnm = (int)sizes.size();
    for (int q = 0; q < P.gnm; ++q) P.gsize[q] = sizes[q].first;
    P.gnpx = npx;
    P.gnpy = npy;
    P.gather = e == cudaSuccess;
    return e;
}

// The t slab as 3D tensor maps -- k (kp, contiguous) x i (nx, stride kp) x plane
// (chunk * ny, stride ps) -- one per box size.
cudaError_t build_gather_maps(spect_plan_s& P)
{
    if (!P.gather) return cudaSuccess;
    const Geometry& g = P.g;
    const int kc = gather_kc(P);
    const cuuint64_t dims[3] = {(cuuint64_t)g.kp, (cuuint64_t)g.nx, (cuuint64_t)P.chunk * g.ny};
    const cuuint64_t strides[2] = {(cuuint64_t)g.kp * 4, (cuuint64_t)P.ps * 4};
    const cuuint32_t estr[3] = {1, 1, 1};
    for (int q = 0; q < P.gnm; ++q) {
        const cuuint32_t box[3] = {(cuuint32_t)kc, (cuuint32_t)P.gsize[q], (cuuint32_t)P.gsize[q]};
        if (encode_fn()(&P.gmaps.m[q], CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, P.slab, dims, strides, box, estr,
                        CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                        CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return cudaErrorInvalidValue;
    }
    return cudaSuccess;
}

namespace {
// The gather's arguments for views [l0, l0 + nv), the first at view s0 of the slab.
void gather_setup(const spect_plan_s& P, int l0, int nv, int s0, GatherArgs* a)
{
    const Geometry& g = P.g;
    const int kc = gather_kc(P), top = P.gsize[P.gnm - 1];
    a->g = g;
    a->npx = P.gnpx;
    a->kc = kc;
    a->box_floats = top * top * kc;
    a->ent_bytes = kPatch * kPatch * P.adj_max * (int)sizeof(AdjEntry);
    a->stage_floats = stage_floats(a->box_floats, a->ent_bytes);
    a->l0 = l0;
    a->nv = nv;
    a->s0 = s0;
    a->nkc = (g.kp + kc - 1) / kc;
    a->segs = P.adj_chunk >= g.nview ? P.gsegs : 1;
    a->seglen = (nv + a->segs - 1) / a->segs;
    a->seg = P.part;  // free between the depth-group reduce and the next forward blur
    a->count = P.gcount;
}
}  // namespace

cudaError_t launch_adj_gather(const spect_plan_s& P, int l0, int nv, int s0, float* out, PassState pass, EmArgs em,
                              cudaStream_t st)
{
    GatherArgs a;
    gather_setup(P, l0, nv, s0, &a);
    const size_t smem = gather_smem(a.box_floats, a.ent_bytes);
    const dim3 grid(P.gnpx * P.gnpy * a.nkc, a.segs);  // (patch, k run), the k runs of a patch adjacent
    switch (P.adj_max) {
#define SPECT_GK(M, KC)                                                                                         \
    {                                                                                                           \
        cudaError_t e = cudaFuncSetAttribute(k_adj_gather<M, KC>, cudaFuncAttributeMaxDynamicSharedMemorySize,  \
                                             (int)smem);                                                        \
        if (e != cudaSuccess) return e;                                                                         \
        return launch_chained(k_adj_gather<M, KC>, grid, 16 * KC + 32, smem, st, P.gmaps, a, P.gboxes, P.gent, out, \
                              pass, em, P.err);                                                                 \
    }
#define SPECT_G(M)                     \
    case M:                            \
        if (a.kc == 32) SPECT_GK(M, 32) \
        else SPECT_GK(M, 16)
        SPECT_G(1) SPECT_G(2) SPECT_G(3) SPECT_G(4) SPECT_G(5) SPECT_G(6) SPECT_G(7) SPECT_G(8)
#undef SPECT_GK
#undef SPECT_G
        default: return cudaErrorInvalidValue;
    }
}

// The grouped gather of a batch: per adjacency-list length, one launch over
// every plan's (patch, k run) blocks, largest plans first; each plan's MLEM
// update (beta = 0) in the epilogue, as in its own EM step.
cudaError_t build_grouped_gather(const std::vector<spect_plan_s*>& plans, GroupedBatch& B,
                                 std::vector<GroupLaunch>& out)
{
    (void)B;
    for (int mk = 2; mk <= 17; ++mk) {  // per list length and k run
        const int maxe = mk / 2, kc = mk % 2 ? 32 : 16;
        std::vector<int> idx;
        for (int i = 0; i < (int)plans.size(); ++i)
            if (plans[i]->adj_max == maxe && gather_kc(*plans[i]) == kc) idx.push_back(i);
        std::stable_sort(idx.begin(), idx.end(), [&](int x, int y) {
            const auto w = [](const spect_plan_s* P) { return (size_t)P->g.nx * P->g.ny * P->g.nz * P->g.nview; };
            return w(plans[x]) > w(plans[y]);
        });
        for (size_t c0 = 0; c0 < idx.size(); c0 += kGroupMax) {
            const size_t c1 = std::min(idx.size(), c0 + (size_t)kGroupMax);
            GroupGathers gg{};
            size_t smem = 0;
            for (size_t m = c0; m < c1; ++m) {
                const spect_plan_s& P = *plans[idx[m]];
                GroupGather& q = gg.p[m - c0];
                gather_setup(P, 0, P.g.nview, 0, &q.a);
                q.maps = P.gmaps;
                q.boxes = P.gboxes;
                q.pent = P.gent;
                q.out = P.et;
                q.em.x = P.xt;
                q.em.s = P.st;
                q.em.u = nullptr;
                q.em.beta = 0.f;
                q.err = P.err;
                smem = std::max(smem, gather_smem(q.a.box_floats, q.a.ent_bytes));
                // the gather's grid: (run of kc depth rows, patch, view segment), the k runs of a patch adjacent
                const int mm = (int)(m - c0), nkc = q.a.nkc;
                if (mm == 0) gg.grid.first[0] = 0;
                gg.grid.gx[mm] = nkc;
                gg.grid.gy[mm] = P.gnpx * P.gnpy;
                gg.grid.first[mm + 1] = gg.grid.first[mm] + P.gnpx * P.gnpy * nkc * q.a.segs;
                gg.grid.n = mm + 1;
            }
            const unsigned nb = (unsigned)gg.grid.first[gg.grid.n];
            GroupLaunch L;
            switch (mk) {
#define SPECT_GG(M, KC)                                                                                        \
    case 2 * M + (KC == 32):                                                                                   \
        L = [gg, nb, smem](cudaStream_t st) -> cudaError_t {                                                   \
            cudaError_t e2 = cudaFuncSetAttribute(k_adj_gather_grp<M, KC>,                                     \
                                                  cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);     \
            if (e2 != cudaSuccess) return e2;                                                                  \
            k_adj_gather_grp<M, KC><<<nb, 16 * KC + 32, smem, st>>>(gg);                                       \
            return cudaGetLastError();                                                                         \
        };                                                                                                     \
        break;
#define SPECT_GG2(M) SPECT_GG(M, 16) SPECT_GG(M, 32)
                SPECT_GG2(1) SPECT_GG2(2) SPECT_GG2(3) SPECT_GG2(4) SPECT_GG2(5) SPECT_GG2(6) SPECT_GG2(7) SPECT_GG2(8)
#undef SPECT_GG2
#undef SPECT_GG
                default: return cudaErrorInvalidValue;
            }
            out.push_back(L);
        }
    }
    return cudaSuccess;
}

}  // namespace spect
