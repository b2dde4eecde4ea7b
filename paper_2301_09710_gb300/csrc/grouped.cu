// grouped.cu -- EM iterations of many plans as grouped launches (the batch
// interface spect_batch_*): one launch per stage and kernel variant over a work
// list that spans every plan of the batch, instead of one launch per stage and
// plan.  Stages of one EM iteration (Eqs. (7)-(8), beta = 0):
//   rotation + attenuation (all plans),
//   blur + depth-group sums (per bucket), depth-group reduce with
//   the EM ratio (all plans), blur adjoint + attenuation (per bucket, tiled or
//   not), adjoint rotation + view sum + MLEM update (gather.cu, per list length),
// plus the layout transposes of the iterates before the first and after the
// last iteration.  A block finds its plan and its coordinates in that plan's own
// grid from blockIdx.x (the plans' block ranges are in the launch parameters);
// the plan's arguments come from a __grid_constant__ parameter array, and the block runs
// the same device body as the plan's own launch (fused_body.cuh), so every plan
// gets bitwise the values it gets alone.  The largest plans' blocks come first,
// so their long blocks start early and small plans fill the tail.
#include <algorithm>
#include <numeric>

#include "fused_body.cuh"

namespace spect {

namespace {

struct GroupPlan {
    Geometry g;
    RotDims dr;        // rotation launch shape
    AdjDims da;        // adjoint launch shape
    FwdDims df;        // forward launch shape
    const float* rtab;
    const float* xt;
    const float* mubar;
    float* slab;
    const float* frec;
    float* part;
    const float* arec;
    float* ratio;
    const float* y;
    const float* rbar;
    size_t nproj;
    int* err;
};
struct GroupPlans {
    GroupPlan p[kGroupMax];
    CUtensorMap fmap[kGroupMax];                  // the slabs' plane images (forward blur)
    CUtensorMap mmap[kGroupMax], tmap[kGroupMax], vmap[kGroupMax];  // factors, t planes, ratios (blur adjoint)
    GroupGrid grid;
};

struct GroupT {
    const float* in;
    float* out;
    int R, C, ip, op;
};
struct GroupTs {
    GroupT p[kGroupMax];
    GroupGrid grid;
};

__global__ void __launch_bounds__(kRotThreads, 5) k_rot_fwd_grp(const __grid_constant__ GroupPlans gp)
{
    const int4 w = group_item(gp.grid);
    const GroupPlan q = gp.p[w.x];  // by value: the fields live in registers, not re-read from parameter space
    rot_body<4>(q.g, q.dr, q.rtab, q.xt, q.mubar, q.slab, 0, w.y, w.z);
}

template <int P, bool RACC>
__global__ void __launch_bounds__(FwdBlock<P>::T, FwdBlock<P>::B) k_fwd_sep_grp(const __grid_constant__ GroupPlans gp)
{
    const int4 w = group_item(gp.grid);
    const GroupPlan q = gp.p[w.x];  // by value: the fields live in registers, not re-read from parameter space
    const int grp = w.y / q.df.nT;
    fwd_sep_body<P, RACC, false>(q.g, q.df, &gp.fmap[w.x], q.frec, q.part, 0, q.g.nview, q.err, grp, w.z, w.y - grp * q.df.nT);
}

template <int P>
__global__ void __launch_bounds__(AdjBlock<P>::T, AdjBlock<P>::B) k_adj_sep_grp(const __grid_constant__ GroupPlans gp)
{
    const int4 w = group_item(gp.grid);
    const GroupPlan q = gp.p[w.x];  // by value: the fields live in registers, not re-read from parameter space
    const int grp = w.y / q.da.nT;
    adj_sep_body<P>(q.g, q.da, &gp.mmap[w.x], &gp.tmap[w.x], &gp.vmap[w.x], q.arec, 0, 0, q.err, grp, w.z,
                    w.y - grp * q.da.nT);
}

// v = sum over depth groups (fixed order), then the EM ratio y / (v + rbar): k_fwd_reduce per plan
constexpr int kReduceThreads = 256;
__global__ void __launch_bounds__(kReduceThreads) k_fwd_reduce_grp(const __grid_constant__ GroupPlans gp)
{
    const int4 w = group_item(gp.grid);
    const GroupPlan q = gp.p[w.x];  // by value: the fields live in registers, not re-read from parameter space
    const size_t o = (size_t)w.y * kReduceThreads + threadIdx.x;
    if (o >= q.nproj) return;
    const float s = group_sum(q.part + o, nullptr, q.df.G, q.nproj);
    const float yb = s + (q.rbar ? q.rbar[o] : 0.f);
    const int nx = q.g.nx, np = q.g.np;
    q.ratio[np == nx ? o : o + o / nx * (np - nx)] = yb > 0.f ? q.y[o] / yb : 0.f;
}

__global__ void k_transpose_grp(const __grid_constant__ GroupTs gt)
{
    const int4 w = group_item(gt.grid);
    const GroupT& q = gt.p[w.x];
    transpose_body(q.in, q.out, q.R, q.C, q.ip, q.op, w.y, w.z);
}

size_t plan_work(const spect_plan_s* P)
{
    return (size_t)P->g.nx * P->g.ny * P->g.nz * P->g.nview;
}

// chunks of at most kGroupMax plan indices, largest plans first
std::vector<std::vector<int>> chunks_of(std::vector<int> idx, const std::vector<spect_plan_s*>& plans)
{
    std::stable_sort(idx.begin(), idx.end(),
                     [&](int a, int b) { return plan_work(plans[a]) > plan_work(plans[b]); });
    std::vector<std::vector<int>> out;
    for (size_t i = 0; i < idx.size(); i += kGroupMax)
        out.emplace_back(idx.begin() + i, idx.begin() + std::min(idx.size(), i + (size_t)kGroupMax));
    return out;
}

template <int P>
void fill_plan(GroupPlan& q, const spect_plan_s* Pl, const float* y, const float* rbar)
{
    q.g = Pl->g;
    q.df = fwd_dims<P>(Pl->g, Pl->fused_J, Pl->fwd_nT, (size_t)Pl->smem_optin);
    q.da = adj_dims<P>(Pl->g, Pl->adj_J, Pl->adj_nT, (size_t)Pl->smem_optin);
    q.mubar = Pl->mubar;
    q.slab = Pl->slab;
    q.frec = Pl->frec;
    q.part = Pl->part;
    q.arec = Pl->arec;
    q.ratio = Pl->ratio;
    q.y = y;
    q.rbar = rbar;
    q.nproj = (size_t)Pl->g.nx * Pl->g.nz * Pl->g.nview;
    q.err = Pl->err;
}

// append plan m's grid (gx x gy x gz blocks) to a grouped launch's block ranges
void add_grid(GroupGrid& gg, int m, int gx, int gy, int gz)
{
    if (m == 0) gg.first[0] = 0;
    gg.gx[m] = gx;
    gg.gy[m] = gy;
    gg.first[m + 1] = gg.first[m] + gx * gy * gz;
    gg.n = m + 1;
}

template <class K, class A>
GroupLaunch make_launch(K kern, const A& args, dim3 threads, size_t smem)
{
    const unsigned blocks = (unsigned)args.grid.first[args.grid.n];
    return [=](cudaStream_t st) -> cudaError_t {
        if (smem > 48 * 1024) {
            cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
            if (e != cudaSuccess) return e;
        }
        kern<<<blocks, threads, smem, st>>>(args);
        return cudaGetLastError();
    };
}

// the launches of one stage for the plans `idx` of bucket P
template <int P>
cudaError_t stage_launches(int stage, const std::vector<int>& idx, const std::vector<spect_plan_s*>& plans,
                           const float* const* y, const float* const* rbar, GroupedBatch& /*B*/,
                           std::vector<GroupLaunch>& out)
{
    // sub-groups by kernel variant: the forward blur's sums in registers or not
    std::vector<int> var[2];
    for (int i : idx) {
        bool flag = false;
        if (stage == 1)
            flag = fwd_dims<P>(plans[i]->g, plans[i]->fused_J, plans[i]->fwd_nT, (size_t)plans[i]->smem_optin).racc;
        var[flag ? 1 : 0].push_back(i);
    }
    for (int f = 0; f < 2; ++f) {
        for (const std::vector<int>& ch : chunks_of(var[f], plans)) {
            GroupPlans gp{};
            size_t smem = 0;
            int thr = 0;  // threads per block: the largest of the plans'
            for (int m = 0; m < (int)ch.size(); ++m) {
                const spect_plan_s* Pl = plans[ch[m]];
                fill_plan<P>(gp.p[m], Pl, y[ch[m]], rbar ? rbar[ch[m]] : nullptr);
                const GroupPlan& q = gp.p[m];
                if (stage == 1) {  // the forward blur's grid: (depth group and column tile, view)
                    smem = std::max(smem, smem_fwd<P>(q.df));
                    thr = std::max(thr, q.df.T);
                    gp.fmap[m] = Pl->fmap;
                    add_grid(gp.grid, m, q.df.G * q.df.nT, q.g.nview, 1);
                } else {           // the adjoint's grid: (depth group and column tile, view)
                    smem = std::max(smem, smem_adj<P>(q.da));
                    thr = std::max(thr, q.da.T);
                    gp.mmap[m] = Pl->amap_mu;
                    gp.tmap[m] = Pl->amap_t;
                    const cudaError_t e = encode_v_map(Pl->g, q.da, Pl->ratio, &gp.vmap[m]);
                    if (e != cudaSuccess) return e;
                    add_grid(gp.grid, m, q.da.G * q.da.nT, q.g.nview, 1);
                }
            }
            if (ch.empty()) continue;
            if (stage == 1)
                out.push_back(f ? make_launch(k_fwd_sep_grp<P, true>, gp, dim3(thr), smem)
                                : make_launch(k_fwd_sep_grp<P, false>, gp, dim3(thr), smem));
            else
                out.push_back(make_launch(k_adj_sep_grp<P>, gp, dim3(thr), smem));
        }
    }
    return cudaSuccess;
}

cudaError_t stage_by_bucket(int stage, const std::vector<spect_plan_s*>& plans, const float* const* y,
                            const float* const* rbar, GroupedBatch& B, std::vector<GroupLaunch>& out)
{
    for (int b : kBuckets) {
        std::vector<int> idx;
        for (int i = 0; i < (int)plans.size(); ++i)
            if (plans[i]->bucket == b) idx.push_back(i);
        if (idx.empty()) continue;
        cudaError_t e = cudaErrorInvalidValue;
        switch (b) {
#define SPECT_GB(B_)                                                      \
    case B_: e = stage_launches<B_>(stage, idx, plans, y, rbar, B, out); \
        break;
            SPECT_GB(3) SPECT_GB(5) SPECT_GB(7) SPECT_GB(9) SPECT_GB(11) SPECT_GB(13) SPECT_GB(15) SPECT_GB(17)
            SPECT_GB(21) SPECT_GB(25) SPECT_GB(29) SPECT_GB(33) SPECT_GB(37)
#undef SPECT_GB
            default: break;
        }
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

// the depth-group reduce with the EM ratio, all plans (any bucket)
cudaError_t reduce_launches(const std::vector<spect_plan_s*>& plans, const float* const* y, const float* const* rbar,
                            GroupedBatch& /*B*/, std::vector<GroupLaunch>& out)
{
    std::vector<int> all(plans.size());
    std::iota(all.begin(), all.end(), 0);
    for (const std::vector<int>& ch : chunks_of(all, plans)) {
        GroupPlans gp{};
        for (int m = 0; m < (int)ch.size(); ++m) {
            const spect_plan_s* Pl = plans[ch[m]];
            GroupPlan& q = gp.p[m];
            q.g = Pl->g;
            q.df.G = fused_groups(*Pl);
            q.part = Pl->part;
            q.ratio = Pl->ratio;
            q.y = y[ch[m]];
            q.rbar = rbar ? rbar[ch[m]] : nullptr;
            q.nproj = (size_t)Pl->g.nx * Pl->g.nz * Pl->g.nview;
            add_grid(gp.grid, m, (int)((q.nproj + kReduceThreads - 1) / kReduceThreads), 1, 1);
        }
        out.push_back(make_launch(k_fwd_reduce_grp, gp, dim3(kReduceThreads), 0));
    }
    return cudaSuccess;
}

// rotation + attenuation, all plans (any bucket): the grid is (planes and column run, view)
cudaError_t rotate_launches(const std::vector<spect_plan_s*>& plans, std::vector<GroupLaunch>& out)
{
    std::vector<int> all(plans.size());
    std::iota(all.begin(), all.end(), 0);
    for (const std::vector<int>& ch : chunks_of(all, plans)) {
        GroupPlans gp{};
        for (int m = 0; m < (int)ch.size(); ++m) {
            const spect_plan_s* Pl = plans[ch[m]];
            GroupPlan& q = gp.p[m];
            q.g = Pl->g;
            q.dr = rot_dims(Pl->g, Pl->ps, Pl->ts, Pl->g.nview, Pl->sms);
            q.rtab = Pl->rtab;
            q.xt = Pl->xt;
            q.mubar = Pl->mubar;
            q.slab = Pl->slab;
            add_grid(gp.grid, m, q.dr.nb * ((q.g.ny + q.dr.JP - 1) / q.dr.JP), q.g.nview, 1);
        }
        out.push_back(make_launch(k_rot_fwd_grp, gp, dim3(kRotThreads), 0));
    }
    return cudaSuccess;
}

// x (image layout) <-> x_t ([j][i][k]) for every plan: to_internal / from_internal
cudaError_t transpose_launches(const std::vector<spect_plan_s*>& plans, float* const* x, bool to_internal,
                               GroupedBatch& /*B*/, std::vector<GroupLaunch>& out)
{
    std::vector<int> all(plans.size());
    std::iota(all.begin(), all.end(), 0);
    for (const std::vector<int>& ch : chunks_of(all, plans)) {
        GroupTs gt{};
        for (int m = 0; m < (int)ch.size(); ++m) {
            const spect_plan_s* Pl = plans[ch[m]];
            const int nxy = Pl->g.nx * Pl->g.ny, nz = Pl->g.nz;
            GroupT& q = gt.p[m];
            q.in = to_internal ? x[ch[m]] : Pl->xt;
            q.out = to_internal ? Pl->xt : x[ch[m]];
            q.R = to_internal ? nz : nxy;
            q.C = to_internal ? nxy : nz;
            q.ip = to_internal ? nxy : Pl->g.kp;
            q.op = to_internal ? Pl->g.kp : nxy;
            add_grid(gt.grid, m, (q.C + 31) / 32, (q.R + 31) / 32, 1);
        }
        out.push_back(make_launch(k_transpose_grp, gt, dim3(32, 8), 0));
    }
    return cudaSuccess;
}

}  // namespace

bool groupable(const spect_plan_s& P)
{
    return P.fast && P.separable && !P.rot3 && !P.recompute && P.gather && P.bucket > 0 && P.chunk >= P.g.nview &&
           P.adj_chunk >= P.g.nview;
}

cudaError_t build_grouped(const std::vector<spect_plan_s*>& plans, float* const* x, const float* const* y,
                          const float* const* rbar, GroupedBatch& B)
{
    cudaError_t e = transpose_launches(plans, x, true, B, B.head);
    if (e == cudaSuccess) e = rotate_launches(plans, B.iter);
    if (e == cudaSuccess) e = stage_by_bucket(1, plans, y, rbar, B, B.iter);
    if (e == cudaSuccess) e = reduce_launches(plans, y, rbar, B, B.iter);
    if (e == cudaSuccess) e = stage_by_bucket(2, plans, y, rbar, B, B.iter);
    if (e == cudaSuccess) e = build_grouped_gather(plans, B, B.iter);
    if (e == cudaSuccess) e = transpose_launches(plans, const_cast<float* const*>(x), false, B, B.tail);
    return e;
}

void free_grouped(GroupedBatch& B)
{
    B.head.clear();
    B.iter.clear();
    B.tail.clear();
}

}  // namespace spect
