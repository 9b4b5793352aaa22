// Host plan of the neighbour-list path (ksg_lists.cu): every group of a batch
// in a few launches, with the lists of at most kListPoolBytes of query points
// in device memory at a time.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstring>
#include <map>
#include <tuple>
#include <utility>
#include <vector>

#include "ksg_lists.h"
#include "te_runtime.h"

namespace teksg {

namespace {

// Lists in device memory at once: enough points to fill the chip several
// times over at the longest lists (48 KB a point), small beside the X values.
constexpr size_t kListPoolBytes = (size_t)256 << 20;

size_t align256(size_t b) { return (b + 255) & ~(size_t)255; }

// Groups of one walk variant.
struct ClassPlan {
    int first_group = 0;
    ListShape shape{};
    size_t smem = 0;
};

// Segments whose lists are in the pool together: one build and one walk launch.
struct Chunk {
    int cls = 0, first_seg = 0, n_segs = 0;
    long long build_items = 0, walk_items = 0;
    int queries = 1, cap_a = 0, cap_b = 0;
};

}  // namespace

te_status launch_groups_lists(te_ctx *ctx, const std::vector<HostGroup> &groups, int n_out,
                              int dbg_out, float *dbg_eps, int *dbg_nxz, int *dbg_nyz,
                              int *dbg_nz)
{
    te_status st;
    int sms = 0;
    CK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, ctx->device),
       "cudaDeviceGetAttribute");
    std::map<ListShape, std::vector<const HostGroup *>> classes;
    for (const HostGroup &g : groups)
        if (!g.members.empty())
            classes[list_shape(g.data->T - g.max_lag, g.dx, (int)g.z.size(), g.k,
                               g.members.size())]
                .push_back(&g);

    std::vector<ListGroup> lg;
    std::vector<MemberDesc> mdesc;
    std::vector<std::pair<size_t, int>> msorted;       // (member, job)
    std::vector<int> cols;
    std::vector<ListSeg> segs;
    std::vector<size_t> seg_off;                       // bytes into the pool
    std::vector<Chunk> chunks;
    std::vector<ClassPlan> plans;
    // sorted columns: (data, column, points) -> job; a job's sorted values and
    // its ranks lie at job_off and job_off + N (rounded up) words of ws_vsort
    std::vector<RankSortJob> vjobs;
    std::vector<size_t> vjob_off;
    std::map<std::tuple<const te_data *, int, int>, int> vsorted;
    std::vector<std::pair<size_t, int>> zjob;          // (group, job)
    size_t vs_words = 0, pool = 0;
    uint64_t pair_evals = 0, members_total = 0;
    for (auto &kv : classes) {
        ClassPlan cp;
        cp.first_group = (int)lg.size();
        cp.shape = kv.first;
        for (const HostGroup *g : kv.second)
            cp.smem = std::max(cp.smem, list_walk_x_bytes(g->data->T - g->max_lag, g->dx,
                                                          (int)g->z.size(), g->k,
                                                          cp.shape.width));
        Chunk ch;
        size_t used = 0;
        auto close_chunk = [&]() {
            ch.queries = list_build_queries(ch.cap_a, ch.cap_b);
            long long blocks = 0;
            int max_nq = 1;
            for (int s = ch.first_seg; s < ch.first_seg + ch.n_segs; ++s) {
                blocks += lg[cp.first_group + segs[s].group].n_mblocks;
                max_nq = std::max(max_nq, segs[s].nq);
            }
            const int splits = list_splits(blocks, max_nq, cp.smem, sms);
            for (int s = ch.first_seg; s < ch.first_seg + ch.n_segs; ++s) {
                segs[s].build_item = ch.build_items;
                ch.build_items += (segs[s].nq + ch.queries - 1) / ch.queries;
                segs[s].walk_item = ch.walk_items;
                segs[s].per_cta = (segs[s].nq + splits - 1) / splits;
                segs[s].n_splits = (segs[s].nq + segs[s].per_cta - 1) / segs[s].per_cta;
                ch.walk_items += (long long)segs[s].n_splits *
                                 lg[cp.first_group + segs[s].group].n_mblocks;
            }
            if (ch.n_segs) chunks.push_back(ch);
            pool = std::max(pool, used);
            ch = Chunk();
            used = 0;
        };
        for (const HostGroup *hg : kv.second) {
            const HostGroup &g = *hg;
            const te_data *d = g.data;
            const int N = d->T - g.max_lag;
            auto off = [&](te_var v) { return v.proc * d->T + g.max_lag - v.lag; };
            ListGroup G{};
            G.base = d->d_series;
            G.N = N;
            G.k = g.k;
            G.theiler = g.theiler;
            G.dy = (int)g.y.size();
            G.dz = (int)g.z.size();
            G.dx = g.dx;
            G.ycol = (int)cols.size();
            for (te_var v : g.y) cols.push_back(off(v));
            G.zcol = (int)cols.size();
            for (te_var v : g.z) cols.push_back(off(v));
            const int xbase = (int)cols.size();
            for (te_var v : g.xvars) cols.push_back(off(v));
            auto sorted_job = [&](int column) {
                auto ins = vsorted.emplace(std::make_tuple(d, column, N), (int)vjobs.size());
                if (ins.second) {
                    vjobs.push_back(RankSortJob{d->d_series + column, nullptr, nullptr, N, 0});
                    vjob_off.push_back(vs_words);
                    vs_words += 2 * (((size_t)N + 3) & ~(size_t)3);
                }
                return ins.first->second;
            };
            if (G.dz == 1) zjob.emplace_back(lg.size(), sorted_job(off(g.z[0])));
            // empty Z and one X variable: n_xz is a range count in the sorted
            // X column (a permutation only reorders its values)
            const bool xsorted = g.z.empty() && g.dx == 1;
            G.member_begin = (int)mdesc.size();
            G.n_members = (int)g.members.size();
            G.n_mblocks = (G.n_members + cp.shape.width - 1) / cp.shape.width;
            for (const HostMember &hm : g.members) {
                if (xsorted)
                    msorted.emplace_back(mdesc.size(), sorted_job(off(g.xvars[hm.xcol_first])));
                mdesc.push_back(MemberDesc{hm.perm, xbase + hm.xcol_first, hm.out, nullptr});
            }
            list_caps(N, g.k, g.dx, G.dy, G.dz, &G.cap_a, &G.cap_b);
            lg.push_back(G);
            const size_t row = list_row_bytes(G.cap_a, G.cap_b);
            for (int q0 = 0; q0 < N;) {
                const size_t room = kListPoolBytes - std::min(kListPoolBytes, used + 256);
                int nq = (int)std::min<size_t>((size_t)(N - q0), room / row);
                if (nq < N - q0) nq &= ~31;
                if (nq <= 0) {
                    close_chunk();
                    continue;
                }
                if (!ch.n_segs) {
                    ch.cls = (int)plans.size();
                    ch.first_seg = (int)segs.size();
                }
                ListSeg s{};
                s.group = (int)lg.size() - 1 - cp.first_group;
                s.q0 = q0;
                s.nq = nq;
                segs.push_back(s);
                seg_off.push_back(used);
                used += align256(nq * row);
                ch.n_segs++;
                ch.cap_a = std::max(ch.cap_a, G.cap_a);
                ch.cap_b = std::max(ch.cap_b, G.cap_b);
                q0 += nq;
            }
            pair_evals += (uint64_t)g.members.size() * 2ull * (uint64_t)N * (uint64_t)(N - 1);
            members_total += g.members.size();
        }
        close_chunk();
        plans.push_back(cp);
    }
    if (plans.empty()) {
        CK(launch_finalize((const unsigned long long *)ctx->ws_acc.p, (long long *)ctx->ws_keys.p,
                           n_out, ctx->stream),
           "finalize launch");
        return TE_OK;
    }

    // workspaces, then the pointers into them, then one upload of all tables
    if ((st = ensure_dev(ctx, ctx->ws_lists, pool))) return st;
    if (vs_words && (st = ensure_dev(ctx, ctx->ws_vsort, vs_words * 4))) return st;
    int vitems = 0;
    for (size_t a = 0; a < vjobs.size(); ++a) {
        RankSortJob &J = vjobs[a];
        J.sorted = (float *)ctx->ws_vsort.p + vjob_off[a];
        J.rank = (int *)(J.sorted + (((size_t)J.N + 3) & ~(size_t)3));
        J.item = vitems;
        vitems += rank_sort_items(J.N);
    }
    for (auto &z : zjob) {
        lg[z.first].zs = vjobs[z.second].sorted;
        lg[z.first].rank = vjobs[z.second].rank;
    }
    for (size_t a = 0; a < segs.size(); ++a)
        segs[a].rows = (unsigned char *)ctx->ws_lists.p + seg_off[a];
    for (auto &ms : msorted) mdesc[ms.first].xsorted = vjobs[ms.second].sorted;
    struct Table {
        const void *src;
        size_t bytes, at;
    } tab[] = {{lg.data(), lg.size() * sizeof(ListGroup), 0},
               {segs.data(), segs.size() * sizeof(ListSeg), 0},
               {mdesc.data(), mdesc.size() * sizeof(MemberDesc), 0},
               {vjobs.data(), vjobs.size() * sizeof(RankSortJob), 0},
               {cols.data(), cols.size() * sizeof(int), 0}};
    size_t bytes = 0;
    for (Table &t : tab) {
        t.at = bytes;
        bytes += (t.bytes + 15) & ~(size_t)15;
    }
    if ((st = ensure_pin(ctx, bytes))) return st;
    if ((st = ensure_dev(ctx, ctx->ws_groups, bytes))) return st;
    for (const Table &t : tab)
        if (t.bytes) std::memcpy((char *)ctx->pin + t.at, t.src, t.bytes);
    CK(copy_h2d(ctx, ctx->ws_groups.p, ctx->pin, bytes), "cudaMemcpyAsync");
    char *dtab = (char *)ctx->ws_groups.p;
    for (const Chunk &ch : chunks)
        CK(list_prepare(plans[ch.cls].shape, ch.queries, &ctx->prepared_lists),
           "cudaFuncSetAttribute");

    const bool graph = ctx->opt_graph != 0;
    auto device_work = [&]() -> te_status {
        if (!vjobs.empty()) {
            CK(launch_rank_sort((const RankSortJob *)(dtab + tab[3].at), (int)vjobs.size(), vitems,
                                ctx->stream),
               "column sort launch");
            ctx->stats.launches++;
        }
        CK(cudaMemsetAsync(ctx->work_dev, 0, 3 * sizeof(unsigned long long), ctx->stream),
           "cudaMemsetAsync");
        if (!graph) CK(cudaEventRecord(ctx->ev_a, ctx->stream), "cudaEventRecord");
        auto launch_args = [&](const ClassPlan &cp) {
            ListLaunch L{};
            L.groups = (const ListGroup *)(dtab + tab[0].at) + cp.first_group;
            L.members = (const MemberDesc *)(dtab + tab[2].at);
            L.cols = (const int *)(dtab + tab[4].at);
            L.q = ctx->q_dev;
            L.acc = (unsigned long long *)ctx->ws_acc.p;
            L.dbg_eps = dbg_eps;
            L.dbg_nxz = dbg_nxz;
            L.dbg_nyz = dbg_nyz;
            L.dbg_nz = dbg_nz;
            L.dbg_out = dbg_out;
            L.work = ctx->work_dev;
            return L;
        };
        for (const Chunk &ch : chunks) {
            const ClassPlan &cp = plans[ch.cls];
            ListLaunch L = launch_args(cp);
            L.segs = (const ListSeg *)(dtab + tab[1].at) + ch.first_seg;
            L.n_segs = ch.n_segs;
            CK(launch_list_build(L, ch.build_items, ch.queries, ch.cap_a, ch.cap_b, ctx->stream),
               "list build launch");
            CK(launch_list_walk(L, ch.walk_items, cp.shape, cp.smem, ctx->stream),
               "list walk launch");
            ctx->stats.launches += 2;
            ctx->stats.ksg_launches++;
        }
        if (!graph) CK(cudaEventRecord(ctx->ev_b, ctx->stream), "cudaEventRecord");
        CK(copy_d2h(ctx, ctx->work_host, ctx->work_dev, 3 * sizeof(unsigned long long)),
           "cudaMemcpyAsync");
        CK(launch_finalize((const unsigned long long *)ctx->ws_acc.p,
                           (long long *)ctx->ws_keys.p, n_out, ctx->stream),
           "finalize launch");
        ctx->stats.launches++;
        return TE_OK;
    };
    if ((st = submit_work(ctx, device_work))) return st;
    ctx->pend_timed = 1;
    ctx->pend_pair_evals = pair_evals;
    ctx->pend_members = members_total;
    return TE_OK;
}

}  // namespace teksg
