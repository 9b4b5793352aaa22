// Host plan of the neighbour-list path (ksg_lists.cu): every group of a batch
// in a few launches, with at most ctx->list_pool bytes of lists in device memory
// at a time.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <map>
#include <tuple>
#include <utility>
#include <vector>

#include "ksg_lists.h"
#include "te_runtime.h"

namespace teksg {

namespace {

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

static bool list_serves_other_k(const ListCall &c, int n_groups, bool full);

// mean n_yz of a member's k nearest: how deep in list A they lie
static double list_depth(const ListCall &c)
{
    return c.N * std::pow((double)c.k / c.N, (double)(c.dy + c.dz) / (c.dx + c.dy + c.dz));
}

// Measured line between the two paths (whole calls on one GB300, member-lane
// or fused kernel / lists, microseconds).  Lists pay for themselves by a row
// per point that all members of the group walk; the member-lane kernel shares
// its tiles among 32 members (64 from 64 on) and wins
// - over an empty Z, where n_z needs no list and n_xz is a range count for
//   either, once the chip is full: 2000 members at N = 10^4 13,700 / 15,800, 9045
//   57,900 / 66,700, 401 2940 / 2120; 12 groups of 64 at N = 2000 719 / 1572;
// - where few members share a row and there are many groups: 64 groups of 21,
//   N = 4000: one Z 8005 / 12,670, two 8323 / 21,559 (their lists are the longest),
//   three 9317 / 13,002, five 12,134 / 9605; one group of 21 933 / 401, 64 of 201
//   at N = 1000 and two Z 7095 / 4901.
// Several X variables: a member's neighbours lie the deeper in list A the fewer
// Y and Z variables there are, and pairs beyond its capacity scan all points.
// The line is at the expected depth: 201 members at N = 9000, k = 4, empty Z, two X
// variables (depth 686) 17,220 / 18,689, four (1922) 28,342 / 147,900; one Z and four
// (686) equal; two Z 3.3 to 7 times in the lists' favour.
bool list_serves(const ListCall &c, int n_groups, long long rows, long long pairs)
{
    const int N = c.N, dz = c.dz;
    const long long m = (long long)c.members;
    if (!list_fits(N, c.dx, dz, c.k)) return false;
    const bool full = rows >= 24000;   // points of all groups: several waves of CTAs
    if (c.dx == 1 && (c.theiler > 0 || N > kMaxOrderN))
        return true;   // the member lanes cannot prune then
    // (a point's X values one by one in shared memory: as with another k)
    if (c.k != 4 || list_shape(N, c.dx, dz, c.k, c.members).dxp == 0)
        return list_serves_other_k(c, n_groups, full);
    if (c.dx > 1)
        return dz > 1 || m < 8 || list_depth(c) <= (dz == 1 ? 680 : m >= 64 ? 650 : 1150);
    const bool block = m <= 32 || (m >= 48 && m <= 64);   // one well-filled block of members
    if (n_groups >= 200 && m <= 8 && N <= 700 && dz > 0) return false;
    if (N < 250) return true;
    switch (dz) {
    case 0:
        return !((pairs >= 1600LL * N && N >= 700) ||
                 (n_groups >= 4 && rows >= 8000 && m >= 16 && (N >= 350 || m <= 64)) ||
                 (full && (m >= 4 || N <= 3000) && (N >= 350 || m <= 64)));
    case 1:
        return !(full && block && n_groups >= (m >= 16 ? 10 : 32) && (m >= 4 || N <= 3000));
    case 2:
        return !(full && (block || (m < 64 && N >= 3500)) &&
                 n_groups >= (m >= 16 ? (N >= 3500 ? 5 : 10)
                                      : N >= 3500 ? 8 : N >= 1500 ? 16 : 32));
    case 3:
        return !(full && block && n_groups >= (m >= 16 && N >= 3500 ? 12 : 32));
    case 4:
    case 5:
        return !(full && m <= 32 && n_groups >= 64 && N <= (dz == 4 ? 1500 : 700));
    default:
        return !(full && m <= 32 && n_groups >= 200 && N <= 700);
    }
}

// With another k the member-lane kernel keeps its k smallest by insertion and
// takes about 1.6 times as long as with four, the lists hardly longer; the fused
// kernel serves two members at a time and, from k = 9 on, its longer buffer. The
// lines are those of 2130 measured sizes (k 1 to 16, one to six X variables, 1 to
// 9045 members): 11 of them are 6 to 12% faster on the other side.
// Member lanes / lists, one X variable: 9 groups of 201, N = 4000, empty Z, k = 3
// and 9: 1.90 and 1.43; 64 of 5, N = 9990 0.90 and 1.02; 64 of 21, N = 8000, two Z
// 0.70 and 0.86, three 1.30 and 0.94, five 2.5 and 2.0. Fused / lists: four X,
// one Z, 201 members, N = 2200, k = 3 and 9 0.67 and 1.47; 21 members 1.24 and 1.89;
// three X, empty Z, 12 members, N = 2200, 4000, 9000, k = 5 1.92, 1.48, 0.53; five X,
// empty Z, k = 4, 29 members, N = 2500 1.46, 201, N = 700 0.75.
static bool list_serves_other_k(const ListCall &c, int n_groups, bool full)
{
    const int N = c.N, dz = c.dz, k = c.k;
    const double m = (double)c.members;
    if (c.dx == 1) {
        if (dz == 0)
            return !(full && m >= 4 && m < 16 && N >= 1500 &&
                     k <= (N < 3000 ? 8 : N < 6000 ? 6 : 3));
        return !(dz == 2 && k > 1 && k <= 9 && full && N >= 3500 && m >= 4 && m <= 32 &&
                 n_groups >= 8);
    }
    if (dz > 1 || m < 8 || N < 150) return true;
    const double depth = list_depth(c);
    if (dz == 0) {
        if (m <= 100) return depth * m * N <= 6.5e7;
        return (k == 4 && N < 400) || (N <= (c.dx == 2 ? 2500 : 1500) && (c.dx <= 3 || k > 8));
    }
    if (k > 8) return m >= 48 ? depth <= 860 : depth * N <= 8e6;
    if (m < 48) return depth * N <= 6.5e6;
    if (m < 100) return c.dx == 2 || N < 600 || (c.dx == 3 && (N < 1500 || (N > 3000 && k <= 3)));
    return c.dx == 2 && (k <= 2 || N >= 5000);
}

size_t list_bytes(const ListCall &c)
{
    int cap_a, cap_b;
    list_caps(c.N, c.k, c.dx, c.dy, c.dz, &cap_a, &cap_b);
    return (size_t)c.N * list_row_bytes(cap_a, cap_b) + 512;   // a piece begins at 256 bytes
}

te_status prepare_lists(te_ctx *ctx, const std::vector<const HostGroup *> &groups,
                        const KsgDebug &dbg, KsgPart &part)
{
    te_status st;
    std::map<ListShape, std::vector<const HostGroup *>> classes;
    for (const HostGroup *g : groups)
        classes[list_shape(g->data->T - g->max_lag, g->dx, (int)g->z.size(), g->k,
                           g->members.size())]
            .push_back(g);

    std::vector<ListGroup> lg;
    std::vector<const HostGroup *> order;              // lg's groups
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
            const int splits = list_splits(blocks, max_nq, cp.smem, ctx->sms);
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
            order.push_back(hg);
            const size_t row = list_row_bytes(G.cap_a, G.cap_b);
            for (int q0 = 0; q0 < N;) {
                const size_t room = ctx->list_pool - std::min(ctx->list_pool, used + 256);
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
    // workspaces, then the pointers into them, then one upload of all tables
    if ((st = ensure_dev(ctx, ctx->ws_lists, pool, ctx->list_pool))) return st;
    if (vs_words && (st = ensure_dev(ctx, ctx->ws_lsort, vs_words * 4))) return st;
    int vitems = 0;
    for (size_t a = 0; a < vjobs.size(); ++a) {
        RankSortJob &J = vjobs[a];
        J.sorted = (float *)ctx->ws_lsort.p + vjob_off[a];
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
    const std::vector<unsigned> bad(lg.size(), 0);   // groups given up
    struct Table {
        const void *src;
        size_t bytes, at;
    } tab[] = {{lg.data(), lg.size() * sizeof(ListGroup), 0},
               {segs.data(), segs.size() * sizeof(ListSeg), 0},
               {mdesc.data(), mdesc.size() * sizeof(MemberDesc), 0},
               {vjobs.data(), vjobs.size() * sizeof(RankSortJob), 0},
               {cols.data(), cols.size() * sizeof(int), 0},
               {bad.data(), bad.size() * sizeof(unsigned), 0}};
    size_t bytes = 0;
    for (Table &t : tab) {
        t.at = bytes;
        bytes += (t.bytes + 15) & ~(size_t)15;
    }
    if ((st = ensure_pin_lists(ctx, bytes))) return st;
    if ((st = ensure_dev(ctx, ctx->ws_ltables, bytes))) return st;
    for (const Table &t : tab)
        if (t.bytes) std::memcpy((char *)ctx->pin_lists + t.at, t.src, t.bytes);
    CK(copy_h2d(ctx, ctx->ws_ltables.p, ctx->pin_lists, bytes), "cudaMemcpyAsync");
    char *dtab = (char *)ctx->ws_ltables.p;
    for (const Chunk &ch : chunks)
        CK(list_prepare(plans[ch.cls].shape, ch.queries, &ctx->prepared_lists),
           "cudaFuncSetAttribute");

    part.pair_evals = pair_evals;
    part.members = members_total;
    if (!vjobs.empty())
        part.before = [ctx, jobs = (const RankSortJob *)(dtab + tab[3].at),
                       n = (int)vjobs.size(), vitems]() -> te_status {
            CK(launch_rank_sort(jobs, n, vitems, ctx->stream), "column sort launch");
            ctx->stats.launches++;
            return TE_OK;
        };
    ListLaunch base{};
    base.groups = (const ListGroup *)(dtab + tab[0].at);
    base.segs = (const ListSeg *)(dtab + tab[1].at);
    base.members = (const MemberDesc *)(dtab + tab[2].at);
    base.cols = (const int *)(dtab + tab[4].at);
    base.q = ctx->q_dev;
    base.acc = (unsigned long long *)ctx->ws_acc.p;
    base.dbg_eps = dbg.eps;
    base.dbg_nxz = dbg.nxz;
    base.dbg_nyz = dbg.nyz;
    base.dbg_nz = dbg.nz;
    base.dbg_out = dbg.out;
    base.work = ctx->work_dev;
    if (!ctx->opt_lists) {
        base.bad = (unsigned *)(dtab + tab[5].at);
        base.n_bad = ctx->work_dev + 4;
        ctx->pend_bad = base.bad;
        ctx->pend_lists = std::move(order);
    }
    part.kernels = [ctx, plans = std::move(plans), chunks = std::move(chunks),
                    base]() -> te_status {
        for (const Chunk &ch : chunks) {
            const ClassPlan &cp = plans[ch.cls];
            ListLaunch L = base;
            L.groups += cp.first_group;
            if (L.bad) L.bad += cp.first_group;
            L.segs += ch.first_seg;
            L.n_segs = ch.n_segs;
            CK(launch_list_build(L, ch.build_items, ch.queries, ch.cap_a, ch.cap_b, ctx->stream),
               "list build launch");
            CK(launch_list_walk(L, ch.walk_items, cp.shape, cp.smem, ctx->stream),
               "list walk launch");
            ctx->stats.launches += 2;
            ctx->stats.ksg_launches++;
        }
        return TE_OK;
    };
    return TE_OK;
}

}  // namespace teksg
