// Neighbour-list form of the KSG estimator: interface between the host plans
// (te_lists.cu, te_static.cu) and the kernels (ksg_lists.cu).
#pragma once

#include <tuple>

#include "ksg_internal.h"

namespace teksg {

// Lists of one query point, one row of memory (list_row_bytes):
//   ListNear | A skip | B skip | A distances | A points | B distances | B points
// A holds exactly the valid points with d_YZ < ra, ascending by d_YZ, B those
// with d_Z < rb, ascending by d_Z; distances are float, points byte offsets
// into a row of X values (as the walk's shared-memory loads take them).  Both are padded to a
// multiple of 32 entries with (+inf, 0).  skip[b] is a list's distance 32 b,
// +inf past its end.  ListNear repeats the beginning of both (+inf past their
// ends): what most points need, in one piece that the walk copies ahead.
//
// Point j's place in a row of X values is j, and for one Z variable its rank
// in the Z column: the points with d_Z < eps are then consecutive, and the
// group has no list B.
constexpr int kNearA = 32, kNearB = 64;
struct __align__(16) ListNear {
    float ra, rb;
    uint16_t na, nb;   // entries, padding included
    float far_a, far_b;   // A's distance kNearA, B's distance kNearB (+inf past their ends)
    uint32_t place;       // byte offset of the query point itself
    uint32_t pad[2];
    float da[kNearA];
    uint32_t oa[kNearA];
    float db[kNearB];
    uint32_t ob[kNearB];
};
static_assert(sizeof(ListNear) % 16 == 0, "copied in 16-byte pieces");
constexpr int kListCapA = 2048, kListCapB = 4096;   // largest lists
constexpr int kSkipA = kListCapA / 32, kSkipB = kListCapB / 32;
constexpr size_t kListWalkSmem = 164 * 1024;   // X values of a walking CTA
constexpr size_t kListHalfSmem = 72 * 1024;    // of each of two CTAs on an SM

__host__ __device__ inline size_t list_row_bytes(int cap_a, int cap_b)
{
    return sizeof(ListNear) + 4 * (kSkipA + kSkipB) + 8 * (size_t)(cap_a + cap_b);
}

// A group of members (as GroupDesc) on the list path; member block b holds
// members b * width .. of the group.
struct ListGroup {
    const float *base;
    int N, k, theiler;
    int dy, dz, dx;
    int ycol, zcol;          // first index into cols[] of the Y / Z column offsets
    int member_begin, n_members, n_mblocks;
    int cap_a, cap_b;        // list capacities, multiples of 32; cap_b = 0 when dz < 2
    const float *zs;         // dz == 1: the Z column ascending, every point's rank in it
    const int *rank;
};

// Query points q0 .. q0 + nq - 1 of one group, whose lists are in the pool at
// once (a launch works through the points in such segments).
struct ListSeg {
    int group, q0, nq;
    int per_cta;             // query points per walking CTA
    int n_splits;            // walking CTAs per member block
    long long build_item, walk_item;   // first CTA in the build / walk launch
    unsigned char *rows;     // nq rows
};

struct ListLaunch {
    const ListGroup *groups;
    const ListSeg *segs;
    int n_segs;
    const MemberDesc *members;
    const int *cols;
    const int64_t *q;
    unsigned long long *acc;
    float *dbg_eps;
    int *dbg_nxz, *dbg_nyz, *dbg_nz;
    int dbg_out;
    unsigned long long *work;   // as KsgLaunch::work [0], [1]; nullptr: not counted
    // per group of the launch: set by a walking CTA that gives it up because more
    // than its share of pairs (list_slow_limit) lies beyond the radii; n_bad:
    // groups given up.  nullptr: none is.
    unsigned *bad;
    unsigned long long *n_bad;
    unsigned *nonfinite;        // set if a value is not finite; nullptr: checked by the caller
};

constexpr int kListBuildThreads = 512;
constexpr int kListWalkThreads = 1024;   // of all walking CTAs on an SM

// Pairs beyond the lists' radii that a walking CTA with `pairs` of them scans,
// before it gives its group of m members up. A scan visits every point twice;
// what the other kernel takes a pair depends on how well it fills the chip and
// prunes (not with a Theiler window or past kMaxOrderN), and on the data, whose
// tails slow it too.  The shares are where lists and scans lost to it in most
// of 5568 measured groups (normal, heavy-tailed, rounded, zero-inflated, binary
// values). Member lanes / lists below and above the share, medians: m >= 61, N >=
// 6000 1.2 / 0.22, 800 to 6000 1.3 / 0.1; m of 13 to 60 1.3 / 0.2; 2 to 12 1.7 /
// 0.35 (unpruned 1.6 / 0.5); one member 2.5 / 0.9 (unpruned 1.4 at every share);
// several X variables, N >= 3000, m >= 61 1.4 / 0.25, 13 to 60 1.3 / 0.4, 2 to 12 1.8 / 0.5.
__host__ __device__ inline int list_slow_limit(int pairs, int N, int dx, int m, bool pruned)
{
    float share = 2.f;   // never
    if (dx == 1) {
        if (m >= 13) share = N < 800 ? 0.5f : m >= 61 && N >= 6000 ? 0.12f : 0.2f;
        else if (m > 1) share = N < 800 ? 0.5f : pruned ? 0.3f : 0.4f;
        else if (pruned) share = 0.6f;
    } else if (m >= 13) {
        share = m >= 61 ? (N >= 3000 ? 0.45f : N >= 800 ? 0.6f : 0.9f) : N >= 3000 ? 0.5f : 0.9f;
    } else if (m > 1 && N >= 3000) {
        share = 0.8f;
    }
    // (a CTA of few pairs needs most of them to judge by)
    return max(pairs < 256 ? 16 : 64, (int)((float)pairs * (pairs < 256 ? fmaxf(share, 0.5f) : share)));
}

// capacities of the two lists for a group
void list_caps(int N, int k, int dx, int dy, int dz, int *cap_a, int *cap_b);
// Walk variant of a group: lanes per (point, member) pair, members per CTA, X
// storage (1, 2, 4: a point's dimensions together; 0: a row per dimension),
// k = 4.
struct ListShape {
    int lanes, width, dxp;
    bool k4;
    bool operator<(const ListShape &o) const
    {
        return std::tie(lanes, width, dxp, k4) < std::tie(o.lanes, o.width, o.dxp, o.k4);
    }
};
ListShape list_shape(int N, int dx, int dz, int k, size_t members);
// shared memory of a walking CTA: X values of width members, and every 16th
// value of the sorted columns that the group's counts search
size_t list_walk_x_bytes(int N, int dx, int dz, int k, int width);
// whether neighbour lists are the faster path for a group of a batch of
// n_groups with `rows` points and `pairs` (member, point) pairs in all
struct ListCall {
    int N, k, theiler, dx, dy, dz;
    size_t members;
};
bool list_serves(const ListCall &c, int n_groups, long long rows, long long pairs);
size_t list_bytes(const ListCall &c);   // of the group's lists, all in the pool
// A batch whose lists do not all fit the pool needs this much of it: smaller
// pieces leave the chip idle at the end of each. Member lanes / lists with
// 64, 32 and 16 MiB, ms: 40 groups of 201 members, N = 10^4, two Z variables 128 /
// 120, 163, 247 (one group 5.9 / 3.2, 4.3, 6.3; 45 candidates 102 / 40, 45, 55),
// N = 3000 20.6 / 16.3, 19.8, 26.2; one group of 41 3.0 / 2.1, 2.9, 4.3.
constexpr size_t kListPoolLeast = (size_t)64 << 20;
// whether a group can take the list path
bool list_fits(int N, int dx, int dz, int k);
// Parts into which the walk splits the points of a launch, given its member
// blocks, the most points of a segment, its CTAs' X bytes and the SM count
int list_splits(long long blocks, int max_nq, size_t smem, int sms);
// queries per CTA of the build kernel
int list_build_queries(int cap_a, int cap_b);

// Ascending copies of columns (sorted) and the points' ranks in them (rank;
// either may be nullptr), equal values in the order of their points.
struct RankSortJob {
    const float *src;
    float *sorted;
    int *rank;
    int N;
    int item;   // first CTA of the job: rank_sort_items(N) each
};
inline int rank_sort_items(int N) { return (N + 63) / 64; }
cudaError_t launch_rank_sort(const RankSortJob *jobs, int n_jobs, int n_items, cudaStream_t st);

// Kernel attributes before the first launch on a device: of every kernel, or
// of those a chunk uses that are not marked in *done yet (loading all of them
// takes longer than a small call).
cudaError_t list_prepare_attributes();
cudaError_t list_prepare(const ListShape &s, int queries, uint64_t *done);
cudaError_t launch_list_build(const ListLaunch &L, long long n_items, int queries, int cap_a,
                              int cap_b, cudaStream_t st);
// smem: the largest list_walk_x_bytes of the launch's groups, all of shape s
cudaError_t launch_list_walk(const ListLaunch &L, long long n_items, const ListShape &s,
                             size_t smem, cudaStream_t st);

}  // namespace teksg
