// Neighbour lists for the KSG estimator (sm_103a).
//
// The members of a group (candidates x surrogates) share Y, Z and the points
// and differ in X only.  So for every query point the points near it in (Y, Z)
// and in Z are found once per group and kept as two sorted lists; each
// member then needs only a prefix of them:
//   list A, ascending d_YZ: the joint distance is max(d_X, d_YZ) >= d_YZ, so
//     a member's k nearest joint distances are known as soon as the next d_YZ
//     is not below its k-th smallest so far; n_yz is a rank in this list;
//   list B, ascending d_Z: n_z is a rank in it, n_xz a count over the prefix
//     with d_Z < eps.
// A list holds every valid point below its radius and no other, so a result
// is exact whenever the member's k-th distance is at most the radius; the few
// (member, point) pairs beyond it scan all points.  Masked points (the point
// itself, the Theiler band) are in no list.
//
// Per member and point the estimate needs the points inside eps only: 9 for
// the neighbours and 21 for n_z with eight Z variables at N = 10^4, 38 and 229
// with two, 71 and 781 with one, against 900 to 10,000 visited by tiles that
// are pruned for 64 members at once.  Measured on one GB300, tiled member-lane
// kernel -> lists, whole calls: 89 candidates x 201 members, 8 Z variables,
// N = 9995: 277 -> 22.9 ms; 45 x 201, 2 Z: 104 -> 35.9 ms; one call of 201, 1 Z:
// 5.7 -> 2.1 ms; 9 x 201, Theiler window 12, N = 2994: 9.8 -> 1.5 ms.
#include <cuda_runtime.h>
#include <math_constants.h>
#include <stdint.h>

#include <algorithm>
#include <cmath>

#include "ksg_lists.h"

namespace teksg {

namespace {

constexpr int kBins = 1024;          // counting-sort bins per list
constexpr int kSample = 1024;        // points sampled for a list's radius
constexpr int kBuildWarps = kListBuildThreads / 32;
constexpr unsigned kFull = 0xffffffffu;

struct Entry {   // 64 bits: unsigned order is (distance, point) order (distances are >= 0)
    uint32_t j;
    float d;
};

__device__ __forceinline__ uint64_t entry_key(Entry e)
{
    return ((uint64_t)__float_as_uint(e.d) << 32) | e.j;
}

template <typename F>
__device__ __forceinline__ int last_at_or_below(int n, long long item, F first)
{
    int lo = 0, hi = n - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (first(mid) <= item) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

struct RowPtrs {
    ListNear *near;
    float *skip_a, *skip_b, *d_a, *d_b;
    uint32_t *j_a, *j_b;
};

__device__ __forceinline__ RowPtrs row_ptrs(unsigned char *rows, int row, int cap_a, int cap_b)
{
    RowPtrs r;
    unsigned char *p = rows + (size_t)row * list_row_bytes(cap_a, cap_b);
    r.near = reinterpret_cast<ListNear *>(p);
    r.skip_a = reinterpret_cast<float *>(p + sizeof(ListNear));
    r.skip_b = r.skip_a + kSkipA;
    r.d_a = r.skip_b + kSkipB;
    r.j_a = reinterpret_cast<uint32_t *>(r.d_a + cap_a);
    r.d_b = reinterpret_cast<float *>(r.j_a + cap_a);
    r.j_b = reinterpret_cast<uint32_t *>(r.d_b + cap_b);
    return r;
}

// ---------------- list construction ----------------
// d_Z and d_YZ of point j to Q query points (0 over an empty Z, whose list is
// not built).  qv holds the query values dimension by dimension (Y first), so
// that a column's value is loaded once for all queries.  The maximum starts at
// 0, so that no difference of non-finite values leaves a distance below it.
template <int Q>
__device__ __forceinline__ void list_dist(const float *const *col, int dy, int dz, int j,
                                          const float (*qv)[Q], float (&vz)[Q], float (&vyz)[Q])
{
#pragma unroll
    for (int q = 0; q < Q; ++q) vz[q] = 0.f;
#pragma unroll 2
    for (int d = dy; d < dy + dz; ++d) {
        const float v = __ldg(col[d] + j);
#pragma unroll
        for (int q = 0; q < Q; ++q) vz[q] = fmaxf(vz[q], fabsf(__fsub_rn(qv[d][q], v)));
    }
#pragma unroll
    for (int q = 0; q < Q; ++q) vyz[q] = vz[q];
    for (int d = 0; d < dy; ++d) {
        const float v = __ldg(col[d] + j);
#pragma unroll
        for (int q = 0; q < Q; ++q) vyz[q] = fmaxf(vyz[q], fabsf(__fsub_rn(qv[d][q], v)));
    }
}

// A team's barrier (team t: threads kTeam t .. of the CTA)
constexpr int kTeam = 128;
constexpr int kTeams = kListBuildThreads / kTeam;
__device__ __forceinline__ void team_sync(int t)
{
    asm volatile("bar.sync %0, %1;" ::"r"(t + 1), "n"(kTeam) : "memory");
}

// One team sorts n entries (any order) ascending into its list of row R, pads
// the list to a multiple of 32 and writes its near part and skip row.
// Counting sort into kBins equal parts of [0, top] (the bin is a
// non-decreasing function of the distance), then every entry's rank inside
// its bin by comparison.  bins: kBins ints, idx: n shorts.  Returns the
// padded length.
__device__ int team_list_sort(const Entry *ent, int n, float top, int *bins, uint16_t *idx,
                              const RowPtrs &R, bool list_b, const int *__restrict__ rank, int team)
{
    const int tid = threadIdx.x % kTeam;
    float *d = list_b ? R.d_b : R.d_a, *nd = list_b ? R.near->db : R.near->da;
    uint32_t *j = list_b ? R.j_b : R.j_a, *no = list_b ? R.near->ob : R.near->oa;
    float *skip = list_b ? R.skip_b : R.skip_a;
    const int n_near = list_b ? kNearB : kNearA, n_skip = list_b ? kSkipB : kSkipA;
    const float scale = top > 0.f && top < 3e38f ? (float)kBins / top : 0.f;
    auto bin_of = [&](float v) { return min((int)(v * scale), kBins - 1); };
    for (int b = tid; b < kBins; b += kTeam) bins[b] = 0;
    for (int b = tid; b < n_skip; b += kTeam) skip[b] = CUDART_INF_F;
    float *far = list_b ? &R.near->far_b : &R.near->far_a;
    if (tid == 0) *far = CUDART_INF_F;
    for (int b = n + tid; b < n_near; b += kTeam) {
        nd[b] = CUDART_INF_F;
        no[b] = 0;
    }
    team_sync(team);
    for (int e = tid; e < n; e += kTeam) atomicAdd(&bins[bin_of(ent[e].d)], 1);
    team_sync(team);
    if (tid < 32) {
        int carry = 0;
        for (int b0 = 0; b0 < kBins; b0 += 128) {   // exclusive scan in place, 4 bins per lane
            int4 c = *reinterpret_cast<int4 *>(bins + b0 + 4 * tid);
            const int t = c.x + c.y + c.z + c.w;
            int s = t;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int u = __shfl_up_sync(kFull, s, o);
                if (tid >= o) s += u;
            }
            const int before = carry + s - t;
            *reinterpret_cast<int4 *>(bins + b0 + 4 * tid) =
                make_int4(before, before + c.x, before + c.x + c.y, before + c.x + c.y + c.z);
            carry += __shfl_sync(kFull, s, 31);
        }
    }
    team_sync(team);
    for (int e = tid; e < n; e += kTeam) idx[atomicAdd(&bins[bin_of(ent[e].d)], 1)] = (uint16_t)e;
    team_sync(team);
    // bins[b] is now the end of bin b, so bin b starts at bins[b - 1]
    for (int p = tid; p < n; p += kTeam) {
        const Entry me = ent[idx[p]];
        const int b = bin_of(me.d);
        const int lo = b ? bins[b - 1] : 0, hi = bins[b];
        const uint64_t key = entry_key(me);
        int r = lo;
        for (int u = lo; u < hi; ++u) r += entry_key(ent[idx[u]]) < key ? 1 : 0;
        const uint32_t place = 4u * (rank ? (uint32_t)__ldg(rank + me.j) : me.j);
        d[r] = me.d;
        j[r] = place;
        if (r < n_near) {
            nd[r] = me.d;
            no[r] = place;
        }
        if ((r & 31) == 0) skip[r >> 5] = me.d;
        if (r == n_near) *far = me.d;
    }
    const int padded = (n + 31) & ~31;
    if (tid < padded - n) {
        d[n + tid] = CUDART_INF_F;
        j[n + tid] = 0;
    }
    team_sync(team);   // bins and idx are free again
    return padded;
}

// One CTA builds the lists of Q consecutive query points.  The radius of a
// list is chosen from a sample of the points so that about 0.7 of its capacity
// is used; a list that overflows is collected again with a smaller radius.
template <int Q>
__global__ void __launch_bounds__(kListBuildThreads) list_build_kernel(const ListLaunch L,
                                                                       int smem_a, int smem_b)
{
    extern __shared__ __align__(16) unsigned char lsm[];
    // per team bins and the sort's index row; per query smem_a + smem_b
    // entries (the sample before that)
    const int per_q = smem_a + smem_b, idx_n = max(smem_a, smem_b);
    int *bins = reinterpret_cast<int *>(lsm);
    Entry *ent = reinterpret_cast<Entry *>(bins + kTeams * kBins);
    uint16_t *idx = reinterpret_cast<uint16_t *>(ent + (size_t)Q * per_q);
    __shared__ __align__(16) float qv[32][Q];
    __shared__ const float *col[32];
    __shared__ float s_r[Q][2];
    __shared__ int s_cnt[Q][2];
    __shared__ unsigned s_todo;

    const long long item = blockIdx.x;
    const ListSeg &S = L.segs[last_at_or_below(L.n_segs, item,
                                               [&](int a) { return L.segs[a].build_item; })];
    const ListGroup &G = L.groups[S.group];
    const int N = G.N, w = G.theiler, dy = G.dy, dz = G.dz, dyz = dy + dz;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int r0 = (int)(item - S.build_item) * Q, nq = S.nq;   // first row of the segment
    const unsigned given_up = L.bad ? L.bad[S.group] : 0u;   // by the walk of an earlier launch
    const int i0 = S.q0 + r0;
    const int cap[2] = {G.cap_a, G.cap_b};
    for (int e = tid; e < Q * dyz; e += kListBuildThreads) {
        const int q = e / dyz, d = e - q * dyz;
        const float *c = G.base + (d < dy ? L.cols[G.ycol + d] : L.cols[G.zcol + d - dy]);
        const float v = c[i0 + min(q, nq - 1 - r0)];
        qv[d][q] = v;
        if (L.nonfinite && !(fabsf(v) < CUDART_INF_F)) *L.nonfinite = 1;
        if (q == 0) col[d] = c;
    }
    const int ns = min(N, kSample);
    if (tid < 2 * Q) {
        s_r[tid >> 1][tid & 1] = CUDART_INF_F;
        s_cnt[tid >> 1][tid & 1] = 0;
    }
    if (given_up) return;
    __syncthreads();
    auto masked = [&](int q, int j) { return abs(j - (i0 + q)) <= w; };
    // per query [A sample | B sample], floats, in the entries' space
    auto samp = [&](int q, int l) {
        return reinterpret_cast<float *>(ent + (size_t)q * per_q) + l * kSample;
    };
    const bool sample[2] = {N > cap[0], cap[1] > 0 && N > cap[1]};
    if (sample[0] || sample[1]) {
        for (int s = tid; s < ns; s += kListBuildThreads) {
            const int j = (int)((long long)s * N / ns);
            float vz[Q], vyz[Q];
            list_dist<Q>(col, dy, dz, j, qv, vz, vyz);
#pragma unroll
            for (int q = 0; q < Q; ++q) {
                const bool m = masked(q, j);
                samp(q, 0)[s] = m ? CUDART_INF_F : vyz[q];
                samp(q, 1)[s] = m ? CUDART_INF_F : vz[q];
            }
        }
        __syncthreads();
        for (int t = warp; t < 2 * Q; t += kBuildWarps) {
            const int q = t >> 1, l = t & 1;
            if (!sample[l]) continue;
            float v[kSample / 32];
#pragma unroll
            for (int a = 0; a < kSample / 32; ++a) {
                const int s = a * 32 + lane;
                v[a] = s < ns ? samp(q, l)[s] : CUDART_INF_F;
            }
            // largest radius (to 8 bits of mantissa) with at most `target`
            // samples below it
            const int target = (int)(0.7f * (float)cap[l] * (float)ns / (float)N);
            unsigned lo = 0;
            for (int bit = 30; bit >= 15; --bit) {
                const unsigned c = lo | (1u << bit);
                const float f = __uint_as_float(c);
                int n = 0;
#pragma unroll
                for (int a = 0; a < kSample / 32; ++a) n += v[a] < f ? 1 : 0;
                const int below = (int)__reduce_add_sync(kFull, n);
                if (c <= 0x7f800000u && below <= target) lo = c;
            }
            if (lane == 0) s_r[q][l] = __uint_as_float(lo);
        }
        __syncthreads();
    }
    // B is needed up to A's radius only: a member beyond that scans all points
    if (tid < Q) s_r[tid][1] = fminf(s_r[tid][1], s_r[tid][0]);
    __syncthreads();
    unsigned todo = 0;   // bit 2q + l: list still to be collected
#pragma unroll
    for (int b = 0; b < 2 * Q; ++b) todo |= (b & 1) && cap[1] == 0 ? 0u : 1u << b;
    for (int sweep = 0; todo; ++sweep) {
        float r[Q][2];
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            // -inf: not collected in this sweep
            r[q][0] = (todo >> (2 * q)) & 1u ? s_r[q][0] : -CUDART_INF_F;
            r[q][1] = (todo >> (2 * q + 1)) & 1u ? s_r[q][1] : -CUDART_INF_F;
        }
        for (int j = tid; j < N; j += kListBuildThreads) {
            float vz[Q], vyz[Q];
            list_dist<Q>(col, dy, dz, j, qv, vz, vyz);
#pragma unroll
            for (int q = 0; q < Q; ++q) {
                const bool ok = !masked(q, j);
                if (ok && vyz[q] < r[q][0]) {
                    const int at = atomicAdd(&s_cnt[q][0], 1);
                    if (at < cap[0]) ent[(size_t)q * per_q + at] = Entry{(uint32_t)j, vyz[q]};
                }
                if (ok && vz[q] < r[q][1]) {
                    const int at = atomicAdd(&s_cnt[q][1], 1);
                    if (at < cap[1])
                        ent[(size_t)q * per_q + smem_a + at] = Entry{(uint32_t)j, vz[q]};
                }
            }
        }
        if (tid == 0) s_todo = 0;
        __syncthreads();
        if (tid < 2 * Q && ((todo >> tid) & 1u)) {
            const int q = tid >> 1, l = tid & 1;
            if (s_cnt[q][l] > cap[l]) {
                // too many: a smaller radius (the count goes with at most the
                // dimension's power of it); an empty list in the end
                const float f = 0.8f * (float)cap[l] / (float)s_cnt[q][l];
                const float c = 1.f - (1.f - f) / (float)(l ? dz : dyz);
                const float rn = s_r[q][l] * c;
                s_r[q][l] = sweep < 8 && rn < s_r[q][l] ? rn : 0.f;
                s_cnt[q][l] = 0;
                atomicOr(&s_todo, 1u << tid);
            }
        }
        __syncthreads();
        todo = s_todo;
        __syncthreads();
    }
    const int team = tid / kTeam;
    for (int t = team; t < 2 * Q; t += kTeams) {
        const int q = t >> 1, l = t & 1;
        if (r0 + q >= nq || (l && cap[1] == 0)) continue;
        const Entry *src = ent + (size_t)q * per_q + (l ? smem_a : 0);
        const RowPtrs R = row_ptrs(S.rows, r0 + q, cap[0], cap[1]);
        const int n = s_cnt[q][l];
        float top = s_r[q][l];
        if (!(top < 3e38f)) {   // no radius: the largest distance (each warp finds it)
            float mx = 0.f;
            for (int e = lane; e < n; e += 32) mx = fmaxf(mx, src[e].d);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(kFull, mx, o));
            top = mx;
        }
        const int padded = team_list_sort(src, n, top, bins + team * kBins,
                                          idx + (size_t)team * idx_n, R, l, G.rank, team);
        if (tid % kTeam == 0) {
            if (l) {
                R.near->rb = s_r[q][1];
                R.near->nb = (uint16_t)padded;
            } else {
                R.near->ra = s_r[q][0];
                R.near->na = (uint16_t)padded;
                R.near->place = 4u * (uint32_t)(G.rank ? __ldg(G.rank + i0 + q) : i0 + q);
                if (cap[1] == 0) {
                    R.near->rb = CUDART_INF_F;
                    R.near->nb = 0;
                    R.near->far_b = CUDART_INF_F;
                }
            }
        }
    }
}

// ---------------- sorted columns ----------------
// A point's rank is the number of points before it in (value, index) order:
// one CTA counts 64 points' against every point, staged in shared memory
// (2^13 points sort in a few microseconds over all SMs; a sort by one CTA
// takes a few hundred).
__global__ void __launch_bounds__(256) rank_sort_kernel(const RankSortJob *jobs, int n_jobs)
{
    constexpr int T = 1024;
    __shared__ __align__(16) float v[T];
    __shared__ int s_rank[64];
    const int item = blockIdx.x;
    const RankSortJob J =
        jobs[last_at_or_below(n_jobs, item, [&](int a) { return (long long)jobs[a].item; })];
    const int p = (item - J.item) * 64 + (threadIdx.x & 63), part = threadIdx.x >> 6;
    const float mine = p < J.N ? J.src[p] : 0.f;
    if (threadIdx.x < 64) s_rank[threadIdx.x] = 0;
    int r = 0;
    for (int t0 = 0; t0 < J.N; t0 += T) {
        __syncthreads();
        for (int e = threadIdx.x; e < T; e += 256)
            v[e] = t0 + e < J.N ? J.src[t0 + e] : CUDART_INF_F;
        __syncthreads();
        const int a0 = part * (T / 4);
#pragma unroll 4
        for (int a = a0; a < a0 + T / 4; a += 4) {
            const float4 x = *reinterpret_cast<const float4 *>(v + a);
            const int j = t0 + a;
            r += (x.x < mine || (x.x == mine && j < p)) ? 1 : 0;
            r += (x.y < mine || (x.y == mine && j + 1 < p)) ? 1 : 0;
            r += (x.z < mine || (x.z == mine && j + 2 < p)) ? 1 : 0;
            r += (x.w < mine || (x.w == mine && j + 3 < p)) ? 1 : 0;
        }
    }
    atomicAdd(&s_rank[threadIdx.x & 63], r);
    __syncthreads();
    if (threadIdx.x < 64 && p < J.N) {
        const int k = s_rank[threadIdx.x];
        if (J.sorted) J.sorted[k] = mine;
        if (J.rank) J.rank[p] = k;
    }
}

// ---------------- the walk ----------------
// Ascending sort of the G lanes' values inside every group of G lanes.
template <int G>
__device__ __forceinline__ float group_sort(float v)
{
    const int u = threadIdx.x & (G - 1);
#pragma unroll
    for (int kk = 2; kk <= G; kk <<= 1)
#pragma unroll
        for (int jj = kk >> 1; jj > 0; jj >>= 1) {
            const float o = __shfl_xor_sync(kFull, v, jj);
            const bool low = ((u & jj) == 0) == ((u & kk) == 0 || kk == G);
            v = low ? fminf(v, o) : fmaxf(v, o);
        }
    return v;
}

// The G smallest of buf (ascending over the group's lanes) and the lanes' new
// values, ascending.
template <int G>
__device__ __forceinline__ float group_merge(float buf, float v)
{
    const int u = threadIdx.x & (G - 1);
    v = group_sort<G>(v);
    v = fminf(buf, __shfl_xor_sync(kFull, v, G - 1));   // lane u against the new lane G - 1 - u
#pragma unroll
    for (int jj = G >> 1; jj > 0; jj >>= 1) {
        const float o = __shfl_xor_sync(kFull, v, jj);
        v = (u & jj) == 0 ? fminf(v, o) : fmaxf(v, o);
    }
    return v;
}

// Per group of G lanes, the number of d[0, n) (ascending) below e: G-ary
// search, the whole warp together.
template <int G>
__device__ __forceinline__ int group_rank(const float *__restrict__ d, int n, float e)
{
    const int lane = threadIdx.x & 31, u = lane & (G - 1), shift = lane & ~(G - 1);
    const unsigned mask = G == 32 ? kFull : (1u << G) - 1u;
    int lo = 0;
    while (__any_sync(kFull, n > 0)) {
        const int step = (n + G - 1) / G;
        const int at = u * step;
        const bool below = at < n && d[lo + at] < e;
        const int c = __popc((__ballot_sync(kFull, below) >> shift) & mask);
        const int end = lo + n;
        if (c) lo += (c - 1) * step + 1;
        n = c ? min(step - 1, end - lo) : 0;
    }
    return lo;
}

// The places of an ascending column's values within e of v: rounding is
// monotone, so fl(v - z) >= e holds for its first lo values and fl(z - v) < e
// for its first hi, and the values within are lo .. hi - 1 (none for e <= 0).
// Even lanes of a group find lo, odd lanes hi, over every 16th value (coarse,
// nc of them, in shared memory); then the group reads 16 values for each.
template <int G>
__device__ __forceinline__ void group_window(const float *__restrict__ z, int n,
                                             const float *coarse, int nc, float v, float e, int &lo,
                                             int &hi)
{
    const int u = threadIdx.x & (G - 1);
    const bool up = u & 1;
    int a = 0, b = nc;   // entries for which the test holds: a prefix
    while (__any_sync(kFull, a < b)) {
        const int mid = min((a + b) >> 1, nc - 1);
        const float x = coarse[mid];
        const bool in = up ? __fsub_rn(x, v) < e : __fsub_rn(v, x) >= e;
        if (a < b) {
            if (in) a = mid + 1;
            else b = mid;
        }
    }
    const int cl = __shfl_sync(kFull, a, 0, G), ch = __shfl_sync(kFull, a, 1, G);
    const int bl = 16 * max(cl - 1, 0), bh = 16 * max(ch - 1, 0);
    int fl = 0, fh = 0;
#pragma unroll
    for (int t = u; t < 16; t += G) {
        if (bl + t < n) fl += __fsub_rn(v, __ldg(z + bl + t)) >= e ? 1 : 0;
        if (bh + t < n) fh += __fsub_rn(__ldg(z + bh + t), v) < e ? 1 : 0;
    }
    int s = fl | (fh << 16);   // both below 17
#pragma unroll
    for (int o = G >> 1; o > 0; o >>= 1) s += __shfl_xor_sync(kFull, s, o);
    lo = bl + (s & 0xffff);
    hi = bh + (s >> 16);
    if (!(e > 0.f) || hi < lo) hi = lo;   // hi < lo: values out of order (not finite)
}

// Work counters of one pair's scan over all points: the search, then the counts
__device__ __forceinline__ void count_scan(const ListLaunch &L, int N, bool search)
{
    if (!L.work) return;
    atomicAdd(&L.work[0], (search ? 2ull : 1ull) * (unsigned)N);
    atomicAdd(&L.work[1], (search ? 10ull : 7ull) * (unsigned)N);
}

// One member at query point i over all points, by the whole CTA: its k-th
// smallest joint distance and the three counts, added to the accumulators.
// Blocks of 32 points go round the warps, four of a warp's in flight; every
// warp keeps the smallest distances it meets, and the warps' k smallest are
// merged through shared memory.  xm: the member's X values in shared memory,
// dimension d of point j at sp * (j's place) + d * sd; col and q: the Y then Z columns and
// the point's values in them; top: 32 * k floats, cnt: three ints.
__device__ __noinline__ void scan_member(const ListLaunch &L, const ListGroup &G,
                                         const float *const *col, const float *q, int i,
                                         const float *xm, int sp, int sd, int out, float *top,
                                         int *cnt)
{
    constexpr int U = 4;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, n_warps = blockDim.x >> 5;
    const int N = G.N, dx = G.dx, dy = G.dy, dyz = G.dy + G.dz, k = G.k, w = G.theiler;
    const int stride = 32 * n_warps;
    const int pi = G.rank ? G.rank[i] : i;
    auto dist = [&](int j0, float (&vx)[U], float (&vz)[U], float (&vyz)[U]) {
        int j[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            j[u] = min(j0 + stride * u, N - 1);
            vz[u] = -CUDART_INF_F;
            const int pj = G.rank ? __ldg(G.rank + j[u]) : j[u];
            vx[u] = fabsf(__fsub_rn(xm[sp * pi], xm[sp * pj]));
            for (int d = 1; d < dx; ++d)
                vx[u] = fmaxf(vx[u],
                              fabsf(__fsub_rn(xm[sp * pi + d * sd], xm[sp * pj + d * sd])));
        }
#pragma unroll 2
        for (int d = dy; d < dyz; ++d) {
            const float *c = col[d];
            const float qd = q[d];
#pragma unroll
            for (int u = 0; u < U; ++u)
                vz[u] = fmaxf(vz[u], fabsf(__fsub_rn(qd, __ldg(c + j[u]))));
        }
#pragma unroll
        for (int u = 0; u < U; ++u) vyz[u] = vz[u];
        for (int d = 0; d < dy; ++d) {
            const float *c = col[d];
            const float qd = q[d];
#pragma unroll
            for (int u = 0; u < U; ++u)
                vyz[u] = fmaxf(vyz[u], fabsf(__fsub_rn(qd, __ldg(c + j[u]))));
        }
#pragma unroll
        for (int u = 0; u < U; ++u)   // masked points: beyond every distance
            if (j0 + stride * u >= N || abs(j[u] - i) <= w)
                vx[u] = vz[u] = vyz[u] = CUDART_INF_F;
    };
    float buf = CUDART_INF_F, eps = CUDART_INF_F;
    for (int j0 = 32 * warp + lane; j0 - lane < N; j0 += U * stride) {
        float vx[U], vz[U], vyz[U];
        dist(j0, vx, vz, vyz);
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const float D = fmaxf(vx[u], vyz[u]);
            if (__any_sync(kFull, D < eps)) {
                buf = group_merge<32>(buf, D);
                eps = __shfl_sync(kFull, buf, k - 1);
            }
        }
    }
    if (lane < k) top[warp * k + lane] = buf;
    if (threadIdx.x < 3) cnt[threadIdx.x] = 0;
    __syncthreads();
    buf = CUDART_INF_F;
    for (int a = 0; a < k; ++a)
        buf = group_merge<32>(buf, lane < n_warps ? top[lane * k + a] : CUDART_INF_F);
    eps = __shfl_sync(kFull, buf, k - 1);
    int cxz = 0, cyz = 0, cz = 0;
    for (int j0 = 32 * warp + lane; j0 - lane < N; j0 += U * stride) {
        float vx[U], vz[U], vyz[U];
        dist(j0, vx, vz, vyz);
#pragma unroll
        for (int u = 0; u < U; ++u) {
            cz += vz[u] < eps ? 1 : 0;
            cxz += fmaxf(vx[u], vz[u]) < eps ? 1 : 0;
            cyz += vyz[u] < eps ? 1 : 0;
        }
    }
    cz = (int)__reduce_add_sync(kFull, cz);
    cxz = (int)__reduce_add_sync(kFull, cxz);
    cyz = (int)__reduce_add_sync(kFull, cyz);
    if (lane == 0) {
        atomicAdd(&cnt[0], cz);
        atomicAdd(&cnt[1], cxz);
        atomicAdd(&cnt[2], cyz);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        count_scan(L, N, true);
        // an empty Z: d_Z is below every eps for every point that is not masked
        if (G.dz == 0) cnt[0] = N - (min(i + w, N - 1) - max(i - w, 0) + 1);
        const long long t = L.q[cnt[0] + 1] - L.q[cnt[1] + 1] - L.q[cnt[2] + 1];
        atomicAdd(&L.acc[2 * (size_t)out], (unsigned long long)t & 0xffffffffull);
        atomicAdd(&L.acc[2 * (size_t)out + 1], (unsigned long long)(t >> 32));
        if (L.dbg_eps && out == L.dbg_out) {
            L.dbg_eps[i] = eps;
            L.dbg_nz[i] = cnt[0];
            L.dbg_nxz[i] = cnt[1];
            L.dbg_nyz[i] = cnt[2];
        }
    }
    __syncthreads();
}

// Pairs whose k-th distance lies beyond the radius of one of their lists, put
// aside by the walk: `pair` as in its bit mask, `eps` the k-th distance over
// list A; kExact: it lies within A's radius, so that only counts are missing,
// otherwise it is an upper bound.
struct Aside {
    uint32_t pair;
    float eps;
};
constexpr uint32_t kExact = 0x80000000u;
constexpr int kAside = kListWalkSmem / 4 / 32 / 2;   // as large as the bit mask
constexpr int kScanPairs = 32;    // pairs scanned together
constexpr int kScanNear = 64;     // distances up to the bound that a pair can keep
struct ScanScratch {
    float q[kScanPairs][32];      // the pairs' points: their Y and Z values
    float near[kScanPairs][kScanNear];
    float eps[kScanPairs];
    int n_near[kScanPairs];
    int n[kScanPairs][3];         // d_Z, max(d_X, d_Z), d_YZ below eps
};

// The pairs aside[0, n), over all points, by the whole CTA, kScanPairs at a
// time: the distances up to a pair's bound are collected and its k-th is found
// by one warp, then everything is counted.  The warps meet four times a batch
// and take its pairs one after another without waiting for each other, where
// scan_member meets four times a pair and sorts as it goes.  10^4 points and a
// few pairs in a thousand: 45 candidates of 201 members 40.0 -> 36.0 ms, one
// 2.43 -> 2.18, three X variables 8.5 -> 6.7.  A pair with more than kScanNear distances up to its bound
// is set in `left`, for scan_member.  xs: X values, member m's at xs + m * sm.
__device__ __noinline__ void scan_aside(const ListLaunch &L, const ListGroup &G,
                                        const float *const *col, const Aside *aside, int n,
                                        int i_first, int width, int member0, const float *xs,
                                        int sm, int sp, int sd, ScanScratch &W, uint32_t *left)
{
    constexpr int U = 2;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, n_warps = blockDim.x >> 5;
    const int N = G.N, dx = G.dx, dy = G.dy, dyz = G.dy + G.dz, k = G.k, w = G.theiler;
    const int stride = 32 * n_warps;
    // distances of the U points j0, j0 + stride to pair e's point i
    auto dist = [&](int e, int i, const float *xm, int j0, float (&vx)[U], float (&vz)[U],
                    float (&vyz)[U]) {
        int j[U];
        const int pi = G.rank ? __ldg(G.rank + i) : i;
#pragma unroll
        for (int u = 0; u < U; ++u) {
            j[u] = min(j0 + stride * u, N - 1);
            vz[u] = -CUDART_INF_F;
            const int pj = G.rank ? __ldg(G.rank + j[u]) : j[u];
            vx[u] = fabsf(__fsub_rn(xm[sp * pi], xm[sp * pj]));
            for (int d = 1; d < dx; ++d)
                vx[u] = fmaxf(vx[u],
                              fabsf(__fsub_rn(xm[sp * pi + d * sd], xm[sp * pj + d * sd])));
        }
#pragma unroll 2
        for (int d = dy; d < dyz; ++d) {
            const float *c = col[d];
            const float qd = W.q[e][d];
#pragma unroll
            for (int u = 0; u < U; ++u)
                vz[u] = fmaxf(vz[u], fabsf(__fsub_rn(qd, __ldg(c + j[u]))));
        }
#pragma unroll
        for (int u = 0; u < U; ++u) vyz[u] = vz[u];
        for (int d = 0; d < dy; ++d) {
            const float *c = col[d];
            const float qd = W.q[e][d];
#pragma unroll
            for (int u = 0; u < U; ++u)
                vyz[u] = fmaxf(vyz[u], fabsf(__fsub_rn(qd, __ldg(c + j[u]))));
        }
#pragma unroll
        for (int u = 0; u < U; ++u)   // masked points: beyond every distance
            if (j0 + stride * u >= N || abs(j[u] - i) <= w)
                vx[u] = vz[u] = vyz[u] = CUDART_INF_F;
    };
    for (int base = 0; base < n; base += kScanPairs) {
        const int ne = min(kScanPairs, n - base);
        auto point = [&](int e) { return i_first + (int)(aside[base + e].pair & ~kExact) / width; };
        auto member = [&](int e) { return (int)(aside[base + e].pair & ~kExact) % width; };
        __syncthreads();
        for (int t = threadIdx.x; t < ne * 32; t += blockDim.x)
            if ((t & 31) < dyz) W.q[t >> 5][t & 31] = __ldg(col[t & 31] + point(t >> 5));
        if (threadIdx.x < ne) {
            W.eps[threadIdx.x] = aside[base + threadIdx.x].eps;
            W.n_near[threadIdx.x] = 0;
            for (int a = 0; a < 3; ++a) W.n[threadIdx.x][a] = 0;
        }
        __syncthreads();
        for (int e = 0; e < ne; ++e) {
            if (aside[base + e].pair & kExact) continue;
            const int i = point(e);
            const float *xm = xs + member(e) * sm;
            const float bound = W.eps[e];
            for (int j0 = 32 * warp + lane; j0 - lane < N; j0 += U * stride) {
                float vx[U], vz[U], vyz[U];
                dist(e, i, xm, j0, vx, vz, vyz);
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const float D = fmaxf(vx[u], vyz[u]);
                    if (D <= bound) {
                        const int a = atomicAdd(&W.n_near[e], 1);
                        if (a < kScanNear) W.near[e][a] = D;
                    }
                }
            }
        }
        __syncthreads();
        for (int e = warp; e < ne; e += n_warps) {
            if (aside[base + e].pair & kExact) continue;
            const int c = W.n_near[e];
            float v = group_sort<32>(lane < c ? W.near[e][lane] : CUDART_INF_F);
            v = group_merge<32>(v, lane + 32 < min(c, kScanNear) ? W.near[e][lane + 32]
                                                                 : CUDART_INF_F);
            const float eps = __shfl_sync(kFull, v, k - 1);
            if (lane == 0) W.eps[e] = eps;
        }
        __syncthreads();
        for (int e = 0; e < ne; ++e) {
            const int i = point(e);
            const float *xm = xs + member(e) * sm;
            const float eps = W.eps[e];
            int cz = 0, cxz = 0, cyz = 0;
            for (int j0 = 32 * warp + lane; j0 - lane < N; j0 += U * stride) {
                float vx[U], vz[U], vyz[U];
                dist(e, i, xm, j0, vx, vz, vyz);
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    cz += vz[u] < eps ? 1 : 0;
                    cxz += fmaxf(vx[u], vz[u]) < eps ? 1 : 0;
                    cyz += vyz[u] < eps ? 1 : 0;
                }
            }
            cz = (int)__reduce_add_sync(kFull, cz);
            cxz = (int)__reduce_add_sync(kFull, cxz);
            cyz = (int)__reduce_add_sync(kFull, cyz);
            if (lane < 3) atomicAdd(&W.n[e][lane], lane == 0 ? cz : lane == 1 ? cxz : cyz);
        }
        __syncthreads();
        if (threadIdx.x < ne) {
            const int e = threadIdx.x, i = point(e);
            count_scan(L, N, !(aside[base + e].pair & kExact));
            if (W.n_near[e] > kScanNear) {
                const uint32_t b = aside[base + e].pair & ~kExact;
                atomicOr(&left[b >> 5], 1u << (b & 31));
            } else {
                // an empty Z: d_Z is below every eps for every point that is not masked
                const int nz = G.dz == 0 ? N - (min(i + w, N - 1) - max(i - w, 0) + 1) : W.n[e][0];
                const int out = L.members[member0 + member(e)].out;
                const long long t = L.q[nz + 1] - L.q[W.n[e][1] + 1] - L.q[W.n[e][2] + 1];
                atomicAdd(&L.acc[2 * (size_t)out], (unsigned long long)t & 0xffffffffull);
                atomicAdd(&L.acc[2 * (size_t)out + 1], (unsigned long long)(t >> 32));
                if (L.dbg_eps && out == L.dbg_out) {
                    L.dbg_eps[i] = W.eps[e];
                    L.dbg_nz[i] = nz;
                    L.dbg_nxz[i] = W.n[e][1];
                    L.dbg_nyz[i] = W.n[e][2];
                }
            }
        }
    }
    __syncthreads();
}

// E consecutive distances (E = 1, 2 or 4, aligned to E)
template <int E>
__device__ __forceinline__ void load_vec(const float *dp, float (&d)[E])
{
    if constexpr (E == 4) {
        const float4 v = *reinterpret_cast<const float4 *>(dp);
        d[0] = v.x; d[1] = v.y; d[2] = v.z; d[3] = v.w;
    } else if constexpr (E == 2) {
        const float2 v = *reinterpret_cast<const float2 *>(dp);
        d[0] = v.x; d[1] = v.y;
    } else {
        d[0] = *dp;
    }
}

// E consecutive entries of a list (E = 1, 2 or 4, aligned to E)
template <int E>
__device__ __forceinline__ void load_entries(const float *dp, const uint32_t *op, float (&d)[E],
                                             uint32_t (&o)[E])
{
    if constexpr (E == 4) {
        const float4 v = *reinterpret_cast<const float4 *>(dp);
        const uint4 w = *reinterpret_cast<const uint4 *>(op);
        d[0] = v.x; d[1] = v.y; d[2] = v.z; d[3] = v.w;
        o[0] = w.x; o[1] = w.y; o[2] = w.z; o[3] = w.w;
    } else if constexpr (E == 2) {
        const float2 v = *reinterpret_cast<const float2 *>(dp);
        const uint2 w = *reinterpret_cast<const uint2 *>(op);
        d[0] = v.x; d[1] = v.y;
        o[0] = w.x; o[1] = w.y;
    } else {
        d[0] = *dp;
        o[0] = *op;
    }
}

// The 4 smallest of two ascending lists of 4, ascending, into b.
__device__ __forceinline__ void cmpx(float &a, float &b)
{
    const float lo = fminf(a, b);
    b = fmaxf(a, b);
    a = lo;
}
__device__ __forceinline__ void merge4(float (&b)[4], const float (&o)[4])
{
#pragma unroll
    for (int a = 0; a < 4; ++a) b[a] = fminf(b[a], o[3 - a]);   // bitonic
    cmpx(b[0], b[2]);
    cmpx(b[1], b[3]);
    cmpx(b[0], b[1]);
    cmpx(b[2], b[3]);
}

// A member's k smallest joint distances so far.  K4 (k = 4): all four in
// every lane of the member's group; otherwise the a-th in the group's lane a.
template <int G, bool K4>
struct Nearest {
    float b[K4 ? 4 : 1];
    float thr;   // the k-th
    __device__ __forceinline__ Nearest()
    {
        thr = CUDART_INF_F;
#pragma unroll
        for (float &v : b) v = CUDART_INF_F;
    }
    // the lanes' E = 32 / G new distances each
    __device__ __forceinline__ void add(const float (&D)[32 / G], int k)
    {
        constexpr int E = 32 / G;
        if constexpr (K4) {
            // sorted in the lane, then pairwise over the group's lanes
            float v[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) v[e] = e < E ? D[e < E ? e : 0] : CUDART_INF_F;
            if constexpr (E == 4) {
                cmpx(v[0], v[1]);
                cmpx(v[2], v[3]);
                cmpx(v[0], v[2]);
                cmpx(v[1], v[3]);
                cmpx(v[1], v[2]);
            } else if constexpr (E == 2) {
                cmpx(v[0], v[1]);
            }
#pragma unroll
            for (int o = 1; o < G; o <<= 1) {
                float t[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) t[e] = __shfl_xor_sync(kFull, v[e], o);
                merge4(v, t);
            }
            merge4(b, v);
            thr = b[3];
        } else {
#pragma unroll
            for (int e = 0; e < E; ++e)
                if (__any_sync(kFull, D[e] < thr)) {
                    b[0] = group_merge<G>(b[0], D[e]);
                    thr = __shfl_sync(kFull, b[0], k - 1, G);
                }
        }
    }
};

// One CTA: `width` members of one group, their X values in shared memory, x a
// range of query points.  A warp serves NG = 32 / G (point, member) pairs at a
// time, G lanes each and 32 list entries at a time: `width` members at
// NG / width points.  Only a long prefix (n_xz) goes over the whole warp, 128
// entries at a time.  With NG members (NEAR) the warp's one point has its
// near lists copied a point ahead; the digamma values that end a pair's work
// are added a point later: in a small call a warp's time is a chain of memory
// and shuffle latencies.  In a large one (45 x 201 members, N = 9995, 2 Z: 33.9
// ms) the kernel issues in 75% of the slots, 344 warp instructions a pair, with the
// shared-memory pipe busy 72%, 63% of its load wavefronts bank conflicts of gathers.
// DXP: X variables as stored, dimensions of a point together: 1, 2 or 4 (three
// or four variables), so that a point's values are one load; 0: any number, a
// row per dimension.
// bytes before the X values of a walking CTA
__host__ __device__ constexpr size_t list_walk_head(bool near, int n_warps)
{
    const size_t b = near ? 2 * (size_t)n_warps * sizeof(ListNear) : 0;
    return b > sizeof(ScanScratch) ? b : (sizeof(ScanScratch) + 15) & ~(size_t)15;
}

template <int G, bool NEAR, int DXP, bool K4>
__global__ void __launch_bounds__(kListWalkThreads) list_walk_kernel(const ListLaunch L,
                                                                     const int width)
{
    constexpr int NG = 32 / G;
    constexpr int E = 32 / G;       // entries per lane of a 32-entry step
    constexpr int XR = DXP > 0 ? DXP : 1;
    // NEAR: [2][warps] ListNear, otherwise room for ScanScratch; X of every
    // member; coarse sorted columns
    extern __shared__ __align__(16) unsigned char wsm[];
    __shared__ const float *s_col[32];
    __shared__ float s_q[32];                     // a point's Y and Z values
    __shared__ float s_top[32 * 16];
    __shared__ int s_cnt[3];
    // pairs beyond the lists' radii: (point of the CTA) * width + member, put
    // aside, and as bits of a mask once that is full
    __shared__ uint32_t s_slow[kListWalkSmem / 4 / 32 + 1];
    __shared__ Aside s_aside[kAside];
    __shared__ int s_n_aside;
    __shared__ unsigned s_given_up;
    __shared__ int s_slow_limit;
    const long long item = blockIdx.x;
    const ListSeg &S = L.segs[last_at_or_below(L.n_segs, item,
                                               [&](int a) { return L.segs[a].walk_item; })];
    const ListGroup &Gr = L.groups[S.group];
    const int N = Gr.N, dx = DXP == 1 ? 1 : Gr.dx, w = Gr.theiler, k = K4 ? 4 : Gr.k, dz = Gr.dz;
    const int dyz = Gr.dy + dz;
    const long long local = item - S.walk_item;
    const int mb = (int)(local / S.n_splits), split = (int)(local % S.n_splits);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, n_warps = blockDim.x >> 5;
    const int u = lane & (G - 1), g = lane / G;
    const int gm = NEAR ? g : g & (width - 1);         // the group's member and
    const int qw = NEAR ? 1 : NG / width;              // point, of qw at a time
    const int cap_a = Gr.cap_a, cap_b = Gr.cap_b;
    const int nm = min(width, Gr.n_members - mb * width);
    const int xd = (N + 3) & ~3;
    const int xn = (DXP > 0 ? DXP : dx) * xd;          // X values of a member
    const int sp = XR, sd = DXP > 0 ? 1 : xd;          // strides of a point, of a dimension
    ListNear *near_buf = reinterpret_cast<ListNear *>(wsm) + 2 * warp;
    float *xs = reinterpret_cast<float *>(wsm + list_walk_head(NEAR, n_warps));
    float *coarse = xs + width * xn;
    const int nc = (N + 15) / 16;
    const bool xsorted = DXP == 1 && dz == 0;
    unsigned given_up = 0;   // by another CTA
    if (threadIdx.x == 0 && L.bad) given_up = *(volatile unsigned *)(L.bad + S.group);

    for (int m = 0; m < width; ++m) {
        // past the last member: the last one again, its results dropped
        const MemberDesc md = L.members[Gr.member_begin + mb * width + min(m, nm - 1)];
        for (int d = 0; d < dx; ++d) {
            const float *src = Gr.base + L.cols[md.xcol + d];
            float *dst = xs + m * xn + d * sd;
            bool finite = true;
#pragma unroll 4
            for (int j = threadIdx.x; j < N; j += blockDim.x) {
                const float v = __ldg(src + (md.perm ? __ldg(md.perm + j) : j));
                dst[sp * (dz == 1 ? __ldg(Gr.rank + j) : j)] = v;
                finite = finite && fabsf(v) < CUDART_INF_F;
            }
            if (!finite && L.nonfinite) *L.nonfinite = 1;
        }
        if (DXP > 2 && dx < DXP)   // the unused dimensions add nothing to a maximum
            for (int j = threadIdx.x; j < N; j += blockDim.x)
                for (int d = dx; d < DXP; ++d) xs[m * xn + DXP * j + d] = 0.f;
        if (xsorted)
            for (int c = threadIdx.x; c < nc; c += blockDim.x)
                coarse[m * nc + c] = __ldg(md.xsorted + 16 * c);
    }
    if (dz == 1)
        for (int c = threadIdx.x; c < nc; c += blockDim.x) coarse[c] = __ldg(Gr.zs + 16 * c);
    if (threadIdx.x < dyz)
        s_col[threadIdx.x] = Gr.base + (threadIdx.x < Gr.dy
                                            ? L.cols[Gr.ycol + threadIdx.x]
                                            : L.cols[Gr.zcol + threadIdx.x - Gr.dy]);
    const int q_first = split * S.per_cta, q_last = min(S.nq, q_first + S.per_cta);
    const int n_words = (q_last - q_first) * width / 32 + 1;
    for (int a = threadIdx.x; a < n_words; a += blockDim.x) s_slow[a] = 0;
    if (threadIdx.x == 0) {
        s_n_aside = 0;
        s_given_up = given_up;
        s_slow_limit = L.bad ? list_slow_limit((q_last - q_first) * nm, N, dx, Gr.n_members,
                                               w == 0 && N <= kMaxOrderN)
                             : 0x7fffffff;
    }
    const char *xm = reinterpret_cast<const char *>(xs + gm * xn);
    // A pair's sum of digamma values: its group's lanes 0, 1, 2 sum those of
    // n_z, -n_xz and -n_yz (the low 32 bits and the rest apart, as the
    // accumulators keep them: a long run would not fit in one int64).
    unsigned long long sum_lo = 0;
    long long sum_hi = 0, q_last_term = 0;
    unsigned evals = 0;   // member-pairs evaluated by the warp
    __syncthreads();
    if (s_given_up) return;

    // the X values at byte offset o of the row x
    auto load_x = [&](const char *x, uint32_t o, float (&v)[XR]) {
        if constexpr (DXP == 4) {
            const float4 t = *reinterpret_cast<const float4 *>(x + 4 * o);
            v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
        } else if constexpr (DXP == 2) {
            const float2 t = *reinterpret_cast<const float2 *>(x + 2 * o);
            v[0] = t.x; v[1] = t.y;
        } else {
            v[0] = *reinterpret_cast<const float *>(x + o);
        }
    };
    // d_X between the query point (values xi, byte offset oi) and the point at o
    auto dist_x = [&](const char *x, const float (&xi)[XR], uint32_t oi, uint32_t o) {
        float t[XR];
        load_x(x, o, t);
        float v = fabsf(__fsub_rn(xi[0], t[0]));
#pragma unroll
        for (int d = 1; d < XR; ++d) v = fmaxf(v, fabsf(__fsub_rn(xi[d], t[d])));
        if (DXP == 0)
            for (int d = 1; d < dx; ++d) {
                const char *r = x + 4 * d * xd;
                v = fmaxf(v, fabsf(__fsub_rn(*reinterpret_cast<const float *>(r + oi),
                                             *reinterpret_cast<const float *>(r + o))));
            }
        return v;
    };
    auto group_sum = [&](int v) {
#pragma unroll
        for (int o = G >> 1; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
        return v;
    };
    unsigned char *const rows = S.rows;
    const int q0 = S.q0;
    // copy a row's near part into buffer `half` (past the end: the last row again)
    auto fetch = [&](int r, int half) {
        const RowPtrs R = row_ptrs(rows, min(r, q_last - 1), cap_a, cap_b);
        const uint32_t dst = (uint32_t)__cvta_generic_to_shared(near_buf + half);
        for (int e = 16 * lane; e < (int)sizeof(ListNear); e += 512)
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + e),
                         "l"(reinterpret_cast<const char *>(R.near) + e)
                         : "memory");
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    auto add_term = [&]() {
        sum_lo += (unsigned long long)q_last_term & 0xffffffffull;
        sum_hi += q_last_term >> 32;
    };
    int half = 0;
    if (NEAR) fetch(q_first + warp, 0);
    for (int first_row = q_first + warp * qw; first_row < q_last;
         first_row += n_warps * qw, half ^= 1) {
        // a group past the last point repeats it, its result dropped
        const int row_g = NEAR ? first_row : first_row + g / width;
        const int row = NEAR ? first_row : min(row_g, q_last - 1);
        const bool live = gm < nm && row_g < q_last;
        const int i = q0 + row;
        const RowPtrs R = row_ptrs(rows, row, cap_a, cap_b);
        if (NEAR) {
            __syncwarp();   // the other half's readers are done
            fetch(first_row + n_warps, half ^ 1);
            asm volatile("cp.async.wait_group 1;" ::: "memory");
            __syncwarp();
        }
        const ListNear &h = NEAR ? near_buf[half] : *R.near;
        const int na = h.na, nb = h.nb;
        const uint32_t oi = h.place;
        float xi[XR];
        load_x(xm, oi, xi);

        // ---- k nearest joint distances over list A ----
        Nearest<G, K4> near;
        int c = 0, p = 32;
        float da[E];   // the first 32 entries' d_YZ
        float d[E];
        uint32_t o[E];
        {
            float D[E];
            load_entries<E>(h.da + E * u, h.oa + E * u, da, o);
#pragma unroll
            for (int e = 0; e < E; ++e) D[e] = fmaxf(dist_x(xm, xi, oi, o[e]), da[e]);
            near.add(D, k);
            evals += 32 * E;
        }
        if (__any_sync(kFull, h.far_a < near.thr))
            for (; NEAR ? p < na : __any_sync(kFull, p < na); p += 32) {
                float D[E], dmin = CUDART_INF_F;
                if (NEAR || p < na) {
                    load_entries<E>(R.d_a + p + E * u, R.j_a + p + E * u, d, o);
                } else {
#pragma unroll
                    for (int e = 0; e < E; ++e) {
                        d[e] = CUDART_INF_F;
                        o[e] = 0;
                    }
                }
                if (!__any_sync(kFull, d[0] < near.thr)) break;
                evals += 32 * E;
#pragma unroll
                for (int e = 0; e < E; ++e) {
                    D[e] = fmaxf(dist_x(xm, xi, oi, o[e]), d[e]);
                    dmin = fminf(dmin, D[e]);
                }
                if (__any_sync(kFull, dmin < near.thr)) near.add(D, k);
            }

        // ---- n_yz: a rank in A ----
        const float eps = near.thr;
        const bool slow = eps > h.ra || (dz > 1 && eps > h.rb);
        const float ec = slow ? -1.f : eps;   // below every distance for pairs that scan
        int nz = 0, nyz = 0, nxz = 0;
        int n[NG];
        int from = 0;   // n_z: the entries before the 32 that hold its end
        const bool far = dz > 1 && __any_sync(kFull, ec > h.far_b);
        if constexpr (NEAR) {
            // the last skip distance below eps, then the 32 entries from it
            int fa = 0;
            const bool far_a = p > 32;
            float2 ska = make_float2(CUDART_INF_F, CUDART_INF_F);
            float4 skb = make_float4(CUDART_INF_F, CUDART_INF_F, CUDART_INF_F, CUDART_INF_F);
            if (far_a) ska = *reinterpret_cast<const float2 *>(R.skip_a + 2 * lane);
            if (far) skb = *reinterpret_cast<const float4 *>(R.skip_b + 4 * lane);
#pragma unroll
            for (int m = 0; m < NG; ++m) {
                const float e = __shfl_sync(kFull, ec, m * G);
                if (far_a) {
                    const int t = __popc(__ballot_sync(kFull, ska.x < e)) +
                                  __popc(__ballot_sync(kFull, ska.y < e));
                    if (g == m) fa = 32 * max(t - 1, 0);
                }
                if (far) {
                    const int t = (int)__reduce_add_sync(
                        kFull, (skb.x < e ? 1 : 0) + (skb.y < e ? 1 : 0) + (skb.z < e ? 1 : 0) +
                                   (skb.w < e ? 1 : 0));
                    if (g == m) from = 32 * max(t - 1, 0);
                }
            }
            if (far_a) load_vec<E>(R.d_a + fa + E * u, da);
            if (far) load_vec<E>(R.d_b + from + E * u, d);
#pragma unroll
            for (int e = 0; e < E; ++e) nyz += da[e] < ec ? 1 : 0;
            nyz = fa + group_sum(nyz);
        } else {
#pragma unroll
            for (int e = 0; e < E; ++e) nyz += da[e] < ec ? 1 : 0;
            nyz = group_sum(nyz);
            if (p > 32) nyz += group_rank<G>(R.d_a + 32, max(min(p, na) - 32, 0), ec);
            if (far) {
                from = 32 * max(group_rank<G>(R.skip_b, kSkipB, ec) - 1, 0);
                load_vec<E>(R.d_b + from + E * u, d);
            }
        }

        // ---- n_z and n_xz ----
        if (dz > 1 && !far) {
            // every prefix of B ends within kNearB entries: counted by the groups
            int cz = 0, cx = 0;
            for (int b = 0; b < kNearB; b += 32) {
                load_entries<E>(h.db + b + E * u, h.ob + b + E * u, d, o);
                if (!__any_sync(kFull, d[0] < ec)) break;
#pragma unroll
                for (int e = 0; e < E; ++e) {
                    cz += d[e] < ec ? 1 : 0;
                    cx += fmaxf(dist_x(xm, xi, oi, o[e]), d[e]) < ec ? 1 : 0;
                }
                evals += 32 * E;
            }
            nz = group_sum(cz);
            nxz = group_sum(cx);
        } else if (dz > 1) {
            uint4 o_next = make_uint4(0, 0, 0, 0);
            if (NEAR && DXP == 1)
                o_next = *reinterpret_cast<const uint4 *>(R.j_b + min(4 * lane, nb - 4));
#pragma unroll
            for (int e = 0; e < E; ++e) c += d[e] < ec ? 1 : 0;
            c = group_sum(c);
            nz = nb ? from + c : 0;
            int nmax = 0;
#pragma unroll
            for (int m = 0; m < NG; ++m) {
                n[m] = __shfl_sync(kFull, nz, m * G);
                nmax = max(nmax, n[m]);
                evals += n[m];
            }
            if constexpr (NEAR && DXP == 1) {   // one list: its entries are read once
                float e[NG], xq[NG][1];
                int cm[NG];
#pragma unroll
                for (int m = 0; m < NG; ++m) {
                    e[m] = __shfl_sync(kFull, ec, m * G);
                    xq[m][0] = __shfl_sync(kFull, xi[0], m * G);
                    cm[m] = 0;
                }
                for (int b = 0; b < nmax; b += 128) {
                    const int at = b + 4 * lane;
                    const uint4 o = o_next;
                    if (b + 128 < nmax)
                        o_next = *reinterpret_cast<const uint4 *>(R.j_b + min(at + 128, nb - 4));
#pragma unroll
                    for (int m = 0; m < NG; ++m) {
                        if (b >= n[m]) continue;
                        const char *x = reinterpret_cast<const char *>(xs + m * xn);
                        const float d0 = dist_x(x, xq[m], oi, o.x), d1 = dist_x(x, xq[m], oi, o.y);
                        const float d2 = dist_x(x, xq[m], oi, o.z), d3 = dist_x(x, xq[m], oi, o.w);
                        if (b + 128 <= n[m]) {
                            cm[m] += (d0 < e[m] ? 1 : 0) + (d1 < e[m] ? 1 : 0) +
                                     (d2 < e[m] ? 1 : 0) + (d3 < e[m] ? 1 : 0);
                        } else {
                            cm[m] += (at < n[m] && d0 < e[m] ? 1 : 0) +
                                     (at + 1 < n[m] && d1 < e[m] ? 1 : 0) +
                                     (at + 2 < n[m] && d2 < e[m] ? 1 : 0) +
                                     (at + 3 < n[m] && d3 < e[m] ? 1 : 0);
                        }
                    }
                }
#pragma unroll
                for (int m = 0; m < NG; ++m) {
                    const int t = (int)__reduce_add_sync(kFull, cm[m]);
                    if (g == m) nxz = t;
                }
            } else {
#pragma unroll 1
                for (int m = 0; m < NG; ++m) {
                    const int nn = __shfl_sync(kFull, nz, m * G);
                    if (nn == 0) continue;
                    const float e = __shfl_sync(kFull, ec, m * G);
                    const uint32_t oq = __shfl_sync(kFull, oi, m * G);
                    float xq[XR];
#pragma unroll
                    for (int d = 0; d < XR; ++d) xq[d] = __shfl_sync(kFull, xi[d], m * G);
                    const uint32_t *list =
                        row_ptrs(rows, __shfl_sync(kFull, row, m * G), cap_a, cap_b).j_b;
                    const char *x = reinterpret_cast<const char *>(
                        xs + (NEAR ? m : m & (width - 1)) * xn);
                    int cm = 0;
                    for (int b = 0; b < nn; b += 128) {
                        const int at = b + 4 * lane;
                        if (at >= nn) continue;
                        const uint4 o = *reinterpret_cast<const uint4 *>(list + at);
                        cm += dist_x(x, xq, oq, o.x) < e ? 1 : 0;
                        cm += at + 1 < nn && dist_x(x, xq, oq, o.y) < e ? 1 : 0;
                        cm += at + 2 < nn && dist_x(x, xq, oq, o.z) < e ? 1 : 0;
                        cm += at + 3 < nn && dist_x(x, xq, oq, o.w) < e ? 1 : 0;
                    }
                    cm = (int)__reduce_add_sync(kFull, cm);
                    if (g == m) nxz = cm;
                }
            }
        } else if (dz == 1) {
            // the points with d_Z < eps are consecutive places
            const float zi = __ldg(s_col[Gr.dy] + i);
            int lo, hi;
            group_window<G>(Gr.zs, N, coarse, nc, zi, ec, lo, hi);
            nz = hi - lo;
#pragma unroll
            for (int m = 0; m < NG; ++m) {
                const int l = __shfl_sync(kFull, lo, m * G), n = __shfl_sync(kFull, nz, m * G);
                const float e = __shfl_sync(kFull, ec, m * G);
                const uint32_t oq = __shfl_sync(kFull, oi, m * G);
                float xq[XR];
#pragma unroll
                for (int d = 0; d < XR; ++d) xq[d] = __shfl_sync(kFull, xi[d], m * G);
                const char *x = reinterpret_cast<const char *>(
                    xs + (NEAR ? m : m & (width - 1)) * xn);
                int cm = 0;
                for (int b = l & ~3; b < l + n; b += 128) {
                    const int at = min(b + 4 * lane, xd - 4);
                    float v[4];
                    if constexpr (DXP == 1) {
                        const float4 t = *reinterpret_cast<const float4 *>(x + 4 * at);
                        v[0] = fabsf(__fsub_rn(xq[0], t.x));
                        v[1] = fabsf(__fsub_rn(xq[0], t.y));
                        v[2] = fabsf(__fsub_rn(xq[0], t.z));
                        v[3] = fabsf(__fsub_rn(xq[0], t.w));
                    } else {
#pragma unroll
                        for (int a = 0; a < 4; ++a) v[a] = dist_x(x, xq, oq, 4u * (at + a));
                    }
                    if (b >= l && b + 128 <= l + n) {
#pragma unroll
                        for (int a = 0; a < 4; ++a) cm += v[a] < e ? 1 : 0;
                    } else {
                        const unsigned f = b + 4 * lane - l;
#pragma unroll
                        for (int a = 0; a < 4; ++a)
                            cm += f + a < (unsigned)n && v[a] < e ? 1 : 0;
                    }
                }
                cm = (int)__reduce_add_sync(kFull, cm);
                evals += n;
                if (g == m) nxz = cm;
            }
            // less the point itself and its Theiler band
            if (w == 0) {
                if (ec > 0.f) {
                    --nz;
                    --nxz;
                }
            } else {
                const int first = max(i - w, 0), last = min(i + w, N - 1);
                int cz = 0, cx = 0;
                for (int j = first + u; j <= last; j += G) {
                    const float d = fabsf(__fsub_rn(zi, __ldg(s_col[Gr.dy] + j)));
                    const float v = dist_x(xm, xi, oi, 4u * (uint32_t)__ldg(Gr.rank + j));
                    cz += d < ec ? 1 : 0;
                    cx += fmaxf(d, v) < ec ? 1 : 0;
                }
                __syncwarp();
                evals += NG * (last - first + 1);
                nz -= group_sum(cz);
                nxz -= group_sum(cx);
            }
        } else {
            const int first = max(i - w, 0), last = min(i + w, N - 1);
            nz = N - (last - first + 1);
            if (xsorted) {
                // the member's X values are its column's, in another order: a
                // window of the sorted column, less the point itself and its band
                int lo, hi;
                group_window<G>(
                    L.members[Gr.member_begin + mb * width + min(gm, nm - 1)].xsorted, N,
                    coarse + gm * nc, nc, xi[0], ec, lo, hi);
                c = 0;
                for (int j = first + u; j <= last; j += G)
                    c += dist_x(xm, xi, oi, 4u * j) < ec ? 1 : 0;
                evals += NG * (last - first + 1);
                __syncwarp();
                nxz = hi - lo - group_sum(c);
            } else {
                c = 0;
                for (int j = u; j < N; j += G)
                    if (j < first || j > last) c += dist_x(xm, xi, oi, 4u * j) < ec ? 1 : 0;
                evals += NG * nz;
                __syncwarp();
                nxz = group_sum(c);
            }
        }
        if (__any_sync(kFull, slow)) {
            bool give_up = false;
            if (slow && u == 0 && live) {
                const int bit = (row - q_first) * width + gm;
                const int at = atomicAdd(&s_n_aside, 1);
                if (at < kAside)
                    s_aside[at] = Aside{(uint32_t)bit | (eps > h.ra ? 0u : kExact), eps};
                else
                    atomicOr(&s_slow[bit >> 5], 1u << (bit & 31));
                give_up = at >= s_slow_limit;
            }
            // the group's sums are not used: no further point
            if (__any_sync(kFull, give_up)) first_row = q_last;
        }
        if (slow || !live) nz = nxz = nyz = -1;   // the digamma table's first value, 0
        add_term();
        // (a band can hold more than the window of values that are not finite)
        q_last_term = L.q[max(u == 0 ? nz : u == 1 ? nxz : nyz, -1) + 1];
        if (u > 0) q_last_term = -q_last_term;
        if (L.dbg_eps && u == 0 && live && !slow &&
            L.members[Gr.member_begin + mb * width + gm].out == L.dbg_out) {
            L.dbg_eps[i] = eps;
            L.dbg_nxz[i] = nxz;
            L.dbg_nyz[i] = nyz;
            L.dbg_nz[i] = nz;
        }
    }
    if (NEAR) asm volatile("cp.async.wait_group 0;" ::: "memory");
    add_term();
    if (u < 3 && gm < nm) {
        const int out = L.members[Gr.member_begin + mb * width + gm].out;
        atomicAdd(&L.acc[2 * (size_t)out], sum_lo);
        atomicAdd(&L.acc[2 * (size_t)out + 1], (unsigned long long)sum_hi);
    }
    if (L.work && lane == 0) {
        atomicAdd(&L.work[0], (unsigned long long)evals);
        atomicAdd(&L.work[1], 3ull * evals);
    }
    // ---- pairs beyond the lists' radii: over all points, by the whole CTA ----
    __syncthreads();
    if (L.bad && s_n_aside > min(32, s_slow_limit)) {   // are so many scans still wanted?
        if (threadIdx.x == 0) {
            if (s_n_aside > s_slow_limit && atomicExch(L.bad + S.group, 1u) == 0u)
                atomicAdd(L.n_bad, 1ull);
            s_given_up = *(volatile unsigned *)(L.bad + S.group);
        }
        __syncthreads();
        if (s_given_up) return;
    }
    if (s_n_aside)
        scan_aside(L, Gr, s_col, s_aside, min(s_n_aside, kAside), q0 + q_first, width,
                   Gr.member_begin + mb * width, xs, xn, sp, sd,
                   *reinterpret_cast<ScanScratch *>(wsm), s_slow);
    for (int w0 = 0; w0 < n_words; w0 += 32) {   // the same in every warp
        const uint32_t mine = w0 + lane < n_words ? s_slow[w0 + lane] : 0;
        unsigned words = __ballot_sync(kFull, mine != 0);
        while (words) {
            const int src = __ffs(words) - 1;
            words &= words - 1;
            uint32_t bits = __shfl_sync(kFull, mine, src);
            while (bits) {
                const int b = 32 * (w0 + src) + __ffs(bits) - 1;
                bits &= bits - 1;
                const int i = q0 + q_first + b / width, m = b % width;
                if (threadIdx.x < dyz) s_q[threadIdx.x] = __ldg(s_col[threadIdx.x] + i);
                __syncthreads();
                scan_member(L, Gr, s_col, s_q, i, xs + m * xn, sp, sd,
                            L.members[Gr.member_begin + mb * width + m].out, s_top, s_cnt);
            }
        }
    }
}

}  // namespace

void list_caps(int N, int k, int dx, int dy, int dz, int *cap_a, int *cap_b)
{
    // Expected counts when the joint space has m independent dimensions: a
    // per-dimension slab of probability (k / N)^(1/m) holds the neighbours.
    // The margins cover the members whose X value lies in a sparse region.
    // Half of either, N = 10^4: one call of 201 members 2.15 -> 2.19 ms, 45
    // candidates 35.8 -> 44.9; more of either changes nothing.
    // From eight dimensions on shorter lists A: 201 members, N = 10^4, 6 to 10 Z
    // variables, coupled maps 0.90 .. 0.96 ms, with 56 0.94 .. 1.00 (their batches, and any
    // N below 6000, the same); VAR data would gain by 56: 1.37 .. 1.52 -> 1.19 .. 1.33, 45
    // candidates 26.7 -> 20.1.
    const double m = dx + dy + dz;
    const double slab = std::pow((double)k / (double)N, 1.0 / m);
    const double nyz = N * std::pow(slab, (double)(dy + dz));
    const double nz = N * std::pow(slab, (double)dz);
    auto cap = [&](double c, int hi) {
        const int all = (N + 31) & ~31;
        const int v = ((int)std::min(c, 1e6) + 31) & ~31;
        return std::min(all, std::max(128, std::min(v, hi)));
    };
    *cap_a = cap((m >= 8 ? 32.0 : 56.0) * nyz, kListCapA);
    *cap_b = dz > 1 ? cap(28.0 * nz, kListCapB) : 0;
}

// X variables as stored for the walk (its DXP): the dimensions of a
// point together where that fits, a row per dimension (0) otherwise
static int list_dxp(int N, int dx, int k)
{
    if (dx == 1) return 1;
    const int p = dx == 2 ? 2 : 4;
    return k == 4 && dx <= 4 && (size_t)p * (((size_t)N + 3) & ~(size_t)3) * 4 <= kListWalkSmem ? p
                                                                                               : 0;
}

size_t list_walk_x_bytes(int N, int dx, int dz, int k, int width)
{
    const int dxp = list_dxp(N, dx, k);
    const size_t coarse = (((size_t)N + 15) / 16 * 4 + 15) & ~(size_t)15;
    return (size_t)width * (dxp ? dxp : dx) * (((size_t)N + 3) & ~(size_t)3) * 4 +
           (dz == 1 ? coarse : dz == 0 && dx == 1 ? width * coarse : 0);
}

ListShape list_shape(int N, int dx, int dz, int k, size_t members)
{
    // G lanes serve a pair and must hold its k neighbours; as many of a
    // warp's pairs as shared memory allows are members of one point
    ListShape s;
    s.dxp = list_dxp(N, dx, k);
    s.k4 = k == 4;
    s.lanes = k <= 8 ? 8 : 16;
    s.width = 32 / s.lanes;
    // one member: a warp per point (so few pairs leave warps idle, and a point's
    // chain of steps is shorter over 32 lanes)
    if (members == 1) {
        s.lanes = 32;
        s.width = 1;
        return s;
    }
    while (s.width > 1 && (list_walk_x_bytes(N, dx, dz, k, s.width) > kListWalkSmem ||
                           (size_t)s.width / 2 >= members))
        s.width /= 2;
    return s;
}

bool list_fits(int N, int dx, int dz, int k)
{
    return list_walk_x_bytes(N, dx, dz, k, 1) <= kListWalkSmem;
}

int list_splits(long long blocks, int max_nq, size_t smem, int sms)
{
    // CTAs that fill whole waves; a CTA first loads its members' X values,
    // which costs about 1/32 of a walk over all points
    const long long resident = (long long)sms * (smem > kListHalfSmem ? 1 : 2);
    int splits = 1;
    double best = 1e300;
    for (int t = 1; t <= std::min(512, (max_nq + 15) / 16); ++t) {
        const double waves = (double)((blocks * t + resident - 1) / resident);
        const double cost = waves * (1.0 / t + 1.0 / 32.0);
        if (cost < 0.98 * best) {
            best = cost;
            splits = t;
        }
    }
    return splits;
}

static size_t list_build_smem(int cap_a, int cap_b, int queries)
{
    // a query's space also holds its sample: kSample distances of either kind
    const int a = std::max(cap_a, kSample - cap_b), b = cap_b;
    return (size_t)queries * (a + b) * sizeof(Entry) +
           (size_t)kTeams * (kBins * 4 + 2 * (size_t)std::max(a, b));
}

int list_build_queries(int cap_a, int cap_b)
{
    for (int q = 8; q > 2; q >>= 1)
        if (list_build_smem(cap_a, cap_b, q) <= 110 * 1024) return q;
    return 2;
}

template <int G, bool NEAR>
static const void *walk_kernel_g(const ListShape &s)
{
    if (s.k4) {
        if constexpr (G != 16) {
            switch (s.dxp) {
            case 1: return reinterpret_cast<const void *>(&list_walk_kernel<G, NEAR, 1, true>);
            case 2: return reinterpret_cast<const void *>(&list_walk_kernel<G, NEAR, 2, true>);
            case 4: return reinterpret_cast<const void *>(&list_walk_kernel<G, NEAR, 4, true>);
            default: return reinterpret_cast<const void *>(&list_walk_kernel<G, NEAR, 0, true>);
            }
        }
        return nullptr;
    }
    if (s.dxp == 1) return reinterpret_cast<const void *>(&list_walk_kernel<G, NEAR, 1, false>);
    return reinterpret_cast<const void *>(&list_walk_kernel<G, NEAR, 0, false>);
}

static const void *walk_kernel(const ListShape &s)
{
    if (s.lanes == 32) return walk_kernel_g<32, true>(s);
    if (s.lanes == 8) return s.width == 4 ? walk_kernel_g<8, true>(s) : walk_kernel_g<8, false>(s);
    return s.width == 2 ? walk_kernel_g<16, true>(s) : walk_kernel_g<16, false>(s);
}

static cudaError_t prepare_build(int queries)
{
    const void *f = queries == 2   ? reinterpret_cast<const void *>(&list_build_kernel<2>)
                    : queries == 4 ? reinterpret_cast<const void *>(&list_build_kernel<4>)
                                   : reinterpret_cast<const void *>(&list_build_kernel<8>);
    return cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, 220 * 1024);
}

static cudaError_t prepare_walk(const ListShape &s)
{
    const void *f = walk_kernel(s);
    if (!f) return cudaSuccess;   // no group has this shape
    return cudaFuncSetAttribute(
        f, cudaFuncAttributeMaxDynamicSharedMemorySize,
        (int)(kListWalkSmem + list_walk_head(true, kListWalkThreads / 32)));
}

cudaError_t list_prepare(const ListShape &s, int queries, uint64_t *done)
{
    const int near = s.width == 32 / s.lanes;
    const int bit = ((s.lanes / 16 * 2 + near) * 5 + s.dxp) * 2 + (s.k4 ? 1 : 0);   // below 60
    const int build = 60 + queries / 4;   // 2, 4 or 8
    cudaError_t e = cudaSuccess;
    if (!(*done >> build & 1)) e = prepare_build(queries);
    if (e == cudaSuccess && !(*done >> bit & 1)) e = prepare_walk(s);
    if (e == cudaSuccess) *done |= 1ull << build | 1ull << bit;
    return e;
}

cudaError_t list_prepare_attributes()
{
    cudaError_t e = cudaSuccess;
    for (int queries = 2; queries <= 8 && e == cudaSuccess; queries *= 2)
        e = prepare_build(queries);
    for (int lanes = 8; lanes <= 32; lanes *= 2)
        for (int width = 32 / lanes; width >= 1; width /= 2)
            for (int dxp : {1, 2, 4, 0})
                for (int k4 = 0; k4 < 2 && e == cudaSuccess; ++k4)
                    e = prepare_walk(ListShape{lanes, width, dxp, k4 != 0});
    return e;
}

cudaError_t launch_list_build(const ListLaunch &L, long long n_items, int queries, int cap_a,
                              int cap_b, cudaStream_t st)
{
    if (n_items <= 0) return cudaSuccess;
    const size_t smem = list_build_smem(cap_a, cap_b, queries);
    if (n_items > 0x7fffffffLL || smem > 220 * 1024) return cudaErrorInvalidValue;
    const int a = std::max(cap_a, kSample - cap_b), b = cap_b;
    const unsigned grid = (unsigned)n_items;
    if (queries == 8) list_build_kernel<8><<<grid, kListBuildThreads, smem, st>>>(L, a, b);
    else if (queries == 4) list_build_kernel<4><<<grid, kListBuildThreads, smem, st>>>(L, a, b);
    else if (queries == 2) list_build_kernel<2><<<grid, kListBuildThreads, smem, st>>>(L, a, b);
    else return cudaErrorInvalidValue;
    return cudaGetLastError();
}

cudaError_t launch_list_walk(const ListLaunch &L, long long n_items, const ListShape &s,
                             size_t smem, cudaStream_t st)
{
    if (n_items <= 0) return cudaSuccess;
    const void *f = walk_kernel(s);
    if (!f || n_items > 0x7fffffffLL || smem > kListWalkSmem) return cudaErrorInvalidValue;
    // one CTA per SM where its X values fill the shared memory, else two
    const int threads = smem > kListHalfSmem ? kListWalkThreads : kListWalkThreads / 2;
    smem += list_walk_head(s.width == 32 / s.lanes, threads / 32);
    ListLaunch arg = L;
    int width = s.width;
    void *args[] = {&arg, &width};
    return cudaLaunchKernel(f, dim3((unsigned)n_items), dim3(threads), args, smem, st);
}

cudaError_t launch_rank_sort(const RankSortJob *jobs, int n_jobs, int n_items, cudaStream_t st)
{
    if (n_items <= 0) return cudaSuccess;
    rank_sort_kernel<<<n_items, 256, 0, st>>>(jobs, n_jobs);
    return cudaGetLastError();
}

}  // namespace teksg
