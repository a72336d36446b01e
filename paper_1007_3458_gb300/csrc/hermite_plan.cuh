// hermite_plan.cuh -- the schedule of the Hermite's sets, by one CTA of 1024
// threads: at the end of the one-CTA set builder (encounter.cu), or in a kernel of
// its own (hermite.cu) after the set builder of larger inputs.
#pragma once

#include "qym_internal.cuh"

namespace qym {

#ifndef QYM_HERM_NBIG
#define QYM_HERM_NBIG 24
#endif
constexpr int NBIG = QYM_HERM_NBIG;  // sets of at least this many members use a whole cluster

// The Hermite kernel's schedule for this step. A set's chain of block steps
// runs on one CTA (or one cluster) from start to end, so the step lasts as
// long as its longest set; which set that is can be foreseen, since a close
// pair stays close over consecutive steps. A set's predicted cost is the
// largest count of block steps among its members' sets of the previous step
// (hcost; 0 for rows that were in no set), raised per member by the set
// builder into hsetcost, which the plan reads and clears. Sets of at least
// NBIG members with the highest predicted cost (then the most members, then
// the lowest index) take the ncl clusters, one each; the other sets form the
// per-CTA queue in descending predicted cost, so the longest chains start
// first. With more than kPlanCap sets the queue keeps the set order and no
// cluster is used.
// One CTA of 1024 threads; the sets are ordered by a bitonic sort of 64-bit
// keys in shared memory.
constexpr int kPlanCap = 4096;
// When a system's step is split over several GPUs (own_hi > 0) this context
// integrates only the sets whose lowest row is its own: sets are numbered in
// the order of their lowest rows, so those are the index range [s_lo, s_hi).
__device__ __forceinline__ void hermite_plan(const Dev &d, int ncl) {
    __shared__ unsigned long long key[kPlanCap];
    __shared__ int wsum[32];
    __shared__ int s_range[2];
    const int tid = threadIdx.x;
    const int nall = (int)min((unsigned long long)d.max_sets, d.ctr[C_NSETS]);
    if (tid == 0) {
        int lo = 0, hi = nall;
        if (d.own_hi > 0) {
            // first set whose root is >= own_lo, and >= own_hi (roots ascend)
            int a = 0, b = nall;
            while (a < b) { const int m = (a + b) >> 1; if (d.set_root[m] < d.own_lo) a = m + 1; else b = m; }
            lo = a;
            b = nall;
            while (a < b) { const int m = (a + b) >> 1; if (d.set_root[m] < d.own_hi) a = m + 1; else b = m; }
            hi = a;
        }
        s_range[0] = lo;
        s_range[1] = hi;
    }
    __syncthreads();
    const int s_lo = s_range[0];
    const int nsets = s_range[1] - s_lo;
    if (ncl > kHermMaxClusters) ncl = kHermMaxClusters;
    for (int c = tid; c < kHermMaxClusters; c += blockDim.x) d.hcl[c] = -1;
    for (int k = tid; k < nall; k += blockDim.x)
        if (k < s_lo || k >= s_lo + nsets) d.hsetcost[k] = 0;
    if (nsets > kPlanCap) {
        for (int k = tid; k < nsets; k += blockDim.x) {
            d.hq[k] = s_lo + k;
            d.hsetcost[s_lo + k] = 0;
        }
        if (tid == 0) d.ctr[C_HNQ] = (unsigned long long)nsets;
        return;
    }
    int P = 1;
    while (P < nsets) P <<= 1;
    // key: predicted cost (31 bits) | members (16 bits) | 0xffff - set index
    // (set indices relative to s_lo)
    for (int k = tid; k < P; k += blockDim.x) {
        unsigned long long kk = 0;
        if (k < nsets) {
            const int sk = s_lo + k;
            const int n = d.set_start[sk + 1] - d.set_start[sk];
            const int cost = d.hsetcost[sk];
            d.hsetcost[sk] = 0;
            kk = ((unsigned long long)min(max(cost, 0), 0x7fffffff) << 32) |
                 ((unsigned long long)min(max(n, 0), 0xffff) << 16) | (unsigned long long)(0xffff - k);
        }
        key[k] = kk;
    }
    __syncthreads();
    // descending bitonic sort (padding keys are 0 and sink to the end)
    for (int size = 2; size <= P; size <<= 1) {
        for (int stride = size >> 1; stride > 0; stride >>= 1) {
            for (int k = tid; k < P; k += blockDim.x) {
                const int o = k ^ stride;
                if (o > k) {
                    const bool desc = (k & size) == 0;
                    const unsigned long long a = key[k], b = key[o];
                    if (desc ? a < b : a > b) {
                        key[k] = b;
                        key[o] = a;
                    }
                }
            }
            __syncthreads();
        }
    }
    // in sorted order: eligible = at least NBIG members; the first ncl
    // eligible sets go to the clusters, the rest keep their order in the queue
    constexpr int PER = kPlanCap / 1024;
    const int k0 = tid * PER;
    int e[PER], cnt = 0;
    for (int i = 0; i < PER; ++i) {
        const int k = k0 + i;
        e[i] = (k < nsets && (int)((key[k] >> 16) & 0xffff) >= NBIG) ? 1 : 0;
        cnt += e[i];
    }
    // exclusive prefix of cnt over the threads
    const int lane = tid & 31, w = tid >> 5;
    int incl = cnt;
    for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += t;
    }
    if (lane == 31) wsum[w] = incl;
    __syncthreads();
    int before = incl - cnt;
    for (int k = 0; k < w; ++k) before += wsum[k];
    int total = 0;
    for (int k = 0; k < 32; ++k) total += wsum[k];
    for (int i = 0; i < PER; ++i) {
        const int k = k0 + i;
        if (k >= nsets) break;
        const int set = s_lo + 0xffff - (int)(key[k] & 0xffff);
        if (e[i] && before < ncl) {
            d.hcl[before] = set;
        } else {
            d.hq[k - min(before, ncl)] = set;
        }
        before += e[i];
    }
    if (tid == 0) d.ctr[C_HNQ] = (unsigned long long)(nsets - min(total, ncl));
}

}  // namespace qym
