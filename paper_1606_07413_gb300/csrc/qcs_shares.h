// qcs_shares.h -- how the CTAs of a batched launch share the jobs' walks and
// merges (the tensor-core kernels of qcs_engine4.cu and qcs_quad.cu).  Plain
// integer arithmetic on the launch's lists, so that the host can run it too.
#pragma once

#include <cstdint>

#include "qcs_internal.h"

namespace qcs {

__host__ __device__ inline int bits_of(uint64_t v)
{
#ifdef __CUDA_ARCH__
    return __popcll(v);
#else
    return __builtin_popcountll(v);
#endif
}

// A job's merges in a batched re-walk's work list: the carried ones, then the round's.
__host__ __device__ inline uint64_t job_merges(const WalkLaunch &w)
{
    const uint32_t queued = *w.qhead;
    return w.pend_in_n + (queued < w.qcap ? queued : w.qcap);
}

// A batched re-walk's shares: the CTAs take equal parts of all jobs' work, a
// merge of a job counting about its evaluations of f: three trail lengths, or
// the budget.  (By merges alone the CTAs that met the jobs of small theta, 64
// evaluations to a merge, took three times as long as the others.)
__host__ __device__ inline uint64_t merge_weight(const WalkLaunch &w)
{
    const int d = bits_of(w.lv.maskL) - w.lv.dshift; // theta = 2^-d
    const uint64_t len = 3ull << (d < 20 ? d : 20);
    return w.rewalk_budget && w.rewalk_budget < len ? (uint64_t)w.rewalk_budget : len;
}

// Few jobs: every CTA works for one of them alone.  A job gets one CTA and of
// the others a part in proportion to its weight, and its CTAs share its items
// evenly, in units of `unit`.  A CTA that takes up two jobs runs them one after
// the other, each as long as its longest chain (a re-walk: up to 64 dependent
// evaluations) with its slots partly empty.  With fewer CTAs to a job the
// one CTA more or less that a job gets would cost as much.  (13 n = 4 and 11
// n = 3 jobs, ms a round: walks 1.42 -> 1.33 and 0.46 -> 0.31, re-walks 0.74 ->
// 0.51 and 0.43 -> 0.36.)  job is ~0 if there is no item for this CTA; false:
// more than a job to ctas_per_job CTAs.  items(w, count, weight) tells a job's
// items.
struct JobShare {
    uint32_t job, p0, p1;
};
template <class Items>
__host__ __device__ __forceinline__ bool own_job(const BatchArgs &a, uint32_t cta, uint32_t ctas,
                                                 uint32_t ctas_per_job, uint32_t unit, Items items, JobShare &s)
{
    const uint32_t nj = *a.n_jobs;
    uint64_t total = 0;
    uint32_t n = 0;
    for (uint32_t j = 0; j < nj; j++) {
        uint64_t cnt, wt;
        items(a.jobs[a.job_ids[j]], cnt, wt);
        total += cnt * wt;
        n += cnt != 0;
    }
    s.job = ~0u;
    if (n * ctas_per_job > ctas) return false;
    const uint64_t spare = ctas - n;
    uint64_t base = 0;
    uint32_t i = 0;
    for (uint32_t j = 0; j < nj; j++) {
        uint64_t cnt, wt;
        items(a.jobs[a.job_ids[j]], cnt, wt);
        if (cnt == 0) continue;
        const uint32_t c0 = i + (uint32_t)(base * spare / total);
        base += cnt * wt;
        const uint32_t c1 = ++i + (uint32_t)(base * spare / total);
        if (cta < c0 || cta >= c1) continue;
        const uint64_t units = (cnt + unit - 1) / unit, r = cta - c0, c = c1 - c0, end = units * (r + 1) / c * unit;
        s.p0 = (uint32_t)(units * r / c) * unit;
        s.p1 = (uint32_t)(cnt < end ? cnt : end);
        if (s.p0 < s.p1) s.job = a.job_ids[j];
    }
    return true;
}

// Walk a CTA's share of the jobs' walks: run(job, first walk, number) for every
// job that it meets, in order.  Few jobs: own_job; else a contiguous range of
// tasks of per_task walks, neighbouring ones of one job together.  Where run
// returns false (a bounded wait ran out and the CTA cannot go on), lost(job)
// is told for that job and for every further one of the share: their round is
// not complete.
template <class Run, class Lost>
__host__ __device__ __forceinline__ void walk_shares(const BatchArgs &a, uint32_t cta, uint32_t ctas, uint32_t unit,
                                                     uint32_t per_task, Run run, Lost lost)
{
    JobShare s;
    if (own_job(a, cta, ctas, 8, unit,
                [](const WalkLaunch &w, uint64_t &cnt, uint64_t &wt) {
                    cnt = (uint64_t)w.n_walks;
                    wt = w.steps; // of every walk as many
                },
                s)) {
        if (s.job != ~0u && !run(s.job, s.p0, s.p1 - s.p0)) lost(s.job);
        return;
    }
    const uint32_t nt = *a.n_tasks, t_end = (uint32_t)(((uint64_t)nt * (cta + 1)) / ctas);
    bool ok = true;
    for (uint32_t task = (uint32_t)(((uint64_t)nt * cta) / ctas); task < t_end;) {
        const uint32_t job = a.tasks[2 * task], first = a.tasks[2 * task + 1];
        uint32_t last = task + 1;
        while (last < t_end && a.tasks[2 * last] == job) last++;
        ok = ok && run(job, first, (last - task) * per_task);
        if (!ok) lost(job);
        task = last;
    }
}

// The same for the jobs' merges: run(job, its first merge, the end of its merges).
template <class Run, class Lost>
__host__ __device__ __forceinline__ void merge_shares(const BatchArgs &a, uint32_t cta, uint32_t ctas, Run run,
                                                      Lost lost)
{
    JobShare s;
    if (own_job(a, cta, ctas, 4, 1,
                [](const WalkLaunch &w, uint64_t &cnt, uint64_t &wt) {
                    cnt = job_merges(w);
                    wt = merge_weight(w);
                },
                s)) {
        if (s.job != ~0u && !run(s.job, s.p0, s.p1)) lost(s.job);
        return;
    }
    const uint32_t nj = *a.n_jobs;
    uint64_t total = 0;
    for (uint32_t j = 0; j < nj; j++) {
        const WalkLaunch &w = a.jobs[a.job_ids[j]];
        total += job_merges(w) * merge_weight(w);
    }
    const uint64_t lo = total / ctas * cta + total % ctas * cta / ctas;
    const uint64_t hi = total / ctas * (cta + 1) + total % ctas * (cta + 1) / ctas;
    uint64_t base = 0;
    bool ok = true;
    for (uint32_t j = 0; j < nj && base < hi; j++) {
        const uint32_t job = a.job_ids[j];
        const WalkLaunch &w = a.jobs[job];
        const uint64_t cnt = job_merges(w), wt = merge_weight(w), at = base;
        base += cnt * wt;
        if (base <= lo) continue;
        // a merge belongs to the share its first unit lies in
        const uint64_t p0 = lo > at ? (lo - at + wt - 1) / wt : 0, p1 = hi < base ? (hi - at + wt - 1) / wt : cnt;
        if (p0 >= p1) continue;
        ok = ok && run(job, (uint32_t)p0, (uint32_t)p1);
        if (!ok) lost(job);
    }
}

} // namespace qcs
