"""How the CTAs of a batched launch share the jobs' walks and merges, run on
the host for made-up job lists: every walk and every merge in exactly one
share, and where a CTA has to give up, every job of the rest of its share is
reported (and no other)."""
import os
import subprocess

import pytest

from paper_1606_07413_gb300 import build as B

SRC = r"""
#include <cstdio>
#include <cstdlib>
#include <random>
#include <set>
#include <vector>
#include "qcs_shares.h"
using namespace qcs;

static int bad(const char *what, int trial) { printf("%s, trial %d\n", what, trial); return 1; }

int main()
{
    std::mt19937_64 rng(20240607);
    auto pick = [&](uint64_t n) { return (uint32_t)(rng() % n); };
    for (int trial = 0; trial < 400; trial++) {
        const uint32_t ctas = trial % 3 ? 152 : 1 + pick(40), nj = 1 + pick(trial & 1 ? 20 : 90), per = trial & 2 ? 24 : 16;
        const bool merges = trial & 4;
        std::vector<WalkLaunch> jobs(nj + 3);
        std::vector<uint32_t> heads(nj + 3), ids, tasks;
        for (uint32_t j = 0; j < jobs.size(); j++) {
            WalkLaunch &w = jobs[j];
            w = WalkLaunch{};
            w.lv.maskL = ~0ull >> 16;
            w.lv.dshift = 48 - (int)pick(13);
            w.steps = 1 + pick(64);
            w.n_walks = (int32_t)(16 * (1 + pick(trial & 8 ? 2 : 40)));
            w.qcap = 400;
            heads[j] = pick(3) ? pick(500) : pick(2);
            w.qhead = &heads[j];
            w.rewalk_budget = pick(3) ? 64 : 0;
            w.pend_in_n = pick(2) ? pick(50) : 0;
        }
        for (uint32_t j = 0; j < nj; j++) {
            const uint32_t job = (j * 7 + 3) % jobs.size(); // some slots unused, ids in no order
            bool seen = false;
            for (uint32_t k : ids) seen = seen || k == job;
            if (seen) continue;
            ids.push_back(job);
            for (int f = 0; f < jobs[job].n_walks; f += (int)per) {
                tasks.push_back(job);
                tasks.push_back((uint32_t)f);
            }
        }
        uint32_t n_tasks = (uint32_t)tasks.size() / 2, n_jobs = (uint32_t)ids.size();
        BatchArgs a{jobs.data(), tasks.data(), &n_tasks, ids.data(), &n_jobs};
        std::vector<std::vector<int>> times(jobs.size());
        for (uint32_t j : ids) times[j].assign(merges ? job_merges(jobs[j]) : (size_t)jobs[j].n_walks, 0);
        for (uint32_t cta = 0; cta < ctas; cta++) {
            // pass 0: all runs succeed.  pass 1: the CTA's runs from the stop-th on would fail
            std::vector<uint32_t> met, lost;
            const uint32_t stop = pick(4);
            for (int pass = 0; pass < 2; pass++) {
                uint32_t runs = 0;
                bool gone = false, again = false;
                auto run = [&](uint32_t job, uint32_t p0, uint32_t p1) {
                    if (!merges) p1 = std::min(p0 + p1, (uint32_t)jobs[job].n_walks);
                    again = again || gone; // called once more after it gave up
                    gone = pass == 1 && runs++ >= stop;
                    if (pass == 0) {
                        met.push_back(job);
                        for (uint32_t p = p0; p < p1; p++) times[job][p]++;
                    }
                    return !gone;
                };
                auto lose = [&](uint32_t job) { lost.push_back(job); };
                if (merges) merge_shares(a, cta, ctas, run, lose);
                else walk_shares(a, cta, ctas, per == 24 ? 1 : 8, per, run, lose);
                if (again) return bad("run after it gave up", trial);
                if (pass == 0 && !lost.empty()) return bad("lost without a failure", trial);
            }
            std::vector<uint32_t> want;
            if (stop < met.size()) want.assign(met.begin() + stop, met.end());
            if (lost != want) return bad("jobs of the rest of the share not reported", trial);
        }
        for (uint32_t j : ids)
            for (int t : times[j])
                if (t != 1) return bad("an item in no share or in two", trial);
    }
    puts("ok");
    return 0;
}
"""


def test_every_item_once_and_every_lost_job_reported(tmp_path):
    src, exe = tmp_path / "shares.cpp", tmp_path / "shares"
    src.write_text("#include <algorithm>\n" + SRC)
    subprocess.check_call([B.nvcc(), "-O1", "-std=c++17", "-I", B.CSRC, "-I", B.INCLUDE, str(src), "-o", str(exe)])
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout
