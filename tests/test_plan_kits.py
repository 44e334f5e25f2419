"""The pool of the plans' page-locked words and events (plan_kits.cuh), compiled
here against a fake of the CUDA calls that it makes: a kit whose stream was not
known to be idle, or whose context a device reset has ended, is never handed out
again, the pool stays bounded, and a failed creation leaves nothing behind."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDA = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")

SOURCE = r'''
#include <cassert>
#include <cstdio>
#include <cstdlib>
#include <set>
#include "plan_kits.cuh"

static std::set<void *> words, events;         // what lives in the fake context
static int made = 0, fail_after = -1;
static unsigned long long now = 1;             // its id (0: reset, none yet)
extern "C" {
cudaError_t cudaMallocHost(void **p, size_t n) {
    if (fail_after == 0) return cudaErrorMemoryAllocation;
    if (fail_after > 0) fail_after--;
    words.insert(*p = malloc(n));
    made++;
    return cudaSuccess;
}
cudaError_t cudaFreeHost(void *p) {
    assert(words.erase(p) == 1);
    free(p);
    return cudaSuccess;
}
cudaError_t cudaEventCreate(cudaEvent_t *e) {
    if (fail_after == 0) return cudaErrorMemoryAllocation;
    if (fail_after > 0) fail_after--;
    *e = (cudaEvent_t)malloc(1);
    events.insert((void *)*e);
    return cudaSuccess;
}
cudaError_t cudaEventDestroy(cudaEvent_t e) {
    assert(events.erase((void *)e) == 1);      // not one of a context that has ended
    free((void *)e);
    return cudaSuccess;
}
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes *a, const void *p) {
    a->type = words.count((void *)p) ? cudaMemoryTypeHost : cudaMemoryTypeUnregistered;
    return cudaSuccess;
}
static int get_id(void *, unsigned long long *id) { *id = now; return now ? 0 : 709; }
cudaError_t cudaGetDriverEntryPointByVersion(const char *, void **f, unsigned, unsigned long long,
                                             cudaDriverEntryPointQueryResult *r) {
    *f = (void *)get_id;
    *r = cudaDriverEntryPointSuccess;
    return cudaSuccess;
}
static unsigned long long next_id = 1;
cudaError_t cudaFree(void *) { if (!now) now = ++next_id; return cudaSuccess; }
cudaError_t cudaGetLastError(void) { return cudaSuccess; }
}
static void device_reset() { words.clear(); events.clear(); now = 0; }

using namespace spg;
int main() {
    PlanKits pool(100);
    PlanKit a, b;
    assert(context_id() == 1);
    // back from an idle stream: handed out again
    assert(pool.take(context_id(), 50, &a) == cudaSuccess && a.words == 100 && made == 1);
    pool.give(a, true, context_id());
    assert(pool.take(context_id(), 100, &b) == cudaSuccess && b.pinned == a.pinned && made == 1);
    // the wait for its stream failed: its words and events are freed instead
    pool.give(b, false, context_id());
    assert(words.empty() && events.empty());
    assert(pool.take(context_id(), 50, &a) == cudaSuccess && made == 2);
    // two plans at a time never share one
    assert(pool.take(context_id(), 50, &b) == cudaSuccess && b.pinned != a.pinned && made == 3);
    pool.give(a, true, context_id());
    pool.give(b, true, context_id());
    // more words than usual: made for the plan, not kept
    assert(pool.take(context_id(), 101, &a) == cudaSuccess && a.words == 101 && made == 4);
    pool.give(a, true, context_id());
    assert(words.size() == 2 && events.size() == 36);
    // a device reset ends what is kept: a new context gets new kits, and nothing of
    // the old one is handed out or destroyed
    assert(pool.take(context_id(), 50, &a) == cudaSuccess && made == 4);
    device_reset();
    const unsigned long long fresh = context_id();
    assert(fresh != 1 && fresh != 0);
    assert(pool.take(fresh, 50, &b) == cudaSuccess && made == 5 && words.count(b.pinned) == 1);
    pool.give(a, true, fresh);      // a plan that outlived the reset
    pool.give(b, true, fresh);
    assert(pool.take(fresh, 50, &a) == cudaSuccess && a.pinned == b.pinned && made == 5);
    pool.give(a, true, fresh);
    // bounded, also with the ended context's kits in it
    PlanKit many[40];
    for (auto &k : many) assert(pool.take(fresh, 50, &k) == cudaSuccess);
    for (auto &k : many) pool.give(k, true, fresh);
    assert(words.size() == PlanKits::kMost && events.size() == 18 * PlanKits::kMost);
    // a creation that fails half-way leaves nothing behind
    for (int at = 0; at < 19; at++) {
        PlanKits other(100);
        const size_t w = words.size(), e = events.size();
        fail_after = at;
        assert(other.take(fresh, 50, &a) == cudaErrorMemoryAllocation);
        fail_after = -1;
        assert(words.size() == w && events.size() == e);
    }
    // no context id to be had: nothing is kept
    PlanKits blind(100);
    assert(blind.take(0, 50, &a) == cudaSuccess);
    blind.give(a, true, 0);
    assert(words.count(a.pinned) == 0);
    puts("kits ok");
}
'''


@pytest.mark.skipif(not shutil.which("g++") or not os.path.isdir(CUDA), reason="needs g++ and CUDA's headers")
def test_kits_of_failed_waits_and_ended_contexts_are_not_reused(tmp_path):
    src, exe = tmp_path / "kits.cpp", tmp_path / "kits"
    src.write_text(SOURCE)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", CUDA, "-I",
                    os.path.join(ROOT, "paper_2408_14558_gb300", "csrc"), str(src), "-o", str(exe), "-pthread"],
                   check=True, timeout=300)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0 and "kits ok" in r.stdout, r.stdout + r.stderr
