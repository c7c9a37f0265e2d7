"""The pools of pinned status words and FFT plans, with the runtime's calls
replaced by counting ones: handles and plans of several contexts, destroyed in
every order, resets and contexts that nothing is kept for."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <algorithm>
#include <cstdio>
#include <cstdlib>
#include <map>
#include <vector>
#include "kbc_pools.cuh"

#define CHECK(c) do { if (!(c)) { std::printf("line %d: %s\n", __LINE__, #c); std::exit(1); } } while (0)

struct Rt {
    using Plan = int;
    static kbc::Context now;
    static std::map<int*, size_t> pinned;                      // live allocations
    static std::map<int, unsigned long long> plans;            // live plans, their context
    static int next_plan, allocs;
    static kbc::Context context() { return now; }
    static int* host_alloc(size_t bytes, bool)
    {
        int* p = static_cast<int*>(std::calloc(1, bytes));
        pinned[p] = bytes;
        ++allocs;
        return p;
    }
    static void host_free(int* p)
    {
        CHECK(pinned.count(p) == 1);  // a base address, freed once
        pinned.erase(p);
        std::free(p);
    }
    static bool plan_create(int n, int* plan, size_t* work)
    {
        *plan = ++next_plan;
        *work = n;
        plans[*plan] = now.id;
        return true;
    }
    static void plan_destroy(int plan)
    {
        CHECK(plans.count(plan) == 1 && plans[plan] == now.id);  // live, in its own context
        plans.erase(plan);
    }
};
kbc::Context Rt::now;
std::map<int*, size_t> Rt::pinned;
std::map<int, unsigned long long> Rt::plans;
int Rt::next_plan = 0, Rt::allocs = 0;

static kbc::Context ctx(int device, unsigned long long id)
{
    kbc::Context c;
    c.device = device;
    c.id = id;
    return c;
}

static bool live(const int* p)
{
    for (auto& a : Rt::pinned)
        if (p >= a.first && p + 4 <= a.first + a.second / sizeof(int)) return true;
    return false;
}

int main()
{
    using Flags = kbc::FlagPool<Rt>;
    using Plans = kbc::PlanPool<Rt>;
    const kbc::Context dev[3] = {ctx(0, 11), ctx(1, 12), ctx(0, 0)};  // two devices, a context of a program's own
    {
        // handles made on the contexts in turn, destroyed in every order
        static Flags pool;
        std::vector<int> order = {0, 1, 2, 3, 4, 5};
        do {
            kbc::FlagWords w[6];
            for (int k = 0; k < 6; ++k) {
                Rt::now = dev[k % 3];
                w[k] = pool.get();
                for (int j = 0; j < k; ++j) CHECK(w[j].p + 4 <= w[k].p || w[k].p + 4 <= w[j].p);
            }
            for (int j = 0; j < 6; ++j) {
                Rt::now = dev[order[j] % 3];
                pool.put(w[order[j]]);
                for (int i = j + 1; i < 6; ++i) CHECK(live(w[order[i]].p));
            }
            CHECK(Rt::pinned.size() == 2);  // the devices' pages, nothing else
        } while (std::next_permutation(order.begin(), order.end()));
        // more handles than a page has slots, on both devices
        std::vector<kbc::FlagWords> many;
        for (int k = 0; k < 2 * Flags::kSlots + 40; ++k) {
            Rt::now = dev[k & 1];
            many.push_back(pool.get());
        }
        CHECK(Rt::pinned.size() == 2 + 40);
        for (size_t k = 0; k < many.size(); ++k) {
            pool.put(many[k]);
            for (size_t j = k + 1; j < many.size(); ++j) CHECK(live(many[j].p));
        }
        CHECK(Rt::pinned.size() == 2);
        // device 0 is reset: its page goes with the context, the handle's words too
        Rt::now = dev[0];
        kbc::FlagWords before = pool.get();
        Rt::now = ctx(0, 21);
        kbc::FlagWords after = pool.get(), other = pool.get();
        CHECK(!(after.p <= before.p && before.p < after.p + Flags::kSlots * 4));
        pool.put(before);  // frees no slot of the new page
        kbc::FlagWords third = pool.get();
        CHECK(third.p != after.p && third.p != other.p && live(third.p));
        pool.put(after);
        pool.put(other);
        pool.put(third);
        pool.put(kbc::FlagWords());
    }
    {
        static Plans pool;
        auto use = [](kbc::Context c, int n) {
            Plans::Entry e;
            Rt::now = c;
            const int made = Rt::next_plan;
            CHECK(pool.get(n, &e) && Rt::plans.count(e.plan) == 1 && (int)e.work == n);
            pool.put(e);
            return Rt::next_plan == made;  // whether it was kept from before
        };
        // more sizes than places on two devices: bounded, and no plan is lost
        for (int k = 0; k < 20; ++k)
            for (int d = 0; d < 2; ++d) use(dev[d], 2 + 2 * k);
        CHECK((int)Rt::plans.size() <= Plans::kPlans);
        CHECK(use(dev[0], 40));  // the latest size
        CHECK(!use(dev[0], 2));
        for (int k = 0; k < 3; ++k) CHECK(!use(dev[2], 8));  // not kept, not leaked
        CHECK((int)Rt::plans.size() <= Plans::kPlans);
        // both devices are reset: their plans went with the contexts, the new ones' are kept
        Rt::plans.clear();
        for (int k = 0; k < 2 * Plans::kPlans; ++k) use(ctx(0, 31), 2 + 2 * k);
        CHECK(use(ctx(0, 31), 4 * Plans::kPlans));
        use(ctx(1, 32), 6);
        CHECK((int)Rt::plans.size() <= Plans::kPlans);
        // a plan that is in use is nobody else's
        Plans::Entry a, b;
        Rt::now = ctx(0, 31);
        use(Rt::now, 100);
        CHECK(pool.get(100, &a) && pool.get(100, &b) && a.plan != b.plan);
        pool.put(a);
        pool.put(b);
    }
    std::puts("ok");
    return 0;
}
"""


def test_pools_over_several_contexts(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host compiler")
    src = tmp_path / "pools.cpp"
    src.write_text(PROGRAM)
    exe = tmp_path / "pools"
    csrc = os.path.join(ROOT, "paper_1507_02509_gb300", "csrc")
    subprocess.run([cxx, "-std=c++17", "-O1", "-Wall", "-Werror", "-I", csrc, str(src), "-o", str(exe), "-pthread"],
                   check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout + r.stderr
