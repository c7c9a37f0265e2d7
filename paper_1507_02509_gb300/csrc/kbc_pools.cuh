// Host resources kept between objects and calls, because making them costs
// more than a small problem computes.  Both pools are bounded, hand a resource
// to one owner at a time under a lock, and keep only what was made in a
// device's primary context, which is the one whose end can be told: a device
// has one at a time, so another id means that the device was reset and that
// what was kept went with the old one.  Contexts of several devices live side
// by side.  In a context that a program made itself nothing is kept.
//
// Rt supplies the runtime's calls:
//   Context context()                  the current context
//   int* host_alloc(size_t, bool)      pinned memory (true: for all contexts) or nullptr
//   void host_free(int*)
//   Plan, bool plan_create(int n, Plan*, size_t* work), void plan_destroy(Plan)
#pragma once

#include <cstddef>
#include <mutex>

namespace kbc {

// id: unique over the process's contexts; 0: not a primary context
struct Context {
    int device = -1;
    unsigned long long id = 0;
};

// Pinned status words of a handle, and where they came from: the page of a
// context, or (ctx 0) an allocation of their own.
struct FlagWords {
    int* p = nullptr;
    int device = -1;
    unsigned long long ctx = 0;
};

// 256 handles' status words in one page per device, kept for as long as the
// device's context (the first pinned allocation of a process without one takes
// 230 us); handles beyond them, and those of other contexts, have an
// allocation of their own.
template <class Rt>
class FlagPool {
public:
    static constexpr int kSlots = 256, kInts = 4, kDevices = 64;

    FlagWords get()
    {
        const Context c = Rt::context();
        if (c.id != 0 && c.device >= 0 && c.device < kDevices) {
            std::lock_guard<std::mutex> lk(mu_);
            Page& pg = page_[c.device];
            if (pg.ctx != c.id) {  // none yet, or it went with the context before this one
                pg = Page();
                pg.base = Rt::host_alloc(kSlots * kInts * sizeof(int), true);
                if (pg.base) pg.ctx = c.id;
            }
            for (int k = 0; pg.base && k < kSlots; ++k)
                if (!pg.used[k]) {
                    pg.used[k] = true;
                    return {pg.base + k * kInts, c.device, c.id};
                }
        }
        return {Rt::host_alloc(kInts * sizeof(int), false), -1, 0};
    }
    // the caller has waited for every copy into them
    void put(const FlagWords& w)
    {
        if (!w.p) return;
        if (w.ctx == 0) {
            Rt::host_free(w.p);
            return;
        }
        std::lock_guard<std::mutex> lk(mu_);
        Page& pg = page_[w.device];
        if (pg.ctx == w.ctx) pg.used[(w.p - pg.base) / kInts] = false;
    }

private:
    struct Page {
        int* base = nullptr;
        unsigned long long ctx = 0;
        bool used[kSlots] = {};
    };
    std::mutex mu_;
    Page page_[kDevices];
};

// FFT plans of kbc_spectrum by size (making one takes 0.3 to 0.5 ms, more than
// the transform of a 1024^2 field); the work area is the call's own.
template <class Rt>
class PlanPool {
public:
    static constexpr int kPlans = 8;
    using Plan = typename Rt::Plan;
    struct Entry {
        Plan plan{};
        size_t work = 0;
        int n = 0, device = -1;
        unsigned long long ctx = 0, age = 0;
        bool held = false;
    };

    // a plan that nobody else uses until put(); false when it cannot be made
    bool get(int n, Entry* out)
    {
        const Context c = Rt::context();
        if (c.id != 0) {
            std::lock_guard<std::mutex> lk(mu_);
            for (Entry& x : e_)
                if (x.held && x.n == n && x.ctx == c.id) {
                    *out = x;
                    x = Entry();
                    return true;
                }
        }
        Entry x;
        if (!Rt::plan_create(n, &x.plan, &x.work)) return false;
        x.n = n;
        x.device = c.device;
        x.ctx = c.id;
        *out = x;
        return true;
    }
    // In the context of get(); the caller has waited for the plan's work.
    // Takes a free place, that of a plan which went with its context, or that
    // of this context's least recently used plan, which is destroyed; plans of
    // other devices stay, and where those fill the pool x is destroyed.
    void put(Entry x)
    {
        Entry old = x;
        old.held = true;  // to be destroyed
        if (x.ctx != 0) {
            std::lock_guard<std::mutex> lk(mu_);
            Entry* to = nullptr;
            for (Entry& y : e_) {
                if (!y.held || (y.device == x.device && y.ctx != x.ctx)) {
                    y = Entry();
                    to = &y;
                    break;
                }
                if (y.ctx == x.ctx && (!to || y.age < to->age)) to = &y;
            }
            if (to) {
                old = *to;
                x.held = true;
                x.age = ++clock_;
                *to = x;
            }
        }
        if (old.held) Rt::plan_destroy(old.plan);
    }

private:
    std::mutex mu_;
    Entry e_[kPlans];
    unsigned long long clock_ = 0;
};

}  // namespace kbc
