// Scratch memory and transform plans that a handle keeps from one call to the next.
//
// Bounded: the scratch and the kept plans' work areas together stay within `limit` bytes, and at
// most kMaxPlans plans are kept; what does not fit is allocated for the call and released by it.
// Given back: by release(), which an allocation that fails calls before it is tried again (retry),
// so that what a handle keeps never makes one of its own calls fail.
//
// Api provides the device calls (bool: success): alloc(void**, size_t), free(void*),
// plan(int N, Plan*, size_t* work_bytes), destroy(Plan).  Host code without CUDA, so that it runs
// against a fake Api.
#pragma once
#include <stddef.h>

#include <utility>
#include <vector>

namespace clk {

template <typename Api>
class KeptScratch {
public:
    using Plan = typename Api::Plan;
    // One call's scratch and plan; release(Use&) after the call.
    struct Use {
        void* mem = nullptr;
        Plan plan{};
        bool has_plan = false, own_mem = false, own_plan = false;
    };
    enum Result { OK, NO_MEMORY, NO_PLAN };
    static constexpr size_t kMaxPlans = 8;

    explicit KeptScratch(size_t limit) : limit_(limit) {}
    KeptScratch(const KeptScratch&) = delete;
    KeptScratch& operator=(const KeptScratch&) = delete;
    ~KeptScratch() { release(); }

    Result acquire(int N, size_t bytes, Use* u)
    {
        *u = Use{};
        if (mem_ && bytes <= bytes_) {
            u->mem = mem_;
        } else if (bytes + plan_bytes() <= limit_) {
            free_mem();
            if (!retry([&] { return Api::alloc(&mem_, bytes); })) {
                mem_ = nullptr;
                return NO_MEMORY;
            }
            bytes_ = bytes;
            u->mem = mem_;
        } else {
            if (!retry([&] { return Api::alloc(&u->mem, bytes); })) {
                u->mem = nullptr;
                return NO_MEMORY;
            }
            u->own_mem = true;
        }
        for (const Kept& k : plans_)
            if (k.N == N) {
                u->plan = k.plan;
                u->has_plan = true;
                return OK;
            }
        size_t work = 0;
        if (!Api::plan(N, &u->plan, &work)) {
            // the other sizes' plans, and the scratch unless this call has it
            drop_plans();
            if (u->own_mem) free_mem();
            if (!Api::plan(N, &u->plan, &work)) return NO_PLAN;
        }
        u->has_plan = true;
        if (plans_.size() < kMaxPlans && bytes_ + plan_bytes() + work <= limit_) plans_.push_back({N, u->plan, work});
        else u->own_plan = true;
        return OK;
    }
    void release(Use& u)
    {
        if (u.own_plan) Api::destroy(u.plan);
        if (u.own_mem) Api::free(u.mem);
        u = Use{};
    }
    void release()
    {
        free_mem();
        drop_plans();
    }
    // An allocation `f` (true: success) of the handle that keeps this: tried again without it.
    template <typename F>
    bool retry(F f)
    {
        if (f()) return true;
        if (!mem_ && plans_.empty()) return false;
        release();
        return f();
    }
    size_t kept_bytes() const { return bytes_ + plan_bytes(); }

private:
    struct Kept {
        int N;
        Plan plan;
        size_t work;
    };
    size_t plan_bytes() const
    {
        size_t b = 0;
        for (const Kept& k : plans_) b += k.work;
        return b;
    }
    void free_mem()
    {
        if (mem_) Api::free(mem_);
        mem_ = nullptr;
        bytes_ = 0;
    }
    void drop_plans()
    {
        for (const Kept& k : plans_) Api::destroy(k.plan);
        plans_.clear();
    }
    const size_t limit_;
    void* mem_ = nullptr;
    size_t bytes_ = 0;
    std::vector<Kept> plans_;
};

}  // namespace clk
