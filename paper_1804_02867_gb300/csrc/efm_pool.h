// efm_pool.h -- which memory pool a call's work area comes from.  Plain C++
// over an Api of two functions, so that the bookkeeping is tested on the host.
//
// Work areas have stream-ordered pools of their own, one per context, which
// keep what a call frees for the next.  In the default pool the small buffers
// that outlive a call (networks, results) come to lie between the large ones,
// and a call then has its arenas mapped anew: in a process with a dozen
// networks four genome-shaped targets took 35.6 ms a call, and take 22.6 with a
// pool of their own (alone in a process 22.7 either way).
//
// A pool belongs to the context it was made in and is found by that context's
// id, which is never used twice: after a device is reset its old pool is not
// looked at again.
#pragma once
#include <cstdint>
#include <mutex>

namespace efm {

// Api: using Pool (a pointer type); bool context(uint64_t &id), the current
// context's id; Pool create(), nullptr if there is none to be had; void
// trim(Pool, size_t keep).
template <typename Api>
class WorkPools {
public:
    static constexpr int kMax = 64;

    // The current context's pool, made at its first use; nullptr: the default
    // pool (no context, no pool, or more contexts than there are entries).
    typename Api::Pool get()
    {
        uint64_t id = 0;
        if (!api.context(id)) return nullptr;
        std::lock_guard<std::mutex> lock(mu_);
        Entry *e = find(id, true);
        if (!e) return nullptr;
        if (!e->made) {
            e->pool = api.create();
            e->made = true;
        }
        return e->pool;
    }

    Api api;

private:
    struct Entry {
        uint64_t id;
        typename Api::Pool pool;
        bool made;
    };
    Entry *find(uint64_t id, bool add)
    {
        for (int i = 0; i < n_; ++i)
            if (e_[i].id == id) return &e_[i];
        if (!add || n_ == kMax) return nullptr;
        e_[n_] = Entry{id, nullptr, false};
        return &e_[n_++];
    }
    std::mutex mu_;
    Entry e_[kMax];
    int n_ = 0;
};

}  // namespace efm
