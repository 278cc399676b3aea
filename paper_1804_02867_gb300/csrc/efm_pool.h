// efm_pool.h -- which memory pool a call's work area comes from.  Plain C++
// over an Api of four functions, so that the bookkeeping is tested on the host.
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
// looked at again.  What a pool holds unused is bounded: an eighth of the
// device's memory while networks are loaded (a 2^26 budget on a core-shaped
// network takes 26 GB of 288), a thirty-second once the last one is freed
// (9 GB: mapping memory anew costs about 1 ms a GB and giving it back 1.4, so
// a program that loads a network for each query of up to 2^24 states does not
// pay; at a 2^26 budget such a query of 67 ms takes 115).
#pragma once
#include <cstdint>
#include <mutex>

namespace efm {

// Api: using Pool (a pointer type); bool context(uint64_t &id), the current
// context's id; Pool create(), nullptr if there is none to be had; void
// trim(Pool), to what an idle pool may keep.
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

    // A network is loaded: returns its context's id, for release().
    uint64_t retain()
    {
        uint64_t id = 0;
        if (!api.context(id)) return 0;
        std::lock_guard<std::mutex> lock(mu_);
        Entry *e = find(id, true);
        if (e) ++e->users;
        return e ? id : 0;
    }

    // It is freed: the last one gives the pool's memory back.  A pool whose
    // context is not the current one is left alone (it may be gone).
    void release(uint64_t id)
    {
        if (id == 0) return;
        uint64_t now = 0;
        const bool known = api.context(now);
        std::lock_guard<std::mutex> lock(mu_);
        Entry *e = find(id, false);
        if (!e || --e->users > 0) return;
        if (known && now == id && e->pool) api.trim(e->pool);
    }

    Api api;

private:
    struct Entry {
        uint64_t id;
        typename Api::Pool pool;
        int users;
        bool made;
    };
    Entry *find(uint64_t id, bool add)
    {
        for (int i = 0; i < n_; ++i)
            if (e_[i].id == id) return &e_[i];
        if (!add || n_ == kMax) return nullptr;
        e_[n_] = Entry{id, nullptr, 0, false};
        return &e_[n_++];
    }
    std::mutex mu_;
    Entry e_[kMax];
    int n_ = 0;
};

}  // namespace efm
