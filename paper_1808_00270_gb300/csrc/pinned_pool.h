// pinned_pool.h -- page-locked staging of results read back, kept for the next
// read of any context: allocating it costs more than most reads.  At most `most`
// bytes are kept, the rest is freed when it is given back, and all of it with the
// last context.  Safe with several host threads.
#pragma once

#include <cstddef>
#include <mutex>
#include <vector>

namespace gld {

struct Pinned {
    char* p = nullptr;
    size_t cap = 0;
};

class PinnedPool {
public:
    using Alloc = void* (*)(size_t);  // nullptr: no room
    using Free = void (*)(void*);
    PinnedPool(Alloc a, Free f, size_t most) : alloc(a), free_(f), most(most) {}
    PinnedPool(const PinnedPool&) = delete;
    PinnedPool& operator=(const PinnedPool&) = delete;

    void enter()
    {
        std::lock_guard<std::mutex> lock(mu);
        ++users;
    }

    void leave()
    {
        std::vector<Pinned> last;
        {
            std::lock_guard<std::mutex> lock(mu);
            if (--users > 0) return;
            last.swap(kept);
        }
        for (const Pinned& b : last) free_(b.p);
    }

    Pinned take(size_t bytes)
    {
        Pinned b;
        {
            std::lock_guard<std::mutex> lock(mu);
            size_t best = kept.size();
            for (size_t k = 0; k < kept.size(); ++k)
                if (kept[k].cap >= bytes && (best == kept.size() || kept[k].cap < kept[best].cap)) best = k;
            if (best < kept.size()) {
                b = kept[best];
                kept.erase(kept.begin() + (long)best);
                return b;
            }
        }
        b.cap = bytes > ((size_t)1 << 16) ? bytes : (size_t)1 << 16;
        b.p = (char*)alloc(b.cap);
        return b.p ? b : Pinned{};
    }

    void give(Pinned b)
    {
        if (!b.p) return;
        {
            std::lock_guard<std::mutex> lock(mu);
            size_t all = b.cap;
            for (const Pinned& x : kept) all += x.cap;
            if (users > 0 && all <= most) {
                kept.push_back(b);
                return;
            }
        }
        free_(b.p);
    }

private:
    Alloc alloc;
    Free free_;
    size_t most;
    std::mutex mu;
    std::vector<Pinned> kept;
    int users = 0;
};

}  // namespace gld
