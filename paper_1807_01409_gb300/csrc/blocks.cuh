// The bookkeeping of a context's block cache (host code, no CUDA calls).
//
// Device blocks a context has freed and hands out again without a driver call (a
// plan on a small store makes some thirty small allocations per operator chain).
// Everything a context does is ordered on its one stream, so a block may be
// reused by the next launch.  Sizes are rounded up to a class (four per power of
// two); larger blocks, and blocks freed while MAX_HELD bytes are held, go back to
// the pool.  Measured on GB300, with the freed sets' events kept as well: a lookup in
// a 1M-triple store 41.5 -> 36.0 us, eight plans on it 2.53 -> 2.38 ms.
#pragma once

#include <stddef.h>

#include <mutex>
#include <new>
#include <unordered_map>

namespace tid {

class BlockCache {
  public:
    static constexpr size_t MAX_BLOCK = (size_t)64 << 20, MAX_HELD = (size_t)256 << 20;
    static constexpr int CLASSES = 4 * 18 + 1;  // 256 B << 18 = 64 MB
    static constexpr int LARGE = -1;

    // Class c holds blocks of (4 + c % 4) / 4 * 256 << (c / 4) bytes.
    static size_t class_bytes(int c) { return ((size_t)64 << (c / 4)) * (4 + c % 4); }
    static int class_of(size_t bytes) {
        int c = 0;
        while (class_bytes(c) < bytes) ++c;
        return c;
    }

    // A held block of the class, or null.
    void *take(int cls) {
        std::lock_guard<std::mutex> lk(mu_);
        Node *n = free_[cls];
        if (!n) return nullptr;
        free_[cls] = n->second.next;
        n->second.state = USED;
        held_ -= class_bytes(cls);
        return n->first;
    }

    // A block from the pool, of class_bytes(cls), is in use (LARGE: above the classes).  Without host memory for
    // the entry the block stays unknown and is freed to the pool.
    void add(void *p, int cls) noexcept {
        std::lock_guard<std::mutex> lk(mu_);
        try {
            known_[p] = Block{cls, USED, nullptr};
        } catch (const std::bad_alloc &) {
        }
    }

    // What becomes of a freed block: KEPT here; POOL, the caller's to give back; TWICE, freed
    // though nobody has it (never held twice: two owners would share it).
    // aside: freed while a graph is captured, which may read it at every run: not
    // handed out again and not the pool's either, until the context goes.
    enum Freed { KEPT, POOL, TWICE };
    Freed put(void *p, bool aside = false) noexcept {  // allocates nothing: freeing cannot fail
        std::lock_guard<std::mutex> lk(mu_);
        auto it = known_.find(p);
        if (it == known_.end()) return POOL;
        Block &b = it->second;
        if (b.state != USED) return TWICE;
        if (aside) {
            b.state = ASIDE;
            return KEPT;
        }
        const size_t bytes = b.cls == LARGE ? MAX_HELD + 1 : class_bytes(b.cls);
        if (held_ + bytes > MAX_HELD) {
            known_.erase(it);
            return POOL;
        }
        b.state = HELD;
        b.next = free_[b.cls];
        free_[b.cls] = &*it;
        held_ += bytes;
        return KEPT;
    }

    // Gives back(p) every held block (all: those set aside too); false if there are none.
    template <class Back>
    bool drop(Back back, bool all = false) {
        std::lock_guard<std::mutex> lk(mu_);
        bool any = false;
        for (auto it = known_.begin(); it != known_.end();) {
            if (it->second.state == HELD || (all && it->second.state == ASIDE)) {
                back(it->first);
                it = known_.erase(it);
                any = true;
            } else {
                ++it;
            }
        }
        for (Node *&f : free_) f = nullptr;
        held_ = 0;
        return any;
    }

    size_t held() const { return held_; }

  private:
    enum State { USED, HELD, ASIDE };
    struct Block;
    using Node = std::pair<void *const, Block>;  // an element of known_: stays where it is
    struct Block {
        int cls;
        State state;
        Node *next;  // in the class's free list
    };
    std::unordered_map<void *, Block> known_;  // blocks of a class, in use or held
    Node *free_[CLASSES] = {nullptr};
    size_t held_ = 0;
    std::mutex mu_;
};

}  // namespace tid
