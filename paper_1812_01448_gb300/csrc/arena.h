// Device memory of a mesh without allocator callbacks.  A cudaMalloc and its cudaFree cost about
// 60 us and a setup makes some 27 of them: blocks are cut, best fit, from a few chunks, those that a
// build keeps (the first chunk as large as a setup's arrays) apart from those made for what one call takes
// and returns, so that a call's work space, where it does not fit in what a build has left over, never
// makes a build's chunks grow.
// - A released block joins its free neighbours, and is reused only after the device has gone idle, as
//   cudaFree waits too: work on another stream that still reads it is safe.
// - Chunks that calls have returned go back to the device beyond kKeep bytes of them, and all of them
//   before a larger one is taken.
// - Blocks from kOwn on have a chunk each, and builds beyond 2 kGrow take chunks of kGrow: in one chunk for
//   all its arrays a 1M-triangle mesh's blocked plasma step took 6.54 to 6.61 us, so 6.37 us, as with a
//   cudaMalloc per array.  Its first build takes 170 us longer for it (1,500 us; 5,150 us with those).
// - Before an allocation fails, every chunk that is wholly free goes back.
// - A rebuild starts from the last build's chunks, unless they are less than half used or belong to
//   another device.
// Host only; the device is reached through Ops.
#pragma once

#include <algorithm>
#include <cstddef>
#include <vector>

namespace ue {

class Arena {
public:
    struct Ops {
        void* (*get)(size_t bytes);   // nullptr when refused
        void (*put)(void* p);
        void (*idle)();               // returns when nothing runs on the device
        int (*device)();              // the current device
    };
    static constexpr size_t kAlign = 256, kChunk = (size_t)2 << 20, kOwn = (size_t)16 << 20, kGrow = (size_t)64 << 20,
                            kKeep = (size_t)64 << 20;

    explicit Arena(const Ops& o) : ops_(o) {}
    Arena(const Arena&) = delete;
    Arena& operator=(const Arena&) = delete;
    ~Arena() { reset(false); }

    // The total of a build's blocks below kOwn: chunks for them are as large, or kGrow each, while it lasts.
    void reserve(size_t bytes) {
        size_t have = 0;
        for (const Chunk& c : chunks_) have += !c.temp && !c.own ? c.bytes : 0;
        reserve_ = bytes > have ? bytes - have : 0;
        first_ = reserve_ <= 2 * kGrow ? 2 * kGrow : kGrow;
    }

    // temp: a call's own, released before it returns.
    void* alloc(size_t bytes, bool temp) {
        bytes = up(bytes, kAlign);
        const bool own = !temp && bytes >= kOwn;
        if (void* p = cut(bytes, temp, own)) return p;
        size_t want = up(bytes, kChunk);
        if (temp) {   // room for a call's other blocks too
            trim(true, 0);
            want = std::max(want, up(std::min(held(false) / 8, kKeep / 4), kChunk));
        } else if (!own) {
            want = std::max(want, up(std::max(std::min(held(false) / 4, kGrow), std::min(reserve_, first_)), kChunk));
            reserve_ -= std::min(reserve_, want);
        }
        if (!grow(want, temp, own)) {   // little memory left: no more than asked for, then any place
            give_back();
            if (!grow(want, temp, own) && (want == bytes || !grow(bytes, temp, own))) return cut(bytes, temp, !own);
        }
        return cut(bytes, temp, own);
    }

    // False when p is not a block of this arena.
    bool release(void* p) {
        for (Chunk& c : chunks_)
            for (size_t i = 0; i < c.used.size(); ++i) {
                if (c.p + c.used[i].off != p) continue;
                ops_.idle();
                const Span s = c.used[i];
                c.used[i] = c.used.back();
                c.used.pop_back();
                size_t k = 0;
                while (k < c.free.size() && c.free[k].off < s.off) ++k;
                c.free.insert(c.free.begin() + k, s);
                join(c, k);
                if (k > 0) join(c, k - 1);
                if (!c.temp) live_ -= s.bytes;
                else if (c.used.empty()) trim(true, kKeep);
                return true;
            }
        return false;
    }

    // Chunks that are wholly free, back to the device.
    void give_back() {
        trim(true, 0);
        trim(false, 0);
    }

    // All blocks free again.  keep: what the last build took stays for the next.
    void reset(bool keep) {
        for (Chunk& c : chunks_) {
            c.used.clear();
            c.free.assign(1, Span{0, c.bytes});
        }
        trim(true, keep ? kKeep : 0);
        const bool most = held(false) <= std::max(2 * peak_, kChunk);
        live_ = peak_ = reserve_ = 0;
        bool here = true;
        for (const Chunk& c : chunks_) here = here && c.device == ops_.device();
        if (keep && most && here) ops_.idle();
        else give_back();
    }

    size_t held() const { return held(false) + held(true); }

private:
    struct Span {
        size_t off, bytes;
    };
    struct Chunk {
        char* p;
        size_t bytes;
        bool temp, own;   // own: of one block from kOwn on
        int device;
        std::vector<Span> free, used;   // free: by offset, no two adjacent
    };
    Ops ops_;
    std::vector<Chunk> chunks_;
    size_t reserve_ = 0, first_ = 0, live_ = 0, peak_ = 0;   // live, peak: of the builds' chunks, in use, and most since reset

    static size_t up(size_t n, size_t to) { return (std::max<size_t>(n, 1) + to - 1) / to * to; }
    static void join(Chunk& c, size_t k) {   // free spans k and k + 1, if they touch
        if (k + 1 >= c.free.size() || c.free[k].off + c.free[k].bytes != c.free[k + 1].off) return;
        c.free[k].bytes += c.free[k + 1].bytes;
        c.free.erase(c.free.begin() + k + 1);
    }
    size_t held(bool temp) const {
        size_t n = 0;
        for (const Chunk& c : chunks_) n += c.temp == temp ? c.bytes : 0;
        return n;
    }
    bool grow(size_t bytes, bool temp, bool own) {
        void* p = ops_.get(bytes);
        if (!p) return false;
        chunks_.push_back(Chunk{(char*)p, bytes, temp, own, ops_.device(), {Span{0, bytes}}, {}});
        return true;
    }
    void* cut(size_t bytes, bool temp, bool own) {
        Chunk* best = nullptr;
        size_t at = 0;
        for (Chunk& c : chunks_)
            for (size_t k = 0; k < c.free.size(); ++k)
                if ((temp || (!c.temp && c.own == own)) && c.free[k].bytes >= bytes && (!best || c.free[k].bytes < best->free[at].bytes)) {
                    best = &c;
                    at = k;
                }
        if (!best) return nullptr;
        Span& f = best->free[at];
        const Span s{f.off, bytes};
        f.off += bytes;
        f.bytes -= bytes;
        if (f.bytes == 0) best->free.erase(best->free.begin() + at);
        best->used.push_back(s);
        if (!best->temp) peak_ = std::max(peak_, live_ += bytes);
        return best->p + s.off;
    }
    // wholly free chunks of one kind back to the device, the newest first, until `keep` bytes of them are left
    void trim(bool temp, size_t keep) {
        size_t spare = 0;
        for (const Chunk& c : chunks_) spare += c.temp == temp && c.used.empty() ? c.bytes : 0;
        for (size_t i = chunks_.size(); i-- > 0 && spare > keep;) {
            if (chunks_[i].temp != temp || !chunks_[i].used.empty()) continue;
            spare -= chunks_[i].bytes;
            ops_.put(chunks_[i].p);
            chunks_.erase(chunks_.begin() + i);
        }
    }
};

}  // namespace ue
