// Device memory that a scene keeps for the calls on one stream, and when it may
// move.
//
// A call made while its stream is being captured leaves its buffers' addresses
// in the captured graph, which may be replayed for as long as the scene lives.
// Such a buffer is never freed before the scene: where a larger one takes its
// place it is retired.  A buffer of no captured call is freed then, after the
// stream has drained.
//
// Mem is where the memory comes from: int alloc(void**, size_t) (0, kNoMemory
// or another error of its own), void release(void*), int drain() (waits for
// the stream's queued work; 0 or an error), size_t spare() (what optional
// memory may take now).
#pragma once
#include <stddef.h>

#include <new>
#include <vector>

namespace qrt {

constexpr int kNoMemory = -1, kCapturing = -2;

struct StreamBuffer {
    void* ptr = nullptr;
    size_t bytes = 0;
    bool captured = false;             // its address is in a captured graph
    size_t refused = ~size_t(0);       // the least optional size that could not be had
};

// Lets go of b's memory (the stream has drained).
template <class Mem>
void let_go(StreamBuffer& b, std::vector<void*>& retired, Mem& mem) {
    if (b.ptr && b.captured) {
        try {
            retired.push_back(b.ptr);
        } catch (const std::bad_alloc&) {  // stays allocated, with nobody to free it
        }
    } else if (b.ptr) {
        mem.release(b.ptr);
    }
    b.ptr = nullptr;
    b.bytes = 0;
    b.captured = false;
}

// Makes b hold at least `bytes`; kCapturing where that takes an allocation
// during a capture.
template <class Mem>
int need(StreamBuffer& b, size_t bytes, bool capturing, std::vector<void*>& retired, Mem& mem) {
    if (b.bytes >= bytes) {
        b.captured = b.captured || capturing;
        return 0;
    }
    if (capturing) return kCapturing;
    int e = b.ptr ? mem.drain() : 0;
    if (e) return e;
    let_go(b, retired, mem);
    e = mem.alloc(&b.ptr, bytes);
    if (e) {
        b.ptr = nullptr;
        return e;
    }
    b.bytes = bytes;
    return 0;
}

// Makes b hold `count` times `unit` bytes, or as many as may be spared, if that
// memory can be had outside a capture, and leaves it as it is otherwise.  A
// size that was refused, or cut, is not tried again.
template <class Mem>
int want(StreamBuffer& b, size_t unit, size_t count, bool capturing, std::vector<void*>& retired, Mem& mem) {
    size_t bytes = unit * count;
    if (b.bytes >= bytes || capturing || bytes >= b.refused) {
        b.captured = b.captured || (capturing && b.ptr);
        return 0;
    }
    const size_t spare = mem.spare();
    if (bytes > spare) {
        b.refused = bytes;
        bytes = spare / unit * unit;
        if (bytes <= b.bytes) return 0;
    }
    void* p = nullptr;
    int e = mem.alloc(&p, bytes);
    if (e == kNoMemory) {
        b.refused = bytes < b.refused ? bytes : b.refused;
        return 0;
    }
    if (e) return e;
    if (b.ptr && (e = mem.drain())) {
        mem.release(p);
        return e;
    }
    let_go(b, retired, mem);
    b.ptr = p;
    b.bytes = bytes;
    return 0;
}

}  // namespace qrt
