// Device memory of handles, kept for the next handle.
//
// A handle's tables take tens of KB, and a program that asks one question per set of tables makes and
// destroys a handle per question: cudaMalloc and cudaFree (which maps, unmaps and waits for the device)
// were most of such a question's time (504 configs, answer read on the host: 830 to 2,300 us by box, 150-170
// with the memory kept and the tables uploaded in one copy instead of ten).
//
// What is kept: at most PER_CONTEXT blocks of at most BYTES each per context, the ones given back last, and TOTAL blocks in
// all; larger ones, and any beyond these numbers, are freed, and so are all of a context's when an allocation in it
// fails and those of the context then current when the library is unloaded.
//
// A block carries the context it was allocated in and is handed out under that context only: an address means nothing
// under another one.  Blocks of other contexts stay where they are (those of a context that is gone are never asked
// for again: a context's id is not used twice).
//
// A destroyed handle's kernels may still be running, and nothing waits for them here (waiting for the device is an error while any
// stream is being captured, and ends the capture; so a handle may be destroyed meanwhile).  A block therefore remembers the one stream
// its handle was used on and is handed out for an upload on that stream only, which comes after them.  Blocks of
// handles used on several streams, or in a capture (a graph may run anywhere), are freed, and freeing waits.
//
// Dev is the device behind it (guide_api.cu: the CUDA runtime), all static:
//   context(make)        id of the calling thread's current context (make: one is made current if there is none); 0: not to be had
//   alloc(&p, bytes)     0, or an error code;   out_of_memory(code);   release(p): once nothing on the device uses it
#pragma once
#include <cstddef>
#include <mutex>

namespace guide {

struct TableBlock {
    void *p = nullptr;
    size_t bytes = 0;
    unsigned long long context = 0;
    unsigned long long stream = 0;             // id of the stream that has used it since its upload (0: none has)
    bool one_stream = true;

    // id 0: a stream that is being captured, or whose id is not to be had
    void used_on(unsigned long long id) {
        if (id == 0 || (stream != 0 && stream != id)) one_stream = false;
        stream = id;
    }
};

template <class Dev>
class TablePool {
public:
    static constexpr size_t PER_CONTEXT = 4, BYTES = 1u << 20, TOTAL = 64, GRAIN = 64 * 1024;

    // for an upload on the stream of that id, which the caller waits for
    int take(size_t need, unsigned long long stream, TableBlock *out) {
        *out = TableBlock();
        const unsigned long long ctx = Dev::context(true);
        if (ctx) {
            std::lock_guard<std::mutex> lock(mu);
            size_t best = n;
            for (size_t i = 0; i < n; i++)
                if (kept[i].context == ctx && kept[i].bytes >= need && (kept[i].stream == 0 || kept[i].stream == stream) &&
                    (best == n || kept[i].bytes < kept[best].bytes)) best = i;
            if (best < n) {
                out->p = kept[best].p; out->bytes = kept[best].bytes; out->context = ctx;
                remove(best);
                return 0;
            }
        }
        out->bytes = (need + GRAIN - 1) / GRAIN * GRAIN;       // so that a block suits the next handle of about that size
        out->context = ctx;
        int e = Dev::alloc(&out->p, out->bytes);
        if (e && Dev::out_of_memory(e)) {
            drop(ctx);
            e = Dev::alloc(&out->p, out->bytes);
        }
        return e;
    }

    // back from a destroyed handle
    void give(const TableBlock &b) {
        void *freed = b.p;
        if (b.context != 0 && b.one_stream && b.bytes <= BYTES && Dev::context(false) == b.context) {
            std::lock_guard<std::mutex> lock(mu);
            size_t mine = 0, oldest = n;
            for (size_t i = n; i-- > 0;)
                if (kept[i].context == b.context) { mine++; oldest = i; }
            freed = nullptr;
            if (mine == PER_CONTEXT) { freed = kept[oldest].p; remove(oldest); }
            if (n < TOTAL) kept[n++] = b; else freed = b.p;
        }
        if (freed) Dev::release(freed);
    }

    ~TablePool() { drop(Dev::context(false)); }

    // frees the blocks of one context, which is the calling thread's
    void drop(unsigned long long ctx) {
        if (!ctx) return;
        std::lock_guard<std::mutex> lock(mu);
        for (size_t i = n; i-- > 0;)
            if (kept[i].context == ctx) { Dev::release(kept[i].p); remove(i); }
    }

private:
    void remove(size_t i) {                                    // oldest first
        for (n--; i < n; i++) kept[i] = kept[i + 1];
    }
    std::mutex mu;
    TableBlock kept[TOTAL];                                    // a fixed array: nothing here allocates host memory or throws
    size_t n = 0;
};

}  // namespace guide
