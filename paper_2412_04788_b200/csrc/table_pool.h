// Device memory of handles, kept for the next handle.
//
// A handle's tables take tens of KB, and a program that asks one question per set of tables makes and
// destroys a handle per question: cudaMalloc and cudaFree (which maps, unmaps and waits for the device)
// were most of such a question's time (504 configs, answer read on the host: 830 to 2,300 us by box, 150-170
// with the memory kept and the tables uploaded in one copy instead of ten).
//
// What is kept: at most PER_CONTEXT blocks of at most BYTES each per context, TOTAL blocks in all; larger
// ones, and any beyond these numbers, are freed, and so are all of a context's when an allocation in it fails and
// those of the context then current when the library is unloaded.
//
// A block carries the context it was allocated in and is handed out under that context only: an address means nothing
// under another one.  Blocks of other contexts stay where they are (those of a context that is gone are never asked
// for again: a context's id is not used twice).
//
// Dev is the device behind it (guide_api.cu: the CUDA runtime), all static:
//   context(make)        id of the calling thread's current context (make: one is made current if there is none); 0: not to be had
//   alloc(&p, bytes)     0, or an error code;   out_of_memory(code);   release(p)
//   wait()               everything queued on the device has completed; false: could not be waited for
#pragma once
#include <cstddef>
#include <mutex>

namespace guide {

struct TableBlock {
    void *p = nullptr;
    size_t bytes = 0;
    unsigned long long context = 0;
};

template <class Dev>
class TablePool {
public:
    static constexpr size_t PER_CONTEXT = 4, BYTES = 1u << 20, TOTAL = 64, GRAIN = 64 * 1024;

    int take(size_t need, TableBlock *out) {
        const unsigned long long ctx = Dev::context(true);
        if (ctx) {
            std::lock_guard<std::mutex> lock(mu);
            size_t best = n;
            for (size_t i = 0; i < n; i++)
                if (kept[i].context == ctx && kept[i].bytes >= need && (best == n || kept[i].bytes < kept[best].bytes)) best = i;
            if (best < n) {
                *out = kept[best];
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

    // Back from a destroyed handle: kept once the device has been waited for, as freeing it would have done, so whoever
    // gets it next may write it on any stream.
    void give(const TableBlock &b) {
        if (b.context != 0 && b.bytes <= BYTES && Dev::context(false) == b.context && Dev::wait()) {
            std::lock_guard<std::mutex> lock(mu);
            size_t mine = 0;
            for (size_t i = 0; i < n; i++) mine += kept[i].context == b.context;
            if (mine < PER_CONTEXT && n < TOTAL) { kept[n++] = b; return; }
        }
        Dev::release(b.p);
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
    void remove(size_t i) { kept[i] = kept[--n]; }
    std::mutex mu;
    TableBlock kept[TOTAL];                                    // a fixed array: nothing here allocates host memory or throws
    size_t n = 0;
};

}  // namespace guide
