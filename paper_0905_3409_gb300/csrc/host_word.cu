// host_word.cu -- page-locked words from slabs.
//
// cudaMallocHost and cudaFreeHost take 0.24 ms and more, whatever the size: with a word of its
// own each, creating and destroying a 64^2 grid took 482 us, with shared ones 154.  So words
// come from slabs of 1024 (one page), one list of slabs per context, because a slab goes with
// its context (cudaDeviceReset).  The last slab of a context is kept for the next handle, one
// that falls empty beside another is freed.
#include <cstdint>
#include <mutex>
#include <new>

#include "host_word.h"

namespace gals {

namespace {

constexpr int kWords = 1024, kBits = 64;

struct Slab {
    unsigned long long context;
    int *words;
    int used;
    uint64_t taken[kWords / kBits];
    Slab *next;
};

std::mutex g_mutex;
Slab *g_slabs = nullptr;

int take(Slab &s)
{
    for (int q = 0; q < kWords / kBits; ++q)
        for (int k = 0; k < kBits && ~s.taken[q]; ++k)
            if (!(s.taken[q] >> k & 1)) {
                s.taken[q] |= 1ull << k;
                ++s.used;
                return q * kBits + k;
            }
    return -1;
}

}  // namespace

unsigned long long current_context_id()
{
    // reached through the runtime's driver entry points, so that the library links against the
    // runtime only
    typedef int (*CtxGetCurrent)(void **);
    typedef int (*CtxGetId)(void *, unsigned long long *);
    auto entry = [](const char *name) -> void * {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion(name, &p, 12000, cudaEnableDefault, &q) != cudaSuccess ||
            q != cudaDriverEntryPointSuccess)
            return nullptr;
        return p;
    };
    static CtxGetCurrent get_current = reinterpret_cast<CtxGetCurrent>(entry("cuCtxGetCurrent"));
    static CtxGetId get_id = reinterpret_cast<CtxGetId>(entry("cuCtxGetId"));
    void *ctx = nullptr;
    unsigned long long id = 0;
    if (!get_current || !get_id || get_current(&ctx) != 0 || !ctx || get_id(ctx, &id) != 0) return 0;
    return id;
}

cudaError_t acquire_host_word(HostWord *word)
{
    *word = HostWord{};
    std::lock_guard<std::mutex> lock(g_mutex);
    unsigned long long context = current_context_id();
    for (Slab *s = g_slabs; s && context; s = s->next)
        if (s->context == context && s->used < kWords) {
            *word = HostWord{s->words + take(*s), context};
            return cudaSuccess;
        }
    int *words = nullptr;
    const cudaError_t e = cudaMallocHost(&words, kWords * sizeof(int));
    if (e != cudaSuccess) return e;
    context = current_context_id();  // the allocation makes one current
    Slab *s = new (std::nothrow) Slab{context, words, 0, {}, g_slabs};
    if (!s) {
        cudaFreeHost(words);
        return cudaErrorMemoryAllocation;
    }
    g_slabs = s;
    *word = HostWord{words + take(*s), context};
    return cudaSuccess;
}

void release_host_word(const HostWord &word)
{
    if (!word.at) return;
    std::lock_guard<std::mutex> lock(g_mutex);
    for (Slab **p = &g_slabs; *p; p = &(*p)->next) {
        Slab *s = *p;
        if (s->context != word.context || word.at < s->words || word.at >= s->words + kWords) continue;
        const int k = (int)(word.at - s->words);
        s->taken[k / kBits] &= ~(1ull << (k % kBits));
        if (--s->used > 0) return;
        bool other = false;
        for (Slab *o = g_slabs; o; o = o->next) other = other || (o != s && o->context == s->context);
        // freed only where its context is known to live: kept otherwise
        if (other && (s->context == 0 || current_context_id() == s->context)) {
            *p = s->next;
            cudaFreeHost(s->words);
            delete s;
        }
        return;
    }
}

}  // namespace gals
