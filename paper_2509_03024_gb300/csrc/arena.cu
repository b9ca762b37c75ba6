// arena.cu — the pinned descriptor arena (Arena in core.cuh). Host code only.
#include <algorithm>
#include <cstring>

#include "core.cuh"

namespace fhe {

void Arena::reset(cudaStream_t s) {
    Half& used = halves[h];
    if (!used.done) CK(cudaEventCreateWithFlags(&used.done, cudaEventDisableTiming));
    CK(cudaEventRecord(used.done, s));
    used.pending = true;
    h ^= 1;
    Half& next = halves[h];
    if (next.pending) {
        CK(cudaEventSynchronize(next.done));  // its tables and staging may be overwritten now
        next.pending = false;
    }
    for (auto& b : next.blocks) b.used = 0;
    next.cur = 0;
}

void* Arena::push(const void* data, size_t bytes, cudaStream_t s) {
    Half& hf = halves[h];
    const size_t span = std::max<size_t>((bytes + 255) & ~(size_t)255, 256);
    while (hf.cur < hf.blocks.size() && hf.blocks[hf.cur].used + span > hf.blocks[hf.cur].cap) {
        if (gathering) upload_block(s);
        hf.cur++;
        from = hf.cur < hf.blocks.size() ? hf.blocks[hf.cur].used : 0;
    }
    if (hf.cur == hf.blocks.size()) {
        Block b;
        b.cap = std::max<size_t>(span, (size_t)4 << 20);
        CK(cudaMallocHost((void**)&b.host, b.cap));
        CK(cudaMalloc((void**)&b.dev, b.cap));
        hf.blocks.push_back(b);
    }
    Block& b = hf.blocks[hf.cur];
    char* hp = b.host + b.used;
    char* d = b.dev + b.used;
    b.used += span;
    if (bytes) {
        std::memcpy(hp, data, bytes);
        if (!gathering) CK(cudaMemcpyAsync(d, hp, bytes, cudaMemcpyHostToDevice, s));
    }
    return d;
}

void Arena::upload_block(cudaStream_t s) {
    Half& hf = halves[h];
    if (hf.cur >= hf.blocks.size()) return;
    Block& b = hf.blocks[hf.cur];
    if (b.used > from) CK(cudaMemcpyAsync(b.dev + from, b.host + from, b.used - from, cudaMemcpyHostToDevice, s));
    from = b.used;
}

void Arena::gather() {
    if (gathering++) return;  // an inner scope: the outer one's staged tables stay in [from, used)
    const Half& hf = halves[h];
    from = hf.cur < hf.blocks.size() ? hf.blocks[hf.cur].used : 0;
}

void Arena::upload(cudaStream_t s) {
    gathering--;
    upload_block(s);
}

Arena::~Arena() {
    for (auto& hf : halves) {
        if (hf.pending) cudaEventSynchronize(hf.done);
        if (hf.done) cudaEventDestroy(hf.done);
        for (auto& b : hf.blocks) {
            if (b.host) cudaFreeHost(b.host);
            if (b.dev) cudaFree(b.dev);
        }
    }
}

}  // namespace fhe
