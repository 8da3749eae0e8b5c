// lanes.cpp -- the fibers, collectives and memory checks behind lanes.h, and stand-ins for the CUDA calls of the host
// side (one device of 152 multiprocessors whose memory is the host's).
#include <ucontext.h>

#include <cstdlib>
#include <cstring>
#include <unordered_map>
#include <vector>

#include "lanes.h"

uint3 threadIdx, blockIdx;
dim3 blockDim, gridDim;

namespace {

constexpr size_t kStack = 256 * 1024;
enum Wait { kRunning, kWarp, kBlock, kDone };
struct Fiber {
    ucontext_t ctx;
    Wait wait;
    uint64_t in;
    uint64_t warp_epoch, block_epoch;  // __syncwarp and __syncthreads passed, __syncthreads passed
};
std::vector<Fiber> fibers;
std::vector<std::vector<uint64_t>> out;  // of each warp's last exchange
char* stacks = nullptr;
size_t stacks_bytes = 0;
std::vector<char> shared;  // dynamic, of the block that runs
ucontext_t scheduler;
int current = -1;
uint64_t block_value = 0;
const std::function<void()>* body = nullptr;
int order = 0;           // 0: ascending threads, 1: descending, else: from lane `order` on, around
long long races = 0, stuck = 0;

// what has touched a word since the launch began: its last write, and per warp the lanes that read it in their epoch
struct Access {
    int thread = -1;
    uint64_t warp_epoch = 0, block_epoch = 0;
};
struct Word {
    Access write;
    std::unordered_map<int, std::pair<Access, uint32_t>> reads;  // by warp: an access and the lanes of its epoch
};
std::unordered_map<uintptr_t, Word> words;

bool unordered(const Access& a, const Fiber& f, int thread)
{
    if (a.thread < 0 || a.thread == thread) return false;
    return a.thread / 32 == thread / 32 ? a.warp_epoch == f.warp_epoch : a.block_epoch == f.block_epoch;
}

void touch(const void* p, size_t bytes, bool write)
{
    if (current < 0 || ((const char*)p >= stacks && (const char*)p < stacks + stacks_bytes)) return;
    if (p == (const void*)&threadIdx || p == (const void*)&blockIdx || p == (const void*)&blockDim) return;
    Fiber& f = fibers[current];
    const int warp = current / 32;
    const uint32_t me = 1u << (current & 31);
    const uintptr_t first = bytes == 1 ? (uintptr_t)p * 2 + 1 : ((uintptr_t)p / 4) * 2;
    for (uintptr_t key = first; key < first + (bytes == 1 ? 1 : bytes / 2); key += 2) {
        Word& w = words[key];
        bool bad = unordered(w.write, f, current);
        if (write) {
            for (const auto& r : w.reads) {
                const Access& a = r.second.first;
                bad = bad || (r.first == warp ? a.warp_epoch == f.warp_epoch && (r.second.second & ~me) != 0
                                              : a.block_epoch == f.block_epoch);
            }
            w.reads.clear();
            w.write = {current, f.warp_epoch, f.block_epoch};
        } else {
            auto& r = w.reads[warp];
            if (r.first.thread < 0 || r.first.warp_epoch != f.warp_epoch) r.second = 0;
            r.first = {current, f.warp_epoch, f.block_epoch};
            r.second |= me;
        }
        races += bad;
    }
}

void yield(Wait w)
{
    Fiber& f = fibers[current];
    f.wait = w;
    swapcontext(&f.ctx, &scheduler);
}

void entry()
{
    (*body)();
    fibers[current].wait = kDone;
    swapcontext(&fibers[current].ctx, &scheduler);
}

}  // namespace

namespace lanes {

const uint64_t* warp_exchange(uint64_t v)
{
    const int me = current;
    fibers[me].in = v;
    yield(kWarp);
    return out[me / 32].data();
}

void warp_order()
{
    warp_exchange(0);
    ++fibers[current].warp_epoch;
}

uint64_t block_or(uint64_t v)
{
    fibers[current].in = v;
    yield(kBlock);
    ++fibers[current].warp_epoch;
    ++fibers[current].block_epoch;
    return block_value;
}

void* dynamic_shared() { return shared.data(); }

void launch(int64_t blocks, int threads, size_t dynamic_bytes, const std::function<void()>& thread)
{
    shared.assign(dynamic_bytes, 0);
    body = &thread;
    gridDim = dim3((unsigned)blocks);
    blockDim = dim3((unsigned)threads);
    stacks_bytes = kStack * (size_t)threads;
    stacks = (char*)std::malloc(stacks_bytes);
    words.clear();
    for (int64_t b = 0; b < blocks; ++b) {
        blockIdx = {(unsigned)b, 0, 0};
        fibers.assign(threads, Fiber{});
        out.assign((threads + 31) / 32, std::vector<uint64_t>(32));
        for (auto& w : words) w.second = Word{};  // blocks here are independent of one another
        for (int t = 0; t < threads; ++t) {
            getcontext(&fibers[t].ctx);
            fibers[t].ctx.uc_stack.ss_sp = stacks + kStack * t;
            fibers[t].ctx.uc_stack.ss_size = kStack;
            fibers[t].ctx.uc_link = nullptr;
            makecontext(&fibers[t].ctx, entry, 0);
        }
        for (;;) {
            bool ran = false;
            for (int i = 0; i < threads; ++i) {
                const int t = order == 0 ? i : order == 1 ? threads - 1 - i : (i & ~31) | ((i + order) & 31);
                if (fibers[t].wait != kRunning) continue;
                ran = true;
                current = t;
                threadIdx = {(unsigned)t, 0, 0};
                swapcontext(&scheduler, &fibers[t].ctx);
                current = -1;
            }
            if (ran) continue;
            bool moved = false;
            for (int w = 0; w < (threads + 31) / 32; ++w) {  // a warp whose lanes have all come to an exchange
                bool all = true;
                for (int l = 0; l < 32; ++l) all = all && fibers[w * 32 + l].wait == kWarp;
                if (!all) continue;
                for (int l = 0; l < 32; ++l) {
                    out[w][l] = fibers[w * 32 + l].in;
                    fibers[w * 32 + l].wait = kRunning;
                }
                moved = true;
            }
            if (moved) continue;
            int at_barrier = 0, done = 0;
            uint64_t v = 0;
            for (auto& f : fibers) {
                at_barrier += f.wait == kBlock;
                done += f.wait == kDone;
                if (f.wait == kBlock) v |= f.in;
            }
            if (done == threads) break;
            if (at_barrier + done != threads) {  // lanes of a warp wait for different collectives, for ever
                ++stuck;
                break;
            }
            block_value = v;
            for (auto& f : fibers)
                if (f.wait == kBlock) f.wait = kRunning;
        }
    }
    std::free(stacks);
    stacks = nullptr;
    stacks_bytes = 0;
}

}  // namespace lanes

uint32_t atomicAdd(uint32_t* p, uint32_t v)  // not among the accesses that need an order
{
    const uint32_t was = *p;
    *p = was + v;
    return was;
}

extern "C" {

void lanes_order(int o) { order = o; }
// since the last call: accesses that no barrier orders, and blocks whose lanes waited for different collectives
long long lanes_faults(long long* blocks)
{
    const long long r = races;
    *blocks = stuck;
    races = stuck = 0;
    return r;
}

cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) { *v = 152; return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaMemsetAsync(void* p, int v, size_t n, cudaStream_t) { std::memset(p, v, n); return cudaSuccess; }

#define LANES_HOOK(n)                                               \
    void __tsan_read##n(void* p) { touch(p, n, false); }            \
    void __tsan_write##n(void* p) { touch(p, n, true); }            \
    void __tsan_unaligned_read##n(void* p) { touch(p, n, false); }  \
    void __tsan_unaligned_write##n(void* p) { touch(p, n, true); }
LANES_HOOK(1)
LANES_HOOK(2)
LANES_HOOK(4)
LANES_HOOK(8)
LANES_HOOK(16)
void __tsan_read_range(void* p, size_t n) { touch(p, n, false); }
void __tsan_write_range(void* p, size_t n) { touch(p, n, true); }
void __tsan_init() {}
void __tsan_func_entry(void*) {}
void __tsan_func_exit() {}
void __tsan_vptr_read(void**) {}
void __tsan_vptr_update(void**, void*) {}

}  // extern "C"
