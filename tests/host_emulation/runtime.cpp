// Fibers, warp and block wide operations and launches of the host emulation.
#include <setjmp.h>
#include <stdio.h>
#include <ucontext.h>

#include <algorithm>
#include <mutex>
#include <random>
#include <vector>

#include "cuda_runtime.h"

namespace emu {

dim3 thread_idx, block_idx, block_dim, grid_dim;
int sms = 1, syncs = 0, fail_alloc = 0;

namespace {

constexpr size_t STACK = 256 << 10;

struct Fiber {
    ucontext_t start;
    jmp_buf at;
    std::vector<char> stack;
    int tid = 0;
    bool started = false, waits = false, ended = true;
};
struct Warp {
    unsigned alive = 0, here = 0, want = 0;
    unsigned long long in[32], out[32];
};

std::vector<Fiber *> fibers;
std::vector<Warp> warps;
std::vector<unsigned long long> dyn;
Fiber *self = nullptr;
jmp_buf sched;
const std::function<void()> *body = nullptr;
long long barriers = 0;   // block wide barriers passed
int order = 0, nthreads = 0, block_here = 0, block_alive = 0, block_acc = 0, block_out = 0;
std::mt19937 rng(1);
std::mutex one;

__attribute__((noinline)) void yield() {
    if (!_setjmp(self->at)) _longjmp(sched, 1);
}

void warp_done(Warp &w, int first) {
    if (!w.here || w.here != (w.want & w.alive)) return;
    memcpy(w.out, w.in, sizeof(w.out));
    for (int l = 0; l < 32; l++)
        if ((w.here >> l) & 1u) fibers[(size_t)(first + l)]->waits = false;
    w.here = 0;
}

void block_done() {
    if (!block_here || block_here != block_alive) return;
    barriers++;
    block_out = block_acc;
    block_acc = block_here = 0;
    for (int i = 0; i < nthreads; i++) fibers[(size_t)i]->waits = false;
}

void entry() {
    (*body)();
    self->ended = true;
    Warp &w = warps[(size_t)(self->tid / 32)];
    w.alive &= ~(1u << (self->tid & 31));
    block_alive--;
    warp_done(w, self->tid / 32 * 32);
    block_done();
    _longjmp(sched, 1);
}

__attribute__((noinline)) void resume(Fiber *f) {
    self = f;
    thread_idx.x = (unsigned)f->tid;
    if (_setjmp(sched)) return;
    if (f->started) _longjmp(f->at, 1);
    f->started = true;
    setcontext(&f->start);
}

void run_block() {
    warps.assign((size_t)(nthreads + 31) / 32, Warp());
    for (int i = 0; i < nthreads; i++) {
        Fiber *f = fibers[(size_t)i];
        f->tid = i;
        f->started = f->waits = f->ended = false;
        getcontext(&f->start);
        f->start.uc_stack.ss_sp = f->stack.data();
        f->start.uc_stack.ss_size = f->stack.size();
        f->start.uc_link = nullptr;
        makecontext(&f->start, entry, 0);
        warps[(size_t)(i / 32)].alive |= 1u << (i & 31);
    }
    block_alive = nthreads;
    block_here = block_acc = 0;
    std::vector<int> turn((size_t)nthreads);
    const bool back = order == 1 || order == 4;
    const int last_lane = back ? 0 : 31;
    for (int i = 0; i < nthreads; i++) turn[(size_t)i] = back ? nthreads - 1 - i : i;
    while (block_alive > 0) {
        if (order == 2) std::shuffle(turn.begin(), turn.end(), rng);
        bool ran = false;
        for (int i : turn) {
            Fiber *f = fibers[(size_t)i];
            if (f->ended || f->waits) continue;
            resume(f);
            ran = true;
            // one warp at a time: back to the first once a warp's lanes have had their turn
            if (order >= 3 && (i & 31) == last_lane) break;
        }
        if (!ran) {
            fprintf(stderr, "emulation: block %u waits for ever (%d of %d threads at a barrier)\n", block_idx.x, block_here, block_alive);
            for (const Warp &w : warps) fprintf(stderr, "  warp: lanes %08x of %08x\n", w.here, w.want & w.alive);
            abort();
        }
    }
}

}  // namespace

char *dynamic_shared() { return reinterpret_cast<char *>(dyn.data()); }

unsigned long long now_ns() { return 1; }   // (the emulation is slow: no shot runs out of time)

int lane() { return self->tid & 31; }

const unsigned long long *exchange(unsigned mask, unsigned long long v) {
    static unsigned long long alone[32];
    const int l = self->tid & 31;
    if (mask == 1u << l) {
        alone[l] = v;
        return alone;
    }
    Warp &w = warps[(size_t)(self->tid / 32)];
    w.in[l] = v;
    w.want = mask;
    w.here |= 1u << l;
    self->waits = true;
    warp_done(w, self->tid / 32 * 32);
    if (self->waits) yield();
    return w.out;
}

int block_or(int v) {
    block_acc |= v != 0;
    block_here++;
    self->waits = true;
    block_done();
    if (self->waits) yield();
    return block_out;
}

void launch(long long grid, int block, size_t smem, const std::function<void()> &kernel) {
    std::lock_guard<std::mutex> lock(one);
    nthreads = block;
    while ((int)fibers.size() < block) {
        fibers.push_back(new Fiber());
        fibers.back()->stack.resize(STACK);
    }
    body = &kernel;
    grid_dim.x = (unsigned)grid;
    block_dim.x = (unsigned)block;
    for (long long b = 0; b < grid; b++) {
        block_idx.x = (unsigned)b;
        dyn.assign(smem / 8 + 2, 0xa5a5a5a5a5a5a5a5ull);
        run_block();
    }
}

}  // namespace emu

extern "C" {
// 0: lanes in order, 1: last lane first, 2: any order (seeded), 3 and 4: one warp
// as far as it gets before the next, first or last warp first
void emu_order(int order, unsigned seed) {
    emu::order = order;
    emu::rng.seed(seed);
}
void emu_sms(int n) { emu::sms = n; }
void emu_fail_alloc(int n) { emu::fail_alloc = n; }   // the n-th allocation from now on fails
int emu_syncs() { return emu::syncs; }   // waits for the whole device
long long emu_barriers() { return emu::barriers; }
}
