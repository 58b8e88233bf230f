// One CTA of a tcgen05 kernel on the host, for what its warps tell each other: the kernel's own source is compiled against this
// instead of csrc/sm100.cuh (tests/test_cta_protocol.py), a warp is a fiber that stands for its first lane, and copies and products
// are events that complete at any later time.  Numbers are not computed.  What is looked at:
//   - named barriers: nobody arrives twice in a phase, the numbers of participants agree, nothing is left over, nobody waits for good;
//   - what is asynchronous has finished when the CTA leaves: loads, reads of stores, products, arrivals of commits;
//   - tensor memory is allocated when it is touched, idle when it is released, and released;
//   - a warp that waits for a time has waited for the kernel before this one first (where the launch asks for that).
// Warps run in a random order with random, very different speeds; an unsatisfied wait expires with a given probability a poll.
#pragma once
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>
#include <stdio.h>
#include <stdlib.h>
#include <ucontext.h>

#include <algorithm>
#include <cmath>
#include <deque>
#include <functional>
#include <map>
#include <random>
#include <set>
#include <string>
#include <vector>

#include "internal.h"

using std::max;
using std::min;

namespace emu {

struct Fiber {
    ucontext_t ctx;
    std::vector<char> stack;
    dim3 idx;
    bool done = false, blocked = false, dep_waited = false;
    double speed = 1;
    int uncommitted = 0;               // bulk stores issued, of the present group
    std::deque<int> groups;            // committed groups whose source may still be read
};
struct Bar { int count = 0, pending = 0; long tx = 0; unsigned phase = 0; bool lost = false; };
struct Named { int arrived = 0, count = 0; std::set<int> who; std::vector<int> waiting; };
struct Load { Bar* bar; long bytes; bool lost; };
struct Op { Bar* commit; };            // null: a product

struct Cta {
    std::vector<Fiber> warps;
    std::map<const void*, Bar> bars;
    std::map<int, Named> named;
    std::vector<Load> loads;
    std::deque<Op> tensor;             // products and commits, in order
    int cur = 0, threads = 0;
    bool tmem = false, tmem_ever = false, need_dep = true;
    double expire = 0;                 // per unsatisfied poll
    double lose = 0;                   // per load: it never arrives
    std::string error;
    std::mt19937 rng;
    ucontext_t main;
};
inline Cta* c;
inline bool c_expired;             // of the last run
inline dim3 block, blockDim_, gridDim_;
alignas(1024) inline unsigned char smem[256 * 1024];

inline double rnd() { return std::uniform_real_distribution<double>(0, 1)(c->rng); }
inline Fiber& me() { return c->warps[c->cur]; }
inline void yield() { swapcontext(&me().ctx, &c->main); }
inline void fail(const std::string& what) {
    if (c->error.empty()) c->error = "warp " + std::to_string(c->cur) + ": " + what;
    swapcontext(&me().ctx, &c->main);   // the run ends here
}

inline void settle(Bar& b) { if (b.pending == 0 && b.tx == 0) { ++b.phase; b.pending = b.count; } }
inline void arrive(Bar& b) { --b.pending; settle(b); }
inline Bar& bar(const void* p) {
    auto it = c->bars.find(p);
    if (it == c->bars.end()) { fail("barrier used before its initialisation"); abort(); }
    return it->second;
}

// bar.sync / bar.arrive of one warp
inline void named(int id, int count, bool sync) {
    yield();
    Named& n = c->named[id];
    if (n.who.count(c->cur)) return fail("arrives twice in one phase of named barrier " + std::to_string(id));
    if (n.arrived && n.count != count) return fail("another number of participants at named barrier " + std::to_string(id));
    n.who.insert(c->cur);
    n.count = count;
    n.arrived += 32;
    if (n.arrived > count) return fail("too many arrivals at named barrier " + std::to_string(id));
    if (n.arrived == count) {
        for (int w : n.waiting) c->warps[w].blocked = false;
        n = Named{};
        if (sync) yield();
        return;
    }
    if (sync) { n.waiting.push_back(c->cur); me().blocked = true; yield(); }
}

// something asynchronous completes; false: nothing can
inline bool event() {
    std::vector<int> can;
    for (int i = 0; i < (int)c->loads.size(); ++i) if (!c->loads[i].lost) can.push_back(i);
    const bool t = !c->tensor.empty();
    if (can.empty() && !t) return false;
    const int k = (int)(rnd() * (can.size() + (t ? 1 : 0)));
    if (k < (int)can.size()) {
        const Load l = c->loads[can[k]];
        c->loads.erase(c->loads.begin() + can[k]);
        l.bar->tx -= l.bytes;
        settle(*l.bar);
    } else {
        const Op o = c->tensor.front();
        c->tensor.pop_front();
        if (o.commit) arrive(*o.commit);
    }
    return true;
}

inline std::function<void()> body;
inline void entry() { body(); me().done = true; swapcontext(&me().ctx, &c->main); }

struct Scenario { unsigned seed; double expire, lose; bool need_dep; };

// Runs one CTA of `threads` threads; "" or what went wrong.
inline std::string run(const Scenario& s, int threads, dim3 blk, dim3 grid, std::function<void()> kernel) {
    Cta cta;
    c = &cta;
    c_expired = false;
    cta.rng.seed(s.seed);
    cta.expire = s.expire; cta.lose = s.lose; cta.need_dep = s.need_dep;
    cta.threads = threads;
    block = blk; gridDim_ = grid; blockDim_ = dim3(threads);
    body = kernel;
    const int n = threads / 32;
    cta.warps.resize(n);
    for (int i = 0; i < n; ++i) {
        Fiber& f = cta.warps[i];
        f.stack.resize(96 * 1024);
        f.idx = dim3(32 * i, 0, 0);
        f.speed = std::pow(10., -3 * rnd());
        getcontext(&f.ctx);
        f.ctx.uc_stack.ss_sp = f.stack.data();
        f.ctx.uc_stack.ss_size = f.stack.size();
        f.ctx.uc_link = nullptr;
        makecontext(&f.ctx, entry, 0);
    }
    if (rnd() < 0.5) cta.warps[(int)(rnd() * n)].speed = s.expire > 0 ? 1e-7 : 1e-4;      // one that hardly moves, for a while
    const double events = std::pow(10., 1 - 3 * rnd());
    for (long step = 0;; ++step) {
        if (step > 20000000) return "does not end";
        double sum = 0;
        bool alive = false;
        for (Fiber& f : cta.warps) { alive |= !f.done; if (!f.done && !f.blocked) sum += f.speed; }
        if (!alive) break;
        if (sum == 0) {
            if (event()) continue;
            std::string w = "every warp waits at a named barrier:";
            for (auto& b : cta.named) if (!b.second.waiting.empty()) w += " " + std::to_string(b.first) + " (" + std::to_string(b.second.arrived) + " of " + std::to_string(b.second.count) + ")";
            return w;
        }
        if (rnd() * (events + 1) > 1) { if (event()) continue; }
        if (rnd() < 0.002) cta.warps[(int)(rnd() * n)].speed = std::pow(10., -3 * rnd());
        double at = rnd() * sum;
        int w = 0;
        for (int i = 0; i < n; ++i) {
            if (cta.warps[i].done || cta.warps[i].blocked) continue;
            w = i;
            if ((at -= cta.warps[i].speed) <= 0) break;
        }
        cta.cur = w;
        swapcontext(&cta.main, &cta.warps[w].ctx);
        if (!cta.error.empty()) return cta.error;
    }
    for (auto& b : cta.named) if (b.second.arrived) return "arrivals left over at named barrier " + std::to_string(b.first);
    for (const Load& l : cta.loads) if (!l.lost) return "leaves with a load in flight";
    for (const Op& o : cta.tensor) return o.commit ? "leaves with the arrival of a commit to come" : "leaves with a product in flight";
    for (int i = 0; i < n; ++i) if (cta.warps[i].uncommitted || !cta.warps[i].groups.empty()) return "leaves with a store that is still reading";
    if (cta.tmem || !cta.tmem_ever) return "tensor memory not released";
    return "";
}

inline void touch_tmem(const char* what) {
    yield();
    if (!c->tmem) fail(std::string(what) + " of tensor memory that is not allocated");
}

}  // namespace emu

#define threadIdx (emu::me().idx)
#define blockIdx emu::block
#define gridDim emu::gridDim_

// ---- what the compiler for the device has built in ---------------------------------------------------------------------------
inline void __syncwarp(unsigned = 0xffffffffu) { emu::yield(); }
inline void __syncthreads() { emu::named(0, emu::c->threads, true); }
template <class T> T __shfl_sync(unsigned, T x, int, int = 32) { return x; }
template <class T> T __shfl_xor_sync(unsigned, T x, int, int = 32) { return x; }
template <class T> T __shfl_up_sync(unsigned, T x, int, int = 32) { return x; }
template <class T> T __shfl_down_sync(unsigned, T x, int, int = 32) { return x; }
inline int __all_sync(unsigned, int x) { emu::yield(); return x; }
inline int __any_sync(unsigned, int x) { emu::yield(); return x; }
template <class T> T __ldcg(const T* p) { return *p; }
inline unsigned atomicAdd(unsigned* p, unsigned x) { const unsigned o = *p; *p += x; return o; }
inline float __expf(float x) { return std::exp(x); }
inline float rsqrtf(float x) { return 1.f / std::sqrt(x); }
inline uint32_t __float_as_uint(float x) { uint32_t u; __builtin_memcpy(&u, &x, 4); return u; }
inline float __uint_as_float(uint32_t u) { float x; __builtin_memcpy(&x, &u, 4); return x; }

namespace qd {
inline void tf32_split(float, uint32_t& hi, uint32_t& lo) { hi = lo = 0; }
inline void mma_tf32(float*, const uint32_t*, const uint32_t*) {}

namespace sm100 {
inline uint32_t smem_u32(const void*) { return 0; }
inline void mbar_init(uint64_t* b, uint32_t count) { emu::c->bars[b] = emu::Bar{(int)count, (int)count, 0, 0}; }
inline void mbar_init_fence() {}
inline void mbar_expect_tx(uint64_t* b, uint32_t bytes) { emu::bar(b).tx += bytes; emu::arrive(emu::bar(b)); emu::yield(); }
inline void mbar_arrive(uint64_t* b) { emu::arrive(emu::bar(b)); emu::yield(); }
inline bool mbar_try_wait(uint64_t* b, uint32_t parity) {
    emu::yield();
    if (emu::c->need_dep && !emu::me().dep_waited) emu::fail("a bounded wait before the kernel before this one has completed");
    return (emu::bar(b).phase & 1) != parity;
}
inline bool expires() { return emu::rnd() < emu::c->expire; }
// as in a kernel's own waits: may expire at any poll
inline bool mbar_wait(uint64_t* b, uint32_t parity, uint32_t = 0) {
    for (;;) {
        if (mbar_try_wait(b, parity)) return true;
        if (expires()) { emu::c_expired = true; return false; }
    }
}
inline bool wait_on(uint64_t* b, uint32_t parity, volatile int& s_abort, unsigned* status) {
    while (!s_abort) {
        if (mbar_try_wait(b, parity)) return true;
        if (expires()) { s_abort = 1; *status = QD_ERR_TIMEOUT; emu::c_expired = true; }
    }
    return false;
}
// what is in flight comes within the limit, unless it never does
inline bool mbar_drain(uint64_t* b, uint32_t parity) {
    for (int polls = 0; !(emu::bar(b).lost && polls > 1000); ++polls)
        if (mbar_try_wait(b, parity)) return true;
    return false;
}
inline void mbar_drain_ring(uint64_t* bars, int depth, int loads) {
    for (int i = 0; i < depth && i < loads; ++i) mbar_drain(&bars[i], (uint32_t)((loads - 1 - i) / depth) & 1);
}
inline void grid_dep_wait() { emu::yield(); emu::me().dep_waited = true; }
inline void grid_dep_launch() {}
inline void fence_proxy_async() {}
inline void tc_fence_before() {}
inline void tc_fence_after() {}

// a map's first word holds the bytes of its box
inline void tma_load(const CUtensorMap* map, uint64_t* b) {
    const bool lost = emu::rnd() < emu::c->lose;
    emu::bar(b).lost |= lost;
    emu::c->loads.push_back({&emu::bar(b), (long)map->opaque[0], lost});
    emu::yield();
}
inline void tma_load_2d(void*, const CUtensorMap* map, int, int, uint64_t* b) { tma_load(map, b); }
inline void tma_load_3d(void*, const CUtensorMap* map, int, int, int, uint64_t* b) { tma_load(map, b); }
inline void tma_store_2d(const CUtensorMap*, const void*, int, int) { ++emu::me().uncommitted; }
inline void tma_store_3d(const CUtensorMap*, const void*, int, int, int) { ++emu::me().uncommitted; }
inline void tma_prefetch_2d(const CUtensorMap*, int, int) {}
inline void tma_prefetch_3d(const CUtensorMap*, int, int, int) {}
inline void tma_store_commit() { emu::me().groups.push_back(emu::me().uncommitted); emu::me().uncommitted = 0; }
template <int N> void tma_store_wait_read_n() { emu::yield(); while ((int)emu::me().groups.size() > N) emu::me().groups.pop_front(); }
inline void tma_store_wait_read() { tma_store_wait_read_n<0>(); }
inline void tma_store_wait_all() { tma_store_wait_read_n<0>(); }

inline void tmem_alloc(uint32_t* slot, uint32_t) { *slot = 0; emu::c->tmem = emu::c->tmem_ever = true; }
inline void tmem_relinquish() {}
inline void tmem_dealloc(uint32_t, uint32_t) {
    emu::touch_tmem("release");
    for (const emu::Op& o : emu::c->tensor) if (!o.commit) emu::fail("tensor memory released under a product");
    emu::c->tmem = false;
}
inline void tmem_ld_wait() {}
inline void tmem_st_wait() {}
template <int N> void tmem_ld(float* v) { emu::touch_tmem("load"); for (int i = 0; i < N; ++i) v[i] = 0.f; }
inline void tmem_ld32(uint32_t, float* v) { tmem_ld<32>(v); }
inline void tmem_ld16(uint32_t, float* v) { tmem_ld<16>(v); }
inline void tmem_ld8(uint32_t, float* v) { tmem_ld<8>(v); }
inline void tmem_ld_frag(uint32_t, float* v) { tmem_ld<4>(v); }
inline void tmem_ld_frag2(uint32_t, float* v) { tmem_ld<8>(v); }
inline void tmem_ld_frag4(uint32_t, float* v) { tmem_ld<16>(v); }
inline void tmem_st8(uint32_t, const uint32_t*) { emu::touch_tmem("store"); }
inline void tmem_st_frag2(uint32_t, const uint32_t*) { emu::touch_tmem("store"); }
inline void tmem_st_frag4(uint32_t, const uint32_t*) { emu::touch_tmem("store"); }
inline uint32_t tmem_addr(uint32_t base, uint32_t, uint32_t) { return base; }
template <bool T> void ldsm4(const void*, uint32_t* r) { for (int i = 0; i < 4; ++i) r[i] = 0; }
template <bool T> void stsm4(void*, const uint32_t*) {}

inline int warp_index() { return threadIdx.x >> 5; }
inline uint32_t uniform(uint32_t x) { return x; }
inline uint32_t elect_lane() { return 1; }
inline void product() { emu::touch_tmem("product"); emu::c->tensor.push_back({nullptr}); }
inline void umma_commit_w(uint64_t* b, uint32_t) { emu::c->tensor.push_back({&emu::bar(b)}); emu::yield(); }
template <bool A_MN, bool B_MN, int M = 128>
void umma_product_w(uint32_t, uint32_t, uint32_t, uint32_t, uint32_t, int, int, bool, uint32_t, bool = false) { product(); }
template <bool B_MN, int M = 128>
void umma_product_ts_w(uint32_t, uint32_t, uint32_t, uint32_t, int, int, bool, uint32_t, bool = false) { product(); }

inline uint32_t sw128_chunk(uint32_t line, uint32_t ch) { return line * 128u + (((ch ^ line) & 7u) << 4); }
inline void sts128(void*, uint4) {}
inline void sts16(void*, __nv_bfloat16) {}
inline void sts32(void*, float) {}
inline uint32_t pack_bf16(float, float) { return 0; }
inline void load8(const unsigned char*, float* f) { for (int i = 0; i < 8; ++i) f[i] = 0.f; }
inline uint4 pack8(const float*) { return make_uint4(0, 0, 0, 0); }
inline void nb_arrive(int id, int count) { emu::named(id, count, false); }
inline void nb_sync(int id, int count) { __syncwarp(); emu::named(id, count, true); }
}  // namespace sm100
}  // namespace qd
