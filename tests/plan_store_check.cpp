// Checks the store of device plan copies (csrc/plan_store.h) against a fake
// of the CUDA runtime calls it makes: a copy whose upload fails half-way
// leaves nothing behind, states share one copy, it is freed behind the work of
// all that held it, and nothing piles up.  Prints "ok" or the first
// violation (exit status 1).
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <set>
#include <string>
#include <thread>

#include "../paper_2105_13484_gb300/csrc/plan_store.h"

using namespace sse;

// ---- the fake: allocations, events and what each stream waited for
static std::mutex g;
static std::set<void *> allocs;
struct Ev { cudaStream_t on; bool done; };
static std::set<Ev *> events;
static std::map<cudaStream_t, std::set<cudaStream_t>> waited;   // stream -> streams it waited for
static bool busy = true;                                        // recorded events are unfinished
static int fail_alloc = -1, fail_copy = -1, fail_event = -1, syncs = 0;
static std::vector<std::set<cudaStream_t>> freed_behind;

extern "C" {
cudaError_t cudaMallocAsync(void **p, size_t n, cudaStream_t) {
    std::lock_guard<std::mutex> lk(g);
    if (fail_alloc >= 0 && fail_alloc-- == 0) return cudaErrorMemoryAllocation;
    allocs.insert(*p = malloc(n));
    return cudaSuccess;
}
cudaError_t cudaFreeAsync(void *p, cudaStream_t s) {
    std::lock_guard<std::mutex> lk(g);
    if (!allocs.erase(p)) { printf("freed twice\n"); exit(1); }
    freed_behind.push_back(waited[s]);
    free(p);
    return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind, cudaStream_t) {
    if (fail_copy >= 0 && fail_copy-- == 0) return cudaErrorUnknown;
    memcpy(d, s, n);
    return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t) { syncs++; return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned) {
    waited[s].insert(((Ev *)e)->on);
    return cudaSuccess;
}
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) {
    if (fail_event >= 0 && fail_event-- == 0) return cudaErrorMemoryAllocation;
    Ev *x = new Ev{nullptr, false};
    events.insert(x);
    *e = (cudaEvent_t)x;
    return cudaSuccess;
}
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) { ((Ev *)e)->on = s; return cudaSuccess; }
cudaError_t cudaEventQuery(cudaEvent_t) { return busy ? cudaErrorNotReady : cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t e) {
    if (!events.erase((Ev *)e)) { printf("event destroyed twice\n"); exit(1); }
    delete (Ev *)e;
    return cudaSuccess;
}
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaGetDevice(int *d) { *d = 0; return cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
}

struct View { const int *a, *b, *c; };
static void fill(PlanUpload &u, View &v) {
    v.a = u.put(std::vector<int>(100, 7));
    v.b = u.put(std::vector<int>());
    v.c = u.put(std::vector<int>(1, 9));
}
#define CHECK(x) do { if (!(x)) { printf("violation: %s (line %d)\n", #x, __LINE__); return 1; } } while (0)

int main() {
    const auto st = [](int i) { return (cudaStream_t)(uintptr_t)(i * 16); };
    const PlanStore::Key k{1, 4, 152, 0}, k2{1, 8, 152, 0};
    PlanStore S(0);
    View v{}, w{};
    CHECK(S.size<View>(k, fill) == 512 + 256 + 256 && allocs.empty());
    // an upload that fails anywhere leaves nothing, and the next one works
    for (int i = 0; i < 3; i++) {
        fail_alloc = i;
        CHECK(S.acquire(k, st(1), v, fill) == cudaErrorMemoryAllocation);
        CHECK(allocs.empty() && S.resident() == 0);
    }
    for (int i = 0; i < 2; i++) {
        fail_copy = i;
        CHECK(S.acquire(k, st(1), v, fill) != cudaSuccess && allocs.empty() && S.resident() == 0);
    }
    fail_alloc = fail_copy = -1;
    // one copy for two states, another for the other precision
    const int s0 = syncs;
    CHECK(S.acquire(k, st(1), v, fill) == cudaSuccess && syncs == s0 + 1 && allocs.size() == 3);
    CHECK(v.a[99] == 7 && v.c[0] == 9 && S.resident() == 1024);
    CHECK(S.acquire(k, st(2), w, fill) == cudaSuccess && w.a == v.a && allocs.size() == 3);
    CHECK(S.acquire(k2, st(2), w, fill) == cudaSuccess && w.a != v.a && S.resident() == 2048);
    S.release(k2, st(2));
    CHECK(S.resident() == 2048 && S.idle() == 1024 && allocs.size() == 6);
    // both leave with work in flight: the copy stays, a later state finds it,
    // and trim frees it behind all of their work
    S.release(k, st(1));
    CHECK(S.idle() == 1024 && S.trim() == 1024);   // the other precision's copy; k is held
    S.release(k, st(2));
    CHECK(allocs.size() == 3 && S.idle() == 1024 && S.resident() == 1024);
    CHECK(S.acquire(k, st(3), w, fill) == cudaSuccess && w.a == v.a && S.idle() == 0 && S.trim() == 0);
    S.release(k, st(3));
    freed_behind.clear();
    CHECK(S.trim() == 1024 && allocs.empty() && events.empty() && S.resident() == 0);
    CHECK(freed_behind.size() == 3);
    for (auto &b : freed_behind) CHECK(b.count(st(1)) && b.count(st(2)) && b.count(st(3)));
    // without an event to be had, the leaving stream is waited for
    S.acquire(k, st(1), v, fill); S.acquire(k, st(3), v, fill);
    fail_event = 0;
    const int s1 = syncs;
    S.release(k, st(3));
    CHECK(syncs == s1 + 1 && events.empty());
    fail_event = -1;
    // states that come and go pile up nothing
    busy = false;
    for (int i = 0; i < 1000; i++) { S.acquire(k, st(4), v, fill); S.release(k, st(4)); }
    CHECK(events.size() <= 1 && allocs.size() == 3);
    S.release(k, st(1));
    S.trim();
    CHECK(allocs.empty() && events.empty());
    // what is to be kept is kept
    S.acquire(k, st(1), v, fill); S.release(k, st(1));
    const auto keep = S.keys();
    S.acquire(k2, st(1), v, fill); S.release(k2, st(1));
    CHECK(keep.size() == 1 && S.trim(keep) == 1024 && S.keys() == keep && S.idle() == 1024);
    CHECK(S.trim() == 1024 && allocs.empty() && events.empty());
    // a store that goes frees what is left
    {
        PlanStore T(0);
        T.acquire(k, st(1), v, fill);
        T.release(k, st(1));
        CHECK(allocs.size() == 3);
    }
    CHECK(allocs.empty() && events.empty());
    // several threads
    std::vector<std::thread> ts;
    for (int t = 0; t < 8; t++)
        ts.emplace_back([&, t] {
            for (int i = 0; i < 500; i++) {
                View x{};
                const PlanStore::Key key{1, 4, i % 3, 0};
                if (S.acquire(key, st(10 + t), x, fill) != cudaSuccess || x.a[0] != 7) abort();
                S.release(key, st(10 + t));
                if (i % 7 == 0) S.trim();
            }
        });
    for (auto &t : ts) t.join();
    S.trim();
    CHECK(allocs.empty() && events.empty() && S.resident() == 0);
    printf("ok\n");
    return 0;
}
