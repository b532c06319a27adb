// A stand-in for the CUDA runtime and the kernels, for tests of the library's host side (capi.cu)
// without a GPU: linked with the objects of capi.cu and host_graph.cpp in place of the kernels'
// objects and cudart.
//
// "Device" memory is host memory.  A stream is a queue whose work runs as late as the CUDA rules
// allow: only when something waits for it (a stream or event wait, a synchronous copy, cudaFree).
// So a host read or write that is not ordered after queued work sees the memory as it was.  The
// decode launches give simple results that depend on every word of a shot's syndrome, check that
// each shot is in the list (or class) of its defect count, and can be made to fail on the host.
#include <cuda_runtime.h>

#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <deque>
#include <functional>
#include <map>
#include <memory>
#include <mutex>
#include <vector>

#include "device.cuh"

namespace {

std::recursive_mutex mu;
#define LOCK std::lock_guard<std::recursive_mutex> lk(mu)

struct Stream;
struct Rec {
    bool done = false;
    Stream* s = nullptr;
};
struct Stream {
    int id = 0, prio = 0;
    bool blocking = true;
    std::deque<std::function<void()>> q;
};
struct Event {
    std::shared_ptr<Rec> rec;
};

Stream legacy;
std::vector<Stream*> streams;  // created and not destroyed
int next_id = 1;
std::map<uintptr_t, size_t> device_mem, pinned_mem;
cudaError_t last_error = cudaSuccess;
int fail_launch = 0;      // the n-th launch from now fails
int fail_create = -1;     // this many more streams can be created
int max_streams = 0, list_errors = 0;
struct Launch {
    int kind, list, stream, prio;
};
std::vector<Launch> launches;

cudaError_t err(cudaError_t e) {
    if (e != cudaSuccess) last_error = e;
    return e;
}
Stream* of(cudaStream_t s) { return s == nullptr || s == cudaStreamLegacy ? &legacy : reinterpret_cast<Stream*>(s); }
Event* of(cudaEvent_t e) { return reinterpret_cast<Event*>(e); }

void step(Stream* s) {
    auto f = std::move(s->q.front());
    s->q.pop_front();
    f();
}
void drain(Stream* s) {
    while (!s->q.empty()) step(s);
}
void finish(const std::shared_ptr<Rec>& r) {
    while (r && !r->done) step(r->s);
}
std::shared_ptr<Rec> mark(Stream* s) {
    auto r = std::make_shared<Rec>();
    r->s = s;
    s->q.push_back([r] { r->done = true; });
    return r;
}
void after(Stream* s, const std::shared_ptr<Rec>& r) {
    s->q.push_back([r] { finish(r); });
}
// work in the legacy stream follows all earlier work of blocking streams and precedes their later work
void put(Stream* s, std::function<void()> f) {
    if (s == &legacy) {
        for (Stream* t : streams)
            if (t->blocking && !t->q.empty()) after(s, mark(t));
    } else if (s->blocking && !legacy.q.empty()) {
        after(s, mark(&legacy));
    }
    s->q.push_back(std::move(f));
}
void drain_all() {
    drain(&legacy);
    for (Stream* t : streams) drain(t);
}
bool within(const std::map<uintptr_t, size_t>& m, const void* p) {
    auto it = m.upper_bound((uintptr_t)p);
    if (it == m.begin()) return false;
    --it;
    return (uintptr_t)p < it->first + it->second;
}

cudaError_t new_stream(cudaStream_t* out, unsigned flags, int prio) {
    LOCK;
    if (fail_create == 0) return err(cudaErrorMemoryAllocation);
    if (fail_create > 0) --fail_create;
    Stream* s = new Stream();
    s->id = next_id++;
    s->prio = prio;
    s->blocking = !(flags & cudaStreamNonBlocking);
    streams.push_back(s);
    max_streams = std::max(max_streams, (int)streams.size());
    *out = reinterpret_cast<cudaStream_t>(s);
    return cudaSuccess;
}

}  // namespace

extern "C" {

// ---- test controls
void fake_reset() {
    LOCK;
    drain_all();
    launches.clear();
    fail_launch = 0;
    fail_create = -1;
    list_errors = 0;
    last_error = cudaSuccess;
    max_streams = (int)streams.size();
}
void fake_fail_launch(int n) { fail_launch = n; }
void fake_fail_stream_create(int left) { fail_create = left; }
int fake_pending() {
    LOCK;
    int n = (int)legacy.q.size();
    for (Stream* t : streams) n += (int)t->q.size();
    return n;
}
int fake_streams() { return (int)streams.size(); }
int fake_max_streams() { return max_streams; }
int fake_list_errors() { return list_errors; }
int fake_launches(int* out, int cap) {  // (kind, list, stream, priority) each
    LOCK;
    for (int k = 0; k < cap && k < (int)launches.size(); ++k) std::memcpy(out + 4 * k, &launches[k], sizeof(Launch));
    return (int)launches.size();
}
void fake_enqueue_write(void* stream, void* dst, const void* src, size_t n) {
    LOCK;
    std::vector<char> v((const char*)src, (const char*)src + n);
    put(of((cudaStream_t)stream), [dst, v] { std::memcpy(dst, v.data(), v.size()); });
}

// ---- runtime
cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) { *v = 8; return cudaSuccess; }
cudaError_t cudaDeviceGetStreamPriorityRange(int* least, int* greatest) { *least = 0; *greatest = -5; return cudaSuccess; }
cudaError_t cudaMemGetInfo(size_t* f, size_t* t) { *f = *t = (size_t)200 << 30; return cudaSuccess; }
cudaError_t cudaGetLastError() { cudaError_t e = last_error; last_error = cudaSuccess; return e; }
cudaError_t cudaPeekAtLastError() { return last_error; }
const char* cudaGetErrorName(cudaError_t) { return "fake error"; }
const char* cudaGetErrorString(cudaError_t) { return "from the stand-in runtime"; }
cudaError_t cudaMalloc(void** p, size_t n) {
    LOCK;
    *p = std::malloc(std::max<size_t>(n, 1));
    std::memset(*p, 0xCD, std::min<size_t>(n, 1 << 20));
    device_mem[(uintptr_t)*p] = n;
    return cudaSuccess;
}
cudaError_t cudaFree(void* p) {
    LOCK;
    if (!p) return cudaSuccess;
    drain_all();
    device_mem.erase((uintptr_t)p);
    std::free(p);
    return cudaSuccess;
}
cudaError_t cudaMallocHost(void** p, size_t n) {
    LOCK;
    *p = std::malloc(std::max<size_t>(n, 1));
    pinned_mem[(uintptr_t)*p] = n;
    return cudaSuccess;
}
cudaError_t cudaFreeHost(void* p) {
    LOCK;
    if (!p) return cudaSuccess;
    drain_all();
    pinned_mem.erase((uintptr_t)p);
    std::free(p);
    return cudaSuccess;
}
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes* a, const void* p) {
    LOCK;
    std::memset(a, 0, sizeof(*a));
    a->type = within(device_mem, p) ? cudaMemoryTypeDevice : within(pinned_mem, p) ? cudaMemoryTypeHost : cudaMemoryTypeUnregistered;
    return cudaSuccess;
}
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) {
    LOCK;
    put(&legacy, [] {});
    drain(&legacy);
    std::memcpy(d, s, n);
    return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t st) {
    LOCK;
    const bool staged = !(within(device_mem, d) || within(pinned_mem, d)) || !(within(device_mem, s) || within(pinned_mem, s));
    put(of(st), [d, s, n] { std::memcpy(d, s, n); });
    if (staged) drain(of(st));  // pageable memory on either side: the call returns when it has been copied
    return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t st) {
    LOCK;
    put(of(st), [d, v, n] { std::memset(d, v, n); });
    return cudaSuccess;
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned flags) { return new_stream(s, flags, 0); }
cudaError_t cudaStreamCreateWithPriority(cudaStream_t* s, unsigned flags, int prio) { return new_stream(s, flags, prio); }
cudaError_t cudaStreamGetPriority(cudaStream_t s, int* p) { *p = of(s)->prio; return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t st) {
    LOCK;
    Stream* s = of(st);
    drain(s);
    for (size_t k = 0; k < streams.size(); ++k)
        if (streams[k] == s) streams.erase(streams.begin() + (std::ptrdiff_t)k);
    return cudaSuccess;  // (kept allocated: records may name it)
}
cudaError_t cudaStreamSynchronize(cudaStream_t s) { LOCK; drain(of(s)); return cudaSuccess; }
cudaError_t cudaDeviceSynchronize() { LOCK; drain_all(); return cudaSuccess; }
cudaError_t cudaStreamQuery(cudaStream_t s) { LOCK; return of(s)->q.empty() ? cudaSuccess : cudaErrorNotReady; }
cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned) {
    LOCK;
    auto r = of(e)->rec;
    put(of(s), [r] { finish(r); });
    return cudaSuccess;
}
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { *e = reinterpret_cast<cudaEvent_t>(new Event()); return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t* e) { return cudaEventCreateWithFlags(e, 0); }
cudaError_t cudaEventDestroy(cudaEvent_t e) { delete of(e); return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) {
    LOCK;
    put(of(s), [] {});  // (orders the record as any other work of the stream)
    of(e)->rec = mark(of(s));
    return cudaSuccess;
}
cudaError_t cudaEventSynchronize(cudaEvent_t e) { LOCK; finish(of(e)->rec); return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) { *ms = 1.f; return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return err(cudaErrorNotSupported); }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t*) { return err(cudaErrorNotSupported); }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t*, cudaGraph_t, unsigned long long) { return err(cudaErrorNotSupported); }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return err(cudaErrorNotSupported); }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }

// capi.cu's one kernel (flags -> converged)
static thread_local cudaStream_t call_stream;
unsigned __cudaPushCallConfiguration(dim3, dim3, size_t, CUstream_st* st) { call_stream = st; return 0; }
cudaError_t __cudaPopCallConfiguration(dim3*, dim3*, size_t*, void* st) { *(cudaStream_t*)st = call_stream; return cudaSuccess; }
cudaError_t __cudaGetKernel(cudaKernel_t*, const void*) { return cudaSuccess; }
cudaError_t __cudaLaunchKernel(cudaKernel_t, dim3, dim3, void** args, size_t, cudaStream_t st) {
    LOCK;
    const uint8_t* flags = *(const uint8_t**)args[0];
    const int64_t n = *(int64_t*)args[1];
    uint8_t* conv = *(uint8_t**)args[2];
    put(of(st), [=] {
        for (int64_t k = 0; k < n; ++k) conv[k] = flags[k] & bp4m::F_CONVERGED;
    });
    return cudaSuccess;
}
cudaError_t cudaLaunchKernel(const void*, dim3, dim3, void** args, size_t n, cudaStream_t st) {
    return __cudaLaunchKernel(nullptr, dim3(), dim3(), args, n, st);
}
void** __cudaRegisterFatBinary(void*) { static void* h; return &h; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char*, char*, const char*, int, uint3*, uint3*, dim3*, dim3*, int*) {}

}  // extern "C"

// ---- kernels
namespace bp4m {

namespace {

enum { CLASSIFY = 0, LIST = 1, GLOBAL = 2, PARTITION = 3, OTHER = 4 };
const int kRows[kGlobalList] = {8, 16, 24, 32, 48, 64, 80, 96, 112, 128, 144, 160};
const int kRows64[kGlobalList] = {32, 32, 32, 32, 64, 64, 112, 112, 112, 112, 112, 112};

cudaError_t launch(int kind, int list, cudaStream_t st, std::function<void()> f) {
    LOCK;
    if (fail_launch > 0 && --fail_launch == 0) return err(cudaErrorLaunchOutOfResources);
    launches.push_back(Launch{kind, list, of(st)->id, of(st)->prio});
    put(of(st), std::move(f));
    return cudaSuccess;
}

int defects(const uint32_t* row, int nw) {
    int s = 0;
    for (int k = 0; k < nw; ++k) s += __builtin_popcount(row[k]);
    return s;
}

// What stands for a decode: obs from a hash of the row, converged unless s % 5 == 0, iterations s
void decode(const DecodeArgs& a, int64_t shot, int lo, int hi) {
    const uint32_t* row = a.synd + shot * a.tb.n_words;
    const int s = defects(row, a.tb.n_words);
    if (s <= lo || s > hi) ++list_errors;
    uint32_t h = 0;
    for (int k = 0; k < a.tb.n_words; ++k) h = (h ^ row[k]) * 2654435761u;
    if (a.obs_pred) a.obs_pred[shot] = (uint8_t)(h >> 31);
    if (a.flags) a.flags[shot] = s % 5 ? F_CONVERGED : F_FORCED_RAN;
    if (a.iters) a.iters[shot] = (int16_t)s;
}

}  // namespace

TierPlan tier_plan(int precision, bool) {
    TierPlan p{};
    for (int c = 0; c < kGlobalList; ++c) p.smax[c] = precision == 0 ? kRows64[c] : kRows[c];
    p.smax[kGlobalList] = 0x7fffffff;
    return p;
}
cudaError_t prepare_decode_kernels(int) { return cudaSuccess; }
cudaError_t launch_classify(const uint32_t* synd, int64_t shots, int nw, const TierPlan& plan, int32_t* lists, int32_t* counts,
                            int32_t* max_s, uint8_t* obs, uint8_t* flags, int16_t* iters, int32_t* trd, const uint8_t* skip,
                            const uint8_t* skip_obs, const int16_t* skip_iters, cudaStream_t st, int64_t stride, int32_t base) {
    if (stride == 0) stride = shots;
    return launch(CLASSIFY, 0, st, [=] {
        for (int64_t k = 0; k < shots; ++k) {
            const int s = defects(synd + k * nw, nw);
            if (trd) trd[k] = s;
            if (s == 0 || (skip && skip[k])) {
                if (obs) obs[k] = s && skip_obs ? skip_obs[k] : 0;
                if (flags) flags[k] = F_CONVERGED;
                if (iters) iters[k] = s && skip_iters ? skip_iters[k] : 0;
                continue;
            }
            *max_s = std::max(*max_s, s);
            int c = 0;
            while (c < kGlobalList && s > plan.smax[c]) ++c;
            const int64_t pos = counts[c]++;
            lists[(int64_t)list_slot(c) * stride + (list_back(c) ? stride - 1 - pos : pos)] = base | (int32_t)k;
        }
    });
}
cudaError_t launch_decode_list(int precision, int list, const DecodeArgs& a, int, cudaStream_t st) {
    return launch(LIST, list, st, [=] {
        const TierPlan p = tier_plan(precision);
        if (a.max_items > 0 && a.max_items != *a.count) ++list_errors;
        for (int k = 0; k < *a.count; ++k) decode(a, a.list[(int64_t)k * a.list_dir], list ? p.smax[list - 1] : 0, p.smax[list]);
    });
}
cudaError_t launch_decode_list_rw(int, int list, const DecodeArgs& a, int, cudaStream_t st) {
    return launch(LIST, list, st, [=] {
        for (int k = 0; k < *a.count; ++k) decode(a, a.list[(int64_t)k * a.list_dir], 0, 1 << 20);
    });
}
cudaError_t launch_decode_global(int precision, const DecodeArgs& a, int slots, int, cudaStream_t st) {
    return launch(GLOBAL, a.gsmax, st, [=] {
        // every slot is written before and checked after, as a block that owns it would
        for (int q = 0; q < slots; ++q) ((volatile char*)a.gscratch)[(size_t)q * a.gslot_elems] = (char)q;
        for (int k = 0; k < *a.count; ++k) decode(a, a.list[k], tier_plan(precision ? 1 : 0).smax[kGlobalList - 1], a.gsmax);
    });
}
GlobalClasses global_classes(int precision, int max_s) {
    GlobalClasses gc{};
    for (int w : {192, 256, 320, 384, 448, 512, 640, 768, 896, 1024}) {
        if (precision == 0 && w != 256 && w != 512) continue;
        gc.smax[gc.n++] = w;
        if (max_s <= w) return gc;
    }
    gc.smax[gc.n++] = max_s;
    return gc;
}
size_t global_slot_bytes(int, int max_s, int* gsmax) {
    *gsmax = max_s;
    return (size_t)max_s * 24;  // (the launch touches the first byte of each slot's matrices)
}
int global_blocks_per_sm(int, int) { return 1; }
cudaError_t launch_partition_global(const DecodeArgs& a, const GlobalClasses& gc, int32_t* sub, int64_t stride, int32_t* cnt,
                                    int64_t, int, cudaStream_t st) {
    return launch(PARTITION, 0, st, [=] {
        for (int k = 0; k < *a.count; ++k) {
            const int s = defects(a.synd + (int64_t)a.list[k] * a.tb.n_words, a.tb.n_words);
            int c = 0;
            while (c + 1 < gc.n && s > gc.smax[c]) ++c;
            sub[c * stride + cnt[c]++] = a.list[k];
        }
    });
}
int stream_cluster_for(int, int, int, int64_t, int) { return 1; }
int stream_cluster_capacity_of(int, int, int) { return 0; }
size_t rw_scratch_bytes(int, int, int, int, int, int64_t* slot) { *slot = 256; return 256; }
cudaError_t launch_qbp(int, const QbpArgs& a, int, cudaStream_t st) {
    return launch(OTHER, 0, st, [=] { std::memset(a.qconv, 0, (size_t)a.shots); });
}
cudaError_t launch_rw_flip(const RwFlipArgs& a, int, cudaStream_t st) {
    return launch(OTHER, 1, st, [=] {
        for (int t = 0; t < 2; ++t) std::memcpy(a.out[t], a.synd[t], (size_t)a.shots * a.n_words[t] * 4);
    });
}
cudaError_t launch_rw_base(uint8_t*, const uint8_t*, const uint8_t*, int64_t, cudaStream_t st) { return launch(OTHER, 2, st, [] {}); }
cudaError_t sample(const SampleArgs& a, cudaStream_t st) {
    return launch(OTHER, 3, st, [=] {
        size_t words = 0;
        for (int t = 0; t < a.n_types; ++t) words += (size_t)a.shots * a.n_words[t];
        for (size_t k = 0; k < words; ++k) a.synd[k] = k % 7 ? 0u : (uint32_t)(1u << (k % 13));
        std::memset(a.obs, 0, (size_t)a.shots * a.n_types);
    });
}
cudaError_t launch_sample_circuit(const SampleArgs& a, cudaStream_t st) { return sample(a, st); }
cudaError_t launch_sample_code_capacity(const SampleArgs& a, cudaStream_t st) { return sample(a, st); }
cudaError_t launch_count(const uint8_t*, const uint8_t*, const uint8_t*, int64_t shots, int, unsigned long long* ctr, cudaStream_t st) {
    return launch(OTHER, 4, st, [=] { ctr[C_SHOTS] += (unsigned long long)shots; });
}
cudaError_t launch_decode_noalloc(int, DecodeArgs, int64_t, cudaStream_t, int*) { return cudaErrorNotSupported; }
int noalloc_max_defects() { return 1; }
int64_t noalloc_max_shots() { return 1; }
cudaError_t launch_mufu_probe(int, int, int, long long*, float*, cudaStream_t) { return cudaErrorNotSupported; }
int mufu_probe_ops_per_thread(int, int) { return 1; }

}  // namespace bp4m
