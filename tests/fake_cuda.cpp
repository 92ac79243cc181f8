// A CUDA runtime on host threads, for tests of the library's host code on a
// machine without a GPU: linked with the library's own host objects (the
// context, the served loop, the allocation-free call) in place of the runtime
// and of the kernels.  "Device" memory is host memory; a stream is a thread
// that runs its operations in order; a kernel is an entry in the log, written
// when the stream reaches it, with what its batch table holds at that time.
// Calls that may wait for the device in the real runtime (allocations, frees,
// synchronous copies) wait here for every host function enqueued before them.
#include <cuda_runtime.h>

#include <atomic>
#include <chrono>
#include <condition_variable>
#include <cstdlib>
#include <cstring>
#include <deque>
#include <functional>
#include <map>
#include <memory>
#include <mutex>
#include <set>
#include <string>
#include <thread>
#include <vector>

#include "ft_internal.h"

namespace {

struct Flag {
    std::mutex m;
    std::condition_variable cv;
    bool up = false;
    void raise()
    {
        {
            std::lock_guard<std::mutex> l(m);
            up = true;
        }
        cv.notify_all();
    }
    void wait()
    {
        std::unique_lock<std::mutex> l(m);
        cv.wait(l, [&] { return up; });
    }
};

struct Graph {
    std::vector<std::function<void()>> ops;
};

struct Stream {
    std::mutex m;
    std::condition_variable cv;
    std::deque<std::function<void()>> q;
    bool busy = false, stop = false;
    Graph *capture = nullptr;
    std::thread worker;
    Stream() : worker([this] { run(); }) {}
    ~Stream()
    {
        {
            std::lock_guard<std::mutex> l(m);
            stop = true;
        }
        cv.notify_all();
        worker.join();
    }
    void run()
    {
        std::unique_lock<std::mutex> l(m);
        for (;;) {
            cv.wait(l, [&] { return stop || !q.empty(); });
            if (q.empty()) return;
            auto f = std::move(q.front());
            q.pop_front();
            busy = true;
            l.unlock();
            f();
            l.lock();
            busy = false;
            cv.notify_all();
        }
    }
    void put(std::function<void()> f)
    {
        if (capture) {
            capture->ops.push_back(std::move(f));
            return;
        }
        {
            std::lock_guard<std::mutex> l(m);
            q.push_back(std::move(f));
        }
        cv.notify_all();
    }
    void drain()
    {
        std::unique_lock<std::mutex> l(m);
        cv.wait(l, [&] { return q.empty() && !busy; });
    }
};

struct Event {
    std::shared_ptr<Flag> last;
    double at = 0;
};

std::mutex g_mu;                                // log, failures, host functions
std::condition_variable g_cv;
std::vector<std::string> g_log;
std::map<std::string, int> g_fail;              // name -> calls that still succeed before one fails
std::set<long> g_host;                          // host functions enqueued and not yet returned
long g_next = 0;
std::atomic<int> g_host_delay_us{0}, g_table_kernels{0};
std::atomic<double> g_clock_ms{0};               // by the one-frame launches so far
std::atomic<int> g_fast_strip{0}, g_last_strip{0};
std::atomic<double> g_fast_ms{1};
thread_local cudaError_t t_error = cudaSuccess;

Stream &stream_of(cudaStream_t s)
{
    static Stream *legacy = new Stream();
    return s ? *reinterpret_cast<Stream *>(s) : *legacy;
}

void log(std::string s)
{
    std::lock_guard<std::mutex> l(g_mu);
    g_log.push_back(std::move(s));
}

cudaError_t result(const char *name)
{
    std::lock_guard<std::mutex> l(g_mu);
    auto it = g_fail.find(name);
    if (it == g_fail.end() || it->second-- > 0) return cudaSuccess;
    g_fail.erase(it);
    return t_error = cudaErrorLaunchFailure;
}

// what a call that synchronizes with the device waits for
void wait_for_host_functions()
{
    std::unique_lock<std::mutex> l(g_mu);
    const long upto = g_next;
    g_cv.wait(l, [&] { return g_host.empty() || *g_host.begin() >= upto; });
}

cudaError_t kernel(const char *name, cudaStream_t s, std::function<std::string()> what)
{
    const cudaError_t e = result(name);
    if (e != cudaSuccess) return e;
    stream_of(s).put([=] { log(std::string(name) + " " + what()); });
    return cudaSuccess;
}

std::string frames_of(const ft::BatchHeader *h) { return std::to_string(h->nframes); }

}  // namespace

// ---------------------------------------------------------------- control from the test
extern "C" {
// the (after + 1)-th call of `name` from now on fails, once
void fake_fail(const char *name, int after)
{
    std::lock_guard<std::mutex> l(g_mu);
    g_fail[name] = after;
}
void fake_host_delay(int us) { g_host_delay_us = us; }
// a one-frame launch takes 1 ms, with strips of `rows` rows `ms`
void fake_fast_strip(int rows, double ms) { g_fast_strip = rows, g_fast_ms = ms; }
int fake_last_strip() { return g_last_strip; }     // of the first frame of the last launch that ran
int fake_table_kernels() { return g_table_kernels; }
void *fake_gate(cudaStream_t s)                 // the stream stands here until the gate opens
{
    auto *f = new std::shared_ptr<Flag>(std::make_shared<Flag>());
    stream_of(s).put([g = *f] { g->wait(); });
    return f;
}
void fake_open(void *gate) { (*static_cast<std::shared_ptr<Flag> *>(gate))->raise(); }
int fake_log(char *out, int max)                // the entries so far, one a line
{
    std::lock_guard<std::mutex> l(g_mu);
    std::string s;
    for (auto &e : g_log) s += e + "\n";
    if ((int)s.size() + 1 > max) return -1;
    std::memcpy(out, s.c_str(), s.size() + 1);
    return (int)g_log.size();
}

// ---------------------------------------------------------------- the runtime
cudaError_t cudaGetDeviceCount(int *n) { return *n = 1, cudaSuccess; }
cudaError_t cudaGetDevice(int *d) { return *d = 0, cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaGetDeviceProperties(cudaDeviceProp *p, int)
{
    std::memset(p, 0, sizeof(*p));
    p->multiProcessorCount = 152;
    return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr, int) { return *v = 152, cudaSuccess; }
cudaError_t cudaDeviceGetStreamPriorityRange(int *lo, int *hi) { return *lo = 0, *hi = -5, cudaSuccess; }
cudaError_t cudaDeviceSynchronize() { return cudaSuccess; }
cudaError_t cudaGetLastError()
{
    const cudaError_t e = t_error;
    t_error = cudaSuccess;
    return e;
}
const char *cudaGetErrorString(cudaError_t e) { return e == cudaSuccess ? "no error" : "made by the test"; }
cudaError_t cudaMalloc(void **p, size_t n)
{
    wait_for_host_functions();
    return *p = std::aligned_alloc(256, (n + 255) / 256 * 256), cudaSuccess;
}
cudaError_t cudaHostAlloc(void **p, size_t n, unsigned)
{
    wait_for_host_functions();
    return *p = std::aligned_alloc(256, (n + 255) / 256 * 256), cudaSuccess;
}
cudaError_t cudaFree(void *p) { return wait_for_host_functions(), std::free(p), cudaSuccess; }
cudaError_t cudaFreeHost(void *p) { return wait_for_host_functions(), std::free(p), cudaSuccess; }
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, cudaMemcpyKind)
{
    return wait_for_host_functions(), std::memcpy(d, s, n), cudaSuccess;
}
cudaError_t cudaMemset(void *d, int v, size_t n) { return wait_for_host_functions(), std::memset(d, v, n), cudaSuccess; }
cudaError_t cudaMemcpy2D(void *d, size_t dp, const void *s, size_t sp, size_t w, size_t h, cudaMemcpyKind)
{
    wait_for_host_functions();
    for (size_t y = 0; y < h; ++y)
        std::memcpy(static_cast<char *>(d) + y * dp, static_cast<const char *>(s) + y * sp, w);
    return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind, cudaStream_t st)
{
    const cudaError_t e = result("memcpy_async");
    if (e == cudaSuccess) stream_of(st).put([=] { std::memcpy(d, s, n); });
    return e;
}
cudaError_t cudaMemsetAsync(void *d, int v, size_t n, cudaStream_t st)
{
    return stream_of(st).put([=] { std::memset(d, v, n); }), cudaSuccess;
}
cudaError_t cudaGetSymbolAddress(void **p, const void *)
{
    static char *mem = static_cast<char *>(std::aligned_alloc(256, (size_t)2 << 20));
    return *p = mem, cudaSuccess;
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned)
{
    return *s = reinterpret_cast<cudaStream_t>(new Stream()), cudaSuccess;
}
cudaError_t cudaStreamCreateWithPriority(cudaStream_t *s, unsigned f, int) { return cudaStreamCreateWithFlags(s, f); }
cudaError_t cudaStreamDestroy(cudaStream_t s) { return delete reinterpret_cast<Stream *>(s), cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t s) { return stream_of(s).drain(), cudaSuccess; }
cudaError_t cudaStreamQuery(cudaStream_t s)
{
    Stream &st = stream_of(s);
    std::lock_guard<std::mutex> l(st.m);
    return st.q.empty() && !st.busy ? cudaSuccess : t_error = cudaErrorNotReady;
}
cudaError_t cudaStreamIsCapturing(cudaStream_t s, cudaStreamCaptureStatus *c)
{
    *c = stream_of(s).capture ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
    return cudaSuccess;
}
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned)
{
    return *e = reinterpret_cast<cudaEvent_t>(new Event()), cudaSuccess;
}
cudaError_t cudaEventCreate(cudaEvent_t *e) { return cudaEventCreateWithFlags(e, 0); }
cudaError_t cudaEventDestroy(cudaEvent_t e) { return delete reinterpret_cast<Event *>(e), cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s)
{
    auto f = std::make_shared<Flag>();
    reinterpret_cast<Event *>(e)->last = f;
    reinterpret_cast<Event *>(e)->at = g_clock_ms;
    stream_of(s).put([f] { f->raise(); });
    return cudaSuccess;
}
cudaError_t cudaEventSynchronize(cudaEvent_t e)
{
    if (auto f = reinterpret_cast<Event *>(e)->last) f->wait();
    return cudaSuccess;
}
cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned)
{
    if (auto f = reinterpret_cast<Event *>(e)->last) stream_of(s).put([f] { f->wait(); });
    return cudaSuccess;
}
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t a, cudaEvent_t b)
{
    return *ms = (float)(reinterpret_cast<Event *>(b)->at - reinterpret_cast<Event *>(a)->at), cudaSuccess;
}
cudaError_t cudaLaunchHostFunc(cudaStream_t s, cudaHostFn_t fn, void *arg)
{
    const cudaError_t e = result("host_func");
    if (e != cudaSuccess) return e;
    long id;
    {
        std::lock_guard<std::mutex> l(g_mu);
        id = g_next++;
        g_host.insert(id);
    }
    stream_of(s).put([=] {
        std::this_thread::sleep_for(std::chrono::microseconds(g_host_delay_us.load()));
        fn(arg);
        {
            std::lock_guard<std::mutex> l(g_mu);
            g_host.erase(id);
        }
        g_cv.notify_all();
    });
    return cudaSuccess;
}
cudaError_t cudaStreamBeginCapture(cudaStream_t s, cudaStreamCaptureMode)
{
    return stream_of(s).capture = new Graph(), cudaSuccess;
}
cudaError_t cudaStreamEndCapture(cudaStream_t s, cudaGraph_t *g)
{
    *g = reinterpret_cast<cudaGraph_t>(stream_of(s).capture);
    stream_of(s).capture = nullptr;
    return cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t *x, cudaGraph_t g, unsigned long long)
{
    log("graph made");
    return *x = reinterpret_cast<cudaGraphExec_t>(new Graph(*reinterpret_cast<Graph *>(g))), cudaSuccess;
}
cudaError_t cudaGraphDestroy(cudaGraph_t g) { return delete reinterpret_cast<Graph *>(g), cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t g) { return delete reinterpret_cast<Graph *>(g), cudaSuccess; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t g, cudaStream_t s)
{
    stream_of(s).put([] { log("graph"); });
    for (auto &f : reinterpret_cast<Graph *>(g)->ops) stream_of(s).put(f);
    return cudaSuccess;
}
// registration and launches of the objects' own kernels (none runs here)
void **__cudaRegisterFatBinary(void *) { return nullptr; }
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterFunction(void **, const char *, char *, const char *, int, uint3 *, uint3 *, dim3 *, dim3 *, int *) {}
void __cudaRegisterVar(void **, char *, char *, const char *, int, size_t, int, int) {}
unsigned __cudaPushCallConfiguration(dim3, dim3, size_t, void *) { return 1; }
cudaError_t __cudaPopCallConfiguration(dim3 *, dim3 *, size_t *, void *) { return cudaErrorLaunchFailure; }
cudaError_t __cudaGetKernel(cudaKernel_t *, const void *) { return cudaErrorLaunchFailure; }
cudaError_t __cudaLaunchKernel(cudaKernel_t, dim3, dim3, void **, size_t, cudaStream_t) { return cudaErrorLaunchFailure; }
}

// ---------------------------------------------------------------- the kernels' launchers
namespace ft {
cudaError_t launch_fused(const BatchHeader *h, int, cudaStream_t s, bool)
{
    return kernel("fused", s, [=] { return g_last_strip = h->frames[0].strip_rows, frames_of(h); });
}
cudaError_t launch_fused(const FrameCall &call, int, cudaStream_t s, bool)
{
    g_clock_ms = g_clock_ms + (call.f.strip_rows == g_fast_strip ? g_fast_ms.load() : 1.0);
    return kernel("fused", s, [n = call.f.strip_rows] { return g_last_strip = n, std::string("one"); });
}
cudaError_t launch_pose(const BatchHeader *h, int n, cudaStream_t s)
{
    return n > 0 ? kernel("pose", s, [=] { return frames_of(h); }) : cudaSuccess;
}
cudaError_t launch_pose(const FrameCall &, cudaStream_t s)
{
    return kernel("pose", s, [] { return std::string("one"); });
}
cudaError_t launch_fisheye(const BatchHeader *h, int n, int blocks, cudaStream_t s, bool)
{
    return n > 0 && blocks > 0 ? kernel("fisheye", s, [=] { return frames_of(h); }) : cudaSuccess;
}
cudaError_t launch_fisheye(const FrameCall &, int blocks, cudaStream_t s)
{
    return blocks > 0 ? kernel("fisheye", s, [] { return std::string("one"); }) : cudaSuccess;
}
cudaError_t launch_pyramids(const BatchHeader *h, int n, int, int, cudaStream_t s)
{
    return n > 0 ? kernel("pyramids", s, [=] { return frames_of(h); }) : cudaSuccess;
}
cudaError_t launch_pyramids(const FrameCall &, int, cudaStream_t s)
{
    return kernel("pyramids", s, [] { return std::string("one"); });
}
cudaError_t launch_orb(const OrbHeader *h, int n, int, int, int, cudaStream_t s)
{
    return n > 0 ? kernel("orb", s, [=] { return std::to_string(h->nimages); }) : cudaSuccess;
}
cudaError_t launch_table_copy(void *dst, const void *src, size_t bytes, cudaStream_t s)
{
    ++g_table_kernels;
    stream_of(s).put([=] { std::memcpy(dst, src, bytes); });
    return cudaSuccess;
}
int fisheye_blocks(int nl) { return (nl + 127) / 128; }
cudaError_t fisheye_setup() { return cudaSuccess; }
cudaError_t pyramid_setup() { return cudaSuccess; }
cudaError_t fused_occupancy(int *n) { return *n = 3, cudaSuccess; }
}  // namespace ft
