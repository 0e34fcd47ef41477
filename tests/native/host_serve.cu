// The server's host code on the fake runtime: kernels end at once (or when the
// test lets them) and report what the test wants.
#include <chrono>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <functional>
#include <memory>
#include <string>
#include <sys/mman.h>
#include <thread>

#include "api_internal.h"
#include "fake_cuda.h"
#include "fan.h"

using namespace sssp;

// ------------------------------------------------------------- launches --

struct Launch {
    char kind;            // 'W' cluster, 'T' grid, 'F' side by side, 'M' slice
    const int2* graph;    // its span: tells the graphs apart
    int nq;
};
static std::vector<Launch> launches;
static std::function<cudaError_t(const Launch&, Ctrl*)> on_launch;

static cudaError_t launched(const Launch& l, Ctrl* ctrl) {
    std::unique_lock<std::mutex> lk(fake::mu);
    launches.push_back(l);
    lk.unlock();
    if (on_launch) {
        const cudaError_t e = on_launch(l, ctrl);
        if (e != cudaSuccess || ctrl->error) return e;
    }
    ctrl->finished = l.nq;
    ctrl->stats[kStIter] = 10;
    return cudaSuccess;
}
static size_t count(char kind, const int2* graph = nullptr) {
    std::lock_guard<std::mutex> lk(fake::mu);
    size_t k = 0;
    for (const Launch& l : launches) k += l.kind == kind && (!graph || l.graph == graph);
    return k;
}

namespace sssp {
cudaError_t launch_wave(int, int, const WaveParams& p, int nq, int, size_t, cudaStream_t) {
    return launched({'W', p.span, nq}, p.ctrl);
}
cudaError_t launch_tide(int, int, const WaveParams& p, int, int, cudaStream_t) { return launched({'T', p.span, 1}, p.ctrl); }
cudaError_t launch_fan(int, const FanParams& p, int, cudaStream_t) { return launched({'F', p.span, p.nq}, p.ctrl); }
cudaError_t launch_fan_out(const uint32_t*, int32_t, int32_t, uint32_t*, int, cudaStream_t) { return cudaSuccess; }
#define INSTANCE(name)                                                                                             \
    cudaError_t launch_mlmq_##name(const KernelKey&, dim3, dim3, size_t, cudaStream_t, const KParams& p) {         \
        return launched({'M', nullptr, p.nq}, p.ctrl);                                                             \
    }                                                                                                              \
    cudaError_t occupancy_mlmq_##name(const KernelKey&, int, size_t, int* b) {                                     \
        *b = 1;                                                                                                    \
        return cudaSuccess;                                                                                        \
    }
INSTANCE(u32)
INSTANCE(u32x)
INSTANCE(f32)
INSTANCE(f32x)
}  // namespace sssp

// --------------------------------------------------------------- graphs --

// A graph in pages of its own, so that a read after its end faults.
static Graph* make_graph(int32_t n, int64_t m, double max_deg) {
    static uint64_t uid = 1000;
    void* p = mmap(nullptr, sizeof(Graph), PROT_READ | PROT_WRITE, MAP_PRIVATE | MAP_ANONYMOUS, -1, 0);
    Graph* g = new (p) Graph();
    g->uid = uid++;
    g->sms = 152;
    g->n = g->nv = n;
    g->m = g->mv = m;
    g->wtype = SSSP_W_U32;
    g->feat.avg_w = 4.0;
    g->feat.min_w = 1.0;
    g->feat.avg_deg = (double)m / n;
    g->feat.max_deg = max_deg;
    g->layout_req = kDefaultSplit;
    g->span = reinterpret_cast<int2*>(g->uid * 64);
    sssp_config_default(&g->defaults);
    return g;
}
// hubs and many arcs: one query on the grid, eight or more side by side
static Graph* grid_graph() { return make_graph(1 << 12, 1 << 20, 900.0); }
static Graph* small_graph() { return make_graph(1000, 6000, 20.0); }
static void end_graph(Graph* g) {
    graph_pins_wait(g->uid);
    mprotect(g, sizeof(Graph), PROT_NONE);
}
static sssp_graph* handle(Graph* g) { return reinterpret_cast<sssp_graph*>(g); }

struct Out {
    std::vector<uint32_t> d;
    std::vector<int32_t> p;
    uint64_t ticket = 0;
    Out(sssp_server* s, Graph* g, bool pred = false) : d(g->n), p(pred ? g->n : 0) {
        CHECK(sssp_serve_submit(s, handle(g), 1, d.data(), pred ? p.data() : nullptr, &ticket) == SSSP_OK);
    }
};
static int wait_state(sssp_server* s, const Out& o, int ms = 10000, int32_t* status = nullptr) {
    int32_t state = -1, st = 0;
    if (sssp_serve_wait(s, o.ticket, ms, &state, &st) == SSSP_E_TIMEOUT) return -1;
    if (status) *status = st;
    return state;
}
static sssp_server* server(void (*set)(sssp_serve_options*) = nullptr) {
    sssp_serve_options opt;
    sssp_serve_options_default(&opt);
    if (set) set(&opt);
    sssp_server* s = nullptr;
    CHECK(sssp_serve_create(&opt, &s) == SSSP_OK);
    return s;
}
static void sleep_ms(int ms) { std::this_thread::sleep_for(std::chrono::milliseconds(ms)); }
template <typename F>
static bool soon(F&& f) {
    for (int i = 0; i < 5000; i++, sleep_ms(1))
        if (f()) return true;
    return false;
}

// ---------------------------------------------------------------- tests --

// A graph that ended after its queries did is not read again; one whose
// cancelled query still runs ends after the job.
static void destroyed() {
    sssp_server* s = server();
    Graph *a = grid_graph(), *b = small_graph(), *c = grid_graph();
    {
        Out q(s, a);
        CHECK(wait_state(s, q) == SSSP_Q_DONE);
        end_graph(a);
    }
    for (int i = 0; i < 3; i++) {
        Out q(s, i % 2 ? c : b);
        CHECK(wait_state(s, q) == SSSP_Q_DONE);
    }
    for (Graph* g : {b, c}) {
        fake::busy = true;
        const size_t had = count('W') + count('T');
        Out q(s, g);
        CHECK(soon([&] { return count('W') + count('T') > had; }));
        CHECK(sssp_serve_cancel(s, q.ticket) == SSSP_OK);
        std::atomic<bool> ended{false};
        std::thread t([&] {
            end_graph(g);
            ended = true;
        });
        sleep_ms(50);
        CHECK(!ended);
        fake::busy = false;
        t.join();
    }
    Graph* d = grid_graph();
    Out q(s, d);
    CHECK(wait_state(s, q) == SSSP_Q_DONE);
    sssp_serve_destroy(s);
}

// One lane has always queries waiting; a query on another graph, and one on the
// same graph without predecessors, each get the grid in their turn.
static void turns() {
    sssp_server* s = server();
    Graph *a = grid_graph(), *b = grid_graph(), *c = grid_graph();
    a->feat.min_w = 0.0;   // strict-improvement predecessors: one by one
    std::vector<std::unique_ptr<Out>> more;
    std::atomic<int> left{300};
    on_launch = [&](const Launch& l, Ctrl*) {
        if (l.graph == a->span && left > 0) {
            left--;
            more.emplace_back(new Out(s, a, true));
        }
        return cudaSuccess;
    };
    fake::busy = true;
    for (int i = 0; i < 4; i++) more.emplace_back(new Out(s, a, true));
    CHECK(soon([&] { return count('T', a->span) == 1; }));
    Out q1(s, b), q2(s, c, true), q3(s, a);
    fake::busy = false;
    CHECK(wait_state(s, q1) == SSSP_Q_DONE && wait_state(s, q2) == SSSP_Q_DONE && wait_state(s, q3) == SSSP_Q_DONE);
    CHECK(left > 250);
    left = 0;
    CHECK(soon([&] {
        sssp_serve_stats st;
        sssp_serve_get_stats(s, &st);
        return st.completed == st.submitted;
    }));
    sssp_serve_destroy(s);
}

// A server that waits for the grid has its place among the solves that do, and
// gives it up when nobody waits any more.
static void places() {
    sssp_server* s = server();
    Graph* a = grid_graph();
    GridTurns& t = grid_turns(0);
    uint64_t later = 0;
    on_launch = [&](const Launch&, Ctrl*) {
        CHECK(!t.mine(later));
        return cudaSuccess;
    };
    for (int i = 0; i < 3; i++) {
        const uint64_t first = t.take();
        Out q(s, a);
        sleep_ms(30);
        CHECK(count('T') == (size_t)i);
        later = t.take();
        t.leave(first);
        CHECK(wait_state(s, q) == SSSP_Q_DONE && count('T') == (size_t)i + 1);
        CHECK(soon([&] { return t.mine(later); }));
        t.leave(later);
    }
    on_launch = nullptr;
    const uint64_t first = t.take();
    {
        Out q(s, a);
        sleep_ms(30);
        CHECK(sssp_serve_cancel(s, q.ticket) == SSSP_OK);
    }
    later = t.take();
    t.leave(first);
    CHECK(soon([&] { return t.mine(later); }));
    t.leave(later);
    // a place that is given up before its turn is passed over
    const uint64_t x = t.take(), y = t.take(), z = t.take();
    t.leave(y);
    CHECK(t.mine(x) && !t.mine(z));
    t.leave(x);
    CHECK(t.mine(z));
    t.leave(z);
    // the solves of two threads and a server's queries side by side
    std::atomic<int> solves{0};
    std::vector<std::thread> ts;
    for (int k = 0; k < 2; k++)
        ts.emplace_back([&] {
            Graph* g = grid_graph();
            std::vector<uint32_t> d(g->n);
            for (int i = 0; i < 200; i++, solves++)
                CHECK(sssp_solve(handle(g), i, d.data(), nullptr, nullptr, nullptr) == SSSP_OK);
        });
    for (int i = 0; i < 50; i++) {
        Out q(s, a);
        CHECK(wait_state(s, q) == SSSP_Q_DONE);
    }
    for (std::thread& th : ts) th.join();
    CHECK(solves == 400);
    sssp_serve_destroy(s);
}

// A solve on a stream that is busy holds up neither another graph's solve nor a
// server; one whose stream waits for another's solve ends after it.
static void busy_stream() {
    Graph *a = grid_graph(), *b = grid_graph(), *c = grid_graph();
    int mine;
    const cudaStream_t st = (cudaStream_t)&mine;
    std::vector<uint32_t> da(a->n), db(b->n);
    fake::busy_stream = st;
    std::atomic<bool> done{false};
    std::thread t([&] {
        CHECK(sssp_solve(handle(a), 1, da.data(), nullptr, nullptr, st) == SSSP_OK);
        done = true;
    });
    sleep_ms(50);
    CHECK(!done);
    std::atomic<bool> other{false};
    std::thread u([&] {
        CHECK(sssp_solve(handle(b), 1, db.data(), nullptr, nullptr, nullptr) == SSSP_OK);
        other = true;
    });
    CHECK(soon([&] { return other.load(); }));
    u.join();
    sssp_server* s = server();
    Out q(s, c);
    CHECK(wait_state(s, q) == SSSP_Q_DONE);
    sssp_serve_destroy(s);
    CHECK(!done);
    fake::busy_stream = nullptr;
    t.join();
}

// A lane without memory concerns its own queries: they wait for the lanes that
// are at work, then fail; the server and its other lanes go on.
static void no_memory() {
    sssp_server* s = server();
    Graph *a = grid_graph(), *b = small_graph();
    fake::busy = true;
    Out qb(s, b);
    CHECK(soon([&] { return count('W') == 1; }));
    fake::largest_malloc = 8 << 10;
    Out qa(s, a, true);
    sleep_ms(50);
    CHECK(wait_state(s, qa, 0) == -1);
    fake::busy = false;
    CHECK(wait_state(s, qb) == SSSP_Q_DONE);
    int32_t status = 0;
    CHECK(wait_state(s, qa, 10000, &status) == SSSP_Q_ERROR && status == SSSP_E_NOMEM);
    Out again(s, b);
    CHECK(wait_state(s, again) == SSSP_Q_DONE);
    fake::largest_malloc = ~(size_t)0;
    Out qc(s, a, true), qd(s, a);
    CHECK(wait_state(s, qc) == SSSP_Q_DONE && wait_state(s, qd) == SSSP_Q_DONE);
    CHECK(count('M') == 0);
    sssp_serve_destroy(s);
}

// A job of 32 queries that finds no room becomes smaller ones.
static void smaller_jobs() {
    sssp_server* s = server();
    Graph* a = make_graph(1 << 20, 1 << 22, 900.0);
    fake::busy = true;
    std::vector<std::unique_ptr<Out>> qs;
    qs.emplace_back(new Out(s, a));
    CHECK(soon([&] { return count('T') == 1; }));
    fake::largest_malloc = (size_t)100 << 20;   // the rows of a group are 134 MB
    for (int i = 0; i < 40; i++) qs.emplace_back(new Out(s, a));
    fake::busy = false;
    for (auto& q : qs) CHECK(wait_state(s, *q) == SSSP_Q_DONE);
    CHECK(count('F') == 0 && count('M') == 0 && count('T') == 41);
    fake::largest_malloc = ~(size_t)0;
    sssp_serve_destroy(s);
}

// Launches that the device refuses beside a running job wait for its end; refused
// with nothing running they go by slices.
static void refused_launches() {
    for (const bool always : {false, true}) {
        sssp_server* s = server();
        Graph* a = small_graph();
        launches.clear();
        std::atomic<bool> refuse{false};
        on_launch = [&](const Launch& l, Ctrl*) {
            return refuse && l.kind == 'W' ? cudaErrorLaunchOutOfResources : cudaSuccess;
        };
        fake::busy = true;
        Out q1(s, a);
        CHECK(soon([&] { return count('W') == 1; }));
        refuse = true;
        Out q2(s, a);
        if (!always) {
            // (the refused launch waits for its stream first)
            std::thread t([&] { sleep_ms(50); refuse = false; fake::busy = false; });
            CHECK(wait_state(s, q2) == SSSP_Q_DONE);
            t.join();
        } else {
            sleep_ms(20);
            fake::busy = false;
            CHECK(wait_state(s, q2) == SSSP_Q_DONE && count('M') > 0);
        }
        CHECK(wait_state(s, q1) == SSSP_Q_DONE);
        sssp_serve_destroy(s);
    }
    on_launch = nullptr;
}

// A job that runs into its kernels' time limit is not the query's end: a server
// without a limit of its own goes on in slices.
static void time_limit() {
    sssp_server* s = server();
    for (Graph* a : {grid_graph(), small_graph()}) {
        launches.clear();
        on_launch = [&](const Launch& l, Ctrl* c) {
            if (l.kind == 'W' || l.kind == 'T') c->error = kErrTimeout;
            return cudaSuccess;
        };
        Out q1(s, a), q2(s, a, true);
        CHECK(wait_state(s, q1) == SSSP_Q_DONE && wait_state(s, q2) == SSSP_Q_DONE);
        CHECK(count('M') >= 2);
    }
    // without room for slices the query ends, and is not run over and over
    Graph* b = grid_graph();
    launches.clear();
    on_launch = [&](const Launch& l, Ctrl* c) {
        if (l.kind == 'T') c->error = kErrTimeout;
        fake::largest_malloc = 8 << 10;
        return cudaSuccess;
    };
    Out q(s, b, true);
    int32_t status = 0;
    CHECK(wait_state(s, q, 10000, &status) == SSSP_Q_ERROR && status == SSSP_E_NOMEM && count('T') == 1);
    fake::largest_malloc = ~(size_t)0;
    on_launch = nullptr;
    sssp_serve_destroy(s);
}

// The engines are timed alike: a first launch that takes long (memory, loading)
// does not make the wavefront kernels the slower ones.
static void autotune() {
    Graph* a = grid_graph();
    bool first = true;
    on_launch = [&](const Launch& l, Ctrl*) {
        sleep_ms(l.kind == 'M' ? 3 : first ? 40 : 0);
        if (l.kind != 'M') first = false;
        return cudaSuccess;
    };
    std::vector<int32_t> srcs(20, 1);
    sssp_config c;
    CHECK(sssp_autotune(handle(a), srcs.data(), 1, 30, &c) == SSSP_OK);
    CHECK(!first && !a->tuned_queues);
    first = true;
    CHECK(sssp_autotune_batch(handle(a), srcs.data(), 20, 30, &c) == SSSP_OK);
    CHECK(!first && count('F') == 2 && a->batch_tuned.size() == 1 && !a->batch_tuned[0].queues);
    on_launch = [&](const Launch& l, Ctrl*) {   // and the other way round
        sleep_ms(l.kind == 'M' ? 0 : 10);
        return cudaSuccess;
    };
    CHECK(sssp_autotune(handle(a), srcs.data(), 1, 30, &c) == SSSP_OK && a->tuned_queues);
    CHECK(sssp_autotune_batch(handle(a), srcs.data(), 20, 30, &c) == SSSP_OK && a->batch_tuned[0].queues);
    on_launch = nullptr;
}

// Where the device has no room for a cluster, the fixed scratch serves the grid.
static void noalloc_without_clusters() {
    std::vector<int32_t> rp(1001), d(1000), p(1000);
    std::vector<uint32_t> arcs(12000);
    on_launch = [&](const Launch& l, Ctrl*) { return l.kind == 'W' ? cudaErrorLaunchOutOfResources : cudaSuccess; };
    for (int32_t* pred : {p.data(), (int32_t*)nullptr}) {
        launches.clear();
        CHECK(sssp_solve_noalloc(rp.data(), arcs.data(), 1000, 6000, SSSP_W_U32, 3, d.data(), pred, nullptr) == SSSP_OK);
        CHECK(count('W') == 1 && count('T') == 1);
    }
    on_launch = [&](const Launch&, Ctrl*) { return cudaErrorLaunchOutOfResources; };
    CHECK(sssp_solve_noalloc(rp.data(), arcs.data(), 1000, 6000, SSSP_W_U32, 3, d.data(), nullptr, nullptr) == SSSP_E_CUDA);
    on_launch = nullptr;
}

// A front that is too wide for a cluster sends a job to the grid, and the graph
// remembers it.
static void wide_fronts() {
    sssp_server* s = server();
    Graph* a = make_graph(200000, 800000, 4.0);
    on_launch = [&](const Launch& l, Ctrl* c) {
        if (l.kind == 'W') c->error = kErrWide;
        return cudaSuccess;
    };
    for (int i = 0; i < 2; i++) {
        Out q(s, a);
        CHECK(wait_state(s, q) == SSSP_Q_DONE);
        CHECK(a->wide && count('W') == 1 && count('T') == (size_t)i + 1);
    }
    on_launch = nullptr;
    sssp_serve_destroy(s);
}

// After a device fault every query ends with it, and the server can be destroyed:
// jobs, slices and the grid's turn are given up.
static void fault() {
    for (const bool slices : {false, true}) {
        sssp_server* s = slices ? server([](sssp_serve_options* o) { o->query_timeout_ms = 1000000; }) : server();
        Graph *a = grid_graph(), *b = small_graph();
        launches.clear();
        if (slices) {
            on_launch = [](const Launch&, Ctrl*) {
                fake::busy = true;   // (a lane is opened on a quiet stream)
                return cudaSuccess;
            };
        } else {
            fake::busy = true;
        }
        Out q1(s, a);
        CHECK(soon([&] { return count(slices ? 'M' : 'T') == 1; }));
        Out q2(s, b), q3(s, a);
        on_launch = nullptr;
        fake::event_fault = true;
        sleep_ms(20);
        // what still runs is waited for
        CHECK(wait_state(s, q1, 0) == -1 && wait_state(s, q2, 0) == -1);
        fake::busy = false;
        int32_t status = 0;
        for (Out* q : {&q1, &q2, &q3})
            CHECK(wait_state(s, *q, 10000, &status) == SSSP_Q_ERROR && status == SSSP_E_CUDA);
        fake::event_fault = false;
        uint64_t t;
        CHECK(sssp_serve_submit(s, handle(b), 0, q2.d.data(), nullptr, &t) == SSSP_E_CUDA);
        sssp_serve_destroy(s);
        const uint64_t place = grid_turns(0).take();
        CHECK(grid_turns(0).mine(place));
        grid_turns(0).leave(place);
        end_graph(a);
        end_graph(b);
    }
}

int main(int argc, char** argv) {
    const std::string what = argc > 1 ? argv[1] : "";
    if (what == "destroyed") destroyed();
    else if (what == "turns") turns();
    else if (what == "places") places();
    else if (what == "busy_stream") busy_stream();
    else if (what == "no_memory") no_memory();
    else if (what == "smaller_jobs") smaller_jobs();
    else if (what == "refused_launches") refused_launches();
    else if (what == "fault") fault();
    else if (what == "wide_fronts") wide_fronts();
    else if (what == "noalloc_without_clusters") noalloc_without_clusters();
    else if (what == "autotune") autotune();
    else if (what == "time_limit") time_limit();
    else CHECK(!"a test's name");
    std::puts("ok");
    return 0;
}
