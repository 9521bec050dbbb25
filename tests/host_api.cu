// Checks of the library's host code on the CPU: every object of liblbm.so linked
// with tests/host_runtime.cpp in place of the CUDA runtime.
//
//   host_api <check> [arguments]     prints its findings; see tests/test_host_api.py
#include <cstdio>
#include <cstdlib>
#include <string>
#include <vector>

#include "host_runtime.h"
#include "lbm.h"
#include "lbm_kernels.cuh"

namespace {

lbm_handle make(int nx, int ny, int nz, int pair, int storage, int forcing = LBM_SHAN_CHEN)
{
    lbm_params p;
    lbm_params_from_physics(&p, nx, ny, nz, pair, forcing, 100.0, 1.0, 1.0, 0.04);
    p.storage = storage;
    lbm_handle h = nullptr;
    if (lbm_create_params(&h, &p)) std::printf("create: %s\n", lbm_last_error());
    return h;
}

void start(lbm_handle h)
{
    const double field = 1.0;   // copies are recorded, not made
    if (lbm_init_fields(h, &field, &field, &field, nullptr, nullptr, 0.0)) std::printf("init: %s\n", lbm_last_error());
}

// A record after a failed one: the k-th allocation of the first call fails, the
// second call has everything in place. One line per k until no call fails.
int record_scratch(int fused)
{
    for (int k = 0;; ++k) {
        lbm_handle h = make(16, 16, 16, LBM_D3Q19_D3Q7, LBM_FP32);
        start(h);
        lbm_diag d;
        auto record = [&] { return fused ? lbm_step_diagnostics(h, 1, &d) : lbm_diagnostics(h, &d); };
        g_work.clear();
        g_fail_in = k;
        const int first = record();
        const bool failed = g_fail_in < 0;
        g_fail_in = -1;
        size_t launches = 0;
        for (const Work& w : g_work) launches += w.kind == Work::kLaunch;
        const int second = record();
        bool scratch = true;
        std::set<void*> cleared;
        for (size_t i = 0; i < g_work.size(); ++i) {
            const Work& w = g_work[i];
            if (w.kind == Work::kMemset) cleared.insert(w.at);
            if (w.kind != Work::kLaunch || !w.launch.is("k_diag_gradients")) continue;
            const lbm::DiagArgs& a = w.launch.as<lbm::DiagArgs>();
            auto live = [&](const void* p) {
                cudaPointerAttributes t;
                return cudaPointerGetAttributes(&t, p) == cudaSuccess && t.type == cudaMemoryTypeDevice;
            };
            scratch = scratch && live(a.fields) && live(a.partials) && live(a.grad_rows) && live(a.finished) &&
                      g_other.count(a.out) && cleared.count(a.finished);
        }
        lbm_destroy(h);
        std::printf("%d first %d launches %zu second %d scratch %d left %zu\n", k, first, failed ? launches : (size_t)0,
                    second, scratch ? 1 : 0, g_device.size() + g_other.size());
        if (!failed) return 0;
    }
}

// A per-instance batch call of 12 lattices whose k-th allocation (streams and
// events among them) fails, and the same call again. One line per k until no
// call fails. `open`: streams whose launches of the failed call the batch's
// stream was not made to wait for; `null`: launches of either call on no stream.
int batch_calls(const std::string& call)
{
    for (int k = 0;; ++k) {
        std::vector<lbm_params> ps;
        for (int n : {32, 16, 24, 20, 16, 32, 24, 20, 16, 16, 40, 8}) {
            lbm_params p;
            lbm_params_from_physics(&p, n, n, n, LBM_D3Q19_D3Q7, LBM_GUO, 100.0, 1.0, 1.0, 0.04);
            ps.push_back(p);
        }
        lbm_batch b = nullptr;
        lbm_batch_create(&b, ps.data(), (int)ps.size());
        lbm_batch_set_mode(b, LBM_BATCH_INSTANCES, 100);
        lbm_batch_init_tgv(b, 1, 1e-3);
        lbm_handle h = nullptr;
        void* own = nullptr;
        lbm_batch_instance(b, 0, &h);
        lbm_get_stream(h, &own);
        std::vector<lbm_diag> d(ps.size());
        auto run = [&] { return call == "step" ? lbm_batch_step(b, 3) : lbm_batch_diagnostics(b, d.data()); };
        g_work.clear();
        g_fail_in = k;
        const int first = run();
        const bool failed = g_fail_in < 0;
        g_fail_in = -1;
        std::map<cudaStream_t, bool> joined;
        std::map<void*, cudaStream_t> recorded;
        for (const Work& w : g_work) {
            if (w.kind == Work::kLaunch && w.stream != own) joined[w.stream] = false;
            if (w.kind == Work::kRecord) recorded[w.at] = w.stream;
            if (w.kind == Work::kWait && w.stream == own) joined[recorded[w.at]] = true;
        }
        int open = 0;
        for (const auto& j : joined) open += !j.second;
        const int second = run();
        int null = 0;
        std::set<cudaStream_t> used;
        for (const Work& w : g_work) {
            null += w.kind == Work::kLaunch && w.stream == nullptr;
            if (w.kind == Work::kLaunch) used.insert(w.stream);
        }
        lbm_batch_destroy(b);
        std::printf("%d first %d open %d second %d null %d streams %zu left %zu\n", k, first, open, second, null,
                    used.size(), g_device.size() + g_other.size());
        if (!failed) return 0;
    }
}

// Pack and unpack with buffers that end `short_by` bytes before lbm_halo_bytes,
// one of the two at a time: statuses and launches.
int halo_buffers(long short_by)
{
    lbm_handle h = make(33, 9, 6, LBM_D3Q27_D3Q19, LBM_FP16_DEV);
    start(h);
    lbm_set_slab(h, 1);
    size_t bytes = 0;
    lbm_halo_bytes(h, &bytes);
    void *whole = nullptr, *cut = nullptr;
    cudaMalloc(&whole, bytes + 64);
    cudaMalloc(&cut, bytes + 64);
    char* w = static_cast<char*>(whole) + 64;
    char* c = static_cast<char*>(cut) + 64 + short_by;
    for (int phase = 0; phase < 2; ++phase)
        for (int side = 0; side < 2; ++side) {
            g_work.clear();
            const int p = lbm_halo_pack(h, phase, side ? w : c, side ? c : w);
            const int u = lbm_halo_unpack(h, phase, side ? w : c, side ? c : w);
            std::printf("pack %d unpack %d launches %zu\n", p, u, g_work.size());
        }
    cudaFree(whole);
    cudaFree(cut);
    lbm_destroy(h);
    return 0;
}

// The launches of two single steps: threads of a block, whether rows are
// numbered through, whether the launch overlaps the one before.
int step_launches(int nx, int ny, int nz, int pair, int storage)
{
    lbm_handle h = make(nx, ny, nz, pair, storage);
    start(h);
    g_work.clear();
    lbm_step(h, 1);
    lbm_step(h, 1);
    for (const Work& w : g_work)
        if (w.kind == Work::kLaunch)
            std::printf("%u %s %s\n", w.launch.block.x * w.launch.block.y, w.launch.as<lbm::StepArgs>().flat ? "flat" : "shaped",
                        w.launch.overlapped ? "overlapped" : "alone");
    lbm_destroy(h);
    return 0;
}

// Step launches of a lattice for calls of the given step counts: AA parity,
// planes and rows (first, number) and the direction; "graph" in front of a
// replay's. `call` of a number before each call's.
int step_ranges(int nx, int ny, int nz, int pair, int storage, int calls, char** counts)
{
    lbm_handle h = make(nx, ny, nz, pair, storage);
    start(h);
    for (int c = 0; c < calls; ++c) {
        g_work.clear();
        std::printf("call %s\n", counts[c]);
        if (lbm_step(h, std::atoi(counts[c]))) std::printf("%s\n", lbm_last_error());
        for (const Work& w : g_work) {
            if (w.kind != Work::kLaunch) continue;
            const lbm::StepArgs& a = w.launch.as<lbm::StepArgs>();
            const bool odd = w.launch.is("Lb1E");
            std::printf("%s%d %d %u %d %d %d\n", w.replayed ? "graph " : "", odd ? 1 : 0, a.z0, w.launch.grid.z, a.y0, a.rows,
                        a.down);
        }
    }
    lbm_destroy(h);
    return 0;
}

// lbm_autotune where a launch takes `nodes` x the threads' distance from
// `threads` (and 1 more if it is not as flat as `flat`): how many of its step
// launches cover the lattice, what it returns and what 32 steps take after it.
int autotune(int n, int pair, int threads, int flat, int batched)
{
    lbm_handle h = nullptr;
    lbm_batch b = nullptr;
    if (batched) {
        lbm_params p[2];
        for (lbm_params& q : p) lbm_params_from_physics(&q, n, n, n, pair, LBM_GUO, 100.0, 1.0, 1.0, 0.04);
        lbm_batch_create(&b, p, 2);
        lbm_batch_init_tgv(b, 1, 0.0);
        lbm_batch_instance(b, 1, &h);
    } else {
        h = make(n, n, n, pair, LBM_FP32);
        start(h);
    }
    g_cost = [=](const Launch& l) {
        if (!l.is("6k_step")) return l.is("k_batch") ? 1e6 : 0.0;
        const lbm::StepArgs& a = l.as<lbm::StepArgs>();
        const int off = std::abs((int)(l.block.x * l.block.y) - threads) + ((a.flat != 0) != (flat != 0) ? 1 : 0);
        return 1e-9 * n * a.rows * l.grid.z * (1.0 + off);
    };
    g_work.clear();
    double ms = 0.0;
    if (batched ? lbm_batch_autotune(b, 3, &ms) : lbm_autotune(h, 3, &ms)) std::printf("%s\n", lbm_last_error());
    int whole = 0, all = 0;
    for (const Work& w : g_work)
        if (w.kind == Work::kLaunch && w.launch.is("6k_step")) {
            ++all;
            whole += (int)w.launch.grid.z == n && w.launch.as<lbm::StepArgs>().rows == n;
        }
    g_work.clear();
    batched ? lbm_batch_step(b, 32) : lbm_step(h, 32);
    double spent = 0.0;
    for (const Work& w : g_work)
        if (w.kind == Work::kLaunch) spent += g_cost(w.launch);
    std::printf("%d %d %.9g %.9g\n", whole, all, ms, spent / 32);
    batched ? lbm_batch_destroy(b) : lbm_destroy(h);
    return 0;
}

// lbm_launch_count against the launches recorded, after each of: steps, a fused
// record with more steps, a record.
int launch_count(int n, int pair, int storage)
{
    lbm_handle h = make(n, n, n, pair, storage);
    start(h);
    lbm_diag d;
    g_work.clear();
    for (int k : {1, 70, 33, 300}) {
        lbm_step(h, k);
        lbm_step_diagnostics(h, k, &d);
        lbm_diagnostics(h, &d);
        int64_t launches = 0, recorded = 0;
        lbm_launch_count(h, &launches);
        for (const Work& w : g_work) recorded += w.kind == Work::kLaunch;
        std::printf("%lld %lld\n", (long long)launches, (long long)recorded);
    }
    lbm_destroy(h);
    return 0;
}

}  // namespace

int main(int argc, char** argv)
{
    const std::string what = argc > 1 ? argv[1] : "";
    g_arg_bytes = [](const std::string& kernel) {
        const auto has = [&](const char* k) { return kernel.find(k) != std::string::npos; };
        return has("k_step") && !has("staged") ? sizeof(lbm::StepArgs) : has("k_diag_gradients") ? sizeof(lbm::DiagArgs) : 0;
    };
    if (what == "record") return record_scratch(std::atoi(argv[2]));
    if (what == "batch") return batch_calls(argv[2]);
    if (what == "halo") return halo_buffers(std::atol(argv[2]));
    const auto arg = [&](int i) { return std::atoi(argv[i]); };
    if (what == "launches") return step_launches(arg(2), arg(3), arg(4), arg(5), arg(6));
    if (what == "steps") return step_ranges(arg(2), arg(3), arg(4), arg(5), arg(6), argc - 7, argv + 7);
    if (what == "autotune") return autotune(arg(2), arg(3), arg(4), arg(5), arg(6));
    if (what == "count") return launch_count(arg(2), arg(3), arg(4));
    std::printf("unknown check '%s'\n", what.c_str());
    return 2;
}
