// C ABI (include/lbm.h): handle management, parameter mapping, launches,
// CUDA-graph replay of the AA step pair, diagnostics, autotuning.
#include <cuda.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <limits>
#include <mutex>
#include <new>
#include <string>
#include <vector>

#include "../../include/lbm.h"
#include "lbm_dispatch.h"
#include "lbm_halo.cuh"
#include "lbm_kernels.cuh"
#include "lbm_stage.cuh"

using namespace lbm;

namespace {

thread_local std::string g_last_error;

int fail(int code, const char* fmt, ...)
{
    char buf[512];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, sizeof(buf), fmt, ap);
    va_end(ap);
    g_last_error = buf;
    return code;
}

int cuda_fail(cudaError_t e, const char* what)
{
    return fail(LBM_ECUDA, "%s: %s", what, cudaGetErrorString(e));
}

#define LBM_CUDA(call, what)                                   \
    do {                                                       \
        cudaError_t e_ = (call);                               \
        if (e_ != cudaSuccess) return cuda_fail(e_, what);     \
    } while (0)

struct PairInfo {
    int qf, qg;
};

bool pair_info(int pair, PairInfo* out)
{
    static const PairInfo t[7] = {{27, 19}, {19, 7}, {27, 27}, {19, 19}, {19, 15}, {15, 7}, {7, 27}};
    if (pair < 0 || pair > 6) return false;
    *out = t[pair];
    return true;
}

double cs2_of(int q) { return q == 7 ? 0.25 : 1.0 / 3.0; }

size_t elem_size(int storage) { return storage == LBM_FP32 ? 4 : 2; }

constexpr int kGraphSteps = 64;   // even number: the graph starts and ends in natural layout

// Looks up (again) the device address of the allocation-free diagnostics
// scratch on `device`, which must be current; defined with the array below.
void static_scratch_refresh(int device);

// What a lattice may take of L2: as it comes; steps beside others of its batch,
// whole lattices only; has the GPU to itself in its batch.
enum class L2Use { unknown, shared, alone };

}  // namespace

struct lbm_ctx {
    lbm_params p{};
    PairInfo q{};
    Geometry geo{};
    Phys ph{};
    const KernelSet* ks = nullptr;
    int device = 0;
    int num_sms = 0;
    cudaStream_t stream = nullptr;
    bool own_stream = false;
    void* store = nullptr;
    size_t store_bytes = 0;
    bool own_store = false;
    bool initialized = false;
    int64_t step = 0;
    int odd = 0;           // layout parity of the store
    int bx = 0, by = 0;      // launch shape of the even AA steps
    int bxo = 0, byo = 0;    // and of the odd ones
    int pairing = LBM_PAIRING_ALL;   // two nodes per thread (16-bit storage, even nx)
    int flat[2] = {0, 0};            // threads per block of flat launches, per AA parity; 0: shaped (bx x by)
    size_t l2_bytes = 0;
    bool mirrored = false;           // direction of the latest group of skewed steps
    cudaGraphExec_t skew_graph = nullptr;   // kSkewGraphSteps skewed steps from the natural layout
    int skew_eager = 0;              // skewed steps launched one by one (counted up to the graph's due)
    L2Use l2 = L2Use::unknown;
    bool tile_staging = false;        // bulk-copy staged kernel where it applies
    bool slab = false;                // z-slab: planes 0 and nz - 1 are ghost planes (lbm_set_slab)
    bool stage_used = false;          // the staged kernel, the one that can raise d_err, has been launched
    int stage_grid = 0;               // persistent grid of the staged kernel (0: not derived yet)
    int* d_err = nullptr;             // device flag raised by a bounded wait that ran out
    uint32_t stage_spin = 1u << 22;   // mbarrier polls per wait
    uint32_t stage_extra_tx = 0;      // test hook: bytes a barrier of their own expects and no copy delivers
    // diagnostics scratch
    float* diag_fields = nullptr;
    double* diag_partials = nullptr;
    int diag_rows = 0;                 // rows of kDNumSlots the partials hold
    cudaEvent_t diag_event = nullptr;  // totals written to diag_host
    double* diag_grad = nullptr;       // pass-2 rows, then the count of finished blocks
    double* diag_host = nullptr;       // pinned; the totals, written by the last kernel itself
    // host<->device staging
    double* staging = nullptr;
    size_t staging_bytes = 0;
    cudaEvent_t copy_event = nullptr;   // host->device copies of lbm_init_fields done
    // lbm_prefetch_fields / lbm_init_prefetched: two device buffers of the
    // five FP64 fields, filled on a copy stream while the lattice steps
    double* pre[2] = {nullptr, nullptr};
    cudaStream_t copy_stream = nullptr;
    cudaEvent_t pre_done[2] = {nullptr, nullptr};   // copies into pre[b] complete
    cudaEvent_t pre_free[2] = {nullptr, nullptr};   // the init that read pre[b] complete
    bool pre_free_recorded[2] = {false, false};
    int pre_next = 0;     // buffer the next prefetch fills
    int pre_ready = -1;   // buffer holding a prefetch not yet used, or -1
    // CUDA graph of kGraphSteps steps starting from the natural layout
    bool graphs = true;
    cudaGraphExec_t graph = nullptr;
    cudaStream_t graph_stream = nullptr;
    int64_t launches = 0;                             // kernels of steps and records, replayed ones too
    int64_t graph_launches = 0, skew_launches = 0;    // of a replay of `graph`, `skew_graph`
};

namespace {

void derive_phys(lbm_ctx* h)
{
    const lbm_params& p = h->p;
    Phys& ph = h->ph;
    ph.delta_f = (float)((2.0 * p.tau_f - 1.0) / p.tau_f);
    ph.delta_g = (float)((2.0 * p.tau_g - 1.0) / p.tau_g);
    ph.G = (float)p.G;
    ph.beta = (float)p.beta;
    ph.rho0 = (float)p.rho0;
    const double c_mom = (p.scalar_mode == LBM_SCALAR_PRINTED) ? 0.5 * (1.0 - 1.0 / (2.0 * p.tau_g)) : 0.5;
    const double c_lbe = (p.scalar_mode == LBM_SCALAR_PRINTED) ? 1.0 : 1.0 - 1.0 / (2.0 * p.tau_g);
    ph.kappa = (float)(c_mom * -p.beta);
    ph.c_lbe = (float)c_lbe;
    ph.guo_pref = (float)(1.0 - 1.0 / (2.0 * p.tau_f));
    ph.guo_tau = (float)(p.tau_f - 0.5);
    ph.sc_tau = (float)(p.sc_shift * p.tau_f);
    h->geo.nx = p.nx;
    h->geo.ny = p.ny;
    h->geo.nz = p.nz;
    h->geo.n3 = (uint32_t)((size_t)p.nx * p.ny * p.nz);
}

// Tile width of the staged kernel (a multiple of 64 that divides nx), or 0
// where it does not apply: FP32 storage, nx not a multiple of 64, or a store
// not 16-byte aligned (bulk copies need 16-byte aligned rows).
int stage_width(const lbm_ctx* h)
{
    if (!h->tile_staging || h->slab || h->ks->staged[h->p.forcing][0] == nullptr || h->store == nullptr) return 0;
    if (reinterpret_cast<uintptr_t>(h->store) % 16 != 0) return 0;
    const int nx = h->p.nx;
    return nx % 256 == 0 ? 256 : nx % 128 == 0 ? 128 : nx % 64 == 0 ? 64 : 0;
}

bool uses_pairs(const lbm_ctx* h, int odd)
{
    const bool wanted = h->pairing == LBM_PAIRING_ALL || (h->pairing == LBM_PAIRING_EVEN && !odd);
    return wanted && h->ks->step2[h->p.forcing][0][0] != nullptr && (h->p.nx % 2) == 0;
}

// Waves of resident blocks that one step of one node per thread takes.
double step_waves(const lbm_ctx* h)
{
    const int qsum = h->q.qf + h->q.qg;
    const int per_sm = 256 * (qsum > 46 ? 2 : qsum <= 26 ? 4 : 3);
    return (double)h->geo.n3 / ((double)per_sm * h->num_sms);
}

// Less than one wave of the longer kernels: every step is one block's latency.
bool one_short_wave(const lbm_ctx* h) { return h->q.qf + h->q.qg >= 38 && step_waves(h) <= 1.0; }

// Whether a step's blocks may wait on the SMs for the end of the step before
// (launch_overlapped). Nearly always the faster: 64^3 FP32 D3Q27xD3Q19 11.7
// against 12.2 us per step, 32^3 D3Q19xD3Q7 2.2 against 2.7, D3Q19xD3Q19 2.69
// against 3.15, D3Q27xD3Q19 FP16 3.2 against 3.8 and at 20^3 3.1 against 3.6.
// Not for the longest FP32 kernels between two 64-thread blocks per SM and one
// wave: there the waiting blocks take their places unevenly (D3Q27xD3Q27 FP32
// 24^3 2.75 against 3.05 us, but 28^3 3.57 against 3.40 and 32^3 3.80 against
// 3.72; D3Q27xD3Q19 32^3 3.2 to 3.3 against 3.4 to 3.6 on some GPUs, up to 3.9 on
// another).
bool overlaps_steps(const lbm_ctx* h)
{
    const bool longest = h->p.storage == LBM_FP32 && h->q.qf + h->q.qg >= 46;
    return !(longest && one_short_wave(h) && h->geo.n3 > 2u * 64u * (uint32_t)h->num_sms);
}

// Default launch shape of one AA parity, from per-parity sweeps of the
// candidate shapes at 256^3: the two-nodes-per-thread kernel runs best in
// 128-thread blocks of 64 x 2, except on the odd steps of D3Q27xD3Q19, where
// one row of 128 is faster (FP16 0.462 against 0.465 ms, BF16 0.462 against
// 0.467 ms); the one-node kernels in one row of 256 threads on even steps
// and on the odd steps of the pairs with 38 to 46 populations per node, one
// row of 128 on the odd steps of the smaller pairs (D3Q19xD3Q7 0.515 / 0.528
// ms, D3Q19xD3Q19 0.751 / 0.768 ms, against 0.520 / 0.528 and 0.758 / 0.776
// as 128 on both), and for D3Q27xD3Q27 (two 128-register blocks per SM) one
// row of 64 on even steps and 128 on odd steps (1.058 / 1.096 ms against
// 1.072 / 1.155 ms as 256). Below 20 waves 128 threads: the last, partly filled
// wave then weighs less than the row order gains (27x19 / 19x7 FP32 at 64^3 11.9
// / 7.5 us against 12.9 / 7.7 with 256, at 128^3 117.3 / 67.1 against 118.4 /
// 67.3), and below one wave of the longer kernels 64 (27x19 Guo FP32 shaped, 64 /
// 256 threads, us per step: 16^3 2.92 / 3.21, 24^3 3.05 / 3.40, 28^3 3.31 / 3.62,
// 32^3 3.60 / 3.66; at 31^3, where 256 fill 124 SMs evenly, 3.89 / 3.77).
void pick_block(const lbm_ctx* h, int odd, int& bx, int& by)
{
    const bool pairs = uses_pairs(h, odd);
    const int xunits = pairs ? h->p.nx / 2 : h->p.nx;
    const int qsum = h->q.qf + h->q.qg;
    const bool big = qsum >= 46;
    const int threads = pairs                                ? 128
                        : qsum <= 46 && one_short_wave(h)    ? 64
                        : qsum <= 46 && step_waves(h) < 20.0 ? 128
                        : qsum > 46                          ? (odd ? 128 : 64)
                        : (odd && qsum <= 34)                ? 128
                                                             : 256;
    const int want = pairs ? ((odd && big) ? 128 : 64) : threads;
    bx = 32;
    while (bx * 2 <= want && bx * 2 <= xunits) bx *= 2;
    by = threads / bx;
    while (by > 1 && by / 2 >= h->p.ny) by /= 2;
    while (bx * by < 256 && (h->p.ny + by - 1) / by > 65535) by *= 2;   // rows of blocks within the grid's limit
}

// Threads per block of a flat launch (the plane's units numbered through, row
// after row) where it leaves clearly fewer lanes idle than the shape bx x by;
// 0 where the shape stays. A shape rounds every row up to whole blocks: FP32
// D3Q27xD3Q19 us per step shaped / flat at 48^3 7.7 / 6.1, 65^3 21.5 / 14.2,
// 72^3 25.0 / 17.0, 96^3 55.9 / 52.6, 160^3 243 / 229. Where a row fills its
// blocks the flat order costs its division (128^3 118.2 / 119.7), hence the
// 4 %. 128 threads against 256: up to 26 % faster, at most 2 % slower (16^3 to
// 225 x 150 x 75, six pairs and storages). D3Q27xD3Q27 FP32 keeps its shape
// up to three 64-thread blocks per SM, where idle lanes cost less than the
// division (16^3 to 28^3 2.44, 2.51, 2.75, 3.40 us against 2.63, 2.60, 2.82,
// 3.47; at 7 blocks per SM 33^3 5.78 against 4.43).
int pick_flat(const lbm_ctx* h, int odd, int bx, int by)
{
    const int row = uses_pairs(h, odd) ? h->p.nx / 2 : h->p.nx;
    const int64_t plane = (int64_t)row * h->p.ny;
    if (row < 2) return 0;
    const int64_t blocks = (int64_t)((row + bx - 1) / bx) * ((h->p.ny + by - 1) / by) * h->p.nz;
    if (h->p.storage == LBM_FP32 && h->q.qf + h->q.qg > 46 && blocks * bx * by <= (int64_t)(3 * 64) * h->num_sms) return 0;
    int64_t best = (int64_t)((row + bx - 1) / bx) * ((h->p.ny + by - 1) / by) * (bx * by) * 100 / 104;
    int pick = 0;
    for (int t = 128; t >= 64; t /= 2) {
        const int64_t lanes = (plane + t - 1) / t * t;
        if (lanes < best) {
            best = lanes * 100 / 104;
            pick = t;
        }
    }
    return pick;
}

void default_block(lbm_ctx* h)
{
    pick_block(h, 0, h->bx, h->by);
    pick_block(h, 1, h->bxo, h->byo);
    h->flat[0] = pick_flat(h, 0, h->bx, h->by);
    h->flat[1] = pick_flat(h, 1, h->bxo, h->byo);
}

dim3 step_block(const lbm_ctx* h, int odd)
{
    if (h->flat[odd]) return dim3((unsigned)h->flat[odd]);
    return odd ? dim3((unsigned)h->bxo, (unsigned)h->byo) : dim3((unsigned)h->bx, (unsigned)h->by);
}

void drop_graph(lbm_ctx* h)
{
    if (h->graph) cudaGraphExecDestroy(h->graph);
    h->graph = nullptr;
    if (h->skew_graph) cudaGraphExecDestroy(h->skew_graph);
    h->skew_graph = nullptr;
}

size_t store_need(const lbm_ctx* h)
{
    return (size_t)(h->q.qf + h->q.qg) * h->geo.n3 * elem_size(h->p.storage);
}

int ensure_store(lbm_ctx* h)
{
    if (h->store) return LBM_OK;
    const size_t bytes = store_need(h);
    void* ptr = nullptr;
    cudaError_t e = cudaMalloc(&ptr, bytes);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return fail(LBM_ENOMEM, "cudaMalloc of %zu bytes for the population store failed: %s", bytes,
                    cudaGetErrorString(e));
    }
    h->store = ptr;
    h->store_bytes = bytes;
    h->own_store = true;
    return LBM_OK;
}

void* f_ptr(lbm_ctx* h) { return h->store; }
void* g_ptr(lbm_ctx* h)
{
    return static_cast<char*>(h->store) + (size_t)h->q.qf * h->geo.n3 * elem_size(h->p.storage);
}

int ensure_staging(lbm_ctx* h, size_t bytes)
{
    if (!h->copy_event && cudaEventCreateWithFlags(&h->copy_event, cudaEventDisableTiming) != cudaSuccess) {
        cudaGetLastError();
        return fail(LBM_ECUDA, "event creation failed");
    }
    if (h->staging_bytes >= bytes) return LBM_OK;
    if (h->staging) cudaFree(h->staging);
    h->staging = nullptr;
    h->staging_bytes = 0;
    cudaError_t e = cudaMalloc(&h->staging, bytes);
    if (e != cudaSuccess) {
        cudaGetLastError();
        h->staging = nullptr;
        return fail(LBM_ENOMEM, "cudaMalloc of %zu staging bytes failed: %s", bytes, cudaGetErrorString(e));
    }
    h->staging_bytes = bytes;
    return LBM_OK;
}

// Consecutive steps and diagnostics passes overlap their launches: the kernel
// starts with wait_prerequisites (griddepcontrol.wait) and touches nothing
// that an earlier one writes before it.
cudaError_t launch_overlapped(const void* k, dim3 grid, dim3 block, void** args, cudaStream_t s, bool overlap = true)
{
    cudaLaunchAttribute pdl{};
    pdl.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    pdl.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.stream = s;
    cfg.attrs = &pdl;
    cfg.numAttrs = overlap && s != nullptr ? 1u : 0u;
    return cudaLaunchKernelExC(&cfg, k, args);
}

// Pass 1 on its own: four blocks per SM (D3Q27xD3Q27, whose kernel fits three,
// runs the fourth in a second wave), or one per 256 nodes of a small lattice.
uint32_t moment_blocks(const lbm_ctx* h, uint32_t nodes)
{
    return std::min(4u * (uint32_t)h->num_sms, (nodes + kDiagBlock - 1) / kDiagBlock);
}

// Pass 2: planes per thread, at most 32 and few enough for 6 blocks per SM. A
// run pays for the march's three loads ahead and for its block's FP64 sums once:
// records of D3Q27xD3Q19 at 128^3 98 us (104 with runs for 8 blocks per SM), at
// 256^3 605 (614 with at most 16 planes), of D3Q19xD3Q7 at 384^3 1324 (1360).
dim3 gradient_grid(const lbm_ctx* h, int& planes)
{
    const int64_t bx = ((int64_t)h->p.nx * h->p.ny + kDiagBlock - 1) / kDiagBlock;
    planes = (int)std::min<int64_t>(32, std::max<int64_t>(1, bx * h->p.nz / (6 * (int64_t)h->num_sms)));
    return dim3((unsigned)bx, (unsigned)((h->p.nz + planes - 1) / planes));
}

// Diagnostics scratch: FP32 fields for pass 2, pass-1 partials (at least
// `rows` rows), pass-2 rows, the totals in pinned memory and their event.
int ensure_diag(lbm_ctx* h, int rows)
{
    if (!h->diag_event) {   // the handle gets all of it or, where a part fails, nothing
        int planes = 0;
        const dim3 g = gradient_grid(h, planes);
        const size_t sums = (size_t)g.x * g.y * kDiagPass2;
        float* fields = nullptr;
        double* grad = nullptr;
        double* host = nullptr;
        cudaEvent_t event = nullptr;
        if (cudaMalloc(&fields, 4 * (size_t)h->geo.n3 * sizeof(float)) != cudaSuccess ||
            cudaMalloc(&grad, (sums + 1) * sizeof(double)) != cudaSuccess ||
            cudaMemsetAsync(grad + sums, 0, sizeof(double), h->stream) != cudaSuccess ||
            cudaMallocHost(&host, 16 * sizeof(double)) != cudaSuccess ||
            cudaEventCreateWithFlags(&event, cudaEventDisableTiming) != cudaSuccess) {
            cudaGetLastError();
            if (fields) cudaFree(fields);
            if (grad) cudaFree(grad);
            if (host) cudaFreeHost(host);
            return fail(LBM_ENOMEM, "diagnostics scratch allocation failed");
        }
        h->diag_fields = fields;
        h->diag_grad = grad;
        h->diag_host = host;
        h->diag_event = event;
    }
    if (h->diag_rows < rows) {
        if (h->diag_partials) {
            cudaStreamSynchronize(h->stream);
            cudaFree(h->diag_partials);
            h->diag_partials = nullptr;
            h->diag_rows = 0;
        }
        if (cudaMalloc(&h->diag_partials, (size_t)rows * kDNumSlots * sizeof(double)) != cudaSuccess) {
            cudaGetLastError();
            return fail(LBM_ENOMEM, "diagnostics partials allocation failed");
        }
        h->diag_rows = rows;
    }
    return LBM_OK;
}

// DiagArgs of the current state (scales of Eqs. 22-26 from the parameters).
DiagArgs diag_args(lbm_ctx* h)
{
    const lbm_params& p = h->p;
    const double cs2f = cs2_of(h->q.qf), cs2g = cs2_of(h->q.qg);
    const double gn2 = (p.beta != 0.0) ? (-p.G * p.rho0 / p.beta) : 1.0;
    const double nu = cs2f * (p.tau_f - 0.5), D = cs2g * (p.tau_g - 0.5);
    DiagArgs a;
    a.f = f_ptr(h);
    a.g = g_ptr(h);
    a.geo = h->geo;
    a.ph = h->ph;
    a.odd = h->odd;
    a.ep_scale = (float)(0.5 * gn2 / (p.rho0 * p.rho0));
    a.epsk_scale = (float)(2.0 * nu);
    a.s_scale = (float)(-1.0 / (2.0 * cs2f * p.tau_f));
    a.epsp_scale = (float)(D * gn2 / (p.rho0 * p.rho0));
    a.nu = (float)nu;
    a.fields = h->diag_fields;
    a.partials = h->diag_partials;
    const uint32_t plane = (uint32_t)p.nx * (uint32_t)p.ny;
    a.idx0 = h->slab ? plane : 0u;
    a.idx1 = h->slab ? h->geo.n3 - plane : h->geo.n3;
    a.rows = 0;
    const dim3 g = gradient_grid(h, a.planes);
    a.grad_rows = h->diag_grad;
    a.finished = reinterpret_cast<unsigned*>(h->diag_grad + (size_t)g.x * g.y * kDiagPass2);
    a.out = h->diag_host;
    return a;
}

// Nodes the diagnostics cover: every node, or a z-slab's own planes.
double owned_nodes(const lbm_ctx* h)
{
    const double plane = (double)h->p.nx * (double)h->p.ny;
    return h->slab ? (double)h->geo.n3 - 2.0 * plane : (double)h->geo.n3;
}

// The paper-unit block of a record (Section 2.4: U = L = 1, so one
// convective time is L / U0 steps): t = step U0 / L, energies / U0^2,
// dissipation rates * L / U0^3; NaN without a positive U0 and L.
void fill_phys(const lbm_params& p, lbm_diag* out)
{
    const bool ok = p.U0 > 0.0 && p.L > 0.0 && std::isfinite(p.U0) && std::isfinite(p.L);
    const double nan = std::numeric_limits<double>::quiet_NaN();
    const double e = ok ? 1.0 / (p.U0 * p.U0) : nan;
    const double r = ok ? p.L / (p.U0 * p.U0 * p.U0) : nan;
    out->t = ok ? (double)out->step * p.U0 / p.L : nan;
    out->Ek_phys = out->Ek * e;
    out->Ep_phys = out->Ep * e;
    out->eps_k_phys = out->eps_k * r;
    out->eps_p_phys = out->eps_p * r;
    out->eps_k_curl_phys = out->eps_k_curl * r;
}

// Totals (diag_host) -> lbm_diag of the state at `step`.
int fill_diag(const lbm_ctx* h, int64_t step, lbm_diag* out)
{
    const double* s = h->diag_host;
    const double nodes = owned_nodes(h);
    const double inv = 1.0 / nodes;
    const double nan = std::numeric_limits<double>::quiet_NaN();
    out->Ek = s[kDEk] * inv;
    out->Ep = s[kDEp] * inv;
    out->eps_k = s[kDEpsK] * inv;
    // a z-slab has no neighbour fields for the central differences
    out->eps_p = h->slab ? nan : s[kDEpsP] * inv;
    out->eps_k_curl = h->slab ? nan : s[kDEpsKCurl] * inv;
    out->mass_f = nodes + s[kDDrho];
    out->mass_g = nodes * h->p.rho0 + s[kDA];
    out->mom[0] = s[kDJx];
    out->mom[1] = s[kDJy];
    out->mom[2] = s[kDJz];
    out->umax = s[kDUmax];
    out->step = step;
    fill_phys(h->p, out);
    const int checked = h->slab ? kDiagPass1 : kDNumSlots;
    for (int q = 0; q < checked; ++q)
        if (!std::isfinite(s[q])) return fail(LBM_ENONFINITE, "non-finite diagnostics at step %lld", (long long)step);
    return LBM_OK;
}

cudaError_t launch_staged(lbm_ctx* h, int odd, int W, cudaStream_t s)
{
    const void* k = h->ks->staged[h->p.forcing][odd];
    const size_t smem = stage_smem_bytes(h->q.qf + h->q.qg, W);
    StageArgs a{};
    a.f = f_ptr(h);
    a.g = g_ptr(h);
    a.geo = h->geo;
    a.ph = h->ph;
    a.W = W;
    a.ntx = h->p.nx / W;
    a.ntiles = (uint32_t)a.ntx * (uint32_t)h->p.ny * (uint32_t)h->p.nz;
    a.err = h->d_err;
    a.spin_limit = h->stage_spin;
    a.extra_tx = h->stage_extra_tx;
    if (h->stage_grid == 0) {
        cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e == cudaSuccess) e = cudaFuncSetAttribute(h->ks->staged[h->p.forcing][odd ^ 1],
                                                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        int occ = 0;
        if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k, stage_threads(W), smem);
        if (e != cudaSuccess) return e;
        if (occ < 1) return cudaErrorInvalidConfiguration;
        const size_t cap = (size_t)h->num_sms * (size_t)occ;
        h->stage_grid = (int)(a.ntiles < cap ? a.ntiles : cap);
    }
    h->stage_used = true;
    ++h->launches;
    void* args[] = {&a};
    return cudaLaunchKernel(k, dim3((unsigned)h->stage_grid), dim3((unsigned)stage_threads(W)), args, smem, s);
}

// A box of planes and rows of the lattice (round the periodic ends), and the
// order of its planes.
struct StepRange {
    int z0, planes, y0, rows, down;
};
StepRange whole_range(const lbm_ctx* h)
{
    // a z-slab updates its own planes 1 .. nz - 2; the ghost planes are only
    // read and written by the boundary planes' odd steps (never wrapped)
    if (h->slab) return StepRange{1, h->p.nz - 2, 0, h->p.ny, 0};
    return StepRange{0, h->p.nz, 0, h->p.ny, 0};
}

dim3 step_grid(const lbm_ctx* h, int odd, const StepRange& r)
{
    const int xunits = uses_pairs(h, odd) ? h->p.nx / 2 : h->p.nx;
    const dim3 b = step_block(h, odd);
    if (h->flat[odd])
        return dim3((unsigned)(((int64_t)xunits * r.rows + b.x - 1) / b.x), 1u, (unsigned)r.planes);
    return dim3((unsigned)((xunits + (int)b.x - 1) / (int)b.x), (unsigned)((r.rows + (int)b.y - 1) / (int)b.y),
                (unsigned)r.planes);
}

StepArgs step_args(lbm_ctx* h, int odd, const StepRange& r)
{
    StepArgs a{};
    a.f = f_ptr(h);
    a.g = g_ptr(h);
    a.geo = h->geo;
    a.ph = h->ph;
    a.z0 = r.z0;
    a.y0 = r.y0;
    a.rows = r.rows;
    a.down = r.down;
    if (h->flat[odd]) {
        // ceil(2^(31 + s) / row) with 2^s >= row divides exactly below 2^31
        a.flat_row = (uint32_t)(uses_pairs(h, odd) ? h->p.nx / 2 : h->p.nx);
        a.flat = a.flat_row * (uint32_t)r.rows;
        uint32_t sh = 1;
        while ((1ull << sh) < a.flat_row) ++sh;
        a.flat_mul = (uint32_t)(((1ull << (31 + sh)) + a.flat_row - 1) / a.flat_row);
        a.flat_shift = sh - 1;
    }
    return a;
}

cudaError_t launch_range(lbm_ctx* h, int odd, const StepRange& r, cudaStream_t s)
{
    StepArgs a = step_args(h, odd, r);
    ++h->launches;
    void* args[] = {&a};
    const int flat = h->flat[odd] ? 1 : 0;
    const void* k = uses_pairs(h, odd) ? h->ks->step2[h->p.forcing][odd][flat] : h->ks->step[h->p.forcing][odd][flat];
    return launch_overlapped(k, step_grid(h, odd, r), step_block(h, odd), args, s, overlaps_steps(h));
}

cudaError_t launch_step(lbm_ctx* h, int odd, cudaStream_t s)
{
    const int W = stage_width(h);
    if (W > 0) return launch_staged(h, odd, W, s);
    StepRange r = whole_range(h);
    // of a lattice that L2 does not hold well a step starts where the one before
    // ended, in what is there; a smaller one keeps its blocks on their SMs. One
    // way / alternating, us per step of FP32 27x19 Guo: 32^3 (0.05 L2) 3.38 / 3.50,
    // 44^3 5.80 / 5.89, 56^3 8.90 / 8.98, 64^3 (0.36) 11.94 / 11.95, 72^3 (0.51)
    // 16.49 either way, 80^3 (0.70) 25.6 / 23.2; 19x7 32^3 2.17 / 2.31, 64^3 7.18 /
    // 7.21
    r.down = odd && 2 * store_need(h) > h->l2_bytes;
    return launch_range(h, odd, r, s);
}

// Skewed stepping of a lattice larger than L2. A step of the whole lattice
// moves every population through HBM; here a strip (some planes and rows, that
// L2 holds) runs `depth` steps before the next strip starts, so that a
// population crosses HBM about once in `depth` steps and the strip's launches
// work from L2. Step s of a node needs step s - 1 of its neighbours and nothing
// else (in the AA pattern a node's step reads and writes locations of its own),
// so a strip's range moves down by one plane and one row a step, into what the
// strips before it have left one step behind; along each axis the first strip
// shrinks by one at both ends and the last takes what it left, round the
// periodic end. The launches are the plain step kernels in stream order: the
// same operations on the same values. A strip is swept back and forth and every
// other group of steps runs mirrored, so that a launch starts where the one
// before it ended, in what L2 holds.
//
// us per step, whole lattice swept one way (the form before) / back and forth /
// skewed in strips of about 3/4 of L2: D3Q27xD3Q19 FP32 96^3 50.4 / 43.0 / 40.8,
// 128^3 115.4 / 107.0 / 97.6, 192^3 384 / 379 / 364, 256^3 905 / 897 / 824-829,
// 512^3 7124 / - / 6653; D3Q19xD3Q7 FP32 256^3 516 / 510 / 455; D3Q27xD3Q19 FP16
// 128^3 60.0 / 54.1 / 53.0, 256^3 451.5 / 446.8 / 446. From L2 a step runs at 20
// to 22 G nodes/s FP32, 37 to 39 FP16, two thirds of the issue slots busy.
struct SkewPlan {
    int jz, jy, depth;   // strips along z and y, steps per strip; depth 1: whole-lattice steps
};

constexpr int kSkewDepth = 16;   // deeper gains under 0.3 %, and the ranges move further
constexpr int kSkewSteps = 4;    // fewer steps in a call run whole

// Strips of at most 3/4 or 0.4 of L2 in FP32. Alone on the GPU the larger ones
// are the faster, beside another lattice stepped on its own stream, which then
// shares L2, the smaller: 50 steps and a record at 128^3 in strips of 0.4 / 0.75
// of L2 5.13 / 4.98 ms alone and 5.29 / 5.61 beside another (whole-lattice steps
// 5.44 and 5.60), 100 at 256^3 88.5 / 82.9 alone and 84.9 / 88.5 beside (89.5 and
// 90.1), at 160^3 as good either way. Which it is, a handle does not know (but for
// an instance with a round of its batch to itself): lattices of up to 6 L2 take
// the smaller strips, of which several are likelier to be stepped at a time, and
// no faster choice was measured between 160^3 and 256^3. One L2 in 16 bits,
// where only deep strips gain (256^3 in 96 / 129 MB strips 449.7 / 446.4 us per
// step). Along z alone while the strips are 16 planes thick, else about square
// in y and z.
SkewPlan skew_plan(const lbm_ctx* h)
{
    const SkewPlan whole{1, 1, 1};
    const double bytes = (double)store_need(h);
    const double l2 = (double)h->l2_bytes;
    const double strip = h->p.storage != LBM_FP32 ? l2 : bytes > 6.0 * l2 || h->l2 == L2Use::alone ? 0.75 * l2 : 0.4 * l2;
    // (72^3 FP32 D3Q27xD3Q19, 69 MB: whole steps 16.4 us from L2)
    if (strip <= 0.0 || bytes <= std::max(strip, 0.75 * l2) || h->slab || stage_width(h) > 0) return whole;
    // 16 bits with one node per thread (odd nx) are bound by issue: strips' last
    // waves cost more than HBM traffic saves (27x19 FP16 171^3 167 against 176 us
    // whole, 225^3 480 against 470, 401^3 2740 against 2641)
    if (h->p.storage != LBM_FP32 && !uses_pairs(h, 0) && bytes > 6.0 * l2) return whole;
    const int nz = h->p.nz, ny = h->p.ny;
    const int64_t want = (int64_t)std::ceil(bytes / strip);
    SkewPlan p{1, 1, kSkewDepth};
    if (want <= nz / kSkewDepth) {
        p.jz = (int)want;
    } else {
        const double side = std::sqrt((double)want * nz / ny);
        p.jz = (int)std::min<double>(std::max(1.0, std::round(side)), std::max(1, nz / kSkewDepth));
        p.jy = (int)std::min<int64_t>((want + p.jz - 1) / p.jz, std::max(1, ny / kSkewDepth));
    }
    // a box too flat for strips that L2 holds, or for two of them
    if (p.jz * p.jy == 1 || (int64_t)p.jz * p.jy * 2 < want) return whole;
    return p;
}

// Range of strip j of `strips` along an axis of n, at step l of a group of k
// (n / strips >= k, or one strip).
void skewed_range(int n, int strips, int j, int k, int l, bool mirrored, int& first, int& count)
{
    auto cut = [&](int i) { return (int)((int64_t)i * n / strips) + k - 1; };
    first = 0;
    count = n;
    if (strips > 1) {
        first = j == 0 ? l : cut(j) - l;
        count = (j == strips - 1 ? n + l : cut(j + 1) - l) - first;
        if (first >= n) first -= n;
    }
    if (mirrored) first = (2 * n - first - count) % n;
}

// One group of k steps from AA parity `odd`.
cudaError_t launch_group(lbm_ctx* h, const SkewPlan& p, int k, int odd, bool mirrored, cudaStream_t s)
{
    for (int z = 0; z < p.jz; ++z)
        for (int y = 0; y < p.jy; ++y)
            for (int l = 0; l < k; ++l) {
                StepRange r{};
                skewed_range(h->p.nz, p.jz, z, k, l, mirrored, r.z0, r.planes);
                skewed_range(h->p.ny, p.jy, y, k, l, mirrored, r.y0, r.rows);
                r.down = (int)mirrored ^ (l & 1);
                const cudaError_t e = launch_range(h, odd ^ (l & 1), r, s);
                if (e != cudaSuccess) return e;
            }
    return cudaSuccess;
}

// Captures `record` on the stream and instantiates it; null where the stream
// cannot be captured (the caller then launches eagerly). `launches` gets the
// number of its kernels.
template <class Record>
cudaGraphExec_t capture_graph(lbm_ctx* h, cudaStream_t s, int64_t* launches, Record&& record)
{
    const int64_t before = h->launches;
    cudaGraph_t g = nullptr;
    cudaGraphExec_t x = nullptr;
    cudaError_t e = cudaStreamBeginCapture(s, cudaStreamCaptureModeThreadLocal);
    if (e == cudaSuccess) {
        e = record();
        const cudaError_t e2 = cudaStreamEndCapture(s, &g);
        if (e == cudaSuccess) e = e2;
    }
    if (e == cudaSuccess) e = cudaGraphInstantiate(&x, g, 0);
    if (g) cudaGraphDestroy(g);
    *launches = h->launches - before;
    h->launches = before;
    if (e == cudaSuccess) return x;
    cudaGetLastError();
    return nullptr;
}

// A lattice stepped in strips takes 10 to 250 launches a step. Two groups, one
// mirrored, make a graph, so that a long call does not fill the launch queue
// and wait in it; it is built once as many steps as kSkewGraphAfter such pairs
// have run (256^3: 1152 nodes, a few ms), before that and beside it groups are
// launched one by one, which keeps ahead of kernels of 14 to 25 us.
constexpr int kSkewGraphSteps = 2 * kSkewDepth;
constexpr int kSkewGraphAfter = 4;

cudaError_t step_skewed(lbm_ctx* h, const SkewPlan& p, int64_t nsteps, cudaStream_t s)
{
    while (nsteps > 0) {
        const bool graphs = h->graphs && s != nullptr && nsteps >= kSkewGraphSteps &&
                            h->skew_eager >= kSkewGraphAfter * kSkewGraphSteps;
        if (graphs && h->odd == 0) {
            if (!h->skew_graph)
                h->skew_graph = capture_graph(h, s, &h->skew_launches, [&] {
                    const cudaError_t e = launch_group(h, p, kSkewDepth, 0, true, s);
                    return e != cudaSuccess ? e : launch_group(h, p, kSkewDepth, 0, false, s);
                });
            if (h->skew_graph) {
                const cudaError_t e = cudaGraphLaunch(h->skew_graph, s);
                if (e != cudaSuccess) return e;
                h->mirrored = false;
                h->launches += h->skew_launches;
                h->step += kSkewGraphSteps;
                nsteps -= kSkewGraphSteps;
                continue;
            }
            h->graphs = false;
        }
        // an odd group brings the natural layout that the graph starts from;
        // else the steps left are dealt to groups of about equal length
        const int64_t groups = (nsteps + p.depth - 1) / p.depth;
        const int k = graphs && h->odd ? kSkewDepth - 1 : (int)((nsteps + groups - 1) / groups);
        h->mirrored = !h->mirrored;
        const cudaError_t e = launch_group(h, p, k, h->odd, h->mirrored, s);
        if (e != cudaSuccess) return e;
        h->odd ^= k & 1;
        h->step += k;
        h->skew_eager = std::min(h->skew_eager + k, kSkewGraphAfter * kSkewGraphSteps);
        nsteps -= k;
    }
    return cudaSuccess;
}

// What follows pass 1, whose `rows` rows are in h->diag_partials: more than
// kDirectRows of them are first added up on every SM (into the rows behind
// them), then pass 2 totals what is left beside its own sums; a z-slab has no
// pass 2.
constexpr int kDirectRows = 1024;
cudaError_t launch_totals(lbm_ctx* h, DiagArgs a, int rows)
{
    double* at = h->diag_partials;
    double* mid = at + (size_t)rows * kDNumSlots;
    cudaError_t e = cudaSuccess;
    if (rows > kDirectRows) {
        void* args[] = {&at, &rows, &mid};
        e = launch_overlapped(diag_rows_kernel(), dim3((unsigned)h->num_sms), dim3(kDiagBlock), args, h->stream);
        if (e != cudaSuccess) return e;
        ++h->launches;
        at = mid;
        rows = h->num_sms;
    }
    ++h->launches;
    if (h->slab) {
        void* args[] = {&at, &rows, &a.out};
        return launch_overlapped(diag_totals_kernel(), dim3(kDiagPass1), dim3(kDiagBlock), args, h->stream);
    }
    a.partials = at;
    a.rows = rows;
    dim3 grid = gradient_grid(h, a.planes);
    grid.y += (kDiagPass1 + grid.x - 1) / grid.x;   // the blocks that total the pass-1 slots
    void* args[] = {&a};
    return launch_overlapped(diag_gradients_kernel(), grid, dim3(kDiagBlock), args, h->stream);
}

// Pass 1 and what follows it, for the current state.
int enqueue_diagnostics(lbm_ctx* h)
{
    const uint32_t blocks = moment_blocks(h, (uint32_t)owned_nodes(h));
    if (int rc = ensure_diag(h, (int)blocks + h->num_sms)) return rc;
    DiagArgs a = diag_args(h);
    void* args[] = {&a};
    LBM_CUDA(cudaLaunchKernel(h->ks->diag_moments, dim3(blocks), dim3(kDiagBlock), args, 0, h->stream), "diag pass 1");
    ++h->launches;
    LBM_CUDA(launch_totals(h, a, (int)blocks), "diag pass 2");
    return LBM_OK;
}

// One 256-thread block per 256 nodes.
dim3 node_grid(const lbm_ctx* h) { return dim3((h->geo.n3 + 255u) / 256u); }

int flat_grid(const lbm_ctx* h)
{
    size_t blocks = ((size_t)h->geo.n3 + 255) / 256;
    size_t cap = (size_t)h->num_sms * 16;
    return (int)(blocks < cap ? blocks : cap);
}

int check_handle(lbm_ctx* h)
{
    if (!h) return fail(LBM_EINVAL, "null handle");
    cudaError_t e = cudaSetDevice(h->device);
    if (e != cudaSuccess) return cuda_fail(e, "cudaSetDevice");
    return LBM_OK;
}

int validate_params(const lbm_params* p, PairInfo* q)
{
    if (!p) return fail(LBM_EINVAL, "null parameters");
    if (p->nx < 1 || p->ny < 1 || p->nz < 1) return fail(LBM_EINVAL, "lattice sizes must be >= 1");
    size_t n3 = (size_t)p->nx * p->ny * p->nz;
    if (n3 > 0x7fffffffull) return fail(LBM_EINVAL, "nx*ny*nz = %zu exceeds 2^31 - 1 nodes", n3);
    if (p->nz > 65535) return fail(LBM_EINVAL, "nz must be <= 65535");
    if (!pair_info(p->pair, q)) return fail(LBM_EINVAL, "unknown stencil pair %d", p->pair);
    if ((size_t)(q->qf > q->qg ? q->qf : q->qg) * n3 > 0xffffffffull)
        return fail(LBM_EINVAL, "Q * nx*ny*nz = %zu exceeds the 32-bit element offsets of the store",
                    (size_t)(q->qf > q->qg ? q->qf : q->qg) * n3);
    if (p->forcing < 0 || p->forcing > 3) return fail(LBM_EINVAL, "unknown forcing scheme %d", p->forcing);
    if (p->storage < 0 || p->storage > 2) return fail(LBM_EINVAL, "unknown storage %d", p->storage);
    if (p->scalar_mode < 0 || p->scalar_mode > 1) return fail(LBM_EINVAL, "unknown scalar mode %d", p->scalar_mode);
    if (!(p->tau_f > 0.5) || !(p->tau_g > 0.5) || !std::isfinite(p->tau_f) || !std::isfinite(p->tau_g))
        return fail(LBM_EINVAL, "relaxation times must be finite and > 1/2 (tau_f=%g, tau_g=%g)", p->tau_f,
                    p->tau_g);
    if (!std::isfinite(p->G) || !std::isfinite(p->beta) || !std::isfinite(p->rho0) || !std::isfinite(p->sc_shift))
        return fail(LBM_EINVAL, "non-finite physical parameter");
    return LBM_OK;
}

int after_init(lbm_ctx* h)
{
    h->initialized = true;
    h->step = 0;
    h->odd = 0;
    return LBM_OK;
}

// Slots of velocity set q (this library's order) whose e_z equals sign,
// into slots[] (may be null); returns their number.
int halo_slots(int q, int sign, int* slots)
{
    auto pick = [&](auto lat) {
        using L = decltype(lat);
        int n = 0;
        for (int i = 0; i < L::kQ; ++i)
            if (L::ez(i) == sign) {
                if (slots) slots[n] = i;
                ++n;
            }
        return n;
    };
    switch (q) {
    case 7: return pick(Lattice<7>{});
    case 15: return pick(Lattice<15>{});
    case 19: return pick(Lattice<19>{});
    default: return pick(Lattice<27>{});
    }
}

// Whether [p, p + bytes) is allocated device memory as far as the driver tells.
// A range may span several mappings (a buffer in expandable memory).
bool device_range(const void* p, size_t bytes)
{
    using Query = CUresult (*)(CUdeviceptr*, size_t*, CUdeviceptr);
    static const Query query = [] {
        void* f = nullptr;
        cudaDriverEntryPointQueryResult found;
        const cudaError_t e =
            cudaGetDriverEntryPointByVersion("cuMemGetAddressRange", &f, 3020, cudaEnableDefault, &found);
        if (e != cudaSuccess || found != cudaDriverEntryPointSuccess) {
            cudaGetLastError();
            f = nullptr;
        }
        return reinterpret_cast<Query>(f);
    }();
    CUdeviceptr at = reinterpret_cast<CUdeviceptr>(p);
    for (bool first = true; bytes > 0; first = false) {
        CUdeviceptr base = 0;
        size_t size = 0;
        if (!query || query(&base, &size, at) != CUDA_SUCCESS) return first;   // memory without an extent of its own
        const size_t here = (size_t)(base + size - at);
        if (here == 0) return false;
        if (here >= bytes) return true;
        at += here;
        bytes -= here;
    }
    return true;
}

// LBM_OK if p is `bytes` of device memory on the handle's device. The halo
// kernel takes the buffers as they are, so their extent is looked at here.
int check_device_buffer(const lbm_ctx* h, const void* p, size_t bytes)
{
    cudaPointerAttributes attr;
    cudaError_t e = cudaPointerGetAttributes(&attr, p);
    if (e != cudaSuccess || attr.type != cudaMemoryTypeDevice || attr.device != h->device) {
        cudaGetLastError();
        return fail(LBM_EINVAL, "halo buffers must be device memory on the handle's device");
    }
    if (!device_range(p, bytes))
        return fail(LBM_EINVAL, "a halo buffer is shorter than the %zu bytes of lbm_halo_bytes", bytes);
    return LBM_OK;
}

// One side of a halo copy: plane z of the store's f slots with e_z = sign, then
// of its g slots with e_z = sign, nx*ny elements each (one contiguous run per
// slot and plane in the store). Returns the number of runs.
int halo_side(lbm_ctx* h, int z, int sign, const void* buf, HaloSide* out)
{
    const size_t es = elem_size(h->p.storage);
    const size_t plane = (size_t)h->p.nx * (size_t)h->p.ny * es;
    int slots[27];
    int runs = 0;
    for (int part = 0; part < 2; ++part) {
        const int q = part ? h->q.qg : h->q.qf;
        char* base = static_cast<char*>(part ? g_ptr(h) : f_ptr(h));
        const int n = halo_slots(q, sign, slots);
        for (int k = 0; k < n; ++k) out->run[runs++] = base + ((size_t)slots[k] * h->geo.n3) * es + (size_t)z * plane;
    }
    out->buffer = static_cast<char*>(const_cast<void*>(buf));
    return runs;
}

// Both halo buffers of a slab in one launch: `lower` holds the slots of sign
// `sl` at plane zl, `upper` those of sign su at zu. Buffers of a pack that
// overlap take one launch each, in order, so that the upper one's bytes stand.
int halo_copy(lbm_ctx* h, int zl, int sl, const void* lower, int zu, int su, const void* upper, bool pack)
{
    HaloArgs a{};
    a.plane = (size_t)h->p.nx * (size_t)h->p.ny * elem_size(h->p.storage);
    a.pack = pack ? 1 : 0;
    const int runs = halo_side(h, zl, sl, lower, &a.side[0]);
    halo_side(h, zu, su, upper, &a.side[1]);
    // the widest type that every address is a multiple of: the runs lie at
    // whole planes from the store's start (and the g part at whole elements)
    uintptr_t bits = (uintptr_t)a.plane;
    for (const HaloSide& s : a.side) {
        bits |= (uintptr_t)s.buffer;
        for (int k = 0; k < runs; ++k) bits |= (uintptr_t)s.run[k];
    }
    const int width = bits % 16 == 0 ? 16 : bits % 4 == 0 ? 4 : bits % 2 == 0 ? 2 : 1;
    const size_t n = a.plane / (size_t)width;
    const size_t want = (n + 4 * kHaloThreads - 1) / (4 * kHaloThreads);
    const unsigned bx = (unsigned)(want < 1024 ? want : 1024);
    const char* b0 = a.side[0].buffer;
    const char* b1 = a.side[1].buffer;
    const size_t bytes = (size_t)runs * a.plane;
    const bool overlap = pack && b0 < b1 + bytes && b1 < b0 + bytes;
    for (int launch = 0; launch < (overlap ? 2 : 1); ++launch) {
        if (launch) a.side[0] = a.side[1];
        void* args[] = {&a};
        LBM_CUDA(cudaLaunchKernel(halo_kernel(width), dim3(bx, (unsigned)runs, overlap ? 1u : 2u), dim3(kHaloThreads),
                                  args, 0, h->stream),
                 "halo copy");
    }
    return LBM_OK;
}

}  // namespace

extern "C" {

const char* lbm_last_error(void) { return g_last_error.c_str(); }

const char* lbm_version(void) { return "paper_2605_14505_gb300 lbm 0.1 (sm_103a)"; }

int lbm_velocity_set(int q, int* e, double* w, double* cs2)
{
    auto fill = [&](auto lat) {
        using L = decltype(lat);
        for (int i = 0; i < L::kQ; ++i) {
            if (e) {
                e[3 * i + 0] = L::ex(i);
                e[3 * i + 1] = L::ey(i);
                e[3 * i + 2] = L::ez(i);
            }
            if (w) w[i] = L::wd(i);
        }
        if (cs2) *cs2 = L::cs2d;
        return L::kQ;
    };
    switch (q) {
    case 7: return fill(Lattice<7>{});
    case 15: return fill(Lattice<15>{});
    case 19: return fill(Lattice<19>{});
    case 27: return fill(Lattice<27>{});
    default: return fail(LBM_EINVAL, "unknown velocity set Q%d", q);
    }
}

int lbm_params_from_physics(lbm_params* p, int nx, int ny, int nz, int pair, int forcing, double Re,
                            double Fr, double Pr, double U0)
{
    PairInfo q;
    if (!p) return fail(LBM_EINVAL, "null parameters");
    if (nx < 1 || ny < 1 || nz < 1) return fail(LBM_EINVAL, "lattice sizes must be >= 1");
    if (!pair_info(pair, &q)) return fail(LBM_EINVAL, "unknown stencil pair %d", pair);
    if (!(Re > 0) || !(Pr > 0) || !(U0 > 0) || !(Fr > 0) || std::isnan(Fr))
        return fail(LBM_EINVAL, "Re, Fr, Pr and U0 must be positive");
    std::memset(p, 0, sizeof(*p));
    const double two_pi = 6.283185307179586476925286766559;
    const double L = nx / two_pi;
    const double nu = U0 * L / Re;
    const double D = nu / Pr;
    const double N = std::isinf(Fr) ? 0.0 : U0 / (Fr * L);
    p->nx = nx;
    p->ny = ny;
    p->nz = nz;
    p->pair = pair;
    p->forcing = forcing;
    p->storage = LBM_FP32;
    p->scalar_mode = LBM_SCALAR_PRINTED;
    p->tau_f = nu / cs2_of(q.qf) + 0.5;
    p->tau_g = D / cs2_of(q.qg) + 0.5;
    p->rho0 = 1.0;
    p->G = N / 1024.0;
    p->beta = N > 0 ? -N * N * p->rho0 / p->G : 0.0;
    p->sc_shift = 1.0;
    p->U0 = U0;
    p->L = L;
    return LBM_OK;
}

int lbm_create_params(lbm_handle* out, const lbm_params* p)
{
    if (!out) return fail(LBM_EINVAL, "null output handle");
    *out = nullptr;
    PairInfo q;
    int rc = validate_params(p, &q);
    if (rc) return rc;
    const KernelSet* ks = kernel_set(p->pair, p->storage);
    if (!ks) return fail(LBM_EUNSUPPORTED, "stencil pair %d with storage %d is not compiled in", p->pair, p->storage);
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return cuda_fail(e, "cudaGetDevice");
    lbm_ctx* h = new (std::nothrow) lbm_ctx();
    if (!h) return fail(LBM_ENOMEM, "host allocation failed");
    h->p = *p;
    h->q = q;
    h->ks = ks;
    h->device = dev;
    cudaDeviceGetAttribute(&h->num_sms, cudaDevAttrMultiProcessorCount, dev);
    if (h->num_sms < 1) h->num_sms = 1;
    int l2 = 0;
    if (cudaDeviceGetAttribute(&l2, cudaDevAttrL2CacheSize, dev) == cudaSuccess && l2 > 0) h->l2_bytes = (size_t)l2;
    // a device reset ends every handle, so looking the scratch address up
    // again here keeps the cached one valid for every handle in use
    static_scratch_refresh(dev);
    derive_phys(h);
    default_block(h);
    e = cudaStreamCreateWithFlags(&h->stream, cudaStreamNonBlocking);
    if (e != cudaSuccess) {
        delete h;
        return cuda_fail(e, "cudaStreamCreate");
    }
    h->own_stream = true;
    if (cudaMalloc(&h->d_err, sizeof(int)) != cudaSuccess || cudaMemset(h->d_err, 0, sizeof(int)) != cudaSuccess) {
        cudaGetLastError();
        if (h->d_err) cudaFree(h->d_err);
        cudaStreamDestroy(h->stream);
        delete h;
        return fail(LBM_ENOMEM, "device error-flag allocation failed");
    }
    *out = h;
    return LBM_OK;
}

int lbm_create(lbm_handle* out, int nx, int ny, int nz, int pair, int forcing, double Re, double Fr, double Pr,
               double U0)
{
    lbm_params p;
    int rc = lbm_params_from_physics(&p, nx, ny, nz, pair, forcing, Re, Fr, Pr, U0);
    if (rc) return rc;
    return lbm_create_params(out, &p);
}

int lbm_get_params(lbm_handle h, lbm_params* p)
{
    if (!h || !p) return fail(LBM_EINVAL, "null argument");
    *p = h->p;
    return LBM_OK;
}

int lbm_set_storage(lbm_handle h, int storage)
{
    if (!h) return fail(LBM_EINVAL, "null handle");
    if (h->store) return fail(LBM_ESTATE, "storage can only change before the store exists");
    if (storage < 0 || storage > 2) return fail(LBM_EINVAL, "unknown storage %d", storage);
    const KernelSet* ks = kernel_set(h->p.pair, storage);
    if (!ks) return fail(LBM_EUNSUPPORTED, "storage %d is not compiled in for pair %d", storage, h->p.pair);
    h->p.storage = storage;
    h->ks = ks;
    h->stage_grid = 0;
    default_block(h);
    drop_graph(h);
    return LBM_OK;
}

int lbm_set_stream(lbm_handle h, void* stream)
{
    int rc = check_handle(h);
    if (rc) return rc;
    if (h->own_stream) {
        cudaStreamSynchronize(h->stream);
        cudaStreamDestroy(h->stream);
    }
    h->stream = static_cast<cudaStream_t>(stream);
    h->own_stream = false;
    return LBM_OK;
}

int lbm_get_stream(lbm_handle h, void** stream)
{
    if (!h || !stream) return fail(LBM_EINVAL, "null argument");
    *stream = h->stream;
    return LBM_OK;
}

int lbm_required_bytes(lbm_handle h, size_t* bytes)
{
    if (!h || !bytes) return fail(LBM_EINVAL, "null argument");
    *bytes = store_need(h);
    return LBM_OK;
}

int lbm_attach(lbm_handle h, void* device_ptr, size_t bytes)
{
    int rc = check_handle(h);
    if (rc) return rc;
    if (h->store) return fail(LBM_ESTATE, "a population store is already in place");
    size_t need;
    lbm_required_bytes(h, &need);
    if (!device_ptr) return fail(LBM_EINVAL, "null device pointer");
    if (bytes < need) return fail(LBM_EINVAL, "store of %zu bytes is smaller than the %zu required", bytes, need);
    if (reinterpret_cast<uintptr_t>(device_ptr) % 256 != 0) return fail(LBM_EINVAL, "store must be 256-byte aligned");
    cudaPointerAttributes attr;
    cudaError_t e = cudaPointerGetAttributes(&attr, device_ptr);
    if (e != cudaSuccess || attr.type != cudaMemoryTypeDevice || attr.device != h->device) {
        cudaGetLastError();
        return fail(LBM_EINVAL, "store must be device memory on the handle's device");
    }
    h->store = device_ptr;
    h->store_bytes = bytes;
    h->own_store = false;
    return LBM_OK;
}

int lbm_init_tgv(lbm_handle h, uint64_t seed, double noise_amp)
{
    int rc = check_handle(h);
    if (rc) return rc;
    if (h->slab) return fail(LBM_EINVAL, "a z-slab is initialised from the global field's planes (lbm_init_fields "
                                         "or lbm_set_populations), not by lbm_init_tgv");
    if (h->p.nx != h->p.ny || h->p.nx != h->p.nz) return fail(LBM_EINVAL, "the Taylor-Green box needs nx = ny = nz");
    if (!std::isfinite(noise_amp)) return fail(LBM_EINVAL, "non-finite noise amplitude");
    if ((rc = ensure_store(h))) return rc;
    // sin and cos of x_i = 2 pi i / n for the kernel, in the staging buffer
    const int n = h->p.nx;
    std::vector<double> trig(2 * (size_t)n);
    for (int i = 0; i < n; ++i) {
        const double x = 6.283185307179586476925286766559 * i / n;
        trig[i] = std::sin(x);
        trig[n + i] = std::cos(x);
    }
    if ((rc = ensure_staging(h, trig.size() * sizeof(double)))) return rc;
    LBM_CUDA(cudaMemcpyAsync(h->staging, trig.data(), trig.size() * sizeof(double), cudaMemcpyHostToDevice, h->stream),
             "copy trig table");
    LBM_CUDA(cudaEventRecord(h->copy_event, h->stream), "init_tgv event");
    TgvArgs a;
    a.f = f_ptr(h);
    a.g = g_ptr(h);
    a.geo = h->geo;
    a.trig = h->staging;
    a.U0 = h->p.U0;
    a.noise = noise_amp;
    a.seed = seed;
    a.rho0 = h->p.rho0;
    void* args[] = {&a};
    LBM_CUDA(cudaLaunchKernel(h->ks->init_tgv, dim3(flat_grid(h)), dim3(256), args, 0, h->stream), "init_tgv launch");
    LBM_CUDA(cudaEventSynchronize(h->copy_event), "init_tgv");   // the table's host copy may go
    return after_init(h);
}

int lbm_init_fields(lbm_handle h, const double* rho, const double* u, const double* rho_p, const double* xi_f,
                    const double* xi_g, double amp)
{
    int rc = check_handle(h);
    if (rc) return rc;
    if (!rho || !u || !rho_p) return fail(LBM_EINVAL, "rho, u and rho_p are required");
    if ((rc = ensure_store(h))) return rc;
    const size_t n3 = h->geo.n3;
    size_t ndoubles = 5 * n3 + (xi_f ? 27 * n3 : 0) + (xi_g ? 27 * n3 : 0);
    if ((rc = ensure_staging(h, ndoubles * sizeof(double)))) return rc;
    double* d = h->staging;
    LBM_CUDA(cudaMemcpyAsync(d, rho, n3 * sizeof(double), cudaMemcpyHostToDevice, h->stream), "copy rho");
    LBM_CUDA(cudaMemcpyAsync(d + n3, u, 3 * n3 * sizeof(double), cudaMemcpyHostToDevice, h->stream), "copy u");
    LBM_CUDA(cudaMemcpyAsync(d + 4 * n3, rho_p, n3 * sizeof(double), cudaMemcpyHostToDevice, h->stream), "copy rho_p");
    double* dxf = nullptr;
    double* dxg = nullptr;
    size_t off = 5 * n3;
    if (xi_f) {
        dxf = d + off;
        off += 27 * n3;
        LBM_CUDA(cudaMemcpyAsync(dxf, xi_f, 27 * n3 * sizeof(double), cudaMemcpyHostToDevice, h->stream), "copy xi_f");
    }
    if (xi_g) {
        dxg = d + off;
        LBM_CUDA(cudaMemcpyAsync(dxg, xi_g, 27 * n3 * sizeof(double), cudaMemcpyHostToDevice, h->stream), "copy xi_g");
    }
    InitArgs a;
    a.f = f_ptr(h);
    a.g = g_ptr(h);
    a.geo = h->geo;
    a.rho = d;
    a.u = d + n3;
    a.rho_p = d + 4 * n3;
    a.xi_f = dxf;
    a.xi_g = dxg;
    a.amp_f = (float)amp;
    a.rho0 = h->p.rho0;
    void* args[] = {&a};
    // the host arrays may be reused once the copies are done; the
    // initialisation itself completes in stream order
    LBM_CUDA(cudaEventRecord(h->copy_event, h->stream), "init_fields event");
    LBM_CUDA(cudaLaunchKernel(h->ks->init_fields, dim3(flat_grid(h)), dim3(256), args, 0, h->stream),
             "init_fields launch");
    LBM_CUDA(cudaEventSynchronize(h->copy_event), "init_fields");
    return after_init(h);
}

int lbm_prefetch_fields(lbm_handle h, const double* rho, const double* u, const double* rho_p)
{
    int rc = check_handle(h);
    if (rc) return rc;
    if (!rho || !u || !rho_p) return fail(LBM_EINVAL, "rho, u and rho_p are required");
    if (h->pre_ready >= 0) return fail(LBM_ESTATE, "a prefetch is already waiting for lbm_init_prefetched");
    const size_t n3 = h->geo.n3;
    if (!h->copy_stream) {
        if (cudaStreamCreateWithFlags(&h->copy_stream, cudaStreamNonBlocking) != cudaSuccess) {
            cudaGetLastError();
            return fail(LBM_ECUDA, "copy stream creation failed");
        }
        for (int b = 0; b < 2; ++b) {
            if (cudaEventCreateWithFlags(&h->pre_done[b], cudaEventDisableTiming) != cudaSuccess ||
                cudaEventCreateWithFlags(&h->pre_free[b], cudaEventDisableTiming) != cudaSuccess ||
                cudaMalloc(&h->pre[b], 5 * n3 * sizeof(double)) != cudaSuccess) {
                cudaGetLastError();
                return fail(LBM_ENOMEM, "prefetch buffer allocation failed");
            }
        }
    }
    const int b = h->pre_next;
    if (h->pre_free_recorded[b])
        LBM_CUDA(cudaStreamWaitEvent(h->copy_stream, h->pre_free[b], 0), "prefetch wait");
    double* d = h->pre[b];
    LBM_CUDA(cudaMemcpyAsync(d, rho, n3 * sizeof(double), cudaMemcpyHostToDevice, h->copy_stream), "prefetch rho");
    LBM_CUDA(cudaMemcpyAsync(d + n3, u, 3 * n3 * sizeof(double), cudaMemcpyHostToDevice, h->copy_stream), "prefetch u");
    LBM_CUDA(cudaMemcpyAsync(d + 4 * n3, rho_p, n3 * sizeof(double), cudaMemcpyHostToDevice, h->copy_stream),
             "prefetch rho_p");
    LBM_CUDA(cudaEventRecord(h->pre_done[b], h->copy_stream), "prefetch event");
    h->pre_ready = b;
    h->pre_next = b ^ 1;
    return LBM_OK;
}

int lbm_init_prefetched(lbm_handle h)
{
    int rc = check_handle(h);
    if (rc) return rc;
    if (h->pre_ready < 0) return fail(LBM_ESTATE, "lbm_init_prefetched without a prefetch");
    if ((rc = ensure_store(h))) return rc;
    const int b = h->pre_ready;
    const size_t n3 = h->geo.n3;
    LBM_CUDA(cudaStreamWaitEvent(h->stream, h->pre_done[b], 0), "init wait");
    InitArgs a{};
    a.f = f_ptr(h);
    a.g = g_ptr(h);
    a.geo = h->geo;
    a.rho = h->pre[b];
    a.u = h->pre[b] + n3;
    a.rho_p = h->pre[b] + 4 * n3;
    a.rho0 = h->p.rho0;
    void* args[] = {&a};
    LBM_CUDA(cudaLaunchKernel(h->ks->init_fields, dim3(flat_grid(h)), dim3(256), args, 0, h->stream),
             "init_prefetched launch");
    LBM_CUDA(cudaEventRecord(h->pre_free[b], h->stream), "init event");
    h->pre_free_recorded[b] = true;
    h->pre_ready = -1;
    // the caller's host arrays of this prefetch may be reused from here on
    LBM_CUDA(cudaEventSynchronize(h->pre_done[b]), "prefetch copies");
    return after_init(h);
}

int lbm_step(lbm_handle h, int64_t nsteps)
{
    int rc = check_handle(h);
    if (rc) return rc;
    if (nsteps < 0) return fail(LBM_EINVAL, "negative step count");
    if (!h->initialized) return fail(LBM_ESTATE, "lbm_step before initialisation");
    if (nsteps >= kSkewSteps && h->l2 != L2Use::shared) {
        const SkewPlan plan = skew_plan(h);
        if (plan.depth > 1) {
            LBM_CUDA(step_skewed(h, plan, nsteps, h->stream), "step launch");
            return LBM_OK;
        }
    }
    while (nsteps > 0) {
        if (h->graphs && h->stream != nullptr && h->odd == 0 && nsteps >= kGraphSteps) {
            if (!h->graph)
                h->graph = capture_graph(h, h->stream, &h->graph_launches, [&] {
                    cudaError_t e = cudaSuccess;
                    for (int s = 0; s < kGraphSteps && e == cudaSuccess; ++s) e = launch_step(h, s & 1, h->stream);
                    return e;
                });
            if (!h->graph) {
                h->graphs = false;  // fall back to eager launches
                continue;
            }
            LBM_CUDA(cudaGraphLaunch(h->graph, h->stream), "graph launch");
            h->launches += h->graph_launches;
            h->step += kGraphSteps;
            nsteps -= kGraphSteps;
            continue;
        }
        LBM_CUDA(launch_step(h, h->odd, h->stream), "step launch");
        h->odd ^= 1;
        h->step += 1;
        nsteps -= 1;
    }
    return LBM_OK;
}

int lbm_synchronize(lbm_handle h)
{
    int rc = check_handle(h);
    if (rc) return rc;
    LBM_CUDA(cudaStreamSynchronize(h->stream), "stream synchronize");
    if (h->copy_stream) LBM_CUDA(cudaStreamSynchronize(h->copy_stream), "copy stream synchronize");
    // only the staged kernel raises the flag: other handles are spared its copy
    if (!h->stage_used) return LBM_OK;
    int err = 0;
    LBM_CUDA(cudaMemcpy(&err, h->d_err, sizeof(int), cudaMemcpyDeviceToHost), "error flag read");
    if (err) {
        LBM_CUDA(cudaMemset(h->d_err, 0, sizeof(int)), "error flag reset");
        return fail(LBM_ETIMEOUT, "a shared-memory staging wait of the step kernel ran out; the lattice state "
                                  "is not valid");
    }
    return LBM_OK;
}

int lbm_diagnostics(lbm_handle h, lbm_diag* out)
{
    int rc = check_handle(h);
    if (rc) return rc;
    if (!out) return fail(LBM_EINVAL, "null output");
    if (!h->initialized) return fail(LBM_ESTATE, "diagnostics before initialisation");
    if ((rc = enqueue_diagnostics(h))) return rc;
    LBM_CUDA(cudaStreamSynchronize(h->stream), "diagnostics");
    return fill_diag(h, h->step, out);
}

int lbm_step_diagnostics(lbm_handle h, int64_t nsteps, lbm_diag* out)
{
    int rc = check_handle(h);
    if (rc) return rc;
    if (!out) return fail(LBM_EINVAL, "null output");
    if (nsteps < 1) return fail(LBM_EINVAL, "lbm_step_diagnostics needs at least one step");
    if (!h->initialized) return fail(LBM_ESTATE, "lbm_step_diagnostics before initialisation");
    if (h->slab) return fail(LBM_EUNSUPPORTED, "a z-slab steps with lbm_step and reports with lbm_diagnostics");
    const int odd = h->odd;
    const bool pairs = uses_pairs(h, odd);
    const StepRange range = whole_range(h);
    const dim3 grid = step_grid(h, odd, range);
    const int rows = (int)(grid.x * grid.y * grid.z);
    if ((rc = ensure_diag(h, rows + h->num_sms))) return rc;
    const DiagArgs da = diag_args(h);
    StepArgs a = step_args(h, odd, range);
    a.dg = DiagSink{da.ep_scale, da.epsk_scale, da.s_scale, h->diag_fields, h->diag_partials};
    void* args[] = {&a};
    const void* k = pairs ? h->ks->step2_diag[h->p.forcing][odd] : h->ks->step_diag[h->p.forcing][odd];
    LBM_CUDA(cudaLaunchKernel(k, grid, step_block(h, odd), args, 0, h->stream), "diagnosing step");
    const int64_t step0 = h->step;
    ++h->launches;
    h->odd ^= 1;
    h->step += 1;
    LBM_CUDA(launch_totals(h, da, rows), "diag pass 2");
    LBM_CUDA(cudaEventRecord(h->diag_event, h->stream), "diag event");
    if ((rc = lbm_step(h, nsteps - 1))) return rc;
    LBM_CUDA(cudaEventSynchronize(h->diag_event), "diagnostics");
    return fill_diag(h, step0, out);
}

int lbm_get_fields(lbm_handle h, double* rho, double* u, double* rho_p)
{
    int rc = check_handle(h);
    if (rc) return rc;
    if (!h->initialized) return fail(LBM_ESTATE, "fields requested before initialisation");
    const size_t n3 = h->geo.n3;
    if ((rc = ensure_staging(h, 5 * n3 * sizeof(double)))) return rc;
    FieldArgs a;
    a.f = f_ptr(h);
    a.g = g_ptr(h);
    a.geo = h->geo;
    a.ph = h->ph;
    a.odd = h->odd;
    a.rho = h->staging;
    a.u = h->staging + n3;
    a.rho_p = h->staging + 4 * n3;
    void* args[] = {&a};
    LBM_CUDA(cudaLaunchKernel(h->ks->get_fields, node_grid(h), dim3(256), args, 0, h->stream), "get_fields");
    if (rho) LBM_CUDA(cudaMemcpyAsync(rho, a.rho, n3 * sizeof(double), cudaMemcpyDeviceToHost, h->stream), "copy rho");
    if (u) LBM_CUDA(cudaMemcpyAsync(u, a.u, 3 * n3 * sizeof(double), cudaMemcpyDeviceToHost, h->stream), "copy u");
    if (rho_p)
        LBM_CUDA(cudaMemcpyAsync(rho_p, a.rho_p, n3 * sizeof(double), cudaMemcpyDeviceToHost, h->stream), "copy rho_p");
    LBM_CUDA(cudaStreamSynchronize(h->stream), "get_fields");
    return LBM_OK;
}

int lbm_get_fields_device(lbm_handle h, double* rho, double* u, double* rho_p)
{
    int rc = check_handle(h);
    if (rc) return rc;
    if (!h->initialized) return fail(LBM_ESTATE, "fields requested before initialisation");
    double* outs[3] = {rho, u, rho_p};
    for (double* p : outs) {
        if (!p) continue;
        cudaPointerAttributes attr;
        cudaError_t e = cudaPointerGetAttributes(&attr, p);
        if (e != cudaSuccess || attr.type != cudaMemoryTypeDevice || attr.device != h->device) {
            cudaGetLastError();
            return fail(LBM_EINVAL, "field outputs must be device memory on the handle's device");
        }
    }
    FieldArgs a;
    a.f = f_ptr(h);
    a.g = g_ptr(h);
    a.geo = h->geo;
    a.ph = h->ph;
    a.odd = h->odd;
    a.rho = rho;
    a.u = u;
    a.rho_p = rho_p;
    void* args[] = {&a};
    LBM_CUDA(cudaLaunchKernel(h->ks->get_fields, node_grid(h), dim3(256), args, 0, h->stream),
             "get_fields_device");
    return LBM_OK;
}

int lbm_get_populations(lbm_handle h, double* f, double* g)
{
    int rc = check_handle(h);
    if (rc) return rc;
    if (!f || !g) return fail(LBM_EINVAL, "null output");
    if (!h->initialized) return fail(LBM_ESTATE, "populations requested before initialisation");
    const size_t n3 = h->geo.n3;
    const size_t nq = (size_t)h->q.qf + h->q.qg;
    if ((rc = ensure_staging(h, nq * n3 * sizeof(double)))) return rc;
    PopArgs a;
    a.f = f_ptr(h);
    a.g = g_ptr(h);
    a.geo = h->geo;
    a.fout = h->staging;
    a.gout = h->staging + (size_t)h->q.qf * n3;
    a.rho0 = h->p.rho0;
    a.odd = h->odd;
    void* args[] = {&a};
    LBM_CUDA(cudaLaunchKernel(h->ks->get_pops, dim3(flat_grid(h)), dim3(256), args, 0, h->stream), "get_pops");
    LBM_CUDA(cudaMemcpyAsync(f, a.fout, (size_t)h->q.qf * n3 * sizeof(double), cudaMemcpyDeviceToHost, h->stream),
             "copy f");
    LBM_CUDA(cudaMemcpyAsync(g, a.gout, (size_t)h->q.qg * n3 * sizeof(double), cudaMemcpyDeviceToHost, h->stream),
             "copy g");
    LBM_CUDA(cudaStreamSynchronize(h->stream), "get_populations");
    return LBM_OK;
}

int lbm_sample_populations(lbm_handle h, const int64_t* nodes, int64_t count, double* f, double* g)
{
    int rc = check_handle(h);
    if (rc) return rc;
    if (count < 0 || (count > 0 && (!nodes || !f || !g))) return fail(LBM_EINVAL, "invalid sample arguments");
    if (!h->initialized) return fail(LBM_ESTATE, "populations requested before initialisation");
    if (count == 0) return LBM_OK;
    for (int64_t s = 0; s < count; ++s)
        if (nodes[s] < 0 || nodes[s] >= (int64_t)h->geo.n3)
            return fail(LBM_EINVAL, "node index %lld out of range", (long long)nodes[s]);
    const size_t nq = (size_t)h->q.qf + h->q.qg;
    const size_t bytes = (size_t)count * (nq * sizeof(double) + sizeof(int64_t));
    if ((rc = ensure_staging(h, bytes))) return rc;
    SampleArgs a;
    a.f = f_ptr(h);
    a.g = g_ptr(h);
    a.geo = h->geo;
    a.fout = h->staging;
    a.gout = h->staging + (size_t)count * h->q.qf;
    int64_t* dnodes = reinterpret_cast<int64_t*>(h->staging + (size_t)count * nq);
    a.nodes = dnodes;
    a.count = count;
    a.rho0 = h->p.rho0;
    a.odd = h->odd;
    LBM_CUDA(cudaMemcpyAsync(dnodes, nodes, (size_t)count * sizeof(int64_t), cudaMemcpyHostToDevice, h->stream),
             "copy nodes");
    void* args[] = {&a};
    const unsigned blocks = (unsigned)((count + 255) / 256 < 4096 ? (count + 255) / 256 : 4096);
    LBM_CUDA(cudaLaunchKernel(h->ks->sample_pops, dim3(blocks), dim3(256), args, 0, h->stream), "sample_pops");
    LBM_CUDA(cudaMemcpyAsync(f, a.fout, (size_t)count * h->q.qf * sizeof(double), cudaMemcpyDeviceToHost, h->stream),
             "copy f");
    LBM_CUDA(cudaMemcpyAsync(g, a.gout, (size_t)count * h->q.qg * sizeof(double), cudaMemcpyDeviceToHost, h->stream),
             "copy g");
    LBM_CUDA(cudaStreamSynchronize(h->stream), "sample_populations");
    return LBM_OK;
}

int lbm_set_populations(lbm_handle h, const double* f, const double* g)
{
    int rc = check_handle(h);
    if (rc) return rc;
    if (!f || !g) return fail(LBM_EINVAL, "null input");
    if ((rc = ensure_store(h))) return rc;
    const size_t n3 = h->geo.n3;
    const size_t nq = (size_t)h->q.qf + h->q.qg;
    if ((rc = ensure_staging(h, nq * n3 * sizeof(double)))) return rc;
    PopArgs a;
    a.f = f_ptr(h);
    a.g = g_ptr(h);
    a.geo = h->geo;
    a.fout = h->staging;
    a.gout = h->staging + (size_t)h->q.qf * n3;
    a.rho0 = h->p.rho0;
    a.odd = 0;
    LBM_CUDA(cudaMemcpyAsync(a.fout, f, (size_t)h->q.qf * n3 * sizeof(double), cudaMemcpyHostToDevice, h->stream),
             "copy f");
    LBM_CUDA(cudaMemcpyAsync(a.gout, g, (size_t)h->q.qg * n3 * sizeof(double), cudaMemcpyHostToDevice, h->stream),
             "copy g");
    void* args[] = {&a};
    LBM_CUDA(cudaLaunchKernel(h->ks->set_pops, dim3(flat_grid(h)), dim3(256), args, 0, h->stream), "set_pops");
    LBM_CUDA(cudaStreamSynchronize(h->stream), "set_populations");
    h->initialized = true;
    h->odd = 0;
    return LBM_OK;
}

int lbm_step_count(lbm_handle h, int64_t* step)
{
    if (!h || !step) return fail(LBM_EINVAL, "null argument");
    *step = h->step;
    return LBM_OK;
}

int lbm_launch_count(lbm_handle h, int64_t* launches)
{
    if (!h || !launches) return fail(LBM_EINVAL, "null argument");
    *launches = h->launches;
    return LBM_OK;
}

int lbm_set_block(lbm_handle h, int bx, int by)
{
    if (!h) return fail(LBM_EINVAL, "null handle");
    if (bx < 32 || bx % 32 != 0 || by < 1 || bx * by > 256)
        return fail(LBM_EINVAL, "block (%d, %d): bx must be a positive multiple of 32 and bx*by <= 256", bx, by);
    h->bx = h->bxo = bx;
    h->by = h->byo = by;
    h->flat[0] = h->flat[1] = 0;
    drop_graph(h);
    return LBM_OK;
}

int lbm_get_block(lbm_handle h, int* bx, int* by)
{
    if (!h || !bx || !by) return fail(LBM_EINVAL, "null argument");
    *bx = h->bx;
    *by = h->by;
    return LBM_OK;
}

int lbm_autotune(lbm_handle h, int reps, double* best_ms_per_step)
{
    int rc = check_handle(h);
    if (rc) return rc;
    if (!h->initialized) return fail(LBM_ESTATE, "autotune needs an initialised state");
    if (reps < 1) return fail(LBM_EINVAL, "reps must be >= 1");
    // shapes, then flat launches (by = 0) of that many threads
    static const int cand[][2] = {{32, 1}, {32, 2}, {32, 4}, {32, 8}, {64, 1}, {64, 2}, {64, 4},
                                  {128, 1}, {128, 2}, {256, 1}, {64, 0}, {128, 0}, {256, 0}};
    void* backup = nullptr;
    const size_t bytes = store_need(h);
    LBM_CUDA(cudaMalloc(&backup, bytes), "autotune backup allocation");
    // one event between consecutive launches, so that each launch is timed
    // on its own and the two AA parities get their own best shape
    std::vector<cudaEvent_t> ev(2 * (size_t)reps + 1, nullptr);
    for (cudaEvent_t& e : ev) cudaEventCreate(&e);
    cudaMemcpyAsync(backup, h->store, bytes, cudaMemcpyDeviceToDevice, h->stream);
    const int save_bx = h->bx, save_by = h->by, save_bxo = h->bxo, save_byo = h->byo, save_odd = h->odd;
    const int save_flat[2] = {h->flat[0], h->flat[1]};
    double best[2] = {1e300, 1e300};
    int bbx[2] = {save_bx, save_bxo}, bby[2] = {save_by, save_byo}, bflat[2] = {save_flat[0], save_flat[1]};
    cudaError_t err = cudaSuccess;
    // A lattice that lbm_step advances in strips: a launch of a strip takes a
    // fraction of a step and starts in what the one before left in L2, so whole
    // groups of steps are timed, with one shape at both parities and, before and
    // after those (the first timings run on a GPU that is still speeding up), with
    // the shapes as set.
    const SkewPlan plan = h->l2 == L2Use::shared ? SkewPlan{1, 1, 1} : skew_plan(h);
    const bool strips = plan.depth > 1;
    auto time_strips = [&] {
        const int groups = (2 * reps + plan.depth - 1) / plan.depth;   // of an even number of steps
        for (int g = -1; g < groups && err == cudaSuccess; ++g) {      // one to warm up
            if (g == 0) err = cudaEventRecord(ev[0], h->stream);
            if (err == cudaSuccess) err = launch_group(h, plan, plan.depth, save_odd, (g & 1) != 0, h->stream);
        }
        if (err == cudaSuccess) err = cudaEventRecord(ev[1], h->stream);
        if (err == cudaSuccess) err = cudaEventSynchronize(ev[1]);
        float ms = 0.f;
        if (err == cudaSuccess) err = cudaEventElapsedTime(&ms, ev[0], ev[1]);
        return (double)ms / (groups * plan.depth);
    };
    if (strips) best[0] = best[1] = time_strips();
    for (const auto& c : cand) {
        if (err != cudaSuccess) break;
        const bool flat = c[1] == 0;
        if (flat && h->p.nx < 4) continue;               // a row of one unit has no division
        if (!flat && c[0] > 32 && c[0] / 2 >= h->p.nx) continue;  // wider than the row
        if (c[1] > 1 && (c[1] / 2) >= h->p.ny) continue;
        h->flat[0] = h->flat[1] = flat ? c[0] : 0;
        if (!flat) {
            h->bx = h->bxo = c[0];
            h->by = h->byo = c[1];
        }
        double t[2] = {0.0, 0.0};
        if (strips) {
            t[0] = t[1] = time_strips();
            if (err != cudaSuccess) break;
        } else {
            // warm-up pair, then timed pairs
            for (int s = 0; s < 2 && err == cudaSuccess; ++s) err = launch_step(h, (save_odd + s) & 1, h->stream);
            if (err == cudaSuccess) err = cudaEventRecord(ev[0], h->stream);
            for (int s = 0; s < 2 * reps && err == cudaSuccess; ++s) {
                err = launch_step(h, (save_odd + s) & 1, h->stream);
                if (err == cudaSuccess) err = cudaEventRecord(ev[s + 1], h->stream);
            }
            if (err == cudaSuccess) err = cudaEventSynchronize(ev[2 * reps]);
            if (err != cudaSuccess) break;
            for (int s = 0; s < 2 * reps; ++s) {
                float ms = 0.f;
                cudaEventElapsedTime(&ms, ev[s], ev[s + 1]);
                t[(save_odd + s) & 1] += ms / reps;
            }
        }
        for (int par = 0; par < 2; ++par)
            if (t[par] < best[par]) {
                best[par] = t[par];
                bflat[par] = flat ? c[0] : 0;
                bbx[par] = flat ? (par ? save_bxo : save_bx) : c[0];
                bby[par] = flat ? (par ? save_byo : save_by) : c[1];
            }
    }
    auto as_set = [&] {
        h->flat[0] = save_flat[0];
        h->flat[1] = save_flat[1];
        h->bx = save_bx;
        h->by = save_by;
        h->bxo = save_bxo;
        h->byo = save_byo;
    };
    as_set();
    if (strips && err == cudaSuccess) {
        const double t = time_strips();
        if (err == cudaSuccess && t <= best[0]) {
            best[0] = best[1] = t;
            for (int par = 0; par < 2; ++par) {
                bflat[par] = save_flat[par];
                bbx[par] = par ? save_bxo : save_bx;
                bby[par] = par ? save_byo : save_by;
            }
        }
    }
    cudaMemcpyAsync(h->store, backup, bytes, cudaMemcpyDeviceToDevice, h->stream);
    cudaError_t e2 = cudaStreamSynchronize(h->stream);
    cudaFree(backup);
    for (cudaEvent_t e : ev) cudaEventDestroy(e);
    h->odd = save_odd;
    if (err != cudaSuccess) return cuda_fail(err, "autotune");
    if (e2 != cudaSuccess) return cuda_fail(e2, "autotune restore");
    h->flat[0] = bflat[0];
    h->flat[1] = bflat[1];
    h->bx = bbx[0];
    h->by = bby[0];
    h->bxo = bbx[1];
    h->byo = bby[1];
    drop_graph(h);
    if (best_ms_per_step) *best_ms_per_step = 0.5 * (best[0] + best[1]);
    return LBM_OK;
}

int lbm_set_pairing(lbm_handle h, int mode)
{
    if (!h) return fail(LBM_EINVAL, "null handle");
    if (mode < LBM_PAIRING_OFF || mode > LBM_PAIRING_EVEN) return fail(LBM_EINVAL, "pairing mode must be 0, 1 or 2");
    h->pairing = mode;
    default_block(h);
    drop_graph(h);
    return LBM_OK;
}

int lbm_set_tile_staging(lbm_handle h, int enable)
{
    if (!h) return fail(LBM_EINVAL, "null handle");
    h->tile_staging = enable != 0;
    h->stage_grid = 0;
    drop_graph(h);
    return LBM_OK;
}

int lbm_uses_tile_staging(lbm_handle h, int* width)
{
    if (!h || !width) return fail(LBM_EINVAL, "null argument");
    *width = stage_width(h);
    return LBM_OK;
}

int lbm_set_stage_test(lbm_handle h, unsigned extra_tx_bytes, unsigned spin_limit)
{
    if (!h) return fail(LBM_EINVAL, "null handle");
    if (spin_limit == 0) return fail(LBM_EINVAL, "spin_limit must be positive");
    if (extra_tx_bytes >= (1u << 20)) return fail(LBM_EINVAL, "extra_tx_bytes must be below 2^20 (mbarrier tx count)");
    h->stage_extra_tx = extra_tx_bytes;
    h->stage_spin = spin_limit;
    drop_graph(h);
    return LBM_OK;
}

int lbm_set_slab(lbm_handle h, int enable)
{
    if (!h) return fail(LBM_EINVAL, "null handle");
    if (enable && h->p.nz < 3) return fail(LBM_EINVAL, "a z-slab needs nz >= 3 (two ghost planes and one of its own)");
    h->slab = enable != 0;
    h->stage_grid = 0;
    drop_graph(h);
    return LBM_OK;
}

int lbm_halo_bytes(lbm_handle h, size_t* bytes)
{
    if (!h || !bytes) return fail(LBM_EINVAL, "null argument");
    *bytes = (size_t)(halo_slots(h->q.qf, 1, nullptr) + halo_slots(h->q.qg, 1, nullptr)) * (size_t)h->p.nx *
             (size_t)h->p.ny * elem_size(h->p.storage);
    return LBM_OK;
}

int lbm_halo_pack(lbm_handle h, int phase, void* to_lower, void* to_upper)
{
    int rc = check_handle(h);
    if (rc) return rc;
    if (!h->slab) return fail(LBM_ESTATE, "halo exchange without lbm_set_slab");
    if (!h->store) return fail(LBM_ESTATE, "halo exchange before the store exists");
    if (phase != 0 && phase != 1) return fail(LBM_EINVAL, "phase must be 0 (before an odd step) or 1 (after it)");
    if (!to_lower || !to_upper) return fail(LBM_EINVAL, "null buffer");
    size_t bytes = 0;
    lbm_halo_bytes(h, &bytes);
    if ((rc = check_device_buffer(h, to_lower, bytes)) || (rc = check_device_buffer(h, to_upper, bytes))) return rc;
    const int top = h->p.nz - 1;
    // phase 0: own boundary planes (plane 1: e_z = +1 slots; plane nz-2: e_z = -1)
    // phase 1: ghost planes (plane 0: e_z = -1 slots; plane nz-1: e_z = +1)
    return halo_copy(h, phase ? 0 : 1, phase ? -1 : +1, to_lower, phase ? top : top - 1, phase ? +1 : -1, to_upper,
                     true);
}

int lbm_halo_unpack(lbm_handle h, int phase, const void* from_lower, const void* from_upper)
{
    int rc = check_handle(h);
    if (rc) return rc;
    if (!h->slab) return fail(LBM_ESTATE, "halo exchange without lbm_set_slab");
    if (!h->store) return fail(LBM_ESTATE, "halo exchange before the store exists");
    if (phase != 0 && phase != 1) return fail(LBM_EINVAL, "phase must be 0 (before an odd step) or 1 (after it)");
    if (!from_lower || !from_upper) return fail(LBM_EINVAL, "null buffer");
    size_t bytes = 0;
    lbm_halo_bytes(h, &bytes);
    if ((rc = check_device_buffer(h, from_lower, bytes)) || (rc = check_device_buffer(h, from_upper, bytes)))
        return rc;
    const int top = h->p.nz - 1;
    // phase 0: into the ghost planes (plane 0: e_z = -1 slots; plane nz-1: e_z = +1)
    // phase 1: into the own boundary planes (plane 1: e_z = +1; plane nz-2: e_z = -1)
    return halo_copy(h, phase ? 1 : 0, phase ? +1 : -1, from_lower, phase ? top - 1 : top, phase ? -1 : +1, from_upper,
                     false);
}

int lbm_set_graphs(lbm_handle h, int enable)
{
    if (!h) return fail(LBM_EINVAL, "null handle");
    h->graphs = enable != 0;
    if (!h->graphs) drop_graph(h);
    return LBM_OK;
}

}  // extern "C"

// ---------------------------------------------------------------------------
// Allocation-free diagnostics: the block partials of the moment pass and the
// final sums live in this file-scope device array instead of cudaMalloc'ed
// scratch. Host code cannot use the array's name as a device address, so the
// address is looked up with the device current and cached per device: when a
// handle is created (lbm_create_params) and, if still missing, on the first
// allocation-free call. A device reset destroys every handle, and the handles
// made after it look the address up again when they are created.
// ---------------------------------------------------------------------------
namespace {
constexpr int kStaticMaxBlocks = 4096;
constexpr uint32_t kStaticNodesPerBlock = 32768;
constexpr size_t kStaticOutOffset = (size_t)kStaticMaxBlocks * kDNumSlots;
constexpr int kStaticMaxDevices = 64;
std::mutex g_static_mutex;
double* g_static_addr[kStaticMaxDevices] = {};
}  // namespace

static __device__ __align__(256) double g_static_scratch[kStaticOutOffset + 16];

namespace {
void static_scratch_refresh(int device)
{
    if (device < 0 || device >= kStaticMaxDevices) return;
    void* p = nullptr;
    cudaError_t e = cudaGetSymbolAddress(&p, g_static_scratch);
    if (e != cudaSuccess) cudaGetLastError();
    std::lock_guard<std::mutex> lock(g_static_mutex);
    g_static_addr[device] = (e == cudaSuccess) ? static_cast<double*>(p) : nullptr;
}

int static_scratch_address(int device, double** out)
{
    if (device < 0 || device >= kStaticMaxDevices) return fail(LBM_EUNSUPPORTED, "device %d out of range", device);
    std::lock_guard<std::mutex> lock(g_static_mutex);
    if (!g_static_addr[device]) {
        void* p = nullptr;
        cudaError_t e = cudaGetSymbolAddress(&p, g_static_scratch);
        if (e != cudaSuccess || !p) return cuda_fail(e, "cudaGetSymbolAddress of the static diagnostics scratch");
        g_static_addr[device] = static_cast<double*>(p);
    }
    *out = g_static_addr[device];
    return LBM_OK;
}
}  // namespace

extern "C" {

int lbm_diagnostics_noalloc(lbm_handle h, lbm_diag* out)
{
    int rc = check_handle(h);
    if (rc) return rc;
    if (!out) return fail(LBM_EINVAL, "null output");
    const uint32_t n3 = h->geo.n3;
    const uint32_t min_blocks = (n3 + kStaticNodesPerBlock - 1) / kStaticNodesPerBlock;
    if (min_blocks > (uint32_t)kStaticMaxBlocks)
        return fail(LBM_EINVAL,
                    "lattice of %u nodes exceeds the static diagnostics scratch (at most %u nodes); "
                    "use lbm_diagnostics",
                    n3, (unsigned)kStaticMaxBlocks * kStaticNodesPerBlock);
    if (!h->initialized) return fail(LBM_ESTATE, "diagnostics before initialisation");
    if (h->slab) return fail(LBM_EUNSUPPORTED, "allocation-free diagnostics of a z-slab (use lbm_diagnostics)");
    double* scratch = nullptr;
    if ((rc = static_scratch_address(h->device, &scratch))) return rc;
    // a row of the array per block, as lbm_diagnostics within the array's rows
    const uint32_t blocks = std::min((uint32_t)kStaticMaxBlocks, std::max(min_blocks, moment_blocks(h, n3)));
    const lbm_params& p = h->p;
    const double cs2f = cs2_of(h->q.qf);
    const double gn2 = (p.beta != 0.0) ? (-p.G * p.rho0 / p.beta) : 1.0;
    const double nu = cs2f * (p.tau_f - 0.5);
    DiagArgs a{};
    a.f = f_ptr(h);
    a.g = g_ptr(h);
    a.geo = h->geo;
    a.ph = h->ph;
    a.odd = h->odd;
    a.ep_scale = (float)(0.5 * gn2 / (p.rho0 * p.rho0));
    a.epsk_scale = (float)(2.0 * nu);
    a.s_scale = (float)(-1.0 / (2.0 * cs2f * p.tau_f));
    a.epsp_scale = 0.f;
    a.nu = (float)nu;
    a.fields = nullptr;      // no field scratch: the central-difference pass is skipped
    a.partials = scratch;    // every block overwrites its own record, nothing needs clearing
    a.idx0 = 0;
    a.idx1 = n3;
    void* args[] = {&a};
    LBM_CUDA(cudaLaunchKernel(h->ks->diag_moments, dim3(blocks), dim3(kDiagBlock), args, 0, h->stream),
             "static diag pass 1");
    const double* pp = scratch;
    int nb = (int)blocks;
    double* dout = scratch + kStaticOutOffset;
    void* fargs[] = {&pp, &nb, &dout};
    LBM_CUDA(cudaLaunchKernel(diag_totals_kernel(), dim3(kDiagPass1), dim3(kDiagBlock), fargs, 0, h->stream),
             "static diag pass 2");
    double s[kDiagPass1];
    LBM_CUDA(cudaMemcpyAsync(s, dout, sizeof(s), cudaMemcpyDeviceToHost, h->stream), "static diag copy");
    LBM_CUDA(cudaStreamSynchronize(h->stream), "static diagnostics");
    const double inv = 1.0 / (double)n3;
    const double nan = std::numeric_limits<double>::quiet_NaN();
    out->Ek = s[kDEk] * inv;
    out->Ep = s[kDEp] * inv;
    out->eps_k = s[kDEpsK] * inv;
    out->eps_p = nan;
    out->eps_k_curl = nan;
    out->mass_f = (double)n3 + s[kDDrho];
    out->mass_g = (double)n3 * p.rho0 + s[kDA];
    out->mom[0] = s[kDJx];
    out->mom[1] = s[kDJy];
    out->mom[2] = s[kDJz];
    out->umax = s[kDUmax];
    out->step = h->step;
    fill_phys(p, out);
    for (int q = 0; q < kDiagPass1; ++q)
        if (!std::isfinite(s[q])) return fail(LBM_ENONFINITE, "non-finite diagnostics at step %lld", (long long)h->step);
    return LBM_OK;
}

int lbm_destroy(lbm_handle h)
{
    if (!h) return LBM_OK;
    cudaSetDevice(h->device);
    if (h->stream) cudaStreamSynchronize(h->stream);
    drop_graph(h);
    if (h->own_store && h->store) cudaFree(h->store);
    if (h->staging) cudaFree(h->staging);
    if (h->diag_fields) cudaFree(h->diag_fields);
    if (h->diag_partials) cudaFree(h->diag_partials);
    if (h->diag_grad) cudaFree(h->diag_grad);
    if (h->diag_host) cudaFreeHost(h->diag_host);
    if (h->diag_event) cudaEventDestroy(h->diag_event);
    if (h->copy_event) cudaEventDestroy(h->copy_event);
    if (h->copy_stream) cudaStreamSynchronize(h->copy_stream);
    for (int b = 0; b < 2; ++b) {
        if (h->pre[b]) cudaFree(h->pre[b]);
        if (h->pre_done[b]) cudaEventDestroy(h->pre_done[b]);
        if (h->pre_free[b]) cudaEventDestroy(h->pre_free[b]);
    }
    if (h->copy_stream) cudaStreamDestroy(h->copy_stream);
    if (h->d_err) cudaFree(h->d_err);
    if (h->own_stream && h->stream) cudaStreamDestroy(h->stream);
    delete h;
    return LBM_OK;
}

}  // extern "C"

// ---------------------------------------------------------------------------
// Batched instances: many independent lattices advanced by one launch.
// ---------------------------------------------------------------------------
struct lbm_batch_ctx {
    std::vector<lbm_ctx*> inst;
    int device = 0;
    int num_sms = 0;
    cudaStream_t stream = nullptr;
    bool own_stream = false;
    BatchInstance* d_inst = nullptr;
    uint16_t* d_tile = nullptr;
    unsigned* d_sync = nullptr;
    uint32_t ntiles = 0;
    uint32_t vbeg[8] = {}, vend[8] = {};   // tiles of each (pair, forcing) variant
    // per-variant streams and events: the captured graph runs each variant's
    // chain of steps as its own branch (variants share no instance)
    cudaStream_t vstream[8] = {};
    cudaEvent_t vjoin[8] = {};
    cudaEvent_t vfork = nullptr;
    // per-instance driver: instances, largest store first; rounds of those
    // that L2 holds together, which run all steps of a call before the next
    // round's; streams and join events, created as they are needed
    std::vector<int> order;
    std::vector<std::vector<int>> rounds;
    std::vector<cudaStream_t> cstream;
    std::vector<cudaEvent_t> cjoin;
    int bx = 32, by = 8;
    int mode = LBM_BATCH_PERSISTENT;
    int chunk = 100;
    int persistent_grid = 0;
    unsigned spin_limit = 1u << 22;   // ~0.3-1 s of polling at 64 ns naps
    unsigned extra_dep = 0;           // test hook: completions a dependency wait expects that never come
    // persistent driver: one step's tile list, its tile size, the queue and
    // completion counters, the kernel variant and its graphs (one per parity)
    uint16_t* d_flow_inst = nullptr;
    unsigned* d_flow = nullptr;
    uint32_t flow_tiles = 0;
    uint32_t flow_nodes = 2048;
    bool guo_sc_only = false;
    FlowArgs* flow_args = nullptr;   // the persistent launch's parameter block (descriptors by value)
    cudaGraphExec_t pgraph[2] = {nullptr, nullptr};
    int pgraph_steps[2] = {0, 0};
    bool initialized = false;
    int64_t step = 0;
    int odd = 0;
    cudaGraphExec_t graph = nullptr;
};

namespace {

constexpr int kBatchGraphSteps = 64;
constexpr int kMaxChains = 128;   // streams of the per-instance driver
constexpr int kRecordChains = 8;  // and of a batch's records

void batch_drop_graph(lbm_batch_ctx* b)
{
    if (b->graph) cudaGraphExecDestroy(b->graph);
    b->graph = nullptr;
    for (int k = 0; k < 2; ++k) {
        if (b->pgraph[k]) cudaGraphExecDestroy(b->pgraph[k]);
        b->pgraph[k] = nullptr;
        b->pgraph_steps[k] = 0;
    }
}

int batch_build_tiles(lbm_batch_ctx* b)
{
    std::vector<BatchInstance> hi(b->inst.size());
    std::vector<uint16_t> tiles;
    uint32_t t0 = 0;
    // tiles listed variant by variant, so that each per-variant launch covers one range
    std::vector<size_t> order(b->inst.size());
    for (size_t i = 0; i < order.size(); ++i) order[i] = i;
    std::stable_sort(order.begin(), order.end(), [&](size_t a, size_t c) {
        return 4 * b->inst[a]->p.pair + b->inst[a]->p.forcing < 4 * b->inst[c]->p.pair + b->inst[c]->p.forcing;
    });
    for (int v = 0; v < 8; ++v) b->vbeg[v] = b->vend[v] = 0;
    for (size_t i : order) {
        lbm_ctx* h = b->inst[i];
        BatchInstance& I = hi[i];
        I.f = f_ptr(h);
        I.g = g_ptr(h);
        I.geo = h->geo;
        I.ph = h->ph;
        I.variant = 4 * h->p.pair + h->p.forcing;
        I.tx = (uint32_t)((h->p.nx + b->bx - 1) / b->bx);
        I.ty = (uint32_t)((h->p.ny + b->by - 1) / b->by);
        I.tile0 = t0;
        const uint64_t n = (uint64_t)I.tx * I.ty * (uint64_t)h->p.nz;
        if ((uint64_t)t0 + n > 0xffffffffull) return fail(LBM_EINVAL, "batch tile count exceeds 2^32");
        tiles.insert(tiles.end(), (size_t)n, (uint16_t)i);
        const int v = I.variant;
        if (b->vend[v] == b->vbeg[v]) b->vbeg[v] = t0;
        t0 += (uint32_t)n;
        b->vend[v] = t0;
    }
    b->ntiles = t0;
    // persistent driver: runs of flow_nodes consecutive nodes, instances with
    // the most bytes per step first
    std::vector<size_t> big(b->inst.size());
    for (size_t i = 0; i < big.size(); ++i) big[i] = i;
    std::stable_sort(big.begin(), big.end(),
                     [&](size_t a, size_t c) { return b->inst[a]->store_bytes > b->inst[c]->store_bytes; });
    std::vector<uint16_t> flow;
    b->guo_sc_only = true;
    for (size_t i : big) {
        BatchInstance& I = hi[i];
        I.flow0 = (uint32_t)flow.size();
        I.nflow = (I.geo.n3 + b->flow_nodes - 1) / b->flow_nodes;
        flow.insert(flow.end(), (size_t)I.nflow, (uint16_t)i);
        if (b->inst[i]->p.forcing != LBM_GUO && b->inst[i]->p.forcing != LBM_SHAN_CHEN) b->guo_sc_only = false;
    }
    if (flow.size() > 0x7fffffffull) return fail(LBM_EINVAL, "batch tile count exceeds 2^31");
    b->flow_tiles = (uint32_t)flow.size();
    if (hi.size() <= (size_t)kFlowMaxInst) {
        if (!b->flow_args) b->flow_args = new (std::nothrow) FlowArgs();
        if (!b->flow_args) return fail(LBM_ENOMEM, "host allocation failed");
        for (size_t i = 0; i < hi.size(); ++i) b->flow_args->inst[i] = hi[i];
    }
    if (b->d_inst) cudaFree(b->d_inst);
    if (b->d_tile) cudaFree(b->d_tile);
    if (b->d_flow_inst) cudaFree(b->d_flow_inst);
    if (b->d_flow) cudaFree(b->d_flow);
    b->d_inst = nullptr;
    b->d_tile = nullptr;
    b->d_flow_inst = nullptr;
    b->d_flow = nullptr;
    if (cudaMalloc(&b->d_inst, hi.size() * sizeof(BatchInstance)) != cudaSuccess ||
        cudaMalloc(&b->d_tile, tiles.size() * sizeof(uint16_t)) != cudaSuccess ||
        cudaMalloc(&b->d_flow_inst, flow.size() * sizeof(uint16_t)) != cudaSuccess ||
        cudaMalloc(&b->d_flow, (1 + hi.size()) * sizeof(unsigned)) != cudaSuccess) {
        cudaGetLastError();
        return fail(LBM_ENOMEM, "batch descriptor allocation failed");
    }
    LBM_CUDA(cudaMemcpy(b->d_inst, hi.data(), hi.size() * sizeof(BatchInstance), cudaMemcpyHostToDevice),
             "copy batch descriptors");
    LBM_CUDA(cudaMemcpy(b->d_tile, tiles.data(), tiles.size() * sizeof(uint16_t), cudaMemcpyHostToDevice),
             "copy batch tiles");
    LBM_CUDA(cudaMemcpy(b->d_flow_inst, flow.data(), flow.size() * sizeof(uint16_t), cudaMemcpyHostToDevice),
             "copy batch tile list");
    int per_sm = 0;
    LBM_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, batch_flow_kernel(b->guo_sc_only), 256, 0),
             "batch occupancy");
    if (per_sm < 1) return fail(LBM_EUNSUPPORTED, "persistent batch kernel does not fit on an SM");
    b->persistent_grid = per_sm * b->num_sms;
    batch_drop_graph(b);
    return LBM_OK;
}

BatchArgs batch_args(const lbm_batch_ctx* b, int steps, int odd0, unsigned grid)
{
    BatchArgs a;
    a.inst = b->d_inst;
    a.tile_inst = b->d_tile;
    a.ntiles = b->ntiles;
    a.tile_begin = 0;
    a.tile_end = b->ntiles;
    a.steps = steps;
    a.odd0 = odd0;
    a.sync = b->d_sync;
    a.spin_limit = b->spin_limit;
    a.flow_inst = b->d_flow_inst;
    a.flow_tiles = b->flow_tiles;
    a.flow_nodes = b->flow_nodes;
    a.flow = b->d_flow;
    a.extra_dep = b->extra_dep;
    (void)grid;
    return a;
}

cudaError_t batch_launch_variant(lbm_batch_ctx* b, int v, int odd, cudaStream_t s)
{
    const uint32_t n = b->vend[v] - b->vbeg[v];
    if (n == 0) return cudaSuccess;
    // one tile per block: the block scheduler then overlaps the descriptor
    // loads that start every tile (measured 2 % faster than a strided loop)
    const unsigned grid = (unsigned)n;
    BatchArgs a = batch_args(b, 1, odd, grid);
    a.tile_begin = b->vbeg[v];
    a.tile_end = b->vend[v];
    void* args[] = {&a};
    return cudaLaunchKernel(batch_variant_kernel(v, odd), dim3(grid), dim3(b->bx, b->by), args, 0, s);
}

cudaError_t batch_launch_step(lbm_batch_ctx* b, int odd, cudaStream_t s)
{
    for (int v = 0; v < 8; ++v) {
        cudaError_t e = batch_launch_variant(b, v, odd, s);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

// Streams and join events of the per-instance driver, at least `count` of them;
// after a failure those that are complete stay.
cudaError_t batch_ensure_streams(lbm_batch_ctx* b, size_t count)
{
    while (b->cjoin.size() < count) {
        cudaStream_t s = nullptr;
        cudaEvent_t done = nullptr;
        cudaError_t e = cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking);
        if (e == cudaSuccess) e = cudaEventCreateWithFlags(&done, cudaEventDisableTiming);
        if (e != cudaSuccess) {
            if (s) cudaStreamDestroy(s);
            return e;
        }
        b->cstream.push_back(s);
        b->cjoin.push_back(done);
    }
    return cudaSuccess;
}

// Instances dealt to at most `most` chains.
std::vector<std::vector<int>> deal_chains(const std::vector<int>& instances, size_t most)
{
    std::vector<std::vector<int>> chains(std::min(instances.size(), most));
    for (size_t k = 0; k < instances.size(); ++k) chains[k % chains.size()].push_back(instances[k]);
    return chains;
}

// Rounds of the per-instance driver: instances in order of size, as many to a
// round as 3/4 of L2 holds, at least one. All 64 lattices of a size, pair,
// forcing and Froude number sweep (32^3 to 96^3, 2.6 GB) at once leave nothing
// in L2 from step to step (885 us a step of all of them, 98 % of the copy
// bandwidth); in rounds all but the 96^3 D3Q27xD3Q19 ones step from L2, and
// those, one to a round, in skewed strips: 728 us.
void batch_build_rounds(lbm_batch_ctx* b)
{
    if (!b->rounds.empty()) return;
    std::vector<int> order(b->inst.size());
    for (size_t i = 0; i < order.size(); ++i) order[i] = (int)i;
    std::stable_sort(order.begin(), order.end(),
                     [&](int a, int c) { return b->inst[a]->store_bytes > b->inst[c]->store_bytes; });
    b->order = order;
    const size_t budget = b->inst[0]->l2_bytes / 4 * 3;
    size_t held = 0;
    for (int i : order) {
        const size_t bytes = b->inst[i]->store_bytes;
        if (b->rounds.empty() || (budget > 0 && held + bytes > budget)) {
            b->rounds.emplace_back();
            held = 0;
        }
        b->rounds.back().push_back(i);
        held += bytes;
    }
}

// work(h) for the instances of each chain with h on the chain's stream, the
// chains forked from and joined back to b->stream, a chain whose work failed too.
template <class Work>
int batch_run_chains(lbm_batch_ctx* b, const std::vector<std::vector<int>>& chains, Work&& work)
{
    LBM_CUDA(cudaEventRecord(b->vfork, b->stream), "batch fork");
    int rc = LBM_OK;
    for (size_t c = 0; c < chains.size() && rc == LBM_OK; ++c) {
        LBM_CUDA(cudaStreamWaitEvent(b->cstream[c], b->vfork, 0), "batch fork wait");
        for (int i : chains[c]) {
            lbm_ctx* h = b->inst[i];
            h->stream = b->cstream[c];
            rc = work(h);
            h->stream = b->stream;
            if (rc) break;
        }
        LBM_CUDA(cudaEventRecord(b->cjoin[c], b->cstream[c]), "batch join");
        LBM_CUDA(cudaStreamWaitEvent(b->stream, b->cjoin[c], 0), "batch join wait");
    }
    return rc;
}

// A call of one step keeps nothing in L2 and runs all instances at once (the
// sweep above in calls of 1 / 2 / 4 / 100 steps: 970 / 956 / 821 / 728 us a step;
// 4 steps all at once 1007).
constexpr int64_t kRoundSteps = 2;

int batch_step_instances(lbm_batch_ctx* b, int64_t nsteps)
{
    const size_t most = std::min<size_t>(b->inst.size(), kMaxChains);
    LBM_CUDA(batch_ensure_streams(b, most), "batch chain streams");
    batch_build_rounds(b);
    // lbm_step on the chain's stream: the instance's own graph replays, eager steps outside them
    if (nsteps < kRoundSteps)
        return batch_run_chains(b, deal_chains(b->order, most), [&](lbm_ctx* h) { return lbm_step(h, nsteps); });
    for (const std::vector<int>& round : b->rounds) {
        const int rc = batch_run_chains(b, deal_chains(round, most), [&](lbm_ctx* h) {
            if (round.size() == 1) h->l2 = L2Use::alone;
            const int r = lbm_step(h, nsteps);
            h->l2 = L2Use::shared;
            return r;
        });
        if (rc) return rc;
    }
    return LBM_OK;
}

// Records `steps` steps (from the natural layout) into the capture running on
// b->stream: each variant's chain on its own stream, forked from and joined
// back to b->stream.
cudaError_t batch_capture_steps(lbm_batch_ctx* b, int steps)
{
    cudaError_t e = cudaEventRecord(b->vfork, b->stream);
    for (int v = 0; v < 8 && e == cudaSuccess; ++v) {
        if (b->vend[v] == b->vbeg[v]) continue;
        e = cudaStreamWaitEvent(b->vstream[v], b->vfork, 0);
        for (int s = 0; s < steps && e == cudaSuccess; ++s) e = batch_launch_variant(b, v, s & 1, b->vstream[v]);
        if (e == cudaSuccess) e = cudaEventRecord(b->vjoin[v], b->vstream[v]);
        if (e == cudaSuccess) e = cudaStreamWaitEvent(b->stream, b->vjoin[v], 0);
    }
    return e;
}

// One persistent launch of `steps` steps: clear the queue and completion
// counters, then the kernel (a plain launch: see lbm_batch.cu).
cudaError_t batch_launch_persistent(lbm_batch_ctx* b, int steps, int odd, cudaStream_t s)
{
    const unsigned grid = (unsigned)b->persistent_grid;
    // the descriptors travel in the parameter block (b->flow_args, filled by
    // batch_build_tiles); the launch copies it
    FlowArgs& fa = *b->flow_args;
    fa.a = batch_args(b, steps, odd, grid);
    cudaError_t e = cudaMemsetAsync(b->d_flow, 0, (1 + b->inst.size()) * sizeof(unsigned), s);
    if (e != cudaSuccess) return e;
    void* args[] = {&fa};
    return cudaLaunchKernel(batch_flow_kernel(b->guo_sc_only), dim3(grid), dim3(256), args, 0, s);
}

// The same launch replayed from a CUDA graph (one per starting parity).
cudaError_t batch_persistent_graph(lbm_batch_ctx* b, int steps, int odd)
{
    if (!b->pgraph[odd] || b->pgraph_steps[odd] != steps) {
        if (b->pgraph[odd]) cudaGraphExecDestroy(b->pgraph[odd]);
        b->pgraph[odd] = nullptr;
        cudaGraph_t g = nullptr;
        cudaError_t e = cudaStreamBeginCapture(b->stream, cudaStreamCaptureModeThreadLocal);
        if (e == cudaSuccess) {
            e = batch_launch_persistent(b, steps, odd, b->stream);
            cudaError_t e2 = cudaStreamEndCapture(b->stream, &g);
            if (e == cudaSuccess) e = e2;
        }
        if (e == cudaSuccess) e = cudaGraphInstantiate(&b->pgraph[odd], g, 0);
        if (g) cudaGraphDestroy(g);
        if (e != cudaSuccess) return e;
        b->pgraph_steps[odd] = steps;
    }
    return cudaGraphLaunch(b->pgraph[odd], b->stream);
}

void batch_sync_instances(lbm_batch_ctx* b)
{
    for (lbm_ctx* h : b->inst) {
        h->step = b->step;
        h->odd = b->odd;
        h->initialized = b->initialized;
    }
}

int batch_check(lbm_batch_ctx* b)
{
    if (!b) return fail(LBM_EINVAL, "null batch");
    cudaError_t e = cudaSetDevice(b->device);
    if (e != cudaSuccess) return cuda_fail(e, "cudaSetDevice");
    return LBM_OK;
}

}  // namespace

extern "C" {

int lbm_batch_create(lbm_batch* out, const lbm_params* params, int count)
{
    if (!out) return fail(LBM_EINVAL, "null output");
    *out = nullptr;
    if (!params || count < 1 || count > 65535) return fail(LBM_EINVAL, "count must be in [1, 65535]");
    for (int i = 0; i < count; ++i) {
        if (params[i].storage != LBM_FP32)
            return fail(LBM_EUNSUPPORTED, "batched instances use FP32 storage (instance %d)", i);
        if (params[i].pair != LBM_D3Q27_D3Q19 && params[i].pair != LBM_D3Q19_D3Q7)
            return fail(LBM_EUNSUPPORTED, "batched instances use D3Q27xD3Q19 or D3Q19xD3Q7 (instance %d)", i);
    }
    lbm_batch_ctx* b = new (std::nothrow) lbm_batch_ctx();
    if (!b) return fail(LBM_ENOMEM, "host allocation failed");
    int rc = LBM_OK;
    cudaGetDevice(&b->device);
    cudaDeviceGetAttribute(&b->num_sms, cudaDevAttrMultiProcessorCount, b->device);
    if (cudaStreamCreateWithFlags(&b->stream, cudaStreamNonBlocking) != cudaSuccess) {
        cudaGetLastError();
        delete b;
        return fail(LBM_ECUDA, "stream creation failed");
    }
    b->own_stream = true;
    bool streams_ok = cudaEventCreateWithFlags(&b->vfork, cudaEventDisableTiming) == cudaSuccess;
    for (int v = 0; v < 8 && streams_ok; ++v) {
        streams_ok = cudaStreamCreateWithFlags(&b->vstream[v], cudaStreamNonBlocking) == cudaSuccess &&
                     cudaEventCreateWithFlags(&b->vjoin[v], cudaEventDisableTiming) == cudaSuccess;
    }
    if (!streams_ok) {
        cudaGetLastError();
        rc = fail(LBM_ECUDA, "batch stream or event creation failed");
    }
    for (int i = 0; i < count && rc == LBM_OK; ++i) {
        lbm_handle h = nullptr;
        rc = lbm_create_params(&h, &params[i]);
        if (rc) break;
        b->inst.push_back(h);
        h->l2 = L2Use::shared;
        if ((rc = lbm_set_stream(h, b->stream))) break;
        if ((rc = ensure_store(h))) break;
    }
    if (rc == LBM_OK && (cudaMalloc(&b->d_sync, 4 * sizeof(unsigned)) != cudaSuccess ||
                         cudaMemset(b->d_sync, 0, 4 * sizeof(unsigned)) != cudaSuccess)) {
        cudaGetLastError();
        rc = fail(LBM_ENOMEM, "batch barrier allocation failed");
    }
    if (rc == LBM_OK) rc = batch_build_tiles(b);
    if (rc == LBM_OK && b->inst.size() > (size_t)kFlowMaxInst) b->mode = LBM_BATCH_PER_STEP;
    if (rc) {
        std::string msg = g_last_error;
        lbm_batch_destroy(b);
        g_last_error = msg;
        return rc;
    }
    *out = b;
    return LBM_OK;
}

int lbm_batch_count(lbm_batch b, int* count)
{
    if (!b || !count) return fail(LBM_EINVAL, "null argument");
    *count = (int)b->inst.size();
    return LBM_OK;
}

int lbm_batch_instance(lbm_batch b, int i, lbm_handle* h)
{
    if (!b || !h) return fail(LBM_EINVAL, "null argument");
    if (i < 0 || i >= (int)b->inst.size()) return fail(LBM_EINVAL, "instance %d out of range", i);
    *h = b->inst[i];
    return LBM_OK;
}

int lbm_batch_set_stream(lbm_batch b, void* stream)
{
    int rc = batch_check(b);
    if (rc) return rc;
    if (b->own_stream) {
        cudaStreamSynchronize(b->stream);
        cudaStreamDestroy(b->stream);
    }
    b->stream = static_cast<cudaStream_t>(stream);
    b->own_stream = false;
    for (lbm_ctx* h : b->inst) h->stream = b->stream;
    batch_drop_graph(b);
    return LBM_OK;
}

int lbm_batch_set_mode(lbm_batch b, int mode, int steps_per_launch)
{
    if (!b) return fail(LBM_EINVAL, "null batch");
    if (mode != LBM_BATCH_PERSISTENT && mode != LBM_BATCH_PER_STEP && mode != LBM_BATCH_INSTANCES)
        return fail(LBM_EINVAL, "unknown mode %d", mode);
    if (steps_per_launch < 1) return fail(LBM_EINVAL, "steps per launch must be >= 1");
    if (mode == LBM_BATCH_PERSISTENT && b->inst.size() > (size_t)kFlowMaxInst)
        return fail(LBM_EUNSUPPORTED, "the persistent driver takes at most %d instances (batch has %zu)", kFlowMaxInst,
                    b->inst.size());
    if (mode != b->mode) batch_drop_graph(b);   // the graph holds one driver's launches
    b->mode = mode;
    b->chunk = steps_per_launch;
    return LBM_OK;
}

int lbm_batch_set_block(lbm_batch b, int bx, int by)
{
    int rc = batch_check(b);
    if (rc) return rc;
    if (!(bx == 16 || bx == 32 || bx == 64 || bx == 128) || by < 1 || bx * by > 256 || (bx * by) % 32 != 0)
        return fail(LBM_EINVAL, "batch block (%d, %d): bx in {16, 32, 64, 128}, bx*by a multiple of 32 <= 256", bx, by);
    b->bx = bx;
    b->by = by;
    return batch_build_tiles(b);
}

int lbm_batch_get_config(lbm_batch b, int* bx, int* by, int* mode, int* grid)
{
    if (!b) return fail(LBM_EINVAL, "null batch");
    if (bx) *bx = b->bx;
    if (by) *by = b->by;
    if (mode) *mode = b->mode;
    if (grid) *grid = b->mode == LBM_BATCH_PERSISTENT ? b->persistent_grid : (int)b->ntiles;   // tiles: also per instance
    return LBM_OK;
}

int lbm_batch_init_tgv(lbm_batch b, uint64_t seed, double noise_amp)
{
    int rc = batch_check(b);
    if (rc) return rc;
    for (lbm_ctx* h : b->inst)
        if ((rc = lbm_init_tgv(h, seed, noise_amp))) return rc;
    b->initialized = true;
    b->step = 0;
    b->odd = 0;
    batch_sync_instances(b);
    return LBM_OK;
}

int lbm_batch_step(lbm_batch b, int64_t nsteps)
{
    int rc = batch_check(b);
    if (rc) return rc;
    if (nsteps < 0) return fail(LBM_EINVAL, "negative step count");
    if (!b->initialized) return fail(LBM_ESTATE, "batch step before initialisation");
    if (b->mode == LBM_BATCH_INSTANCES && nsteps > 0) {
        // no stream: every instance in turn on the legacy stream
        if (b->stream == nullptr) {
            for (lbm_ctx* h : b->inst)
                if ((rc = lbm_step(h, nsteps))) return rc;
        } else if ((rc = batch_step_instances(b, nsteps))) {
            return rc;
        }
        b->odd ^= (int)(nsteps & 1);
        b->step += nsteps;
        nsteps = 0;
    }
    while (nsteps > 0) {
        if (b->mode == LBM_BATCH_PERSISTENT) {
            // queue positions are 32-bit: steps * tiles per step (plus the
            // grid's claims past the end) must stay below 2^32
            const int64_t kmax = (int64_t)((0xffffffffull - 2ull * (uint64_t)b->persistent_grid) / b->flow_tiles);
            const int64_t chunk = std::min<int64_t>(b->chunk, std::max<int64_t>(kmax, 1));
            const int k = (int)(nsteps < chunk ? nsteps : chunk);
            if (b->stream != nullptr && k == chunk)
                LBM_CUDA(batch_persistent_graph(b, k, b->odd), "persistent batch graph");
            else
                LBM_CUDA(batch_launch_persistent(b, k, b->odd, b->stream), "persistent batch launch");
            b->odd ^= (k & 1);
            b->step += k;
            nsteps -= k;
            continue;
        }
        if (b->stream != nullptr && b->odd == 0 && nsteps >= kBatchGraphSteps) {
            if (!b->graph) {
                cudaGraph_t g = nullptr;
                cudaError_t e = cudaStreamBeginCapture(b->stream, cudaStreamCaptureModeThreadLocal);
                if (e == cudaSuccess) {
                    e = batch_capture_steps(b, kBatchGraphSteps);
                    cudaError_t e2 = cudaStreamEndCapture(b->stream, &g);
                    if (e == cudaSuccess) e = e2;
                }
                if (e == cudaSuccess) e = cudaGraphInstantiate(&b->graph, g, 0);
                if (g) cudaGraphDestroy(g);
                if (e != cudaSuccess) return cuda_fail(e, "batch graph capture");
            }
            LBM_CUDA(cudaGraphLaunch(b->graph, b->stream), "batch graph launch");
            b->step += kBatchGraphSteps;
            nsteps -= kBatchGraphSteps;
            continue;
        }
        LBM_CUDA(batch_launch_step(b, b->odd, b->stream), "batch step launch");
        b->odd ^= 1;
        b->step += 1;
        nsteps -= 1;
    }
    batch_sync_instances(b);
    return LBM_OK;
}

int lbm_batch_synchronize(lbm_batch b)
{
    int rc = batch_check(b);
    if (rc) return rc;
    LBM_CUDA(cudaStreamSynchronize(b->stream), "batch synchronize");
    unsigned flags[4];
    LBM_CUDA(cudaMemcpy(flags, b->d_sync, sizeof(flags), cudaMemcpyDeviceToHost), "read barrier state");
    if (flags[2] != 0u) {
        cudaMemset(b->d_sync, 0, 4 * sizeof(unsigned));
        return fail(LBM_ETIMEOUT, "a dependency wait of the persistent batch kernel ran out; "
                                  "the state of the batch is undefined");
    }
    return LBM_OK;
}

int lbm_batch_diagnostics(lbm_batch b, lbm_diag* out)
{
    int rc = lbm_batch_synchronize(b);
    if (rc) return rc;
    if (!out) return fail(LBM_EINVAL, "null output");
    for (lbm_ctx* h : b->inst) {
        if (!h->initialized) return fail(LBM_ESTATE, "diagnostics before initialisation");
    }
    // every instance's kernels first, on several streams, then one wait (one
    // instance after the other with a wait each: 64 instances 3.3 ms)
    if (b->stream != nullptr) {
        const size_t most = std::min<size_t>(b->inst.size(), kRecordChains);
        LBM_CUDA(batch_ensure_streams(b, most), "batch chain streams");
        batch_build_rounds(b);
        rc = batch_run_chains(b, deal_chains(b->order, most), enqueue_diagnostics);
        if (rc) return rc;
    } else {
        for (lbm_ctx* h : b->inst)
            if ((rc = enqueue_diagnostics(h))) return rc;
    }
    int worst = LBM_OK;
    for (size_t i = 0; i < b->inst.size(); ++i) {
        LBM_CUDA(cudaStreamSynchronize(b->inst[i]->stream), "diagnostics");
        rc = fill_diag(b->inst[i], b->inst[i]->step, &out[i]);
        if (rc == LBM_ENONFINITE) worst = rc;
        else if (rc) return rc;
    }
    return worst;
}

int lbm_batch_autotune(lbm_batch b, int reps, double* best_ms_per_step)
{
    int rc = batch_check(b);
    if (rc) return rc;
    if (!b->initialized) return fail(LBM_ESTATE, "autotune needs an initialised batch");
    if (reps < 1) return fail(LBM_EINVAL, "reps must be >= 1");
    if ((rc = lbm_batch_synchronize(b))) return rc;
    std::vector<void*> backup(b->inst.size(), nullptr);
    for (size_t i = 0; i < b->inst.size(); ++i) {
        if (cudaMalloc(&backup[i], b->inst[i]->store_bytes) != cudaSuccess) {
            cudaGetLastError();
            for (void* p : backup) if (p) cudaFree(p);
            return fail(LBM_ENOMEM, "autotune backup allocation failed");
        }
        cudaMemcpyAsync(backup[i], b->inst[i]->store, b->inst[i]->store_bytes, cudaMemcpyDeviceToDevice, b->stream);
    }
    static const int cand[][2] = {{16, 8}, {32, 2}, {32, 4}, {32, 8}, {64, 2}, {64, 4}, {128, 1}, {128, 2}};
    static const int flow_cand[] = {1024, 2048, 4096, 8192};
    const int save_bx = b->bx, save_by = b->by, save_mode = b->mode, save_odd = b->odd;
    const uint32_t save_flow = b->flow_nodes;
    const int64_t save_step = b->step;
    double best = 1e300;
    int bbx = save_bx, bby = save_by, bmode = save_mode;
    uint32_t bflow = save_flow;
    cudaEvent_t e0, e1;
    cudaEventCreate(&e0);
    cudaEventCreate(&e1);
    // one candidate as lbm_batch_step runs it: a warm-up span (which also
    // builds the graphs), then `reps` spans timed with events; a span is one
    // 64-step graph (per-step and per-instance drivers) or one persistent launch
    auto time_mode = [&](int mode, double* per) {
        b->mode = mode;
        const int64_t span = (mode == LBM_BATCH_PERSISTENT) ? b->chunk : kBatchGraphSteps;
        int r = lbm_batch_step(b, span);
        if (r) return r;
        cudaEventRecord(e0, b->stream);
        r = lbm_batch_step(b, span * (int64_t)reps);
        cudaEventRecord(e1, b->stream);
        if (r) return r;
        if ((r = lbm_batch_synchronize(b))) return r;
        float ms = 0.f;
        cudaEventElapsedTime(&ms, e0, e1);
        *per = ms / (double)(span * reps);
        return LBM_OK;
    };
    for (const auto& c : cand) {
        b->bx = c[0];
        b->by = c[1];
        if ((rc = batch_build_tiles(b))) break;
        double per = 0.0;
        if ((rc = time_mode(LBM_BATCH_PER_STEP, &per))) break;
        if (per < best) {
            best = per;
            bbx = c[0];
            bby = c[1];
            bmode = LBM_BATCH_PER_STEP;
        }
    }
    b->bx = save_bx;
    b->by = save_by;
    const bool flow_ok = b->inst.size() <= (size_t)kFlowMaxInst;
    for (size_t k = 0; flow_ok && k < sizeof(flow_cand) / sizeof(flow_cand[0]) && rc == LBM_OK; ++k) {
        b->flow_nodes = (uint32_t)flow_cand[k];
        if ((rc = batch_build_tiles(b))) break;
        double per = 0.0;
        if ((rc = time_mode(LBM_BATCH_PERSISTENT, &per))) break;
        if (per < best) {
            best = per;
            bbx = save_bx;
            bby = save_by;
            bflow = b->flow_nodes;
            bmode = LBM_BATCH_PERSISTENT;
        }
    }
    b->flow_nodes = save_flow;
    if (rc == LBM_OK) {
        // per-instance driver: every instance's own launch shape, then whole
        // 64-step graphs of all chains
        batch_sync_instances(b);
        batch_build_rounds(b);
        for (const std::vector<int>& round : b->rounds) {
            for (int i : round) {
                lbm_ctx* h = b->inst[i];
                if (round.size() == 1) h->l2 = L2Use::alone;   // as batch_step_instances steps it
                rc = lbm_autotune(h, reps, nullptr);
                h->l2 = L2Use::shared;
                if (rc) break;
            }
            if (rc) break;
        }
        b->mode = LBM_BATCH_INSTANCES;
        batch_drop_graph(b);
        if (rc == LBM_OK) rc = lbm_batch_step(b, kBatchGraphSteps);   // warm-up, builds the graph
        if (rc == LBM_OK) {
            cudaEventRecord(e0, b->stream);
            rc = lbm_batch_step(b, kBatchGraphSteps * (int64_t)reps);
            cudaEventRecord(e1, b->stream);
        }
        if (rc == LBM_OK) rc = lbm_batch_synchronize(b);
        if (rc == LBM_OK) {
            float ms = 0.f;
            cudaEventElapsedTime(&ms, e0, e1);
            const double per = ms / (double)(kBatchGraphSteps * reps);
            if (per < best) {
                best = per;
                bbx = b->bx;
                bby = b->by;
                bflow = b->flow_nodes;
                bmode = LBM_BATCH_INSTANCES;
            }
        }
    }
    for (size_t i = 0; i < b->inst.size(); ++i) {
        cudaMemcpyAsync(b->inst[i]->store, backup[i], b->inst[i]->store_bytes, cudaMemcpyDeviceToDevice, b->stream);
    }
    cudaStreamSynchronize(b->stream);
    for (void* p : backup) cudaFree(p);
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    b->odd = save_odd;
    b->step = save_step;
    b->bx = bbx;
    b->by = bby;
    b->flow_nodes = bflow;
    b->mode = bmode;
    int rc2 = batch_build_tiles(b);
    batch_sync_instances(b);
    if (rc) return rc;
    if (rc2) return rc2;
    if (best_ms_per_step) *best_ms_per_step = best;
    return LBM_OK;
}

int lbm_batch_set_barrier_test(lbm_batch b, unsigned extra_completions, unsigned spin_limit)
{
    if (!b) return fail(LBM_EINVAL, "null batch");
    if (spin_limit < 1) return fail(LBM_EINVAL, "spin limit must be >= 1");
    b->extra_dep = extra_completions;
    b->spin_limit = spin_limit;
    batch_drop_graph(b);
    return LBM_OK;
}

int lbm_batch_partition(const lbm_params* params, int count, int nranks, int32_t* owner, double* imbalance)
{
    if (!params || !owner || count < 1 || count > 65535 || nranks < 1)
        return fail(LBM_EINVAL, "lbm_batch_partition: null argument, count outside [1, 65535] or nranks < 1");
    std::vector<double> bytes(count);
    for (int i = 0; i < count; ++i) {
        PairInfo q;
        int rc = validate_params(&params[i], &q);
        if (rc) return rc;
        bytes[i] = (double)(q.qf + q.qg) * (double)params[i].nx * params[i].ny * params[i].nz *
                   (double)elem_size(params[i].storage);
    }
    // longest first (ties: lower index first), each to the least-loaded rank (ties: lower rank)
    std::vector<int> order(count);
    for (int i = 0; i < count; ++i) order[i] = i;
    std::stable_sort(order.begin(), order.end(), [&](int a, int c) { return bytes[a] > bytes[c]; });
    std::vector<double> load(nranks, 0.0);
    for (int i : order) {
        int r = 0;
        for (int k = 1; k < nranks; ++k)
            if (load[k] < load[r]) r = k;
        owner[i] = r;
        load[r] += bytes[i];
    }
    if (imbalance) {
        double total = 0.0, mx = 0.0;
        for (double l : load) {
            total += l;
            mx = std::max(mx, l);
        }
        *imbalance = mx / (total / nranks);
    }
    return LBM_OK;
}

int lbm_batch_set_flow_nodes(lbm_batch b, int nodes)
{
    int rc = batch_check(b);
    if (rc) return rc;
    if (nodes < 256 || nodes > 65536 || nodes % 256 != 0)
        return fail(LBM_EINVAL, "nodes per tile must be a multiple of 256 in [256, 65536] (got %d)", nodes);
    b->flow_nodes = (uint32_t)nodes;
    return batch_build_tiles(b);
}

int lbm_batch_get_flow_nodes(lbm_batch b, int* nodes)
{
    if (!b || !nodes) return fail(LBM_EINVAL, "null argument");
    *nodes = (int)b->flow_nodes;
    return LBM_OK;
}

int lbm_batch_destroy(lbm_batch b)
{
    if (!b) return LBM_OK;
    cudaSetDevice(b->device);
    if (b->stream) cudaStreamSynchronize(b->stream);
    batch_drop_graph(b);
    for (lbm_ctx* h : b->inst) {
        h->stream = nullptr;
        h->own_stream = false;
        lbm_destroy(h);
    }
    if (b->d_inst) cudaFree(b->d_inst);
    if (b->d_tile) cudaFree(b->d_tile);
    if (b->d_flow_inst) cudaFree(b->d_flow_inst);
    if (b->d_flow) cudaFree(b->d_flow);
    delete b->flow_args;
    if (b->d_sync) cudaFree(b->d_sync);
    for (int v = 0; v < 8; ++v) {
        if (b->vstream[v]) cudaStreamDestroy(b->vstream[v]);
        if (b->vjoin[v]) cudaEventDestroy(b->vjoin[v]);
    }
    if (b->vfork) cudaEventDestroy(b->vfork);
    for (cudaStream_t cs : b->cstream)
        if (cs) cudaStreamDestroy(cs);
    for (cudaEvent_t ce : b->cjoin)
        if (ce) cudaEventDestroy(ce);
    if (b->own_stream && b->stream) cudaStreamDestroy(b->stream);
    delete b;
    return LBM_OK;
}

}  // extern "C"

// ---------------------------------------------------------------------------
// The 16-bit storage rule (host logic on a few numbers per sample).
// ---------------------------------------------------------------------------
namespace {

// max_s |c_s - r_s| / max_s |r_s| of one diagnostics quantity; +inf when the
// candidate is not finite, 0 for an all-zero reference matched exactly.
template <class Get>
double series_dev(const lbm_diag* ref, const lbm_diag* cand, int64_t count, Get get)
{
    double scale = 0.0, worst = 0.0;
    for (int64_t s = 0; s < count; ++s) {
        const double r = get(ref[s]), c = get(cand[s]);
        if (!std::isfinite(c)) return std::numeric_limits<double>::infinity();
        scale = std::max(scale, std::fabs(r));
        worst = std::max(worst, std::fabs(c - r));
    }
    if (scale > 0.0) return worst / scale;
    return worst > 0.0 ? std::numeric_limits<double>::infinity() : 0.0;
}

}  // namespace

extern "C" {

int lbm_storage_rule(const lbm_diag* ref, const lbm_diag* cand, int64_t count, int candidate_storage, double tol,
                     lbm_storage_report* report)
{
    if (!ref || !cand || count < 1) return fail(LBM_EINVAL, "lbm_storage_rule needs two series of >= 1 samples");
    if (candidate_storage < LBM_FP32 || candidate_storage > LBM_BF16_DEV)
        return fail(LBM_EINVAL, "unknown storage %d", candidate_storage);
    if (!(tol > 0.0) || !std::isfinite(tol)) return fail(LBM_EINVAL, "tol must be finite and > 0");
    for (int64_t s = 0; s < count; ++s) {
        if (ref[s].step != cand[s].step)
            return fail(LBM_EINVAL, "sample %lld: reference step %lld, candidate step %lld", (long long)s,
                        (long long)ref[s].step, (long long)cand[s].step);
        if (!std::isfinite(ref[s].Ek) || !std::isfinite(ref[s].Ep) || !std::isfinite(ref[s].eps_k) ||
            !std::isfinite(ref[s].eps_p))
            return fail(LBM_EINVAL, "reference sample %lld is not finite", (long long)s);
    }
    lbm_storage_report r{};
    r.dev_Ek = series_dev(ref, cand, count, [](const lbm_diag& d) { return d.Ek; });
    r.dev_Ep = series_dev(ref, cand, count, [](const lbm_diag& d) { return d.Ep; });
    r.dev_eps_k = series_dev(ref, cand, count, [](const lbm_diag& d) { return d.eps_k; });
    r.dev_eps_p = series_dev(ref, cand, count, [](const lbm_diag& d) { return d.eps_p; });
    // the two highest interior local maxima of the reference eps_k + eps_p
    auto eps = [](const lbm_diag& d) { return d.eps_k + d.eps_p; };
    int64_t p1 = -1, p2 = -1;
    for (int64_t s = 1; s + 1 < count; ++s) {
        const double e = eps(ref[s]);
        if (!(e > eps(ref[s - 1]) && e >= eps(ref[s + 1]))) continue;
        if (p1 < 0 || e > eps(ref[p1])) {
            p2 = p1;
            p1 = s;
        } else if (p2 < 0 || e > eps(ref[p2])) {
            p2 = s;
        }
    }
    const double nan = std::numeric_limits<double>::quiet_NaN();
    auto peak_dev = [&](int64_t s) {
        if (s < 0) return nan;
        const double c = eps(cand[s]);
        if (!std::isfinite(c)) return std::numeric_limits<double>::infinity();
        return std::fabs(c - eps(ref[s])) / std::fabs(eps(ref[s]));
    };
    r.dev_peak1 = peak_dev(p1);
    r.dev_peak2 = peak_dev(p2);
    r.step_peak1 = p1 < 0 ? -1 : ref[p1].step;
    r.step_peak2 = p2 < 0 ? -1 : ref[p2].step;
    bool pass = r.dev_Ek <= tol && r.dev_Ep <= tol && r.dev_eps_k <= tol && r.dev_eps_p <= tol;
    if (p1 >= 0) pass = pass && r.dev_peak1 <= tol;
    if (p2 >= 0) pass = pass && r.dev_peak2 <= tol;
    r.pass = pass ? 1 : 0;
    r.selected = pass ? candidate_storage : LBM_FP32;
    if (report) *report = r;
    return r.selected;
}

}  // extern "C"
