// C ABI of the batched stability sweep (lbm_batch_* in include/lbm.h): instance layout in one
// slab, batched equilibrium initialisation, the graph-captured persistent launch, results,
// and the autotuner that picks the kernel's (vector width, CTA size).
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <functional>
#include <new>
#include <numeric>
#include <queue>
#include <vector>

#include "lbm.h"
#include "lbm_batch.cuh"
#include "lbm_internal.h"

using lbm::BatchInstance;
using lbm::BatchState;

struct lbm_batch {
    int n = 0;
    int storage = LBM_F32;
    double rho0 = 1.0;
    cudaStream_t stream = nullptr;
    std::vector<BatchInstance> inst;
    std::vector<long long> node_off;   // dense node offset of each instance (concatenated fields)
    long long nodes = 0;
    BatchInstance* d_inst = nullptr;
    BatchState* d_state = nullptr;
    int* d_order = nullptr;
    int* d_queue = nullptr;
    long long* d_node_off = nullptr;
    void* slab = nullptr;
    size_t slab_bytes = 0;
    double* stage = nullptr;           // host-pointer staging for init (lazy)
    size_t stage_elems = 0;
    int vec = 0, block = 0, grid = 0;
    bool fused = false;                // the kernel with the marches
    int smem = 0;                      // its dynamic shared memory
    int per_sm = 0, sms = 0;           // resident CTAs per SM of the kernel; SMs
    bool models = false;               // instances of several models
    bool own_shape = true;             // the shape is the library's choice
    int shape_check = -1;              // check interval the kernel was chosen for
    std::vector<int> order;            // largest instances first
    std::vector<int> bands;            // of a march, by instance
    const void* kernel = nullptr;
    cudaGraphExec_t exec = nullptr;
    long long g_target = -1;
    int g_check = -1;
    double g_growth = -1.0;
    const void* g_kernel = nullptr;
    char err[512] = {0};
};

namespace {

int berr(lbm_batch* b, int code, const char* fmt, ...) {
    if (b) {
        va_list ap;
        va_start(ap, fmt);
        vsnprintf(b->err, sizeof(b->err), fmt, ap);
        va_end(ap);
    }
    return code;
}

#define LBM_BCK(b, call)                                                                         \
    do {                                                                                         \
        cudaError_t e_ = (call);                                                                 \
        if (e_ != cudaSuccess)                                                                   \
            return berr((b), e_ == cudaErrorMemoryAllocation ? LBM_ERR_NOMEM : LBM_ERR_CUDA,     \
                        "%s failed: %s", #call, cudaGetErrorString(e_));                         \
    } while (0)

const void* pick_batch_kernel(int storage, int vec, int block, bool fused) {
    switch (storage) {
        case LBM_F64: return lbm::batch_kernel_f64(vec, block);
        case LBM_F32: return lbm::batch_kernel_f32(vec, block, fused);
        case LBM_F16: return lbm::batch_kernel_f16(vec, block, fused);
        case LBM_BF16: return lbm::batch_kernel_bf16(vec, block, fused);
        default: return nullptr;
    }
}

// dynamic shared memory of a batch kernel: the fused marches' of its warps (none for FP64)
int batch_smem(int storage, int block) {
    if (storage == LBM_F64) return 0;
    return block / 32 * (storage == LBM_F32 ? lbm::march_smem_bytes<float, true> : lbm::march_smem_bytes<__half, true>);
}

// ---- which instances march, and how many threads a CTA has --------------------------------------
// Estimated us a step of an instance with `block` threads, `resident` such CTAs at work on its SM;
// `spill`: the instances at work together exceed the L2.  Fitted to 17 shapes of 16 x 16 to 256 x 256,
// 3 x 2000 to 2000 x 3, alone and 152, 304, 608 at a time, FP32 and FP16, mostly within a tenth.
// One step at a time: latency a sweep, then nodes at the rate of so many warps, of a full SM or of HBM.
double one_step_us(const BatchInstance& I, int vec, int block, int resident, bool spill) {
    const double nodes = (double)I.a.ny * ((I.a.nx + vec - 1) / vec * vec);
    const double alone = 0.7 + nodes / (block >= 512 ? 1020.0 : (block >= 256 ? 850.0 : 630.0));
    return std::max(alone, 0.8 + nodes * resident / (spill ? 630.0 : 1040.0));
}
// Bands of a marching instance, as batch_march picks them.
int fused_bands(const BatchInstance& I, int block) {
    const int warps = block / 32, most = lbm::MarchForm<float>::TMAX;
    const int strips = (I.a.nx + lbm::march_width(most) - 1) / lbm::march_width(most);
    long long least = 1ll << 40;
    int bands = 1;
    for (int b = 1; b <= 2 * warps; ++b) {
        const long long cost = ((long long)strips * b + warps - 1) / warps * ((I.a.ny + b - 1) / b + most - 1);
        if (cost < least) {
            least = cost;
            bands = b;
        }
    }
    return bands;
}
// t steps fused, a step: rounds of the CTA's warps over strips and bands.
double fused_us(const BatchInstance& I, int bands, int block, int resident, int t) {
    const int warps = block / 32;
    const long long tasks = (long long)((I.a.nx + lbm::march_width(t) - 1) / lbm::march_width(t)) * bands;
    const double rows = (double)((tasks + warps - 1) / warps) * ((I.a.ny + bands - 1) / bands + t - 1);
    const int load = warps * resident;   // warps of the SM: a level row takes so long
    const double row = load <= 4 ? 0.26 : (load <= 8 ? 0.36 : 0.69);
    return 0.5 + rows * row * (0.8 + 0.8 / t);
}
// what a check adds to a step: the folds of the diagnostics in FP64
double check_us(const BatchInstance& I, int block, int resident) {
    const double nodes = (double)I.a.nx * I.a.ny;
    if (block >= 512) return 7.1 + nodes / 1100.0;
    return block >= 256 ? (resident > 1 ? 4.0 + nodes / 900.0 : 4.5 + nodes / 870.0) : 3.5 + nodes * resident / 1100.0;
}
int resident_ctas(const lbm_batch* b) { return std::max(1, std::min(b->per_sm, (b->n + b->sms - 1) / b->sms)); }
bool spills(const lbm_batch* b) {
    const double together = std::min<double>(b->n, (double)b->sms * resident_ctas(b)) / b->n;
    return (double)b->slab_bytes * together > 110e6;
}
// one_step_us in the kernel of the batch's shape: accesses below 16 bytes, and instances of several
// models on an SM or beside the marches, which cost one another the instruction cache (800 of 96^2 in
// BF16: 256 threads 98 us against 61 fused, 128 threads 149 against 56).
double sweep_us(const lbm_batch* b, const BatchInstance& I) {
    const int resident = resident_ctas(b);
    double us = one_step_us(I, b->vec, b->block, resident, spills(b));
    if (b->vec * lbm::storage_bytes(b->storage) < 16) us *= 1.25;
    if (!b->models) return us;
    if (b->storage == LBM_F32) return us * (b->fused ? (resident > 1 ? 1.35 : 1.1) : 1.0);
    return us * (resident > 1 ? 1.7 : (b->fused ? 1.25 : 1.0));
}
// Least check interval from which marching instance I is quicker (kNeverMarch: never): the fewest
// steps t that pay fused are what lies between two checks.
int march_from(const lbm_batch* b, const BatchInstance& I, int bands) {
    const double one = sweep_us(b, I);
    int from = lbm::kNeverMarch;
    for (int t = lbm::MarchForm<float>::TMAX; t >= 1 && fused_us(I, bands, b->block, resident_ctas(b), t) < one; --t)
        from = t + 1;
    return from;
}

bool is_device_ptr(const void* p) {
    cudaPointerAttributes at;
    if (cudaPointerGetAttributes(&at, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return at.type == cudaMemoryTypeDevice || at.type == cudaMemoryTypeManaged;
}

// The kernel of (vec, block), with the marches or without, and what of it suits the instances.
int set_shape(lbm_batch* b, int vec, int block, bool fused) {
    const void* k = pick_batch_kernel(b->storage, vec, block, fused);
    if (!k) return berr(b, LBM_ERR_UNSUPPORTED, "no batch kernel with vec=%d block=%d for this storage", vec, block);
    int dev = 0, per_sm = 0;
    LBM_BCK(b, cudaGetDevice(&dev));
    LBM_BCK(b, cudaDeviceGetAttribute(&b->sms, cudaDevAttrMultiProcessorCount, dev));
    const int smem = fused ? batch_smem(b->storage, block) : 0;
    LBM_BCK(b, cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    LBM_BCK(b, cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, block, smem));
    if (per_sm < 1) return berr(b, LBM_ERR_UNSUPPORTED, "batch kernel cannot be resident");
    b->kernel = k;
    b->vec = vec;
    b->block = block;
    b->fused = fused;
    b->smem = smem;
    b->per_sm = per_sm;
    // resident CTAs only (a persistent grid); never more CTAs than instances
    b->grid = std::min(b->sms * per_sm, b->n);
    b->bands.resize(b->n);
    for (int i = 0; i < b->n; ++i) {
        BatchInstance& I = b->inst[i];
        b->bands[i] = fused ? fused_bands(I, block) : 1;
        I.march_from = fused ? march_from(b, I, b->bands[i]) : lbm::kNeverMarch;
    }
    return LBM_OK;
}

// Estimated us a step of all instances in runs checked every `check_every` steps: each to the CTA that
// is free first, largest first, as the queue hands them out.
double shape_us(const lbm_batch* b, int check_every) {
    const int resident = resident_ctas(b);
    const int apart = check_every > 0 ? check_every : 1 << 20;   // steps from check to check
    const int t = std::min(apart - 1, (int)lbm::MarchForm<float>::TMAX);
    std::priority_queue<double, std::vector<double>, std::greater<double>> busy;
    double last = 0.0;
    for (int i : b->order) {
        const BatchInstance& I = b->inst[i];
        const double one = sweep_us(b, I);
        const double rest = lbm::batch_fused(I.march_from, check_every) ? fused_us(I, b->bands[i], b->block, resident, t) : one;
        double us = rest + (one - rest + check_us(I, b->block, resident)) / apart;
        if ((int)busy.size() == b->grid) {
            us += busy.top();
            busy.pop();
        }
        busy.push(us);
        last = std::max(last, us);
    }
    return last;
}

// The kernel for runs checked every `check_every` steps.  With the shape left to the library, CTAs of
// 512 threads (FP64 256), or of 256 where that is clearly quicker: two of 256 overlap one another's
// barriers, loads and checks, one of 512 has an instance done sooner (us a step, 512 / 256: 300 of
// 32^2 3.7 / 2.8, 800 of 96^2 60 / 54, 200 of 32..128 squared 21 / 37, 1024 of 32..256 147 / 162).
int choose_shape(lbm_batch* b, int check_every) {
    if (b->kernel && (b->storage == LBM_F64 || b->shape_check == check_every)) return LBM_OK;
    const int own = 16 / lbm::storage_bytes(b->storage), given = b->block, vec = b->own_shape ? own : b->vec;
    struct {
        int block;
        bool fused;
        double worth;
    } best = {0, false, 1e300}, all[] = {{512, true, 1.0}, {512, false, 1.0}, {256, false, 1.0}, {256, true, 1.0}};
    if (b->storage == LBM_F64) {
        best.block = 256;
    } else {
        for (auto& c : all) {
            if (!b->own_shape) {
                if (c.block == 256) continue;
                c.block = given;
            }
            const int rc = set_shape(b, vec, c.block, c.fused);
            if (rc != LBM_OK) return rc;
            c.worth = shape_us(b, check_every) * (c.block == 256 ? (b->n > b->sms ? 1.06 : 1.035) : 1.0);
            if (c.worth < best.worth) best = c;
        }
    }
    const int rc = set_shape(b, vec, best.block, best.fused);
    if (rc != LBM_OK) return rc;
    b->shape_check = check_every;
    // (in the order of the stream, so after the runs before)
    LBM_BCK(b, cudaMemcpyAsync(b->d_inst, b->inst.data(), sizeof(BatchInstance) * b->n, cudaMemcpyHostToDevice, b->stream));
    return LBM_OK;
}
// A shape asked for: its kernel of the check interval in use.
int ask_shape(lbm_batch* b, int vec, int block) {
    if (!pick_batch_kernel(b->storage, vec, block, false))
        return berr(b, LBM_ERR_UNSUPPORTED, "no batch kernel with vec=%d block=%d for this storage", vec, block);
    const int check = b->shape_check < 0 ? 100 : b->shape_check;
    b->own_shape = false;
    b->vec = vec;
    b->block = block;
    if (b->storage == LBM_F64) return set_shape(b, vec, block, false);
    b->shape_check = -1;
    return choose_shape(b, check);
}
// Equilibrium initialisation of every instance from concatenated dense fields.
template <typename S>
__global__ void batch_init_kernel(S* slab, const BatchInstance* __restrict__ inst, const BatchState* __restrict__ st,
                                  const long long* __restrict__ node_off, int n, long long nodes,
                                  const double* __restrict__ rho, const double* __restrict__ ux,
                                  const double* __restrict__ uy) {
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < nodes;
         k += (long long)gridDim.x * blockDim.x) {
        int lo = 0, hi = n - 1;   // last instance whose node_off <= k
        while (lo < hi) {
            const int mid = (lo + hi + 1) / 2;
            if (node_off[mid] <= k) lo = mid; else hi = mid - 1;
        }
        const BatchInstance& I = inst[lo];
        const lbm::StepArgs& a = I.a;
        const long long local = k - node_off[lo];
        const int y = (int)(local / a.nx), x = (int)(local - (long long)y * a.nx);
        S* buf = slab + I.off + (long long)st[lo].cur * 9 * a.plane;
        S g[9];
        lbm::equilibrium_node<S>(rho[k], ux[k], uy[k], a.rho0, a.urx, a.ury, I.eq, g);
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            int xs = x - lbm::ex_of(i), ys = y - lbm::ey_of(i);
            xs = xs < 0 ? xs + a.nx : (xs >= a.nx ? xs - a.nx : xs);
            ys = ys < 0 ? ys + a.ny : (ys >= a.ny ? ys - a.ny : ys);
            buf[(long long)i * a.plane + (long long)ys * a.pitch + xs] = g[i];
        }
    }
}

cudaError_t launch_batch_init(lbm_batch* b, const double* r, const double* x, const double* y) {
    const int block = 256;
    long long g = (b->nodes + block - 1) / block;
    if (g > 152 * 32) g = 152 * 32;
    switch (b->storage) {
        case LBM_F64: batch_init_kernel<double><<<(int)g, block, 0, b->stream>>>((double*)b->slab, b->d_inst, b->d_state, b->d_node_off, b->n, b->nodes, r, x, y); break;
        case LBM_F32: batch_init_kernel<float><<<(int)g, block, 0, b->stream>>>((float*)b->slab, b->d_inst, b->d_state, b->d_node_off, b->n, b->nodes, r, x, y); break;
        case LBM_F16: batch_init_kernel<__half><<<(int)g, block, 0, b->stream>>>((__half*)b->slab, b->d_inst, b->d_state, b->d_node_off, b->n, b->nodes, r, x, y); break;
        default: batch_init_kernel<__nv_bfloat16><<<(int)g, block, 0, b->stream>>>((__nv_bfloat16*)b->slab, b->d_inst, b->d_state, b->d_node_off, b->n, b->nodes, r, x, y); break;
    }
    return cudaGetLastError();
}

int reset_states(lbm_batch* b) {
    std::vector<BatchState> s(b->n);
    for (auto& x : s) {
        x.steps = 0; x.blowup_step = -1; x.pert0 = -1.0;
        x.pert = x.ke = x.rho_min = x.nonfinite = 0.0;
        x.status = 0; x.cur = 0;
    }
    LBM_BCK(b, cudaMemcpyAsync(b->d_state, s.data(), sizeof(BatchState) * b->n, cudaMemcpyHostToDevice, b->stream));
    LBM_BCK(b, cudaStreamSynchronize(b->stream));
    return LBM_OK;
}

// records {queue = 0; persistent kernel} into a graph for the current parameters
int record_run(lbm_batch* b, long long target, int check_every, double growth) {
    if (b->exec && b->g_target == target && b->g_check == check_every && b->g_growth == growth &&
        b->g_kernel == b->kernel)
        return LBM_OK;
    if (b->exec) {
        cudaGraphExecDestroy(b->exec);
        b->exec = nullptr;
    }
    cudaStream_t cap = nullptr;
    LBM_BCK(b, cudaStreamCreateWithFlags(&cap, cudaStreamNonBlocking));
    cudaError_t e = cudaStreamBeginCapture(cap, cudaStreamCaptureModeThreadLocal);
    if (e == cudaSuccess) {
        cudaMemsetAsync(b->d_queue, 0, sizeof(int), cap);
        void* slab = b->slab;
        const BatchInstance* di = b->d_inst;
        BatchState* ds = b->d_state;
        const int* dord = b->d_order;
        int n = b->n;
        int* dq = b->d_queue;
        long long tg = target;
        int ce = check_every;
        double gr = growth;
        void* args[] = {&slab, &di, &ds, &dord, &n, &dq, &tg, &ce, &gr};
        cudaLaunchKernel(b->kernel, dim3(b->grid), dim3(b->block), args, b->smem, cap);
        cudaGraph_t graph = nullptr;
        e = cudaStreamEndCapture(cap, &graph);
        if (e == cudaSuccess) {
            e = cudaGraphInstantiate(&b->exec, graph, 0);
            cudaGraphDestroy(graph);
        }
    }
    cudaStreamDestroy(cap);
    if (e != cudaSuccess) {
        b->exec = nullptr;
        return berr(b, LBM_ERR_CUDA, "batch graph: %s", cudaGetErrorString(e));
    }
    b->g_target = target;
    b->g_check = check_every;
    b->g_growth = growth;
    b->g_kernel = b->kernel;
    return LBM_OK;
}

}  // namespace

extern "C" {

const char* lbm_batch_last_error(const lbm_batch* b) { return b ? b->err : "null batch"; }

int lbm_batch_create(lbm_batch** out, int n, const lbm_instance_desc* desc, int storage, double rho0,
                     void* cuda_stream) {
    if (!out) return LBM_ERR_INVALID_ARG;
    *out = nullptr;
    if (n < 1 || !desc || storage < LBM_F64 || storage > LBM_BF16 || !(rho0 > 0.0) || !std::isfinite(rho0))
        return LBM_ERR_INVALID_ARG;
    const int esz = lbm::storage_bytes(storage);
    const int align_elems = 32 / esz;   // 32-byte rows: every 16-byte vector stays aligned
    long long off = 0, nodes = 0;
    std::vector<BatchInstance> inst(n);
    std::vector<long long> node_off(n);
    for (int k = 0; k < n; ++k) {
        const lbm_instance_desc& d = desc[k];
        if (d.nx < 3 || d.ny < 3 || (long long)d.nx * d.ny > (1LL << 31)) return LBM_ERR_INVALID_ARG;
        if (d.model < LBM_BGK || d.model > LBM_K_EQ) return LBM_ERR_INVALID_ARG;
        const lbm_rates& r = d.rates;
        for (double w : {r.omega_nu, r.omega3, r.omega4})
            if (!(std::isfinite(w) && w > 0.0 && w < 2.0)) return LBM_ERR_INVALID_ARG;
        if (!std::isfinite(d.ux_ref) || !std::isfinite(d.uy_ref) || std::fabs(d.ux_ref) >= 1.0 ||
            std::fabs(d.uy_ref) >= 1.0 || !std::isfinite(d.ke_ref) || !std::isfinite(d.ke_factor))
            return LBM_ERR_INVALID_ARG;
        BatchInstance& I = inst[k];
        I.a.nx = d.nx;
        I.a.ny = d.ny;
        I.a.pitch = (d.nx + align_elems - 1) / align_elems * align_elems;
        I.a.nseg = 0;
        I.a.plane = (long long)d.ny * I.a.pitch;
        I.a.w_nu = r.omega_nu;
        I.a.w3 = d.model == LBM_PR ? 1.0 : r.omega3;
        I.a.w4 = d.model == LBM_PR ? 1.0 : r.omega4;
        I.a.rho0 = rho0;
        I.a.urx = d.ux_ref;
        I.a.ury = d.uy_ref;
        // the cumulant readings LBM_K_PRE / LBM_K_EQ: the kernels of LBM_K, other constants
        I.a.kread = d.model == LBM_K_PRE ? 1 : (d.model == LBM_K_EQ ? 2 : 0);
        lbm::fill_consts(I.a);
        I.model = (d.model == LBM_K_PRE || d.model == LBM_K_EQ) ? LBM_K : d.model;
        I.march_from = lbm::kNeverMarch;
        I.ke_ref = d.ke_ref;
        I.ke_factor = d.ke_factor;
        I.eq = lbm::equilibrium_consts(d.ux_ref, d.uy_ref);
        off = (off + 127) / 128 * 128;   // 256-byte aligned or better for every storage type
        I.off = off;
        off += 2 * 9 * I.a.plane;
        node_off[k] = nodes;
        nodes += (long long)d.nx * d.ny;
    }
    lbm_batch* b = new (std::nothrow) lbm_batch();
    if (!b) return LBM_ERR_NOMEM;
    b->n = n;
    b->storage = storage;
    b->rho0 = rho0;
    b->stream = (cudaStream_t)cuda_stream;
    b->inst = inst;
    b->node_off = node_off;
    b->nodes = nodes;
    b->slab_bytes = (size_t)off * esz;
    // largest instances first (longest-processing-time order for the dynamic queue)
    std::vector<int> order(n);
    std::iota(order.begin(), order.end(), 0);
    std::stable_sort(order.begin(), order.end(), [&](int a, int c) {
        return (long long)inst[a].a.nx * inst[a].a.ny > (long long)inst[c].a.nx * inst[c].a.ny;
    });
    int rc = LBM_OK;
    cudaError_t e = cudaMalloc(&b->slab, b->slab_bytes);
    if (e == cudaSuccess) e = cudaMemsetAsync(b->slab, 0, b->slab_bytes, b->stream);
    if (e == cudaSuccess) e = cudaMalloc(&b->d_inst, sizeof(BatchInstance) * n);
    if (e == cudaSuccess) e = cudaMalloc(&b->d_state, sizeof(BatchState) * n);
    if (e == cudaSuccess) e = cudaMalloc(&b->d_order, sizeof(int) * n);
    if (e == cudaSuccess) e = cudaMalloc(&b->d_queue, sizeof(int));
    if (e == cudaSuccess) e = cudaMalloc(&b->d_node_off, sizeof(long long) * n);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(b->d_inst, inst.data(), sizeof(BatchInstance) * n, cudaMemcpyHostToDevice, b->stream);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(b->d_order, order.data(), sizeof(int) * n, cudaMemcpyHostToDevice, b->stream);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(b->d_node_off, node_off.data(), sizeof(long long) * n, cudaMemcpyHostToDevice, b->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(b->stream);
    if (e != cudaSuccess) {
        rc = e == cudaErrorMemoryAllocation ? LBM_ERR_NOMEM : LBM_ERR_CUDA;
    } else {
        rc = reset_states(b);
        b->order = order;
        for (const BatchInstance& I : inst) b->models = b->models || I.model != inst[0].model;
        if (rc == LBM_OK) rc = choose_shape(b, 100);
    }
    if (rc != LBM_OK) {
        lbm_batch_destroy(b);
        return rc;
    }
    *out = b;
    return LBM_OK;
}

void lbm_batch_destroy(lbm_batch* b) {
    if (!b) return;
    cudaStreamSynchronize(b->stream);
    if (b->exec) cudaGraphExecDestroy(b->exec);
    cudaFree(b->slab);
    cudaFree(b->d_inst);
    cudaFree(b->d_state);
    cudaFree(b->d_order);
    cudaFree(b->d_queue);
    cudaFree(b->d_node_off);
    cudaFree(b->stage);
    delete b;
}

long long lbm_batch_nodes(const lbm_batch* b) { return b ? b->nodes : -1; }

int lbm_batch_init_equilibrium(lbm_batch* b, const double* rho, const double* ux, const double* uy) {
    if (!b || !rho || !ux || !uy) return b ? berr(b, LBM_ERR_INVALID_ARG, "null field") : LBM_ERR_INVALID_ARG;
    int rc = reset_states(b);
    if (rc) return rc;
    const double* in[3] = {rho, ux, uy};
    const double* dev[3];
    const size_t n = (size_t)b->nodes;
    for (int k = 0; k < 3; ++k) {
        if (is_device_ptr(in[k])) {
            dev[k] = in[k];
            continue;
        }
        if (b->stage_elems < 3 * n) {
            cudaFree(b->stage);
            b->stage = nullptr;
            b->stage_elems = 0;
            LBM_BCK(b, cudaMalloc(&b->stage, 3 * n * sizeof(double)));
            b->stage_elems = 3 * n;
        }
        LBM_BCK(b, cudaMemcpyAsync(b->stage + k * n, in[k], n * sizeof(double), cudaMemcpyHostToDevice, b->stream));
        dev[k] = b->stage + k * n;
    }
    LBM_BCK(b, launch_batch_init(b, dev[0], dev[1], dev[2]));
    LBM_BCK(b, cudaStreamSynchronize(b->stream));
    return LBM_OK;
}

int lbm_batch_run(lbm_batch* b, long long target_steps, int check_every, double growth) {
    if (!b) return LBM_ERR_INVALID_ARG;
    if (target_steps < 0 || check_every < 0 || !(growth > 1.0) || !std::isfinite(growth))
        return berr(b, LBM_ERR_INVALID_ARG, "invalid run parameters");
    int rc = choose_shape(b, check_every);
    if (rc) return rc;
    rc = record_run(b, target_steps, check_every, growth);
    if (rc) return rc;
    LBM_BCK(b, cudaGraphLaunch(b->exec, b->stream));
    return LBM_OK;
}

int lbm_batch_status(lbm_batch* b, int* status, long long* blowup_step, long long* steps, double* diag4) {
    if (!b) return LBM_ERR_INVALID_ARG;
    std::vector<BatchState> s(b->n);
    LBM_BCK(b, cudaMemcpyAsync(s.data(), b->d_state, sizeof(BatchState) * b->n, cudaMemcpyDeviceToHost, b->stream));
    LBM_BCK(b, cudaStreamSynchronize(b->stream));
    for (int k = 0; k < b->n; ++k) {
        if (status) status[k] = s[k].status;
        if (blowup_step) blowup_step[k] = s[k].blowup_step;
        if (steps) steps[k] = s[k].steps;
        if (diag4) {
            diag4[4 * k + 0] = s[k].pert;
            diag4[4 * k + 1] = s[k].ke;
            diag4[4 * k + 2] = s[k].rho_min;
            diag4[4 * k + 3] = s[k].pert0;
        }
    }
    return LBM_OK;
}

int lbm_batch_get_populations(lbm_batch* b, int index, double* f) {
    if (!b || !f || index < 0 || index >= b->n)
        return b ? berr(b, LBM_ERR_INVALID_ARG, "bad instance index or null output") : LBM_ERR_INVALID_ARG;
    const BatchInstance& I = b->inst[index];
    lbm::FieldArgs a;
    a.nx = I.a.nx; a.ny = I.a.ny; a.pitch = I.a.pitch; a.plane = I.a.plane; a.rho0 = I.a.rho0;
    a.urx = I.a.urx; a.ury = I.a.ury;
    // the kernel reads which of the two buffers is current: no round trip to the host before it
    a.which = &b->d_state[index].cur;
    a.other = 9 * I.a.plane;
    const char* base = static_cast<const char*>(b->slab) + (size_t)I.off * lbm::storage_bytes(b->storage);
    const size_t n = (size_t)I.a.nx * I.a.ny;
    double* dst = f;
    double* tmp = nullptr;
    if (!is_device_ptr(f)) {
        LBM_BCK(b, cudaMalloc(&tmp, 9 * n * sizeof(double)));
        dst = tmp;
    }
    cudaError_t e = lbm::launch_gather(b->storage, base, a, dst, nullptr, nullptr, nullptr, nullptr, nullptr,
                                       nullptr, b->stream);
    if (e == cudaSuccess && tmp) e = cudaMemcpyAsync(f, tmp, 9 * n * sizeof(double), cudaMemcpyDeviceToHost, b->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(b->stream);
    if (tmp) cudaFree(tmp);
    if (e != cudaSuccess) return berr(b, LBM_ERR_CUDA, "get_populations: %s", cudaGetErrorString(e));
    return LBM_OK;
}

int lbm_batch_set_shape(lbm_batch* b, int vec, int block) {
    if (!b) return LBM_ERR_INVALID_ARG;
    return ask_shape(b, vec, block);
}

int lbm_batch_get_shape(const lbm_batch* b, int* vec, int* block, int* grid) {
    if (!b) return LBM_ERR_INVALID_ARG;
    if (vec) *vec = b->vec;
    if (block) *block = b->block;
    if (grid) *grid = b->grid;
    return LBM_OK;
}

int lbm_batch_autotune(lbm_batch* b, long long trial_steps, int check_every, int* vec, int* block, double* best_ms) {
    if (!b || trial_steps < 1 || check_every < 0) return b ? berr(b, LBM_ERR_INVALID_ARG, "bad trial") : LBM_ERR_INVALID_ARG;
    static const int cand[][2] = {{2, 128}, {2, 256}, {2, 512}, {4, 128}, {4, 256}, {4, 512}, {8, 128}, {8, 256}, {8, 512}};
    // save the state, time each shape from it, restore it after every trial
    std::vector<BatchState> s0(b->n);
    LBM_BCK(b, cudaMemcpyAsync(s0.data(), b->d_state, sizeof(BatchState) * b->n, cudaMemcpyDeviceToHost, b->stream));
    LBM_BCK(b, cudaStreamSynchronize(b->stream));
    long long start = 0;
    for (const auto& x : s0) start = std::max(start, x.steps);
    void* saved = nullptr;
    LBM_BCK(b, cudaMalloc(&saved, b->slab_bytes));
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    cudaEventCreate(&e0);
    cudaEventCreate(&e1);
    cudaError_t e = cudaMemcpyAsync(saved, b->slab, b->slab_bytes, cudaMemcpyDeviceToDevice, b->stream);
    const int v0 = b->vec, k0 = b->block;
    int best_v = v0, best_b = k0;
    double best = 1e300;
    int rc = LBM_OK;
    for (const auto& c : cand) {
        if (e != cudaSuccess) break;
        if (!pick_batch_kernel(b->storage, c[0], c[1], false)) continue;
        if (ask_shape(b, c[0], c[1]) != LBM_OK || choose_shape(b, check_every) != LBM_OK) continue;
        rc = record_run(b, start + trial_steps, check_every, 1e4);
        if (rc != LBM_OK) break;
        cudaEventRecord(e0, b->stream);
        e = cudaGraphLaunch(b->exec, b->stream);
        cudaEventRecord(e1, b->stream);
        if (e == cudaSuccess) e = cudaStreamSynchronize(b->stream);
        float ms = 0.f;
        if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, e0, e1);
        if (e == cudaSuccess && ms < best) { best = ms; best_v = c[0]; best_b = c[1]; }
        if (e == cudaSuccess) e = cudaMemcpyAsync(b->slab, saved, b->slab_bytes, cudaMemcpyDeviceToDevice, b->stream);
        if (e == cudaSuccess)
            e = cudaMemcpyAsync(b->d_state, s0.data(), sizeof(BatchState) * b->n, cudaMemcpyHostToDevice, b->stream);
        if (e == cudaSuccess) e = cudaStreamSynchronize(b->stream);
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    cudaFree(saved);
    if (rc != LBM_OK) return rc;
    if (e != cudaSuccess) return berr(b, LBM_ERR_CUDA, "autotune: %s", cudaGetErrorString(e));
    rc = ask_shape(b, best_v, best_b);
    if (rc) return rc;
    if (vec) *vec = best_v;
    if (block) *block = best_b;
    if (best_ms) *best_ms = best;
    return LBM_OK;
}

}  // extern "C"
