// lb_api.cu — the C ABI of liblbsc.so (include/lb.h): parameter validation,
// device memory of a state, launch sequencing on the caller's stream, and
// host<->device transfers at the boundary.
#include <cmath>
#include <cstdlib>
#include <cstring>
#include <atomic>
#include <new>
#include <vector>

#include "lb_internal.h"

using namespace lbsc;

namespace lbsc {

// Test hook: allocations left before one is made to fail (-1: never).
static std::atomic<int> g_fail_allocs_after{-1};

// Allocate blocks of at most kBlockBytes for whole buffers in order (a larger buffer is a
// block of its own) and set up their guards; nothing is allocated if that fails.
static bool alloc_blocks(lb_state* s, const std::vector<Buffer>& buffers)
{
    const size_t had_allocs = s->allocs.size(), had_blocks = s->blocks.size();
    auto room = [](const Buffer& b) { return guarded_size(b.bytes) + 2 * kGuardBytes; };
    bool ok = true;
    for (size_t k = 0; ok && k < buffers.size();) {
        size_t end = k + 1, total = room(buffers[k]);
        while (end < buffers.size() && total + room(buffers[end]) <= kBlockBytes)
            total += room(buffers[end++]);
        void* block = nullptr;
        ok = cudaMalloc(&block, total) == cudaSuccess;
        if (!ok) break;
        s->blocks.push_back(block);
        // the guards: one fill over small buffers and all, otherwise one at each end and
        // where two buffers meet
        char* at = static_cast<char*>(block);
        auto fill = [&](char* p, size_t n) {
            ok = ok && cudaMemsetAsync(p, kGuardByte, n, s->stream) == cudaSuccess;
        };
        const bool small = total <= (64u << 10);
        fill(at, small ? total : kGuardBytes);
        for (; k < end; ++k) {
            const size_t body = guarded_size(buffers[k].bytes);
            *buffers[k].ptr = at + kGuardBytes;
            s->allocs.push_back({at, body});
            if (!small) fill(at + kGuardBytes + body, (k + 1 < end ? 2 : 1) * kGuardBytes);
            at += body + 2 * kGuardBytes;
        }
    }
    if (ok) return true;
    cudaGetLastError();
    for (size_t k = had_blocks; k < s->blocks.size(); ++k) cudaFree(s->blocks[k]);
    s->blocks.resize(had_blocks);
    s->allocs.resize(had_allocs);
    for (const Buffer& b : buffers) *b.ptr = nullptr;
    return false;
}

bool state_alloc(lb_state* s, std::vector<Buffer> buffers, size_t spare)
{
    const size_t needed = buffers.size() - spare;
    auto leave_out_spare = [&]() {
        for (; buffers.size() > needed; buffers.pop_back()) *buffers.back().ptr = nullptr;
    };
    for (size_t k = 0; k < buffers.size(); ++k) {
        int left = g_fail_allocs_after.load();
        while (left >= 0 && !g_fail_allocs_after.compare_exchange_weak(left, left - 1)) {
        }
        if (left != 0) continue;
        // the hook's failure (counter is now -1: disarmed)
        if (k < needed) return false;
        leave_out_spare();
    }
    if (alloc_blocks(s, buffers)) return true;
    if (buffers.size() == needed) return false;
    leave_out_spare();
    return alloc_blocks(s, buffers);
}

Couplings couplings(double G1, double G2)
{
    // Table 1 weights; p_s0 = 1 - sum of the 24 link weights (Eq. weights_1)
    const double p1 = 4.0 / 63.0, p2 = 4.0 / 135.0, p4 = 1.0 / 180.0, p5 = 2.0 / 945.0,
                 p8 = 1.0 / 15120.0;
    const double p0 = 1.0 - (4 * p1 + 4 * p2 + 4 * p4 + 8 * p5 + 4 * p8);
    Couplings c;
    c.K0 = G1 * (4.0 / 9.0) + G2 * p0;
    c.K1 = G1 * (1.0 / 9.0) + G2 * p1;
    c.K2 = G1 * (1.0 / 36.0) + G2 * p2;
    c.K4 = G2 * p4;
    c.K5 = G2 * p5;
    c.K8 = G2 * p8;
    return c;
}

// Where a kernel can read or write an array directly: device (or managed) memory
// as it is, pinned host memory through its device alias (read or written over
// the host link by the kernel, no staging copy); nullptr for pageable host memory.
double* device_view(double* p)
{
    if (!p) return nullptr;
    cudaPointerAttributes at;
    if (cudaPointerGetAttributes(&at, p) != cudaSuccess) {
        cudaGetLastError();
        return nullptr;
    }
    if (at.type == cudaMemoryTypeDevice || at.type == cudaMemoryTypeManaged) return p;
    if (at.type == cudaMemoryTypeHost && at.devicePointer)
        return static_cast<double*>(at.devicePointer);
    return nullptr;
}

}  // namespace lbsc

namespace {

lb_status validate(const lb_params* p)
{
    if (!p) return LB_ERR_ARG;
    if (p->nx < 5 || p->ny < 5) return LB_ERR_ARG;
    if ((long long)p->nx * p->ny * 9 >= (1LL << 31)) return LB_ERR_ARG;
    if (g_elems(p->nx, p->ny) >= (1LL << 31)) return LB_ERR_ARG;   // 32-bit indices in the steps
    if (!(p->omega > 0.0 && p->omega < 2.0)) return LB_ERR_ARG;
    if (!std::isfinite(p->G1) || !std::isfinite(p->G2)) return LB_ERR_ARG;
    if (!(p->rho0 > 0.0) || !std::isfinite(p->rho0)) return LB_ERR_ARG;
    if (p->psi_form != LB_PSI_SC_EXP) return LB_ERR_ARG;
    if (p->prec != LB_FP32 && p->prec != LB_FP64 && p->prec != LB_FP16_DELTA) return LB_ERR_ARG;
    if (p->trace_every < 0) return LB_ERR_ARG;
    if (!std::isfinite(p->rho_ref)) return LB_ERR_ARG;
    if (p->device < 0) return LB_ERR_ARG;
    return LB_OK;
}

// Default launch shape: the register-prefetch pipeline (measured faster than
// the bulk-copy rings on GB300 for the 8192^2 lattice; the tuner may still pick
// the rings) with 128-thread strips, or 64-thread strips for lattices whose
// state fits in L2 (512^2: 11.1 us per step against 12.5 us); rows chosen for
// about five waves of 40 resident warps per SM on a 152-SM part (8192^2: 72
// rows, 4.95 waves, the tuned shape), at least 8
// (small lattices have few columns, so short chunks are what gives them enough
// CTAs: 512^2 steps in 11.1 us with 8-row chunks against 15.2 us with 16).
Fp32Launch default_launch(int nx, int ny, lb_precision prec)
{
    (void)prec;
    Fp32Launch L{128, 64, 0};
    if (!beyond_l2((long long)nx * ny)) L.block_x = 64;
    const long long strips = (nx + L.block_x - 3) / (L.block_x - 2);
    const long long target = 152LL * (40 * 32 / L.block_x) * 5;
    long long rows = (strips * ny + target - 1) / target;
    if (rows < 8) rows = 8;
    if (rows > 512) rows = 512;
    L.rows = (int)rows;
    return L;
}

// CTA count of a launch shape (the CTA-partial buffer is sized for the largest)
size_t step_blocks(const lb_state* s, Fp32Launch L)
{
    if (L.pipeline == 1)
        return (size_t)bulk_grid_blocks(s->p.nx, s->p.ny, (int)elem_size(s->p.prec), L);
    return (size_t)fp32_grid_blocks(s->p.nx, s->p.ny, L);
}

template <typename T>
StepArgs<T> make_args(const lb_state* s)
{
    return lbsc::state_args<T>(s, s->cur);
}

}  // namespace

namespace lbsc {

template <typename T>
StepArgs<T> state_args(const lb_state* s, int cur)
{
    const lb_params& p = s->p;
    const Couplings K = couplings(p.G1, p.G2);
    StepArgs<T> a{};
    a.g_in = static_cast<const T*>(s->g[cur]);
    a.g_out = static_cast<T*>(s->g[cur ^ 1]);
    a.dpsi_in = s->dpsi[cur];
    a.dpsi_out = s->dpsi[cur ^ 1];
    a.nx = p.nx;
    a.ny = p.ny;
    a.rows = s->launch.rows;
    a.N = s->N;
    a.pitch = g_pitch(p.nx);
    a.npitch = (int)g_elems(p.nx, p.ny);
    a.omega = (float)p.omega;
    a.omc = (float)(1.0 - p.omega);
    a.inv_omega = (float)(1.0 / p.omega);
    a.w0 = (float)(4.0 / 9.0);
    a.w1 = (float)(1.0 / 9.0);
    a.w2 = (float)(1.0 / 36.0);
    a.K0 = (float)K.K0;
    a.K1 = (float)K.K1;
    a.K2 = (float)K.K2;
    a.K4 = (float)K.K4;
    a.K5 = (float)K.K5;
    a.K8 = (float)K.K8;
    a.rho_ref = (float)s->rho_ref;
    a.psi_ref = (float)(std::sqrt(p.rho0) * -std::expm1(-s->rho_ref / p.rho0));
    a.cpsi = (float)(-std::sqrt(p.rho0) * std::exp(-s->rho_ref / p.rho0));
    a.inv_rho0 = (float)(1.0 / p.rho0);
    a.half_A1 = (float)(0.5 * (p.G1 + p.G2));
    a.partials = s->partials;
    a.counter = s->counter;
    a.trace = s->trace;
    a.trace_count = s->trace_count;
    a.t = s->t;
    a.err = s->err;
    a.wait_cycles = s->wait_cycles;
    a.skip_unit0 = s->skip_unit0;
    a.dev = s->dev;
    return a;
}

template StepArgs<float> state_args<float>(const lb_state*, int);
template StepArgs<__half> state_args<__half>(const lb_state*, int);

size_t elem_size(lb_precision p) { return p == LB_FP16_DELTA ? 2 : 4; }

}  // namespace lbsc

namespace {

lb_status fail_cuda(lb_state* s)
{
    if (s) s->poisoned = true;
    cudaGetLastError();
    return LB_ERR_CUDA;
}

// The state's control words into c (synchronises the stream): a strided copy of the words
// without the guards between them (13.9 us with a kernel before it, 15.9 us for all bytes).
cudaError_t copy_control(lb_state* s, Control& c)
{
    char h[4][sizeof(c.res)];
    cudaError_t e = cudaMemcpy2DAsync(h, sizeof(h[0]), s->res, kControlPitch, sizeof(h[0]), 4,
                                      cudaMemcpyDeviceToHost, s->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s->stream);
    if (e != cudaSuccess) return e;
    std::memcpy(c.res, h[0], sizeof(c.res));
    std::memcpy(&c.err, h[1], sizeof(int));
    std::memcpy(&c.trace_count, h[2], sizeof(int));
    std::memcpy(&c.flag, h[3], sizeof(int));
    return cudaSuccess;
}

// Read them and the kernels' error flags among them: bit 1, a bounded wait ran out (the
// state is poisoned); bit 2, a fused reduction produced a non-finite mass or energy (the
// lattice has blown up).
lb_status read_control(lb_state* s, Control& c)
{
    if (copy_control(s, c) != cudaSuccess) return fail_cuda(s);
    if (c.err & 1) {
        s->poisoned = true;
        return LB_ERR_TIMEOUT;
    }
    return c.err & 2 ? LB_ERR_NONFINITE : LB_OK;
}

lb_status check_err(lb_state* s)
{
    Control c;
    return read_control(s, c);
}

#define LB_CUDA(s, call)                          \
    do {                                          \
        if ((call) != cudaSuccess) return fail_cuda(s); \
    } while (0)

void free_state(lb_state* s)
{
    if (!s) return;
    DeviceScope dev(s->p.device);
    cudaStreamSynchronize(s->stream);
    for (void* b : s->blocks) cudaFree(b);
    cudaGetLastError();
    delete s;
}

// Steps of a small lattice that stay on the SMs (lb_resident.cu), as many per launch as the
// trace rows they append can be kept. `left` receives the steps not taken: too few for a
// launch at the end, or all from the launch on that the stream refused.
lb_status step_held(lb_state* s, long n, long& left)
{
    ResidentBuf& b = s->res_buf;
    const int least = held_least(b.tw * b.th, (float)s->p.omega == 1.0f);
    while (left = n, n >= least) {
        long m = n;
        if (b.trace_every > 0) {
            const long long te = b.trace_every;
            const long long first = (s->t + te - 1) / te * te;   // next trace row
            const long long room = first + te * b.max_rows - s->t;
            if (m > room) m = (long)room;
        }
        if (m > (1L << 20)) m = 1L << 20;
        if (s->in_graphs && m % 2 == 0) --m;   // a launch swaps the buffers once
        if (m < least) return LB_OK;
        const cudaError_t e =
            s->p.prec == LB_FP32
                ? fp32_resident(make_args<float>(s), b, s->launch.block_x, (int)m, s->stream)
                : fp16_resident(make_args<__half>(s), b, s->launch.block_x, (int)m, s->stream);
        if (launch_refused(e)) {
            cudaGetLastError();
            b.gx = 0;
            return LB_OK;
        }
        if (e != cudaSuccess) return fail_cuda(s);
        s->cur ^= 1;
        s->t += m;
        n -= m;
    }
    return LB_OK;
}

// Steps t and t + 1, and the trace row of state t if it has one.
template <typename T>
cudaError_t pair_step(lb_state* s, bool traced)
{
    const StepArgs<T> a = make_args<T>(s);
    cudaError_t e;
    if constexpr (sizeof(T) == 4) e = fp32_step_pair(a, traced, s->stream);
    else e = fp16_step_pair(a, traced, s->stream);
    if (e != cudaSuccess || !traced) return e;
    const TraceRows r{a.dpsi_in, a.dev, 0, 1, s->t, 1, s->launch.block_x, s->partials, s->counter};
    return trace_rows<T>(a, r, s->stream);
}

// n steps in launches of their own or (`pairs`) two at a time (lb_pair.cu): the same
// fields bit for bit, half the memory traffic.
lb_status step_streamed(lb_state* s, long n, bool pairs)
{
    const int te = s->p.trace_every;
    const bool bulk = s->launch.pipeline == 1;
    pairs = pairs && pairs_pay(s->p.nx, s->p.ny, s->launch.block_x, (int)elem_size(s->p.prec));
    // one pair fewer if the buffers would not swap as single steps swap them
    const bool traced = s->dev && traced_pairs_pay(s->p.nx, s->p.ny, s->launch.block_x,
                                                   (int)elem_size(s->p.prec));
    int singles = pairs && s->in_graphs && pairs_made(s->t, n, te, traced) % 2 != 0 ? 2 : 0;
    while (n > 0) {
        const bool reduce = te > 0 && s->t % te == 0;
        bool pair = pairs && pair_at(s->t, n, te, traced);
        if (singles == 1 || (singles == 2 && pair)) {
            --singles;
            pair = false;
        }
        cudaError_t e;
        if (s->p.prec == LB_FP32)
            e = pair   ? pair_step<float>(s, reduce)
                : bulk ? fp32_step_bulk(make_args<float>(s), s->launch, reduce, s->stream)
                       : fp32_step(make_args<float>(s), s->launch, reduce, s->stream);
        else
            e = pair   ? pair_step<__half>(s, reduce)
                : bulk ? fp16_step_bulk(make_args<__half>(s), s->launch, reduce, s->stream)
                       : fp16_step(make_args<__half>(s), s->launch, reduce, s->stream);
        if (e != cudaSuccess) return fail_cuda(s);
        s->cur ^= 1;
        s->t += pair ? 2 : 1;
        n -= pair ? 2 : 1;
    }
    return LB_OK;
}

lb_status step_fp32(lb_state* s, long n)
{
    // in a stream capture every step is a launch of its own, so that a graph of an even
    // number of steps can be replayed: each step swaps the buffers once
    const bool captures = stream_captures(s->stream);
    s->in_graphs = s->in_graphs || (captures && n > 0);
    const bool many = n >= 2 && s->launch.pipeline == 0 && !captures;
    if (many && s->res_buf.gx > 0) {
        const lb_status st = step_held(s, n, n);
        if (st != LB_OK || n == 0) return st;
    }
    return step_streamed(s, n, many);
}

}  // namespace

lb_status lbsc::advance_delta(lb_state* s, long n) { return step_fp32(s, n); }

namespace {

Fp64Args make64(const lb_state* s)
{
    Fp64Args a;
    a.f_in = s->f64[s->cur];
    a.f_out = s->f64[s->cur ^ 1];
    a.psi = s->psi64;
    a.rho = s->rho64;
    a.nx = s->p.nx;
    a.ny = s->p.ny;
    a.omega = s->p.omega;
    a.G1 = s->p.G1;
    a.G2 = s->p.G2;
    a.rho0 = s->p.rho0;
    return a;
}

lb_status step_fp64(lb_state* s, long n)
{
    for (long k = 0; k < n; ++k) {
        const Fp64Args a = make64(s);
        LB_CUDA(s, fp64_psi(a, s->stream));
        if (s->p.trace_every > 0 && (s->t % s->p.trace_every) == 0)
            LB_CUDA(s, fp64_energy(a, s->partials, s->counter, s->res, s->trace, s->trace_count,
                                   s->t, s->stream));
        LB_CUDA(s, fp64_collide_stream(a, s->stream));
        s->cur ^= 1;
        s->t += 1;
    }
    return LB_OK;
}

}  // namespace

extern "C" {

const char* lb_status_str(lb_status st)
{
    switch (st) {
    case LB_OK: return "ok";
    case LB_ERR_ARG: return "invalid argument";
    case LB_ERR_CUDA: return "CUDA error (state poisoned)";
    case LB_ERR_OOM: return "device allocation failed";
    case LB_ERR_NONFINITE: return "non-finite density or energy";
    case LB_ERR_STATE: return "call not valid in the current state";
    case LB_ERR_TIMEOUT: return "an in-kernel wait ran out (state poisoned)";
    }
    return "unknown status";
}

lb_status lb_init(lb_state** out, const lb_params* p, const double* rho_init, void* stream)
{
    NvtxRange nvtx_range("lb_init");
    return lbsc::state_init(out, p, rho_init, stream, true);
}

}  // extern "C"

lb_status lbsc::state_init(lb_state** out, const lb_params* p, const double* rho_init, void* stream,
                           bool alone)
{
    if (!out) return LB_ERR_ARG;
    *out = nullptr;
    if (validate(p) != LB_OK || !rho_init) return LB_ERR_ARG;
    lb_state* s = new (std::nothrow) lb_state();
    if (!s) return LB_ERR_OOM;
    s->p = *p;
    s->stream = static_cast<cudaStream_t>(stream);
    s->N = (long long)p->nx * p->ny;
    const long long N = s->N;
    DeviceScope dev(p->device);
    if (!dev.ok) {
        delete s;
        return LB_ERR_CUDA;
    }
    s->launch = default_launch(p->nx, p->ny, p->prec);
    size_t nblk_step = (size_t)fp32_grid_blocks(p->nx, p->ny, Fp32Launch{64, kMinRows, 0});
    const size_t nblk_bulk =
        (size_t)bulk_grid_blocks(p->nx, p->ny, (int)elem_size(p->prec), Fp32Launch{64, kMinRows, 1});
    if (nblk_bulk > nblk_step) nblk_step = nblk_bulk;
    s->partials_cap = nblk_step > 152 * 16 ? nblk_step : 152 * 16;
    // the reduction step's grid sum keeps one total per CTA row after the CTA partials
    s->max_cta_rows = (p->ny + kMinRows - 1) / kMinRows;
    s->partials_cap += (size_t)s->max_cta_rows;
    // the control words first, at the distances that kControlPitch states; cleared below
    std::vector<Buffer> buffers = {{(void**)&s->res, 4 * sizeof(double)},
                                   {(void**)&s->err, sizeof(int)},
                                   {(void**)&s->trace_count, sizeof(int)},
                                   {(void**)&s->flag, sizeof(int)},
                                   {(void**)&s->counter, 2 * sizeof(unsigned int)},
                                   {(void**)&s->partials, 4 * sizeof(double) * s->partials_cap},
                                   {(void**)&s->trace, sizeof(double) * kTraceCap * kTraceCols}};
    auto add = [&](auto** ptr, size_t bytes) { buffers.push_back({(void**)ptr, bytes}); };
    if (p->prec == LB_FP64) {
        add(&s->f64[0], 9 * sizeof(double) * N);
        add(&s->f64[1], 9 * sizeof(double) * N);
        add(&s->psi64, sizeof(double) * N);
        add(&s->rho64, sizeof(double) * N);
    } else {
        const size_t gb = elem_size(p->prec) * (size_t)g_elems(p->nx, p->ny);
        add(&s->g[0], gb);
        add(&s->g[1], gb);
        add(&s->dpsi[0], sizeof(float) * N);
        add(&s->dpsi[1], sizeof(float) * N);
    }
    // what only faster ways to step need: without the memory for it the state does without
    const size_t needed = buffers.size();
    if (p->prec != LB_FP64 && p->trace_every > 0) add(&s->dev, sizeof(float) * N);
    ResidentBuf& rb = s->res_buf;
    size_t words4 = 0, words2 = 0;   // bytes of the halo words
    if (alone && p->prec != LB_FP64) {
        int sms = 0;
        const bool om1 = (float)p->omega == 1.0f;
        if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, p->device) != cudaSuccess) {
            cudaGetLastError();
            sms = 0;
        }
        if (resident_plan(p->nx, p->ny, om1, sms, rb)) {
            rb.trace_every = p->trace_every;
            words4 = sizeof(uint4) * 2 * (om1 ? 1 : 3) * (size_t)N;
            words2 = sizeof(uint2) * 2 * (size_t)N;
            add(&rb.llm, words4);
            add(&rb.llp, words2);
            if (p->trace_every > 0) {
                const long long rows = (8LL << 20) / (8 * N);
                const int least = held_least(rb.tw * rb.th, om1) + 1;   // a launch at every state traced
                rb.max_rows = (int)(rows < least ? least : rows > 16 ? 16 : rows);
                // partials of one trace row: of the smallest CTAs a shape may have, and CTA rows
                const size_t row_cap =
                    (size_t)fp32_grid_blocks(p->nx, p->ny, Fp32Launch{64, kMinRows, 0}) +
                    (size_t)s->max_cta_rows;
                add(&rb.counters, sizeof(unsigned int) * (1 + (size_t)rb.max_rows));
                add(&rb.partials, (size_t)rb.max_rows * 4 * sizeof(double) * row_cap);
                add(&rb.dump, (size_t)rb.max_rows * 2 * sizeof(float) * N);
            }
        }
    }
    const bool ok = state_alloc(s, buffers, buffers.size() - needed);
    if (!rb.llm) rb = ResidentBuf{};
    if (!ok) {
        free_state(s);
        return LB_ERR_OOM;
    }
    // rho_init is copied once (one DMA transfer, whatever memory it is in) into the
    // second population buffer, which holds nothing until the first step writes it
    // and is at least 8 N bytes in every precision; the checks and the
    // initialisation then read device memory only.
    double* rho_in = static_cast<double*>(p->prec == LB_FP64 ? (void*)s->f64[1] : s->g[1]);
    auto bail = [&](lb_status st) {
        cudaGetLastError();
        free_state(s);
        return st;
    };
    if (cudaMemcpyAsync(rho_in, rho_init, sizeof(double) * N, cudaMemcpyDefault, s->stream) !=
            cudaSuccess ||
        cudaMemset2DAsync(s->res, kControlPitch, 0, kGuardBytes, 5, s->stream) != cudaSuccess ||
        (rb.gx > 0 && (cudaMemsetAsync(rb.llm, 0, words4, s->stream) != cudaSuccess ||
                       cudaMemsetAsync(rb.llp, 0, words2, s->stream) != cudaSuccess)) ||
        (rb.counters && cudaMemsetAsync(rb.counters, 0, kGuardBytes, s->stream) != cudaSuccess))
        return bail(LB_ERR_CUDA);
    if (rho_check_sum(rho_in, N, s->partials, s->counter, s->res, s->flag, s->stream) !=
        cudaSuccess)
        return bail(LB_ERR_CUDA);
    Control got{};
    // after this synchronisation the caller's rho_init is no longer read
    if (copy_control(s, got) != cudaSuccess) return bail(LB_ERR_CUDA);
    const double sum = got.res[0];
    if (got.flag) return bail(LB_ERR_ARG);
    // The reference density is rounded to FP32 once: the kernels add it in FP32,
    // the deviations at init and the mass/field reconstructions use it in FP64,
    // and all of them must mean the same number.
    s->rho_ref = (double)(float)(p->rho_ref > 0.0 ? p->rho_ref : sum / (double)N);
    const bool padded = p->prec != LB_FP64 && g_pitch(p->nx) != 9 * p->nx;
    const size_t gbytes = elem_size(p->prec) * (size_t)g_elems(p->nx, p->ny);
    if (padded && cudaMemsetAsync(s->g[0], 0, gbytes, s->stream) != cudaSuccess)
        return bail(LB_ERR_CUDA);
    cudaError_t e;
    if (p->prec == LB_FP64)
        e = fp64_init(s->f64[0], rho_in, p->nx, p->ny, s->stream);
    else if (p->prec == LB_FP32)
        e = delta_init<float>(static_cast<float*>(s->g[0]), s->dpsi[0], rho_in, p->nx, p->ny,
                              s->rho_ref, p->rho0, s->stream);
    else
        e = delta_init<__half>(static_cast<__half*>(s->g[0]), s->dpsi[0], rho_in, p->nx, p->ny,
                               s->rho_ref, p->rho0, s->stream);
    if (e != cudaSuccess) return bail(LB_ERR_CUDA);
    // the padding columns of the tiled populations hold zeros in both buffers (nx
    // not a multiple of 32; otherwise every element of g[0] is written by the
    // initialisation and every element of g[1] by the first step); g[1] is
    // cleared after the initialisation has read rho_init from it
    if (padded && cudaMemsetAsync(s->g[1], 0, gbytes, s->stream) != cudaSuccess)
        return bail(LB_ERR_CUDA);
    *out = s;
    return LB_OK;
}

extern "C" {

lb_status lb_step(lb_state* s, long n)
{
    NvtxRange nvtx_range("lb_step");
    if (!s || n < 0) return LB_ERR_ARG;
    if (s->poisoned) return LB_ERR_STATE;
    if (n == 0) return LB_OK;
    DeviceScope dev(s->p.device);
    if (!dev.ok) return fail_cuda(s);
    return s->p.prec == LB_FP64 ? step_fp64(s, n) : step_fp32(s, n);
}

lb_status lb_energy(lb_state* s, double out[4])
{
    NvtxRange nvtx_range("lb_energy");
    if (!s || !out) return LB_ERR_ARG;
    if (s->poisoned) return LB_ERR_STATE;
    DeviceScope dev(s->p.device);
    if (!dev.ok) return fail_cuda(s);
    auto sums = [&](bool wide) -> cudaError_t {
        if (s->p.prec == LB_FP64) {
            const Fp64Args a = make64(s);
            const cudaError_t e = fp64_psi(a, s->stream);
            return e != cudaSuccess ? e
                                    : fp64_energy(a, s->partials, s->counter, s->res, nullptr, nullptr,
                                                  s->t, s->stream);
        }
        if (s->p.prec == LB_FP32) {
            const StepArgs<float> a = make_args<float>(s);
            return delta_energy<float>(a.g_in, a.dpsi_in, s->p.nx, s->p.ny, a, s->res, s->partials,
                                       s->counter, s->flag, wide, s->stream);
        }
        const StepArgs<__half> a = make_args<__half>(s);
        return delta_energy<__half>(a.g_in, a.dpsi_in, s->p.nx, s->p.ny, a, s->res, s->partials,
                                    s->counter, s->flag, wide, s->stream);
    };
    LB_CUDA(s, sums(false));
    Control c;
    lb_status st = read_control(s, c);
    if (st != LB_ERR_CUDA && c.flag) {   // beyond the range of the FP32 pairs
        LB_CUDA(s, cudaMemsetAsync(s->flag, 0, sizeof(int), s->stream));
        LB_CUDA(s, sums(true));
        st = read_control(s, c);
    }
    if (st != LB_OK) return st;
    for (int k = 0; k < 4; ++k) out[k] = c.res[k];
    for (int k = 0; k < 4; ++k)
        if (!std::isfinite(c.res[k])) return LB_ERR_NONFINITE;
    return LB_OK;
}

lb_status lb_objective(lb_state* s, const double* rho_target, double* J)
{
    NvtxRange nvtx_range("lb_objective");
    if (!s || !rho_target || !J) return LB_ERR_ARG;
    if (s->poisoned) return LB_ERR_STATE;
    DeviceScope dev(s->p.device);
    if (!dev.ok) return fail_cuda(s);
    const long long N = s->N;
    // the target where a kernel can read it: in place, or copied into the
    // state's field buffer (allocated on first use, as by lb_fields)
    const double* tgt = device_view(const_cast<double*>(rho_target));
    if (!tgt) {
        if (!s->field_tmp) {
            s->field_tmp = static_cast<double*>(state_alloc(s, sizeof(double) * N));
            if (!s->field_tmp) return LB_ERR_OOM;
        }
        LB_CUDA(s, cudaMemcpyAsync(s->field_tmp, rho_target, sizeof(double) * N,
                                   cudaMemcpyHostToDevice, s->stream));
        tgt = s->field_tmp;
    }
    double h[2] = {0.0, 0.0};
    if (s->p.prec == LB_FP64) {
        // psi and rho of the current state, the Sec. 5 sums, then the misfit
        const Fp64Args a = make64(s);
        LB_CUDA(s, fp64_psi(a, s->stream));
        LB_CUDA(s, fp64_energy(a, s->partials, s->counter, s->res, nullptr, nullptr, s->t,
                               s->stream));
        LB_CUDA(s, cudaMemcpyAsync(h, s->res, 2 * sizeof(double), cudaMemcpyDeviceToHost,
                                   s->stream));
        LB_CUDA(s, misfit64(s->rho64, tgt, N, s->partials, s->counter, s->res, s->stream));
    } else {
        // the terminal sums of lb_adjoint (same kernel, grid and order)
        LB_CUDA(s, objective_delta(s, tgt, s->res, false, s->stream));
    }
    Control c;
    lb_status st = read_control(s, c);
    if (st != LB_ERR_CUDA && c.flag) {   // beyond the range of the FP32 pairs
        LB_CUDA(s, cudaMemsetAsync(s->flag, 0, sizeof(int), s->stream));
        LB_CUDA(s, objective_delta(s, tgt, s->res, true, s->stream));
        st = read_control(s, c);
    }
    if (st == LB_ERR_CUDA) return st;
    *J = s->p.prec == LB_FP64 ? (h[0] + h[1]) + c.res[0] : c.res[0] + c.res[1];
    return st != LB_OK || std::isfinite(*J) ? st : LB_ERR_NONFINITE;
}

static cudaError_t fields_into(lb_state* s, double* r, double* x, double* y)
{
    if (s->p.prec == LB_FP64) return fp64_fields(s->f64[s->cur], s->p.nx, s->p.ny, r, x, y, s->stream);
    if (s->p.prec == LB_FP32)
        return delta_fields<float>(static_cast<const float*>(s->g[s->cur]), s->p.nx, s->p.ny,
                                   s->rho_ref, r, x, y, s->stream);
    return delta_fields<__half>(static_cast<const __half*>(s->g[s->cur]), s->p.nx, s->p.ny,
                                s->rho_ref, r, x, y, s->stream);
}

lb_status lb_fields(lb_state* s, double* rho, double* ux, double* uy)
{
    NvtxRange nvtx_range("lb_fields");
    if (!s) return LB_ERR_ARG;
    if (s->poisoned) return LB_ERR_STATE;
    DeviceScope dev(s->p.device);
    if (!dev.ok) return fail_cuda(s);
    const long long N = s->N;
    double* outs[3] = {rho, ux, uy};
    double* views[3];
    for (int k = 0; k < 3; ++k) views[k] = device_view(outs[k]);
    // every output a kernel can write directly: one pass over the populations
    if (views[0] || views[1] || views[2]) {
        if (fields_into(s, views[0], views[1], views[2]) != cudaSuccess) return fail_cuda(s);
    }
    // pageable host outputs: through a device buffer, one field at a time
    for (int k = 0; k < 3; ++k) {
        if (!outs[k] || views[k]) continue;
        if (!s->field_tmp) {
            s->field_tmp = static_cast<double*>(state_alloc(s, sizeof(double) * N));
            if (!s->field_tmp) {
                cudaGetLastError();
                s->field_tmp = nullptr;
                return LB_ERR_OOM;
            }
        }
        double* t = s->field_tmp;
        if (fields_into(s, k == 0 ? t : nullptr, k == 1 ? t : nullptr, k == 2 ? t : nullptr) !=
            cudaSuccess)
            return fail_cuda(s);
        LB_CUDA(s, cudaMemcpyAsync(outs[k], t, sizeof(double) * N, cudaMemcpyDeviceToHost,
                                   s->stream));
    }
    return check_err(s);
}

lb_status lb_trace(lb_state* s, double* buf, int cap, int* count)
{
    NvtxRange nvtx_range("lb_trace");
    if (!s || !count || cap < 0 || (cap > 0 && !buf)) return LB_ERR_ARG;
    if (s->poisoned) return LB_ERR_STATE;
    DeviceScope dev(s->p.device);
    if (!dev.ok) return fail_cuda(s);
    Control c;
    const lb_status st = read_control(s, c);
    if (st == LB_ERR_CUDA) return st;
    const int total = c.trace_count;
    const int stored = total < kTraceCap ? total : kTraceCap;
    const int n = stored < cap ? stored : cap;
    // rows total-n .. total-1, oldest first; row r lives in ring slot r % kTraceCap,
    // so the rows form at most two contiguous runs of the ring
    int done = 0;
    while (done < n) {
        const int slot = (total - n + done) % kTraceCap;
        int run = kTraceCap - slot;
        if (run > n - done) run = n - done;
        LB_CUDA(s, cudaMemcpyAsync(buf + (size_t)done * kTraceCols,
                                   s->trace + (size_t)slot * kTraceCols,
                                   sizeof(double) * kTraceCols * run, cudaMemcpyDeviceToHost,
                                   s->stream));
        done += run;
    }
    LB_CUDA(s, cudaStreamSynchronize(s->stream));
    *count = n;
    return st;
}

namespace {
struct SavedHeader {
    char magic[8];            // "LBSCSTAT"
    int version, nx, ny, prec;
    long long t;
    double rho_ref;
    long long payload;        // bytes after the header
};
constexpr int kSaveVersion = 4;   // 4: tiled populations of state t (pairs side by side, FP16 too)

size_t payload_bytes(const lb_state* s)
{
    if (s->p.prec == LB_FP64) return sizeof(double) * 9 * (size_t)s->N;
    return elem_size(s->p.prec) * (size_t)g_elems(s->p.nx, s->p.ny) +
           sizeof(float) * (size_t)s->N;
}
}  // namespace

lb_status lb_check_guards(lb_state* s, int* damaged)
{
    NvtxRange nvtx_range("lb_check_guards");
    if (!s || !damaged) return LB_ERR_ARG;
    *damaged = 0;
    DeviceScope dev(s->p.device);
    if (!dev.ok) return fail_cuda(s);
    LB_CUDA(s, cudaStreamSynchronize(s->stream));
    std::vector<unsigned char> h(2 * kGuardBytes);
    for (const lb_state::Alloc& a : s->allocs) {
        const char* b = static_cast<const char*>(a.base);
        LB_CUDA(s, cudaMemcpy(h.data(), b, kGuardBytes, cudaMemcpyDeviceToHost));
        LB_CUDA(s, cudaMemcpy(h.data() + kGuardBytes, b + kGuardBytes + a.bytes, kGuardBytes,
                              cudaMemcpyDeviceToHost));
        for (unsigned char c : h)
            if (c != kGuardByte) {
                ++*damaged;
                break;
            }
    }
    return LB_OK;
}

void lb_debug_fail_alloc(int after)
{
    lbsc::g_fail_allocs_after.store(after < 0 ? -1 : after);
}

lb_status lb_debug_damage_guard(lb_state* s, int buffer)
{
    NvtxRange nvtx_range("lb_debug_damage_guard");
    if (!s || buffer < 0 || buffer >= (int)s->allocs.size()) return LB_ERR_ARG;
    DeviceScope dev(s->p.device);
    if (!dev.ok) return fail_cuda(s);
    const lb_state::Alloc& a = s->allocs[(size_t)buffer];
    char* tail = static_cast<char*>(a.base) + kGuardBytes + a.bytes;
    LB_CUDA(s, cudaMemsetAsync(tail + 17, 0x00, 1, s->stream));
    LB_CUDA(s, cudaStreamSynchronize(s->stream));
    return LB_OK;
}

size_t lb_state_bytes(const lb_state* s)
{
    return s ? sizeof(SavedHeader) + payload_bytes(s) : 0;
}

lb_status lb_save_state(lb_state* s, void* dst, size_t bytes)
{
    NvtxRange nvtx_range("lb_save_state");
    if (!s || !dst || bytes < lb_state_bytes(s)) return LB_ERR_ARG;
    if (s->poisoned) return LB_ERR_STATE;
    DeviceScope dev(s->p.device);
    if (!dev.ok) return fail_cuda(s);
    SavedHeader h{};
    std::memcpy(h.magic, "LBSCSTAT", 8);
    h.version = kSaveVersion;
    h.nx = s->p.nx;
    h.ny = s->p.ny;
    h.prec = (int)s->p.prec;
    h.t = s->t;
    h.rho_ref = s->rho_ref;
    h.payload = (long long)payload_bytes(s);
    char* d = static_cast<char*>(dst);
    const cudaMemcpyKind k = cudaMemcpyDefault;
    LB_CUDA(s, cudaMemcpyAsync(d, &h, sizeof(h), cudaMemcpyDefault, s->stream));
    d += sizeof(h);
    if (s->p.prec == LB_FP64) {
        LB_CUDA(s, cudaMemcpyAsync(d, s->f64[s->cur], sizeof(double) * 9 * s->N, k, s->stream));
    } else {
        const size_t gb = elem_size(s->p.prec) * (size_t)g_elems(s->p.nx, s->p.ny);
        LB_CUDA(s, cudaMemcpyAsync(d, s->g[s->cur], gb, k, s->stream));
        LB_CUDA(s, cudaMemcpyAsync(d + gb, s->dpsi[s->cur], sizeof(float) * s->N, k, s->stream));
    }
    LB_CUDA(s, cudaStreamSynchronize(s->stream));
    return LB_OK;
}

lb_status lb_load_state(lb_state* s, const void* src, size_t bytes)
{
    NvtxRange nvtx_range("lb_load_state");
    if (!s || !src || bytes < sizeof(SavedHeader)) return LB_ERR_ARG;
    if (s->poisoned) return LB_ERR_STATE;
    DeviceScope dev(s->p.device);
    if (!dev.ok) return fail_cuda(s);
    SavedHeader h{};
    LB_CUDA(s, cudaMemcpyAsync(&h, src, sizeof(h), cudaMemcpyDefault, s->stream));
    LB_CUDA(s, cudaStreamSynchronize(s->stream));
    if (std::memcmp(h.magic, "LBSCSTAT", 8) != 0 || h.version != kSaveVersion ||
        h.nx != s->p.nx || h.ny != s->p.ny || h.prec != (int)s->p.prec ||
        h.payload != (long long)payload_bytes(s) || bytes < lb_state_bytes(s) || h.t < 0)
        return LB_ERR_ARG;
    if (s->p.prec != LB_FP64 && h.rho_ref != s->rho_ref) return LB_ERR_ARG;
    const char* d = static_cast<const char*>(src) + sizeof(h);
    const cudaMemcpyKind k = cudaMemcpyDefault;
    if (s->p.prec == LB_FP64) {
        LB_CUDA(s, cudaMemcpyAsync(s->f64[0], d, sizeof(double) * 9 * s->N, k, s->stream));
    } else {
        const size_t gb = elem_size(s->p.prec) * (size_t)g_elems(s->p.nx, s->p.ny);
        LB_CUDA(s, cudaMemcpyAsync(s->g[0], d, gb, k, s->stream));
        LB_CUDA(s, cudaMemcpyAsync(s->dpsi[0], d + gb, sizeof(float) * s->N, k, s->stream));
    }
    LB_CUDA(s, cudaStreamSynchronize(s->stream));
    s->cur = 0;
    s->t = h.t;
    return LB_OK;
}

lb_status lb_get_launch(const lb_state* s, int* block_x, int* rows_per_cta, int* pipeline)
{
    if (!s || !block_x || !rows_per_cta || !pipeline) return LB_ERR_ARG;
    if (s->p.prec == LB_FP64) return LB_ERR_STATE;
    *block_x = s->launch.block_x;
    *rows_per_cta = s->launch.rows;
    *pipeline = s->launch.pipeline;
    return LB_OK;
}

lb_status lb_set_launch(lb_state* s, int block_x, int rows_per_cta, int pipeline)
{
    if (!s) return LB_ERR_ARG;
    if (s->p.prec == LB_FP64) return LB_ERR_STATE;
    if (rows_per_cta < kMinRows || rows_per_cta > kMaxRows) return LB_ERR_ARG;
    if (pipeline == 0) {
        if (block_x != 64 && block_x != 96 && block_x != 128 && block_x != 192 && block_x != 256)
            return LB_ERR_ARG;
    } else if (pipeline == 1) {
        if (block_x != 64 && block_x != 128 && block_x != 256) return LB_ERR_ARG;
        if (!bulk_supported(s->p.nx, s->p.ny, (int)elem_size(s->p.prec), block_x))
            return LB_ERR_ARG;
    } else {
        return LB_ERR_ARG;
    }
    const Fp32Launch L{block_x, rows_per_cta, pipeline};
    // the CTA-partial buffer was sized for the smallest CTAs (64 threads, kMinRows rows)
    // and one row total per CTA row
    if (step_blocks(s, L) + (size_t)s->max_cta_rows > s->partials_cap) return LB_ERR_ARG;
    s->launch = L;
    return LB_OK;
}

lb_status lb_set_wait_limit(lb_state* s, long long cycles, int test_skip_copies)
{
    if (!s || cycles <= 0 || (test_skip_copies != 0 && test_skip_copies != 1)) return LB_ERR_ARG;
    s->wait_cycles = cycles;
    s->skip_unit0 = test_skip_copies;
    return LB_OK;
}

long lb_time(const lb_state* s) { return s ? (long)s->t : -1; }

void lb_destroy(lb_state* s)
{
    NvtxRange nvtx_range("lb_destroy");
    free_state(s);
}

}  // extern "C"
