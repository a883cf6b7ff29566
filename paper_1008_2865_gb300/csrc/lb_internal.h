// lb_internal.h — declarations shared by the translation units of liblbsc.so
// (state layout, launch helpers). Not installed; the public interface is
// include/lb.h.
#pragma once

#include <cuda_runtime.h>
#include <cuda_fp16.h>
#include <cstdint>
#include <utility>
#include <vector>

#include <nvtx3/nvToolsExt.h>

#include "lb.h"

namespace lbsc {

// NVTX range for the duration of an ABI call (visible in Nsight timelines).
struct NvtxRange {
    explicit NvtxRange(const char* name) { nvtxRangePushA(name); }
    ~NvtxRange() { nvtxRangePop(); }
    NvtxRange(const NvtxRange&) = delete;
    NvtxRange& operator=(const NvtxRange&) = delete;
};

// Makes `dev` the calling thread's current device for the duration of an ABI
// call and gives the caller's current device back on return, so that a call on
// a state of another device does not move the caller's thread (a torch caller
// working on device 1 stays on device 1). ok is false if the switch failed.
struct DeviceScope {
    int prev = -1;
    bool ok = false;
    explicit DeviceScope(int dev)
    {
        if (cudaGetDevice(&prev) != cudaSuccess) {
            cudaGetLastError();
            prev = -1;
        }
        ok = prev == dev || cudaSetDevice(dev) == cudaSuccess;
        if (!ok) cudaGetLastError();
    }
    ~DeviceScope()
    {
        int now = -1;
        if (prev >= 0 && (cudaGetDevice(&now) != cudaSuccess || now != prev)) {
            cudaSetDevice(prev);
            cudaGetLastError();
        }
    }
    DeviceScope(const DeviceScope&) = delete;
    DeviceScope& operator=(const DeviceScope&) = delete;
};

// Whether the caller is capturing `s` into a graph.
inline bool stream_captures(cudaStream_t s)
{
    cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(s, &st) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return st != cudaStreamCaptureStatusNone;
}

// Whether a wait that began at clock `first` has lasted longer than `limit` cycles at `now`.
// (The difference, not first + limit, which a limit near the type's largest overflows.)
__host__ __device__ inline bool limit_passed(long long first, long long now, long long limit)
{
    return now - first > limit;
}

constexpr int kTraceCap = 65536;     // rows kept in the device trace ring
constexpr int kTraceCols = 5;        // (t, mass, E_s, E_m, E_bulk)

// Couplings of the 24 links grouped by |c|^2 (Eq. FORCE with Table 1):
//   K1 = G1/9 + 4 G2/63, K2 = G1/36 + 4 G2/135, K4 = G2/180,
//   K5 = 2 G2/945, K8 = G2/15120; K0 = G1 4/9 + G2 p_s0 is the rest coupling
//   of the belt-1 energy (p_s0 = 247/420 from Eq. weights_1).
struct Couplings {
    double K0, K1, K2, K4, K5, K8;
};
Couplings couplings(double G1, double G2);

// Populations of an FP32 / FP16 state ("tiled" layout): rows of 32-column
// tiles of 288 elements; the tile of column x in row y starts at
//   y * g_pitch(nx) + (x / 32) * 288.
// FP32 ("paired"): a tile holds its 32 sites' populations 0, 2 and 4 as three
// runs of 32 (elements 0-31, 32-63, 64-95, at x % 32 within each run), then the
// pairs (1, 3), (5, 6) and (7, 8) as three runs of 32 pairs (elements 96-159,
// 160-223, 224-287, the pair of column x % 32 at 2 (x % 32), first member
// first). The pairs are the populations a thread of the fused step always
// writes together (the two that arrive from the neighbouring columns in one
// row), so each pair is one 8-byte access.
// FP16: the same element layout, so a pair is one 4-byte access (8192^2:
// 92.6k against 91.5k MLUPS with nine runs of 32).
// Columns past nx in the last tile of a row are padding (zero, never read by a
// step).
constexpr int kTileW = 32;
constexpr int kTileElems = 9 * kTileW;
__host__ __device__ inline int g_pitch(int nx) { return kTileElems * ((nx + kTileW - 1) / kTileW); }
__host__ __device__ inline long long g_elems(int nx, int ny) { return (long long)ny * g_pitch(nx); }

// Arguments of the fused FP32 step (deviation storage, see lb.h LB_FP32).
template <typename T>
struct StepArgs {
    const T* __restrict__ g_in;      // tiled f(t) - w rho_ref: populations of state t
    T* __restrict__ g_out;           // tiled f(t+1) - w rho_ref
    const float* __restrict__ dpsi_in;   // [ny][nx] psi(t) - psi_ref
    float* __restrict__ dpsi_out;        // [ny][nx] psi(t+1) - psi_ref
    int nx, ny;
    int rows;                        // output rows per CTA
    long long N;                     // nx*ny
    int pitch;                       // g_pitch(nx): elements per row of g
    int npitch;                      // g_elems(nx, ny): elements per g buffer
    float omega, omc, inv_omega;     // omega, 1-omega, 1/omega
    float w0, w1, w2;                // D2Q9 weights
    float K1, K2, K4, K5, K8;        // force couplings
    float rho_ref, psi_ref, cpsi, inv_rho0;  // dpsi = cpsi * expm1(-(rho-rho_ref)/rho0)
    // energy/mass reduction (REDUCE launches only)
    float K0, half_A1;
    double* partials;                // [gridDim.x*gridDim.y + gridDim.y][4]: CTA, row totals
    unsigned int* counter;           // arrival counter of the grid sums (zero between uses)
    double* trace;                   // [kTraceCap][5] ring
    int* trace_count;                // rows ever written
    long long t;                     // time level of the reduced state
    // bounded waits of the bulk-copy kernel
    int* err;                        // error flags: 1 a wait ran out, 2 a reduction was not finite
    long long wait_cycles;           // clock limit of one wait
    int skip_unit0;                  // test hook: the first row unit's barrier is armed, no copy issued
    float* __restrict__ dev;         // [ny][nx] density deviations of a traced state (pairs of steps)
};

// Output rows per CTA accepted by lb_set_launch / lb_batch_set_launch.
constexpr int kMinRows = 4;
constexpr int kMaxRows = 4096;

// Launchers (lb_fp32.cu). All return the launch's cudaError_t.
struct Fp32Launch {
    int block_x;   // threads per CTA
    int rows;      // output rows per CTA
    int pipeline;  // 0: register prefetch (any shape), 1: bulk-copy rings (nx % 32 == 0)
};
int fp32_grid_blocks(int nx, int ny, Fp32Launch L);
cudaError_t fp32_step(const StepArgs<float>& a, Fp32Launch L, bool reduce, cudaStream_t s);
cudaError_t fp16_step(const StepArgs<__half>& a, Fp32Launch L, bool reduce, cudaStream_t s);
// Batches (lb_fp32.cu kernels, lb_batch.cu host code): one launch advances many
// replicas. tiles[k] = (replica, strip, chunk, alternate), grouped by replica in
// each replica's own CTA order; reps[r] locates replica r's tiles and its trace ring.
struct BatchRep {
    int first_tile, ntiles;
    int ntx;                   // tiles per row chunk
    int first_row;             // slot of the replica's row totals (after all tile partials)
    unsigned int* counter;     // the replica's arrival counter (its state's, zero between uses)
    long long N;
    double rho_ref;
    double* trace;
    int* trace_count;
    int* err;                  // the replica's error flags
};
template <typename T>
struct BatchLaunch {
    const StepArgs<T>* args;   // [nreps] arguments of this step's parity
    const int4* tiles;
    int ntiles;
    double* tile_partials;     // [ntiles + row chunks of all replicas][4]
    const BatchRep* reps;
    int nreps;
    const int2* rowmap;        // [nrows] (replica, row chunk) of each reduction CTA
    int nrows;
    int block_x;
    bool om1;                  // every replica has omega == 1
    int trace_every;
    int num_sms;
    bool alternate;            // some replica marches in alternating directions
};
cudaError_t fp32_batch_step(const BatchLaunch<float>& b, bool reduce, cudaStream_t s);
cudaError_t fp16_batch_step(const BatchLaunch<__half>& b, bool reduce, cudaStream_t s);
// Whether the state of a lattice of n sites exceeds L2.
inline bool beyond_l2(long long n) { return n * 80 > (128LL << 20); }
// Whether the steps of a lattice of n sites march in alternating directions
// (down in even row chunks, up in odd ones): only when its state does not fit in
// L2 (measured: 2% slower at 1024^2, faster from 2048^2 on). A batch replica
// follows the same rule as the lattice run alone.
inline bool marches_alternate(long long n) { return beyond_l2(n); }

// Two plain steps in one pass (lb_pair.cu): CTAs of kPairTH threads, two columns each, and
// kPairCols output columns.
constexpr int kPairTH = 64;
constexpr int kPairCols = 2 * kPairTH - 8;
// Columns computed in a row of nx, halo and idle lanes included: by a pair, and by a step of its
// own in CTAs of block_x threads (block_x - 2 output columns).
inline long long pair_columns(int nx) { return 2LL * kPairTH * ((nx + kPairCols - 1) / kPairCols); }
inline long long single_columns(int nx, int block_x)
{
    return (long long)block_x * ((nx + block_x - 3) / (block_x - 2));
}
// Pairs are for lattices of 2^18 sites on that are not held on the SMs (lb_resident.cu):
// below, their few long chunks take as long as two launches of k_step (us per step, single and
// paired: 250x187 10.1 and 10.2, 512^2 10.3 and 9.3, 700^2 12.3 and 10.2). And not where a
// last strip of few columns makes a pair compute that many more columns than single steps do,
// with 64 threads per CTA up to 1.7 million sites, 128 beyond. Time of paired over single
// steps (FP32 with omega 1 and 0.8, FP16 alike) by that ratio:
//   450,000 sites: 1.33 (140 columns) held, 1.08, held, 0.93; 1.0 (360) held, 0.84, ..
//   600,000: 1.5 (241) 1.00, 1.07, 1.14, 1.12; 1.33 (140) 0.82, 0.88, 0.94, 0.95; 1.0 0.80 to 1.00
//   10^6: 2 (121) 1.15, 1.23, 1.20; 1.5 (241) 0.91, 0.96, 1.11, 1.00; 1.33 0.82, 0.87, 0.87, 0.84
//   1.3 million: 1.5 (241) 0.88, 0.96, 1.04, 0.99, (246) 0.80, 0.88, 0.95, 0.92
//   2^24: 2 (121) 1.09, 1.19, 1.25; 1.5 (241) 0.84, 0.94, 0.95; 1.0 0.57 to 0.69
inline bool pairs_pay(int nx, int ny, int block_x, int elem_bytes)
{
    const long long n = (long long)nx * ny, pair = pair_columns(nx), single = single_columns(nx, block_x);
    return n < (1LL << 18)                            ? false
           : n < (1LL << 19)                          ? 4 * pair <= 5 * single
           : n < (elem_bytes == 4 ? 900000 : 1200000) ? 5 * pair <= 7 * single
                                                      : 2 * pair <= 3 * single;
}
// A pair whose first state has a trace row adds two kernels for the row, where a reduction step
// forms it on the way. That pays where memory traffic bounds the steps (every second state
// traced, paired over single, FP32 and FP16: 740^2 1.15 and 1.10, 900^2 0.96 and 0.96, 1024^2 1.00
// and 1.03, 1024x1269 0.95 and 1.07, 1024x1562 0.84 and 0.97, 1300^2 0.81 and 0.90, 2048^2 0.80 and
// 0.80), again not with that many more columns (ratio 1.14, 425 columns, 1.3 million sites 1.03 and
// 1.14, 1.6 million 0.94 and 1.05; 2^24 sites: ratio 1.5 1.02, 1.33 0.93).
inline bool traced_pairs_pay(int nx, int ny, int block_x, int elem_bytes)
{
    const long long n = (long long)nx * ny, pair = pair_columns(nx), single = single_columns(nx, block_x);
    return beyond_l2(n) ? 5 * pair <= 7 * single
                        : n >= (elem_bytes == 4 ? 1250000 : 1500000) && 5 * pair <= 6 * single;
}
// (traced: the density deviations of state t are left in a.dev)
cudaError_t fp32_step_pair(const StepArgs<float>& a, bool traced, cudaStream_t s);
cudaError_t fp16_step_pair(const StepArgs<__half>& a, bool traced, cudaStream_t s);
// The same for a batch of any size (its single-step tiles are 32 rows high unless the
// caller chose otherwise, so even small batches gain: 27 replicas of up to 69^2, 30.7 ->
// 9.5 us per step; nine 512^2 57.4 -> 28.6; the 96-replica sweep 338 -> 178): `tiles`
// (pair_tiles: replica, first column, first row, end row) on the device; odd: some replica
// has an odd nx
// Estimated time of a batch's pair over that of two single steps. Either takes its CTAs' rows
// one after another, a row in the longer of its latency and the SM's share of the work:
// fitted to 1,200 batches of 2 to 500 lattices from 5^2 to 122x2000 at six shapes (FP32 and
// FP16 separately for the pair), within 10% and 6% on average.
struct BatchWork {
    int tiles, block_x, chunk;        // of the single step; chunk: rows of its tallest CTA
    int pair_tiles, pair_chunk;       // of the pair
    int elem_bytes, num_sms;
};
inline double batch_paired_over_single(const BatchWork& w)
{
    auto most = [](double x, double y) { return x > y ? x : y; };
    const bool half = w.elem_bytes == 2;
    const double warps = w.tiles * (w.block_x / 32.0) / w.num_sms;
    const double single = 4.0 + (w.chunk + 2) * most(0.8, 0.06 * warps);
    const int slots = (half ? 8 : 6) * w.num_sms, waves = (w.pair_tiles + slots - 1) / slots;
    const double pair_warps = 2.0 * w.pair_tiles / w.num_sms;
    const double pair = half ? 6.0 + (w.pair_chunk + 5) * most(1.1 * waves, 0.15 * pair_warps)
                             : 6.0 + (w.pair_chunk + 7) * most(0.7 * waves, 0.14 * pair_warps);
    return pair / (2.0 * single);
}
// Whether a batch takes pairs. With the default tiles of single steps (126 columns, 32 rows) and
// larger ones always: paired over single 0.96 at most (two 5^2, FP16), 0.27 at best; nor do
// 62 columns of 32 rows change that (0.94 at most) unless nearly all of them are idle (fill: sites
// over the columns that single steps compute; 5x20000 up to 1.21). Otherwise the estimate
// decides: where it allows pairs they take 1.00 at most, where it does not up to 1.44 (500 of
// 12x40 in tiles of 62x8) and 0.79 at best.
inline bool batch_pairs_pay(int block_x, int rows, double fill, double estimate)
{
    return (rows >= 32 && (block_x >= 128 || fill >= 0.15)) || estimate <= 1.0;
}
// And whether these take a state with a trace row along (otherwise a reduction step does). Not
// lattices of a few rows (every second state traced: 5^2 1.02 to 1.17, 16^2 0.75), and with
// smaller tiles only by a margin, or where a pair computes few columns more: allowed 1.06 at
// most, otherwise up to 1.45. column_ratio: of pair_columns to single_columns, over all rows.
inline bool batch_traced_pairs_pay(int block_x, int rows, int tallest, double column_ratio,
                                   double estimate)
{
    return tallest >= 16 && ((block_x >= 128 && rows >= 32) || column_ratio <= 1.25 ||
                             estimate <= (rows >= 32 ? 0.9 : 0.7));
}
void pair_tiles(const std::vector<std::pair<int, int>>& sizes, int elem_bytes, int num_sms,
                std::vector<int4>& tiles);
cudaError_t fp32_batch_pair(const BatchLaunch<float>& b, const int4* tiles, int ntiles, bool odd,
                            bool traced, cudaStream_t s);
cudaError_t fp16_batch_pair(const BatchLaunch<__half>& b, const int4* tiles, int ntiles, bool odd,
                            bool traced, cudaStream_t s);
// Trace rows of kept states (lb_trace.cu), as reduction steps of launch width block_x and
// a.rows write them: `count` states `apart` values from one another, at t, t + every, ...
struct TraceRows {
    const float *dpsi, *dev;
    size_t apart;
    int count;
    long long t;
    int every;
    int block_x;
    double* partials;                     // [count][CTA partials, row totals][4]
    unsigned int* counters;               // [1 + count], zero between uses
};
template <typename T>
cudaError_t trace_rows(const StepArgs<T>& a, const TraceRows& r, cudaStream_t s);
// the tile partials of a batch's traced states (from dpsi_in and dev), and their sums
template <typename T>
cudaError_t batch_trace_partials(const BatchLaunch<T>& b, cudaStream_t s);
template <typename T>
cudaError_t batch_reduce(const BatchLaunch<T>& b, cudaStream_t s);
// Shared memory per CTA of the kernels that hold a lattice on the SMs (227 KB at most, less
// their static words).
constexpr int kHeldSmem = 226 * 1024;
// Many steps of a small lattice in one launch (lb_resident.cu): the tiles its CTAs hold
// and the buffers they exchange through.
struct ResidentBuf {
    int gx = 0, gy = 0, tw = 0, th = 0;   // tile grid and tile size; gx = 0: not used
    unsigned tag = 0;                     // steps exchanged so far
    uint2* llp = nullptr;                 // halo words of dpsi
    uint4* llm = nullptr;                 // halo words of the moments or populations
    int trace_every = 0;
    int max_rows = 0;                     // trace rows one launch may dump
    float* dump = nullptr;                // [max_rows][2][N]
    double* partials = nullptr;           // [max_rows][partials of one trace row][4]
    unsigned int* counters = nullptr;     // [1 + max_rows]
};
// A cooperative launch is refused, at once and with nothing started, where the stream has fewer
// SMs than the lattice has tiles (a stream of a green context, a process with a share of
// the GPU). The steps are then taken without holding the lattice.
inline bool launch_refused(cudaError_t e)
{
    return e == cudaErrorCooperativeLaunchTooLarge || e == cudaErrorNotSupported;
}
// Whether the stream takes a held launch of this lattice: one step into the idle buffers. (A
// test for a launch without steps in the kernel costs 1% of every step at 70x45.)
cudaError_t fp32_resident_probe(const StepArgs<float>& a, ResidentBuf& b, cudaStream_t s);
// The fewest steps worth a held launch, by the sites of a tile: it loads them, and sorts its
// work lists, before the first step. Calls of 2, 3, 4, 5 and 6 steps, held over single launches,
// omega = 1: 440^2 (1344 sites) 0.91, 0.74, ..; 512^2 (1728) 1.10, 0.87, ..; 560^2 (2100)
// 1.19, 0.96, 0.83, ..; 600^2 (2432) 1.38, 1.07, 0.91, ..; 680^2 (3096) 1.38, 1.07, 0.92, ..;
// 720^2 (3420) 1.50, 1.17, 1.01, 0.91. Otherwise: 440^2 1.00, 0.81, ..; 512^2 1.20, 0.94, ..;
// 560^2 1.33, 1.07, 0.95, ..; 600^2 1.49, 1.20, 1.09, 1.00, 0.94.
inline int held_least(int tile_sites, bool om1)
{
    if (tile_sites <= 1400) return 2;
    if (om1) return tile_sites <= 2150 ? 3 : tile_sites <= 3200 ? 4 : 5;
    return tile_sites <= 1900 ? 3 : tile_sites <= 2200 ? 4 : 6;
}
bool resident_plan(int nx, int ny, bool om1, int num_sms, ResidentBuf& b);
cudaError_t fp32_resident(const StepArgs<float>& a, ResidentBuf& b, int block_x, int steps,
                          cudaStream_t s);
cudaError_t fp16_resident(const StepArgs<__half>& a, ResidentBuf& b, int block_x, int steps,
                          cudaStream_t s);
// The same without trace rows, every state before its step kept in `states`: [steps][4][N],
// dpsi, density deviation and the momentum negated (x, y).
cudaError_t fp32_resident_kept(const StepArgs<float>& a, ResidentBuf& b, int steps, float* states,
                               cudaStream_t s);
// bulk-copy pipelined step (lb_bulk.cu)
bool bulk_supported(int nx, int ny, int elem_bytes, int block_x);
int bulk_grid_blocks(int nx, int ny, int elem_bytes, Fp32Launch L);
cudaError_t fp32_step_bulk(const StepArgs<float>& a, Fp32Launch L, bool reduce, cudaStream_t s);
cudaError_t fp16_step_bulk(const StepArgs<__half>& a, Fp32Launch L, bool reduce, cudaStream_t s);
template <typename T>
cudaError_t delta_init(T* g, float* dpsi, const double* rho_init, int nx, int ny,
                       double rho_ref, double rho0, cudaStream_t s);
template <typename T>
cudaError_t delta_fields(const T* g, int nx, int ny, double rho_ref, double* rho, double* ux,
                         double* uy, cudaStream_t s);
template <typename T>
cudaError_t delta_energy(const T* g, const float* dpsi, int nx, int ny, const StepArgs<T>& a,
                         double* out4, double* partials, unsigned int* counter, int* narrow,
                         bool wide, cudaStream_t s);

// Input checks and sums (lb_fp32.cu): out[0] = sum rho, flag |= 1 if any rho is
// not finite or <= 0.
cudaError_t rho_check_sum(const double* rho, long long n, double* partials, unsigned int* counter,
                          double* out_sum, int* flag, cudaStream_t s);

// FP64 parity path (lb_fp64.cu, compiled without FMA contraction).
struct Fp64Args {
    double* f_in;        // [9][ny][nx] populations of state t (after streaming)
    double* f_out;       // [9][ny][nx] populations of state t+1
    double* psi;         // [ny][nx] psi(t)
    double* rho;         // [ny][nx] rho(t)
    int nx, ny;
    double omega, G1, G2, rho0;
};
cudaError_t fp64_init(double* f, const double* rho_init, int nx, int ny, cudaStream_t s);
cudaError_t fp64_psi(const Fp64Args& a, cudaStream_t s);
cudaError_t fp64_collide_stream(const Fp64Args& a, cudaStream_t s);
cudaError_t fp64_energy(const Fp64Args& a, double* partials, unsigned int* counter,
                        double* out4, double* trace, int* trace_count, long long t,
                        cudaStream_t s);
cudaError_t fp64_fields(const double* f, int nx, int ny, double* rho, double* ux, double* uy,
                        cudaStream_t s);

}  // namespace lbsc

namespace lbsc {
constexpr size_t kGuardBytes = 256;              // guard region on each side of a buffer
constexpr unsigned char kGuardByte = 0xA5;       // the pattern the guards hold
// The usable size of a guarded buffer: its tail guard starts 256-byte aligned
constexpr size_t guarded_size(size_t bytes)
{
    return (bytes + kGuardBytes - 1) / kGuardBytes * kGuardBytes;
}

// The control words of a state, each a guarded buffer of its own, in one allocation in this
// order, so that the host reads back all but the arrival counters in one transfer.
struct Control {
    double res[4];
    int err, trace_count, flag;
};
constexpr size_t kControlPitch = 3 * kGuardBytes;   // from one word to the next: guards and words
}  // namespace lbsc

// The state behind the opaque lb_state* of the C ABI (lb_api.cu owns its
// lifetime; lb_batch.cu drives several of them with one launch per step).
struct lb_state {
    lb_params p;
    cudaStream_t stream = nullptr;
    long long t = 0;
    bool poisoned = false;
    long long N = 0;
    // FP32 / FP16 deviation storage (g tiled, lbsc::g_elems elements each)
    void* g[2] = {nullptr, nullptr};
    float* dpsi[2] = {nullptr, nullptr};
    float* dev = nullptr;          // density deviations of a traced state; if there was not the
                                   // memory for them, traced states are stepped singly
    int cur = 0;
    double rho_ref = 0.0;
    lbsc::Fp32Launch launch{128, 64, 0};
    int* err = nullptr;            // set by a kernel whose bounded wait ran out
    long long wait_cycles = 2000000000LL;
    int skip_unit0 = 0;            // test hook of lb_set_wait_limit
    lbsc::ResidentBuf res_buf;     // small lattices: tiles held on the SMs over many steps
    bool in_graphs = false;        // steps were captured: n steps swap the buffers as n single ones do
    // FP64 parity storage
    double* f64[2] = {nullptr, nullptr};
    double* psi64 = nullptr;
    double* rho64 = nullptr;
    // reductions, trace, scratch
    double* partials = nullptr;
    size_t partials_cap = 0;       // number of 4-double partials
    int max_cta_rows = 0;          // CTA rows of the step's grid at most (kMinRows-row chunks)
    unsigned int* counter = nullptr;
    double* trace = nullptr;
    int* trace_count = nullptr;
    double* res = nullptr;         // 4 doubles of results; err, trace_count, flag follow (Control)
    int* flag = nullptr;
    double* field_tmp = nullptr;   // N doubles, allocated on the first lb_fields into pageable host memory
    // every device buffer of the state, with a guard region on each side (base: the first
    // guard), and the allocations that they lie in
    struct Alloc {
        void* base;
        size_t bytes;
    };
    std::vector<Alloc> allocs;
    std::vector<void*> blocks;
};

namespace lbsc {
// lb_init; `alone`: the state is stepped by itself (false for a batch's replicas)
lb_status state_init(lb_state** out, const lb_params* p, const double* rho_init, void* stream,
                     bool alone);
// Allocate buffers for a state together, each with guards on both sides (pattern written on
// the state's stream); the usable pointers are stored in order. False, with nothing allocated,
// if there is not the memory. The last `spare` are left out (nullptr) if there is only memory
// for the others. They share blocks of up to kBlockBytes (lb_init, with an allocation for each
// of the larger buffers and with one for all: 70x45 200 and 158 us, 512^2 338 and 162 us, 2050x1999
// 425 and 250 us, but 8192^2 1390 and 2100 us).
constexpr size_t kBlockBytes = size_t(1) << 30;
struct Buffer {
    void** ptr;
    size_t bytes;
};
bool state_alloc(lb_state* s, std::vector<Buffer> buffers, size_t spare = 0);
// one buffer; nullptr if there is not the memory
inline void* state_alloc(lb_state* s, size_t bytes)
{
    void* p = nullptr;
    return state_alloc(s, {{&p, bytes}}) ? p : nullptr;
}
}  // namespace lbsc

namespace lbsc {
// Whether steps t and t + 1 go through a lattice or batch together when `left` steps are
// left: not when state t + 1 has a trace row (every te steps; 0: none), and when state t has
// one only if `traced`.
inline bool pair_at(long long t, long long left, int te, bool traced)
{
    return left >= 2 && !(te > 0 && ((t + 1) % te == 0 || (!traced && t % te == 0)));
}
// How many pairs n steps from t make. A captured graph reads and writes the buffers that
// were in place when it was captured, and its replays are valid after any number of further
// steps that swaps the buffers as often, modulo two, as single steps do: once each. A pair swaps
// them once for two steps, so states whose steps have been captured take an even number of pairs.
inline long long pairs_made(long long t, long long n, int te, bool traced)
{
    long long pairs = 0;
    for (long long k = 0; k < n;) {
        const bool pair = pair_at(t + k, n - k, te, traced);
        pairs += pair;
        k += pair ? 2 : 1;
    }
    return pairs;
}
// Take n steps of an FP32 or FP16 state, several per launch where that pays (lb_step).
lb_status advance_delta(lb_state* s, long n);
template <typename T>
StepArgs<T> state_args(const lb_state* s, int cur);   // arguments of a step from buffers `cur`
size_t elem_size(lb_precision p);
// Where a kernel can read or write a double array directly: device memory as it
// is, pinned host memory through its device alias; nullptr for pageable memory.
double* device_view(double* p);
// Objective sums of lb_adjoint's terminal kernel for an FP32/FP16 state
// (lb_adjoint.cu): acc[0] = E_s + E_m of the current state, acc[1] = sum (rho -
// tgt)^2, acc[2..3] the explicit dE/dG1, dE/dG2; tgt is device memory. wide: in FP64
// throughout, for states that set the state's flag without it (delta_energy's `narrow`).
cudaError_t objective_delta(const lb_state* s, const double* tgt, double* acc, bool wide,
                            cudaStream_t st);
// *out = sum (rho - tgt)^2 over n doubles in device memory, deterministic.
cudaError_t misfit64(const double* rho, const double* tgt, long long n, double* partials,
                     unsigned int* counter, double* out, cudaStream_t st);
}  // namespace lbsc
