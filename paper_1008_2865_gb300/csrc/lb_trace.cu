// lb_trace.cu — trace rows of states whose steps went through a kernel that takes
// several steps (lb_pair.cu, lb_resident.cu): mass and the Sec. 5 energies of state t
// from its dpsi and its density deviations, which those kernels leave in memory.
//
// A reduction step of k_step forms its sums while it steps: per thread in FP32 along the
// thread's march, then per CTA and per grid. The kernels here repeat exactly these sums
// in this order, thread for thread, from 8 bytes per site; the row has the bits of the
// one the reduction step writes. They stream the two fields: 13 of the 25 stencil values
// (one of each pair (c, -c) and the centre) come from L1, and the rows of a march are
// independent loads, four rows in flight (4096^2: 69 us, 50% of the issue slots).
#include "lb_device.cuh"

#include <type_traits>

namespace lbsc {
namespace {

using namespace dev;

// The sums of one thread of the tile with output columns [x0, ..) and rows [y0, +nrows):
// the out-site rows of step_tile_dir, marching up or down, flushed to FP64 as there.
template <int BX, typename T>
__device__ __forceinline__ void trace_tile(const StepArgs<T>& a, const float* __restrict__ dpsi,
                                           const float* __restrict__ dev, int x0, int y0, int nrows,
                                           bool up, double v[4])
{
    const int tid = threadIdx.x, nx = a.nx, ny = a.ny;
    float es = 0.f, em = 0.f, eb = 0.f, ms = 0.f;
#pragma unroll
    for (int q = 0; q < 4; ++q) v[q] = 0.0;
    if (tid < 1 || tid > min(BX - 2, nx - x0)) return;
    const int x = x0 - 1 + tid;
    auto march = [&](auto inner, auto upward) {
        constexpr bool kInner = decltype(inner)::value, kUp = decltype(upward)::value;
        int xc[5];
#pragma unroll
        for (int m = 0; m < 5; ++m) xc[m] = wrapi(x + m - 2, nx);
        // offsets of the five stencil rows; a step of the march needs one new one
        const int first = kUp ? y0 + nrows - 1 : y0, N = (int)a.N;
        int o[5];
#pragma unroll
        for (int r = 0; r < 5; ++r) o[r] = wrapi(first + r - 2, ny) * nx;
        for (int k = 1; k <= nrows;) {
            // up to the row after which k_step flushes; the FP64 sums stay out of the row
            // loop (predicated into it they bound it: 239 instead of 92 us at 4096^2)
            const int end = min(nrows, k | 63);
#pragma unroll 4
            for (; k <= end; ++k) {
                float q[5][5];
#pragma unroll
                for (int r = 0; r < 5; ++r) {
                    const float* row = dpsi + o[r] + (kInner ? x : 0);
#pragma unroll
                    for (int m = 0; m < 5; ++m) q[r][m] = __ldg(row + (kInner ? m - 2 : xc[m]));
                }
                const float* rows[5] = {&q[0][2], &q[1][2], &q[2][2], &q[3][2], &q[4][2]};
                float Sx, Sy;
                force_energy<true>(rows, a, Sx, Sy, 1.f, a.psi_ref + q[2][2], es, em, eb);
                ms = fmaf(1.f, __ldg(dev + o[2] + x), ms);
                if (kUp) {
                    const int next = (o[0] == 0 ? N : o[0]) - nx;
#pragma unroll
                    for (int r = 4; r > 0; --r) o[r] = o[r - 1];
                    o[0] = next;
                } else {
                    const int next = o[4] + nx == N ? 0 : o[4] + nx;
#pragma unroll
                    for (int r = 0; r < 4; ++r) o[r] = o[r + 1];
                    o[4] = next;
                }
            }
            v[0] += es;
            v[1] += em;
            v[2] += eb;
            v[3] += ms;
            es = em = eb = ms = 0.f;
        }
    };
    using Yes = std::true_type;
    using No = std::false_type;
    const bool inside = x >= 2 && x < nx - 2;
    if (up) inside ? march(Yes{}, Yes{}) : march(No{}, Yes{});
    else inside ? march(Yes{}, No{}) : march(No{}, No{});
}

// CTA (bx, by, z) is CTA (bx, by) of k_step's grid for the z-th of the kept states (fields
// `apart` values from one to the next).
template <typename T, int BX>
__global__ void __launch_bounds__(BX)
    k_trace_partial(const StepArgs<T> a, const float* __restrict__ dpsi, const float* __restrict__ dev,
                    size_t apart, double* __restrict__ partials, int stride, bool alternate)
{
    __shared__ double red[4 * BX];
    const size_t z = blockIdx.z;
    const int y0 = blockIdx.y * a.rows;
    double v[4];
    trace_tile<BX>(a, dpsi + z * apart, dev + z * apart, blockIdx.x * (BX - 2), y0, min(a.rows, a.ny - y0),
                   alternate && (blockIdx.y & 1), v);
    block_sum4<BX>(v, red);
    if (threadIdx.x == 0) {
        double* p = partials + 4 * (z * stride + (size_t)blockIdx.y * gridDim.x + blockIdx.x);
#pragma unroll
        for (int q = 0; q < 4; ++q) p[q] = v[q];
    }
}

// The grid sums of kept states: k_step_total for every trace row (blockIdx.y) at once.
template <int NT>
__global__ void __launch_bounds__(NT)
    k_trace_total(const double* __restrict__ cta, double* __restrict__ rows, int stride, int nbx,
                  unsigned int* counters, double* trace, int* trace_count, int* err, long long t,
                  int trace_every, double mass_ref)
{
    __shared__ double red[4 * NT];
    const int nby = gridDim.x, z = blockIdx.y, nz = gridDim.y;
    double w[4];
    if (row_then_total<NT>(cta + 4 * (size_t)z * stride, nbx, nby, blockIdx.x,
                           rows + 4 * (size_t)z * stride, counters + 1 + z, w, red)) {
        const int c = *reinterpret_cast<volatile int*>(trace_count);
        const double mass = mass_ref + w[3];
        double* r = trace + (size_t)((c + z) % kTraceCap) * kTraceCols;
        r[0] = (double)(t + (long long)z * trace_every);
        r[1] = mass;
        r[2] = w[0];
        r[3] = w[1];
        r[4] = w[2];
        if (!isfinite(mass) || !isfinite(w[0]) || !isfinite(w[1])) atomicOr(err, 2);
        __threadfence();
        // the last row to finish counts all of them
        if (atomicAdd(counters, 1u) == (unsigned)nz - 1) {
            *trace_count = c + nz;
            *counters = 0u;
        }
    }
}

// A batch's tiles (k_step_batch's work list), one CTA each; k_batch_reduce follows.
template <typename T, int BX>
__global__ void __launch_bounds__(BX)
    k_trace_batch(const StepArgs<T>* __restrict__ args, const int4* __restrict__ tiles,
                  double* __restrict__ tile_partials)
{
    __shared__ double red[4 * BX];
    const int4 tl = __ldg(tiles + blockIdx.x);      // (replica, strip, chunk, alternate)
    const StepArgs<T>& a = args[tl.x];
    const int y0 = tl.z * a.rows;
    double v[4];
    trace_tile<BX>(a, a.dpsi_in, a.dev, tl.y * (BX - 2), y0, min(a.rows, a.ny - y0),
                   tl.w != 0 && (tl.z & 1), v);
    block_sum4<BX>(v, red);
    if (threadIdx.x == 0) {
#pragma unroll
        for (int q = 0; q < 4; ++q) tile_partials[4 * (size_t)blockIdx.x + q] = v[q];
    }
}

// f(std::integral_constant<int, block_x>) for the CTA widths of the step
template <typename F>
cudaError_t with_width(int block_x, F f)
{
    switch (block_x) {
    case 64: return f(std::integral_constant<int, 64>{});
    case 96: return f(std::integral_constant<int, 96>{});
    case 128: return f(std::integral_constant<int, 128>{});
    case 192: return f(std::integral_constant<int, 192>{});
    case 256: return f(std::integral_constant<int, 256>{});
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace

template <typename T>
cudaError_t trace_rows(const StepArgs<T>& a, const TraceRows& r, cudaStream_t s)
{
    return with_width(r.block_x, [&](auto width) {
        constexpr int BX = decltype(width)::value;
        const dim3 grid((a.nx + BX - 3) / (BX - 2), (a.ny + a.rows - 1) / a.rows, r.count);
        const int stride = (int)(grid.x * grid.y + grid.y);
        k_trace_partial<T, BX><<<grid, BX, 0, s>>>(a, r.dpsi, r.dev, r.apart, r.partials, stride,
                                                   marches_alternate(a.N));
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
        k_trace_total<BX><<<dim3(grid.y, r.count), BX, 0, s>>>(
            r.partials, r.partials + 4 * (size_t)grid.x * grid.y, stride, (int)grid.x, r.counters,
            a.trace, a.trace_count, a.err, r.t, r.every, (double)a.N * (double)a.rho_ref);
        return cudaGetLastError();
    });
}

template <typename T>
cudaError_t batch_trace_partials(const BatchLaunch<T>& b, cudaStream_t s)
{
    return with_width(b.block_x, [&](auto width) {
        constexpr int BX = decltype(width)::value;
        k_trace_batch<T, BX><<<b.ntiles, BX, 0, s>>>(b.args, b.tiles, b.tile_partials);
        return cudaGetLastError();
    });
}

template cudaError_t trace_rows<float>(const StepArgs<float>&, const TraceRows&, cudaStream_t);
template cudaError_t trace_rows<__half>(const StepArgs<__half>&, const TraceRows&, cudaStream_t);
template cudaError_t batch_trace_partials<float>(const BatchLaunch<float>&, cudaStream_t);
template cudaError_t batch_trace_partials<__half>(const BatchLaunch<__half>&, cudaStream_t);

}  // namespace lbsc
