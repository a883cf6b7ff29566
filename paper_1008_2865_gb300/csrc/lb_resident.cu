// lb_resident.cu — many steps of a small lattice in one launch (k_resident), for FP32
// and FP16 states.
//
// A small lattice is bound by latency: a launch of k_step takes 8 to 10 us however few
// its sites, because a CTA marches down ten rows one after another and the next step is
// another launch. Here the lattice is cut into one tile per SM, which stays in shared
// memory from step to step: a step is one collision of all the tile's sites at once, a
// barrier, one streaming. Only the sites next to a tile's edge go through L2. us per
// step, before -> after: 70x45 10.8 -> 1.9, 128^2 8.2 -> 1.8, 250x187 10.1 -> 2.3, 512^2
// 10.3 -> 4.1.
//
// What a step costs now: two passes over the tile at about 0.4 us each (128^2) and the
// halo's way to L2 and back, 0.5 us. The halo is one ring of moments (with omega = 1 a
// collision needs only rho, j and the psi stencil of a site; otherwise one ring of
// populations) and three rings of psi, and the collisions of the ring are computed on
// both sides, so that there is one exchange per step and not two. Its words carry the step's
// number (put_word), so the exchange is data and flag in one access: no grid barrier, no
// fence, and a tile waits only for its neighbours. The collisions that need no halo
// run while it is on its way (512^2: 4.75 -> 4.45 us), the tile's edge sites are streamed
// first. Two sets of words alternate: a tile writes a word again two steps later, and by
// then it has read words that its neighbours wrote after reading the first.
//
// All tiles must be resident together: the launch is cooperative, one CTA per SM at
// most, and starts none of its CTAs before there is room for all. Lattices on streams of
// their own therefore queue for the SMs where single launches share them (us per step of all:
// two, four and eight 512^2 lattices 8.4, 16.6 and 32.9, in single launches 12.9, 17.6
// and 30.6; 400^2 7.0, 13.6 and 26.8, against 12.7, 14.0 and 20.7). Every wait is bounded by the state's wait limit; a tile whose wait runs out
// flags the state and leaves, and so do the others.
//
// Every site's arithmetic is that of k_step, operation by operation, so the fields are
// bit-identical to single steps. States with a trace row leave their dpsi and density
// deviation in a buffer; trace_rows (lb_trace.cu) forms the
// energies from them afterwards, for all rows of the launch at once, in the order of
// k_step's threads.
#include "lb_packed.cuh"

namespace lbsc {
namespace {

using namespace dev;

// Threads at most, by the registers (us per step at 512^2 / 600^2 with 768, 896 and 1024
// threads: 4.25 / 5.32, 4.11 / 5.11, 4.26 / 5.30)
template <bool OM1>
constexpr int kResThreads = OM1 ? 896 : 768;

template <typename T>
struct ResArgs {
    StepArgs<T> a;
    PackedArgs k;
    int gx, tw, th;        // tiles per row of tiles, tile width (even) and height
    int steps;             // steps of this launch
    unsigned tag;          // steps exchanged before this launch
    uint2* llp;            // [2][N] dpsi halo words
    uint4* llm;            // [2][NQ][N] moments (omega = 1) or populations halo words
    float* dump;           // [rows][planes][N] of the states kept: dpsi, density deviation, and
    int planes;            // with four planes the momentum, negated
    int keep_every;        // states t with t % keep_every == 0 are kept; 0: none
};

template <bool OM1>
constexpr int kPlanes = OM1 ? 3 : 9;   // values a site carries from step to step
template <bool OM1>
constexpr int kQuads = OM1 ? 1 : 3;    // halo words of three values each

__host__ __device__ inline int res_lw(int tw) { return tw + 4; }
__host__ __device__ inline int res_lh(int th) { return th + 2; }
__host__ __device__ inline int halo_psi(int tw, int th) { return (tw + 6) * (th + 6) - tw * th; }
__host__ __device__ inline int halo_mom(int tw, int th) { return (tw + 2) * (th + 2) - tw * th; }
inline size_t res_smem(int tw, int th, bool om1)
{
    const size_t site = (size_t)res_lw(tw) * res_lh(th);
    return sizeof(float) * (site * (9 + (om1 ? 3 : 9)) + (size_t)(res_lw(tw) + 4) * (res_lh(th) + 4)) +
           sizeof(int2) * (size_t)(halo_psi(tw, th) + halo_mom(tw, th)) +
           sizeof(int) * (size_t)((tw + 4) / 2 * (th + 2) + tw / 2 * th);
}

__device__ __forceinline__ float2 at2(const float* p) { return *reinterpret_cast<const float2*>(p); }
__device__ __forceinline__ float2 shifted2(const float* p) { return make_float2(p[0], p[1]); }
__device__ __forceinline__ void put2(float* p, float2 v) { *reinterpret_cast<float2*>(p) = v; }

template <typename T>
__device__ __forceinline__ float2 stored2(float2 v);
template <>
__device__ __forceinline__ float2 stored2<float>(float2 v)
{
    return v;
}
template <>
__device__ __forceinline__ float2 stored2<__half>(float2 v)
{
    return __half22float2(__float22half2_rn(v));
}

template <typename T, bool OM1>
__global__ void __launch_bounds__(kResThreads<OM1>, 1) k_resident(const ResArgs<T> A)
{
    const int nt = blockDim.x;
    extern __shared__ __align__(16) float sm[];
    __shared__ int s_fail, s_np, s_nm, s_free;
    const StepArgs<T>& a = A.a;
    const int tid = threadIdx.x;
    const int nx = a.nx, ny = a.ny;
    const int N = (int)a.N;
    const int x0 = (blockIdx.x % A.gx) * A.tw, y0 = (blockIdx.x / A.gx) * A.th;
    const int w = min(A.tw, nx - x0), h = min(A.th, ny - y0);
    const int LW = res_lw(A.tw), LH = res_lh(A.th), S = LW * LH, PW = LW + 4;
    float* G = sm;                                   // [9] post-collision planes
    float* M = G + 9 * S;                            // [kPlanes] state planes
    float* P = M + kPlanes<OM1> * S;                 // dpsi, two columns and rows wider
    int2* hp = reinterpret_cast<int2*>(P + PW * (LH + 4));
    int2* hm = hp + halo_psi(A.tw, A.th);
    int* lc = reinterpret_cast<int*>(hm + halo_mom(A.tw, A.th));   // pairs to collide
    int* lo = lc + (A.tw + 4) / 2 * (A.th + 2);                   // own pairs
    using TL = Tile<T>;

    if (tid == 0) s_fail = s_np = s_nm = 0;
    __syncthreads();
    // ---- dpsi(t) of the tile and three rings around it; lists of the halo sites
    for (int q = tid; q < (w + 8) * (h + 6); q += nt) {
        const int jj = q / (w + 8), ii = q - jj * (w + 8);
        const int site = wrapi(y0 - 3 + jj, ny) * nx + wrapi(x0 - 4 + ii, nx);
        P[jj * PW + ii] = __ldg(a.dpsi_in + site);
        const bool own = jj >= 3 && jj < h + 3 && ii >= 4 && ii < w + 4;
        if (!own && ii >= 1 && ii < w + 7) hp[atomicAdd(&s_np, 1)] = make_int2(jj * PW + ii, site);
    }
    // ---- the state of the tile and one ring
    for (int q = tid; q < (w + 4) * (h + 2); q += nt) {
        const int j = q / (w + 4), i = q - j * (w + 4);
        const int x = wrapi(x0 - 2 + i, nx), y = wrapi(y0 - 1 + j, ny);
        float f[9];
        load_site_xy(f, a.g_in, a.pitch, x, y);
        float* m = M + j * LW + i;
        if (OM1) {
            m[0] = ((f[0] + f[1]) + (f[2] + f[3])) + ((f[4] + f[5]) + (f[6] + f[7])) + f[8];
            m[S] = (f[3] - f[1]) + (f[6] - f[5]) + (f[7] - f[8]);
            m[2 * S] = (f[7] + f[8]) - ((f[2] - f[4]) + (f[5] + f[6]));
        } else {
#pragma unroll
            for (int v = 0; v < 9; ++v) m[v * S] = f[v];
        }
        const bool own = j >= 1 && j <= h && i >= 2 && i < w + 2;
        if (!own && i >= 1 && i < w + 3) hm[atomicAdd(&s_nm, 1)] = make_int2(j * LW + i, y * nx + x);
    }
    // ---- work lists, in row order within each class: the pairs to collide, those that
    // need no halo first; the own pairs, those whose values the neighbours need first
    const int ew = (w + 4) / 2, en = ew * (h + 2);
    const int ow = (w + 1) / 2, on = ow * h;
    auto no_halo = [&](int j, int c) {        // stencil and moments within the tile
        return j >= 3 && j < h - 1 && c >= 2 && 2 * c + 1 < w;
    };
    auto is_edge = [&](int j, int c) {        // within three columns or rows of the edge
        return j < 3 || j >= h - 3 || 2 * c < 3 || 2 * c + 1 >= w - 3;
    };
    if (tid < 64) {
        const bool coll = tid < 32;
        const int lane = tid & 31, n = coll ? en : on, wd = coll ? ew : ow;
        int at = 0;
        for (int pass = 0; pass < 2; ++pass) {
            for (int p0 = 0; p0 < n; p0 += 32) {
                const int p = p0 + lane, j = p / wd, c = p - j * wd;
                const bool first = coll ? no_halo(j, c) : is_edge(j, c);
                const bool take = p < n && first == (pass == 0);
                const unsigned m = __ballot_sync(0xffffffffu, take);
                if (take) (coll ? lc : lo)[at + __popc(m & ((1u << lane) - 1u))] = j << 16 | 2 * c;
                at += __popc(m);
            }
            if (pass == 0 && coll && lane == 0) s_free = at;
        }
    }
    __syncthreads();
    const int np = s_np, nm = s_nm, nfree = s_free;
    int row = 0;                                         // trace rows dumped

    // collision of the pairs [p0, p1) of the list
    auto collide = [&](int p0, int p1, bool traced) {
        for (int p = p0 + tid; p < p1; p += nt) {
            const int e = lc[p], j = e >> 16, i = e & 0xffff;
            float2 Ak[5], Bk[5], Ck[5];
#pragma unroll
            for (int r = 0; r < 5; ++r) {
                const float* src = P + (j + r) * PW + i;
                Ak[r] = at2(src);
                Bk[r] = at2(src + 2);
                Ck[r] = at2(src + 4);
            }
            float2 Sx, Sy;
            force_sums2(Ak, Bk, Ck, A.k, Sx, Sy);
            const float2 pc = add2(A.k.psi_ref, Bk[2]);
            const float* m = M + j * LW + i;
            float2 f[9];
            Moments2 mo;
            if (OM1) {
                mo.d = at2(m);
                mo.jx = at2(m + S);
                mo.jy = at2(m + 2 * S);
            } else {
#pragma unroll
                for (int v = 0; v < 9; ++v) f[v] = at2(m + v * S);
                mo = moments2(f);
            }
            if (traced && j >= 1 && j <= h) {
                float* d0 = A.dump + (size_t)row * A.planes * N + (size_t)(y0 + j - 1) * nx + x0 + i - 2;
                if (i >= 2 && i < w + 2) {
                    d0[0] = Bk[2].x;
                    d0[N] = mo.d.x;
                    if (A.planes == 4) {
                        d0[2 * (size_t)N] = mo.jx.x;
                        d0[3 * (size_t)N] = mo.jy.x;
                    }
                }
                if (i + 1 >= 2 && i + 1 < w + 2) {
                    d0[1] = Bk[2].y;
                    d0[N + 1] = mo.d.y;
                    if (A.planes == 4) {
                        d0[2 * (size_t)N + 1] = mo.jx.y;
                        d0[3 * (size_t)N + 1] = mo.jy.y;
                    }
                }
            }
            float2 gs[9];
            collide2<OM1>(mo, f, mul2(pc, Sx), mul2(pc, Sy), A.k, gs);
            float* g = G + j * LW + i;
#pragma unroll
            for (int v = 0; v < 9; ++v) put2(g + v * S, gs[v]);
        }
    };
    auto is_traced = [&](int s) { return A.keep_every > 0 && (a.t + s) % A.keep_every == 0; };
    bool traced = is_traced(0);
    collide(0, en, traced);
    row += traced;

    for (int s = 0;; ++s) {
        __syncthreads();
        // ---- streaming into the tile: f(t+1), its moments and dpsi(t+1)
        const bool last = s + 1 == A.steps;
        const unsigned tag = A.tag + (unsigned)s + 1u;
        // (test hook: the first tile's words carry a number nobody waits for)
        const unsigned mark = a.skip_unit0 && blockIdx.x == 0 ? tag - 1u : tag;
        uint2* llp = A.llp + (size_t)(tag & 1u) * N;
        uint4* llm = A.llm + (size_t)(tag & 1u) * kQuads<OM1> * N;
        for (int p = tid; p < on; p += nt) {
            const int e = lo[p], jo = e >> 16, io = e & 0xffff;   // within the tile
            const int j = jo + 1, i = io + 2;
            const float* g = G + j * LW + i;
            float2 f[9];
            f[0] = at2(g);
            f[1] = shifted2(g + 1 * S - 1);
            f[2] = at2(g + 2 * S - LW);
            f[3] = shifted2(g + 3 * S + 1);
            f[4] = at2(g + 4 * S + LW);
            f[5] = shifted2(g + 5 * S - LW - 1);
            f[6] = shifted2(g + 6 * S - LW + 1);
            f[7] = shifted2(g + 7 * S + LW + 1);
            f[8] = shifted2(g + 8 * S + LW - 1);
            const float2 ga = add2(f[2], add2(f[5], f[6]));
            const float2 g0 = add2(f[0], add2(f[1], f[3]));
            const float2 gb = add2(f[4], add2(f[8], f[7]));
            const float2 rho1 = add2(add2(ga, g0), gb);
#pragma unroll
            for (int v = 0; v < 9; ++v) f[v] = stored2<T>(f[v]);
            const bool two = io + 1 < w;
            const int y = y0 + jo, x = x0 + io, site = y * nx + x;
            if (last) {
                const float2 dp = make_float2(dpsi_of(rho1.x, a), dpsi_of(rho1.y, a));
                T* gr = a.g_out + (size_t)y * a.pitch;
                for (int q = 0; q < (two ? 2 : 1); ++q) {
                    auto c = [&](int v) { return q ? f[v].y : f[v].x; };
                    const int cs = tsingle(x + q), cp = tpair<T>(x + q);
                    st_(gr + cs + TL::P0, c(0));
                    st_(gr + cs + TL::P2, c(2));
                    st_(gr + cs + TL::P4, c(4));
                    st2<TL::A13, TL::B13>(gr + cp, c(1), c(3));
                    st2<TL::A56, TL::B56>(gr + cp, c(5), c(6));
                    st2<TL::A78, TL::B78>(gr + cp, c(7), c(8));
                    a.dpsi_out[site + q] = q ? dp.y : dp.x;
                }
                continue;
            }
            // (the second column of a pair is the neighbour's if w is odd: not written here)
            const Moments2 mo = moments2(f);
            const bool yedge1 = jo < 1 || jo >= h - 1;
            const bool e1a = yedge1 || io < 1 || io >= w - 1, e1b = two && (yedge1 || io + 1 >= w - 1);
            float* m = M + j * LW + i;
            if (OM1) {
                if (e1a) put_word(llm + site, mo.d.x, mo.jx.x, mo.jy.x, mark);
                if (e1b) put_word(llm + site + 1, mo.d.y, mo.jx.y, mo.jy.y, mark);
                m[0] = mo.d.x;
                m[S] = mo.jx.x;
                m[2 * S] = mo.jy.x;
                if (two) {
                    m[1] = mo.d.y;
                    m[S + 1] = mo.jx.y;
                    m[2 * S + 1] = mo.jy.y;
                }
            } else {
#pragma unroll
                for (int v = 0; v < 3; ++v) {
                    uint4* dst = llm + (size_t)v * N + site;
                    if (e1a) put_word(dst, f[3 * v].x, f[3 * v + 1].x, f[3 * v + 2].x, mark);
                    if (e1b) put_word(dst + 1, f[3 * v].y, f[3 * v + 1].y, f[3 * v + 2].y, mark);
                }
#pragma unroll
                for (int v = 0; v < 9; ++v) {
                    m[v * S] = f[v].x;
                    if (two) m[v * S + 1] = f[v].y;
                }
            }
            const float2 dp = make_float2(dpsi_of(rho1.x, a), dpsi_of(rho1.y, a));
            const bool yedge3 = jo < 3 || jo >= h - 3;
            if (yedge3 || io < 3 || io >= w - 3) put_word(llp + site, dp.x, mark);
            if (two && (yedge3 || io + 1 < 3 || io + 1 >= w - 3)) put_word(llp + site + 1, dp.y, mark);
            float* pp = P + (jo + 3) * PW + io + 4;
            pp[0] = dp.x;
            if (two) pp[1] = dp.y;
        }
        if (last) return;
        __syncthreads();
        // ---- collisions that need no halo, while the neighbours' values arrive
        traced = is_traced(s + 1);
        collide(0, nfree, traced);
        long long t_first = 0;
        unsigned polls = 0;
        auto give_up = [&]() { return wait_over(a, &s_fail, polls, t_first); };
        for (int q = tid; q < nm * kQuads<OM1> + np; q += nt) {
            if (q < nm * kQuads<OM1>) {
                const int u = OM1 ? 0 : q / nm;
                const int2 e = hm[q - u * nm];
                const uint4* src = llm + (size_t)u * N + e.y;
                uint4 v = get_word(src);
                while (v.w != tag && !give_up()) v = get_word(src);
                float* m = M + e.x + 3 * u * S;
                m[0] = __uint_as_float(v.x);
                m[S] = __uint_as_float(v.y);
                m[2 * S] = __uint_as_float(v.z);
            } else {
                const int2 e = hp[q - nm * kQuads<OM1>];
                uint2 v = get_word(llp + e.y);
                while (v.y != tag && !give_up()) v = get_word(llp + e.y);
                P[e.x] = __uint_as_float(v.x);
            }
        }
        __syncthreads();
        if (s_fail) return;
        collide(nfree, en, traced);
        row += traced;
    }
}

template <typename T, bool OM1>
cudaError_t launch_resident(const ResArgs<T>& A, int grid, int threads, size_t smem, cudaStream_t s)
{
    // the limit, not this launch's size: another thread may be launching another lattice
    cudaError_t e = cudaFuncSetAttribute(k_resident<T, OM1>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         kHeldSmem);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeCooperative;   // every tile waits for its neighbours'
    at.val.cooperative = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k_resident<T, OM1>, A);
}

// `steps` steps from a's buffers; states with a trace row, or all of them as four planes
// each, are left in `dump`.
template <typename T>
cudaError_t resident_launch(const StepArgs<T>& a, ResidentBuf& b, int steps, float* dump, int planes,
                            int keep_every, cudaStream_t s)
{
    ResArgs<T> A{};
    A.a = a;
    A.k = packed_args(a);
    A.gx = b.gx;
    A.tw = b.tw;
    A.th = b.th;
    A.steps = steps;
    A.tag = b.tag;
    A.llp = b.llp;
    A.llm = b.llm;
    A.dump = dump;
    A.planes = planes;
    A.keep_every = keep_every;
    const bool om1 = a.omega == 1.0f;
    const size_t smem = res_smem(b.tw, b.th, om1);
    // a thread per collision pair and per halo word, from 256 on (us per step, 256 / 384 /
    // 512 / 768 threads: 128^2 1.80 / 1.81 / 1.86 / 1.96, 250x187 2.49 / 2.31 / 2.36 / 2.48,
    // 512^2 5.43 / 4.47 / 4.48 / 4.28)
    const int pairs = (b.tw + 4) / 2 * (b.th + 2);
    const int words = halo_psi(b.tw, b.th) + (om1 ? 1 : 3) * halo_mom(b.tw, b.th);
    int threads = ((pairs > words ? pairs : words) + 31) / 32 * 32;
    const int most = om1 ? kResThreads<true> : kResThreads<false>;
    threads = threads < 256 ? 256 : threads > most ? most : threads;
    const cudaError_t e = om1 ? launch_resident<T, true>(A, b.gx * b.gy, threads, smem, s)
                              : launch_resident<T, false>(A, b.gx * b.gy, threads, smem, s);
    if (e == cudaSuccess) b.tag += (unsigned)steps;
    return e;
}

template <typename T>
cudaError_t resident_steps(const StepArgs<T>& a, ResidentBuf& b, int block_x, int steps, cudaStream_t s)
{
    const cudaError_t e = resident_launch<T>(a, b, steps, b.dump, 2, b.trace_every, s);
    if (e != cudaSuccess || b.trace_every == 0) return e;
    const long long te = b.trace_every, first = (a.t + te - 1) / te * te;
    const int rows = first < a.t + steps ? (int)((a.t + steps - 1 - first) / te + 1) : 0;
    if (rows == 0) return cudaSuccess;
    TraceRows r{};
    r.dpsi = b.dump;
    r.dev = b.dump + a.N;
    r.apart = 2 * (size_t)a.N;
    r.count = rows;
    r.t = first;
    r.every = b.trace_every;
    r.block_x = block_x;
    r.partials = b.partials;
    r.counters = b.counters;
    return trace_rows(a, r, s);
}

}  // namespace

// Tiles of a lattice for k_resident: one per SM at most; false if it does not fit the
// SMs' shared memory (about 690^2 with omega = 1, 570^2 otherwise, on 152 SMs). The tile
// grid is the one that makes a CTA's step shortest: collisions of the tile and its ring,
// streaming, halo words; tiles of at least 64 sites, below which only the number of
// neighbours grows (16x16: 1.70 us per step with 128 sites, 4.18 with single sites).
bool resident_plan(int nx, int ny, bool om1, int num_sms, ResidentBuf& b)
{
    double best = 1e30;
    b.gx = 0;
    for (int gx = 1; gx <= num_sms; ++gx) {
        const int tw = ((nx + gx - 1) / gx + 1) / 2 * 2;
        if ((nx + tw - 1) / tw != gx) continue;
        for (int gy = 1; gy <= num_sms / gx; ++gy) {
            const int th = (ny + gy - 1) / gy;
            if ((ny + th - 1) / th != gy) continue;
            if (res_smem(tw, th, om1) > kHeldSmem) continue;
            if (tw * th < 64 && gx * gy > 1) continue;
            const double cost = (tw + 4) / 2 * (th + 2) + 0.5 * tw * th / 2 + 0.5 * halo_psi(tw, th);
            if (cost < best) {
                best = cost;
                b.gx = gx;
                b.gy = gy;
                b.tw = tw;
                b.th = th;
            }
        }
    }
    return b.gx > 0;
}

cudaError_t fp32_resident(const StepArgs<float>& a, ResidentBuf& b, int block_x, int steps, cudaStream_t s)
{
    return resident_steps<float>(a, b, block_x, steps, s);
}
cudaError_t fp32_resident_kept(const StepArgs<float>& a, ResidentBuf& b, int steps, float* states,
                               cudaStream_t s)
{
    return resident_launch<float>(a, b, steps, states, 4, 1, s);
}
cudaError_t fp32_resident_probe(const StepArgs<float>& a, ResidentBuf& b, cudaStream_t s)
{
    return resident_launch<float>(a, b, 1, nullptr, 2, 0, s);
}
cudaError_t fp16_resident(const StepArgs<__half>& a, ResidentBuf& b, int block_x, int steps, cudaStream_t s)
{
    return resident_steps<__half>(a, b, block_x, steps, s);
}

}  // namespace lbsc
