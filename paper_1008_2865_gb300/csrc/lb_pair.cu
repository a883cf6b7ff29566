// lb_pair.cu — two plain steps t -> t+2 of the fused update in one pass over the
// lattice (k_step2), for FP32 and FP16 states.
//
// A plain step by itself (k_step, lb_fp32.cu) moves 80 bytes per site and runs at
// 0.95 of the copy bandwidth at 8192^2, so the only way on is fewer passes: here the
// state t+1 never leaves the SM, and a site costs 40 bytes per step. What bounds
// the kernel then is instruction issue (63% of the slots busy, 5.2 TB/s of HBM
// traffic at 4096^2), so every thread works on two adjacent columns with packed FP32
// instructions (lb_packed.cuh): about 190 instructions per site and step, halo
// included, against 343 of k_step. 8192^2, us per plain step: FP32 827 -> 495,
// FP16 717 -> 445; 2050x1999 63.7 -> 37.9; 1024^2 20.5 -> 14.4.
//
// A CTA of TH threads owns 2 TH - 8 output columns (two steps need a halo of four
// collision columns on each side) and marches down its rows. Iteration r: stage 1
// (t -> t+1) streams its collision row r and collides row r+1; dpsi(t+1) of row r-1
// goes to a ring in shared memory; stage 2 (t+1 -> t+2) collides row r-4, whose
// stencil rows r-6 .. r-2 are complete, and streams row r-5 into the output. A chunk
// of rows costs four (stage 1) and one (stage 2) collision rows more at either end.
// With omega = 1 a collision needs only the moments of f(t+1), not the populations:
// they are summed as the speeds arrive, and a row waits in shared memory as three
// values per site instead of nine (496 against 524 us per FP32 step at 8192^2).
//
// Measured and not kept, us per step at 8192^2 (FP32 / FP16; 498 / 445 as it is): strips of
// 184 and 248 columns (TH = 96, 128) 502 / 481 and 517 / 472; 16 instead of 12 resident
// FP32 warps per SM, at 128 registers with 12 bytes spilled, 551 (FP16 fits 128 without
// spills and gains 4%); populations unpacked or loaded later than at the top of the
// iteration 568; the rings' first rows repeated behind the last, so that a stencil is
// one base address, 500 / 456; the row loop unrolled by two 498 / 505; dpsi rows loaded
// an iteration earlier 504 / 498; streaming loads 534 / 449, stores 495 / 449; without the
// L2 prefetch of the population rows 619 (with an earlier form of the rest). Stage 1 alone,
// streamed into the output, as a single step of its own: 920 / 523, and 16.5 at 1024^2
// against 14.4. In a narrow last strip the second warp only keeping the barriers:
// 96-replica batch 192 against 178. Odd nx with the test for split pairs only in the strips
// at the periodic edge, two bodies in one kernel: 46.1 against 41.0 at 2051x1999.
//
// Every site's arithmetic is that of k_step, operation by operation, so the fields
// are bit-identical to two single steps. If state t has a trace row, stage 1 leaves its
// density deviations in memory (4 bytes per site) and the row is formed from them and
// dpsi afterwards (lb_trace.cu): 0.28 ms at 8192^2, against 0.73 ms that a reduction step
// and a plain one cost more than a pair.
#include "lb_packed.cuh"

#include <type_traits>
#include <utility>
#include <vector>

namespace lbsc {
namespace {

using namespace dev;

// Two adjacent values of the population storage type, as they lie in shared memory.
template <typename T>
struct PairOf;
template <>
struct PairOf<float> {
    using type = float2;
};
template <>
struct PairOf<__half> {
    using type = __half2;
};
__device__ __forceinline__ float2 widen(float2 v) { return v; }
__device__ __forceinline__ float2 widen(__half2 v) { return __half22float2(v); }
__device__ __forceinline__ void narrow(float2* p, float2 v) { *p = v; }
__device__ __forceinline__ void narrow(__half2* p, float2 v) { *p = __float22half2_rn(v); }

// The populations of a thread's two columns as loaded. They are taken apart only
// where they are used: a register move of a loaded value waits for the load, so
// unpacking at the load would give away the prefetch.
template <typename T>
struct RawCols;
template <>
struct RawCols<float> {
    float2 s0, s2, s4;          // speeds 0, 2, 4 of both columns
    float4 q13, q56, q78;       // (first column's pair, second column's pair)
    __device__ __forceinline__ void unpack(float2 f[9]) const
    {
        f[0] = s0;
        f[2] = s2;
        f[4] = s4;
        f[1] = make_float2(q13.x, q13.z);
        f[3] = make_float2(q13.y, q13.w);
        f[5] = make_float2(q56.x, q56.z);
        f[6] = make_float2(q56.y, q56.w);
        f[7] = make_float2(q78.x, q78.z);
        f[8] = make_float2(q78.y, q78.w);
    }
};
template <>
struct RawCols<__half> {
    __half2 s0, s2, s4;
    uint2 q13, q56, q78;
    static __device__ __forceinline__ void two(uint2 q, float2& a, float2& b)
    {
        const float2 lo = __half22float2(*reinterpret_cast<const __half2*>(&q.x));
        const float2 hi = __half22float2(*reinterpret_cast<const __half2*>(&q.y));
        a = make_float2(lo.x, hi.x);
        b = make_float2(lo.y, hi.y);
    }
    __device__ __forceinline__ void unpack(float2 f[9]) const
    {
        f[0] = __half22float2(s0);
        f[2] = __half22float2(s2);
        f[4] = __half22float2(s4);
        two(q13, f[1], f[3]);
        two(q56, f[5], f[6]);
        two(q78, f[7], f[8]);
    }
};
__device__ __forceinline__ void st_two(float* p, float2 v) { *reinterpret_cast<float2*>(p) = v; }
__device__ __forceinline__ void st_two(__half* p, float2 v)
{
    *reinterpret_cast<__half2*>(p) = __float22half2_rn(v);
}
__device__ __forceinline__ void st_four(float* p, float2 a, float2 b)
{
    *reinterpret_cast<float4*>(p) = make_float4(a.x, b.x, a.y, b.y);
}
__device__ __forceinline__ void st_four(__half* p, float2 a, float2 b)
{
    const __half2 lo = __floats2half2_rn(a.x, b.x), hi = __floats2half2_rn(a.y, b.y);
    uint2 v;
    v.x = *reinterpret_cast<const unsigned int*>(&lo);
    v.y = *reinterpret_cast<const unsigned int*>(&hi);
    *reinterpret_cast<uint2*>(p) = v;
}

// A thread's two columns in the population tiles. ODD (nx odd): the pair may be
// split by the periodic edge or start at an odd column there; `vec` says that the
// two columns are one aligned pair.
struct Cols {
    int csa, cpa;   // single and pair offsets of the first column
    int csb, cpb;   // of the second (ODD)
    bool vec;
};

template <bool ODD>
__device__ __forceinline__ void load_cols(RawCols<float>& f, const float* __restrict__ row,
                                          const Cols& c)
{
    using L = Tile<float>;
    if (!ODD || c.vec) {
        f.s0 = __ldg(reinterpret_cast<const float2*>(row + c.csa + L::P0));
        f.s2 = __ldg(reinterpret_cast<const float2*>(row + c.csa + L::P2));
        f.s4 = __ldg(reinterpret_cast<const float2*>(row + c.csa + L::P4));
        f.q13 = __ldg(reinterpret_cast<const float4*>(row + c.cpa + L::A13));
        f.q56 = __ldg(reinterpret_cast<const float4*>(row + c.cpa + L::A56));
        f.q78 = __ldg(reinterpret_cast<const float4*>(row + c.cpa + L::A78));
    } else {
        auto pair = [&](int o) { return __ldg(reinterpret_cast<const float2*>(row + o)); };
        f.s0 = make_float2(__ldg(row + c.csa + L::P0), __ldg(row + c.csb + L::P0));
        f.s2 = make_float2(__ldg(row + c.csa + L::P2), __ldg(row + c.csb + L::P2));
        f.s4 = make_float2(__ldg(row + c.csa + L::P4), __ldg(row + c.csb + L::P4));
        const float2 a13 = pair(c.cpa + L::A13), b13 = pair(c.cpb + L::A13);
        const float2 a56 = pair(c.cpa + L::A56), b56 = pair(c.cpb + L::A56);
        const float2 a78 = pair(c.cpa + L::A78), b78 = pair(c.cpb + L::A78);
        f.q13 = make_float4(a13.x, a13.y, b13.x, b13.y);
        f.q56 = make_float4(a56.x, a56.y, b56.x, b56.y);
        f.q78 = make_float4(a78.x, a78.y, b78.x, b78.y);
    }
}

template <bool ODD>
__device__ __forceinline__ void load_cols(RawCols<__half>& f, const __half* __restrict__ row,
                                          const Cols& c)
{
    using L = Tile<__half>;
    if (!ODD || c.vec) {
        f.s0 = __ldg(reinterpret_cast<const __half2*>(row + c.csa + L::P0));
        f.s2 = __ldg(reinterpret_cast<const __half2*>(row + c.csa + L::P2));
        f.s4 = __ldg(reinterpret_cast<const __half2*>(row + c.csa + L::P4));
        f.q13 = __ldg(reinterpret_cast<const uint2*>(row + c.cpa + L::A13));
        f.q56 = __ldg(reinterpret_cast<const uint2*>(row + c.cpa + L::A56));
        f.q78 = __ldg(reinterpret_cast<const uint2*>(row + c.cpa + L::A78));
    } else {
        auto pair = [&](int o) { return __ldg(reinterpret_cast<const unsigned int*>(row + o)); };
        f.s0 = __halves2half2(__ldg(row + c.csa + L::P0), __ldg(row + c.csb + L::P0));
        f.s2 = __halves2half2(__ldg(row + c.csa + L::P2), __ldg(row + c.csb + L::P2));
        f.s4 = __halves2half2(__ldg(row + c.csa + L::P4), __ldg(row + c.csb + L::P4));
        f.q13 = make_uint2(pair(c.cpa + L::A13), pair(c.cpb + L::A13));
        f.q56 = make_uint2(pair(c.cpa + L::A56), pair(c.cpb + L::A56));
        f.q78 = make_uint2(pair(c.cpa + L::A78), pair(c.cpb + L::A78));
    }
}

// dpsi of the two columns at src + xa, src + xb (nx even: one aligned pair)
template <bool ODD>
__device__ __forceinline__ float2 load_dpsi(const float* __restrict__ src, int xa, int xb)
{
    if (!ODD) return __ldg(reinterpret_cast<const float2*>(src + xa));
    return make_float2(__ldg(src + xa), __ldg(src + xb));
}

// Start fetching `bytes` (a multiple of 16, 16-byte aligned) from HBM into L2.
__device__ __forceinline__ void prefetch_l2(const void* p, unsigned bytes)
{
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(bytes) : "memory");
}

template <typename T, int TH, bool OM1>
struct PairShared {
    float2 win[2][8][TH + 2];        // dpsi(t), dpsi(t+1) rows, slot = row & 7
    float exR[2][2][3][TH + 2];      // right-moving f* of the second column: speeds 8, 1, 5
    float exL[2][2][3][TH + 2];      // left-moving f* of the first column: speeds 7, 3, 6
    // f(t+1) of the own columns, slot = row & 3: with OM1 its moments, which are all
    // that stage 2 needs then, otherwise the populations
    float2 mom[OM1 ? 4 : 1][3][OM1 ? TH : 1];
    typename PairOf<T>::type g1[OM1 ? 1 : 4][9][OM1 ? 1 : TH];
};

// A value as the population storage type holds it.
template <typename T>
__device__ __forceinline__ float2 stored(float2 v);
template <>
__device__ __forceinline__ float2 stored<float>(float2 v)
{
    return v;
}
template <>
__device__ __forceinline__ float2 stored<__half>(float2 v)
{
    return __half22float2(__float22half2_rn(v));
}

// A row of f(t+1) before its speeds 4, 7, 8 arrive: the parts of moments2 that the
// others make up (p of d, q of -jx), and the speeds whose sums wait for the missing ones.
struct Half2Row {
    float2 p, q, f2, f5, f6;
};

// What a thread keeps of a collision row for the streaming after the barrier.
struct Own {
    float2 c0, c2, c4;     // speeds 0, 2, 4 (own columns)
    float r8, r1, r5;      // right-moving values of the first column (into the second)
    float l7, l3, l6;      // left-moving values of the second column (into the first)
};

// Collision of a row's two sites from the dpsi ring, their moments and (without OM1)
// the populations f; the
// values leaving the thread's columns go to the exchange buffers.
template <bool OM1, typename T, int TH>
__device__ __forceinline__ void collide_row(const PackedArgs& k, const float2 (*win)[TH + 2], int r,
                                            const Moments2& m, const float2 f[9], float (*exR)[TH + 2], float (*exL)[TH + 2], Own& o)
{
    const int tid = threadIdx.x;
    float2 A[5], B[5], C[5];
#pragma unroll
    for (int j = 0; j < 5; ++j) {
        const float2* w = &win[(r - 2 + j) & 7][tid];
        A[j] = w[0];
        B[j] = w[1];
        C[j] = w[2];
    }
    float2 Sx, Sy;
    force_sums2(A, B, C, k, Sx, Sy);
    const float2 pc = add2(k.psi_ref, B[2]);
    float2 gs[9];
    collide2<OM1>(m, f, mul2(pc, Sx), mul2(pc, Sy), k, gs);
    exR[0][tid + 1] = gs[8].y;
    exR[1][tid + 1] = gs[1].y;
    exR[2][tid + 1] = gs[5].y;
    exL[0][tid + 1] = gs[7].x;
    exL[1][tid + 1] = gs[3].x;
    exL[2][tid + 1] = gs[6].x;
    o.c0 = gs[0];
    o.c2 = gs[2];
    o.c4 = gs[4];
    o.r8 = gs[8].x;
    o.r1 = gs[1].x;
    o.r5 = gs[5].x;
    o.l7 = gs[7].y;
    o.l3 = gs[3].y;
    o.l6 = gs[6].y;
}

template <typename T, int TH, bool OM1, bool ODD, bool TRACE>
__device__ __forceinline__ void pair_tile(const StepArgs<T>& a, const PackedArgs& k, PairShared<T, TH, OM1>& sh, int x0, int y0,
                                          int y1)
{
    constexpr int W = 2 * TH - 8;
    const int tid = threadIdx.x;
    const int nx = a.nx, ny = a.ny;
    const int N = (int)a.N, P = a.pitch, NP = a.npitch;
    using TL = Tile<T>;
    const int xa = wrapi(x0 - 4 + 2 * tid, nx), xb = xa + 1 == nx ? 0 : xa + 1;
    Cols c;
    c.csa = tsingle(xa);
    c.cpa = tpair<T>(xa);
    c.csb = tsingle(xb);
    c.cpb = tpair<T>(xb);
    c.vec = !ODD || (xb == xa + 1 && (xa & 1) == 0);
    const int xlim = min(x0 + W, nx);
    const int xo = x0 - 4 + 2 * tid;                 // output column (threads 2 .. TH - 3)
    const bool outa = tid >= 2 && tid < TH - 2 && xo < xlim;
    const bool outb = !ODD ? outa : outa && xo + 1 < xlim;
    // the two column pairs beyond the threads' own, loaded by threads 0 and 1
    const int xe = tid == 0 ? wrapi(x0 - 6, nx) : wrapi(x0 - 4 + 2 * TH, nx);
    const int xe1 = xe + 1 == nx ? 0 : xe + 1;
    const int slot_e = tid == 0 ? 0 : TH + 1;

    const int rs = y0 - 4;
    for (int rr = rs - 2; rr <= rs + 3; ++rr) {
        const float* src = a.dpsi_in + wrapi(rr, ny) * nx;
        sh.win[0][rr & 7][tid + 1] = load_dpsi<ODD>(src, xa, xb);
        if (tid < 2) sh.win[0][rr & 7][slot_e] = load_dpsi<ODD>(src, xe, xe1);
    }
    int la = wrapi(rs, ny) * P;                       // g row offset of the next load
    int oq = wrapi(rs + 4, ny) * nx;                  // dpsi row offset of the next load
    RawCols<T> f;
    load_cols<ODD>(f, a.g_in + la, c);
    la = la + P == NP ? 0 : la + P;
    __syncthreads();
    Own o1, o2;
    float2 f1[9];
    f.unpack(f1);
    // TRACE: the density deviations of state t at the tile's own sites
    float* dev = TRACE ? a.dev + (long long)(rs + 1) * nx + xa : nullptr;   // row r + 1
    collide_row<OM1, T, TH>(k, sh.win[0], rs, moments2(f1), f1, sh.exR[0][rs & 1], sh.exL[0][rs & 1], o1);
    load_cols<ODD>(f, a.g_in + la, c);
    la = la + P == NP ? 0 : la + P;
    o2.c0 = o2.c2 = o2.c4 = make_float2(0.f, 0.f);
    o2.r8 = o2.r1 = o2.r5 = o2.l7 = o2.l3 = o2.l6 = 0.f;
    const float2 zero = make_float2(0.f, 0.f);
    float2 hb1 = zero, zb1 = zero, hc1 = zero, hb2 = zero, zb2 = zero, hc2 = zero;
    float2 h2 = zero, h5 = zero, h6 = zero;           // speeds 2, 5, 6 of f(t+1) in row r
    Half2Row hr{zero, zero, zero, zero, zero};        // row r - 1 of f(t+1) without speeds 4, 7, 8 (OM1)
    T* gp = a.g_out + (long long)(rs - 5) * P;        // g row of stage 2's collision row

    // the strip's population tiles of a row, [tl, t1), and past the periodic edge
    // [0, t2): one thread has them fetched into L2 three rows ahead of their load (us per
    // step at 8192^2 with two, three, four, eight rows: FP16 446, 442, 451, 448; FP32 495,
    // 497, 501, 536)
    constexpr int kAhead = 3;
    const int tl = wrapi(x0 - 4, nx) >> 5, tiles = (nx + 31) >> 5;
    const int span = (2 * TH + 31 + 31) / 32;
    const int t1 = min(tl + span, tiles), t2 = min(span - (t1 - tl), tl);
    int lp = wrapi(rs + 2 + kAhead, ny) * P;
    // One row: stage 1 streams its collision row r and collides row r + 1, stage 2
    // streams its collision row r - 5 and collides row r - 4. S1, S2: whether the stage
    // still (already) collides; the rows at a chunk's ends where only one stage has work
    // are loops of their own, so that the main loop is free of branches.
    auto body = [&](auto s1, auto s2, int r) {
        constexpr bool S1 = decltype(s1)::value, S2 = decltype(s2)::value;
        __syncthreads();
        const int b = r & 1;
        if (S1 && tid == 32 && r + 2 + kAhead <= y1 + 3) {
            prefetch_l2(a.g_in + lp + tl * kTileElems, (t1 - tl) * kTileElems * sizeof(T));
            if (t2 > 0) prefetch_l2(a.g_in + lp, t2 * kTileElems * sizeof(T));
        }
        lp = lp + P == NP ? 0 : lp + P;
        float2 pn = zero, pe = zero;
        const bool mored = S1 && r + 4 <= y1 + 5;
        if (mored) {
            const float* src = a.dpsi_in + oq;
            pn = load_dpsi<ODD>(src, xa, xb);
            if (tid < 2) pe = load_dpsi<ODD>(src, xe, xe1);
        }
        oq = oq + nx == N ? 0 : oq + nx;

        // moments of stage 1's next row r + 1; the loads of row r + 2 follow at once,
        // a whole iteration ahead of their use
        Moments2 m1;
        if (S1) {
            f.unpack(f1);
            m1 = moments2(f1);
            if (TRACE) {
                if (outa && r + 1 >= y0 && r + 1 < y1) {
                    if (!ODD) {
                        *reinterpret_cast<float2*>(dev) = m1.d;
                    } else {
                        dev[0] = m1.d.x;
                        if (outb) dev[1] = m1.d.y;
                    }
                }
                dev += nx;
            }
        }
        if (S1 && r + 2 <= y1 + 3) load_cols<ODD>(f, a.g_in + la, c);
        la = la + P == NP ? 0 : la + P;

        // stage 2's row r - 4 of f(t+1) (slot of row r; the populations are overwritten below)
        float2 f2[9];
        Moments2 m2;
        if (S2 && OM1) {
            const float2(*m)[TH] = reinterpret_cast<const float2(*)[TH]>(sh.mom[OM1 ? r & 3 : 0]);
            m2.d = m[0][tid];
            m2.jx = m[1][tid];
            m2.jy = m[2][tid];
        } else if (S2) {
#pragma unroll
            for (int i = 0; i < 9; ++i) f2[i] = widen(sh.g1[OM1 ? 0 : r & 3][i][OM1 ? 0 : tid]);
            m2 = moments2(f2);
        }

        // ---- stage 1: stream collision row r; f(t+1) and dpsi(t+1) of row r - 1
        {
            const float (*eR)[TH + 2] = sh.exR[0][b], (*eL)[TH + 2] = sh.exL[0][b];
            const float3 R = make_float3(eR[0][tid], eR[1][tid], eR[2][tid]);
            const float3 L = make_float3(eL[0][tid + 2], eL[1][tid + 2], eL[2][tid + 2]);
            const float2 v8 = make_float2(R.x, o1.r8), v1 = make_float2(R.y, o1.r1),
                         v5 = make_float2(R.z, o1.r5);
            const float2 v7 = make_float2(o1.l7, L.x), v3 = make_float2(o1.l3, L.y),
                         v6 = make_float2(o1.l6, L.z);
            if (OM1) {
                // moments2 of row r - 1, whose speeds 4, 7, 8 are the last to arrive, in
                // its order: what the row's earlier speeds contribute waits in hr
                const float2 f4 = stored<T>(o1.c4), f7 = stored<T>(v7), f8 = stored<T>(v8);
                float2(*m)[TH] = reinterpret_cast<float2(*)[TH]>(sh.mom[OM1 ? (r - 1) & 3 : 0]);
                m[0][tid] = add2(add2(hr.p, add2(add2(f4, hr.f5), add2(hr.f6, f7))), f8);
                m[1][tid] = add2(hr.q, sub2(f7, f8));
                m[2][tid] = sub2(add2(f7, f8), add2(sub2(hr.f2, f4), add2(hr.f5, hr.f6)));
                const float2 f0 = stored<T>(o1.c0), f1 = stored<T>(v1), f3 = stored<T>(v3);
                hr.p = add2(add2(f0, f1), add2(h2, f3));
                hr.q = add2(sub2(f3, f1), sub2(h6, h5));
                hr.f2 = h2;
                hr.f5 = h5;
                hr.f6 = h6;
                h2 = stored<T>(o1.c2);
                h5 = stored<T>(v5);
                h6 = stored<T>(v6);
            } else {
                auto* gm = sh.g1[OM1 ? 0 : (r - 1) & 3];
                auto* gc = sh.g1[OM1 ? 0 : r & 3];
                const int i = OM1 ? 0 : tid;
                narrow(&gm[4][i], o1.c4);
                narrow(&gm[7][i], v7);
                narrow(&gm[8][i], v8);
                narrow(&gc[0][i], o1.c0);
                narrow(&gc[1][i], v1);
                narrow(&gc[3][i], v3);
                narrow(&gc[2][i], h2);
                narrow(&gc[5][i], h5);
                narrow(&gc[6][i], h6);
                h2 = o1.c2;
                h5 = v5;
                h6 = v6;
            }
            const float2 gb = add2(o1.c4, add2(v8, v7));
            const float2 g0 = add2(o1.c0, add2(v1, v3));
            const float2 ga = add2(o1.c2, add2(v5, v6));
            const float2 rho1 = add2(add2(hb1, zb1), gb);
            sh.win[1][(r - 1) & 7][tid + 1] = make_float2(dpsi_of(rho1.x, a), dpsi_of(rho1.y, a));
            hb1 = hc1;
            zb1 = g0;
            hc1 = ga;
        }
        // ---- stage 2: stream collision row p = r - 5 into f(t+2)
        if (S2) {
            const int p = r - 5;
            const float (*eR)[TH + 2] = sh.exR[1][b], (*eL)[TH + 2] = sh.exL[1][b];
            const float3 R = make_float3(eR[0][tid], eR[1][tid], eR[2][tid]);
            const float3 L = make_float3(eL[0][tid + 2], eL[1][tid + 2], eL[2][tid + 2]);
            const float2 v8 = make_float2(R.x, o2.r8), v1 = make_float2(R.y, o2.r1),
                         v5 = make_float2(R.z, o2.r5);
            const float2 v7 = make_float2(o2.l7, L.x), v3 = make_float2(o2.l3, L.y),
                         v6 = make_float2(o2.l6, L.z);
            const bool st_b = outa && p > y0 && p <= y1;
            const bool st_0 = outa && p >= y0 && p < y1;
            const bool st_a = outa && p >= y0 - 1 && p < y1 - 1;
            if (!ODD || outb) {
                if (st_b) {
                    st_two(gp - P + c.csa + TL::P4, o2.c4);
                    st_four(gp - P + c.cpa + TL::A78, v7, v8);
                }
                if (st_0) {
                    st_two(gp + c.csa + TL::P0, o2.c0);
                    st_four(gp + c.cpa + TL::A13, v1, v3);
                }
                if (st_a) {
                    st_two(gp + P + c.csa + TL::P2, o2.c2);
                    st_four(gp + P + c.cpa + TL::A56, v5, v6);
                }
            } else {
                if (st_b) {
                    st_(gp - P + c.csa + TL::P4, o2.c4.x);
                    st2<TL::A78, TL::B78>(gp - P + c.cpa, v7.x, v8.x);
                }
                if (st_0) {
                    st_(gp + c.csa + TL::P0, o2.c0.x);
                    st2<TL::A13, TL::B13>(gp + c.cpa, v1.x, v3.x);
                }
                if (st_a) {
                    st_(gp + P + c.csa + TL::P2, o2.c2.x);
                    st2<TL::A56, TL::B56>(gp + P + c.cpa, v5.x, v6.x);
                }
            }
            const float2 gb = add2(o2.c4, make_float2(v8.x + v7.x, v8.y + v7.y));
            const float2 g0 = add2(o2.c0, make_float2(v1.x + v3.x, v1.y + v3.y));
            const float2 ga = add2(o2.c2, make_float2(v5.x + v6.x, v5.y + v6.y));
            const float2 rho1 = add2(add2(hb2, zb2), gb);
            if (st_b) {
                const float2 d = make_float2(dpsi_of(rho1.x, a), dpsi_of(rho1.y, a));
                float* dst = a.dpsi_out + (p - 1) * nx + xa;
                if (!ODD) {
                    *reinterpret_cast<float2*>(dst) = d;
                } else {
                    dst[0] = d.x;
                    if (outb) dst[1] = d.y;
                }
            }
            hb2 = hc2;
            zb2 = g0;
            hc2 = ga;
        }
        gp += P;
        // ---- the next collision rows of both stages
        if (S2)
            collide_row<OM1, T, TH>(k, sh.win[1], r - 4, m2, f2, sh.exR[1][b ^ 1], sh.exL[1][b ^ 1], o2);
        if (S1)
            collide_row<OM1, T, TH>(k, sh.win[0], r + 1, m1, f1, sh.exR[0][b ^ 1], sh.exL[0][b ^ 1], o1);
        if (mored) {
            sh.win[0][(r + 4) & 7][tid + 1] = pn;
            if (tid < 2) sh.win[0][(r + 4) & 7][slot_e] = pe;
        }
    };
    using Yes = std::true_type;
    using No = std::false_type;
    int r = rs;
    for (; r <= y0 + 2; ++r) body(Yes{}, No{}, r);
    for (; r <= y1 + 2; ++r) body(Yes{}, Yes{}, r);
    for (; r <= y1 + 5; ++r) body(No{}, Yes{}, r);
}

// Resident threads per SM the registers are cut for: 16 warps where the kernel fits
// 128 registers (FP16; with omega != 1 8 bytes are spilled, 494 us per step at 8192^2
// against 522-549 with 12 warps), otherwise 12.
template <typename T>
constexpr int kPairThreads = sizeof(T) == 2 ? 512 : 384;
constexpr int kTH = kPairTH;

template <typename T, int TH, bool OM1, bool ODD, bool TRACE>
__global__ void __launch_bounds__(TH, kPairThreads<T> / TH)
    k_step2(const StepArgs<T> a, const PackedArgs k, int rows)
{
    __shared__ PairShared<T, TH, OM1> sh;
    const int y0 = blockIdx.y * rows;
    pair_tile<T, TH, OM1, ODD, TRACE>(a, k, sh, blockIdx.x * (2 * TH - 8), y0, min(y0 + rows, a.ny));
}

// Output rows per CTA: one wave of resident CTAs, because a chunk's ends cost ten rows
// of one stage or the other (2050x1999, us per step: 37.8 with one wave, 46.3 with two;
// 1500^2 23.6 and 30.7); two waves once that leaves chunks of more than 400 rows, where
// the ends no longer count and CTAs that fall behind do (8192^2: 493 with two waves of
// 316 rows, 532 with one of 631; 6000^2, 334 rows: 263 with one, 268 with two). At
// least 8 rows.
template <typename T>
int pair_rows(int nx, int ny)
{
    const int strips = (nx + kPairCols - 1) / kPairCols;
    const int slots = 152 * (kPairThreads<T> / kTH);
    auto rows_for = [&](int waves) {
        const int chunks = slots * waves / strips;
        return chunks > 1 ? (ny + chunks - 1) / chunks : ny;
    };
    int rows = rows_for(1);
    if (rows > 400) rows = rows_for(2);
    return rows < 8 ? 8 : rows;
}

// f(omega == 1, odd nx, traced) with the three as compile-time constants
template <typename F>
cudaError_t with_flags(bool om1, bool odd, bool traced, F f)
{
    using Y = std::true_type;
    using N = std::false_type;
    if (traced) {
        if (om1) return odd ? f(Y{}, Y{}, Y{}) : f(Y{}, N{}, Y{});
        return odd ? f(N{}, Y{}, Y{}) : f(N{}, N{}, Y{});
    }
    if (om1) return odd ? f(Y{}, Y{}, N{}) : f(Y{}, N{}, N{});
    return odd ? f(N{}, Y{}, N{}) : f(N{}, N{}, N{});
}

template <typename T>
cudaError_t launch_pair(const StepArgs<T>& a, bool traced, cudaStream_t s)
{
    constexpr int W = kPairCols;
    const bool om1 = a.omega == 1.0f;
    const int rows = pair_rows<T>(a.nx, a.ny);
    const dim3 grid((a.nx + W - 1) / W, (a.ny + rows - 1) / rows);
    return with_flags(om1, a.nx & 1, traced, [&](auto o, auto d, auto t) {
        k_step2<T, kTH, decltype(o)::value, decltype(d)::value, decltype(t)::value>
            <<<grid, kTH, 0, s>>>(a, packed_args(a), rows);
        return cudaGetLastError();
    });
}

// The pairs of a batch: a persistent grid strides over a work list of tiles (replica,
// first column, first row, end row) of every replica. The replica's arguments are
// staged in shared memory by warp 0 when the replica changes.
template <typename T, bool OM1, bool ODD, bool TRACE>
__global__ void __launch_bounds__(kTH, kPairThreads<T> / kTH)
    k_step2_batch(const StepArgs<T>* __restrict__ args, const int4* __restrict__ tiles, int ntiles)
{
    __shared__ PairShared<T, kTH, OM1> sh;
    __shared__ StepArgs<T> sa;
    __shared__ PackedArgs sk;
    __shared__ int sa_rep;
    if (threadIdx.x == 0) sa_rep = -1;
    for (int i = blockIdx.x; i < ntiles; i += gridDim.x) {
        const int4 tl = __ldg(tiles + i);
        __syncthreads();                            // previous tile done with the shared memory
        if (threadIdx.x < 32 && tl.x != sa_rep) {
            const int* src = reinterpret_cast<const int*>(args + tl.x);
            int* dst = reinterpret_cast<int*>(&sa);
            for (int w = threadIdx.x; w < (int)(sizeof(StepArgs<T>) / 4); w += 32)
                dst[w] = __ldg(src + w);
            __syncwarp();
            if (threadIdx.x == 0) {
                sk = packed_args(sa);
                sa_rep = tl.x;
            }
        }
        __syncthreads();
        const StepArgs<T> a = sa;
        pair_tile<T, kTH, OM1, ODD, TRACE>(a, sk, sh, tl.y, tl.z, tl.w);
    }
}

template <typename T>
cudaError_t launch_batch_pair(const BatchLaunch<T>& b, const int4* tiles, int ntiles, bool odd,
                              bool traced, cudaStream_t s)
{
    const int per_sm = kPairThreads<T> / kTH;
    const int grid = ntiles < per_sm * b.num_sms ? ntiles : per_sm * b.num_sms;
    return with_flags(b.om1, odd, traced, [&](auto o, auto d, auto t) {
        k_step2_batch<T, decltype(o)::value, decltype(d)::value, decltype(t)::value>
            <<<grid, kTH, 0, s>>>(b.args, tiles, ntiles);
        return cudaGetLastError();
    });
}

}  // namespace

// Work list of a batch's pair kernel. Chunk heights are balanced within a replica;
// the height is the one that makes the estimated time least: waves of resident CTAs,
// each as long as its tallest tile plus nine rows (the two half-busy ends of a tile
// and its prologue).
void pair_tiles(const std::vector<std::pair<int, int>>& sizes, int elem_bytes, int num_sms,
                std::vector<int4>& tiles)
{
    constexpr int W = kPairCols;
    const int threads = elem_bytes == 2 ? kPairThreads<__half> : kPairThreads<float>;
    const long long slots = (long long)(threads / kTH) * num_sms;
    auto chunks_of = [](int ny, int rows) { return (ny + rows - 1) / rows; };
    int tallest = 8;
    for (const auto& s : sizes) tallest = s.second > tallest ? s.second : tallest;
    int best = 8;
    double best_cost = 1e30;
    for (int rows = 8; rows <= tallest && rows <= 1024; ++rows) {
        long long n = 0;
        int high = 0;
        for (const auto& s : sizes) {
            const int c = chunks_of(s.second, rows), h = (s.second + c - 1) / c;
            n += (long long)((s.first + W - 1) / W) * c;
            high = h > high ? h : high;
        }
        const double cost = (double)((n + slots - 1) / slots) * (high + 9);
        if (cost < best_cost) {
            best_cost = cost;
            best = rows;
        }
    }
    for (size_t r = 0; r < sizes.size(); ++r) {
        const int ny = sizes[r].second, c = chunks_of(ny, best), h = (ny + c - 1) / c;
        for (int y = 0; y < ny; y += h)
            for (int x = 0; x < sizes[r].first; x += W)
                tiles.push_back(make_int4((int)r, x, y, y + h < ny ? y + h : ny));
    }
}

cudaError_t fp32_batch_pair(const BatchLaunch<float>& b, const int4* tiles, int ntiles, bool odd,
                            bool traced, cudaStream_t s)
{
    return launch_batch_pair<float>(b, tiles, ntiles, odd, traced, s);
}
cudaError_t fp16_batch_pair(const BatchLaunch<__half>& b, const int4* tiles, int ntiles, bool odd,
                            bool traced, cudaStream_t s)
{
    return launch_batch_pair<__half>(b, tiles, ntiles, odd, traced, s);
}

cudaError_t fp32_step_pair(const StepArgs<float>& a, bool traced, cudaStream_t s)
{
    return launch_pair<float>(a, traced, s);
}
cudaError_t fp16_step_pair(const StepArgs<__half>& a, bool traced, cudaStream_t s)
{
    return launch_pair<__half>(a, traced, s);
}

}  // namespace lbsc
