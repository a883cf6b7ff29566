// lb_adjoint.cu — lb_adjoint: the gradient of
//   J = E_s(T) + E_m(T) + sum_x (rho(x, T) - rho*(x))^2
// (Sec. 5 pseudo-energy of the final state plus a squared misfit to a target
// density) with respect to the initial density field and the couplings G1, G2
// of Eq. FORCE, for an FP32 state, by a hand-written reverse sweep of the
// fused step with sqrt(T) checkpointing.
//
// Forward (Eqs. 1-4, Eq. FORCE):  rho, j = moments of f;  psi(rho);
//   F = -psi(x) S(x), S = sum_c K_c c psi(x+c);  v = (j + F/omega)/rho;
//   f*_i = (1-omega) f_i + omega feq_i(rho, v);  f_i(x + c_i, t+1) = f*_i(x).
// Reverse, with l' = dJ/df(t+1) and l* the streamed-back adjoint
// l*_i(x) = l'_i(x + c_i):
//   pass A (per site x):
//     rho-bar = omega sum_i l*_i feq_i / rho - (v-bar . v) / rho
//     v-bar   = omega rho sum_i l*_i w_i (3 c_i + 9 (c_i.v) c_i - 3 v)
//     j-bar   = v-bar / rho,  F-bar = v-bar / (omega rho)
//     psi-bar(x) gets -F-bar . S (the leading psi(x) of F(x)); Q = psi F-bar
//     dJ/dG1 += -psi F-bar . S_w,  dJ/dG2 += -psi F-bar . S_p  (S = G1 S_w + G2 S_p)
//   pass B (per site y): psi-bar(y) += sum_c K_c c . Q(y + c) (the transpose of the
//     force stencil; K_c = K_{-c}); rho-bar += psi'(rho) psi-bar;
//     l_i(y) = (1 - omega) l*_i(y) + rho-bar(y) + c_i . j-bar(y).
// Terminal: l_i(y, T) = psi'(rho) sum_{c incl. rest} K_c psi(y+c) + 2 (rho - rho*).
// Start: dJ/drho_init(x) = sum_i w_i l_i(x, 0).
// The state and the adjoint are FP32; J and the G1, G2 gradients accumulate
// in FP64 (per-thread, then deterministic CTA and grid sums).
#include <cmath>
#include <new>
#include <vector>

#include "lb_packed.cuh"

using namespace lbsc;
using namespace lbsc::dev;

namespace {

constexpr int kAdjThreads = 256;
constexpr int kAdjMaxBlocks = 152 * (2048 / kAdjThreads);   // one full wave of threads

// Periodic neighbourhood of site (x, y), computed once per site (nx, ny >= 5):
// columns x-2 .. x+2 and row offsets (y-2 .. y+2) * nx.
struct Nbr5 {
    int xo[5];
    int yo[5];
};

__device__ __forceinline__ Nbr5 nbr5(int x, int y, int nx, int ny)
{
    Nbr5 n;
#pragma unroll
    for (int k = 0; k < 5; ++k) {
        int xx = x + k - 2, yy = y + k - 2;
        xx += xx < 0 ? nx : 0;
        xx -= xx >= nx ? nx : 0;
        yy += yy < 0 ? ny : 0;
        yy -= yy >= ny ? ny : 0;
        n.xo[k] = xx;
        n.yo[k] = yy * nx;
    }
    return n;
}

// The 5 x 5 neighbourhood of a periodic FP32 field: v[k][m] = field(x + m - 2, y + k - 2).
// For a column away from the periodic x edges (2 <= x < nx - 2, `xin`) each row is
// one pointer with immediate offsets; otherwise every column offset is wrapped.
__device__ __forceinline__ void gather5(const float* __restrict__ fld, const Nbr5& nb, int x,
                                        bool xin, float v[5][5])
{
    if (xin) {
#pragma unroll
        for (int k = 0; k < 5; ++k) {
            const float* r = fld + nb.yo[k] + x;
#pragma unroll
            for (int m = 0; m < 5; ++m) v[k][m] = __ldg(r + (m - 2));
        }
    } else {
#pragma unroll
        for (int k = 0; k < 5; ++k) {
#pragma unroll
            for (int m = 0; m < 5; ++m) v[k][m] = __ldg(fld + nb.yo[k] + nb.xo[m]);
        }
    }
}

// The same for the (Qx, Qy) pairs of pass B: one 8-byte load per stencil site.
__device__ __forceinline__ void gather5x2(const float2* __restrict__ fld, const Nbr5& nb, int x,
                                          bool xin, float vx[5][5], float vy[5][5])
{
    if (xin) {
#pragma unroll
        for (int k = 0; k < 5; ++k) {
            const float2* r = fld + nb.yo[k] + x;
#pragma unroll
            for (int m = 0; m < 5; ++m) {
                const float2 q = __ldg(r + (m - 2));
                vx[k][m] = q.x;
                vy[k][m] = q.y;
            }
        }
    } else {
#pragma unroll
        for (int k = 0; k < 5; ++k) {
#pragma unroll
            for (int m = 0; m < 5; ++m) {
                const float2 q = __ldg(fld + nb.yo[k] + nb.xo[m]);
                vx[k][m] = q.x;
                vy[k][m] = q.y;
            }
        }
    }
}

// D2Q9 speeds in the order of the populations (compile-time in unrolled loops).
__host__ __device__ constexpr int cx_of(int i)
{
    return (i == 1 || i == 5 || i == 8) ? 1 : (i == 3 || i == 6 || i == 7) ? -1 : 0;
}
__host__ __device__ constexpr int cy_of(int i)
{
    return (i == 2 || i == 5 || i == 6) ? 1 : (i == 4 || i == 7 || i == 8) ? -1 : 0;
}

// Deviations f_i(x, y) - w_i rho_ref of state t, read from the tiled populations.
template <typename T>
__device__ __forceinline__ void site_f(const T* __restrict__ g, int pitch, int x, int y,
                                       float f[9])
{
    load_site_xy(f, g, pitch, x, y);
}

struct AdjArgs {
    StepArgs<float> a;        // couplings, weights, rho_ref, psi_ref, omega of the state
    StepArgs<float> aw;       // couplings replaced by the D2Q9 weights (S_w)
    StepArgs<float> ap;       // couplings replaced by the E(8) weights (S_p)
    float G1, G2;
    float inv_sqrt_rho0;      // 1 / sqrt(rho0): psi'(rho) = exp(-rho/rho0) / sqrt(rho0)
    const float* g;           // tiled f(t) - w rho_ref
    const float* dpsi;        // dpsi(t)
    const float* lam_next;    // [9][N] dJ/df(t+1)
    float* lam;               // [9][N] dJ/df(t)
    float4* lam4;             // instead of lam, with omega = 1: (rho-bar, j-bar x, j-bar y)
    float4* site;             // per site (j-bar x, j-bar y, rho-bar so far, psi'(rho))
    float2* Q;                // per site psi F-bar (x, y), read by pass B as a stencil
    const double* rho_target; // terminal kernel
    double* partials;
    unsigned int* counter;
    double* acc;              // [4] FP64 accumulators
    int* narrow;              // flags of the terminal kernel's sums
};

// s += x with Kahan's compensation c (the rounding error of the previous adds).
// The operations must not be reassociated: nvcc does not, and fmaf is not used.
__device__ __forceinline__ void kahan_add(float& s, float& c, float x)
{
    const float y = __fsub_rn(x, c);
    const float t = __fadd_rn(s, y);
    c = __fsub_rn(__fsub_rn(t, s), y);
    s = t;
}

template <int NT>
__device__ void accumulate_grid(double v[4], const AdjArgs& A)
{
    if (last_block_total<NT>(v, A.partials, A.counter, gridDim.x)) {
#pragma unroll
        for (int k = 0; k < 4; ++k) A.acc[k] += v[k];
    }
}

// Grid sum of two per-thread values added into A.acc[0..1] with little FP64
// work (FP64 issues slowly on this part) and no long dependent chains: the
// CTA's values meet in shared memory, each lane of warp 0 adds NT/32 of them in
// FP32 in a fixed order, the 32 lane sums go to FP64 and a fixed shuffle tree
// adds them; the last CTA to finish sums the CTA partials in FP64 in CTA order
// (loads issued four at a time). Error: each FP32 lane sum adds at most NT/32
// per-thread values, so its relative error is below (NT/32) 2^-24 of the sum of
// their magnitudes; everything above it is FP64.
template <int NT>
__device__ void accumulate_grid2(float v0, float v1, const AdjArgs& A)
{
    __shared__ float sh[2][NT];
    __shared__ bool s_last;
    const int tid = threadIdx.x;
    sh[0][tid] = v0;
    sh[1][tid] = v1;
    __syncthreads();
    if (tid < 32) {
        float a0 = 0.f, a1 = 0.f;
#pragma unroll
        for (int k = tid; k < NT; k += 32) {
            a0 += sh[0][k];
            a1 += sh[1][k];
        }
        double w0 = a0, w1 = a1;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            w0 += __shfl_down_sync(0xffffffffu, w0, o);
            w1 += __shfl_down_sync(0xffffffffu, w1, o);
        }
        if (tid == 0) {
            reinterpret_cast<double2*>(A.partials)[blockIdx.x] = make_double2(w0, w1);
            __threadfence();
            s_last = atomicAdd(A.counter, 1u) == gridDim.x - 1;
        }
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    double w0 = 0.0, w1 = 0.0;
    const double2* p2 = reinterpret_cast<const double2*>(A.partials);
    unsigned int j = tid;
    for (; j + 3 * NT < gridDim.x; j += 4 * NT) {
        double2 q[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) q[u] = __ldcg(p2 + j + u * NT);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            w0 += q[u].x;
            w1 += q[u].y;
        }
    }
    for (; j < gridDim.x; j += NT) {
        const double2 q = __ldcg(p2 + j);
        w0 += q.x;
        w1 += q.y;
    }
    double v[4] = {w0, w1, 0.0, 0.0};
    block_sum4<NT>(v);
    if (tid == 0) {
        A.acc[0] += v[0];
        A.acc[1] += v[1];
        *A.counter = 0u;
    }
}

// J of the state (gT, A.dpsi) and, with GRAD, the terminal adjoint l(T) and the explicit
// dE/dG1, dE/dG2 (lb_objective takes J alone; its sums are the same additions). T is the
// population storage type. Rows of CTAs' sites are read as in k_delta_energy; a thread's
// sums of psi times a class sum are exact FP32 products in two FP32 values (Two), the
// misfit, whose target is FP64, is summed in FP64. A thread whose sums leave the range of Two
// (as in k_delta_energy) sets bit 1 (E) or 2 (the derivatives) of *A.narrow, and these are
// taken again with WIDE, in FP64 and without the adjoint.
template <typename T, bool GRAD, bool WIDE>
__global__ void __launch_bounds__(kAdjThreads) k_adj_terminal(const AdjArgs A,
                                                              const T* __restrict__ gT)
{
    const StepArgs<float>& a = A.a;
    const int nx = a.nx, ny = a.ny, N = (int)a.N;
    Two e{0.f, 0.f}, e1{0.f, 0.f}, e2{0.f, 0.f};
    float most = 0.f, most1 = 0.f;            // largest terms of e and e1
    double mis2 = 0.0, w0 = 0.0, w1 = 0.0, w2 = 0.0;
    for (int s = blockIdx.x * kAdjThreads + threadIdx.x; s < N; s += gridDim.x * kAdjThreads) {
        const int y = s / nx, x = s - y * nx;
        const double target = __ldg(A.rho_target + s);
        float f[9];
        site_f(gT, a.pitch, x, y, f);
        const float d = ((f[0] + f[1]) + (f[2] + f[3])) + ((f[4] + f[5]) + (f[6] + f[7])) + f[8];
        const float rho = a.rho_ref + d;
        const Nbr5 nb = nbr5(x, y, nx, ny);
        const bool xin = x >= 2 && x < nx - 2;
        float p[5][5];
        gather5(A.dpsi, nb, x, xin, p);
        const float pr = a.psi_ref;
        const float pc = pr + p[2][2];
        // class sums of psi (not deviations) around the site
        const float S1 = fmaf(4.f, pr, (p[2][3] + p[2][1]) + (p[3][2] + p[1][2]));
        const float S2 = fmaf(4.f, pr, (p[3][3] + p[3][1]) + (p[1][3] + p[1][1]));
        const float S4 = fmaf(4.f, pr, (p[2][4] + p[2][0]) + (p[4][2] + p[0][2]));
        const float S5 = fmaf(8.f, pr, ((p[3][4] + p[3][0]) + (p[1][4] + p[1][0])) +
                                           ((p[4][3] + p[4][1]) + (p[0][3] + p[0][1])));
        const float S8 = fmaf(4.f, pr, (p[4][4] + p[4][0]) + (p[0][4] + p[0][0]));
        const float dEdpsi = a.K0 * pc + a.K1 * S1 + a.K2 * S2 + a.K4 * S4 + a.K5 * S5 + a.K8 * S8;
        const double mis = (double)rho - target;
        mis2 += mis * mis;
        const float sw = A.aw.K0 * pc + A.aw.K1 * S1 + A.aw.K2 * S2;
        const float sp = A.ap.K0 * pc + A.ap.K1 * S1 + A.ap.K2 * S2 + A.ap.K4 * S4 +
                         A.ap.K5 * S5 + A.ap.K8 * S8;
        if (WIDE) {
            w0 += 0.5 * (double)pc * dEdpsi;
            if (GRAD) {
                w1 += 0.5 * (double)pc * sw;
                w2 += 0.5 * (double)pc * sp;
            }
            continue;
        }
        auto add_product = [&](Two& sum, float u, float v) {
            const float q = __fmul_rn(u, v);
            two_add(sum, q, __fmaf_rn(u, v, -q));
            return fabsf(q);
        };
        most = fmaxf(most, add_product(e, pc, dEdpsi));
        if (GRAD) {
            const float dpr = __expf(-rho * a.inv_rho0) * A.inv_sqrt_rho0;
            const float lam = dpr * dEdpsi + (float)(2.0 * mis);
            if (A.lam4) {
                A.lam4[s] = make_float4(lam, 0.f, 0.f, 0.f);
            } else {
#pragma unroll
                for (int i = 0; i < 9; ++i) A.lam[i * N + s] = lam;
            }
            most1 = fmaxf(most1, add_product(e1, pc, sw));
            add_product(e2, pc, sp);
        }
    }
    if (!WIDE) {
        w0 = 0.5 * value(e);
        w1 = 0.5 * value(e1);
        w2 = 0.5 * value(e2);
        // without couplings E is zero, whatever psi is
        const bool coupled = a.K0 != 0.f || a.K1 != 0.f || a.K2 != 0.f || a.K4 != 0.f;
        int bits = (most >= kNarrowLeast || !coupled) && isfinite(w0) ? 0 : 1;
        if (GRAD && !(most1 >= kNarrowLeast && isfinite(w1) && isfinite(w2))) bits |= 2;
        if (bits && blockIdx.x * kAdjThreads + threadIdx.x < N) atomicOr(A.narrow, bits);
    }
    // E, misfit, dE/dG1, dE/dG2
    double v[4] = {w0, mis2, w1, w2};
    accumulate_grid<kAdjThreads>(v, A);
}

// Pass A of one site: from its stencil p, its density deviation and momentum and the
// streamed-back adjoint ls, the values pass B needs (sv: j-bar x, j-bar y, rho-bar so far,
// psi'(rho); Q = psi F-bar) and the site's terms of dJ/dG1 and dJ/dG2. (One body for both
// callers: the compiler's choice of fused multiply-adds in it decides the last bits. The
// same in packed pairs of sites, with 546 instead of 821 instructions per site and step
// in k_adj_reverse, was 6% faster there but changed them.)
__device__ __forceinline__ void adj_site(const AdjArgs& A, const float p[5][5], float d, float jx,
                                         float jy, const float ls[9], float4& sv, float2& Q,
                                         float& x1, float& x2)
{
    const StepArgs<float>& a = A.a;
    const float om = a.omega;
    const float w[9] = {a.w0, a.w1, a.w1, a.w1, a.w1, a.w2, a.w2, a.w2, a.w2};
    const float rho = a.rho_ref + d;
    const float* rows[5] = {&p[0][2], &p[1][2], &p[2][2], &p[3][2], &p[4][2]};
    float Swx, Swy, Spx, Spy;
    force_sums(rows, A.aw, Swx, Swy);
    force_sums(rows, A.ap, Spx, Spy);
    const float Sx = A.G1 * Swx + A.G2 * Spx, Sy = A.G1 * Swy + A.G2 * Spy;
    const float pc = a.psi_ref + p[2][2];
    const float Fx = -pc * Sx, Fy = -pc * Sy;
    const float inv = __frcp_rn(rho);
    const float vx = fmaf(Fx, a.inv_omega, jx) * inv, vy = fmaf(Fy, a.inv_omega, jy) * inv;
    const float usq = vx * vx + vy * vy;
    // rho-bar gets omega sum_i l*_i feq_i / rho = omega sum_i l*_i w_i (1 + 3 c.v + ...);
    // v-bar = omega rho sum_i l*_i w_i (3 c_i + 9 (c_i.v) c_i - 3 v)
    float rb = 0.f, vbx = 0.f, vby = 0.f;
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        const int ci = cx_of(i), cj = cy_of(i);
        const float lw = w[i] * ls[i];
        const float cu = ci * vx + cj * vy;
        rb += lw * (1.f + 3.f * cu + 4.5f * cu * cu - 1.5f * usq);
        const float t9 = 9.f * cu;
        vbx += lw * (3.f * ci + t9 * ci - 3.f * vx);
        vby += lw * (3.f * cj + t9 * cj - 3.f * vy);
    }
    rb *= om;
    vbx *= om * rho;
    vby *= om * rho;
    const float Fbx = vbx * inv * a.inv_omega, Fby = vby * inv * a.inv_omega;
    rb -= (vbx * vx + vby * vy) * inv;
    const float dpr = __expf(-rho * a.inv_rho0) * A.inv_sqrt_rho0;
    sv = make_float4(vbx * inv, vby * inv, rb + dpr * (-(Fbx * Sx + Fby * Sy)), dpr);
    Q = make_float2(pc * Fbx, pc * Fby);
    x1 = -pc * (Fbx * Swx + Fby * Swy);
    x2 = -pc * (Fbx * Spx + Fby * Spy);
}

__global__ void __launch_bounds__(kAdjThreads) k_adj_pass_a(const AdjArgs A)
{
    const StepArgs<float>& a = A.a;
    const int nx = a.nx, ny = a.ny, N = (int)a.N;
    // dJ/dG1, dJ/dG2: per thread a compensated FP32 sum (Kahan: the running sum
    // stays within about one FP32 rounding of the exact sum of its terms, however
    // many sites the thread visits), then accumulate_grid2
    float f1 = 0.f, f2 = 0.f, c1 = 0.f, c2 = 0.f;
    for (int s = blockIdx.x * kAdjThreads + threadIdx.x; s < N; s += gridDim.x * kAdjThreads) {
        const int y = s / nx, x = s % nx;
        float f[9];
        site_f(A.g, a.pitch, x, y, f);
        const float d = ((f[0] + f[1]) + (f[2] + f[3])) + ((f[4] + f[5]) + (f[6] + f[7])) + f[8];
        const float jx = (f[1] - f[3]) + (f[5] - f[6]) + (f[8] - f[7]);
        const float jy = (f[2] - f[4]) + (f[5] + f[6]) - (f[7] + f[8]);
        const Nbr5 nb = nbr5(x, y, nx, ny);
        const bool xin = x >= 2 && x < nx - 2;
        float p[5][5];
        gather5(A.dpsi, nb, x, xin, p);
        // l*_i(x) = l'_i(x + c_i): the adjoint streamed back
        float ls[9];
#pragma unroll
        for (int i = 0; i < 9; ++i)
            ls[i] = __ldg(A.lam_next + i * N + nb.yo[2 + cy_of(i)] + nb.xo[2 + cx_of(i)]);
        float x1, x2;
        adj_site(A, p, d, jx, jy, ls, A.site[s], A.Q[s], x1, x2);
        kahan_add(f1, c1, x1);
        kahan_add(f2, c2, x2);
    }
    accumulate_grid2<kAdjThreads>(f1, f2, A);
}

__global__ void __launch_bounds__(kAdjThreads) k_adj_pass_b(const AdjArgs A)
{
    const StepArgs<float>& a = A.a;
    const int nx = a.nx, ny = a.ny, N = (int)a.N;
    const float omc = a.omc;
    for (int s = blockIdx.x * kAdjThreads + threadIdx.x; s < N; s += gridDim.x * kAdjThreads) {
        const int y = s / nx, x = s % nx;
        // sum_c K_c c . Q(y + c): the x part is the force stencil of Qx, the y part of
        // Qy (one 8-byte load per stencil site for both)
        const Nbr5 nb = nbr5(x, y, nx, ny);
        const bool xin = x >= 2 && x < nx - 2;
        float qx[5][5], qy[5][5];
        gather5x2(A.Q, nb, x, xin, qx, qy);
        const float* rx[5] = {&qx[0][2], &qx[1][2], &qx[2][2], &qx[3][2], &qx[4][2]};
        const float* ry[5] = {&qy[0][2], &qy[1][2], &qy[2][2], &qy[3][2], &qy[4][2]};
        float sx, sy, tx, ty;
        force_sums(rx, a, sx, sy);
        force_sums(ry, a, tx, ty);
        const float4 sv = __ldg(A.site + s);
        const float rb = sv.z + sv.w * (sx + ty);
        const float jbx = sv.x, jby = sv.y;
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            const int ci = cx_of(i), cj = cy_of(i);
            const float ls = __ldg(A.lam_next + i * N + nb.yo[2 + cj] + nb.xo[2 + ci]);
            A.lam[i * N + s] = fmaf(omc, ls, rb + ci * jbx + cj * jby);
        }
    }
}

// ---- omega = 1 on a lattice that fits the SMs: a segment's reverse steps in one launch.
//
// At 512^2 the two passes took 28 us per step, launches and latency. With omega = 1 pass
// B gives l_i = rho-bar + c_i . j-bar: the adjoint of a site is three numbers, not nine,
// and one kernel holds a tile's adjoint in shared memory over a segment as k_resident
// holds its state (tiles, halo words and their argument as there; the words are the three
// numbers and the step's). A reverse step needs them in three rings around the tile, the
// moments of the state in two (pass A of two rings is recomputed) and dpsi in four; the next
// state is copied in while a step runs. 8.1 us per step at 512^2, bound by instruction
// issue (60% of the slots, 775 instructions per site and step, the rings included). On
// lattices that do not fit, the same kernel with one step per launch took 207 us at 2048^2
// against 175 us of the two passes, which therefore stay, as they do for other omega.
// The terms of dJ/dG are left in a buffer and summed afterwards, in the order of
// k_adj_pass_a's threads (k_adj_sums).
//
// The states are moments and dpsi as k_resident keeps them ([4][N], momentum negated); the
// launch is cooperative and takes `steps` of them, last first.
struct RevArgs {
    AdjArgs A;
    int gx, tw, th;             // tiles per row of tiles, tile size
    int steps;
    unsigned tag;               // steps exchanged before this launch
    const float* states;        // [steps][4][N] in forward order
    const float4* lam_in;       // (rho-bar, j-bar x, j-bar y) after the last state
    float4* lam_out;            // before the first
    uint4* words;               // [2][N] halo words
    float* terms;               // [steps][2][N] of dJ/dG1, dJ/dG2 in reverse order
};

__host__ __device__ inline int rev_floats(int tw, int th)
{
    return 2 * (tw + 8) * (th + 8) + 2 * 3 * (tw + 4) * (th + 4) + 3 * (tw + 8) * (th + 6) +
           2 * (tw + 4) * (th + 4) + tw * th + (tw + 8) * (th + 8) +
           2 * ((tw + 6) * (th + 6) - tw * th);
}

__device__ __forceinline__ void copy_async(float* dst, const float* src)
{
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(d), "l"(src) : "memory");
}

constexpr int kRevThreads = 768;   // at most

__global__ void __launch_bounds__(kRevThreads, 1) k_adj_reverse(const RevArgs R)
{
    extern __shared__ __align__(16) float sm[];
    __shared__ int s_fail, s_nl;
    if (R.steps == 0) return;                            // asked whether the launch is taken
    const AdjArgs& A = R.A;
    const StepArgs<float>& a = A.a;
    const int tid = threadIdx.x, nt = blockDim.x, warps = nt >> 5, warp = tid >> 5, lane = tid & 31;
    const int nx = a.nx, ny = a.ny, N = (int)a.N;
    const int x0 = (blockIdx.x % R.gx) * R.tw, y0 = (blockIdx.x / R.gx) * R.th;
    const int w = min(R.tw, nx - x0), h = min(R.th, ny - y0);
    const int PW = R.tw + 8, QW = R.tw + 4;
    const int PS = PW * (R.th + 8), QS = QW * (R.th + 4), LS = PW * (R.th + 6);
    float* P = sm;                                       // [2] dpsi, four rings
    float* M = P + 2 * PS;                               // [2][3] moments, two rings; then sv
    float2* Q = reinterpret_cast<float2*>(M + 6 * QS);   // two rings
    float* L = reinterpret_cast<float*>(Q + QS);                              // [3] adjoint, three rings (and a column)
    float* D = L + 3 * LS;                               // psi'(rho) of the own sites
    int* ps = reinterpret_cast<int*>(D + R.tw * R.th);   // sites of the dpsi tile
    int2* hl = reinterpret_cast<int2*>(ps + PS);         // halo sites of the adjoint

    if (tid == 0) s_fail = s_nl = 0;
    for (int q = tid; q < (w + 8) * (h + 8); q += nt) {
        const int j = q / (w + 8), i = q - j * (w + 8);
        ps[j * PW + i] = wrapi(y0 - 4 + j, ny) * nx + wrapi(x0 - 4 + i, nx);
    }
    __syncthreads();
    for (int q = tid; q < (w + 6) * (h + 6); q += nt) {
        const int j = q / (w + 6), i = q - j * (w + 6) + 1;
        const int site = ps[(j + 1) * PW + i];
        const float4 l = __ldg(R.lam_in + site);
        float* dst = L + j * PW + i;
        dst[0] = l.x;
        dst[LS] = l.y;
        dst[2 * LS] = l.z;
        if (j < 3 || j >= h + 3 || i < 4 || i >= w + 4) hl[atomicAdd(&s_nl, 1)] = make_int2(j * PW + i, site);
    }
    // dpsi and moments of state k into buffer b, a row per warp
    auto fetch = [&](int k, int b) {
        const float* st = R.states + (size_t)k * 4 * N;
        for (int j = warp; j < h + 8; j += warps) {
            for (int i = lane; i < w + 8; i += 32) {
                const int site = ps[j * PW + i];
                copy_async(P + b * PS + j * PW + i, st + site);
                if (j >= 2 && j < h + 6 && i >= 2 && i < w + 6) {
                    float* m = M + b * 3 * QS + (j - 2) * QW + i - 2;
                    copy_async(m, st + N + site);
                    copy_async(m + QS, st + 2 * (size_t)N + site);
                    copy_async(m + 2 * QS, st + 3 * (size_t)N + site);
                }
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    fetch(R.steps - 1, 0);
    // sites: (row, column) of this thread's first, and the stride to its next
    const int ew = w + 4, en = ew * (h + 4), ow = w, on = ow * h;
    const int ej = tid / ew, ec = tid - ej * ew, edj = nt / ew, edc = nt - edj * ew;
    const int oj = tid / ow, oc = tid - oj * ow, odj = nt / ow, odc = nt - odj * ow;
    for (int r = 0; r < R.steps; ++r) {
        const int b = r & 1;
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncthreads();
        if (s_fail) return;
        const int nl = s_nl;
        if (r + 1 < R.steps) fetch(R.steps - 2 - r, b ^ 1);
        const float* Pb = P + b * PS;
        float* Mb = M + b * 3 * QS;
        // ---- pass A of the tile and two rings
        float* t1 = R.terms + (size_t)r * 2 * N;
        for (int q = tid, j = ej, i = ec; q < en; q += nt) {
            const int site = ps[(j + 2) * PW + i + 2];
            float p[5][5];
#pragma unroll
            for (int k = 0; k < 5; ++k) {
#pragma unroll
                for (int m = 0; m < 5; ++m) p[k][m] = Pb[(j + k) * PW + i + m];
            }
            float* mo = Mb + j * QW + i;
            // l*_k(x) = l_k(x + c_k) = rho-bar + c_k . j-bar there
            float ls[9];
#pragma unroll
            for (int k = 0; k < 9; ++k) {
                const int ci = cx_of(k), cj = cy_of(k);
                const float* l = L + (j + 1 + cj) * PW + i + 2 + ci;
                ls[k] = l[0];
                if (ci) ls[k] = ci > 0 ? ls[k] + l[LS] : ls[k] - l[LS];
                if (cj) ls[k] = cj > 0 ? ls[k] + l[2 * LS] : ls[k] - l[2 * LS];
            }
            float4 sv;
            float2 Qv;
            float x1, x2;
            adj_site(A, p, mo[0], -mo[QS], -mo[2 * QS], ls, sv, Qv, x1, x2);
            Q[j * QW + i] = Qv;
            if (j >= 2 && j < h + 2 && i >= 2 && i < w + 2) {
                mo[0] = sv.x;
                mo[QS] = sv.y;
                mo[2 * QS] = sv.z;
                D[(j - 2) * R.tw + i - 2] = sv.w;
                t1[site] = x1;
                t1[N + site] = x2;
            }
            j += edj;
            i += edc;
            if (i >= ew) {
                i -= ew;
                ++j;
            }
        }
        __syncthreads();
        // ---- pass B of the tile
        const bool last = r + 1 == R.steps;
        const unsigned tag = R.tag + (unsigned)r + 1u;
        const unsigned mark = a.skip_unit0 && blockIdx.x == 0 ? tag - 1u : tag;
        uint4* words = R.words + (size_t)(tag & 1u) * N;
        for (int q = tid, j = oj, i = oc; q < on; q += nt) {
            const int site = ps[(j + 4) * PW + i + 4];
            float qx[5][5], qy[5][5];
#pragma unroll
            for (int k = 0; k < 5; ++k) {
#pragma unroll
                for (int m = 0; m < 5; ++m) {
                    const float2 v = Q[(j + k) * QW + i + m];
                    qx[k][m] = v.x;
                    qy[k][m] = v.y;
                }
            }
            const float* rx[5] = {&qx[0][2], &qx[1][2], &qx[2][2], &qx[3][2], &qx[4][2]};
            const float* ry[5] = {&qy[0][2], &qy[1][2], &qy[2][2], &qy[3][2], &qy[4][2]};
            float sx, sy, tx, ty;
            force_sums(rx, a, sx, sy);
            force_sums(ry, a, tx, ty);
            const float* mo = Mb + (j + 2) * QW + i + 2;
            const float rb = mo[2 * QS] + D[j * R.tw + i] * (sx + ty);
            const float jbx = mo[0], jby = mo[QS];
            if (last) {
                R.lam_out[site] = make_float4(rb, jbx, jby, 0.f);
            } else {
                float* l = L + (j + 3) * PW + i + 4;
                l[0] = rb;
                l[LS] = jbx;
                l[2 * LS] = jby;
                if (j < 3 || j >= h - 3 || i < 3 || i >= w - 3) put_word(words + site, rb, jbx, jby, mark);
            }
            j += odj;
            i += odc;
            if (i >= ow) {
                i -= ow;
                ++j;
            }
        }
        if (last) return;
        long long t_first = 0;
        unsigned polls = 0;
        for (int q = tid; q < nl; q += nt) {
            const int2 e = hl[q];
            uint4 v = get_word(words + e.y);
            while (v.w != tag && !wait_over(a, &s_fail, polls, t_first)) v = get_word(words + e.y);
            float* l = L + e.x;
            l[0] = __uint_as_float(v.x);
            l[LS] = __uint_as_float(v.y);
            l[2 * LS] = __uint_as_float(v.z);
        }
    }
}

// The sums of the steps' dJ/dG terms: CTA (b, r) forms what CTA b of k_adj_pass_a and
// accumulate_grid2 leave for step r; k_adj_sums_total adds the CTAs of each step and then,
// in the last CTA to finish, the steps in order.
__global__ void __launch_bounds__(kAdjThreads)
    k_adj_sums(const float* __restrict__ terms, int N, double2* __restrict__ part)
{
    __shared__ float sh[2][kAdjThreads];
    const int tid = threadIdx.x;
    const float* t = terms + (size_t)blockIdx.y * 2 * N;
    float f1 = 0.f, f2 = 0.f, c1 = 0.f, c2 = 0.f;
    for (int s = blockIdx.x * kAdjThreads + tid; s < N; s += gridDim.x * kAdjThreads) {
        kahan_add(f1, c1, __ldg(t + s));
        kahan_add(f2, c2, __ldg(t + N + s));
    }
    sh[0][tid] = f1;
    sh[1][tid] = f2;
    __syncthreads();
    if (tid >= 32) return;
    float a0 = 0.f, a1 = 0.f;
#pragma unroll
    for (int k = tid; k < kAdjThreads; k += 32) {
        a0 += sh[0][k];
        a1 += sh[1][k];
    }
    double w0 = a0, w1 = a1;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        w0 += __shfl_down_sync(0xffffffffu, w0, o);
        w1 += __shfl_down_sync(0xffffffffu, w1, o);
    }
    if (tid == 0) part[(size_t)blockIdx.y * gridDim.x + blockIdx.x] = make_double2(w0, w1);
}

__global__ void __launch_bounds__(kAdjThreads)
    k_adj_sums_total(const double2* __restrict__ part, int ctas, double2* __restrict__ tot,
                     unsigned int* counter, double* acc)
{
    const int tid = threadIdx.x;
    const double2* p = part + (size_t)blockIdx.x * ctas;
    double v[4] = {0.0, 0.0, 0.0, 0.0};
    for (int j = tid; j < ctas; j += kAdjThreads) {
        const double2 q = __ldg(p + j);
        v[0] += q.x;
        v[1] += q.y;
    }
    block_sum4<kAdjThreads>(v);
    if (tid != 0) return;
    tot[blockIdx.x] = make_double2(v[0], v[1]);
    __threadfence();
    if (atomicAdd(counter, 1u) != gridDim.x - 1) return;
    __threadfence();
    double w0 = acc[0], w1 = acc[1];
    for (unsigned r = 0; r < gridDim.x; ++r) {
        const double2 q = __ldcg(tot + r);
        w0 += q.x;
        w1 += q.y;
    }
    acc[0] = w0;
    acc[1] = w1;
    *counter = 0u;
}

// Tiles of the reverse kernel for one CTA per SM; false if they do not fit.
bool reverse_plan(int nx, int ny, int num_sms, RevArgs& R, int& tiles)
{
    double best = 1e30;
    for (int gx = 1; gx <= num_sms; ++gx) {
        const int tw = ((nx + gx - 1) / gx + 1) / 2 * 2;
        if ((nx + tw - 1) / tw != gx) continue;
        for (int gy = 1; gy <= num_sms / gx; ++gy) {
            const int th = (ny + gy - 1) / gy;
            if ((ny + th - 1) / th != gy || (tw * th < 64 && gx * gy > 1)) continue;
            if (4 * (size_t)rev_floats(tw, th) > kHeldSmem) continue;
            const double cost = (tw + 4) * (th + 4) + 0.5 * tw * th;
            if (cost < best) {
                best = cost;
                R.gx = gx;
                R.tw = tw;
                R.th = th;
                tiles = gx * gy;
            }
        }
    }
    return best < 1e30;
}

cudaError_t launch_reverse(const RevArgs& R, int tiles, cudaStream_t s)
{
    const int sites = (R.tw + 4) * (R.th + 4);
    int threads = (sites + 31) / 32 * 32;
    threads = threads < 256 ? 256 : threads > kRevThreads ? kRevThreads : threads;
    // the limit, not this launch's size: another thread may be launching another lattice
    const cudaError_t e =
        cudaFuncSetAttribute(k_adj_reverse, cudaFuncAttributeMaxDynamicSharedMemorySize, kHeldSmem);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(tiles);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = sizeof(float) * (size_t)rev_floats(R.tw, R.th);
    cfg.stream = s;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeCooperative;   // every tile waits for its neighbours'
    at.val.cooperative = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k_adj_reverse, R);
}

__global__ void k_adj_grad_init(const float* __restrict__ lam, const float4* __restrict__ lam4, int N,
                                float w0, float w1, float w2, double* __restrict__ out)
{
    for (int s = blockIdx.x * blockDim.x + threadIdx.x; s < N; s += gridDim.x * blockDim.x) {
        float l[9];
        if (lam4) {
            const float4 v = __ldg(lam4 + s);
#pragma unroll
            for (int i = 0; i < 9; ++i) {
                l[i] = v.x;
                if (cx_of(i)) l[i] = cx_of(i) > 0 ? l[i] + v.y : l[i] - v.y;
                if (cy_of(i)) l[i] = cy_of(i) > 0 ? l[i] + v.z : l[i] - v.z;
            }
        } else {
#pragma unroll
            for (int i = 0; i < 9; ++i) l[i] = __ldg(lam + (size_t)i * N + s);
        }
        out[s] = (double)w0 * l[0] + (double)w1 * (((double)l[1] + l[2]) + ((double)l[3] + l[4])) +
                 (double)w2 * (((double)l[5] + l[6]) + ((double)l[7] + l[8]));
    }
}

int adj_grid(long long n)
{
    long long b = (n + kAdjThreads - 1) / kAdjThreads;
    if (b > kAdjMaxBlocks) b = kAdjMaxBlocks;
    return (int)(b < 1 ? 1 : b);
}

bool dev_ptr(const void* p)
{
    if (!p) return false;
    cudaPointerAttributes at;
    if (cudaPointerGetAttributes(&at, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return at.type == cudaMemoryTypeDevice || at.type == cudaMemoryTypeManaged;
}

StepArgs<float> with_weights(StepArgs<float> a, bool e8)
{
    // the same stencil code with unit couplings: the D2Q9 weights (belt 1 and
    // rest) or the E(8) weights (both belts and rest, Table 1, Eq. weights_1)
    if (!e8) {
        a.K0 = 4.f / 9.f; a.K1 = 1.f / 9.f; a.K2 = 1.f / 36.f; a.K4 = 0.f; a.K5 = 0.f; a.K8 = 0.f;
    } else {
        a.K0 = (float)(247.0 / 420.0); a.K1 = 4.f / 63.f; a.K2 = 4.f / 135.f;
        a.K4 = 1.f / 180.f; a.K5 = 2.f / 945.f; a.K8 = 1.f / 15120.f;
    }
    return a;
}

}  // namespace

extern "C" lb_status lb_adjoint(lb_state* s, long steps, const double* rho_target,
                                int checkpoint_every, double* J_out, double* grad_rho,
                                double* grad_G)
{
    NvtxRange nvtx_range("lb_adjoint");
    if (!s || steps < 0 || !rho_target || !J_out || !grad_rho || !grad_G || checkpoint_every < 0)
        return LB_ERR_ARG;
    if (s->poisoned) return LB_ERR_STATE;
    if (s->p.prec != LB_FP32 || s->t != 0) return LB_ERR_STATE;
    DeviceScope dev(s->p.device);
    if (!dev.ok) return LB_ERR_CUDA;
    const int N = (int)s->N;
    const long long T = steps;
    long long C = checkpoint_every > 0 ? checkpoint_every : (long long)std::ceil(std::sqrt((double)T));
    if (C < 1) C = 1;
    const long long K = T > 0 ? (T + C - 1) / C : 0;     // checkpoints at t = 0, C, 2C, ...
    const size_t GE = (size_t)g_elems(s->p.nx, s->p.ny);
    // populations (GE floats) then dpsi (N), rounded up so that every state starts
    // 256-byte aligned: the populations are read in pairs, and N may be odd
    const size_t slot = (GE + (size_t)N + 63) / 64 * 64;
    cudaStream_t st = s->stream;

    // ---- working memory of one call (freed on return): checkpoints, two segment
    // buffers (states 1 .. C-1 of a segment; state 0 is its checkpoint), the
    // adjoint ping-pong, per-site scratch, and a second stream with its events
    float *ck = nullptr, *seg = nullptr, *lam = nullptr, *scr = nullptr;
    double *tgt = nullptr, *acc = nullptr, *part = nullptr, *grad_dev = nullptr;
    unsigned int* cnt = nullptr;
    cudaStream_t rs = nullptr;                       // recomputation stream
    cudaEvent_t ev_fwd = nullptr, ev_ready[2] = {nullptr, nullptr}, ev_free[2] = {nullptr, nullptr};
    auto release = [&]() {
        void* ptrs[] = {ck, seg, lam, scr, tgt, acc, part, grad_dev, cnt};
        for (void* q : ptrs)
            if (q) cudaFree(q);
        cudaEvent_t evs[] = {ev_fwd, ev_ready[0], ev_ready[1], ev_free[0], ev_free[1]};
        for (cudaEvent_t e : evs)
            if (e) cudaEventDestroy(e);
        if (rs) cudaStreamDestroy(rs);
        cudaGetLastError();
    };
    // held: omega = 1 and the lattice fits the SMs, so that one launch takes a whole
    // segment back (k_adj_reverse), from the moments that a resident recomputation of it
    // leaves behind
    RevArgs R{};
    int rev_tiles = 0, sms = 0;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, s->p.device) != cudaSuccess) {
        cudaGetLastError();
        sms = 0;
    }
    // (segments too short for a held launch take the two passes: 512^2, 20 steps, with a
    // checkpoint at every step 2.08 ms, held 2.47 ms, at every second 1.89 and 1.97 ms)
    bool held = (float)s->p.omega == 1.0f && s->res_buf.gx > 0 &&
                (T < C ? T : C) >= held_least(s->res_buf.tw * s->res_buf.th, true) &&
                reverse_plan(s->p.nx, s->p.ny, sms, R, rev_tiles);
    if (held) {
        // not where the stream refuses either launch, as found out before anything depends on it
        R.steps = 0;
        cudaError_t e = fp32_resident_probe(state_args<float>(s, s->cur), s->res_buf, s->stream);
        if (e == cudaSuccess) e = launch_reverse(R, rev_tiles, s->stream);
        if (e != cudaSuccess && !launch_refused(e)) {
            s->poisoned = true;
            return LB_ERR_CUDA;
        }
        held = e == cudaSuccess;
        cudaGetLastError();
    }
    const int grid = adj_grid(N);
    const long long rows = T < C ? T : C;                 // steps of a segment at most
    const size_t seg_slots = (size_t)(C > 1 ? C - 1 : 1);
    const size_t seg_floats = held ? (size_t)4 * N * (size_t)(rows > 0 ? rows : 1) : slot * 2 * seg_slots;
    const size_t lam_floats = held ? (size_t)8 * N : (size_t)18 * N;
    // scratch: per-site values of the two passes, or the reverse kernel's halo words, the
    // terms of dJ/dG and their sums
    const size_t word_bytes = held ? sizeof(uint4) * 2 * (size_t)N : 0;
    const size_t scr_bytes = held ? word_bytes + sizeof(double2) * (size_t)(grid + 1) * (size_t)(rows + 1) +
                                       sizeof(float) * 2 * (size_t)N * (size_t)(rows > 0 ? rows : 1)
                                 : sizeof(float) * 6 * (size_t)N;
    const bool grad_on_dev = dev_ptr(grad_rho);
    bool ok = cudaMalloc((void**)&ck, sizeof(float) * slot * (size_t)(K > 0 ? K : 1)) == cudaSuccess &&
              cudaMalloc((void**)&seg, sizeof(float) * seg_floats) == cudaSuccess &&
              cudaMalloc((void**)&lam, sizeof(float) * lam_floats) == cudaSuccess &&
              cudaMalloc((void**)&scr, scr_bytes) == cudaSuccess &&
              cudaMalloc((void**)&tgt, sizeof(double) * N) == cudaSuccess &&
              cudaMalloc((void**)&acc, sizeof(double) * 8) == cudaSuccess &&
              cudaMalloc((void**)&part, sizeof(double) * 4 * kAdjMaxBlocks) == cudaSuccess &&
              cudaMalloc((void**)&cnt, sizeof(unsigned int)) == cudaSuccess &&
              (grad_on_dev || cudaMalloc((void**)&grad_dev, sizeof(double) * N) == cudaSuccess);
    if (!ok) {
        release();
        return LB_ERR_OOM;
    }
    if (cudaStreamCreateWithFlags(&rs, cudaStreamNonBlocking) != cudaSuccess ||
        cudaEventCreateWithFlags(&ev_fwd, cudaEventDisableTiming) != cudaSuccess ||
        cudaEventCreateWithFlags(&ev_ready[0], cudaEventDisableTiming) != cudaSuccess ||
        cudaEventCreateWithFlags(&ev_ready[1], cudaEventDisableTiming) != cudaSuccess ||
        cudaEventCreateWithFlags(&ev_free[0], cudaEventDisableTiming) != cudaSuccess ||
        cudaEventCreateWithFlags(&ev_free[1], cudaEventDisableTiming) != cudaSuccess) {
        release();
        return LB_ERR_CUDA;
    }
    auto fail = [&]() {
        release();
        s->poisoned = true;
        return LB_ERR_CUDA;
    };
    if (cudaMemcpyAsync(tgt, rho_target, sizeof(double) * N, cudaMemcpyDefault, st) != cudaSuccess ||
        cudaMemsetAsync(acc, 0, sizeof(double) * 8, st) != cudaSuccess ||
        cudaMemsetAsync(cnt, 0, sizeof(unsigned int), st) != cudaSuccess ||
        (word_bytes > 0 && cudaMemsetAsync(scr, 0, word_bytes, st) != cudaSuccess))
        return fail();

    auto save = [&](float* dst, int cur) -> bool {
        return cudaMemcpyAsync(dst, s->g[cur], sizeof(float) * GE, cudaMemcpyDeviceToDevice,
                               st) == cudaSuccess &&
               cudaMemcpyAsync(dst + GE, s->dpsi[cur], sizeof(float) * N,
                               cudaMemcpyDeviceToDevice, st) == cudaSuccess;
    };
    // ---- forward, checkpointing the state (g(t), dpsi(t)) at t = kC. Steps taken
    // together, here and in the recomputation, give the bits of single steps of the
    // register-prefetch kernel, so the recomputed states are those of the trajectory.
    const int pipeline = s->launch.pipeline;
    s->launch.pipeline = 0;
    Fp32Launch L = s->launch;
    lb_status fwd = LB_OK;
    for (long long t = 0; t < T && fwd == LB_OK; t += C) {
        if (!save(ck + slot * (t / C), s->cur)) fwd = LB_ERR_CUDA;
        else fwd = advance_delta(s, (long)(T - t < C ? T - t : C));
    }
    s->launch.pipeline = pipeline;
    if (fwd != LB_OK) return fail();

    AdjArgs A{};
    A.a = state_args<float>(s, s->cur);
    A.aw = with_weights(A.a, false);
    A.ap = with_weights(A.a, true);
    A.G1 = (float)s->p.G1;
    A.G2 = (float)s->p.G2;
    A.inv_sqrt_rho0 = (float)(1.0 / std::sqrt(s->p.rho0));
    A.rho_target = tgt;
    A.partials = part;
    A.counter = cnt;
    // the float4 array first, at the allocation's (256-byte aligned) start, then
    // the float2 array at 16 N bytes (8-byte aligned for any N)
    A.site = reinterpret_cast<float4*>(scr);
    A.Q = reinterpret_cast<float2*>(scr + 4 * (size_t)N);
    float* lamA = lam;
    float* lamB = lam + 9 * (size_t)N;
    // ---- terminal: J and l(T)
    A.g = static_cast<const float*>(s->g[s->cur]);
    A.dpsi = s->dpsi[s->cur];
    A.lam = lamA;
    float4* lam4[2] = {reinterpret_cast<float4*>(lam), reinterpret_cast<float4*>(lam) + N};
    A.lam4 = held ? lam4[0] : nullptr;
    A.acc = acc;             // acc[0..3] = E, misfit, dE/dG1, dE/dG2
    A.narrow = s->flag;
    const AdjArgs terminal = A;
    k_adj_terminal<float, true, false><<<grid, kAdjThreads, 0, st>>>(A, A.g);
    if (cudaGetLastError() != cudaSuccess) return fail();

    // ---- reverse over the segments. Segment k (states kC .. kC + n - 1) is
    // recomputed from its checkpoint into segment buffer k & 1 on the second
    // stream while the reverse sweep of segment k + 1 runs on the caller's
    // stream (both are latency-bound on lattices that fit in L2, so the two
    // overlap); events order the buffer reuse and the hand-over.
    A.acc = acc + 4;         // acc[4], acc[5] = the steps' dJ/dG1, dJ/dG2
    const StepArgs<float> base = state_args<float>(s, 0);
    auto seg_len = [&](long long k) { return (k + 1) * C <= T ? C : T - k * C; };
    auto state_at = [&](long long k, long long j) -> float* {
        return j == 0 ? ck + slot * k : seg + slot * ((size_t)(k & 1) * seg_slots + (j - 1));
    };
    bool used[2] = {false, false};
    auto recompute = [&](long long k) -> bool {
        const int b = (int)(k & 1);
        if (used[b] && cudaStreamWaitEvent(rs, ev_free[b], 0) != cudaSuccess) return false;
        used[b] = true;
        for (long long j = 0; j + 1 < seg_len(k); ++j) {
            StepArgs<float> a = base;
            const float* in = state_at(k, j);
            float* out = state_at(k, j + 1);
            a.g_in = in;
            a.g_out = out;
            a.dpsi_in = in + GE;
            a.dpsi_out = out + GE;
            if (fp32_step(a, L, false, rs) != cudaSuccess) return false;
        }
        return cudaEventRecord(ev_ready[b], rs) == cudaSuccess;
    };
    // held: the segment's dJ/dG terms, summed in the order of the steps
    uint4* words = reinterpret_cast<uint4*>(scr);
    double2* sums = reinterpret_cast<double2*>(reinterpret_cast<char*>(scr) + word_bytes);
    double2* tot = sums + (size_t)grid * (size_t)(rows + 1);
    float* terms = reinterpret_cast<float*>(tot + (rows + 1));
    auto add_terms = [&](int n) -> bool {
        for (int r = 0; r < n; r += 32768) {      // within the grid's limit in y
            const int m = n - r < 32768 ? n - r : 32768;
            k_adj_sums<<<dim3(grid, m), kAdjThreads, 0, st>>>(terms + (size_t)2 * N * r, N, sums);
            if (cudaGetLastError() != cudaSuccess) return false;
            k_adj_sums_total<<<m, kAdjThreads, 0, st>>>(sums, grid, tot, cnt, acc + 4);
            if (cudaGetLastError() != cudaSuccess) return false;
        }
        return true;
    };
    int in4 = 0;             // lam4[in4] holds the adjoint
    if (held) {
        // one stream: the recomputation and the reverse sweep each take the whole GPU.
        // The state's idle buffers receive the recomputation's last state, which nobody reads.
        R.A = A;
        R.words = words;
        R.states = seg;
        R.terms = terms;
        for (long long k = K - 1; k >= 0; --k) {
            const int n = (int)seg_len(k);
            StepArgs<float> a = base;
            const float* in = ck + slot * k;
            a.g_in = in;
            a.dpsi_in = in + GE;
            a.g_out = static_cast<float*>(s->g[s->cur ^ 1]);
            a.dpsi_out = s->dpsi[s->cur ^ 1];
            if (fp32_resident_kept(a, s->res_buf, n, seg, st) != cudaSuccess) return fail();
            R.steps = n;
            R.lam_in = lam4[in4];
            R.lam_out = lam4[in4 ^ 1];
            if (launch_reverse(R, rev_tiles, st) != cudaSuccess || !add_terms(n))
                return fail();
            R.tag += (unsigned)n;
            in4 ^= 1;
        }
    } else {
        if (cudaEventRecord(ev_fwd, st) != cudaSuccess || cudaStreamWaitEvent(rs, ev_fwd, 0) != cudaSuccess)
            return fail();
        if (K > 0 && !recompute(K - 1)) return fail();
        for (long long k = K - 1; k >= 0; --k) {
            const long long n = seg_len(k);
            if (k > 0 && !recompute(k - 1)) return fail();
            if (cudaStreamWaitEvent(st, ev_ready[k & 1], 0) != cudaSuccess) return fail();
            for (long long j = n - 1; j >= 0; --j) {
                const float* state = state_at(k, j);
                A.g = state;
                A.dpsi = state + GE;
                A.lam_next = lamA;
                A.lam = lamB;
                k_adj_pass_a<<<grid, kAdjThreads, 0, st>>>(A);
                k_adj_pass_b<<<grid, kAdjThreads, 0, st>>>(A);
                float* tmp = lamA;
                lamA = lamB;
                lamB = tmp;
                if (cudaGetLastError() != cudaSuccess) return fail();
            }
            if (cudaEventRecord(ev_free[k & 1], st) != cudaSuccess) return fail();
        }
    }
    double* gout = grad_on_dev ? grad_rho : grad_dev;
    k_adj_grad_init<<<grid, kAdjThreads, 0, st>>>(
        lamA, held ? lam4[in4] : nullptr, N, A.a.w0, A.a.w1, A.a.w2, gout);
    if (cudaGetLastError() != cudaSuccess) return fail();
    double h[8];
    int flags = 0, narrow = 0;
    if (cudaMemcpyAsync(h, acc, sizeof(h), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaMemcpyAsync(&flags, s->err, sizeof(int), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaMemcpyAsync(&narrow, s->flag, sizeof(int), cudaMemcpyDeviceToHost, st) != cudaSuccess)
        return fail();
    if (!grad_on_dev &&
        cudaMemcpyAsync(grad_rho, grad_dev, sizeof(double) * N, cudaMemcpyDeviceToHost, st) !=
            cudaSuccess)
        return fail();
    if (cudaStreamSynchronize(st) != cudaSuccess) return fail();
    if (narrow && !(flags & 1)) {
        // J or the explicit derivatives beyond the range of the FP32 pairs
        double w[4];
        if (cudaMemsetAsync(s->flag, 0, sizeof(int), st) != cudaSuccess ||
            cudaMemsetAsync(acc, 0, sizeof(w), st) != cudaSuccess)
            return fail();
        k_adj_terminal<float, true, true><<<grid, kAdjThreads, 0, st>>>(terminal, terminal.g);
        if (cudaGetLastError() != cudaSuccess ||
            cudaMemcpyAsync(w, acc, sizeof(w), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
            cudaStreamSynchronize(st) != cudaSuccess)
            return fail();
        if (narrow & 1) h[0] = w[0];
        if (narrow & 2) {
            h[2] = w[2];
            h[3] = w[3];
        }
    }
    release();
    if (flags & 1) {                                 // a bounded wait ran out
        s->poisoned = true;
        return LB_ERR_TIMEOUT;
    }
    *J_out = h[0] + h[1];
    grad_G[0] = h[2] + h[4];
    grad_G[1] = h[3] + h[5];
    if (!std::isfinite(*J_out) || !std::isfinite(grad_G[0]) || !std::isfinite(grad_G[1]))
        return LB_ERR_NONFINITE;
    return LB_OK;
}

namespace {

__global__ void __launch_bounds__(256) k_misfit64(const double* __restrict__ rho,
                                                  const double* __restrict__ tgt, long long n,
                                                  double* partials, unsigned int* counter,
                                                  double* out)
{
    double v[4] = {0.0, 0.0, 0.0, 0.0};
    for (long long s = blockIdx.x * 256LL + threadIdx.x; s < n; s += (long long)gridDim.x * 256) {
        const double m = rho[s] - tgt[s];
        v[0] += m * m;
    }
    if (last_block_total<256>(v, partials, counter, gridDim.x)) *out = v[0];
}

}  // namespace

namespace lbsc {

cudaError_t objective_delta(const lb_state* s, const double* tgt, double* acc, bool wide,
                            cudaStream_t st)
{
    AdjArgs A{};
    A.a = state_args<float>(s, s->cur);
    A.aw = with_weights(A.a, false);
    A.ap = with_weights(A.a, true);
    A.G1 = (float)s->p.G1;
    A.G2 = (float)s->p.G2;
    A.inv_sqrt_rho0 = (float)(1.0 / std::sqrt(s->p.rho0));
    A.dpsi = s->dpsi[s->cur];
    A.rho_target = tgt;
    A.partials = s->partials;
    A.counter = s->counter;
    A.acc = acc;
    A.narrow = s->flag;
    cudaError_t e = cudaMemsetAsync(acc, 0, 4 * sizeof(double), st);
    if (e != cudaSuccess) return e;
    const int grid = adj_grid(s->N);
    auto go = [&](auto kern, auto* g) { kern<<<grid, kAdjThreads, 0, st>>>(A, g); };
    const auto *f = static_cast<const float*>(s->g[s->cur]);
    const auto *h = static_cast<const __half*>(s->g[s->cur]);
    if (s->p.prec == LB_FP16_DELTA)
        wide ? go(k_adj_terminal<__half, false, true>, h) : go(k_adj_terminal<__half, false, false>, h);
    else
        wide ? go(k_adj_terminal<float, false, true>, f) : go(k_adj_terminal<float, false, false>, f);
    return cudaGetLastError();
}

cudaError_t misfit64(const double* rho, const double* tgt, long long n, double* partials,
                     unsigned int* counter, double* out, cudaStream_t st)
{
    long long b = (n + 255) / 256;
    if (b > 152 * 16) b = 152 * 16;
    k_misfit64<<<(int)(b < 1 ? 1 : b), 256, 0, st>>>(rho, tgt, n, partials, counter, out);
    return cudaGetLastError();
}

}  // namespace lbsc
