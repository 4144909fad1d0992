// Differentiable unrolled PnP-ADMM (relaxed DMD masks, Huber-smoothed TV with
// the z-smoothness Gauss-Seidel sweep) and its hand-written reverse pass.
//
// Forward, K iterations of Algorithm 1 on a batch of B volumes [Z][H][W]
// (one shot, R = Z), from u = d = 0:
//   m     = sigmoid(logits)                             relaxed DMD patterns
//   x-update (Eq. v-update, Woodbury with D = sum_r m_r^2):
//         g = u - d,  e = (b - sum_r m_r g_r) / (rho + D),  v_r = g_r + m_r e,
//         w = v + d
//   u-step, n = 0..Z-1 in order (Eq. u-update, newest neighbours, cyclic):
//         h_n = (rho w_n + gamma (u_{n-1} + u_{n+1})) / (rho + 2 gamma)
//         u_n = prox of theta * HuberTV_eps at h_n, theta = lambda/(rho+2gamma),
//               by T steps of projected gradient on its dual from p = 0:
//               q = div p - h/theta,  a = p + tau (grad q - kappa p),
//               p <- a / max(1, |a|),  kappa = eps / theta,
//               u_n = h - theta div p
//   d = w - u.
// The Huber function |x| - eps/2 (|x| > eps), |x|^2/(2 eps) (|x| <= eps) has the
// conjugate eps/2 |p|^2 on |p| <= 1, which is the -kappa p damping above.
// grad: forward differences, zero on the last row / column; div = -grad^T.
//
// Reverse.  The caller gives vbar = dL/dv^K.  The state (u^k, d^k) is stored
// every `ckpt_every` iterations by the forward; the reverse walks the
// segments backwards, recomputes each segment's states from its checkpoint,
// and backpropagates one iteration at a time: the dual update, the
// Gauss-Seidel sweep in reverse slice order (each prox recomputes its T dual
// iterates and runs their adjoint), the x-update.  Gradients: dL/dlogits and
// the three scalars dL/drho, dL/dlambda, dL/dgamma (FP64 accumulators).
//
// The x-update kernels are one-thread-per-pixel passes (a block row of the grid
// per batch item); the u-step runs several dual steps per launch on chip (below).
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <utility>
#include <vector>

#include "internal.cuh"
#include "inv_norm.cuh"
#include "tv_body.cuh"

namespace cslsm {
namespace {

constexpr int kT = 256;
// The three scalar gradients are accumulated in kAccCopies FP64 copies each
// (one atomic per block into copy blockIdx % kAccCopies), summed at the end:
// one address per scalar would serialise tens of thousands of atomics a launch.
constexpr int kAccCopies = 64;

// A sum kept as an unevaluated pair of FP32 numbers (Knuth's two-sum): about 48
// bits, at FP32 rates.  An FP64 addition occupies an SM for 16 cycles a warp
// here, so FP64 block sums took as long as the reverse steps they followed.
struct Pair32 {
    float hi, lo;
    __device__ __forceinline__ void add(float h, float l)
    {
        const float s = hi + h, v = s - hi;
        lo += ((hi - (s - v)) + (h - v)) + l;
        hi = s;
    }
    // adds (h + l) x f, f = (f.x + f.y), products of the leading parts exact
    __device__ __forceinline__ void add_scaled(float h, float l, float2 f)
    {
        const float p = h * f.x;
        add(p, fmaf(h, f.x, -p) + fmaf(l, f.x, h * f.y));
    }
};

// Two such sums side by side, of a lane's two columns.
struct Pairs32 {
    float2 hi, lo;
    __device__ __forceinline__ void add(float2 h, float2 l)
    {
        const float2 s = add2(hi, h), v = sub2(s, hi);
        lo = add2(lo, add2(add2(sub2(hi, sub2(s, v)), sub2(h, v)), l));
        hi = s;
    }
    __device__ __forceinline__ void add(float2 h)
    {
        const float2 s = add2(hi, h), v = sub2(s, hi);
        lo = add2(lo, add2(sub2(hi, sub2(s, v)), sub2(h, v)));
        hi = s;
    }
    __device__ __forceinline__ Pair32 total() const
    {
        Pair32 t = {hi.x, lo.x};
        t.add(hi.y, lo.y);
        return t;
    }
};

// Adds the block's sums of v[0 .. N) to acc[idx[.]][blockIdx.x % kAccCopies].
// Every thread of the block must call it.
template <int N>
__device__ __forceinline__ void block_acc(Pair32 (&v)[N], double *acc, const int (&idx)[N])
{
    __shared__ Pair32 s_part[N][32];
#pragma unroll
    for (int q = 0; q < N; ++q) {
        for (int off = 16; off > 0; off >>= 1)
            v[q].add(__shfl_down_sync(0xffffffffu, v[q].hi, off),
                     __shfl_down_sync(0xffffffffu, v[q].lo, off));
        if ((threadIdx.x & 31) == 0) s_part[q][threadIdx.x >> 5] = v[q];
    }
    __syncthreads();
    if (threadIdx.x < N) {
        Pair32 t = s_part[threadIdx.x][0];
        for (int w = 1; w < (int)(blockDim.x >> 5); ++w)
            t.add(s_part[threadIdx.x][w].hi, s_part[threadIdx.x][w].lo);
        // an infinite sum has no second part
        atomicAdd(acc + idx[threadIdx.x] * kAccCopies + blockIdx.x % kAccCopies,
                  isfinite(t.hi) ? (double)t.hi + (double)t.lo : (double)t.hi);
    }
}

struct Geo {
    int B, Z, H, W;
    __host__ __device__ size_t HW() const { return (size_t)H * W; }
    __host__ __device__ size_t NV() const { return (size_t)Z * H * W; }  // per batch item
};

__device__ __forceinline__ float sigm(float x) { return 1.f / (1.f + expf(-x)); }

// ---- x-update ----------------------------------------------------------------
__global__ void ux_fwd_kernel(const float *__restrict__ U, const float *__restrict__ Dl,
                              const float *__restrict__ logits, const float *__restrict__ b,
                              Geo g, float rho, float *__restrict__ Wb, float *__restrict__ vout)
{
    const size_t p = blockIdx.x * (size_t)kT + threadIdx.x;
    const int bi = blockIdx.y;
    if (p >= g.HW()) return;
    const size_t base = bi * g.NV() + p, HW = g.HW();
    float s = 0.f, D = 0.f;
    for (int r = 0; r < g.Z; ++r) {
        const size_t o = base + r * HW;
        const float m = sigm(logits[o]);
        s += m * (U[o] - Dl[o]);
        D += m * m;
    }
    const float e = (b[bi * HW + p] - s) / (rho + D);
    for (int r = 0; r < g.Z; ++r) {
        const size_t o = base + r * HW;
        const float m = sigm(logits[o]);
        const float v = (U[o] - Dl[o]) + m * e;
        Wb[o] = v + Dl[o];
        if (vout) vout[o] = v;
    }
}

// Reverse of ux_fwd: given vbar (may be null) and wbar = dL/dw, accumulates
// dL/du^k into Uold_bar, writes dL/dd^k into Dbar, adds dL/dlogits into
// lbar, and dL/drho (direct) into acc[0].
__global__ void ux_bwd_kernel(const float *__restrict__ U, const float *__restrict__ Dl,
                              const float *__restrict__ logits, const float *__restrict__ b,
                              Geo g, float rho, const float *__restrict__ vbar,
                              const float *__restrict__ Wbar, float *__restrict__ Uold_bar,
                              float *__restrict__ Dbar, float *__restrict__ lbar,
                              double *__restrict__ acc)
{
    const size_t p = blockIdx.x * (size_t)kT + threadIdx.x;
    const int bi = blockIdx.y;
    Pair32 rho_bar[1] = {};
    if (p < g.HW()) {
        const size_t base = bi * g.NV() + p, HW = g.HW();
        float s = 0.f, D = 0.f, ebar = 0.f;
        for (int r = 0; r < g.Z; ++r) {
            const size_t o = base + r * HW;
            const float m = sigm(logits[o]);
            s += m * (U[o] - Dl[o]);
            D += m * m;
            const float vb = Wbar[o] + (vbar ? vbar[o] : 0.f);  // v feeds w = v + d and v^K
            ebar += m * vb;
        }
        const float den = rho + D;
        const float e = (b[bi * HW + p] - s) / den;
        const float sbar = -ebar / den;
        const float Dbarv = -ebar * e / den;
        rho_bar[0].hi = -ebar * e / den;
        for (int r = 0; r < g.Z; ++r) {
            const size_t o = base + r * HW;
            const float m = sigm(logits[o]);
            const float gr = U[o] - Dl[o];
            const float vb = Wbar[o] + (vbar ? vbar[o] : 0.f);
            const float gbar = vb + sbar * m;
            const float mbar = e * vb + sbar * gr + 2.f * m * Dbarv;
            Uold_bar[o] += gbar;
            Dbar[o] = Wbar[o] - gbar;
            lbar[o] += mbar * m * (1.f - m);
        }
    }
    const int idx[1] = {0};
    block_acc(rho_bar, acc, idx);
}

// ---- u-step: the Huber-TV prox of one slice of every batch item ----------------
// k dual steps per launch.  A CTA owns a TH x TW tile of one item's slice and
// works on a region of NW RPW + 2 rows x 64 columns around it (halo of k + 1
// rows, an even column halo): a warp holds RPW rows in registers, a lane two
// adjacent columns, and only the warps' boundary rows go through shared memory,
// one barrier a step.  Rows and columns of the halo go stale by one a step;
// warps whose rows no later step needs skip.  One launch per dual step, h and u
// apart, was bound by its 23 launches a slice (3.9 us each at 256 x 256) and at 8 x
// 512 x 512 by its passes over memory; now the forward is bound by issue (67 % of
// the slots, 43 us for 7 steps of 8 x 512 x 512), the reverse too (73 %, 86 us for
// 5), and one small slice by the latency of a step and of a launch.  Forward +
// backward, 10 iterations: 16 x 256 x 256 75.8 -> 17.8 ms; 8 x 16 x 512 x 512 with
// the duals kept 242.5 -> 117.7 ms.
//
//   forward  first phase: h = (rho w_n + gamma (u_{n-1} + u_{n+1})) / (rho + 2
//            gamma) on the region (kept for the later phases and the reverse
//            pass), p = 0; each step q = div p - h / theta, a = p + tau (grad q -
//            kappa p), p = a / max(1, |a|); last phase: u_n = h - theta div p,
//            d_n = w_n - u_n.  With `rec` the a of every step is recorded (in place
//            of the dual iterates, which a / max(1, |a|) gives back exactly).
//   reverse  p^{t+1} = proj(a) with a recorded, so the Jacobian of the projection
//            is local: abar = J(a)^T pbar^{t+1}, J = (I - a a^T / |a|^2) / |a|
//            where |a| > 1; then qbar = -tau div abar and pbar^t = (1 - tau
//            kappa) abar - grad qbar, the forward step's stencil once more.
//            hbar = ubar - sum_t qbar / theta.  First phase: pbar^T = theta grad
//            ubar; last phase: hbar to w_n, the neighbour slices and the scalars.
//
// The masks (0 on the last row / column and outside the image) keep p1 = 0 on
// the last row and p2 = 0 on the last column, so div needs no boundary cases.
struct HuberArgs {
    const float *Wn, *A, *C;  // w_n and the neighbour slices, items N_V floats apart
    float *Hb;                // [B][H][W] h
    const float *Pin;         // [B][2][H][W] p (forward) / pbar (reverse) of the last
    float *Pout;              //   phase or null; p / pbar for the next phase or null
    float *rec;               // a of step t: rec + t [B][2][H][W], or null (forward)
    float *Un, *Dn;           // forward, last phase: u_n and d_n (Un null: not wanted)
    const float *Ubar;        // reverse: dL/du_n, items N_V floats apart
    float *Hbar;              // reverse: [B][H][W]
    float *Wbar, *Abar, *Cbar;  // reverse, last phase (Abar may be Cbar: Z = 2)
    double *acc;
    Geo g;
    float rho, gam, theta, inv_theta, tau, kappa;
    float2 it2, kfac;  // 1 / theta^2 and tau eps / theta^2, each in two parts
    int t0, ns;  // steps t0 .. t0 + ns - 1 (reverse: downwards)
    int T;
    int hh, hc, TH, TW, tx;
    int pair;  // W even and the buffers 8-byte aligned: a lane's columns in one access
};

__device__ __forceinline__ float2 ld_pair(const float *p, int off, bool in0, bool in1, int pair)
{
    if (pair) return in0 ? *reinterpret_cast<const float2 *>(p + off) : make_float2(0.f, 0.f);
    return make_float2(in0 ? p[off] : 0.f, in1 ? p[off + 1] : 0.f);
}

__device__ __forceinline__ void st_pair(float *p, int off, float2 v, bool in0, bool in1, int pair)
{
    if (pair) {
        if (in0) *reinterpret_cast<float2 *>(p + off) = v;
    } else {
        if (in0) p[off] = v.x;
        if (in1) p[off + 1] = v.y;
    }
}

// The lane's place in the region (the same for both directions).
template <int NW, int RPW>
struct HuberTile {
    int lane, wp, gi0, gc, r0, j0;
    bool in0, in1, own0, own1, interior;
    bool mc0, mc1;           // the columns have a column to their right in the image
    unsigned inr, ownr, mr;  // bit i: row i in the image / owned / has a row below it
    __device__ __forceinline__ HuberTile(const HuberArgs &a)
    {
        constexpr int RH = NW * RPW + 2;
        const int H = a.g.H, W = a.g.W;
        const int bx = (int)blockIdx.x % a.tx, by = (int)blockIdx.x / a.tx;
        lane = (int)(threadIdx.x & 31);
        wp = (int)(threadIdx.x >> 5);
        gi0 = by * a.TH - a.hh;
        const int gj0 = bx * a.TW - a.hc;
        j0 = 2 * lane;
        gc = gj0 + j0;
        r0 = 1 + wp * RPW;
        in0 = gc >= 0 && gc < W;
        in1 = gc + 1 >= 0 && gc + 1 < W;
        own0 = in0 && j0 >= a.hc && j0 < a.hc + a.TW;
        own1 = in1 && j0 + 1 >= a.hc && j0 + 1 < a.hc + a.TW;
        mc0 = in0 && gc < W - 1;
        mc1 = in1 && gc + 1 < W - 1;
        interior = gi0 >= 0 && gi0 + RH < H && gj0 >= 0 && gj0 + 64 < W;
        inr = ownr = mr = 0;
#pragma unroll
        for (int i = 0; i <= RPW; ++i) {
            const int gi = gi0 + r0 + i;
            if (gi >= 0 && gi < H) inr |= 1u << i;
            if (gi >= 0 && gi < H - 1) mr |= 1u << i;
            if (i < RPW && gi >= 0 && gi < H && r0 + i >= a.hh && r0 + i < a.hh + a.TH)
                ownr |= 1u << i;
        }
    }
    __device__ __forceinline__ int off(int i, int W) const { return (gi0 + r0 + i) * W + gc; }
    __device__ __forceinline__ bool row_in(int i) const { return (inr >> i) & 1u; }
    __device__ __forceinline__ bool row_own(int i) const { return (ownr >> i) & 1u; }
    // zero a row component without a row below, a column component without a column to the right
    __device__ __forceinline__ void mask(int i, float2 &x, float2 &y) const
    {
        if (!((mr >> i) & 1u)) x = make_float2(0.f, 0.f);
        y.x = mc0 ? y.x : 0.f;
        y.y = mc1 ? y.y : 0.f;
    }
};

// Programmatic dependent launch: lets the next launch's blocks start (they wait
// here too), then waits until the launch before has completed and its writes
// are visible.  Every thread calls it before its first access to memory.
__device__ __forceinline__ void pdl_enter()
{
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

// 1 / max(1, |a|) of a lane's two columns.
__device__ __forceinline__ float2 huber_scale(float2 a1, float2 a2)
{
    return inv_norm2(fma2(a1, a1, mul2(a2, a2)));
}

template <bool INTERIOR, int NW, int RPW>
__device__ __forceinline__ void huber_steps(const HuberArgs &a, const HuberTile<NW, RPW> &t,
                                            Bnd<NW> &sb, float2 (&p1)[RPW], float2 (&p2)[RPW],
                                            const float2 (&h)[RPW + 1], float *rec)
{
    constexpr unsigned FULL = 0xffffffffu;
    const size_t step = (size_t)a.g.B * 2 * a.g.HW();
    const int HW = (int)a.g.HW();
    const int lo = a.hh - (a.Pout ? 0 : 1), hi = a.hh + a.TH;
    for (int st = 0; st < a.ns; ++st) {
        const int par = st & 1, nxt = par ^ 1;
        const int e = a.ns - 1 - st;
        if (t.r0 + RPW > lo - e && t.r0 < hi + e) {
            const float2 pu0 = sb.up[par][t.wp][t.lane];
            const float2 dn1 = sb.dn1[par][t.wp][t.lane], dn2 = sb.dn2[par][t.wp][t.lane];
            float2 qc = q_pair(p1[0], pu0, p2[0], __shfl_up_sync(FULL, p2[0].y, 1), h[0],
                               a.inv_theta);
#pragma unroll
            for (int i = 0; i < RPW; ++i) {
                const float2 qn =
                    i + 1 < RPW
                        ? q_pair(p1[i + 1 < RPW ? i + 1 : 0], p1[i], p2[i + 1 < RPW ? i + 1 : 0],
                                 __shfl_up_sync(FULL, p2[i + 1 < RPW ? i + 1 : 0].y, 1), h[i + 1],
                                 a.inv_theta)
                        : q_pair(dn1, p1[RPW - 1], dn2, __shfl_up_sync(FULL, dn2.y, 1), h[RPW],
                                 a.inv_theta);
                const float qr = __shfl_down_sync(FULL, qc.x, 1);
                float2 gx = sub2(qn, qc), gy = make_float2(qc.y - qc.x, qr - qc.y);
                if (!INTERIOR) t.mask(i, gx, gy);
                const float2 a1 = fma2(splat(a.tau), fma2(splat(-a.kappa), p1[i], gx), p1[i]);
                const float2 a2 = fma2(splat(a.tau), fma2(splat(-a.kappa), p2[i], gy), p2[i]);
                if (rec && t.row_own(i)) {
                    float *r = rec + st * step;
                    const int o = t.off(i, a.g.W);
                    st_pair(r, o, a1, t.own0, t.own1, a.pair);
                    st_pair(r + HW, o, a2, t.own0, t.own1, a.pair);
                }
                const float2 sc = huber_scale(a1, a2);
                p1[i] = mul2(a1, sc);
                p2[i] = mul2(a2, sc);
                qc = qn;
            }
            if (t.wp + 1 < NW) sb.up[nxt][t.wp + 1][t.lane] = p1[RPW - 1];
            if (t.wp > 0) {
                sb.dn1[nxt][t.wp - 1][t.lane] = p1[0];
                sb.dn2[nxt][t.wp - 1][t.lane] = p2[0];
            }
        }
        __syncthreads();
    }
}

template <int NW, int RPW>
__global__ void __launch_bounds__(NW * 32, 2) huber_fwd_kernel(const HuberArgs a)
{
    constexpr unsigned FULL = 0xffffffffu;
    constexpr int RH = NW * RPW + 2;
    __shared__ Bnd<NW> sb;
    const HuberTile<NW, RPW> t(a);
    pdl_enter();
    const int W = a.g.W, bi = blockIdx.y, lane = t.lane, wp = t.wp;
    const size_t HW = a.g.HW();
    const float *Wn = a.Wn + bi * a.g.NV(), *A = a.A + bi * a.g.NV(), *C = a.C + bi * a.g.NV();
    float *Hb = a.Hb + bi * HW;
    float2 p1[RPW], p2[RPW], h[RPW + 1];
    float2 f1 = make_float2(0.f, 0.f), f2 = f1;
    if (a.Pin) {
        const float *P1 = a.Pin + (size_t)bi * 2 * HW, *P2 = P1 + HW;
#pragma unroll
        for (int i = 0; i <= RPW; ++i) {
            const bool i0 = t.row_in(i) && t.in0, i1 = t.row_in(i) && t.in1;
            h[i] = ld_pair(Hb, t.off(i, W), i0, i1, a.pair);
            if (i < RPW) {
                p1[i < RPW ? i : 0] = ld_pair(P1, t.off(i, W), i0, i1, a.pair);
                p2[i < RPW ? i : 0] = ld_pair(P2, t.off(i, W), i0, i1, a.pair);
            }
        }
        if (wp == 0 || wp == NW - 1) {  // frozen rows 0 and RH - 1 of the region
            const int gi = t.gi0 + (wp == 0 ? 0 : RH - 1);
            if (gi >= 0 && gi < a.g.H) {
                f1 = ld_pair(P1, gi * W + t.gc, t.in0, t.in1, a.pair);
                f2 = ld_pair(P2, gi * W + t.gc, t.in0, t.in1, a.pair);
            }
        }
    } else {
        const float rho = a.rho, gam = a.gam, den = a.rho + 2.f * a.gam;
#pragma unroll
        for (int i = 0; i <= RPW; ++i) {
            const bool i0 = t.row_in(i) && t.in0, i1 = t.row_in(i) && t.in1;
            const int o = t.off(i, W);
            const float2 w = ld_pair(Wn, o, i0, i1, a.pair);
            float2 s = make_float2(0.f, 0.f);
            if (gam > 0.f) s = add2(ld_pair(A, o, i0, i1, a.pair), ld_pair(C, o, i0, i1, a.pair));
            // the roundings of the numerator are written out: the iterates reach the
            // kink of the projection, where a changed bit can flip a gradient's branch
            h[i].x = __fmaf_rn(gam, s.x, __fmul_rn(rho, w.x)) / den;
            h[i].y = __fmaf_rn(gam, s.y, __fmul_rn(rho, w.y)) / den;
            if (i < RPW && t.row_own(i)) st_pair(Hb, o, h[i], t.own0, t.own1, a.pair);
        }
#pragma unroll
        for (int i = 0; i < RPW; ++i) p1[i] = p2[i] = make_float2(0.f, 0.f);
    }
    if (wp == 0) sb.up[0][0][lane] = sb.up[1][0][lane] = f1;
    if (wp == NW - 1) {
        sb.dn1[0][NW - 1][lane] = sb.dn1[1][NW - 1][lane] = f1;
        sb.dn2[0][NW - 1][lane] = sb.dn2[1][NW - 1][lane] = f2;
    }
    if (wp + 1 < NW) sb.up[0][wp + 1][lane] = p1[RPW - 1];
    if (wp > 0) {
        sb.dn1[0][wp - 1][lane] = p1[0];
        sb.dn2[0][wp - 1][lane] = p2[0];
    }
    __syncthreads();
    float *rec = a.rec ? a.rec + (size_t)bi * 2 * HW : nullptr;
    if (t.interior) huber_steps<true, NW, RPW>(a, t, sb, p1, p2, h, rec);
    else huber_steps<false, NW, RPW>(a, t, sb, p1, p2, h, rec);
    if (a.Pout) {
        float *Q1 = a.Pout + (size_t)bi * 2 * HW, *Q2 = Q1 + HW;
#pragma unroll
        for (int i = 0; i < RPW; ++i)
            if (t.row_own(i)) {
                st_pair(Q1, t.off(i, W), p1[i], t.own0, t.own1, a.pair);
                st_pair(Q2, t.off(i, W), p2[i], t.own0, t.own1, a.pair);
            }
    } else if (a.Un) {
        float *Un = a.Un + bi * a.g.NV(), *Dn = a.Dn + bi * a.g.NV();
        const float2 pu0 = sb.up[a.ns & 1][wp][lane];
#pragma unroll
        for (int i = 0; i < RPW; ++i) {
            const float p2l = __shfl_up_sync(FULL, p2[i].y, 1);
            const float2 dv = add2(sub2(p1[i], i == 0 ? pu0 : p1[i > 0 ? i - 1 : 0]),
                                   sub2(p2[i], make_float2(p2l, p2[i].x)));
            if (!t.row_own(i)) continue;
            const int o = t.off(i, W);
            const float2 u = fma2(splat(-a.theta), dv, h[i]);
            st_pair(Un, o, u, t.own0, t.own1, a.pair);
            st_pair(Dn, o, sub2(ld_pair(Wn, o, t.own0, t.own1, a.pair), u), t.own0, t.own1, a.pair);
        }
    }
}

// The recorded a of the lane's rows, fetched kRing - 1 steps ahead into shared
// memory by asynchronous copies.  Every thread reads back only what it copied
// itself, so a wait on its own copies is all the ordering needed, and the
// fetches cost no registers.
constexpr int kRing = 4;

template <int NW, int RPW>
struct HuberRing {
    static constexpr int kSlot = 2 * RPW * NW * 32;  // float2 per step
    static constexpr size_t bytes() { return sizeof(float2) * kRing * kSlot; }
    float2 *buf;           // the thread's column of the ring
    const float *src[RPW];  // the row in the a of the step to fetch next
    size_t step;           // floats between steps
    int hw, pair;
    unsigned in0, in1;     // bit i: the row's columns are in the image

    __device__ __forceinline__ HuberRing(const HuberArgs &a, const HuberTile<NW, RPW> &t,
                                         const float *rec, int first, float2 *mem)
        : buf(mem + threadIdx.x), step((size_t)a.g.B * 2 * a.g.HW()), hw((int)a.g.HW()),
          pair(a.pair), in0(t.in0 ? t.inr : 0u), in1(t.in1 ? t.inr : 0u)
    {
#pragma unroll
        for (int i = 0; i < RPW; ++i)  // outside the image any valid address (nothing is read)
            src[i] = rec + (size_t)max(first, 0) * step + ((in0 >> i) & 1u ? t.off(i, a.g.W) : 0);
    }
    // Fetches the rows of the next step (going down) as one group of copies into
    // slot `slot`; an empty group when there is none.
    __device__ __forceinline__ void fetch(int slot, bool any)
    {
        if (any) {
            const unsigned d = (unsigned)__cvta_generic_to_shared(buf + slot * kSlot);
#pragma unroll
            for (int i = 0; i < RPW; ++i) {
#pragma unroll
                for (int c = 0; c < 2; ++c) {
                    const unsigned dst = d + (unsigned)((c * RPW + i) * NW * 32 * sizeof(float2));
                    const float *q = src[i] + (c ? hw : 0);
                    if (pair) {
                        asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(dst),
                                     "l"(q), "r"(((in0 >> i) & 1u) * 8)
                                     : "memory");
                    } else {
                        // gc is even, so a second column in the image has the first there too
                        const unsigned x = (in0 >> i) & 1u, y = (in1 >> i) & 1u;
                        asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst),
                                     "l"(q), "r"(x * 4)
                                     : "memory");
                        asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst + 4),
                                     "l"(q + (x & y)), "r"(y * 4)
                                     : "memory");
                    }
                }
                src[i] -= step;
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    }
    // all but the newest kRing - 2 groups of this thread have arrived
    __device__ __forceinline__ void wait() const
    {
        asm volatile("cp.async.wait_group %0;" ::"n"(kRing - 2) : "memory");
    }
    __device__ __forceinline__ float2 get(int slot, int c, int i) const
    {
        return buf[slot * kSlot + (c * RPW + i) * NW * 32];
    }
};

// Reverse of steps t0 + ns - 1 .. t0 on the region.  Needs a of t0 - 1 too (the
// theta partial takes p^{t0}).  Step st's a is group st of the ring.
template <bool INTERIOR, int NW, int RPW>
__device__ __forceinline__ void huber_reverse(const HuberArgs &a, const HuberTile<NW, RPW> &t,
                                              Bnd<NW> &sb, HuberRing<NW, RPW> &ring, int groups,
                                              float2 (&b1)[RPW], float2 (&b2)[RPW],
                                              float2 (&sq)[RPW], float &tk, float &tk_err)
{
    constexpr unsigned FULL = 0xffffffffu;
    const float damp = 1.f - a.tau * a.kappa;
    const int lo = a.hh, hi = a.hh + a.TH;
    float2 a1[RPW], a2[RPW], inv[RPW];  // a of the step, 1 / max(1, |a|)
    ring.wait();
#pragma unroll
    for (int i = 0; i < RPW; ++i) {
        a1[i] = ring.get(0, 0, i);
        a2[i] = ring.get(0, 1, i);
        inv[i] = huber_scale(a1[i], a2[i]);
    }
    int e = a.ns - 1;
    for (int st = 0; st < a.ns; ++st, --e) {
        const int par = st & 1;
        const bool live = t.r0 + RPW > lo - e - 1 && t.r0 < hi + e + 1;
        if (live) {
#pragma unroll
            for (int i = 0; i < RPW; ++i) {
                const float2 dot =
                    mul2(fma2(a1[i], b1[i], mul2(a2[i], b2[i])), mul2(inv[i], inv[i]));
                const float2 nd = mul2(dot, splat(-1.f));
                const float2 o1 = mul2(fma2(a1[i], nd, b1[i]), inv[i]);
                const float2 o2 = mul2(fma2(a2[i], nd, b2[i]), inv[i]);
                // |a| <= 1 (inv = 1): the projection is the identity
                b1[i].x = inv[i].x < 1.f ? o1.x : b1[i].x;
                b1[i].y = inv[i].y < 1.f ? o1.y : b1[i].y;
                b2[i].x = inv[i].x < 1.f ? o2.x : b2[i].x;
                b2[i].y = inv[i].y < 1.f ? o2.y : b2[i].y;
                if (!INTERIOR) t.mask(i, b1[i], b2[i]);
            }
            if (t.wp + 1 < NW) sb.up[par][t.wp + 1][t.lane] = b1[RPW - 1];
            if (t.wp > 0) {
                sb.dn1[par][t.wp - 1][t.lane] = b1[0];
                sb.dn2[par][t.wp - 1][t.lane] = b2[0];
            }
        }
        __syncthreads();
        if (live) {
            // group st + 3 into the slot that group st - 1 has left
            ring.fetch((st + kRing - 1) % kRing, st + kRing - 1 < groups);
            ring.wait();  // group st + 1
            const float2 pu0 = sb.up[par][t.wp][t.lane];
            const float2 dn1 = sb.dn1[par][t.wp][t.lane], dn2 = sb.dn2[par][t.wp][t.lane];
            // p^t = n / max(1, |n|), n the a of the step before: the theta partial
            // <abar, p^t> of the own tile
            float2 part = make_float2(0.f, 0.f);
            const bool more = st + 1 < groups;
#pragma unroll
            for (int i = 0; i < RPW; ++i) {
                a1[i] = a2[i] = make_float2(0.f, 0.f);
                if (more) {
                    a1[i] = ring.get((st + 1) % kRing, 0, i);
                    a2[i] = ring.get((st + 1) % kRing, 1, i);
                }
                inv[i] = huber_scale(a1[i], a2[i]);
                const float2 w = mul2(fma2(b1[i], a1[i], mul2(b2[i], a2[i])), inv[i]);
                if (t.row_own(i)) part = add2(part, w);
            }
            const float p = (t.own0 ? part.x : 0.f) + (t.own1 ? part.y : 0.f);
            const float s = tk + p, v = s - tk;  // two-sum
            tk_err += (tk - (s - v)) + (p - v);
            tk = s;
            auto q_of = [&](float2 x1, float2 up, float2 x2) {
                const float l = __shfl_up_sync(FULL, x2.y, 1);
                return mul2(splat(-a.tau),
                            add2(sub2(x1, up), make_float2(x2.x - l, x2.y - x2.x)));
            };
            float2 qc = q_of(b1[0], pu0, b2[0]);
#pragma unroll
            for (int i = 0; i < RPW; ++i) {
                const float2 qn = i + 1 < RPW ? q_of(b1[i + 1 < RPW ? i + 1 : 0], b1[i],
                                                     b2[i + 1 < RPW ? i + 1 : 0])
                                              : q_of(dn1, b1[RPW - 1], dn2);
                const float qr = __shfl_down_sync(FULL, qc.x, 1);
                float2 gx = sub2(qc, qn), gy = make_float2(qc.x - qc.y, qc.y - qr);  // -grad
                if (!INTERIOR) t.mask(i, gx, gy);
                sq[i] = add2(sq[i], qc);
                b1[i] = fma2(splat(damp), b1[i], gx);
                b2[i] = fma2(splat(damp), b2[i], gy);
                qc = qn;
            }
        }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");  // of warps that stopped early
}

template <int NW, int RPW>
__global__ void __launch_bounds__(NW * 32, RPW == 2 ? 2 : 1) huber_bwd_kernel(const HuberArgs a)
{
    constexpr unsigned FULL = 0xffffffffu;
    __shared__ Bnd<NW> sb;
    const HuberTile<NW, RPW> t(a);
    pdl_enter();
    const int W = a.g.W, H = a.g.H, bi = blockIdx.y, lane = t.lane, wp = t.wp;
    const size_t HW = a.g.HW();
    const float *rec = a.rec + (size_t)bi * 2 * HW;
    extern __shared__ float2 s_ring[];
    // a of steps t0 + ns - 1 down to t0 - 1 (none before step 0)
    const int groups = a.ns + (a.t0 > 0);
    HuberRing<NW, RPW> ring(a, t, rec, a.t0 + a.ns - 1, s_ring);
    for (int q = 0; q < kRing - 1; ++q) ring.fetch(q, q < groups);
    float *Hb = a.Hb + bi * HW, *Hbar = a.Hbar + bi * HW;
    float2 b1[RPW], b2[RPW], sq[RPW], hb[RPW];
    __shared__ Pair32 s_first[NW * 32];  // the thread's -<ubar, div p^T>, over the steps
    Pair32 sum[3] = {};  // theta, and in the last phase rho, gamma
    if (a.Pin) {
        const float *P1 = a.Pin + (size_t)bi * 2 * HW, *P2 = P1 + HW;
#pragma unroll
        for (int i = 0; i < RPW; ++i) {
            const bool i0 = t.row_in(i) && t.in0, i1 = t.row_in(i) && t.in1;
            b1[i] = ld_pair(P1, t.off(i, W), i0, i1, a.pair);
            b2[i] = ld_pair(P2, t.off(i, W), i0, i1, a.pair);
        }
    } else {
        // pbar^T = theta grad ubar; hbar = ubar; -<ubar, div p^T>
        const float *ub = a.Ubar + bi * a.g.NV();
        const float *r = rec + (size_t)max(a.T - 1, 0) * a.g.B * 2 * HW;
        auto proj = [&](int gi, float2 &x1, float2 &x2) {  // p^T of a row (p^0 = 0)
            const bool in = a.T > 0 && gi >= 0 && gi < H;
            const bool i0 = in && t.in0, i1 = in && t.in1;
            x1 = ld_pair(r, gi * W + t.gc, i0, i1, a.pair);
            x2 = ld_pair(r + HW, gi * W + t.gc, i0, i1, a.pair);
            const float2 sc = huber_scale(x1, x2);
            x1 = mul2(x1, sc);
            x2 = mul2(x2, sc);
        };
        float2 u[RPW + 1], up1, up2;
#pragma unroll
        for (int i = 0; i <= RPW; ++i)
            u[i] = ld_pair(ub, t.off(i, W), t.row_in(i) && t.in0, t.row_in(i) && t.in1, a.pair);
        proj(t.gi0 + t.r0 - 1, up1, up2);
        Pairs32 part = {};
#pragma unroll
        for (int i = 0; i < RPW; ++i) {
            float2 x1, x2;
            proj(t.gi0 + t.r0 + i, x1, x2);
            const float l = __shfl_up_sync(FULL, x2.y, 1);
            const float2 dv = add2(sub2(x1, up1), sub2(x2, make_float2(l, x2.x)));
            up1 = x1;
            if (t.row_own(i))
                part.add(make_float2(t.own0 ? -u[i].x * dv.x : 0.f, t.own1 ? -u[i].y * dv.y : 0.f));
            const float ur = __shfl_down_sync(FULL, u[i].x, 1);
            b1[i] = mul2(sub2(u[i + 1], u[i]), splat(a.theta));
            b2[i] = mul2(sub2(make_float2(u[i].y, ur), u[i]), splat(a.theta));
            t.mask(i, b1[i], b2[i]);
        }
        s_first[threadIdx.x] = part.total();
    }
#pragma unroll
    for (int i = 0; i < RPW; ++i) sq[i] = make_float2(0.f, 0.f);
    if (wp == 0) sb.up[0][0][lane] = sb.up[1][0][lane] = make_float2(0.f, 0.f);
    if (wp == NW - 1) {
        sb.dn1[0][NW - 1][lane] = sb.dn1[1][NW - 1][lane] = make_float2(0.f, 0.f);
        sb.dn2[0][NW - 1][lane] = sb.dn2[1][NW - 1][lane] = make_float2(0.f, 0.f);
    }
    float tk = 0.f, tk_err = 0.f;
    if (t.interior) huber_reverse<true, NW, RPW>(a, t, sb, ring, groups, b1, b2, sq, tk, tk_err);
    else huber_reverse<false, NW, RPW>(a, t, sb, ring, groups, b1, b2, sq, tk, tk_err);
    // hbar -= sum qbar / theta and the h / theta partial <qbar, h> / theta^2
    const float *ub = a.Ubar + bi * a.g.NV();
    Pairs32 tqs = {};
    float2 h[RPW];
#pragma unroll
    for (int i = 0; i < RPW; ++i) {
        const bool o0 = t.row_own(i) && t.own0, o1 = t.row_own(i) && t.own1;
        const int o = t.off(i, W);
        h[i] = ld_pair(Hb, o, o0, o1, a.pair);
        hb[i] = ld_pair(a.Pin ? Hbar : ub, o, o0, o1, a.pair);
        hb[i] = fma2(sq[i], splat(-a.inv_theta), hb[i]);
        const float2 q = make_float2(o0 ? sq[i].x : 0.f, o1 ? sq[i].y : 0.f);
        const float2 qh = mul2(q, h[i]);
        tqs.add(qh, fma2(q, h[i], mul2(qh, splat(-1.f))));
    }
    const Pair32 tq = tqs.total();
    // kappa = eps / theta: d/dtheta of -tau kappa <abar, p>
    if (!a.Pin) sum[0] = s_first[threadIdx.x];
    sum[0].add_scaled(tk, tk_err, a.kfac);
    sum[0].add_scaled(tq.hi, tq.lo, a.it2);
    if (a.Pout) {
        float *Q1 = a.Pout + (size_t)bi * 2 * HW, *Q2 = Q1 + HW;
#pragma unroll
        for (int i = 0; i < RPW; ++i)
            if (t.row_own(i)) {
                st_pair(Q1, t.off(i, W), b1[i], t.own0, t.own1, a.pair);
                st_pair(Q2, t.off(i, W), b2[i], t.own0, t.own1, a.pair);
                st_pair(Hbar, t.off(i, W), hb[i], t.own0, t.own1, a.pair);
            }
    } else {
        // hbar -> w_n and the neighbours; direct dL/drho, dL/dgamma
        const float *Wn = a.Wn + bi * a.g.NV(), *A = a.A + bi * a.g.NV(), *C = a.C + bi * a.g.NV();
        float *Wb = a.Wbar + bi * a.g.NV(), *Ab = a.Abar + bi * a.g.NV(),
              *Cb = a.Cbar + bi * a.g.NV();
        const float den = a.rho + 2.f * a.gam, cw = a.rho / den, cn = a.gam / den;
        Pairs32 rb = {}, gb = {};
#pragma unroll
        for (int i = 0; i < RPW; ++i) {
            const bool o0 = t.row_own(i) && t.own0, o1 = t.row_own(i) && t.own1;
            const int o = t.off(i, W);
            const float2 w = ld_pair(Wn, o, o0, o1, a.pair);
            st_pair(Wb, o, fma2(splat(cw), hb[i], ld_pair(Wb, o, o0, o1, a.pair)), o0, o1, a.pair);
            if (a.gam > 0.f) {
                const float2 s = add2(ld_pair(A, o, o0, o1, a.pair), ld_pair(C, o, o0, o1, a.pair));
                st_pair(Ab, o, fma2(splat(cn), hb[i], ld_pair(Ab, o, o0, o1, a.pair)), o0, o1,
                        a.pair);
                st_pair(Cb, o, fma2(splat(cn), hb[i], ld_pair(Cb, o, o0, o1, a.pair)), o0, o1,
                        a.pair);
                gb.add(make_float2(o0 ? hb[i].x * (s.x - 2.f * h[i].x) / den : 0.f,
                                   o1 ? hb[i].y * (s.y - 2.f * h[i].y) / den : 0.f));
            }
            rb.add(make_float2(o0 ? hb[i].x * (w.x - h[i].x) / den : 0.f,
                               o1 ? hb[i].y * (w.y - h[i].y) / den : 0.f));
        }
        sum[1] = rb.total();
        sum[2] = gb.total();
    }
    if (a.Pout) {
        Pair32 one[1] = {sum[0]};
        const int idx[1] = {2};
        block_acc(one, a.acc, idx);
    } else {
        const int idx[3] = {2, 0, 1};
        block_acc(sum, a.acc, idx);
    }
}

// lbar -> dL/dlogits already includes m (1 - m); Uold_bar etc. are plain adds.
__global__ void axpy_kernel(float *__restrict__ y, const float *__restrict__ x, float a,
                            size_t n)
{
    for (size_t i = blockIdx.x * (size_t)kT + threadIdx.x; i < n; i += (size_t)gridDim.x * kT)
        y[i] += a * x[i];
}

// ---- host side ---------------------------------------------------------------
struct Ws {
    float *U, *D, *Wb, *Hb, *Pa, *Pb, *PH, *Useg, *Dseg;
    float *Ubar_new, *Ubar_old, *Wbar, *Dbar, *Hbar, *Pbar_a, *Pbar_b;
    double *acc;  // [3]: rho (direct), gamma (direct), theta (total)
    // keep_duals: the prox inputs h and the a^t of the dual steps of every slice of
    // a checkpoint segment, recorded by the segment's recompute:
    // Hall [S][Z][B][H][W], PHall [S][Z][T + 1][B][2][H][W] (T used); else null
    float *Hall, *PHall;
};

inline size_t al(size_t x) { return (x + 255) & ~size_t(255); }

size_t ws_bytes(const Geo &g, int T, int S, int keep)
{
    const size_t nv = (size_t)g.B * g.NV() * 4, hw = (size_t)g.B * g.HW() * 4;
    size_t n = al(nv) * 3 + al(hw) + 2 * al(2 * hw) + al((size_t)(T + 1) * 2 * hw) +
               2 * al((size_t)(S + 1) * nv) + al(nv) * 4 + al(hw) + 2 * al(2 * hw) +
               al(3 * kAccCopies * sizeof(double));
    if (keep)
        n += al((size_t)S * g.Z * hw) + al((size_t)S * g.Z * (T + 1) * 2 * hw);
    return n;
}

Ws carve(void *base, const Geo &g, int T, int S, int keep)
{
    const size_t nv = (size_t)g.B * g.NV() * 4, hw = (size_t)g.B * g.HW() * 4;
    char *p = (char *)base;
    auto take = [&](size_t n) {
        char *r = p;
        p += al(n);
        return (float *)r;
    };
    Ws w;
    w.U = take(nv);
    w.D = take(nv);
    w.Wb = take(nv);
    w.Hb = take(hw);
    w.Pa = take(2 * hw);
    w.Pb = take(2 * hw);
    w.PH = take((size_t)(T + 1) * 2 * hw);
    w.Useg = take((size_t)(S + 1) * nv);
    w.Dseg = take((size_t)(S + 1) * nv);
    w.Ubar_new = take(nv);
    w.Ubar_old = take(nv);
    w.Wbar = take(nv);
    w.Dbar = take(nv);
    w.Hbar = take(hw);
    w.Pbar_a = take(2 * hw);
    w.Pbar_b = take(2 * hw);
    w.acc = (double *)take(3 * kAccCopies * sizeof(double));
    w.Hall = keep ? take((size_t)S * g.Z * hw) : nullptr;
    w.PHall = keep ? take((size_t)S * g.Z * (T + 1) * 2 * hw) : nullptr;
    return w;
}

struct Prm {
    float rho, lam, gam, tau, eps;
    int K, T, S;
    float theta() const { return lam / (rho + 2.f * gam); }
    // dual steps of a prox: none where theta underflows to 0 (the prox is the identity)
    int steps() const { return theta() > 0.f ? T : 0; }
};

inline dim3 pgrid(const Geo &g) { return dim3((unsigned)((g.HW() + kT - 1) / kT), g.B); }
#define LAUNCH(kid, ...)                    \
    do {                                    \
        LaunchScope ls_((kid), s);          \
        __VA_ARGS__;                        \
        CSLSM_LAUNCHED();                   \
    } while (0)

// Neighbour slices of slice n at its Gauss-Seidel update (newest values): the
// previous slice is already new (old u_{Z-1} for n = 0), the next still old
// (new u_0 for n = Z-1).
inline void neighbours(const Geo &g, int n, float *Uold, float *Unew, float *&A, float *&C)
{
    const size_t HW = g.HW();
    A = n >= 1 ? Unew + (size_t)(n - 1) * HW : Uold + (size_t)(g.Z - 1) * HW;
    C = n < g.Z - 1 ? Uold + (size_t)(n + 1) * HW : Unew;
}

// Region shape (warps, rows per warp) and steps per launch.
struct HuberShape {
    int rpw, k;
};

inline long long huber_tiles(const Geo &g, int rpw, int k)
{
    const int hh = k + 1, hc = hh + (hh & 1), TH = 16 * rpw + 2 - 2 * hh, TW = 64 - 2 * hc;
    return (long long)g.B * ((g.W + TW - 1) / TW) * ((g.H + TH - 1) / TH);
}

// Few steps and large tiles waste less work on halos, many steps need fewer
// launches, and a launch wants a tile for every SM.  16 warps throughout (8 x 2,
// 8 x 4 and 8 x 8 warps x rows lost at every size).  Forward + backward in ms, 5
// iterations of 16 slices (10 for 256 x 256), steps (forward / reverse):
//   8 x 512 x 512: 4 rows x 7 / 2 rows x 5 57.4; forward 2 rows x 7 64.6; reverse
//     2 rows x 10 74.7, 4 rows x 10 63.6
//   1 x 512 x 512: 2 rows x 7 / 4 rows x 7 14.2; forward 4 rows x 10 14.6, 2 rows
//     x 10 15.7; reverse 2 rows x 10 18.0
//   1 x 256 x 256: 2 rows x 10 / 2 rows x 7 17.4; forward 2 rows x 7 21.0, 4 rows
//     x 10 22.0; reverse 2 rows x 10 18.2
HuberShape huber_shape(const Geo &g, int T, bool reverse)
{
    HuberShape h;
    if (reverse) {
        if (huber_tiles(g, 2, 5) >= 600) h = {2, 5};
        else if (huber_tiles(g, 4, 7) >= 100) h = {4, 7};
        else h = {2, 7};
    } else {
        if (huber_tiles(g, 4, 7) >= 300) h = {4, 7};
        else if (huber_tiles(g, 2, 7) >= 152) h = {2, 7};
        else h = {2, 10};
    }
    const int P = std::max(1, (T + h.k - 1) / h.k);  // balanced phases
    h.k = std::max(1, (T + P - 1) / P);
    return h;
}

template <int NW, int RPW>
cslsm_status launch_huber_shape(const HuberArgs &a, dim3 grid, bool reverse, cudaStream_t s)
{
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(NW * 32);
    cfg.stream = s;
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    LaunchScope ls(K_DIFF, s);
    if (reverse) {
        cfg.dynamicSmemBytes = HuberRing<NW, RPW>::bytes();
        CSLSM_CUDA(cudaFuncSetAttribute(huber_bwd_kernel<NW, RPW>,
                                        cudaFuncAttributeMaxDynamicSharedMemorySize,
                                        (int)cfg.dynamicSmemBytes));
        CSLSM_CUDA(cudaLaunchKernelEx(&cfg, huber_bwd_kernel<NW, RPW>, a));
    } else {
        CSLSM_CUDA(cudaLaunchKernelEx(&cfg, huber_fwd_kernel<NW, RPW>, a));
    }
    return CSLSM_OK;
}

cslsm_status launch_huber(HuberArgs a, int rpw, bool reverse, cudaStream_t s)
{
    a.TH = 16 * rpw + 2 - 2 * a.hh;
    a.TW = 64 - 2 * a.hc;
    a.tx = (a.g.W + a.TW - 1) / a.TW;
    const dim3 grid((unsigned)(a.tx * ((a.g.H + a.TH - 1) / a.TH)), a.g.B);
    return rpw == 2 ? launch_huber_shape<16, 2>(a, grid, reverse, s)
                    : launch_huber_shape<16, 4>(a, grid, reverse, s);
}

inline bool pairs_ok(const Geo &g, const void *ws) { return g.W % 2 == 0 && (uintptr_t)ws % 8 == 0; }

HuberArgs huber_args(const Geo &g, const Prm &P, int k, bool pair)
{
    HuberArgs a{};
    a.g = g;
    a.rho = P.rho;
    a.gam = P.gam;
    a.theta = P.theta();
    a.inv_theta = a.theta > 0.f ? 1.f / a.theta : 0.f;
    a.tau = P.tau;
    const double it2 = (double)a.inv_theta * a.inv_theta, kfac = it2 * P.tau * P.eps;
    a.it2 = make_float2((float)it2, (float)(it2 - (float)it2));
    a.kfac = make_float2((float)kfac, (float)(kfac - (float)kfac));
    a.kappa = a.theta > 0.f ? P.eps / a.theta : 0.f;
    a.T = P.steps();
    a.hh = k + 1;
    a.hc = a.hh + (a.hh & 1);
    a.pair = pair;
    return a;
}

// One slice's prox of every batch item from w_n and the neighbour slices A, C:
// h into Hb, a^t into rec [T][B][2][H][W] when given, u_n and d_n into Un, Dn
// when given.  Pa, Pb: [B][2][H][W] scratch.
cslsm_status slice_prox(const Geo &g, const Prm &P, const float *Wn, const float *A,
                        const float *C, float *Hb, float *Pa, float *Pb, float *rec, float *Un,
                        float *Dn, bool pair, cudaStream_t s)
{
    const int T = P.steps();
    const HuberShape sh = huber_shape(g, T, false);
    HuberArgs a = huber_args(g, P, sh.k, pair);
    a.Wn = Wn;
    a.A = A;
    a.C = C;
    a.Hb = Hb;
    const size_t hw2 = (size_t)g.B * 2 * g.HW();
    float *out = Pa;
    for (int t = 0; t == 0 || t < T; t += sh.k) {
        a.ns = std::min(sh.k, T - t);
        const bool last = t + a.ns == T;
        a.Pout = last ? nullptr : out;
        a.rec = rec ? rec + (size_t)t * hw2 : nullptr;
        a.Un = last ? Un : nullptr;
        a.Dn = Dn;
        cslsm_status e = launch_huber(a, sh.rpw, false, s);
        if (e) return e;
        a.Pin = out;
        out = out == Pa ? Pb : Pa;
    }
    return CSLSM_OK;
}

// Its reverse: Ubar (dL/du_n) to Wbar, Abar, Cbar (added) and the scalars.
cslsm_status slice_prox_bwd(const Geo &g, const Prm &P, const float *Wn, const float *A,
                            const float *C, float *Hb, float *rec, const float *Ubar, float *Hbar,
                            float *Pa, float *Pb, float *Wbar, float *Abar, float *Cbar,
                            double *acc, bool pair, cudaStream_t s)
{
    const int T = P.steps();
    const HuberShape sh = huber_shape(g, T, true);
    HuberArgs a = huber_args(g, P, sh.k, pair);
    a.Wn = Wn;
    a.A = A;
    a.C = C;
    a.Hb = Hb;
    a.rec = rec;
    a.Ubar = Ubar;
    a.Hbar = Hbar;
    a.Wbar = Wbar;
    a.Abar = Abar;
    a.Cbar = Cbar;
    a.acc = acc;
    float *out = Pa;
    for (int t = T; t == T || t > 0; t -= sh.k) {
        a.ns = std::min(sh.k, t);
        a.t0 = t - a.ns;
        a.Pout = a.t0 > 0 ? out : nullptr;
        cslsm_status e = launch_huber(a, sh.rpw, true, s);
        if (e) return e;
        a.Pin = out;
        out = out == Pa ? Pb : Pa;
    }
    return CSLSM_OK;
}

// One forward iteration on (U, D) in place; writes v when vout != null.  With
// Hrec / PHrec (keep_duals), slice n's prox input goes to Hrec + n [B][H][W]
// and the a of its dual steps to PHrec + n [T + 1][B][2][H][W].
cslsm_status fwd_iter(const Geo &g, const Prm &P, const float *logits, const float *b, Ws &w,
                      float *vout, bool pair, cudaStream_t s, float *Hrec = nullptr,
                      float *PHrec = nullptr)
{
    const float gam = g.Z > 1 ? P.gam : 0.f;
    LAUNCH(K_DIFF, ux_fwd_kernel<<<pgrid(g), kT, 0, s>>>(w.U, w.D, logits, b, g, P.rho, w.Wb, vout));
    Prm Q = P;
    Q.gam = gam;
    for (int n = 0; n < g.Z; ++n) {
        float *A, *C;
        neighbours(g, n, w.U, w.U, A, C);  // in place: the array holds the newest values
        const size_t off = (size_t)n * g.HW();
        const size_t hwf = (size_t)g.B * g.HW();
        float *Hb = Hrec ? Hrec + (size_t)n * hwf : w.Hb;
        float *PH = PHrec ? PHrec + (size_t)n * (P.T + 1) * 2 * hwf : nullptr;
        cslsm_status e = slice_prox(g, Q, w.Wb + off, A, C, Hb, w.Pa, w.Pb, PH, w.U + off,
                                    w.D + off, pair, s);
        if (e) return e;
    }
    return CSLSM_OK;
}

}  // namespace

size_t unrolled_workspace_bytes(int B, int Z, int H, int W, int T, int S, int keep)
{
    return ws_bytes(Geo{B, Z, H, W}, T, S, keep);
}

cslsm_status unrolled_forward(int B, int Z, int H, int W, float rho, float lam, float gam,
                              int K, int T, float tau, float eps, int S, const float *logits,
                              const float *b, float *vout, float *ckpt, void *ws, cudaStream_t s)
{
    const Geo g{B, Z, H, W};
    const Prm P{rho, lam, gam, tau, eps, K, T, S};
    Ws w = carve(ws, g, T, S, 0);  // the kept duals, if any, lie beyond this part
    const size_t nv = (size_t)B * g.NV();
    CSLSM_CUDA(cudaMemsetAsync(w.U, 0, nv * 4, s));
    CSLSM_CUDA(cudaMemsetAsync(w.D, 0, nv * 4, s));
    for (int k = 0; k < K; ++k) {
        if (k % S == 0 && ckpt) {
            float *c = ckpt + (size_t)(k / S) * 2 * nv;
            CSLSM_CUDA(cudaMemcpyAsync(c, w.U, nv * 4, cudaMemcpyDeviceToDevice, s));
            CSLSM_CUDA(cudaMemcpyAsync(c + nv, w.D, nv * 4, cudaMemcpyDeviceToDevice, s));
        }
        cslsm_status e = fwd_iter(g, P, logits, b, w, k == K - 1 ? vout : nullptr,
                                  pairs_ok(g, ws), s);
        if (e) return e;
    }
    return CSLSM_OK;
}

cslsm_status unrolled_backward(int B, int Z, int H, int W, float rho, float lam, float gam,
                               int K, int T, float tau, float eps, int S, int keep,
                               const float *logits, const float *b, const float *ckpt,
                               const float *vbar, float *logits_bar, double *scal_bar, void *ws,
                               cudaStream_t s)
{
    const Geo g{B, Z, H, W};
    Prm P{rho, lam, gam, tau, eps, K, T, S};
    const float gz = Z > 1 ? gam : 0.f;
    P.gam = gz;
    Ws w = carve(ws, g, T, S, keep);
    const size_t nv = (size_t)B * g.NV(), HW = g.HW(), hw2 = (size_t)B * 2 * HW;
    const size_t hwf = (size_t)B * HW;
    const float den = rho + 2.f * gz;
    const bool pair = pairs_ok(g, ws);
    CSLSM_CUDA(cudaMemsetAsync(w.acc, 0, 3 * kAccCopies * sizeof(double), s));
    CSLSM_CUDA(cudaMemsetAsync(logits_bar, 0, nv * 4, s));
    // adjoint of the state after the last iteration: only v^K is observed
    CSLSM_CUDA(cudaMemsetAsync(w.Ubar_new, 0, nv * 4, s));
    CSLSM_CUDA(cudaMemsetAsync(w.Dbar, 0, nv * 4, s));
    const int nseg = (K + S - 1) / S;
    for (int sg = nseg - 1; sg >= 0; --sg) {
        const int k0 = sg * S, k1 = std::min(K, k0 + S);
        // recompute the segment's states u^k, d^k for k = k0 .. k1
        const float *c = ckpt + (size_t)sg * 2 * nv;
        CSLSM_CUDA(cudaMemcpyAsync(w.U, c, nv * 4, cudaMemcpyDeviceToDevice, s));
        CSLSM_CUDA(cudaMemcpyAsync(w.D, c + nv, nv * 4, cudaMemcpyDeviceToDevice, s));
        for (int k = k0; k <= k1; ++k) {
            const int slot = k - k0;
            CSLSM_CUDA(cudaMemcpyAsync(w.Useg + (size_t)slot * nv, w.U, nv * 4,
                                       cudaMemcpyDeviceToDevice, s));
            CSLSM_CUDA(cudaMemcpyAsync(w.Dseg + (size_t)slot * nv, w.D, nv * 4,
                                       cudaMemcpyDeviceToDevice, s));
            if (k < k1) {
                // keep_duals: record every slice's h and dual iterates of iteration k
                cslsm_status e =
                    fwd_iter(g, P, logits, b, w, nullptr, pair, s,
                             keep ? w.Hall + (size_t)slot * Z * hwf : nullptr,
                             keep ? w.PHall + (size_t)slot * Z * (T + 1) * hw2 : nullptr);
                if (e) return e;
            }
        }
        for (int k = k1 - 1; k >= k0; --k) {
            const int slot = k - k0;
            float *Uo = w.Useg + (size_t)slot * nv, *Do = w.Dseg + (size_t)slot * nv;
            float *Un = w.Useg + (size_t)(slot + 1) * nv;
            // w^{k+1} from (u^k, d^k)
            LAUNCH(K_DIFF, ux_fwd_kernel<<<pgrid(g), kT, 0, s>>>(Uo, Do, logits, b, g, rho, w.Wb,
                                                                   nullptr));
            // d^{k+1} = w - u^{k+1}:  wbar = dbar, ubar_new -= dbar
            CSLSM_CUDA(cudaMemcpyAsync(w.Wbar, w.Dbar, nv * 4, cudaMemcpyDeviceToDevice, s));
            LAUNCH(K_DIFF, axpy_kernel<<<4096, kT, 0, s>>>(w.Ubar_new, w.Dbar, -1.f, nv));
            CSLSM_CUDA(cudaMemsetAsync(w.Ubar_old, 0, nv * 4, s));
            // reverse Gauss-Seidel sweep
            for (int n = Z - 1; n >= 0; --n) {
                float *A, *C;
                neighbours(g, n, Uo, Un, A, C);
                float *Ab, *Cb;
                neighbours(g, n, w.Ubar_old, w.Ubar_new, Ab, Cb);
                const size_t off = (size_t)n * HW;
                // the prox input h and the a^t of its dual steps: kept by the segment's
                // recompute, or recomputed here
                float *Hn = w.Hb, *PHn = w.PH;
                if (keep) {
                    Hn = w.Hall + ((size_t)slot * Z + n) * hwf;
                    PHn = w.PHall + ((size_t)slot * Z + n) * (T + 1) * hw2;
                } else {
                    cslsm_status e = slice_prox(g, P, w.Wb + off, A, C, Hn, w.Pa, w.Pb, PHn,
                                                nullptr, nullptr, pair, s);
                    if (e) return e;
                }
                cslsm_status e = slice_prox_bwd(g, P, w.Wb + off, A, C, Hn, PHn,
                                                w.Ubar_new + off, w.Hbar, w.Pbar_a, w.Pbar_b,
                                                w.Wbar + off, Ab, Cb, w.acc, pair, s);
                if (e) return e;
            }
            // x-update reverse: u^k, d^k adjoints
            LAUNCH(K_DIFF, ux_bwd_kernel<<<pgrid(g), kT, 0, s>>>(
                               Uo, Do, logits, b, g, rho, k == K - 1 ? vbar : nullptr, w.Wbar,
                               w.Ubar_old, w.Dbar, logits_bar, w.acc));
            std::swap(w.Ubar_new, w.Ubar_old);  // adjoint of u^k becomes the next "new"
        }
    }
    // scalars: rho_direct, gamma_direct, theta_total -> (rho, lambda, gamma)
    double copies[3 * kAccCopies], acc[3] = {0.0, 0.0, 0.0};
    CSLSM_CUDA(cudaMemcpyAsync(copies, w.acc, sizeof(copies), cudaMemcpyDeviceToHost, s));
    CSLSM_CUDA(cudaStreamSynchronize(s));
    for (int q = 0; q < 3; ++q)
        for (int c = 0; c < kAccCopies; ++c) acc[q] += copies[q * kAccCopies + c];
    const double dd = (double)den;
    double out[3];
    out[1] = acc[2] / dd;                                   // dtheta/dlambda = 1/den
    out[0] = acc[0] - acc[2] * lam / (dd * dd);             // dtheta/drho = -lambda/den^2
    out[2] = (Z > 1 ? acc[1] - 2.0 * acc[2] * lam / (dd * dd) : 0.0);
    CSLSM_CUDA(cudaMemcpyAsync(scal_bar, out, sizeof(out), cudaMemcpyHostToDevice, s));
    CSLSM_CUDA(cudaStreamSynchronize(s));
    return CSLSM_OK;
}

}  // namespace cslsm
