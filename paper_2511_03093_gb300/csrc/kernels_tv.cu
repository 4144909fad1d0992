// Isotropic-TV prox of the u-step (Eq. u-sub / u-update) by Chambolle's dual
// projection, with the z-smoothness Gauss-Seidel input of Sec. III-C folded
// into the tile load.
//
//   g  = (rho w_n + gamma (u_{n-1} + u_{n+1})) / (rho + 2 gamma)   (gamma > 0)
//      = w_n                                                        (gamma = 0)
//   p^0 = 0,  q^t = div p^t - g / theta,
//   p^{t+1} = (p^t + tau grad q^t) / (1 + tau |grad q^t|),
//   u_n = g - theta div p^T,  d_n = w_n - u_n.
// grad: forward differences, zero on the last row / column; div = -grad^T.
//
// GB300 design: temporal blocking in shared memory.  One CTA owns a TH x TW
// output tile of one slice and loads g on the tile plus a halo of T+1 pixels
// (the dependence cone of T Chambolle steps), so all T steps run on chip and
// the dual field p never touches HBM; one launch performs the whole prox of
// every slice it covers.  HBM/L2 traffic per prox is one read of w (plus the
// two neighbouring u slices when gamma > 0) and one write of u and d.
//
// Inside a step every warp walks a band of rows top to bottom, one row per
// iteration; each lane owns two adjacent columns (float2 shared accesses).
// q of the next row is computed once and carried in registers, the right
// neighbour's q comes from a warp shuffle and the left neighbour's p from the
// float2 holding the two columns to the left (no lane-divergent load), so a
// pixel-step costs 2 shared loads and 1 store.  A warp spans 64 columns
// and owns 62 of them (column chunks overlap by two so that every chunk
// starts on an even column; the last lane only supplies q and p to its
// neighbours).  p is double-buffered in shared memory,
// so one __syncthreads per step suffices, and the row bands are re-balanced
// every step as the valid region shrinks by one pixel per side.  The Neumann
// boundary and the outside of the image are handled without branches:
// gradient components are multiplied by a 0/1 row / column mask, which keeps
// p = 0 wherever the discrete gradient vanishes.
//
// Step counts above kMaxSteps are split into chunks that hand p over through
// a double-buffered global array.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <map>
#include <mutex>
#include <tuple>
#include <vector>

#include "internal.cuh"
#include "storage.cuh"
#include "tv_body.cuh"

namespace cslsm {
namespace {

// ---- phases: the prox in launches of a few steps ------------------------------
// The tile kernel below runs all T steps in one launch on a halo of T + 1 pixels.
// Here a launch runs k of them on a halo of k + 1 with the dual field in registers
// (a warp holds RPW rows, a lane two columns; sweep_steps, one barrier a step) and
// hands p over in global memory, so that a step costs about a third and the halo
// half; programmatic dependent launch hides most of a launch's latency.  Bound by the
// step's dependent chain on small volumes and by issue on large ones.  ADMM iteration
// in us, gamma = 0, T = 20, FP32 (tile kernel / one-item persistent batch / phases):
// 64 x 64 x 8 30 / - / 16; 128 x 128 x 8 32 / 55 / 22; 256 x 256 x 16 110 / 79 / 57; 512 x
// 512 x 16 335 / 196 / 166; 999 x 701 x 24 1227 / 977 / 666; 1024 x 1024 x 32 2450 / 1350 /
// 1221 (BF16 2494 / 1413 / 1541).  The same bits on every path.
struct TvPhase {
    const void *w;  // element type S
    void *u, *d;
    const float *pin;  // [2][nslices][H][W] p of the phase before, or null (p = 0)
    float *pout;       // for the next phase, or null (the last: u and d are written)
    int H, W, Z, n0, nslices;
    int ns, hh, hc, TH, TW, tx;
    float rho, gamma, inv_rho2g, theta, inv_theta, tau;
    int pair;  // W even, buffers aligned: a lane's two columns in one access
    const int *stop;
};

template <typename S>
__device__ __forceinline__ float2 ld_cols(const S *p, int off, bool in0, bool in1, int pair)
{
    if (pair) return in0 ? ld2_l2<S>(p + off) : make_float2(0.f, 0.f);
    return make_float2(in0 ? ld_l2<S>(p + off) : 0.f, in1 ? ld_l2<S>(p + off + 1) : 0.f);
}

template <typename S>
__device__ __forceinline__ void st_cols(S *p, int off, float2 v, bool in0, bool in1, int pair)
{
    if (pair) {
        if (in0) st2<S>(p + off, v);
    } else {
        if (in0) st<S>(p + off, v.x);
        if (in1) st<S>(p + off + 1, v.y);
    }
}

constexpr int kPhaseWarps = 16;

template <int RPW, typename S>
__global__ void __launch_bounds__(kPhaseWarps * 32, 2) tv_phase_kernel(const TvPhase a)
{
    constexpr int NW = kPhaseWarps, RH = NW * RPW + 2;
    constexpr unsigned FULL = 0xffffffffu;
    __shared__ Bnd<NW> sb;
    const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5, H = a.H, W = a.W;
    const int bx = (int)blockIdx.x % a.tx, by = (int)blockIdx.x / a.tx, sl = blockIdx.y;
    const int gi0 = by * a.TH - a.hh, gj0 = bx * a.TW - a.hc;
    const int j0 = 2 * lane, gc = gj0 + j0, r0 = 1 + wp * RPW;
    const bool in0 = gc >= 0 && gc < W, in1 = gc + 1 >= 0 && gc + 1 < W;
    const bool own0 = in0 && j0 >= a.hc && j0 < a.hc + a.TW;
    const bool own1 = in1 && j0 + 1 >= a.hc && j0 + 1 < a.hc + a.TW;
    const float mc0 = in0 && gc < W - 1 ? 1.f : 0.f, mc1 = in1 && gc + 1 < W - 1 ? 1.f : 0.f;
    const bool interior = gi0 >= 0 && gi0 + RH < H && gj0 >= 0 && gj0 + 64 < W;
    unsigned inr = 0, ownr = 0, mr = 0;  // bit i: row i in the image / owned / has one below
#pragma unroll
    for (int i = 0; i <= RPW; ++i) {
        const int gi = gi0 + r0 + i;
        if (gi >= 0 && gi < H) inr |= 1u << i;
        if (gi >= 0 && gi < H - 1) mr |= 1u << i;
        if (i < RPW && gi >= 0 && gi < H && r0 + i >= a.hh && r0 + i < a.hh + a.TH) ownr |= 1u << i;
    }
    // let the next launch's blocks in, then wait for the launch before to complete
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (a.stop && *a.stop) return;
    const int n = a.n0 + sl;
    const size_t HW = (size_t)H * W;
    const S *wn = (const S *)a.w + n * HW;
    const S *um = (const S *)a.u + (size_t)((n + a.Z - 1) % a.Z) * HW;
    const S *up = (const S *)a.u + (size_t)((n + 1) % a.Z) * HW;
    auto off = [&](int i) { return (gi0 + r0 + i) * W + gc; };
    float2 p1[RPW], p2[RPW], g[RPW], gdn;
#pragma unroll
    for (int i = 0; i <= RPW; ++i) {
        const bool i0 = ((inr >> i) & 1u) && in0, i1 = ((inr >> i) & 1u) && in1;
        float2 v = ld_cols<S>(wn, off(i), i0, i1, a.pair);
        if (a.gamma > 0.f) {
            const float2 m = ld_cols<S>(um, off(i), i0, i1, a.pair);
            const float2 q = ld_cols<S>(up, off(i), i0, i1, a.pair);
            v.x = i0 ? (a.rho * v.x + a.gamma * (m.x + q.x)) * a.inv_rho2g : 0.f;
            v.y = i1 ? (a.rho * v.y + a.gamma * (m.y + q.y)) * a.inv_rho2g : 0.f;
        }
        if (i < RPW) g[i < RPW ? i : 0] = v;
        else gdn = v;
    }
    float2 f1 = make_float2(0.f, 0.f), f2 = f1;
    if (a.pin) {
        const float *P1 = a.pin + (size_t)sl * HW, *P2 = a.pin + (size_t)(a.nslices + sl) * HW;
#pragma unroll
        for (int i = 0; i < RPW; ++i) {
            const bool i0 = ((inr >> i) & 1u) && in0, i1 = ((inr >> i) & 1u) && in1;
            p1[i] = ld_cols<float>(P1, off(i), i0, i1, a.pair);
            p2[i] = ld_cols<float>(P2, off(i), i0, i1, a.pair);
        }
        if (wp == 0 || wp == NW - 1) {  // frozen rows 0 and RH - 1 of the region
            const int gi = gi0 + (wp == 0 ? 0 : RH - 1);
            const bool in = gi >= 0 && gi < H;
            f1 = ld_cols<float>(P1, gi * W + gc, in && in0, in && in1, a.pair);
            f2 = ld_cols<float>(P2, gi * W + gc, in && in0, in && in1, a.pair);
        }
    } else {
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
    // exact after the phase: the own tile, and the row above it where u is formed
    const int lo = a.hh - (a.pout ? 0 : 1), hi = a.hh + a.TH;
    if (interior)
        sweep_steps<true, NW, RPW>(sb, p1, p2, g, gdn, mr, mc0, mc1, a.inv_theta, a.tau, a.ns, wp,
                                   lane, lo, hi);
    else
        sweep_steps<false, NW, RPW>(sb, p1, p2, g, gdn, mr, mc0, mc1, a.inv_theta, a.tau, a.ns, wp,
                                    lane, lo, hi);
    if (a.pout) {
        float *Q1 = a.pout + (size_t)sl * HW, *Q2 = a.pout + (size_t)(a.nslices + sl) * HW;
#pragma unroll
        for (int i = 0; i < RPW; ++i) {
            if (!((ownr >> i) & 1u)) continue;
            st_cols<float>(Q1, off(i), p1[i], own0, own1, a.pair);
            st_cols<float>(Q2, off(i), p2[i], own0, own1, a.pair);
        }
        return;
    }
    S *un = (S *)a.u + n * HW, *dn = a.d ? (S *)a.d + n * HW : nullptr;
    const float2 pu0 = sb.up[a.ns & 1][wp][lane];
#pragma unroll
    for (int i = 0; i < RPW; ++i) {
        const float p2l = __shfl_up_sync(FULL, p2[i].y, 1);
        const float2 pu = i == 0 ? pu0 : p1[i > 0 ? i - 1 : 0];
        const float dx = (p1[i].x - pu.x) + (p2[i].x - p2l);
        const float dy = (p1[i].y - pu.y) + (p2[i].y - p2[i].x);
        if (!((ownr >> i) & 1u)) continue;
        const size_t vi = n * HW + (size_t)off(i);
        const float2 ur = make_float2(keep<S>(g[i].x - a.theta * dx, vi, kKeyU),
                                      keep<S>(g[i].y - a.theta * dy, vi + 1, kKeyU));
        st_cols<S>(un, off(i), ur, own0, own1, a.pair);
        if (dn) {
            const float2 wv = ld_cols<S>(wn, off(i), own0, own1, a.pair);
            st_cols<S>(dn, off(i), make_float2(keep<S>(wv.x - ur.x, vi, kKeyD),
                                               keep<S>(wv.y - ur.y, vi + 1, kKeyD)),
                       own0, own1, a.pair);
        }
    }
}

constexpr int kMaxSteps = 24;

inline size_t smem_bytes(int C, int RH) { return tv_smem_bytes(C, RH); }

constexpr size_t kSmemLimit = 227 * 1024;  // per CTA
constexpr size_t kSmemPerSm = 228 * 1024;

// Kernel variants: (column chunks, row bands).
struct Variant {
    int C, B;
};
constexpr Variant kVariants[] = {{1, 12}, {1, 24}, {2, 12}, {2, 16}};
constexpr int kNumVariants = 4;

struct Shape {
    int v, TH, TW, RH;  // variant index, tile rows / columns, region rows
};

std::mutex g_mu;
struct DeviceInfo {
    int sms = 0;
    bool ready = false;
};
std::vector<DeviceInfo> g_dev;
int g_mode = 0;  // 0: cost model, 1: timed autotuning, 2 + k: force variant k
struct Key {
    int dev, H, W, T, ns;
    bool operator<(const Key &o) const
    {
        return std::tie(dev, H, W, T, ns) < std::tie(o.dev, o.H, o.W, o.T, o.ns);
    }
};
std::map<Key, Shape> g_tuned;

template <int C, int B>
cslsm_status set_attr()
{
    const int lim = (int)kSmemLimit;
    CSLSM_CUDA(cudaFuncSetAttribute(tv_tile_kernel<C, B, float>,
                                    cudaFuncAttributeMaxDynamicSharedMemorySize, lim));
    CSLSM_CUDA(cudaFuncSetAttribute(tv_tile_kernel<C, B, __nv_bfloat16>,
                                    cudaFuncAttributeMaxDynamicSharedMemorySize, lim));
    CSLSM_CUDA(cudaFuncSetAttribute(tv_tile_kernel<C, B, __half>,
                                    cudaFuncAttributeMaxDynamicSharedMemorySize, lim));
    return CSLSM_OK;
}

cslsm_status device_info(int &dev, int &sms)
{
    CSLSM_CUDA(cudaGetDevice(&dev));
    std::lock_guard<std::mutex> lk(g_mu);
    if ((int)g_dev.size() <= dev) g_dev.resize(dev + 1);
    DeviceInfo &di = g_dev[dev];
    if (!di.ready) {
        CSLSM_CUDA(cudaDeviceGetAttribute(&di.sms, cudaDevAttrMultiProcessorCount, dev));
        cslsm_status e;
        if ((e = set_attr<1, 12>()) || (e = set_attr<1, 24>()) || (e = set_attr<2, 12>()) ||
            (e = set_attr<2, 16>()))
            return e;
        di.ready = true;
    }
    sms = di.sms;
    return CSLSM_OK;
}

// Best tile rows for one variant under the cost model: waves of CTAs times the
// pixel-steps of one CTA's shrinking region, with a latency penalty when fewer
// than 32 warps share an SM.  Returns the modelled cost (inf if nothing fits).
double model_shape(int vi, int H, int W, int T, int nslices, int sms, Shape &out)
{
    const int C = kVariants[vi].C, B = kVariants[vi].B;
    const int RW = 62 * C + 2, TW = RW - 2 * T - 2;
    double best = 1e300;
    if (TW < 4) return best;
    const int tiles_w = (W + TW - 1) / TW, threads = C * B * 32;
    for (int TH = 4; TH <= 1024; TH += 2) {
        const int RH = TH + 2 * T + 2;
        const size_t sm = smem_bytes(C, RH);
        if (sm > kSmemLimit) break;
        const int per_sm = (int)std::min<size_t>(kSmemPerSm / (sm + 1024), 2048 / threads);
        if (per_sm < 1) break;
        const long long ctas = (long long)tiles_w * ((H + TH - 1) / TH) * nslices;
        const int resident = (int)std::min<long long>(per_sm, (ctas + sms - 1) / sms);
        const double waves = std::ceil((double)ctas / ((double)sms * per_sm));
        double work = 2.0 * RW * RH;  // pixel-steps of one CTA plus its load
        for (int s = 0; s < T; ++s) work += (double)(RW - 2 * s - 3) * (RH - 2 * s - 3);
        const double warps = (double)resident * C * B;
        const double cost = waves * work * per_sm * std::max(1.0, 32.0 / warps);
        if (cost < best) {
            best = cost;
            out = Shape{vi, TH, TW, RH};
        }
        if (TH >= H) break;
    }
    return best;
}

template <typename S>
void launch_variant(int v, dim3 grid, int nt, size_t sm, cudaStream_t st, const TvLaunch &b)
{
    switch (v) {
    case 0: tv_tile_kernel<1, 12, S><<<grid, nt, sm, st>>>(b); break;
    case 1: tv_tile_kernel<1, 24, S><<<grid, nt, sm, st>>>(b); break;
    case 2: tv_tile_kernel<2, 12, S><<<grid, nt, sm, st>>>(b); break;
    default: tv_tile_kernel<2, 16, S><<<grid, nt, sm, st>>>(b); break;
    }
}

cslsm_status launch_tile(const TvLaunch &a, const Shape &sh, cudaStream_t st)
{
    if (sh.RH <= 0) {
        set_error("no TV tile shape fits shared memory for %d steps", a.T);
        return CSLSM_ERR_UNSUPPORTED;
    }
    TvLaunch b = a;
    b.TH = sh.TH;
    b.TW = sh.TW;
    b.RH = sh.RH;
    const Variant v = kVariants[sh.v];
    const dim3 grid((a.W + sh.TW - 1) / sh.TW, (a.H + sh.TH - 1) / sh.TH, a.nslices);
    const size_t sm = smem_bytes(v.C, sh.RH);
    const int nt = v.C * v.B * 32;
    LaunchScope ls(K_TV_TILE, st);
    if (a.storage == CSLSM_STORE_BF16) launch_variant<__nv_bfloat16>(sh.v, grid, nt, sm, st, b);
    else if (a.storage == CSLSM_STORE_FP16) launch_variant<__half>(sh.v, grid, nt, sm, st, b);
    else launch_variant<float>(sh.v, grid, nt, sm, st, b);
    CSLSM_LAUNCHED();
    return CSLSM_OK;
}

// Shape for this launch: forced variant, cached tuning result, cost model, or
// (mode 1, outside stream capture, first use of the key) timed candidates.
cslsm_status choose_shape(const TvLaunch &a, int dev, int sms, cudaStream_t st, bool may_time,
                          Shape &sh)
{
    int mode;
    {
        std::lock_guard<std::mutex> lk(g_mu);
        mode = g_mode;
        if (mode == 1 && !may_time) mode = 0;
        if (mode == 1) {
            auto it = g_tuned.find(Key{dev, a.H, a.W, a.T, a.nslices});
            if (it != g_tuned.end()) {
                sh = it->second;
                return CSLSM_OK;
            }
        }
    }
    Shape cand[kNumVariants];
    double cost[kNumVariants];
    int best = -1;
    for (int v = 0; v < kNumVariants; ++v) {
        cand[v] = Shape{v, 0, 0, 0};
        cost[v] = model_shape(v, a.H, a.W, a.T, a.nslices, sms, cand[v]);
        if (cost[v] < 1e300 && (best < 0 || cost[v] < cost[best])) best = v;
    }
    if (mode >= 2) {
        const int v = (mode - 2) % kNumVariants;
        if (cost[v] < 1e300) best = v;
    }
    if (best < 0) {
        set_error("no TV tile shape fits shared memory for %d steps", a.T);
        return CSLSM_ERR_UNSUPPORTED;
    }
    sh = cand[best];
    if (mode != 1) return CSLSM_OK;
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    CSLSM_CUDA(cudaStreamIsCapturing(st, &cap));
    if (cap != cudaStreamCaptureStatusNone) return CSLSM_OK;
    // time every variant (the launch is idempotent: same inputs, same outputs)
    cudaEvent_t e0, e1;
    CSLSM_CUDA(cudaEventCreate(&e0));
    CSLSM_CUDA(cudaEventCreate(&e1));
    float best_ms = 1e30f;
    for (int v = 0; v < kNumVariants; ++v) {
        if (cost[v] >= 1e300) continue;
        float ms_min = 1e30f;
        for (int rep = 0; rep < 3; ++rep) {
            cudaEventRecord(e0, st);
            cslsm_status e = launch_tile(a, cand[v], st);
            cudaEventRecord(e1, st);
            if (e) {
                cudaEventDestroy(e0);
                cudaEventDestroy(e1);
                return e;
            }
            float ms = 0.f;
            if (cudaEventSynchronize(e1) == cudaSuccess && cudaEventElapsedTime(&ms, e0, e1) ==
                                                               cudaSuccess)
                ms_min = std::min(ms_min, ms);
        }
        if (ms_min < best_ms) {
            best_ms = ms_min;
            sh = cand[v];
        }
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    std::lock_guard<std::mutex> lk(g_mu);
    g_tuned[Key{dev, a.H, a.W, a.T, a.nslices}] = sh;
    return CSLSM_OK;
}

// The exchange of p (16 bytes a voxel) is kept to 1 GB; larger volumes run elsewhere.
constexpr size_t kPhaseMaxFloats = 256ull << 20;
constexpr int kPhaseMaxSlices = 65535;  // a grid's y extent; more slices run elsewhere too

struct PhaseShape {
    int rpw = 0, P = 0, k = 0, hh = 0, hc = 0, TH = 0, TW = 0, tx = 0, ty = 0;
    double us = 1e30;
};

// Candidate with RPW rows per warp and P phases; false if the halo leaves no tile.
bool phase_shape(int rpw, int P, int H, int W, int T, int nslices, int sms, PhaseShape &f)
{
    f.rpw = rpw;
    f.P = P;
    f.k = (T + P - 1) / P;
    f.hh = f.k + 1;
    f.hc = f.hh + (f.hh & 1);  // even: regions start on even columns
    f.TH = kPhaseWarps * rpw + 2 - 2 * f.hh;
    f.TW = 64 - 2 * f.hc;
    if (f.TH < 4 || f.TW < 4) return false;
    f.tx = (W + f.TW - 1) / f.TW;
    f.ty = (H + f.TH - 1) / f.TH;
    // Microseconds, fitted to 93 measured (geometry, rpw, P): 64 x 64 x 8 to 700 x 333 x
    // 20, FP32, T = 20, 5 % rms; its choice is the best one there within 1 %.  A phase
    // runs in rounds of two CTAs per SM (one per SM in the last, if they fit).
    const double active = std::min((double)kPhaseWarps, std::ceil((f.TH + f.k - 1.0) / rpw) + 0.5);
    const double step = 0.137 + 0.0919 * rpw;
    const double t1 = f.k * (step - 0.0016 * active * rpw) + 0.531 * rpw;
    const double t2 = f.k * step + 1.062 * rpw;
    const long long ctas = (long long)f.tx * f.ty * nslices, full = ctas / (2 * sms),
                    rest = ctas - full * 2 * sms;
    f.us = P * (1.64 + full * t2 + (rest > sms ? t2 : rest > 0 ? t1 : 0.0));
    return true;
}

PhaseShape phase_best(int H, int W, int T, int nslices, int sms)
{
    PhaseShape best;
    for (int rpw = 2; rpw <= 4; rpw += 2)
        for (int P = 1; P <= T && (T + P - 1) / P >= std::min(T, 4); ++P) {
            PhaseShape f;
            if (phase_shape(rpw, P, H, W, T, nslices, sms, f) && f.us < best.us) best = f;
        }
    return best;
}

template <int RPW, typename S>
cslsm_status launch_phase(const TvPhase &a, const PhaseShape &f, cudaStream_t st)
{
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)(f.tx * f.ty), (unsigned)a.nslices);
    cfg.blockDim = dim3(kPhaseWarps * 32);
    cfg.stream = st;
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    LaunchScope ls(K_TV_TILE, st);
    CSLSM_CUDA(cudaLaunchKernelEx(&cfg, tv_phase_kernel<RPW, S>, a));
    return CSLSM_OK;
}

template <typename S>
cslsm_status launch_phase_typed(const TvPhase &a, const PhaseShape &f, cudaStream_t st)
{
    return f.rpw == 2 ? launch_phase<2, S>(a, f, st) : launch_phase<4, S>(a, f, st);
}

cslsm_status run_phases(const TvSlices &s, const PhaseShape &f, float *pbuf, cudaStream_t st)
{
    const size_t esz = s.storage == CSLSM_STORE_FP32 ? 4 : 2;
    TvPhase a{};
    a.w = s.w;
    a.u = s.u;
    a.d = s.d;
    a.H = s.H;
    a.W = s.W;
    a.Z = s.Z;
    a.n0 = s.n0;
    a.nslices = s.nslices;
    a.hh = f.hh;
    a.hc = f.hc;
    a.TH = f.TH;
    a.TW = f.TW;
    a.tx = f.tx;
    a.rho = s.rho;
    a.gamma = s.Z > 1 ? s.gamma : 0.f;
    a.inv_rho2g = 1.f / (s.rho + 2.f * a.gamma);
    a.theta = s.theta;
    a.inv_theta = 1.f / s.theta;
    a.tau = s.tau;
    a.pair = s.W % 2 == 0 && ((uintptr_t)s.w | (uintptr_t)s.u | (uintptr_t)s.d) % (2 * esz) == 0;
    a.stop = s.stop;
    const size_t half = 2ull * s.nslices * s.H * s.W;
    for (int t = 0, q = 0; t < s.T; t += f.k, q ^= 1) {
        a.ns = std::min(f.k, s.T - t);
        a.pout = t + a.ns < s.T ? pbuf + q * half : nullptr;
        cslsm_status e;
        if (s.storage == CSLSM_STORE_BF16) e = launch_phase_typed<__nv_bfloat16>(a, f, st);
        else if (s.storage == CSLSM_STORE_FP16) e = launch_phase_typed<__half>(a, f, st);
        else e = launch_phase_typed<float>(a, f, st);
        if (e) return e;
        a.pin = a.pout;
    }
    return CSLSM_OK;
}

}  // namespace

int tv_max_steps_per_launch() { return kMaxSteps; }

cslsm_status tv_query_shape(int H, int W, int T, int nslices, int *out4)
{
    int dev = 0, sms = 0;
    cslsm_status e = device_info(dev, sms);
    if (e) return e;
    TvLaunch a{};
    a.H = H;
    a.W = W;
    a.T = T;
    a.nslices = nslices;
    Shape sh{};
    {
        std::lock_guard<std::mutex> lk(g_mu);
        if (g_mode == 1) {
            auto it = g_tuned.find(Key{dev, H, W, T, nslices});
            if (it != g_tuned.end()) {
                sh = it->second;
                out4[0] = sh.v;
                out4[1] = sh.TH;
                out4[2] = sh.TW;
                out4[3] = sh.RH;
                return CSLSM_OK;
            }
        }
    }
    if ((e = choose_shape(a, dev, sms, nullptr, false, sh))) return e;
    out4[0] = sh.v;
    out4[1] = sh.TH;
    out4[2] = sh.TW;
    out4[3] = sh.RH;
    return CSLSM_OK;
}

bool tv_phases_fit(int H, int W, int nslices)
{
    return nslices <= kPhaseMaxSlices && 4ull * nslices * H * W <= kPhaseMaxFloats;
}

int tv_get_mode()
{
    std::lock_guard<std::mutex> lk(g_mu);
    return g_mode;
}

void tv_set_mode(int mode)
{
    std::lock_guard<std::mutex> lk(g_mu);
    g_mode = mode;
    if (mode != 1) g_tuned.clear();
}

size_t tv_pbuf_floats(int H, int W, int T, int nslices)
{
    const size_t all = 4ull * nslices * H * W;
    if (T > kMaxSteps) return all;
    int dev = 0, sms = 0;
    if (tv_get_mode() > 1 || T < 1 || !tv_phases_fit(H, W, nslices) ||
        device_info(dev, sms) != CSLSM_OK)
        return 0;
    return phase_best(H, W, T, nslices, sms).P > 1 ? all : 0;
}

cslsm_status tv_prox_slices(const TvSlices &s, float *pbuf, size_t pbuf_floats, cudaStream_t st)
{
    int dev = 0, sms = 0;
    cslsm_status e = device_info(dev, sms);
    if (e) return e;
    if (s.theta > 0.f && s.T >= 1 && tv_get_mode() <= 1 && s.nslices <= kPhaseMaxSlices) {
        const PhaseShape f = phase_best(s.H, s.W, s.T, s.nslices, sms);
        const size_t need = f.P > 1 ? 4ull * s.nslices * s.H * s.W : 0;
        if (f.rpw && need <= pbuf_floats) return run_phases(s, f, pbuf, st);
    }
    TvLaunch a{};
    a.storage = s.storage;
    a.stop = s.stop;
    a.w = s.w;
    a.u = s.u;
    a.d = s.d;
    a.H = s.H;
    a.W = s.W;
    a.Z = s.Z;
    a.n0 = s.n0;
    a.nslices = s.nslices;
    a.rho = s.rho;
    a.gamma = s.Z > 1 ? s.gamma : 0.f;
    a.inv_rho2g = 1.f / (s.rho + 2.f * a.gamma);
    a.theta = s.theta;
    a.inv_theta = s.theta > 0.f ? 1.f / s.theta : 0.f;
    a.tau = s.tau;
    const int T = s.theta > 0.f ? s.T : 0;  // zero weight: the prox is the identity
    if (T <= kMaxSteps) {
        a.T = T;
        a.write_final = 1;
        Shape sh{};
        if ((e = choose_shape(a, dev, sms, st, true, sh))) return e;
        return launch_tile(a, sh, st);
    }
    if (!pbuf || pbuf_floats < 4ull * s.nslices * s.H * s.W) {
        set_error("TV prox with %d steps needs the dual buffers", T);
        return CSLSM_ERR_INVALID_ARG;
    }
    const int nch = (T + kMaxSteps - 1) / kMaxSteps;
    const size_t half = 2ull * s.nslices * s.H * s.W;
    const float *pin = nullptr;
    int done = 0;
    for (int c = 0; c < nch; ++c) {
        const int steps = (T - done) / (nch - c);
        a.T = steps;
        a.pin = pin;
        a.write_final = (c == nch - 1);
        a.pout = a.write_final ? nullptr : pbuf + (c % 2) * half;
        Shape sh{};
        if ((e = choose_shape(a, dev, sms, st, false, sh))) return e;
        e = launch_tile(a, sh, st);
        if (e) return e;
        pin = a.pout;
        done += steps;
    }
    return CSLSM_OK;
}

}  // namespace cslsm
