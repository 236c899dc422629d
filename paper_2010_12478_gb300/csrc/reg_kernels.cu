// Device kernels of libreg: the registration operator.
//
// Design (GB300, sm_103a):
//   * One operator application (A or B, Sec. 2.3.1-2.3.2) runs start to finish
//     inside ONE thread-block cluster: every level, every gradient-flow
//     iteration and every Armijo trial.  The C CTAs of the cluster split the
//     rows of each pyramid level; their partial sums meet through distributed
//     shared memory, so an iteration costs two exchanges within the cluster (the
//     rigid model: one) and never a kernel launch or a grid-wide synchronisation.
//   * Per pixel the work is FP32 (warp, sample, derivative, moment products).
//     Sums are accumulated per thread in FP32 over runs of 8 pixels, then carried
//     as float-float pairs (error-free transformations on the FP32 pipes: GB300's
//     FP64 rate is a small fraction of FP32) through the warp and CTA stages, and
//     in FP64 across the cluster.  Reduction order is fixed, so results are bitwise
//     reproducible for a given cluster size.
//   * The step controller (NCC from the moments, gradient, Armijo test, step
//     size, stop rules) is FP64 and runs on one thread (the rigid model: one
//     warp) of every CTA of the cluster on identical totals, so all CTAs take
//     identical decisions.
//   * Images are read through the read-only path; the nonrigid model's control
//     values live in shared memory.
#include <cooperative_groups.h>

#include <algorithm>
#include <cmath>
#include <cstdlib>
#include <cstring>

#include "reg_internal.h"
#include "reg_dev.cuh"
#include "reg_f2.cuh"

namespace cg = cooperative_groups;

namespace reg {

constexpr int kWarps = kThreads / 32;
constexpr int kNM = 16;        // sums per reduction at most
constexpr int kMaxCluster = 16; // CTAs per operator at most (non-portable cluster size)

// ------------------------------------------------------------------ shared state
// Step-controller state, used by thread 0 (rigid: warp 0) of each CTA only: kept in shared memory so it
// does not occupy registers of every thread.  All of it is FP64.  An FP64 instruction, conversions among them,
// takes 64 cycles of its warp on this GPU however many lanes take part, a compare 105, an FP32 one 4: the
// controllers are written for few FP64 instructions.
struct LevelSums {
    double P, invP, sr, Srr;       // pixels; sum of the reference's shifted samples; S'_RR
    double gam;                    // scale of the reference in the difference e = t - gam r
    double least;                  // a centred sum of squares below this is a constant image
};

struct RigidCtl {
    LevelSums ls;
    double th[3], tt[3], d[3];
    double E, slope, m0, inv_m0;
    double accept, rel;            // a trial is accepted up to the first energy, and ends the level from the second
    double tolg2;  // the level's stop tolerance (tol_grad, times tol_coarse above the finest level), squared
    double dp[3];                  // direction of the last accepted step
    double tau, tau_acc;           // length of the trial step, and of the last accepted one
    int nrej, iters, evals, stop, rejects, have_prev;
};

struct FieldCtl {
    LevelSums ls;
    double E, ss, invNc, half_lam; // ss: sum_j m_j |d_j|^2; half_lam: lambda / (2 P)
    double accept, rel;            // a trial is accepted up to the first energy, and ends the level from the second
    double Eold, ss_old;           // before the last accepted step, for its quadratic rule
    double tolss;  // the level's stop tolerance (tol_grad, times tol_coarse above the finest level), squared, times Nc
    double tau, tau_acc;           // length of the trial step, and of the last accepted one as it was taken (FP32)
    int nrej, iters, evals, stop, rejects, have_prev;
};

// x >= 0, false for a NaN, from the bits.
__device__ __forceinline__ bool nonneg(double x)
{
    return (unsigned)__double2hiint(x) <= 0x7ff00000u;
}

// x >= y for y >= 0, false for a NaN, from the bits (those of non-negative values order as integers).
__device__ __forceinline__ bool at_least(double x, double y)
{
    return __double_as_longlong(x) >= __double_as_longlong(y) && nonneg(x);
}

// x < y for a finite x and y > 0, false for a NaN of either sign, from the bits.
__device__ __forceinline__ bool below(double x, double y)
{
    return __double_as_longlong(x) < __double_as_longlong(y) && ((unsigned)__double2hiint(x) & 0x7fffffffu) < 0x7ff00000u;
}

// First trial of a line search after an accepted step (Barzilai and Borwein, "Two-point step size
// gradient methods", 1988, their second step): tau = tau_acc <d_prev, d_prev - d> / |d_prev - d|^2
// in the flow's metric, given num = <d_prev, d_prev - d> and den = |d_prev - d|^2; false without
// positive curvature.  The ratio needs no more than FP32 relative precision.
__device__ __forceinline__ bool bb_tau(double tau_acc, double num, double den, double &tau)
{
    if (!(num > 0.0 && den > 0.0)) return false;
    tau = tau_acc * num * (double)__frcp_rn((float)den);
    return true;
}

struct Smem {
    float2 warp[kWarps][kNM];   // per-warp (hi, lo) partials
    double part[2][kMaxCluster][kNM];   // every CTA's partials, pushed here by each CTA
    double tot[kNM];            // cluster totals
    unsigned wmax[kWarps], pmax[2][kMaxCluster];   // bits of the per-warp and per-CTA maxima
    unsigned long long xbar[2]; // mbarriers of the exchanges, used in turn
    float tmax;
    float pm[16];               // pass parameters broadcast by thread 0
    int action;
    int idata[4];
    PassGeom geom;              // of the level
    long long wait_ns;          // limit of an exchange's wait
    int fail;                   // an exchange's wait ran out: kDevWaitTimeout
    int mute;                   // sends nothing (Params::mute)
    union {
        RigidCtl rctl;
        FieldCtl fctl;
    };
};

// ------------------------------------------------------------------ exchanges within a cluster
// CTAs of a cluster hand each other values by asynchronous stores into the receiver's shared memory
// that count down bytes on an mbarrier there (st.async), and a receiver waits for the bytes it is due.
// An exchange is numbered: number n uses barrier and buffers n mod 2.  A CTA sends for n + 2 only after
// completing n + 1, to which every peer contributes after completing n, so nothing of n + 2 meets
// anything of n.  A cluster barrier here takes about 2,000 cycles (its release and acquire are fences over
// global memory), and its acquire drops the SM's L1 lines, so every pass fetched its pixels from L2
// again (331 cycles a load instead of 75); an exchange takes 500, and comm_wait's acquire some more.
struct Comm {
    unsigned n;   // number of the next exchange
};

__device__ __forceinline__ uint32_t smem_addr(const void *p)
{
    return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ uint32_t peer_addr(const void *p, int rank)
{
    uint32_t r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(smem_addr(p)), "r"(rank));
    return r;
}

// Eight (four) bytes to *p in the shared memory of CTA `rank`, counted on its barrier `bar`.
__device__ __forceinline__ void send8(const void *p, const unsigned long long *bar, int rank, unsigned long long v)
{
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.b64 [%0], %1, [%2];" ::"r"(peer_addr(p, rank)),
                 "l"(v), "r"(peer_addr(bar, rank))
                 : "memory");
}

__device__ __forceinline__ void send8(const void *p, const unsigned long long *bar, int rank, float2 v)
{
    send8(p, bar, rank, (unsigned long long)__float_as_uint(v.x) | ((unsigned long long)__float_as_uint(v.y) << 32));
}

__device__ __forceinline__ void send4(const void *p, const unsigned long long *bar, int rank, unsigned v)
{
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.b32 [%0], %1, [%2];" ::"r"(peer_addr(p, rank)),
                 "r"(v), "r"(peer_addr(bar, rank))
                 : "memory");
}

// One thread, before the cluster's first exchange (a cluster barrier follows).
__device__ __forceinline__ void comm_init(Smem &sm, const Params &p, const cg::cluster_group &cl)
{
    for (int i = 0; i < 2; ++i)
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(&sm.xbar[i])) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    sm.wait_ns = p.wait_ns;
    sm.fail = 0;
    sm.mute = p.mute && cl.block_rank() + 1 == cl.num_blocks();
}

// A CTA that has given up neither waits nor sends in any later exchange: a peer that lacks its part gives up
// too, instead of taking a later one for it, and no barrier gets an arrival beyond the one of its phase.
// The same in every thread of a CTA between two barriers.
__device__ __forceinline__ bool comm_quiet(const Smem &sm)
{
    return sm.fail != 0 || sm.mute != 0;
}

// One thread: this CTA is due `bytes` in exchange n.
__device__ __forceinline__ void comm_expect(Smem &sm, unsigned n, unsigned bytes)
{
    if (sm.fail != 0) return;
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(&sm.xbar[n & 1])), "r"(bytes)
                 : "memory");
}

// Wait until exchange n has brought what is due; the peers run side by side with this CTA, so it ends.  After
// sm.wait_ns of waiting it gives up: sm.fail, which the operator's status and the launch's status word report.
// The time between two looks at the clock counts for kWaitStep at most, so a process that was suspended does not
// give up on what is on its way.
// The wait acquires at cluster scope, as it orders the peers' stores before the reads that follow (a CTA's other
// threads, by the barrier after it); at its default scope, its own CTA, the memory model orders nothing of a
// peer's.  It costs 1.6 % over the timed calls (a rigid scan of 24 frames 848 -> 918 us, a pair of 512x512 276 ->
// 280, scans of hundreds of frames nothing).
constexpr unsigned long long kWaitStep = 50000000ULL;
__device__ __forceinline__ void comm_wait(Smem &sm, unsigned n)
{
    const uint32_t bar = smem_addr(&sm.xbar[n & 1]), parity = (n >> 1) & 1;
    unsigned long long last = 0, spent = 0;
    for (unsigned it = 0; *(volatile int *)&sm.fail == 0; ++it) {
        uint32_t done;
        asm volatile("{\n .reg .pred p;\n mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
                     : "=r"(done)
                     : "r"(bar), "r"(parity)
                     : "memory");
        if (done) return;
        if ((it & 15) == 15) {
            unsigned long long t;
            asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
            if (last != 0) spent += min(t - last, kWaitStep);
            last = t;
            if (spent >= (unsigned long long)sm.wait_ns) *(volatile int *)&sm.fail = kDevWaitTimeout;
        }
    }
}

// Reduce NM per-thread float-float sums over the cluster into sm.tot, in a fixed order, and with MAXV
// the largest of a non-negative value into sm.tmax, by one exchange.  Within a warp the sums are exchanged
// by halves, so a lane carries one of them after log2 steps (9 pair additions for 8 sums instead of 40);
// the warps', then the CTAs' partials of a sum are shared out over the lanes and folded the same way.
// Every CTA sends its partials to every CTA, which adds the same values in the same order: identical
// totals.  `push` is called by every thread after a barrier of the CTA with the exchange's number, to
// send more under it; `due`: bytes of such sends that this CTA gets.
struct NoPush {
    __device__ void operator()(unsigned) const {}
};
template <int NM, bool MAXV, typename Push = NoPush>
__device__ __forceinline__ void cluster_reduce(const float (&hi)[NM], const float (&lo)[NM], float mx, Smem &sm,
                                               Comm &comm, const cg::cluster_group &cl, unsigned due = 0,
                                               Push push = Push())
{
    static_assert(NM <= kNM && kWarps == 8, "reduction slots");
    constexpr int kLog = NM <= 8 ? 3 : 4, N2 = 1 << kLog, kParts = 32 / N2;   // lanes that share a sum
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const bool quiet = comm_quiet(sm);   // before this exchange's wait
    float h[N2], l[N2];
#pragma unroll
    for (int m = 0; m < N2; ++m) { h[m] = m < NM ? hi[m] : 0.f; l[m] = m < NM ? lo[m] : 0.f; }
#pragma unroll
    for (int o = 16, n = N2 / 2; o >= 1; o >>= 1, n >>= 1) {
        if (n >= 1) {
            const bool up = lane & o;
#pragma unroll
            for (int m = 0; m < n; ++m) {
                const float h2 = __shfl_xor_sync(0xffffffffu, up ? h[m] : h[m + n], o);
                const float l2 = __shfl_xor_sync(0xffffffffu, up ? l[m] : l[m + n], o);
                h[m] = up ? h[m + n] : h[m];
                l[m] = up ? l[m + n] : l[m];
                ff_add(h[m], l[m], h2, l2);
            }
        } else {
            const float h2 = __shfl_xor_sync(0xffffffffu, h[0], o), l2 = __shfl_xor_sync(0xffffffffu, l[0], o);
            ff_add(h[0], l[0], h2, l2);
        }
    }
    if (lane % kParts == 0) sm.warp[w][lane / kParts] = make_float2(h[0], l[0]);
    if constexpr (MAXV) {
        const unsigned m = __reduce_max_sync(0xffffffffu, __float_as_uint(mx));   // non-negative: bits order as values
        if (lane == 0) sm.wmax[w] = m;
    }
    __syncthreads();
    const int C = cl.num_blocks(), me = cl.block_rank();
    const int m = lane % N2, q = lane / N2;   // warp 0: lane's sum, and which share of its parts
    const unsigned n = comm.n++, b = n & 1;
    const unsigned long long *bar = &sm.xbar[b];
    if (w == 0) {
        if (lane == 0) comm_expect(sm, n, (unsigned)C * (NM * 8 + (MAXV ? 4 : 0)) + due);
        float2 v = sm.warp[q][m];
#pragma unroll
        for (int k = q + kParts; k < kWarps; k += kParts) ff_add(v.x, v.y, sm.warp[k][m].x, sm.warp[k][m].y);
#pragma unroll
        for (int o = N2; o < 32; o <<= 1) {
            const float h2 = __shfl_xor_sync(0xffffffffu, v.x, o), l2 = __shfl_xor_sync(0xffffffffu, v.y, o);
            ff_add(v.x, v.y, h2, l2);
        }
        const unsigned long long t = __double_as_longlong((double)v.x + (double)v.y);
        if (m < NM && !quiet)
            for (int r = q; r < C; r += kParts) send8(&sm.part[b][me][m], bar, r, t);
    } else if (MAXV && w == 1) {
        const unsigned v = __reduce_max_sync(0xffffffffu, lane < kWarps ? sm.wmax[lane] : 0u);
        if (lane < C && !quiet) send4(&sm.pmax[b][me], bar, lane, v);
    }
    if (!quiet) push(n);
    if (w == 0) {
        comm_wait(sm, n);
        double s = q < C && m < NM ? sm.part[b][q][m] : 0.0;
        for (int r = q + kParts; r < C; r += kParts) s = __dadd_rn(s, m < NM ? sm.part[b][r][m] : 0.0);
#pragma unroll
        for (int o = N2; o < 32; o <<= 1) s = __dadd_rn(s, __shfl_xor_sync(0xffffffffu, s, o));
        if (lane < N2) sm.tot[m] = s;
        if constexpr (MAXV) {
            const unsigned v = __reduce_max_sync(0xffffffffu, lane < C ? sm.pmax[b][lane] : 0u);
            if (lane == 0) sm.tmax = __uint_as_float(v);
        }
    }
    __syncthreads();
}

// ------------------------------------------------------------------ NCC (FP64)
struct Ncc {
    double e;                  // 1 - NCC
    double a, u;               // 1 / sqrt(S'_RR S'_TT), gam S'_RE + S'_EE
    double Srt, Stt, ebar;     // S'_RT, S'_TT, mean of e
};

// NCC and what its gradient follows from, from the shifted sums: of r (LevelSums) and of the difference
// e = t - gam r: sum e, sum e^2, sum r e.  Each image is shifted by its own mean, and gam is the ratio of their
// standard deviations (level_gain), so e is small wherever the images match up to the gain and offset that NCC
// does not see.  With S'_RT = gam S'_RR + S'_RE and S'_TT = gam S'_RT + u, u = gam S'_RE + S'_EE, the rounding of
// the FP32 sums enters 1 - NCC, about (S'_EE - S'_RE^2 / S'_RR) / (2 S'_TT), relative to its own size; sums of t^2
// and r t, or of t - r at another gain or offset, enter it relative to 1.  Restated on the host (512x512
// lattices and noise, 1 - NCC from 7e-6 to 1): off by 1e-13 to 1e-8 at any gain and offset; t - r with one shift
// 3e-13 to 1e-8 at equal ones, but 1e-7 at gains of 3 and 1/5 and 1e-4 at an offset of 100 times the contrast; sums of t^2 and
// r t with every product's rounding kept 1e-9 to 1e-8, 2e-6 and 1e-5.  A constant image has E = 1 and no gradient.
__device__ __forceinline__ Ncc ncc_terms(const LevelSums &L, double se, double see, double sre)
{
    Ncc o;
    o.ebar = __dmul_rn(se, L.invP);
    const double See = __fma_rn(-se, o.ebar, see), Sre = __fma_rn(-L.sr, o.ebar, sre);
    o.Srt = __fma_rn(L.gam, L.Srr, Sre);
    o.u = __fma_rn(L.gam, Sre, See);
    o.Stt = __fma_rn(L.gam, o.Srt, o.u);
    o.a = rsqrt(__dmul_rn(L.Srr, o.Stt));
    o.e = __fma_rn(-o.Srt, o.a, 1.0);
    // e = 0 everywhere (T o phi equals R up to gain and offset: identical inputs) is exactly NCC = 1
    if ((__double_as_longlong(Sre) | __double_as_longlong(See)) << 1 == 0) o.e = 0.0;
    // a constant template has no deviation at all (gam 0), whatever its samples between the pixels round to
    if (below(L.Srr, L.least) || below(o.Stt, L.least) || __double_as_longlong(L.gam) == 0) {
        o.e = 1.0; o.a = 0.0;
    }
    return o;
}

// A level's constants, and the reference's part of its sums (known after the first pass).
__device__ __forceinline__ void set_level(LevelSums &L, int W, int H, float gam)
{
    L.P = (double)W * (double)H;
    L.gam = gam;
    L.invP = 1.0 / L.P;
    L.least = 1e-12 * L.P;
}
__device__ __forceinline__ void set_reference(LevelSums &L, double sr, double srr)
{
    const double rbar = __dmul_rn(sr, L.invP);
    L.sr = sr;
    L.Srr = __fma_rn(-sr, rbar, srr);
}

// ------------------------------------------------------------------ level access
struct Lvl {
    const void *R, *T;
    int W, H, Rp, Tp;
    float cR, cT;   // shift constants: the levels' means
    float gam;      // level_gain
};

__device__ __forceinline__ void strip_rows(int H, int rank, int C, int &r0, int &r1)
{
    int per = (H + C - 1) / C;
    r0 = min(H, rank * per);
    r1 = min(H, r0 + per);
}

constexpr int kFast = 8;   // pixels of a thread in one FP32 run before the float-float fold
// Bilinear sample of T (storage S, pitch Tp) at p = (xi + vx, yi + vy) with clamp-to-edge,
// where (xi, yi) is an integer pixel and (vx, vy) a small FP32 offset.  Splitting the
// position keeps the FP32 fractional part exact to the precision of the offset, not
// of the absolute coordinate.  Cell choice and clamping follow floor(p) clamped to
// [0, W-2]; the derivative along a clamped axis (p < 0 or p > W-1) is 0.
template <typename S>
__device__ __forceinline__ float sample_at(const S *T, int W, int H, int Tp, int xi, int yi, float vx, float vy,
                                           float &dtx, float &dty)
{
    vx = fminf(fmaxf(vx, -1.0e6f), 1.0e6f);   // also maps NaN into range: every access stays in bounds
    vy = fminf(fmaxf(vy, -1.0e6f), 1.0e6f);
    const float flx = floorf(vx), fly = floorf(vy);
    int x = xi + (int)flx, y = yi + (int)fly;
    float fx = vx - flx, fy = vy - fly;
    bool clx = false, cly = false;
    if (x < 0) { x = 0; fx = 0.f; clx = true; }
    else if (x > W - 2) { clx = (x > W - 1) || (fx > 0.f); x = W - 2; fx = 1.f; }
    if (y < 0) { y = 0; fy = 0.f; cly = true; }
    else if (y > H - 2) { cly = (y > H - 1) || (fy > 0.f); y = H - 2; fy = 1.f; }
    const S *row = T + (size_t)y * Tp + x;
    float t00 = ldS<S>(row), t01 = ldS<S>(row + 1);
    float t10 = ldS<S>(row + Tp), t11 = ldS<S>(row + Tp + 1);
    float gx = 1.f - fx, gy = 1.f - fy;
    float top = fmaf(fx, t01, gx * t00);
    float bot = fmaf(fx, t11, gx * t10);
    dtx = clx ? 0.f : fmaf(fy, t11 - t10, gy * (t01 - t00));
    dty = cly ? 0.f : (bot - top);
    return fmaf(fy, bot, gy * top);
}

// x rounded to the nearest integer by adding and subtracting 1.5 2^23: the sum's low bits are the
// integer (kRoundBits + n), with no conversion instruction.  Beyond 2^22 the bits are no longer the
// integer, but they are far above or below every pixel, and so is the position.
constexpr float kRound = 12582912.f;
constexpr unsigned kRoundBits = 0x4B400000u;

// ================================================================== rigid
// One pass over a level's rows [r0, r1) at (cos(alpha) - 1, sin(alpha), translation) gives the moments
// of the energy and the sums the gradient follows from: with the shifted samples t = T(phi(x)) - cT,
// r = R(x) - cR, e = t - gam r, dE/dTw = b e + c r + kappa as in the nonrigid pass, and g_k =
// grad T(phi(x)) . dphi/dtheta_k, k = alpha, Gx, Gy.  Sums in sm.tot: 0 sum e, 1 sum e^2,
// 2 sum r e, with START (a level's first pass) 3 sum r, 4 sum r^2; 5 + k sum e g_k; 8 + k sum r g_k;
// 11 + k sum g_k.
//
// Two columns a lane in packed steps, as in the nonrigid pass: a warp's task is 64 columns over a
// segment of rows, and in a straight run (the cell of every column's sample moves down by one row per
// row) a row loads one tap row and keeps the other.  In a run a column beyond the left or right edge
// keeps its clamped cell; runs that reach the top or bottom edge go row by row through sample_at.
constexpr int kRigidSums = 14, kRigidRows = 4;   // rows whose loads are in flight together
template <typename S, bool START>
__device__ void rigid_pass(const Lvl &L, int r0, int r1, const float *pm, Smem &sm, Comm &comm,
                           const cg::cluster_group &cl)
{
    constexpr int NS = START ? 5 : 3;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // pm: cos(alpha) - 1, sin(alpha), fractional translation (x, y), integer translation (x, y)
    const float cm1 = pm[0], sa = pm[1], gfx = pm[2], gfy = pm[3], ca = 1.f + cm1;
    const int gix = (int)pm[4], giy = (int)pm[5];
    const float cx = 0.5f * (float)(L.W - 1), cy = 0.5f * (float)(L.H - 1);
    const S *R = (const S *)L.R, *T = (const S *)L.T;
    const float2 ncR = f2(-L.cR), ncT = f2(-L.cT), ngam = f2(-L.gam), one = f2(1.f);
    float2 mh[NS], ml[NS], m[NS];   // moments: float-float sums and the current run, per column
    float gh[9], gl[9];             // gradient sums: float-float, and the current run
    float2 g[9];
#pragma unroll
    for (int i = 0; i < NS; ++i) mh[i] = ml[i] = m[i] = f2(0.f);
#pragma unroll
    for (int i = 0; i < 9; ++i) { gh[i] = gl[i] = 0.f; g[i] = f2(0.f); }
    // rows split so that the warps' tasks even out: the least rounds x (rows + the window's first row)
    const int strips = (L.W + 63) / 64, rows = r1 - r0;
    int nseg = 1, least = 0x7fffffff;
    for (int k = 1; k <= 8; k *= 2) {
        const int cost = (strips * k + kWarps - 1) / kWarps * ((rows + k - 1) / k + 2);
        if (cost < least) { least = cost; nseg = k; }
    }
    const int per = (rows + nseg - 1) / nseg;
    for (int task = warp; task < strips * nseg; task += kWarps) {
        const int seg = task / strips, x0 = 64 * (task - seg * strips);
        int y = r0 + seg * per;
        const int ye = min(r1, y + per);
        const bool acta = x0 + lane < L.W, actb = x0 + 32 + lane < L.W;
        const int xa = acta ? x0 + lane : x0, xb = actb ? x0 + 32 + lane : x0;   // an idle column counts for nothing
        const float2 xc = make_float2((float)xa - cx, (float)xb - cx);
        auto flush = [&]() {
#pragma unroll
            for (int i = 0; i < NS; ++i) {
                ff_acc2(mh[i], ml[i], make_float2(acta ? m[i].x : 0.f, actb ? m[i].y : 0.f));
                m[i] = f2(0.f);
            }
#pragma unroll
            for (int i = 0; i < 9; ++i) {
                ff_acc(gh[i], gl[i], (acta ? g[i].x : 0.f) + (actb ? g[i].y : 0.f));
                g[i] = f2(0.f);
            }
        };
        // displacement without the integer translation at row y (small, so FP32 keeps ~1e-7 relative)
        auto shift = [&](int row, float2 &vx, float2 &vy, float &yc) {
            yc = (float)row - cy;
            vx = __ffma2_rn(f2(cm1), xc, f2(fmaf(-sa, yc, gfx)));
            vy = __ffma2_rn(f2(sa), xc, f2(fmaf(cm1, yc, gfy)));
        };
        auto pixel = [&](float2 tw, float2 dx, float2 dy, float2 rv, float yc) {
            const float2 r = __fadd2_rn(rv, ncR), e = __ffma2_rn(ngam, r, __fadd2_rn(tw, ncT));
            m[0] = __fadd2_rn(m[0], e);
            m[1] = __ffma2_rn(e, e, m[1]);
            m[2] = __ffma2_rn(r, e, m[2]);
            if constexpr (START) {
                m[3] = __fadd2_rn(m[3], r);
                m[4] = __ffma2_rn(r, r, m[4]);
            }
            // dphi/dalpha = Rot'(alpha) (x - c) = (-sa xc - ca yc, ca xc - sa yc)
            const float2 px = __ffma2_rn(f2(-sa), xc, f2(-ca * yc)), py = __ffma2_rn(f2(ca), xc, f2(-sa * yc));
            const float2 q[3] = {__ffma2_rn(dy, py, __fmul2_rn(dx, px)), dx, dy};
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                g[i] = __ffma2_rn(e, q[i], g[i]);
                g[3 + i] = __ffma2_rn(r, q[i], g[3 + i]);
                g[6 + i] = __fadd2_rn(g[6 + i], q[i]);
            }
        };
        while (y < ye) {
            float2 v0x, v0y, v1x, v1y;
            float yc;
            const int n = min(ye - y, kFast);
            shift(y, v0x, v0y, yc);
            shift(y + n - 1, v1x, v1y, yc);
            const float2 m0x = f2add_down(v0x, f2(kRound)), m0y = f2add_down(v0y, f2(kRound));
            const float2 m1x = f2add_down(v1x, f2(kRound)), m1y = f2add_down(v1y, f2(kRound));
            const unsigned diff = (__float_as_uint(m0x.x) ^ __float_as_uint(m1x.x)) | (__float_as_uint(m0x.y) ^ __float_as_uint(m1x.y)) |
                                  (__float_as_uint(m0y.x) ^ __float_as_uint(m1y.x)) | (__float_as_uint(m0y.y) ^ __float_as_uint(m1y.y));
            // the cells of the first row; |displacement| < 2^22, as the rounding needs
            const int ua = xa + gix + (int)(__float_as_uint(m0x.x) - kRoundBits), ub = xb + gix + (int)(__float_as_uint(m0x.y) - kRoundBits);
            const int wa = y + giy + (int)(__float_as_uint(m0y.x) - kRoundBits), wb = y + giy + (int)(__float_as_uint(m0y.y) - kRoundBits);
            const bool near = fabsf(v0x.x) < 4.0e6f && fabsf(v0x.y) < 4.0e6f && fabsf(v0y.x) < 4.0e6f && fabsf(v0y.y) < 4.0e6f;
            const bool ok = diff == 0u && near && wa >= 0 && wa + n <= L.H - 1 && wb >= 0 && wb + n <= L.H - 1;
            const S *pa = R + (ptrdiff_t)y * L.Rp + xa, *pb = R + (ptrdiff_t)y * L.Rp + xb;
            if (__all_sync(0xffffffffu, ok)) {
                const bool edge = __any_sync(0xffffffffu, (unsigned)ua > (unsigned)(L.W - 2) || (unsigned)ub > (unsigned)(L.W - 2));
                const S *qa = T + (ptrdiff_t)wa * L.Tp + min(max(ua, 0), L.W - 2), *qb = T + (ptrdiff_t)wb * L.Tp + min(max(ub, 0), L.W - 2);
                const float2 nx = f2sub(m0x, f2(kRound)), ny = f2sub(m0y, f2(kRound));
                // a tap row's sample and difference; beyond the right edge the last sample, at weight 0
                const bool ra = ua > L.W - 2, rb = ub > L.W - 2;
                auto tap = [&](float2 l, float2 r, float2 &t, float2 &d) {
                    d = f2sub(r, l);
                    t = edge ? make_float2(ra ? r.x : l.x, rb ? r.y : l.y) : l;
                };
                float2 t0, d0;
                tap(make_float2(ldS<S>(qa), ldS<S>(qb)), make_float2(ldS<S>(qa + 1), ldS<S>(qb + 1)), t0, d0);
                for (int k = 0; k < n; k += kRigidRows) {
                    float2 q[kRigidRows][2], r[kRigidRows];
#pragma unroll
                    for (int i = 0; i < kRigidRows; ++i) {
                        if (k + i < n) { qa += L.Tp; qb += L.Tp; }   // the last rows of a short run repeat
                        q[i][0] = make_float2(ldS<S>(qa), ldS<S>(qb));
                        q[i][1] = make_float2(ldS<S>(qa + 1), ldS<S>(qb + 1));
                        r[i] = make_float2(ldS<S>(pa), ldS<S>(pb));
                        if (k + i + 1 < n) { pa += L.Rp; pb += L.Rp; }
                    }
#pragma unroll
                    for (int i = 0; i < kRigidRows; ++i) {
                        if (k + i >= n) break;
                        float2 vx, vy;
                        shift(y + k + i, vx, vy, yc);
                        float2 fx = f2sub(vx, nx), on = one;
                        const float2 fy = f2sub(vy, ny);
                        if (edge) {
                            // beyond an edge: its sample, and no derivative along x (on the last column
                            // itself, fx = 0, the cell's own)
                            on = make_float2(ua < 0 || ua > L.W - 1 || (ua == L.W - 1 && fx.x > 0.f) ? 0.f : 1.f,
                                             ub < 0 || ub > L.W - 1 || (ub == L.W - 1 && fx.y > 0.f) ? 0.f : 1.f);
                            fx = make_float2(ua < 0 || ra ? 0.f : fx.x, ub < 0 || rb ? 0.f : fx.y);
                        }
                        float2 t1, d1;
                        tap(q[i][0], q[i][1], t1, d1);
                        const float2 top = __ffma2_rn(fx, d0, t0), dy = f2sub(__ffma2_rn(fx, d1, t1), top);
                        const float2 dx = __fmul2_rn(on, __ffma2_rn(fy, f2sub(d1, d0), d0));
                        pixel(__ffma2_rn(fy, dy, top), dx, dy, r[i], yc);
                        t0 = t1;
                        d0 = d1;
                    }
                }
            } else {
                for (int k = 0; k < n; ++k) {
                    float2 vx, vy, dx, dy, tw;
                    shift(y + k, vx, vy, yc);
                    tw.x = sample_at<S>(T, L.W, L.H, L.Tp, xa + gix, y + k + giy, vx.x, vy.x, dx.x, dy.x);
                    tw.y = sample_at<S>(T, L.W, L.H, L.Tp, xb + gix, y + k + giy, vx.y, vy.y, dx.y, dy.y);
                    pixel(tw, dx, dy, make_float2(ldS<S>(pa), ldS<S>(pb)), yc);
                    pa += L.Rp; pb += L.Rp;
                }
            }
            flush();
            y += n;
        }
    }
    float hi[kRigidSums], lo[kRigidSums];
#pragma unroll
    for (int i = 0; i < 5; ++i) {
        hi[i] = i < NS ? mh[i].x : 0.f;
        lo[i] = i < NS ? ml[i].x : 0.f;
        if (i < NS) ff_add(hi[i], lo[i], mh[i].y, ml[i].y);
    }
#pragma unroll
    for (int i = 0; i < 9; ++i) { hi[5 + i] = gh[i]; lo[5 + i] = gl[i]; }
    cluster_reduce<kRigidSums, false>(hi, lo, 0.f, sm, comm, cl);
}

enum Action { kActGrad = 0, kActTrial = 1, kActDone = 2 };


// Pass parameters of parameter q's value v, written by lanes 0-2 of a warp: cos(alpha) - 1 (without
// cancellation) and sin(alpha); the fractional and the integer part of Gx and Gy.
__device__ __forceinline__ void rigid_param(double v, int q, int lane, float *pm)
{
    const float vf = (float)v, i = fminf(fmaxf(rintf(vf), -4.0e6f), 4.0e6f);
    const float frac = (float)(v - (double)i);
    float h, ch;
    sincosf(q == 0 ? 0.5f * vf : 0.f, &h, &ch);
    if (lane == 0) {
        pm[0] = -2.f * h * h;
        pm[1] = 2.f * h * ch;
    } else if (lane < 3) {
        pm[1 + lane] = frac;
        pm[3 + lane] = i;
    }
}

// Step-size rule of the line search: Armijo backtracking with safeguarded quadratic
// interpolation (Nocedal and Wright, Numerical Optimization, Sec. 3.5).  tq minimises the
// parabola through E(0) = E, E'(0) = slope and E(tau) = Et; a rejected trial retries at tq
// clamped to [0.1 tau, 0.5 tau], an accepted one starts the next search at tq clamped to
// [0.5 tau, 4 tau]; without positive curvature the rule halves / doubles.
__device__ __forceinline__ double next_tau(double E, double slope, double tau, double Et, bool accepted)
{
    const double st = __dmul_rn(slope, tau), den = Et - E - st;
    if (!(den > 0.0)) return accepted ? 2.0 * tau : 0.5 * tau;
    // a step-size estimate needs no more than FP32 relative precision once den is formed
    const double tq = -st * tau * (double)__frcp_rn((float)(2.0 * den));
    return accepted ? fmin(fmax(tq, 0.5 * tau), 4.0 * tau) : fmin(fmax(tq, 0.1 * tau), 0.5 * tau);
}

// Coefficients of the gradient of 1 - NCC: dE/dTw(x) = b (t - tbar) - a (r - rbar) = b e + c r + kappa with
// b = NCC / S'_TT, c = gam b - a = -a u / S'_TT, kappa = -(b ebar + c rbar); 1 / S'_TT = a^2 S'_RR.  c and kappa are
// exact zeros for identical frames.
struct GradCoef {
    double b, c, kappa;
};
__device__ __forceinline__ GradCoef grad_coef(const LevelSums &L, const Ncc &n)
{
    const double w = __dmul_rn(__dmul_rn(n.a, n.a), __dmul_rn(n.a, L.Srr));
    GradCoef o;
    o.b = __dmul_rn(w, n.Srt);
    o.c = -__dmul_rn(w, n.u);
    o.kappa = -__fma_rn(o.b, n.ebar, __dmul_rn(o.c, __dmul_rn(L.sr, L.invP)));
    return o;
}

// Gradient component q at the point of a pass from its sums and the point's NCC terms.
__device__ __forceinline__ double rigid_gradient(const LevelSums &L, const Ncc &n, const double *tot, int q)
{
    const GradCoef k = grad_coef(L, n);
    return __fma_rn(k.b, tot[5 + q], __fma_rn(k.c, tot[8 + q], __dmul_rn(k.kappa, tot[11 + q])));
}

// v of lanes 0, 1 and 2 added in that order, in every lane.
__device__ __forceinline__ double sum3(double v)
{
    return (__shfl_sync(0xffffffffu, v, 0) + __shfl_sync(0xffffffffu, v, 1)) + __shfl_sync(0xffffffffu, v, 2);
}

// Controller after a pass at a level's start or at a trial point: the energy there, the Armijo test, and
// where the point is taken the stop tests, the direction and the next trial.  Returns the next action
// and writes its parameters.  Same rules as the oracle's level loop.  Run by one warp: lane q < 3 has
// parameter q, every lane the scalars.
__device__ int rigid_step(RigidCtl &k, const Config &cfg, const double *tot, bool start, float *pm)
{
    const int lane = threadIdx.x & 31, q = min(lane, 2);
    if (start) {
        if (lane == 0) set_reference(k.ls, tot[3], tot[4]);
        __syncwarp();
    }
    const Ncc n = ncc_terms(k.ls, tot[0], tot[1], tot[2]);
    const double Et = n.e, Eold = k.E, slope_old = k.slope;
    const double tau_old = k.tau;
    double th = k.th[q], d = k.d[q], E = Et, slope = slope_old, accept = k.accept, rel = k.rel;
    double dp = k.dp[q];
    double tau = tau_old, tau_acc = k.tau_acc;
    int evals = k.evals + (start ? 0 : 1), iters = k.iters, have_prev = k.have_prev, nrej = k.nrej, rejects = k.rejects;
    int stop = -1;
    const bool taken = start || nonneg(accept - Et);
    if (!taken) {
        E = Eold;
        tau = next_tau(Eold, slope_old, tau_old, Et, false);
        rejects += 1;
        nrej += 1;
        if (nrej > cfg.max_rejects) stop = REG_STOP_LS;
    } else {
        if (!start) {
            th = k.tt[q];
            dp = d;
            tau_acc = tau_old;
            have_prev = 1;
            iters += 1;
        }
        if (!start && nonneg(Et - rel)) {
            stop = REG_STOP_REL;
        } else {
            evals += 1;
            const double g = rigid_gradient(k.ls, n, tot, q);
            d = q == 0 ? -g * k.inv_m0 : -g;
            slope = sum3(g * d);
            // |g|_M = sqrt(-slope); the tests compare squares
            if (iters >= cfg.max_iter) stop = REG_STOP_MAXIT;
            else if (!at_least(-slope, k.tolg2)) stop = REG_STOP_GRAD;
            else {
                if (have_prev) {
                    const double y = dp - d, wy = q == 0 ? k.m0 * y : y;
                    if (!bb_tau(tau_acc, sum3(dp * wy), sum3(y * wy), tau)) tau = next_tau(Eold, slope_old, tau_old, Et, true);
                }
                if (tau * tau * -slope > cfg.step_cap * cfg.step_cap) tau = cfg.step_cap / sqrt(-slope);
                nrej = 0;
                rel = cfg.tol_rel_e == 0.0 ? E : E - cfg.tol_rel_e * fabs(E);
            }
        }
    }
    __syncwarp();   // every lane has read the state
    if (stop < 0) {
        const double tt = __fma_rn(tau, d, th);
        accept = __fma_rn(cfg.armijo_c * slope, tau, E);
        if (lane < 3) k.tt[q] = tt;
        rigid_param(tt, q, lane, pm);
    }
    if (lane < 3) { k.th[q] = th; k.d[q] = d; k.dp[q] = dp; }
    if (lane == 0) {
        k.E = E; k.slope = slope; k.accept = accept; k.rel = rel;
        k.tau = tau; k.tau_acc = tau_acc;
        k.nrej = nrej; k.rejects = rejects; k.iters = iters; k.evals = evals; k.have_prev = have_prev;
        if (stop >= 0) k.stop = stop;
    }
    __syncwarp();
    return stop >= 0 ? kActDone : kActTrial;
}

// Scale of a reference of standard deviation sr to a template of st; any value gives the same NCC up to rounding,
// 1 where there is none (a constant reference, samples that are not finite).
__device__ __forceinline__ float level_gain(float sr, float st)
{
    const float g = st / sr;
    return sr >= 1e-6f && g <= 1e30f ? g : 1.f;
}

__device__ __forceinline__ Lvl level_of(const Params &p, int ref, int tmpl, int l)
{
    const LevelDesc &a = p.levels[ref * p.cfg.levels + l];
    const LevelDesc &b = p.levels[tmpl * p.cfg.levels + l];
    Lvl L;
    L.R = a.rptr; L.T = b.ptr; L.W = a.W; L.H = a.H; L.Rp = a.rpitch; L.Tp = b.pitch;
    L.cR = a.mean; L.cT = b.mean; L.gam = level_gain(a.sd, b.sd);
    return L;
}

template <typename S>
__device__ void run_rigid(const Params &p, const OpDesc &op, int op_index, Smem &sm, Comm &comm,
                          const cg::cluster_group &cl)
{
    const int tid = threadIdx.x;
    const int C = cl.num_blocks(), rank = cl.block_rank();
    const Config &cfg = p.cfg;
    RigidCtl &k = sm.rctl;
    if (tid == 0) {
        memset(&k, 0, sizeof(k));
        double th0[3] = {0.0, 0.0, 0.0};
        if (op.left >= 0) {
            // B's initial guess phi_jk o phi_ij in centred coordinates (Sec. 2.3.2)
            // node states come from other clusters: read through L2, never a stale L1 line
            const double *pa = p.node_theta + 3 * op.left, *pb = p.node_theta + 3 * op.right;
            double a[3] = {__ldcg(pa), __ldcg(pa + 1), __ldcg(pa + 2)};
            double b[3] = {__ldcg(pb), __ldcg(pb + 1), __ldcg(pb + 2)};
            float s, c;
            sincosf((float)b[0], &s, &c);
            double cb = c, sb = s;
            th0[0] = a[0] + b[0];
            th0[1] = cb * a[1] - sb * a[2] + b[1];
            th0[2] = sb * a[1] + cb * a[2] + b[2];
        } else if (op.init_node >= 0) {
            const double *pa = p.node_theta + 3 * op.init_node;
            th0[0] = __ldcg(pa); th0[1] = __ldcg(pa + 1); th0[2] = __ldcg(pa + 2);
        }
        k.th[0] = th0[0];
        k.th[1] = ldexp(th0[1], -(cfg.levels - 1));
        k.th[2] = ldexp(th0[2], -(cfg.levels - 1));
    }
    int stops[kMaxLevels], iters[kMaxLevels], evals[kMaxLevels];
    for (int l = cfg.levels - 1; l >= 0; --l) {
        const Lvl L = level_of(p, op.ref, op.tmpl, l);
        int r0, r1;
        strip_rows(L.H, rank, C, r0, r1);
        if (tid == 0) {
            set_level(k.ls, L.W, L.H, L.gam);
            double rho = 0.25 * (L.W + L.H);
            k.m0 = rho * rho;
            k.inv_m0 = 1.0 / k.m0;
            k.tau = cfg.tau0;
            k.have_prev = 0;
            k.iters = 0; k.evals = 0; k.stop = REG_STOP_MAXIT;
            // a coarse level only supplies the next level's initial guess: a looser stop
            const double tolg = cfg.tol_grad * (l > 0 ? cfg.tol_coarse : 1.0);
            k.tolg2 = tolg * tolg;
            sm.action = kActTrial;
        }
        __syncthreads();
        if (tid < 32) rigid_param(k.th[min(tid, 2)], min(tid, 2), tid, sm.pm);
        for (bool start = true;; start = false) {
            __syncthreads();
            if (sm.action == kActDone) break;
            float pm[6];
#pragma unroll
            for (int q = 0; q < 6; ++q) pm[q] = sm.pm[q];
            if (start) rigid_pass<S, true>(L, r0, r1, pm, sm, comm, cl);
            else rigid_pass<S, false>(L, r0, r1, pm, sm, comm, cl);
            if (tid < 32) {
                const int act = rigid_step(k, cfg, sm.tot, start, sm.pm);
                if (tid == 0) sm.action = sm.fail ? (int)kActDone : act;
            }
        }
        if (tid == 0) {
            stops[l] = k.stop; iters[l] = k.iters; evals[l] = k.evals;
            if (l > 0) { k.th[1] *= 2.0; k.th[2] *= 2.0; }
        }
        __syncthreads();
    }
    if (tid == 0 && rank == 0) {
        double *o = p.node_theta + 3 * op.out;
        __stcg(o, k.th[0]); __stcg(o + 1, k.th[1]); __stcg(o + 2, k.th[2]);
        OpStats &st = p.stats[op_index];
        st.i = op.ref;
        st.k = op.tmpl;
        for (int l = 0; l < kMaxLevels; ++l) {
            bool v = l < cfg.levels;
            st.iters[l] = v ? iters[l] : 0;
            st.evals[l] = v ? evals[l] : 0;
            st.stop[l] = v ? stops[l] : 0;
        }
        st.rejects = k.rejects;
        st.status = sm.fail;
        st.energy = k.E;
        st.theta[0] = o[0]; st.theta[1] = o[1]; st.theta[2] = o[2];
    }
}

// ================================================================== nonrigid
// Free-form field: u(x) bilinear in control values c_j on a grid of spacing s
// (finest-level pixels), points (jx s, jy s).  At level l a pixel x sits at
// finest coordinate X = 2^l x + (2^l - 1)/2, and the level works on c in its
// own pixels (c / 2^l).
//
// One pass over a level's pixels gives everything an evaluation needs: the moments of the energy
// and, per control point, the sums from which the gradient follows once the moments are known.
// With dE/dTw = b e + c r + kappa (e = t - gam r and r the shifted samples, ncc_terms; b, c, kappa:
// grad_coef), the gradient of the data term is
//     b sum_x w_j e dT/dp + c sum w_j r dT/dp + kappa sum w_j dT/dp,
// three sums per point and axis that do not depend on the moments.  c is small where the energy is, so the
// split loses no precision to cancellation; identical frames give e = 0, c = 0 and kappa = 0 exactly.  An accepted trial
// (three in four and more) thus costs one pass over the pixels, not one for the energy and one for
// the gradient, and a level starts with one pass, which also gives the Gauss-Newton scalar product.
// The gradient sums of a rejected trial are dropped.  With separate passes a scan of 256 frames of
// 512x512 took 28.4 ms and a pair 1,031 us (8 CTAs per operator); fused, with two packed columns a lane
// and sliding windows, 16.5 ms and 513 us; with the exchanges and emissions below 13.9 ms and 390 us.  What
// bounds the pass is the latency of its loads and of dependent packed steps (40 % issue, 16 warps per SM).
//
// A CTA of the cluster holds the control rows of its own band of cell rows and one row on either
// side, assembles the gradient at its own rows (the first one with the last partial row of the CTA
// above, which sends it), and hands the direction of its edge rows to its neighbours.
// With the whole grid in every CTA, each assembled all of it (13,000 cycles of an iteration's 230,000
// at 512x512, most of one at 128x128) and 26 KB a CTA were taken from the L1 cache.

struct Grid {
    int nx, ny, s;   // points per axis, spacing in finest pixels
};

struct GridLvl {
    int W, H, l;     // level size and index
    float scale_inv; // 1 / s in level-coordinate units: g = (2^l x + off) / s
    float off;       // (2^l - 1) / 2
    float pl;        // 2^l
};

__device__ __forceinline__ GridLvl grid_level(const Grid &G, const Lvl &L, int l)
{
    GridLvl g;
    g.W = L.W; g.H = L.H; g.l = l;
    g.pl = ldexpf(1.f, l);
    g.off = 0.5f * (g.pl - 1.f);
    g.scale_inv = 1.f / (float)G.s;
    return g;
}

// Cell rows of one CTA at most: rank k owns cell rows [k q, (k+1) q).
__host__ __device__ __forceinline__ int band_cells(int gny, int C)
{
    return (gny - 1 + C - 1) / C;
}

// Points j = tid, tid + kThreads, ... of rows of nx points as (row, column): the first without a
// division, and it is the only one of a thread where a band has up to kThreads points.
struct PointIter {
    int i0, x0;
    __device__ __forceinline__ explicit PointIter(int nx)
    {
        i0 = (int)threadIdx.x / nx;
        x0 = (int)threadIdx.x - i0 * nx;
    }
    __device__ __forceinline__ static void at(int nx, int j, int &i, int &x)
    {
        i = j / nx;
        x = j - i * nx;
    }
};

// The rows of a CTA: cell rows [cr0, cr1); control rows [cr0, own1) are its own (the last band
// owns the grid's last row too); rows [h0, h1) are held in shared memory.
struct Band {
    int q, cr0, cr1, own1, h0, h1;
};

__device__ __forceinline__ Band grid_band(const Grid &G, int rank, int C)
{
    const int cells = G.ny - 1;
    Band b;
    b.q = band_cells(G.ny, C);
    b.cr0 = min(cells, rank * b.q);
    b.cr1 = min(cells, b.cr0 + b.q);
    const bool any = b.cr0 < b.cr1;
    b.own1 = any ? (b.cr1 == cells ? G.ny : b.cr1) : b.cr0;
    b.h0 = any ? max(0, b.cr0 - 1) : b.cr0;
    b.h1 = any ? min(G.ny, b.own1 + 1) : b.cr0;
    return b;
}

// a / b for a b < 2^31, r = recip31(b): the integer divisions of a pass's set-up take longer than the rows
// of a small frame.  A quotient's rounding is a / 2^31 at most, below 1 / b.  (With 20 bits a band of 1,205 cell
// rows, which two CTAs hold of a 2 x 2,410 grid, was beyond it.)
__host__ __device__ __forceinline__ unsigned recip31(int b)
{
    return (1u << 31) / (unsigned)b + 1u;
}
__host__ __device__ __forceinline__ int div31(int a, unsigned r)
{
    return (int)(((unsigned long long)(unsigned)a * r) >> 31);
}

constexpr int kSlot = 8;   // floats per slot: (e, r, 1) x (x, y), then dT^2 x (x, y)
// The rule of PassGeom.  On the host, once per launch: made by the kernel, per operator and level, it took
// 16 us of a pair of 128x128 frames.
//
// A column's sums run in FP32 over the rows of a segment's cell row.  `exact` takes pieces of at most 8 rows
// where their slots fit: for a gradient that is a result itself (reg_energy, 512x512), 6.1e-8 of its norm off
// the 64-bit value instead of 6.8e-8 when it was chosen (5.1e-8 to 5.8e-8 now), within a microsecond of a call.
static PassGeom pass_geom(int sl, int ncx, int q, bool over, int room, bool exact)
{
    PassGeom P;
    P.sl = sl;
    P.g = sl < 32 ? 32 / sl < ncx ? 32 / sl : ncx : 1;
    P.chunks = (sl + 31) / 32;
    P.past = sl < 32 ? (ncx + P.g - 1) / P.g : ncx * P.chunks;
    for (const bool walk : {false, true}) {
        P.sch = walk ? 1 : P.chunks;
        P.ns = walk ? ncx : P.past;
        P.nst = P.ns + (over ? 1 : 0);
        P.tasks = walk ? P.nst : (P.nst + 1) / 2;
        P.walk = walk ? (P.chunks + 1) / 2 : 1;
        int least = -1;
        const int most = room / ((P.g + 1) * kSlot) / P.nst;   // segments x control rows that fit
        for (int k = 1; k < 2 * q; k *= 2) {
            const int m = (q + k - 1) / k, nseg = (q + m - 1) / m;
            const int cost = (P.tasks * nseg + kWarps - 1) / kWarps * (P.walk * m * sl + 2 * m + 4);
            if ((least < 0 || cost < least) && nseg * (m + 1) <= most) {
                least = cost;
                P.m = m; P.h = 1; P.ph = sl; P.nseg = nseg;
            }
        }
        for (int h = 2; h <= 8 && sl / h >= 2; h *= 2) {
            const int ph = (sl + h - 1) / h;
            const int cost = (P.tasks * q * h + kWarps - 1) / kWarps * (P.walk * ph + 6);
            if ((least < 0 || cost < least || (exact && P.ph > 8)) && q * h * 2 <= most) {
                least = cost;
                P.m = 1; P.h = h; P.ph = ph; P.nseg = q * h;
            }
        }
        if (least >= 0) break;
        P.m = q; P.h = 1; P.ph = sl; P.nseg = 1;   // the fewest slots: they do not fit here, the host refuses
        if (P.chunks == 1) break;
    }
    P.hlog = P.h == 8 ? 3 : P.h >> 1;
    P.rm = recip31(P.m);
    P.rg = recip31(P.g);
    return P;
}

static size_t slot_floats(const PassGeom &P)
{
    return (size_t)P.nseg * P.nst * (P.m + 1) * (P.g + 1) * kSlot;
}

constexpr int kEmitSums = 6, kEmitRow = 36;   // gradient sums of a column; a row of 32 columns, padded against bank conflicts
constexpr int kEmitFloats = 2 * kEmitSums * kEmitRow;   // a warp's emission: 2 strips' sums

// Dynamic shared memory of the nonrigid kernels, in float2 units: c, d, mt (the held rows; mt the
// flow's scalar product per control point and axis), the sums that the CTA above sends for the first own
// row, the warps' rows of an emission, then the slots.  Two staged halo rows of d lie in the place of the
// emissions: a neighbour sends them after a pass's exchange, to which this CTA contributed behind its last
// emission, and they are read before its next pass.  Without that the 3-row grids of 858 to 892 points a row
// (frames of 28,000 x 50 at a spacing of 32), which grid_dims takes, had no split that fits 16 CTAs; now every
// grid that it takes has one.
// With the H1 product mt is the right-hand side of its solve on the whole grid, and the two work
// grids t and u of the solve lie in the place of the slots, which it has read by then.
struct GridLayout {
    int c, d, mt, halo, above, emits, slots;
};
__host__ __device__ __forceinline__ GridLayout grid_layout(int gnx, int gny, int C, bool h1)
{
    const int q = band_cells(gny, C);
    const int rows = q + 2 < gny ? q + 2 : gny;
    GridLayout g;
    g.c = 0;
    g.d = rows * gnx;
    g.mt = 2 * rows * gnx;
    const int edges = q < gny - 1 ? gnx : 0;   // a band has neighbours
    g.above = g.mt + (h1 ? gny : rows) * gnx;
    g.emits = g.above + kSlot / 2 * edges;
    g.emits += g.emits & 1;
    g.halo = g.emits;
    const int warps = kWarps * kEmitFloats / 2;
    g.slots = g.emits + (warps > 2 * edges ? warps : 2 * edges);
    return g;
}

// Floats that a CTA's shared memory holds as slots beside the rest of the layout and the static part.
constexpr int kMostSmem = 227 * 1024 - (int)sizeof(Smem) - 256;
static int slot_room(const GridLayout &g)
{
    return (kMostSmem - (int)sizeof(float2) * g.slots) / (int)sizeof(float);
}

// ------------------------------------------------------------------ a control row's sums
// The emission of a segment's control row: a lane holds its two columns' sums x (kEmitSums of them per
// strip; 2 with SQ), which every cell's columns add up to for the point on its left, weighted 1 - w, and
// on its right, weighted w (SQ: by the squares).  w grows by dw per column from that of the strip's first
// column, wf, in each cell anew.  The sums go through shared memory: a lane writes its columns, and then
// has a cell's columns of one sum to itself (with cells of 8 or 16 columns; of 32, half of them), four at
// a load: right = wf S + dw K, left = wl S + dw L from S = sum x, K = sum k x and L = sum (n - 1 - k) x,
// wl the last column's 1 - w (S - right has the rounding of S where the left share is small).  Exchanging
// the lanes' values by halves took twice the instructions, a chain of some 1,000 cycles.  With this and
// the level's geometry in shared memory (made per operator and held in registers and local memory before)
// a scan of 256 frames of 512x512 went from 15.4 to 14.4 ms, of 1,024 from 65.1 to 59.9, a pair of
// 741x1003 (BF16) from 571 to 531 us, of 128x128 from 218 to 210.

// A unit's columns: left and right sum; wf: the first column's weight.
template <int COLS, bool SQ>
__device__ __forceinline__ void cell_sums(const float *x, float wf, float dw, float &l, float &r)
{
    float4 a = make_float4(0.f, 0.f, 0.f, 0.f), b = a, c = a;
#pragma unroll
    for (int k = 0; k < COLS; k += 4) {
        const float4 v = *(const float4 *)(x + k);
        if constexpr (SQ) {
            const float w0 = fmaf((float)k, dw, wf), w1 = fmaf((float)(k + 1), dw, wf), w2 = fmaf((float)(k + 2), dw, wf),
                        w3 = fmaf((float)(k + 3), dw, wf);
            a.x = fmaf((1.f - w0) * (1.f - w0), v.x, a.x); b.x = fmaf(w0 * w0, v.x, b.x);
            a.y = fmaf((1.f - w1) * (1.f - w1), v.y, a.y); b.y = fmaf(w1 * w1, v.y, b.y);
            a.z = fmaf((1.f - w2) * (1.f - w2), v.z, a.z); b.z = fmaf(w2 * w2, v.z, b.z);
            a.w = fmaf((1.f - w3) * (1.f - w3), v.w, a.w); b.w = fmaf(w3 * w3, v.w, b.w);
        } else {
            a.x += v.x; b.x = fmaf((float)k, v.x, b.x);       c.x = fmaf((float)(COLS - 1 - k), v.x, c.x);
            a.y += v.y; b.y = fmaf((float)(k + 1), v.y, b.y); c.y = fmaf((float)(COLS - 2 - k), v.y, c.y);
            a.z += v.z; b.z = fmaf((float)(k + 2), v.z, b.z); c.z = fmaf((float)(COLS - 3 - k), v.z, c.z);
            a.w += v.w; b.w = fmaf((float)(k + 3), v.w, b.w); c.w = fmaf((float)(COLS - 4 - k), v.w, c.w);
        }
    }
    l = (a.x + a.y) + (a.z + a.w);
    r = (b.x + b.y) + (b.z + b.w);
    if constexpr (!SQ) {
        const float s = l;
        r = fmaf(wf, s, dw * r);
        l = fmaf(1.f - fmaf((float)(COLS - 1), dw, wf), s, dw * ((c.x + c.y) + (c.z + c.w)));
    }
}

// Cells of 8 or 16 columns, or one of 32 (HALF: by halves of 16).  A point between two cells gets both
// shares in one addition.  x: the warp's rows, sum by sum, strip by strip; slot s0 or s1 (points 0 .. last + 1
// of the strip, slot[p kSlot]; none where last < 0), the same one for two chunks of a cell, which `adds`
// to earlier ones.
template <int COLS, bool HALF, bool SQ>
__device__ __forceinline__ void emit_cells(const float *x, int lane, float2 wf, float dw, int2 last, float *s0, float *s1,
                                           int adds)
{
    constexpr int kSums = SQ ? 2 : kEmitSums, kCells = 32 / COLS;
#pragma unroll
    for (int u0 = 0; u0 < 2 * kSums * kCells; u0 += 32) {
        const int u = min(u0 + lane, 2 * kSums * kCells - 1), cell = u % kCells, row = u / kCells;
        const bool second = row >= kSums, mine = u0 + lane == u;
        const int comp = second ? row - kSums : row, lst = second ? last.y : last.x;
        float w = second ? wf.y : wf.x, l, r;
        if (HALF && cell) w = fmaf((float)COLS, dw, w);
        cell_sums<COLS, SQ>(x + row * kEmitRow + cell * COLS, w, dw, l, r);
        float *p = (second ? s1 : s0) + (SQ ? kEmitSums : 0) + comp;
        if (HALF) {
            l += __shfl_xor_sync(0xffffffffu, l, 1);
            r += __shfl_xor_sync(0xffffffffu, r, 1);
            const bool on = mine && cell == 0 && lst >= 0, same = s0 == s1;
            if (on && !(second && same)) {
                p[0] = adds ? p[0] + l : l;
                p[kSlot] = adds ? p[kSlot] + r : r;
            }
            if (same) {   // chunks of one cell
                __syncwarp();
                if (on && second) {
                    p[0] += l;
                    p[kSlot] += r;
                }
            }
        } else {
            const float left = __shfl_up_sync(0xffffffffu, r, 1);
            if (cell) l += left;
            if (mine && cell <= lst) p[cell * kSlot] = l;
            if (mine && cell == lst) p[(cell + 1) * kSlot] = r;
        }
    }
}

// Cells of any width below 32: a lane has a point, and adds the columns of the cells on both sides.
template <bool SQ>
__device__ __forceinline__ void emit_points(const float *x, int lane, int sl, int cells, float2 wf, float dw, int2 last, float *s0,
                                            float *s1)
{
    constexpr int kSums = SQ ? 2 : kEmitSums;
    const unsigned rp = recip31(cells + 1);
    for (int u = lane; u < 2 * kSums * (cells + 1); u += 32) {
        const int row = div31(u, rp), pt = u - row * (cells + 1);
        const bool second = row >= kSums;
        const int comp = second ? row - kSums : row, lst = second ? last.y : last.x;
        if (pt > lst + 1 || lst < 0) continue;
        const float w0 = second ? wf.y : wf.x, *c = x + row * kEmitRow + pt * sl;
        float v = 0.f;
        if (pt > 0)
            for (int k = 0; k < sl; ++k) {
                const float w = fmaf((float)k, dw, w0);
                v = fmaf(SQ ? w * w : w, c[k - sl], v);
            }
        if (pt <= lst)
            for (int k = 0; k < sl; ++k) {
                const float w = 1.f - fmaf((float)k, dw, w0);
                v = fmaf(SQ ? w * w : w, c[k], v);
            }
        ((second ? s1 : s0) + (SQ ? kEmitSums : 0) + comp)[pt * kSlot] = v;
    }
}

template <bool SQ>
__device__ __forceinline__ void emit_any(int sl, const float *x, int lane, int cells, float2 wf, float dw, int2 last, float *s0,
                                         float *s1, int adds)
{
    if (sl == 16) emit_cells<16, false, SQ>(x, lane, wf, dw, last, s0, s1, 0);
    else if (sl >= 32) emit_cells<16, true, SQ>(x, lane, wf, dw, last, s0, s1, adds);
    else if (sl == 8) emit_cells<8, false, SQ>(x, lane, wf, dw, last, s0, s1, 0);
    else emit_points<SQ>(x, lane, sl, cells, wf, dw, last, s0, s1);
}

// Value and twice the gradient of the B-spline model for two samples (.x and .y) from their 3 x 3
// windows t (rows, then columns) at offsets (tx, ty) in [-1/2, 1/2] from the middle sample.  Along an
// axis the taps' weights (1/2 - t)^2 / 2, 3/4 - t^2, (1/2 + t)^2 / 2 are taken as a polynomial in t,
//     S + t/2 (D1 + t D2),   S = (t0 + t2) / 8 + 3/4 t1,   D1 = t2 - t0,   D2 = t0 - 2 t1 + t2,
// its derivative as (D1 + 2 t D2) / 2: S, D1 and D2 of a tap row serve every window that holds it.
struct TapRow {
    float2 S, D1, D2;
};
__device__ __forceinline__ TapRow tap_row(float2 t0, float2 t1, float2 t2)
{
    const float2 s = __fadd2_rn(t0, t2);
    return TapRow{__ffma2_rn(f2(0.125f), s, __fmul2_rn(f2(0.75f), t1)), f2sub(t2, t0), __ffma2_rn(f2(-2.f), t1, s)};
}
__device__ __forceinline__ float2 bspline2(const TapRow &r0, const TapRow &r1, const TapRow &r2, float2 tx, float2 ty,
                                           float2 &dtx2, float2 &dty2)
{
    const float2 hx = __fmul2_rn(f2(0.5f), tx), hy = __fmul2_rn(f2(0.5f), ty);
    const float2 x2 = __fadd2_rn(tx, tx), y2 = __fadd2_rn(ty, ty);
    const float2 a0 = __ffma2_rn(hx, __ffma2_rn(tx, r0.D2, r0.D1), r0.S), b0 = __ffma2_rn(x2, r0.D2, r0.D1);
    const float2 a1 = __ffma2_rn(hx, __ffma2_rn(tx, r1.D2, r1.D1), r1.S), b1 = __ffma2_rn(x2, r1.D2, r1.D1);
    const float2 a2 = __ffma2_rn(hx, __ffma2_rn(tx, r2.D2, r2.D1), r2.S), b2 = __ffma2_rn(x2, r2.D2, r2.D1);
    const TapRow a = tap_row(a0, a1, a2), b = tap_row(b0, b1, b2);
    dtx2 = __ffma2_rn(hy, __ffma2_rn(ty, b.D2, b.D1), b.S);
    dty2 = __ffma2_rn(y2, a.D2, a.D1);
    return __ffma2_rn(hy, __ffma2_rn(ty, a.D2, a.D1), a.S);
}

constexpr int kRunRows = 16;   // rows of a straight run at most; half of it is tried next

// Sums of control point (cr0 + i, jx) over the slots that one CTA with nr cell rows wrote: entries
// first .. first + N - 1, segment by segment and strip by strip (FF: added in float-float).
template <int N, bool FF = false>
__device__ __forceinline__ void slot_sum(const float *slots, const PassGeom &P, int ncx, int nr, int i, int jx,
                                         int first, float (&o)[N])
{
    const int ga = i > 0 ? div31(i - 1, P.rm) : 0, gb = div31(i < nr ? i : nr - 1, P.rm);
    const int srow = (P.g + 1) * kSlot, sstrip = (P.m + 1) * srow, sseg = P.nst * sstrip;
    float e[N];
#pragma unroll
    for (int k = 0; k < N; ++k) e[k] = 0.f;
    auto add = [&](const float *s) {
#pragma unroll
        for (int k = 0; k < N; k += 2) {
            const float2 v = *(const float2 *)(s + k);
            if constexpr (FF) {
                ff_acc(o[k], e[k], v.x);
                ff_acc(o[k + 1], e[k + 1], v.y);
            } else {
                o[k] += v.x;
                o[k + 1] += v.y;
            }
        }
    };
    const int st = div31(jx, P.rg), pt = jx - st * P.g;
    // the strips that hold the point: where it is the last of one, the first or an inner one of another, and
    // where it lies beside the column past the last cell
    const bool narrow = P.sl < 32, over = P.nst > P.ns && jx >= ncx - 1;
    const bool left = narrow && pt == 0 && jx > 0, own = narrow && st < P.ns;
    for (int grp = ga; grp <= gb; ++grp) {
        const float *p = slots + grp * P.h * sseg + (i - grp * P.m) * srow + first;
        const float *po = p + st * sstrip + pt * kSlot, *pl = po - sstrip + P.g * kSlot;
        const float *pv = p + P.ns * sstrip + (jx - (ncx - 1)) * kSlot;
#pragma unroll 4
        for (int piece = 0; piece < P.h; ++piece) {
            if (left) add(pl);
            if (own) add(po);
            if (!narrow)
                for (int q = 0; q < P.sch; ++q) {
                    if (jx > 0) add(p + ((jx - 1) * P.sch + q) * sstrip + kSlot);
                    if (jx < ncx) add(p + (jx * P.sch + q) * sstrip);
                }
            if (over) add(pv);
            p += sseg; po += sseg; pl += sseg; pv += sseg;
        }
    }
    if constexpr (FF)
#pragma unroll
        for (int k = 0; k < N; ++k) o[k] += e[k];
}

// One pass at c (START: a level's first) or at the trial c + tau d: the moments into sm.tot (e =
// t - gam r: 0 sum e, 1 sum e^2, 2 sum r e, with START 3 sum r, 4 sum r^2; 5: sum over control edges of |dct|^2) and the gradient
// sums into the slots.  The trial values are formed where they are read, fmaf(tau, d_j, c_j), the
// expression an accepted step stores into c.
//
// Two columns a lane, every floating-point step on both in one packed instruction.  Where the sample
// positions of every column of the warp move down by one row per row (a straight run: the rounded
// displacement is constant, as it is over most of a smooth field), the window slides: a row loads one
// tap row and keeps two, R rows' loads in flight together.  Elsewhere each row loads its own window.
// A sum of products takes one rounding per product (fmaf), in runs of at most 8 pixels carried on in
// float-float.
template <typename S, bool START, int R>
__device__ void grid_pass(const Lvl &L, const Grid &G, const GridLvl &GL, const PassGeom &P, const Band &B,
                          const float2 *c, const float2 *d, float tau, float *slots, const float *above, float *emits, const PointIter &pi,
                          Smem &sm, Comm &comm, const cg::cluster_group &cl)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int ncx = G.nx - 1, ncy = G.ny - 1, sl = P.sl;
    const S *Rp = (const S *)L.R, *T = (const S *)L.T;
    const float2 ncR = f2(-L.cR), ncT = f2(-L.cT), ngam = f2(-L.gam), dw = f2(GL.pl * GL.scale_inv);
    float *emit = emits + warp * kEmitFloats;
    auto ct = [&](int row, int col) {   // control value of the point evaluated
        const int j = (row - B.h0) * G.nx + col;
        const float2 a = c[j];
        if constexpr (START) {
            return a;
        } else {
            const float2 b = d[j];
            return make_float2(fmaf(tau, b.x, a.x), fmaf(tau, b.y, a.y));
        }
    };
    constexpr int NM = START ? 5 : 3;
    float2 hi2[NM], lo2[NM], a[NM];
#pragma unroll
    for (int i = 0; i < NM; ++i) hi2[i] = lo2[i] = a[i] = f2(0.f);

    const int kw = sl < 32 ? div31(lane, recip31(sl)) : 0;   // the lane's cell in a strip of whole cells
    for (int seg = 0, pr = warp, cp = 0;;) {
        while (pr >= P.tasks) { pr -= P.tasks; ++seg; }
        if (seg >= P.nseg) break;
        // the task's strips from the first to before the last one
        const bool walk = P.sch < P.chunks, past = walk && pr == P.ns;
        const int strip0 = walk ? pr * P.chunks + 2 * cp : 2 * pr;
        const int strips = walk ? past ? P.past + 1 : (pr + 1) * P.chunks : P.nst, slot0 = walk ? pr : strip0;
        const int adds = cp;
        if (++cp == P.walk || past) { cp = 0; pr += kWarps; }
        const int grp = seg >> P.hlog, piece = seg & (P.h - 1);
        const int ca = B.cr0 + grp * P.m, cb = min(ca + P.m, B.cr1);
        if (ca >= cb) continue;
        // this lane's column of either strip; an idle lane repeats the last column and counts for nothing
        int xc[2], cell[2], last[2];
        float wx[2];
        bool act[2];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int strip = strip0 + u;
            const bool over = strip == P.past;    // the column past the last cell
            const int cell0 = over ? ncx - 1 : sl < 32 ? strip * P.g : P.chunks == 1 ? strip : strip / P.chunks;
            const int c0 = min(cell0, ncx - 1);
            last[u] = over || sl >= 32 ? 0 : min(P.g, ncx - c0) - 1;
            const int xs = over ? ncx * sl : sl < 32 ? c0 * sl : c0 * sl + (strip - cell0 * P.chunks) * 32;
            const int xe = over ? L.W : min(L.W, min(c0 * sl + (last[u] + 1) * sl, xs + 32));
            act[u] = strip < strips && xs + lane < xe && kw <= last[u];
            cell[u] = c0 + min(kw, last[u]);
            xc[u] = min(xs + lane, L.W - 1);
            wx[u] = fminf(fmaf(GL.pl, (float)xc[u], GL.off) * GL.scale_inv, (float)ncx) - (float)cell[u];
            if (!act[u]) { xc[u] = min(cell[u] * sl, L.W - 1); wx[u] = 0.f; }
        }
        auto column = [&](int row, float2 &tx, float2 &ty) {   // displacement of a control row at the two columns
            const float2 p0 = ct(row, cell[0]), p1 = ct(row, cell[0] + 1), q0 = ct(row, cell[1]), q1 = ct(row, cell[1] + 1);
            tx = make_float2(fmaf(wx[0], p1.x - p0.x, p0.x), fmaf(wx[1], q1.x - q0.x, q0.x));
            ty = make_float2(fmaf(wx[0], p1.y - p0.y, p0.y), fmaf(wx[1], q1.y - q0.y, q0.y));
        };
        const S *ra = Rp + xc[0], *rb = Rp + xc[1];
        float2 sE[4], sR[4], s1[4], sM[4];   // top x, top y, bottom x, bottom y
#pragma unroll
        for (int i = 0; i < 4; ++i) sE[i] = sR[i] = s1[i] = sM[i] = f2(0.f);
        float2 tx, ty;
        column(ca, tx, ty);
        auto flush = [&]() {
#pragma unroll
            for (int i = 0; i < NM; ++i) {
                ff_acc2(hi2[i], lo2[i], make_float2(act[0] ? a[i].x : 0.f, act[1] ? a[i].y : 0.f));
                a[i] = f2(0.f);
            }
        };
        // one pixel of either column; wy: the weight of the control row below
        auto pixel = [&](const TapRow &t0, const TapRow &t1, const TapRow &t2, float2 fx, float2 fy, float2 r, float2 wy) {
            float2 dx2, dy2;
            const float2 e = __ffma2_rn(ngam, r, __fadd2_rn(bspline2(t0, t1, t2, fx, fy, dx2, dy2), ncT));
            a[0] = __fadd2_rn(a[0], e);
            a[1] = __ffma2_rn(e, e, a[1]);
            a[2] = __ffma2_rn(r, e, a[2]);
            if constexpr (START) {
                a[3] = __fadd2_rn(a[3], r);
                a[4] = __ffma2_rn(r, r, a[4]);
            }
            const float2 wb = __fmul2_rn(f2(0.5f), wy), wt = f2sub(f2(0.5f), wb);   // half of wy and 1 - wy
            const float2 g[4] = {__fmul2_rn(wt, dx2), __fmul2_rn(wt, dy2), __fmul2_rn(wb, dx2), __fmul2_rn(wb, dy2)};
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                sE[i] = __ffma2_rn(e, g[i], sE[i]);
                sR[i] = __ffma2_rn(r, g[i], sR[i]);
                s1[i] = __fadd2_rn(s1[i], g[i]);
                if constexpr (START) sM[i] = __ffma2_rn(g[i], g[i], sM[i]);
            }
        };
        // the window of one row of one column, anywhere: clamped into the level's border
        auto window = [&](float m_x, float m_y, int x, int y) {
            const int wxn = min(max((int)(__float_as_uint(m_x) - kRoundBits + (unsigned)x), -2), L.W + 1);
            const int wyn = min(max((int)(__float_as_uint(m_y) - kRoundBits + (unsigned)y), -2), L.H + 1);
            return T + (ptrdiff_t)(wyn - 1) * L.Tp + wxn;
        };
        auto row = [&](const S *qa, const S *qb) {
            return tap_row(make_float2(ldS<S>(qa - 1), ldS<S>(qb - 1)), make_float2(ldS<S>(qa), ldS<S>(qb)),
                           make_float2(ldS<S>(qa + 1), ldS<S>(qb + 1)));
        };
        for (int cy = ca; cy <= cb; ++cy) {
            if (cy < cb) {
                float2 bx, by;
                column(cy + 1, bx, by);
                const float2 ex = f2sub(bx, tx), ey = f2sub(by, ty);
                const float cyf = (float)cy;
                const int yc = min(L.H, (cy + 1) * sl), y1 = cy == ncy - 1 ? L.H : yc;
                int y = min(y1, cy * sl + piece * P.ph);
                const int ye = piece == P.h - 1 ? y1 : min(y1, y + P.ph);
                while (y < ye) {
                    // the weight of the control row below; a row past the last cell row lies on it
                    const float2 w0 = f2(y < yc ? fmaf(GL.pl, (float)y, GL.off) * GL.scale_inv - cyf : 1.f);
                    const float2 v0x = __ffma2_rn(w0, ex, tx), v0y = __ffma2_rn(w0, ey, ty);
                    const float2 m0x = __fadd2_rn(v0x, f2(kRound)), m0y = __fadd2_rn(v0y, f2(kRound));
                    const int nxa = (int)(__float_as_uint(m0x.x) - kRoundBits + (unsigned)xc[0]);
                    const int nxb = (int)(__float_as_uint(m0x.y) - kRoundBits + (unsigned)xc[1]);
                    const int nya = (int)(__float_as_uint(m0y.x) - kRoundBits + (unsigned)y);
                    const int nyb = (int)(__float_as_uint(m0y.y) - kRoundBits + (unsigned)y);
                    // a straight run of n rows: the rounded displacement is the same in its first and its last
                    // row, and so in every one between (it is monotonic along a column of a cell)
                    auto straight = [&](int n) {
                        const float2 w1 = __ffma2_rn(f2((float)(n - 1)), dw, w0);
                        const float2 m1x = __fadd2_rn(__ffma2_rn(w1, ex, tx), f2(kRound));
                        const float2 m1y = __fadd2_rn(__ffma2_rn(w1, ey, ty), f2(kRound));
                        const unsigned diff = (__float_as_uint(m1x.x) ^ __float_as_uint(m0x.x)) |
                                              (__float_as_uint(m1x.y) ^ __float_as_uint(m0x.y)) |
                                              (__float_as_uint(m1y.x) ^ __float_as_uint(m0y.x)) |
                                              (__float_as_uint(m1y.y) ^ __float_as_uint(m0y.y));
                        return (bool)__all_sync(0xffffffffu, diff == 0u && (unsigned)(nxa + 2) <= (unsigned)(L.W + 3) &&
                                                                 (unsigned)(nxb + 2) <= (unsigned)(L.W + 3) &&
                                                                 nya >= -2 && nya + n <= L.H + 2 && nyb >= -2 &&
                                                                 nyb + n <= L.H + 2);
                    };
                    const int left = min(ye, yc) - y;
                    int n = min(left, kRunRows);
                    bool run = n > 1 && straight(n);
                    if (!run && n > kRunRows / 2) {
                        n = kRunRows / 2;
                        run = straight(n);
                    }
                    const S *rya = ra + (ptrdiff_t)y * L.Rp, *ryb = rb + (ptrdiff_t)y * L.Rp;
                    if (run) {
                        const S *qa = T + (ptrdiff_t)(nya - 1) * L.Tp + nxa, *qb = T + (ptrdiff_t)(nyb - 1) * L.Tp + nxb;
                        const float2 ox = f2sub(tx, f2sub(m0x, f2(kRound))), oy = f2sub(ty, f2sub(m0y, f2(kRound)));
                        TapRow t0 = row(qa, qb);
                        qa += L.Tp; qb += L.Tp;
                        TapRow t1 = row(qa, qb);
                        float2 w = w0;
                        int k = 0;
                        for (; k + R <= n; k += R) {
                            float2 r[R], q[R][3];
#pragma unroll
                            for (int i = 0; i < R; ++i) {
                                qa += L.Tp; qb += L.Tp;
#pragma unroll
                                for (int j = 0; j < 3; ++j) q[i][j] = make_float2(ldS<S>(qa + j - 1), ldS<S>(qb + j - 1));
                                r[i] = make_float2(ldS<S>(rya), ldS<S>(ryb));
                                rya += L.Rp; ryb += L.Rp;
                            }
#pragma unroll
                            for (int i = 0; i < R; ++i) {
                                const float2 wy = i == 0 ? w : __ffma2_rn(f2((float)i), dw, w);
                                const TapRow t2 = tap_row(q[i][0], q[i][1], q[i][2]);
                                pixel(t0, t1, t2, __ffma2_rn(wy, ex, ox), __ffma2_rn(wy, ey, oy), __fadd2_rn(r[i], ncR), wy);
                                t0 = t1;
                                t1 = t2;
                            }
                            w = __ffma2_rn(f2((float)R), dw, w);
                            if ((k & (kFast - R)) == kFast - R) flush();
                        }
                        for (; k < n; ++k) {   // what R does not divide
                            qa += L.Tp; qb += L.Tp;
                            const TapRow t2 = row(qa, qb);
                            const float2 r = make_float2(ldS<S>(rya), ldS<S>(ryb));
                            rya += L.Rp; ryb += L.Rp;
                            pixel(t0, t1, t2, __ffma2_rn(w, ex, ox), __ffma2_rn(w, ey, oy), __fadd2_rn(r, ncR), w);
                            t0 = t1;
                            t1 = t2;
                            w = __fadd2_rn(w, dw);
                        }
                    } else {
                        // every row loads its own window
                        n = min(n, kRunRows / 2);
                        if (n < 1) n = 1;
#pragma unroll 2
                        for (int k = 0; k < n; ++k) {
                            const float2 wy = __ffma2_rn(f2((float)k), dw, w0);
                            const float2 vx = __ffma2_rn(wy, ex, tx), vy = __ffma2_rn(wy, ey, ty);
                            const float2 mx = __fadd2_rn(vx, f2(kRound)), my = __fadd2_rn(vy, f2(kRound));
                            const S *qa = window(mx.x, my.x, xc[0], y + k), *qb = window(mx.y, my.y, xc[1], y + k);
                            const float2 r = make_float2(ldS<S>(rya), ldS<S>(ryb));
                            rya += L.Rp; ryb += L.Rp;
                            const TapRow t0 = row(qa, qb), t1 = row(qa + L.Tp, qb + L.Tp),
                                         t2 = row(qa + 2 * (ptrdiff_t)L.Tp, qb + 2 * (ptrdiff_t)L.Tp);
                            pixel(t0, t1, t2, f2sub(vx, f2sub(mx, f2(kRound))), f2sub(vy, f2sub(my, f2(kRound))),
                                  __fadd2_rn(r, ncR), wy);
                        }
                    }
                    flush();
                    y += n;
                }
                tx = bx;
                ty = by;
            }
            // control row cy: what the cell row above it left and the top sums of the one below
            {
                const float2 wf = make_float2(__shfl_sync(0xffffffffu, wx[0], 0), __shfl_sync(0xffffffffu, wx[1], 0));
                const int2 lst = make_int2(last[0], strip0 + 1 < strips ? last[1] : -1);
                const int strip = (P.m + 1) * (P.g + 1) * kSlot;
                float *slot = slots + (seg * P.nst + slot0) * strip + (cy - ca) * (P.g + 1) * kSlot;
                float *slot1 = walk ? slot : slot + strip;
                auto put = [&](int row, int rows, float2 v) {   // the lane's two columns of a sum
                    emit[row * kEmitRow + lane] = act[0] ? v.x : 0.f;
                    emit[(rows + row) * kEmitRow + lane] = act[1] ? v.y : 0.f;
                };
                __syncwarp();
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    put(i, kEmitSums, sE[i]);
                    put(2 + i, kEmitSums, sR[i]);
                    put(4 + i, kEmitSums, s1[i]);
                }
                __syncwarp();
                emit_any<false>(sl, emit, lane, P.g, wf, dw.x, lst, slot, slot1, adds);
                if constexpr (START) {
                    __syncwarp();
                    put(0, 2, sM[0]);
                    put(1, 2, sM[1]);
                    __syncwarp();
                    emit_any<true>(sl, emit, lane, P.g, wf, dw.x, lst, slot, slot1, adds);
                }
            }
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                sE[i] = sE[2 + i]; sE[2 + i] = f2(0.f);
                sR[i] = sR[2 + i]; sR[2 + i] = f2(0.f);
                s1[i] = s1[2 + i]; s1[2 + i] = f2(0.f);
                sM[i] = sM[2 + i]; sM[2 + i] = f2(0.f);
            }
        }
    }
    float hi[6], lo[6];
#pragma unroll
    for (int i = 0; i < 6; ++i) {
        hi[i] = i < NM ? hi2[i].x : 0.f;
        lo[i] = i < NM ? lo2[i].x : 0.f;
        if (i < NM) ff_add(hi[i], lo[i], hi2[i].y, lo2[i].y);
    }
    // the regulariser's edges from this CTA's own rows: to the right and down
    {
        float e = 0.f;
        int k = 0;
        int i = pi.i0, col = pi.x0;
        for (int j = threadIdx.x; j < (B.own1 - B.cr0) * G.nx; j += kThreads) {
            if (j >= kThreads) PointIter::at(G.nx, j, i, col);
            const int row = B.cr0 + i;
            const float2 v = ct(row, col);
            if (col + 1 < G.nx) {
                const float2 w = ct(row, col + 1);
                e = fmaf(w.x - v.x, w.x - v.x, fmaf(w.y - v.y, w.y - v.y, e));
            }
            if (row + 1 < G.ny) {
                const float2 w = ct(row + 1, col);
                e = fmaf(w.x - v.x, w.x - v.x, fmaf(w.y - v.y, w.y - v.y, e));
            }
            if (++k == kFast) { ff_acc(hi[5], lo[5], e); e = 0.f; k = 0; }
        }
        ff_acc(hi[5], lo[5], e);
    }
    // the last control row's sums, where the CTA below owns that row, go to it
    constexpr int kPairs = START ? 4 : 3;
    const unsigned due = B.cr0 > 0 && B.cr0 < B.cr1 ? (unsigned)(G.nx * kPairs) * 8u : 0u;
    cluster_reduce<6, false>(hi, lo, 0.f, sm, comm, cl, due, [&](unsigned n) {
        if (!(B.cr0 < B.cr1 && B.own1 < G.ny)) return;
        for (int t = threadIdx.x; t < G.nx * kPairs; t += kThreads) {
            const int jx = t / kPairs, i = 2 * (t - jx * kPairs);
            float v[2] = {0.f, 0.f};
            slot_sum<2>(slots, P, ncx, B.q, B.q, jx, i, v);
            send8(above + jx * kSlot + i, &sm.xbar[n & 1], (int)cl.block_rank() + 1, make_float2(v[0], v[1]));
        }
    });
}

// The same over the whole grid: this CTA's slots, and at its first row what the CTA above sent.
template <int N, bool FF = false>
__device__ __forceinline__ void point_sum(const float *slots, const float *above, const PassGeom &P, const Band &B,
                                          int ncx, int row, int jx, int first, float (&o)[N])
{
#pragma unroll
    for (int k = 0; k < N; ++k) o[k] = 0.f;
    if (row == B.cr0 && row > 0)
#pragma unroll
        for (int k = 0; k < N; ++k) o[k] = above[jx * kSlot + first + k];
    slot_sum<N, FF>(slots, P, ncx, B.cr1 - B.cr0, row - B.cr0, jx, first, o);
}

// Buffers of the H1 scalar product (B null: another product): B the right-hand side -Nc dE/dc,
// T and U work grids, q the cosine bases and eigenvalues of the control grid (Qx [nx][nx],
// Qy [ny][ny], lx [nx], ly [ny], device memory), s2 = sigma^2.
struct H1Bufs {
    float2 *B = nullptr, *T = nullptr, *U = nullptr;
    const float *q = nullptr;
    float s2 = 0.f;
};

// U = (I + s2 Lg)^-1 B per axis, Lg the control grid's graph Laplacian, through its eigenbasis:
// Lg = (Qy (x) Qx) diag(ly_m + lx_k) (Qy (x) Qx)^T with Qx, Qy the orthonormal DCT-II bases
// (free-end path graphs), so U = Qy [(Qy^T B Qx) / (1 + s2 (ly_m + lx_k))] Qx^T: four small matrix
// products over the grid, every CTA of the cluster the same work in the same order.
__device__ void h1_solve(const H1Bufs &h, int nx, int ny)
{
    const float *Qx = h.q, *Qy = h.q + nx * nx, *lx = Qy + ny * ny, *ly = lx + nx;
    const int Nc = nx * ny;
    // T = B Qx
    for (int i = threadIdx.x; i < Nc; i += kThreads) {
        const int jy = i / nx, k = i - jy * nx;
        float ax = 0.f, ay = 0.f;
        for (int jx = 0; jx < nx; ++jx) {
            const float qv = __ldg(Qx + jx * nx + k);
            const float2 b = h.B[jy * nx + jx];
            ax = fmaf(b.x, qv, ax);
            ay = fmaf(b.y, qv, ay);
        }
        h.T[i] = make_float2(ax, ay);
    }
    __syncthreads();
    // U = (Qy^T T) / (1 + s2 (ly_m + lx_k))
    for (int i = threadIdx.x; i < Nc; i += kThreads) {
        const int m = i / nx, k = i - m * nx;
        float ax = 0.f, ay = 0.f;
        for (int jy = 0; jy < ny; ++jy) {
            const float qv = __ldg(Qy + jy * ny + m);
            const float2 t = h.T[jy * nx + k];
            ax = fmaf(qv, t.x, ax);
            ay = fmaf(qv, t.y, ay);
        }
        const float den = fmaf(h.s2, __ldg(ly + m) + __ldg(lx + k), 1.f);
        h.U[i] = make_float2(ax / den, ay / den);
    }
    __syncthreads();
    // T = Qy U
    for (int i = threadIdx.x; i < Nc; i += kThreads) {
        const int jy = i / nx, k = i - jy * nx;
        float ax = 0.f, ay = 0.f;
        for (int m = 0; m < ny; ++m) {
            const float qv = __ldg(Qy + jy * ny + m);
            const float2 u = h.U[m * nx + k];
            ax = fmaf(qv, u.x, ax);
            ay = fmaf(qv, u.y, ay);
        }
        h.T[i] = make_float2(ax, ay);
    }
    __syncthreads();
    // U = T Qx^T
    for (int i = threadIdx.x; i < Nc; i += kThreads) {
        const int jy = i / nx, jx = i - jy * nx;
        float ax = 0.f, ay = 0.f;
        for (int k = 0; k < nx; ++k) {
            const float qv = __ldg(Qx + jx * nx + k);
            const float2 t = h.T[jy * nx + k];
            ax = fmaf(t.x, qv, ax);
            ay = fmaf(t.y, qv, ay);
        }
        h.U[i] = make_float2(ax, ay);
    }
    __syncthreads();
}

// The flow's scalar product at c, from the pass's squared-derivative sums: per own control point and
// axis m = dk sum_x w_j(x)^2 (dT/dp)^2 + rk n_j (dk = 1/(P var T), rk = lambda/P, n_j the neighbours
// of j), normalised by the mean of all 2 Nc values and floored at 1e-3 of it, written to mt.
__device__ void grid_metric(const Grid &G, const PassGeom &P, const Band &B, const float *slots, const float *above,
                            const PointIter &pi, float2 *mt, float dk, float rk, Smem &sm, Comm &comm, const cg::cluster_group &cl)
{
    const int n = (B.own1 - B.cr0) * G.nx;
    float hi[1] = {0.f}, lo[1] = {0.f};
    int i = pi.i0, jx = pi.x0;
    for (int j = threadIdx.x; j < n; j += kThreads) {
        if (j >= kThreads) PointIter::at(G.nx, j, i, jx);
        const int row = B.cr0 + i;
        float s[2];
        point_sum<2>(slots, above, P, B, G.nx - 1, row, jx, 6, s);
        const float nb = (float)((jx > 0) + (jx + 1 < G.nx) + (row > 0) + (row + 1 < G.ny));
        const float2 m = make_float2(fmaf(dk, s[0], rk * nb), fmaf(dk, s[1], rk * nb));
        mt[(row - B.h0) * G.nx + jx] = m;
        ff_acc(hi[0], lo[0], m.x + m.y);
    }
    cluster_reduce<1, false>(hi, lo, 0.f, sm, comm, cl);
    const double mean = sm.tot[0] / (2.0 * (G.nx * G.ny));
    const float inv = mean > 0.0 ? (float)(1.0 / mean) : 0.f;
    for (int j = threadIdx.x; j < n; j += kThreads) {
        float2 &m = mt[(B.cr0 - B.h0) * G.nx + j];
        m = mean > 0.0 ? make_float2(fmaxf(m.x * inv, 1e-3f), fmaxf(m.y * inv, 1e-3f)) : make_float2(1.f, 1.f);
    }
}

// The descent direction d = -M^-1 grad E at c with the scalar product mt, from the pass's gradient
// sums: dE/dc_j = (1/P) [bP sE + cP sR + kP s1 + lambda sum_nbrs (c_j - c_k)] (pm: b P, c P, kappa P,
// lambda), at the own rows and, through the neighbours' staged rows, at the held ones.  Leaves
// sum_j m_j |d_j|^2 in sm.tot[0], with the direction d held before the call <d_old, d_old - d>_M in
// sm.tot[1] and |d_old - d|_M^2 in sm.tot[2], max |d_j|^2 in sm.tmax; identical in every CTA.
template <bool FF = false>
__device__ void grid_direction(const Grid &G, const Lvl &L, const PassGeom &P, const Band &B, const float2 *c,
                               float2 *d, float2 *mt, float2 *halo, const float *slots, const float *above,
                               const PointIter &pi, const float *pm, Smem &sm, Comm &comm, const cg::cluster_group &cl, const H1Bufs &h1)
{
    const int Nc = G.nx * G.ny, n = (B.own1 - B.cr0) * G.nx, rank = cl.block_rank();
    const bool quiet = comm_quiet(sm);
    const float bP = pm[0], cP = pm[1], kP = pm[2], lam = pm[3];
    const float scale = -(float)Nc / ((float)L.W * (float)L.H);
    float hi[3] = {0.f, 0.f, 0.f}, lo[3] = {0.f, 0.f, 0.f}, mx = 0.f;
    // -Nc dE/dc at own point j (row i of the own rows)
    auto rhs = [&](int i, int jx) {
        const int row = B.cr0 + i, k = (row - B.h0) * G.nx + jx;
        float s[6];
        point_sum<6, FF>(slots, above, P, B, G.nx - 1, row, jx, 0, s);
        const float gx = fmaf(bP, s[0], fmaf(cP, s[2], kP * s[4]));
        const float gy = fmaf(bP, s[1], fmaf(cP, s[3], kP * s[5]));
        const float2 cj = c[k];
        float lx = 0.f, ly = 0.f;
        if (jx > 0)         { const float2 v = c[k - 1];    lx += cj.x - v.x; ly += cj.y - v.y; }
        if (jx + 1 < G.nx)  { const float2 v = c[k + 1];    lx += cj.x - v.x; ly += cj.y - v.y; }
        if (row > 0)        { const float2 v = c[k - G.nx]; lx += cj.x - v.x; ly += cj.y - v.y; }
        if (row + 1 < G.ny) { const float2 v = c[k + G.nx]; lx += cj.x - v.x; ly += cj.y - v.y; }
        return make_float2(scale * fmaf(lam, lx, gx), scale * fmaf(lam, ly, gy));
    };
    if (h1.B) {
        // H1 product: b = -Nc dE/dc into B of every CTA, d = M^-1 b into U by every CTA; then
        // |d|_M^2 = d.b, and for the first trial <d_prev, y>_M, |y|_M^2 with y = d_prev - d, M y
        // taken as the stencil y + s2 Lg y
        // an exchange of its own; every CTA sends every other one at least a word, as exchanges rely on
        const unsigned xn = comm.n++, C = cl.num_blocks();
        const unsigned long long *xb = &sm.xbar[xn & 1];
        if (threadIdx.x == 0) comm_expect(sm, xn, (unsigned)Nc * 8u + C * 4u);
        if (threadIdx.x < C && !quiet) send4(&sm.pmax[xn & 1][rank], xb, threadIdx.x, 0u);
        int i = pi.i0, jx = pi.x0;
        for (int j = threadIdx.x; j < n; j += kThreads) {
            if (j >= kThreads) PointIter::at(G.nx, j, i, jx);
            const float2 b = rhs(i, jx);
            if (!quiet)
                for (unsigned r = 0; r < C; ++r) send8(h1.B + (B.cr0 + i) * G.nx + jx, xb, r, b);
        }
        if (threadIdx.x < 32) comm_wait(sm, xn);
        __syncthreads();   // B is complete, and this CTA's slots have been read (T and U lie there)
        h1_solve(h1, G.nx, G.ny);
        auto yv = [&](int row, int jx) {
            const float2 a = d[(row - B.h0) * G.nx + jx], b = h1.U[row * G.nx + jx];
            return make_float2(a.x - b.x, a.y - b.y);
        };
        i = pi.i0;
        jx = pi.x0;
        for (int j = threadIdx.x; j < n; j += kThreads) {
            if (j >= kThreads) PointIter::at(G.nx, j, i, jx);
            const int row = B.cr0 + i;
            const float2 dj = h1.U[row * G.nx + jx], bj = h1.B[row * G.nx + jx], dold = d[(row - B.h0) * G.nx + jx];
            const float2 y = yv(row, jx);
            float lx = 0.f, ly = 0.f;
            if (jx > 0)         { const float2 v = yv(row, jx - 1); lx += y.x - v.x; ly += y.y - v.y; }
            if (jx + 1 < G.nx)  { const float2 v = yv(row, jx + 1); lx += y.x - v.x; ly += y.y - v.y; }
            if (row > 0)        { const float2 v = yv(row - 1, jx); lx += y.x - v.x; ly += y.y - v.y; }
            if (row + 1 < G.ny) { const float2 v = yv(row + 1, jx); lx += y.x - v.x; ly += y.y - v.y; }
            const float myx = fmaf(h1.s2, lx, y.x), myy = fmaf(h1.s2, ly, y.y);
            ff_acc(hi[0], lo[0], fmaf(dj.x, bj.x, dj.y * bj.y));
            ff_acc(hi[1], lo[1], fmaf(dold.x, myx, dold.y * myy));
            ff_acc(hi[2], lo[2], fmaf(y.x, myx, y.y * myy));
            mx = fmaxf(mx, fmaf(dj.x, dj.x, dj.y * dj.y));
        }
        __syncthreads();   // every d_prev was read before d is replaced
        for (int j = threadIdx.x; j < (B.h1 - B.h0) * G.nx; j += kThreads) d[j] = h1.U[B.h0 * G.nx + j];
        cluster_reduce<3, true>(hi, lo, mx, sm, comm, cl);
        return;
    }
    // The edge rows go to the neighbours' halo rows (0: the row above the own ones, 1: the row below),
    // not to their d, which a slower neighbour may still read for its accepted step; they count on the
    // exchange of the sums below.
    const unsigned long long *bar = &sm.xbar[comm.n & 1];
    unsigned due = 0;
    if (B.cr0 < B.cr1) due = (unsigned)G.nx * 8u * ((B.cr0 > 0 ? 1u : 0u) + (B.own1 < G.ny ? 1u : 0u));
    int i = pi.i0, jx = pi.x0;
    for (int j = threadIdx.x; j < n; j += kThreads) {
        if (j >= kThreads) PointIter::at(G.nx, j, i, jx);
        const int row = B.cr0 + i, k = (row - B.h0) * G.nx + jx;
        const float2 b = rhs(i, jx), mj = mt[k], dold = d[k];
        const float2 dj = make_float2(b.x / mj.x, b.y / mj.y);
        d[k] = dj;
        if (i == 0 && B.cr0 > 0 && !quiet) send8(halo + G.nx + jx, bar, rank - 1, dj);
        if (row == B.cr1 - 1 && B.own1 < G.ny && !quiet) send8(halo + jx, bar, rank + 1, dj);
        const float yx = dold.x - dj.x, yy = dold.y - dj.y;
        ff_acc(hi[0], lo[0], fmaf(mj.x * dj.x, dj.x, mj.y * dj.y * dj.y));
        ff_acc(hi[1], lo[1], fmaf(mj.x * dold.x, yx, mj.y * dold.y * yy));
        ff_acc(hi[2], lo[2], fmaf(mj.x * yx, yx, mj.y * yy * yy));
        mx = fmaxf(mx, fmaf(dj.x, dj.x, dj.y * dj.y));
    }
    cluster_reduce<3, true>(hi, lo, mx, sm, comm, cl, due);
    for (int j = threadIdx.x; j < 2 * G.nx; j += kThreads) {
        const bool below = j >= G.nx;
        const int row = below ? B.own1 : B.cr0 - 1;
        if (B.cr0 < B.own1 && row >= 0 && row < G.ny) d[(row - B.h0) * G.nx + (below ? j - G.nx : j)] = halo[j];
    }
}

// Parameter slots of the nonrigid passes: gradient coefficients b P, c P, kappa P (grad_coef)
// and lambda; the scalar product's 1/(P var T) and lambda/P; the next trial's step.
enum FieldParam { kPmB = 0, kPmC = 1, kPmK = 2, kPmLam = 3, kPmDk = 4, kPmRk = 5, kPmTau = 6 };

// The coefficients times P, formed in FP64 and rounded once.
__device__ __forceinline__ void field_grad_params(const Ncc &n, const LevelSums &L, const Config &cfg, float *pm)
{
    const GradCoef k = grad_coef(L, n);
    pm[kPmB] = (float)__dmul_rn(k.b, L.P);
    pm[kPmC] = (float)__dmul_rn(k.c, L.P);
    pm[kPmK] = (float)__dmul_rn(k.kappa, L.P);
    pm[kPmLam] = (float)cfg.lambda;
}

// Thread-0 controller of the nonrigid level loop (same rules as the rigid one).  field_eval decides
// on a pass's moments: the level's first point, an accepted trial (`accepted` = 1) or a rejected
// one, whose shorter step it leaves in pm[kPmTau]; kActGrad asks for the direction there.
__device__ int field_eval(FieldCtl &k, const Config &cfg, const double *tot, bool start, float *pm, int &accepted)
{
    accepted = 0;
    if (start) set_reference(k.ls, tot[3], tot[4]);
    const Ncc n = ncc_terms(k.ls, tot[0], tot[1], tot[2]);
    const double Et = __fma_rn(k.half_lam, tot[5], n.e);
    if (start) {
        k.E = Et;
        // the level's scalar product at its initial control values: 1/(P var T) and lambda/P
        const double vt = n.Stt * k.ls.invP;
        pm[kPmDk] = vt > 0.0 ? (float)(k.ls.invP / vt) : 0.f;
        pm[kPmRk] = (float)(2.0 * k.half_lam);
        field_grad_params(n, k.ls, cfg, pm);
        return kActGrad;
    }
    k.evals += 1;
    if (nonneg(k.accept - Et)) {
        accepted = 1;   // c is advanced by the trial's step
        field_grad_params(n, k.ls, cfg, pm);
        k.iters += 1;
        k.Eold = k.E;
        k.ss_old = k.ss;
        k.tau_acc = (double)(float)k.tau;
        k.have_prev = 1;
        k.E = Et;
        if (nonneg(Et - k.rel)) { k.stop = REG_STOP_REL; return kActDone; }
        return kActGrad;
    }
    k.rejects += 1;
    k.nrej += 1;
    const double slope = -k.ss * k.invNc;
    const double tau = next_tau(k.E, slope, k.tau, Et, false);
    k.tau = tau;
    if (k.nrej > cfg.max_rejects) { k.stop = REG_STOP_LS; return kActDone; }
    k.accept = __fma_rn(cfg.armijo_c * slope, tau, k.E);
    pm[kPmTau] = (float)tau;
    return kActTrial;
}

// The stop tests at a point whose direction is known, and the first trial's step.
__device__ int field_grad(FieldCtl &k, const Config &cfg, const double *tot, float dmax2, float *pm)
{
    k.evals += 1;
    if (k.iters >= cfg.max_iter) { k.stop = REG_STOP_MAXIT; return kActDone; }
    // |g| = sqrt(ss / Nc) and the largest control step dmax: compared squared
    const double ss = tot[0];
    k.ss = ss;
    if (!at_least(ss, k.tolss)) { k.stop = REG_STOP_GRAD; return kActDone; }
    // the metric (mean over control points) is a common factor of the two sums; without positive
    // curvature the quadratic rule of the last step
    double tau = k.tau;
    if (k.have_prev && !bb_tau(k.tau_acc, tot[1], tot[2], tau))
        tau = next_tau(k.Eold, -k.ss_old * k.invNc, k.tau, k.E, true);
    if (tau * tau * (double)dmax2 > cfg.step_cap * cfg.step_cap) tau = cfg.step_cap / sqrt((double)dmax2);
    k.tau = tau;
    k.nrej = 0;
    k.accept = __fma_rn(-ss * (cfg.armijo_c * k.invNc), tau, k.E);
    k.rel = cfg.tol_rel_e == 0.0 ? k.E : k.E - cfg.tol_rel_e * fabs(k.E);
    pm[kPmTau] = (float)tau;
    return kActTrial;
}

// FFD value of the grid q (finest-pixel values) at finest coordinate (X, Y), read through L2.
__device__ __forceinline__ float2 grid_eval_global(const float2 *q, const Grid &G, float X, float Y)
{
    float gx = fminf(fmaxf(X / (float)G.s, 0.f), (float)(G.nx - 1));
    float gy = fminf(fmaxf(Y / (float)G.s, 0.f), (float)(G.ny - 1));
    int ix = min((int)gx, G.nx - 2), iy = min((int)gy, G.ny - 2);
    float wx = gx - (float)ix, wy = gy - (float)iy;
    const float2 *p = q + iy * G.nx + ix;
    float2 a = __ldcg(p), b = __ldcg(p + 1), e = __ldcg(p + G.nx), f = __ldcg(p + G.nx + 1);
    float hx = 1.f - wx, hy = 1.f - wy;
    float2 u;
    u.x = fmaf(wy, fmaf(wx, f.x, hx * e.x), hy * fmaf(wx, b.x, hx * a.x));
    u.y = fmaf(wy, fmaf(wx, f.y, hx * e.y), hy * fmaf(wx, b.y, hx * a.y));
    return u;
}

// The level's geometry into shared memory (a barrier follows): read from the parameters by every pass, it
// waits for the constant cache.
__device__ __forceinline__ const PassGeom &level_geom(Smem &sm, const Params &p, int l, bool over)
{
    static_assert(sizeof(PassGeom) % 4 == 0 && sizeof(PassGeom) / 4 <= kThreads, "copied by words");
    if (threadIdx.x < sizeof(PassGeom) / 4) ((int *)&sm.geom)[threadIdx.x] = ((const int *)&p.geom[l][over])[threadIdx.x];
    return sm.geom;
}

template <typename S, int R>
__device__ void run_nonrigid(const Params &p, const OpDesc &op, int op_index, Smem &sm, float2 *gbuf, Comm &comm,
                             const cg::cluster_group &cl)
{
    const int tid = threadIdx.x;
    const int C = cl.num_blocks(), rank = cl.block_rank();
    const Config &cfg = p.cfg;
    const int Lc = cfg.levels;
    const Grid G{p.gnx, p.gny, p.gs};
    const int Nc = G.nx * G.ny;
    const bool h1 = cfg.metric == REG_METRIC_H1;
    const GridLayout lay = grid_layout(G.nx, G.ny, C, h1);
    const Band B = grid_band(G, rank, C);
    const PointIter pi(G.nx);
    const int held = (B.h1 - B.h0) * G.nx, first = B.h0 * G.nx;   // points held, and the first of them
    float2 *c = gbuf + lay.c, *d = gbuf + lay.d, *mt = gbuf + lay.mt, *halo = gbuf + lay.halo;
    float *slots = (float *)(gbuf + lay.slots);
    const float *above = (const float *)(gbuf + lay.above);
    float *emits = (float *)(gbuf + lay.emits);
    const H1Bufs hb{h1 ? mt : nullptr, (float2 *)slots, (float2 *)slots + Nc, p.h1q, (float)(cfg.sigma * cfg.sigma)};
    // initial control values (finest px), scaled to the coarsest level
    {
        const float sc = ldexpf(1.f, -(Lc - 1));
        if (op.left >= 0) {
            // B's initial guess phi_jk o phi_ij at the control points (Sec. 2.3.2)
            const float2 *q1 = p.node_grid + (size_t)Nc * op.left, *q2 = p.node_grid + (size_t)Nc * op.right;
            for (int j = tid; j < held; j += kThreads) {
                const int jy = (first + j) / G.nx, jx = first + j - jy * G.nx;
                const float2 a = __ldcg(q1 + first + j);
                const float2 u = grid_eval_global(q2, G, (float)(jx * G.s) + a.x, (float)(jy * G.s) + a.y);
                c[j] = make_float2(sc * (a.x + u.x), sc * (a.y + u.y));
            }
        } else if (op.init_node >= 0) {
            const float2 *q = p.node_grid + (size_t)Nc * op.init_node;
            for (int j = tid; j < held; j += kThreads) {
                const float2 a = __ldcg(q + first + j);
                c[j] = make_float2(sc * a.x, sc * a.y);
            }
        } else {
            for (int j = tid; j < held; j += kThreads) c[j] = make_float2(0.f, 0.f);
        }
    }
    FieldCtl &k = sm.fctl;
    if (tid == 0) {
        memset(&k, 0, sizeof(k));
        k.invNc = 1.0 / (double)Nc;
    }
    int stops[kMaxLevels], iters[kMaxLevels], evals[kMaxLevels];
    for (int l = Lc - 1; l >= 0; --l) {
        const Lvl L = level_of(p, op.ref, op.tmpl, l);
        const GridLvl GL = grid_level(G, L, l);
        const PassGeom &P = level_geom(sm, p, l, L.W > (G.nx - 1) * (G.s >> l));
        if (cfg.metric == REG_METRIC_MEAN)
            for (int j = tid; j < held; j += kThreads) mt[j] = make_float2(1.f, 1.f);
        if (tid == 0) {
            set_level(k.ls, L.W, L.H, L.gam);
            k.half_lam = 0.5 * cfg.lambda * k.ls.invP;
            k.tau = cfg.tau0;
            k.have_prev = 0;
            k.iters = 0; k.evals = 0; k.stop = REG_STOP_MAXIT;
            // a coarse level only supplies the next level's initial guess: a looser stop
            const double tolg = cfg.tol_grad * (l > 0 ? cfg.tol_coarse : 1.0);
            k.tolss = tolg * tolg * (double)Nc;
        }
        __syncthreads();
        for (bool start = true;; start = false) {
            const float tau = sm.pm[kPmTau];   // not read by a level's first pass
            if (start) grid_pass<S, true, R>(L, G, GL, P, B, c, d, 0.f, slots, above, emits, pi, sm, comm, cl);
            else grid_pass<S, false, R>(L, G, GL, P, B, c, d, tau, slots, above, emits, pi, sm, comm, cl);
            if (tid == 0) {
                sm.action = field_eval(k, cfg, sm.tot, start, sm.pm, sm.idata[0]);
                if (sm.fail) sm.action = kActDone;
            }
            __syncthreads();
            const int act = sm.action;
            if (sm.idata[0]) {
                // the accepted trial, as the pass formed it
                for (int j = tid; j < held; j += kThreads) {
                    const float2 a = c[j], b = d[j];
                    c[j] = make_float2(fmaf(tau, b.x, a.x), fmaf(tau, b.y, a.y));
                }
                __syncthreads();
            }
            if (act == kActDone) break;
            if (act == kActTrial) continue;
            float pm[6];
#pragma unroll
            for (int q = 0; q < 6; ++q) pm[q] = sm.pm[q];
            if (start && cfg.metric == REG_METRIC_GAUSS_NEWTON)
                grid_metric(G, P, B, slots, above, pi, mt, pm[kPmDk], pm[kPmRk], sm, comm, cl);
            grid_direction(G, L, P, B, c, d, mt, halo, slots, above, pi, pm, sm, comm, cl, hb);
            if (tid == 0) {
                sm.action = field_grad(k, cfg, sm.tot, sm.tmax, sm.pm);
                if (sm.fail) sm.action = kActDone;
            }
            __syncthreads();
            if (sm.action == kActDone) break;
        }
        if (tid == 0) { stops[l] = k.stop; iters[l] = k.iters; evals[l] = k.evals; }
        __syncthreads();
        if (l > 0)
            for (int j = tid; j < held; j += kThreads) c[j] = make_float2(2.f * c[j].x, 2.f * c[j].y);
    }
    // the result: every CTA its own rows; the mean displacement over all points
    float hi[2] = {0.f, 0.f}, lo[2] = {0.f, 0.f};
    float2 *o = p.node_grid + (size_t)Nc * op.out + (size_t)B.cr0 * G.nx;
    for (int j = tid; j < (B.own1 - B.cr0) * G.nx; j += kThreads) {
        const float2 v = c[(B.cr0 - B.h0) * G.nx + j];
        __stcg(o + j, v);
        ff_acc(hi[0], lo[0], v.x);
        ff_acc(hi[1], lo[1], v.y);
    }
    __threadfence();   // before the cluster's first CTA publishes the node
    cluster_reduce<2, false>(hi, lo, 0.f, sm, comm, cl);
    if (tid == 0 && rank == 0) {
        double *th = p.node_theta + 3 * op.out;
        th[0] = 0.0;
        th[1] = sm.tot[0] / Nc;
        th[2] = sm.tot[1] / Nc;
        OpStats &st = p.stats[op_index];
        st.i = op.ref;
        st.k = op.tmpl;
        for (int l = 0; l < kMaxLevels; ++l) {
            bool v = l < Lc;
            st.iters[l] = v ? iters[l] : 0;
            st.evals[l] = v ? evals[l] : 0;
            st.stop[l] = v ? stops[l] : 0;
        }
        st.rejects = k.rejects;
        st.status = sm.fail;
        st.energy = k.E;
        st.theta[0] = th[0]; st.theta[1] = th[1]; st.theta[2] = th[2];
    }
}

// ================================================================== kernels
// Mock operator (Sec. 5.1): the two input values are added after a spin of the operator's given
// duration on %globaltimer (at most 100 ms, and a bounded number of sleeps), as the paper's
// artificial operator of fixed or exponentially distributed running time.  left < 0 is the
// identity (0), which the exclusive Blelloch scan feeds in.
__device__ void run_mock(const Params &p, const OpDesc &op, int op_index, const cg::cluster_group &cl)
{
    if (threadIdx.x != 0 || cl.block_rank() != 0) return;
    const double a = op.left >= 0 ? __ldcg(p.node_theta + 3 * op.left) : 0.0;
    const double b = __ldcg(p.node_theta + 3 * op.right);
    const long long dur = (long long)(fminf(fmaxf(p.mock_us[op_index], 0.f), 1.0e5f) * 1000.0f);
    unsigned long long t0, t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t0));
    for (int it = 0; it < (1 << 24); ++it) {
        asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
        if ((long long)(t - t0) >= dur) break;
        __nanosleep(100);
    }
    __stcg(p.node_theta + 3 * op.out, a + b);
    OpStats &st = p.stats[op_index];
    st.i = op.ref;
    st.k = op.tmpl;
    st.status = kDevOk;
    st.energy = a + b;
}

__device__ bool op_valid(const Params &p, const OpDesc &op)
{
    if (p.cfg.mode == kModeMock) {
        auto ok = [&](int n) { return n >= 0 && n < p.n_nodes; };
        return ok(op.out) && ok(op.right) && (op.left < 0 || ok(op.left));
    }
    auto node_ok = [&](int n) { return n >= 0 && n < p.n_nodes; };
    if (p.cfg.mode == REG_NONRIGID && p.cfg.metric == REG_METRIC_H1 && !p.h1q) return false;
    if (op.ref < 0 || op.ref >= p.n_frames || op.tmpl < 0 || op.tmpl >= p.n_frames) return false;
    if (!node_ok(op.out)) return false;
    if (op.left >= 0 && !(node_ok(op.left) && node_ok(op.right))) return false;
    if (op.left < 0 && op.init_node >= 0 && !node_ok(op.init_node)) return false;
    return true;
}

template <int MODE, typename S, int U>
__device__ void run_op(const Params &p, int op_index, Smem &sm, float2 *gbuf, Comm &comm, const cg::cluster_group &cl)
{
    const OpDesc op = p.ops[op_index];
    if (!op_valid(p, op)) {
        if (threadIdx.x == 0 && cl.block_rank() == 0) {
            p.stats[op_index].status = kDevBadOp;
            atomicCAS(p.status, 0, (int)kDevBadOp);
        }
        return;
    }
    if constexpr (MODE == REG_RIGID) run_rigid<S>(p, op, op_index, sm, comm, cl);
    else if constexpr (MODE == kModeMock) run_mock(p, op, op_index, cl);
    else run_nonrigid<S, U / 2>(p, op, op_index, sm, gbuf, comm, cl);
    if constexpr (MODE != kModeMock) {
        if (threadIdx.x == 0 && sm.fail) atomicCAS(p.status, 0, sm.fail);
    }
}

// Batched launch: cluster q of the grid runs operator op_base + q.  MINB: CTAs per SM the register
// budget is sized for.  The nonrigid kernels take 128 registers a thread, two CTAs per SM: at 80 (three
// CTAs) the pass spills in its pixel loop, and a scan of 1,024 frames of 512x512 took 97 ms instead of
// 76 (8 CTAs per operator).  U: pixels in flight per lane in the nonrigid passes (2 or 4, the tile shape
// reg_autotune chooses): two columns of one or two rows.
template <int MODE, typename S, int MINB, int U = 4>
__global__ void __launch_bounds__(kThreads, MINB) op_kernel(const __grid_constant__ Params p)
{
    __shared__ Smem sm;
    extern __shared__ __align__(16) float2 gbuf[];   // nonrigid: grid_layout
    cg::cluster_group cl = cg::this_cluster();
    Comm comm{0};
    if (threadIdx.x == 0) comm_init(sm, p, cl);
    cl.sync();   // every CTA's barriers are set before a peer sends
    const int q = blockIdx.x / cl.num_blocks();
    run_op<MODE, S, U>(p, p.op_base + q, sm, gbuf, comm, cl);
    cl.sync();   // no CTA leaves while a peer may still send to it
}

// Persistent launch: each cluster claims ready operators from the device queue
// until all n_ops have been claimed.  Every wait is bounded by queue.timeout_ns.
template <int MODE, typename S, int MINB, int U = 4>
__global__ void __launch_bounds__(kThreads, MINB) persistent_kernel(const __grid_constant__ Params p)
{
    __shared__ Smem sm;
    extern __shared__ __align__(16) float2 gbuf[];
    cg::cluster_group cl = cg::this_cluster();
    const bool leader = cl.block_rank() == 0 && threadIdx.x == 0;
    Comm comm{0};
    if (threadIdx.x == 0) comm_init(sm, p, cl);   // before the cluster barriers of the first claim
    for (;;) {
        if (leader) {
            // claim the first ready operator of the most urgent non-empty class; every operator
            // claimed (all classes): leave.  Waiting for work gives up after queue.timeout_ns
            // without any operator finishing; the wait for a claimed slot's writer is bounded too.
            const Queue &Q = p.queue;
            volatile int *vh = Q.head, *vt = Q.tail, *vs = Q.slots, *vc = Q.claimed, *vd = Q.done;
            unsigned long long start;
            asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(start));
            unsigned ns = 64;
            int op = -1, seen = *vd;
            // the wait has run out once timeout_ns passed with no operator finishing (the finished
            // count is read only then, so spinning workers do not crowd its line), or on an error
            auto wait_expired = [&](unsigned long long now) {
                if (*((volatile int *)p.status) != 0) return true;
                if ((long long)(now - start) <= Q.timeout_ns) return false;
                const int dn = *vd;
                if (dn == seen) return true;
                seen = dn;
                start = now;
                return false;
            };
            // the mock operator's kernel keeps to the FIFO (the class scan's registers would halve its
            // resident CTAs)
            constexpr bool kClassQueue = MODE != kModeMock;
            if (!kClassQueue || Q.n_class == 1) {
                // one class, a plain FIFO: take a ticket, then wait for that slot to be written (the
                // form for short operators, where polling every class's head would crowd one line)
                const int slot = atomicAdd(Q.head, 1);
                while (slot < p.n_ops && (op = vs[slot]) < 0) {
                    unsigned long long now;
                    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(now));
                    if (wait_expired(now)) {
                        atomicCAS(p.status, 0, (int)kDevQueueTimeout);
                        op = -2;
                        break;
                    }
                    __nanosleep(ns);
                    if (ns < 1024) ns *= 2;
                }
            }
            for (; kClassQueue && Q.n_class > 1;) {
                if (*vc >= p.n_ops) break;
                // every class's head and tail in one round of loads; the first class with a ready
                // operator is claimed by a compare-and-swap on its head, which never passes the tail
                // (with a plain addition, workers that lost a race sat on slots that a later release
                // of that class fills, while ready operators of other classes waited for a worker: the
                // B operators of 4,096 frames of 512x512 on 4 CTAs took 360 ms, in one run of ten 450 to
                // 880)
                int hs[kQueueClasses], ts[kQueueClasses];
#pragma unroll
                for (int c = 0; c < kQueueClasses; ++c) hs[c] = c < Q.n_class ? vh[c] : 0;
#pragma unroll
                for (int c = 0; c < kQueueClasses; ++c) ts[c] = c < Q.n_class ? vt[c] : 0;
                int slot = -1;
#pragma unroll
                for (int c = 0; c < kQueueClasses; ++c)
                    for (int h = hs[c]; slot < 0 && h < ts[c];) {
                        const int was = atomicCAS(Q.head + c, h, h + 1);
                        if (was == h) slot = Q.class_off[c] + h;
                        h = was;
                    }
                if (slot >= 0) {
                    atomicAdd(Q.claimed, 1);
                    // the releaser bumps the tail before it writes the slot
                    while ((op = vs[slot]) < 0) {
                        unsigned long long now;
                        asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(now));
                        if (wait_expired(now)) {
                            atomicCAS(p.status, 0, (int)kDevQueueTimeout);
                            op = -2;
                            break;
                        }
                        __nanosleep(32);
                    }
                    break;
                }
                unsigned long long now;
                asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(now));
                if (wait_expired(now)) {
                    atomicCAS(p.status, 0, (int)kDevQueueTimeout);
                    op = -2;
                    break;
                }
                __nanosleep(ns);
                if (ns < 256) ns *= 2;   // at 1,024 a rigid scan of 128 frames of 512x512 takes 1 % longer
            }
            __threadfence();
            sm.idata[1] = op;
        }
        cl.sync();
        const int op = *cl.map_shared_rank(&sm.idata[1], 0);
        cl.sync();
        if (op < 0) break;
        run_op<MODE, S, U>(p, op, sm, gbuf, comm, cl);
        cl.sync();
        if (cl.block_rank() == 0) {
            // publish the produced node and release its consumers, spread over the CTA's threads (a
            // node of a Ladner-Fischer scan has up to n/2 consumers); the lanes of a warp that make
            // consumers of one class ready claim their slots with one atomic on that class's tail
            const int node = p.ops[op].out;
            const int cb = p.queue.cons_start[node], ce = p.queue.cons_start[node + 1];
            const int lane = threadIdx.x & 31;
            // only warps with consumers take part (most nodes have one or two: warp 0 alone); each
            // orders the cluster's writes of the node, seen through cl.sync, before its releases
            if (cb + (int)(threadIdx.x & ~31) < ce) __threadfence();
            for (int base = cb + (int)(threadIdx.x & ~31); base < ce; base += kThreads) {
                const int e = base + lane;
                int c = -1;
                bool ready = false;
                if (e < ce) {
                    c = p.queue.consumers[e];
                    ready = atomicSub(p.queue.pending + c, 1) == 1;
                }
                if (__ballot_sync(0xffffffffu, ready)) {
                    // lanes releasing into the same class take consecutive slots of it
                    const int cls = ready ? p.queue.op_class[c] : -1;
                    const unsigned grp = __match_any_sync(0xffffffffu, cls);
                    if (ready) {
                        const int first = __ffs(grp) - 1;
                        int t0 = 0;
                        if (lane == first) t0 = atomicAdd(p.queue.tail + cls, __popc(grp));
                        t0 = __shfl_sync(grp, t0, first);
                        atomicExch(p.queue.slots + p.queue.class_off[cls] + t0 + __popc(grp & ((1u << lane) - 1)), c);
                    }
                }
            }
            if (threadIdx.x == 0) atomicAdd(p.queue.done, 1);
        }
    }
    cl.sync();
}

// Energy/gradient at a given deformation for a single pair, on one cluster of kEnergyCtas CTAs that
// split the rows as the operator's do.  It is bound by latency: one pass over the pair, and the call's
// launches.  A call took 801 us for 512x512 (nonrigid) with a single CTA, 126 with 16 in two passes, and takes 79.
// Rigid: theta (device) -> out[0] = E, out[1..3] = dE/dtheta.  Nonrigid: control values cgrid
// (finest px, level 0) -> out[0] = E and grad_c = dE/dc.
template <int MODE, typename S>
__global__ void __launch_bounds__(kThreads) energy_kernel(const __grid_constant__ Params p, const double *theta, const float2 *cgrid,
                                                          double *out, float2 *grad_c)
{
    __shared__ Smem sm;
    extern __shared__ __align__(16) float2 gbuf[];
    cg::cluster_group cl = cg::this_cluster();
    const int tid = threadIdx.x;
    const Lvl L = level_of(p, 0, 1, 0);
    const int C = cl.num_blocks(), rank = cl.block_rank();
    const bool first = tid == 0 && rank == 0;
    Comm comm{0};
    if (tid == 0) comm_init(sm, p, cl);
    cl.sync();
    if constexpr (MODE == REG_RIGID) {
        RigidCtl &k = sm.rctl;
        if (tid == 0) {
            memset(&k, 0, sizeof(k));
            set_level(k.ls, L.W, L.H, L.gam);
        }
        if (tid < 32) rigid_param(theta[min(tid, 2)], min(tid, 2), tid, sm.pm);
        __syncthreads();
        int r0, r1;
        strip_rows(L.H, rank, C, r0, r1);
        float pm[6];
        for (int q = 0; q < 6; ++q) pm[q] = sm.pm[q];
        rigid_pass<S, true>(L, r0, r1, pm, sm, comm, cl);
        if (first) {
            set_reference(k.ls, sm.tot[3], sm.tot[4]);
            const Ncc n = ncc_terms(k.ls, sm.tot[0], sm.tot[1], sm.tot[2]);
            out[0] = n.e;
            for (int q = 0; q < 3; ++q) out[1 + q] = rigid_gradient(k.ls, n, sm.tot, q);
        }
    } else {
        const Grid G{p.gnx, p.gny, p.gs};
        const int Nc = G.nx * G.ny;
        const GridLayout lay = grid_layout(G.nx, G.ny, C, false);
        const Band B = grid_band(G, rank, C);
        const PointIter pi(G.nx);
        float2 *c = gbuf + lay.c, *d = gbuf + lay.d, *mt = gbuf + lay.mt, *halo = gbuf + lay.halo;
        float *slots = (float *)(gbuf + lay.slots);
        const float *above = (const float *)(gbuf + lay.above);
        float *emits = (float *)(gbuf + lay.emits);
        for (int j = tid; j < (B.h1 - B.h0) * G.nx; j += kThreads) {
            c[j] = cgrid[B.h0 * G.nx + j];
            d[j] = make_float2(0.f, 0.f);
            mt[j] = make_float2(1.f, 1.f);
        }
        __syncthreads();
        const GridLvl GL = grid_level(G, L, 0);
        const PassGeom &P = level_geom(sm, p, 0, L.W > (G.nx - 1) * G.s);
        __syncthreads();
        grid_pass<S, true, 2>(L, G, GL, P, B, c, d, 0.f, slots, above, emits, pi, sm, comm, cl);
        FieldCtl &k = sm.fctl;
        if (tid == 0) {
            set_level(k.ls, L.W, L.H, L.gam);
            set_reference(k.ls, sm.tot[3], sm.tot[4]);
            const Ncc n = ncc_terms(k.ls, sm.tot[0], sm.tot[1], sm.tot[2]);
            if (first) out[0] = __fma_rn(0.5 * p.cfg.lambda * k.ls.invP, sm.tot[5], n.e);
            field_grad_params(n, k.ls, p.cfg, sm.pm);
        }
        __syncthreads();
        if (grad_c) {
            float pm[4];
            for (int q = 0; q < 4; ++q) pm[q] = sm.pm[q];
            grid_direction<true>(G, L, P, B, c, d, mt, halo, slots, above, pi, pm, sm, comm, cl, H1Bufs{});
            // d = -Nc dE/dc (unit scalar product)
            const double s = -1.0 / (double)Nc;
            const float2 *own = d + (B.cr0 - B.h0) * G.nx;
            for (int j = tid; j < (B.own1 - B.cr0) * G.nx; j += kThreads)
                grad_c[B.cr0 * G.nx + j] = make_float2((float)(s * (double)own[j].x), (float)(s * (double)own[j].y));
        }
    }
    if (tid == 0 && sm.fail) atomicCAS(p.status, 0, sm.fail);
    cl.sync();   // no CTA leaves while a peer may still send to it
}

// Composition of two control grids at the control points (standalone entry point).
__global__ void grid_compose_kernel(const float2 *q1, const float2 *q2, Grid G, float2 *out)
{
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= G.nx * G.ny) return;
    const int jy = j / G.nx, jx = j - jy * G.nx;
    const float2 a = q1[j];
    const float2 u = grid_eval_global(q2, G, (float)(jx * G.s) + a.x, (float)(jy * G.s) + a.y);
    out[j] = make_float2(a.x + u.x, a.y + u.y);
}

// Dense finest-level fields [2][H][W] of control grids (grid nodes[blockIdx.z]), four pixels per
// thread written with one float4 store per plane where the row allows it.
__global__ void grid_dense_kernel(const float2 *grids, const int *nodes, Grid G, int W, int H, float *out)
{
    const int Nc = G.nx * G.ny;
    const float2 *q = grids + (size_t)Nc * nodes[blockIdx.z];
    float *ox = out + (size_t)blockIdx.z * 2 * W * H, *oy = ox + (size_t)W * H;
    const int r = blockIdx.y, c0 = 4 * (blockIdx.x * blockDim.x + threadIdx.x);
    if (c0 >= W) return;
    float vx[4], vy[4];
#pragma unroll
    for (int t = 0; t < 4; ++t) {
        const float2 u = grid_eval_global(q, G, (float)min(c0 + t, W - 1), (float)r);
        vx[t] = u.x;
        vy[t] = u.y;
    }
    const size_t i = (size_t)r * W + c0;
    if (c0 + 3 < W && (((size_t)(ox + i) | (size_t)(oy + i)) & 15) == 0) {
        __stcs((float4 *)(ox + i), make_float4(vx[0], vx[1], vx[2], vx[3]));
        __stcs((float4 *)(oy + i), make_float4(vy[0], vy[1], vy[2], vy[3]));
    } else {
        for (int t = 0; t < 4 && c0 + t < W; ++t) { ox[i + t] = vx[t]; oy[i + t] = vy[t]; }
    }
}

// Control values sampled from a dense finest-level field [2][H][W] (clamped at the border).
__global__ void grid_from_dense_kernel(const float *u, int W, int H, Grid G, float2 *out)
{
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= G.nx * G.ny) return;
    const int jy = j / G.nx, jx = j - jy * G.nx;
    const int x = min(jx * G.s, W - 1), y = min(jy * G.s, H - 1);
    out[j] = make_float2(u[(size_t)y * W + x], u[(size_t)W * H + (size_t)y * W + x]);
}

// ================================================================== host launchers
// Dynamic shared memory of the nonrigid kernels (layout of grid_layout).
static size_t set_geometry(Params &p, int cluster, bool exact = false)
{
    if (p.cfg.mode != REG_NONRIGID) return 0;
    const bool h1 = p.cfg.metric == REG_METRIC_H1;
    const GridLayout lay = grid_layout(p.gnx, p.gny, cluster, h1);
    size_t slots = h1 ? sizeof(float2) * 2 * (size_t)p.gnx * p.gny : 0;
    for (int l = 0; l < p.cfg.levels; ++l)
        for (const bool over : {false, true}) {   // the frame's width decides, which is not known here
            const PassGeom P = pass_geom(p.gs >> l, p.gnx - 1, band_cells(p.gny, cluster), over, slot_room(lay), exact);
            p.geom[l][over] = P;
            slots = std::max(slots, sizeof(float) * slot_floats(P));
        }
    return sizeof(float2) * (size_t)lay.slots + slots;
}
static size_t grid_smem(const Params &p, int cluster)
{
    Params q = p;
    return set_geometry(q, cluster);
}

// The largest grids do not fit the few CTAs of a small cluster: from the size asked for, the first
// whose control state and slots leave room for the static part.
int fit_cluster(const Params &p, int cluster)
{
    while (cluster < kMaxCluster && grid_smem(p, cluster) > (size_t)kMostSmem) cluster *= 2;
    return cluster;
}

// Limit of an exchange's wait, two seconds: the CTAs of a cluster run side by side, and a pass over the largest
// frame takes milliseconds.  Host-side fault injection for tests: REG_FAULT_INJECT=mute_cta keeps an operator's
// last CTA from sending, so that the waits run out; REG_EXCHANGE_TIMEOUT_MS shortens them.
void set_exchange_limits(Params &p)
{
    p.wait_ns = 2000000000LL;
    if (const char *t = getenv("REG_EXCHANGE_TIMEOUT_MS")) {
        const long long ms = atoll(t);
        if (ms > 0) p.wait_ns = ms * 1000000LL;
    }
    const char *inj = getenv("REG_FAULT_INJECT");
    p.mute = inj && strcmp(inj, "mute_cta") == 0;
}

template <typename K>
static cudaError_t launch_cluster(K kernel, int blocks, int cluster, cudaStream_t s, Params p)
{
    set_exchange_limits(p);
    if (cluster > 8) {
        cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        if (e != cudaSuccess) return e;
    }
    const size_t smem = set_geometry(p, cluster);
    if (smem > 0) {
        cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    cudaLaunchConfig_t lc = {};
    lc.gridDim = dim3(blocks);
    lc.blockDim = dim3(kThreads);
    lc.dynamicSmemBytes = smem;
    lc.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = cluster;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    lc.attrs = attr;
    lc.numAttrs = 1;
    return cudaLaunchKernelEx(&lc, kernel, p);
}

typedef void (*OpKernelFn)(Params);

// The nonrigid kernel for a storage type, launch form and energy-pass unroll.
template <typename S>
static OpKernelFn nonrigid_fn(bool persistent, int unroll)
{
    if (persistent) return unroll == 2 ? persistent_kernel<REG_NONRIGID, S, 2, 2> : persistent_kernel<REG_NONRIGID, S, 2, 4>;
    return unroll == 2 ? op_kernel<REG_NONRIGID, S, 2, 2> : op_kernel<REG_NONRIGID, S, 2, 4>;
}

static OpKernelFn nonrigid_kernel(int storage, bool persistent, int unroll)
{
    switch (storage) {
    case REG_F32: return nonrigid_fn<float>(persistent, unroll);
    case REG_BF16: return nonrigid_fn<__nv_bfloat16>(persistent, unroll);
    case REG_F16: return nonrigid_fn<__half>(persistent, unroll);
    }
    return nullptr;
}

cudaError_t launch_ops(const Params &p, int storage, int cluster, int n_launch_ops, cudaStream_t s)
{
    const int blocks = n_launch_ops * cluster;
    if (p.cfg.mode == kModeMock) return launch_cluster(op_kernel<kModeMock, float, 8>, blocks, cluster, s, p);
    if (p.cfg.mode == REG_RIGID) {
        switch (storage) {
        case REG_F32: return launch_cluster(op_kernel<REG_RIGID, float, 2>, blocks, cluster, s, p);
        case REG_BF16: return launch_cluster(op_kernel<REG_RIGID, __nv_bfloat16, 2>, blocks, cluster, s, p);
        case REG_F16: return launch_cluster(op_kernel<REG_RIGID, __half, 2>, blocks, cluster, s, p);
        }
    } else {
        OpKernelFn k = nonrigid_kernel(storage, false, p.unroll);
        if (k) return launch_cluster(k, blocks, cluster, s, p);
    }
    return cudaErrorInvalidValue;
}

cudaError_t launch_persistent(const Params &p, int storage, int cluster, int workers, cudaStream_t s)
{
    const int blocks = workers * cluster;
    if (p.cfg.mode == kModeMock) return launch_cluster(persistent_kernel<kModeMock, float, 8>, blocks, cluster, s, p);
    if (p.cfg.mode == REG_RIGID) {
        switch (storage) {
        case REG_F32: return launch_cluster(persistent_kernel<REG_RIGID, float, 2>, blocks, cluster, s, p);
        case REG_BF16: return launch_cluster(persistent_kernel<REG_RIGID, __nv_bfloat16, 2>, blocks, cluster, s, p);
        case REG_F16: return launch_cluster(persistent_kernel<REG_RIGID, __half, 2>, blocks, cluster, s, p);
        }
    } else {
        OpKernelFn k = nonrigid_kernel(storage, true, p.unroll);
        if (k) return launch_cluster(k, blocks, cluster, s, p);
    }
    return cudaErrorInvalidValue;
}

template <typename K>
static int resident_clusters(K kernel, int cluster, const Params &p)
{
    if (cluster > 8 && cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess)
        return -1;
    const size_t smem = grid_smem(p, cluster);
    if (smem > 0 && cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
        return -1;
    cudaLaunchConfig_t lc = {};
    lc.gridDim = dim3(cluster);
    lc.blockDim = dim3(kThreads);
    lc.dynamicSmemBytes = smem;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = cluster;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    lc.attrs = attr;
    lc.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, kernel, &lc) != cudaSuccess) return -1;
    return n;
}

int persistent_resident_clusters(const Params &p, int storage, int cluster)
{
    int n = -1;
    if (p.cfg.mode == kModeMock) {
        n = resident_clusters(persistent_kernel<kModeMock, float, 8>, cluster, p);
    } else if (p.cfg.mode == REG_RIGID) {
        switch (storage) {
        case REG_F32: n = resident_clusters(persistent_kernel<REG_RIGID, float, 2>, cluster, p); break;
        case REG_BF16: n = resident_clusters(persistent_kernel<REG_RIGID, __nv_bfloat16, 2>, cluster, p); break;
        case REG_F16: n = resident_clusters(persistent_kernel<REG_RIGID, __half, 2>, cluster, p); break;
        }
    } else {
        OpKernelFn k = nonrigid_kernel(storage, true, p.unroll);
        if (k) n = resident_clusters(k, cluster, p);
    }
    if (n < 0) cudaGetLastError();
    return n;
}

cudaError_t launch_energy(const Params &params, int storage, const double *theta_dev, const float2 *grid_dev,
                          double *out_dev, float2 *grad_dev, cudaStream_t s)
{
    (void)storage;
    constexpr int kEnergyCtas = kMaxCluster;
    Params p = params;
    set_exchange_limits(p);
    const void *kern = p.cfg.mode == REG_RIGID ? (const void *)energy_kernel<REG_RIGID, float>
                                               : (const void *)energy_kernel<REG_NONRIGID, float>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
    const size_t smem = set_geometry(p, kEnergyCtas, true);
    if (smem > 0) {
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    cudaLaunchConfig_t lc = {};
    lc.gridDim = dim3(kEnergyCtas);
    lc.blockDim = dim3(kThreads);
    lc.dynamicSmemBytes = smem;
    lc.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = kEnergyCtas;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    lc.attrs = attr;
    lc.numAttrs = 1;
    if (p.cfg.mode == REG_RIGID)
        return cudaLaunchKernelEx(&lc, energy_kernel<REG_RIGID, float>, p, theta_dev, grid_dev, out_dev, grad_dev);
    return cudaLaunchKernelEx(&lc, energy_kernel<REG_NONRIGID, float>, p, theta_dev, grid_dev, out_dev, grad_dev);
}

cudaError_t launch_grid_compose(const float2 *q1, const float2 *q2, int nx, int ny, int spacing, float2 *out,
                                cudaStream_t s)
{
    const int Nc = nx * ny;
    grid_compose_kernel<<<(Nc + 127) / 128, 128, 0, s>>>(q1, q2, Grid{nx, ny, spacing}, out);
    return cudaGetLastError();
}

cudaError_t launch_grid_dense(const float2 *grids, const int *nodes, int n, int nx, int ny, int spacing, int W,
                              int H, float *out, cudaStream_t s)
{
    if (n <= 0) return cudaSuccess;
    dim3 grid((W / 4 + 1 + 63) / 64, H, n);
    grid_dense_kernel<<<grid, 64, 0, s>>>(grids, nodes, Grid{nx, ny, spacing}, W, H, out);
    return cudaGetLastError();
}

cudaError_t launch_grid_from_dense(const float *u, int W, int H, int nx, int ny, int spacing, float2 *out,
                                   cudaStream_t s)
{
    const int Nc = nx * ny;
    grid_from_dense_kernel<<<(Nc + 127) / 128, 128, 0, s>>>(u, W, H, Grid{nx, ny, spacing}, out);
    return cudaGetLastError();
}

int max_cluster_size() { return 16; }

}  // namespace reg
