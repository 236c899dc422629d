// Internal declarations shared by the kernel and host translation units of libreg.
#pragma once

#include <cstddef>
#include <cstdint>

#include <cuda_runtime.h>

#include "../../include/reg.h"

namespace reg {

constexpr int kMaxLevels = REG_MAX_LEVELS;
constexpr int kThreads = 256;          // threads per CTA of the operator kernels

// One pyramid level of one frame, as the operator kernels read it.
struct LevelDesc {
    const void *ptr;    // template role: storage-typed samples, row-major, pixel (0, 0)
    const void *rptr;   // reference role: the same samples (rigid model) or the B-spline model
                        // at the pixel centres (nonrigid model)
    int W, H, pitch;    // pitch of ptr, in elements
    int rpitch;         // pitch of rptr, in elements
    float mean, sd;     // the level's (LevelStat)
};

// Mean of a level's samples, the shift constant of its moment sums, and their standard deviation, which only
// scales one image to the other where the sums are formed (a few digits do).
struct LevelStat {
    float mean, sd;
};

// Pyramid layout.  The nonrigid model samples the quadratic B-spline of a level's samples
// extended by the level's mean; storing every level of that model with a border of kPad samples
// holding the mean lets a 3x3 tap window at a nearest sample clamped to [-2, W + 1] x [-2, H + 1]
// read without per-tap clamps and still equal the mean-extended model everywhere.
constexpr int kPad = 3;
inline int level_pitch(int W, int pad) { return W + 2 * pad; }
inline size_t level_elems(int W, int H, int pad) { return (size_t)(W + 2 * pad) * (H + 2 * pad); }
inline size_t level_origin(int W, int pad) { return (size_t)pad * (W + 2 * pad) + pad; }

// Where launch_pyramid writes the levels of frame 0 (frame f at + f * stride elements).
struct PyrOut {
    void *raw[kMaxLevels];            // start of level l's block (border included)
    size_t raw_stride[kMaxLevels];
    void *smooth[kMaxLevels];         // B-spline model at the pixel centres, W_l x H_l, or null
    size_t smooth_stride[kMaxLevels];
    int pad;                          // 0, or kPad border samples (the level's mean) around each level
};

// One operator application.  left < 0: A(f_ref, f_tmpl) from the identity (or
// from `init_node` when >= 0); otherwise B(node[left], node[right]).
struct OpDesc {
    int ref, tmpl;     // frame indices
    int left, right;   // input nodes of B, -1 for A
    int out;           // node written
    int init_node;     // A only: node holding the initial deformation, -1 = identity
};

// Per-operator record written by the device (mirrors reg_stats_t).
struct OpStats {
    int32_t i, k;
    int32_t iters[kMaxLevels], evals[kMaxLevels], stop[kMaxLevels];
    int32_t rejects, status;
    double energy;
    double theta[3];
};
static_assert(sizeof(OpStats) == sizeof(reg_stats_t), "stats layout");

// Device-side error codes in OpStats::status and the kernel status word.
enum DevStatus : int32_t {
    kDevOk = 0,
    kDevBadOp = 1,       // operator descriptor out of range / non-adjacent
    kDevQueueTimeout = 2, // bounded wait on the ready queue gave up
    kDevWaitTimeout = 3   // bounded wait on an mbarrier (TMA load, cluster exchange) gave up
};

// Operator model of a launch beyond REG_RIGID / REG_NONRIGID: the mock operator of reg_mock_scan.
constexpr int kModeMock = 2;

struct Config {
    int mode, levels, max_iter, max_rejects;
    double tol_grad, tol_rel_e, armijo_c, tau0, step_cap, lambda;
    int metric;   // nonrigid scalar product: REG_METRIC_MEAN, REG_METRIC_GAUSS_NEWTON or REG_METRIC_H1
    double sigma; // REG_METRIC_H1: smoothing length in control-grid spacings
    double tol_coarse;   // factor on tol_grad at every level above the finest
};

// Ready-queue state of the persistent executor (device memory): one FIFO per priority class,
// class 0 first.  An operator's class is its rank by bottom level (the longest estimated path
// from it to the end of the DAG), so operators on long chains start before ones with slack.
constexpr int kQueueClasses = 16;
struct Queue {
    int *head;         // [kQueueClasses] next slot to claim in each class
    int *tail;         // [kQueueClasses] next slot to fill in each class
    int *slots;        // class c at slots[class_off[c] ...]: op indices in ready order, -1 = not yet filled
    const int *op_class;   // per op: its class
    const int *class_off;  // [kQueueClasses + 1] first slot of each class, then the slot count
    int *pending;      // per op: inputs not yet produced
    int *consumers;    // CSR list of ops consuming each node
    int *cons_start;   // [n_nodes + 1]
    int *done;         // number of finished ops
    int *claimed;      // number of claimed ops, all classes
    int n_class;       // classes in use (1: a plain FIFO)
    long long timeout_ns;
};

// How a pass splits a band's pixels among the warps.  A strip is up to 32 columns: those of g whole cells
// (32 / sl of them, sl the cell width at the level), or from 32 columns a cell on a chunk of one cell; a
// column past the last cell, which a frame of 2^k + 1 columns has, is a strip of its own.  A warp's
// task is two neighbouring strips, a column of each per lane, over the rows of a segment: m cell
// rows, or one h-th of a cell row.  Every strip of every segment has slots of its own for its sums
// (m + 1 control rows of g + 1 points, 8 floats each), so no two warps add to one place and the
// order is fixed.  Long segments are best (a control row inside one is reduced over the lanes once, not
// twice), short ones where there are too few strips for the warps: the rule takes the least number of
// rounds x (pixel rows + about two rows' time per reduction) of the splits whose slots fit `room`
// floats.  Where none does (thousands of chunks), a task is one wide cell, whose chunks a warp walks
// two at a time and adds up in one strip's slots.
struct PassGeom {
    int sl, g, chunks;    // cell width, cells per strip, strips per cell (wide cells)
    int ns, nst;          // strips of cells with slots, strips with slots
    int sch;              // strips with slots per wide cell: chunks, or 1 where a task walks them
    int past;             // the strip past the last cell, counting every chunk
    int tasks, walk;      // tasks of a segment; pairs of strips a task walks
    int m, h, ph;         // cell rows per segment, pieces per cell row (a power of two), pixel rows per piece
    int nseg, hlog;       // segments, log2 of h
    unsigned rm, rg;      // reciprocals for div31: of m and g
};

struct Params {
    Config cfg;
    const LevelDesc *levels;   // [n_frames][cfg.levels]
    int n_frames;
    const OpDesc *ops;
    int n_ops;
    int op_base;               // first op of this launch (batched launches)
    double *node_theta;        // [n_nodes][3]: rigid (alpha, Gx, Gy); nonrigid (0, mean c_x, mean c_y)
    float2 *node_grid;         // nonrigid: [n_nodes][gny * gnx] control values (finest px)
    const float *mock_us;      // mock operator (kModeMock): duration of each operator, microseconds
    const float *h1q;          // REG_METRIC_H1: the control grid's cosine bases and eigenvalues (Qx, Qy, lx, ly)
    int unroll;                // nonrigid passes: pixels in flight per lane (2 or 4; 0 = 4)
    int minb;                  // nonrigid register form as configured (3 or 4; 0 = 3); one kernel serves both
    int gnx, gny, gs;          // nonrigid control grid: points per axis and spacing (finest px)
    PassGeom geom[kMaxLevels][2];   // nonrigid, set at the launch: per level, without and with columns past the last cell
    int n_nodes;
    OpStats *stats;            // [n_ops]
    int *status;               // kernel status word (first device error)
    long long wait_ns;         // set at the launch: limit of a wait for the other CTAs of an operator,
    int mute;                  // and whether a test keeps an operator's last CTA from sending
    Queue queue;               // persistent executor only
};

// Launch shape of the operator kernels (0 = not chosen): CTAs per operator, pixels in flight per lane, and the
// register form as recorded.
struct TileShape {
    int cluster = 0, unroll = 0, minb = 0;
};

// Host launchers (reg_kernels.cu).
// Pyramids of N frames (frame f at frames + f * fstride, rows of `pitch`) into the layout `out`
// (storage-typed); means[f * levels + l] = those of level l of frame f (or null).
cudaError_t launch_pyramid(const float *frames, int N, size_t fstride, int W, int H, int pitch, int levels,
                           int storage, const PyrOut &out, LevelStat *means, cudaStream_t s);
// Kernel launches of one launch_pyramid call.
int pyramid_launches(int levels, bool means, int pad);
// Level table of a batch of frames: frame f's row l is that of frame 0, its pointers f strides on, with
// the level's mean and standard deviation.
struct LevelTable {
    int levels;
    const char *raw[kMaxLevels], *ref[kMaxLevels];         // pixel (0, 0) of frame 0, template and reference role
    size_t raw_stride[kMaxLevels], ref_stride[kMaxLevels]; // bytes between frames
    int W[kMaxLevels], H[kMaxLevels], pitch[kMaxLevels], rpitch[kMaxLevels];
};
cudaError_t launch_level_table(LevelDesc *tab, const LevelTable &t, const LevelStat *means, int frames, cudaStream_t s);

// What one pairwise call needs on the device besides its pyramids, in one block: the operator, its
// nodes (0 the result, 1 the initial guess), and what comes back to the host (through `status`).
struct PairBlock {
    OpStats stats;
    double theta[6];
    int status[4];
    OpDesc op;
    int node0;         // 0: the dense field is that of node 0
};
// Fill the block (statistics and status zero) and the level table of the call's two frames.
cudaError_t launch_pair_setup(PairBlock *b, const OpDesc &op, const double *init3, LevelDesc *tab, const LevelTable &t,
                              const LevelStat *means, cudaStream_t s);
// tab[l].mean and sd = means[l] for l < L (a slot's level table rows after its pyramid build).
cudaError_t launch_set_level_means(LevelDesc *tab, const LevelStat *means, int L, cudaStream_t s);
// CTAs per operator for a launch that asks for `cluster`: more where an operator's control grid does
// not fit the shared memory of so few.
int fit_cluster(const Params &p, int cluster);
// The launchers set wait_ns and mute by this; a caller that compares Params of two launches does so first.
void set_exchange_limits(Params &p);
cudaError_t launch_ops(const Params &p, int storage, int cluster, int n_launch_ops,
                       cudaStream_t s);
cudaError_t launch_persistent(const Params &p, int storage, int cluster, int workers,
                              cudaStream_t s);
// Clusters of `cluster` CTAs of the persistent kernel that fit on the device at once
// (occupancy query), or -1 if the query fails.
int persistent_resident_clusters(const Params &p, int storage, int cluster);

// Registered series (reg_warp): out_k = f_k o phi_{0,k} and their mean.
struct WarpJob {
    const float *frames;       // device [N][H][pitch]
    int N, W, H, pitch;
    int mode;
    const reg_elem_t *elems;   // rigid: N-1 device elements phi_{0,k}, k = 1..N-1
    const float2 *grids;       // nonrigid: N-1 device control grids [ny][nx]
    int nx, ny, s;
    float *out;                // device [N][H][W] or null
    float *mean;               // device [H][W] or null
    void *ws;                  // warp_workspace_bytes() of device memory
    int *status;               // device status word (kDevWaitTimeout on a timed-out load)
    long long timeout_ns;
};
size_t warp_workspace_bytes(int N, int W, int H, bool mean);
// *used_tma = 1 when the source boxes were staged by TMA (aligned frames, pitch % 4 == 0).
cudaError_t launch_warp(const WarpJob &j, cudaStream_t s, int *used_tma);
// dst (device) = bytes of src, host memory the device reads at the same address; both 16-byte
// aligned, bytes a multiple of 16 (else cudaErrorInvalidValue).  `blocks` CTAs of 256 threads.
cudaError_t launch_stage_copy(void *dst, const void *src, size_t bytes, int blocks, cudaStream_t s);
cudaError_t launch_grid_gather(const float2 *src, const int *nodes, int n, int Nc, float2 *dst, cudaStream_t s);
cudaError_t launch_energy(const Params &p, int storage, const double *theta_dev,
                          const float2 *grid_dev, double *out_dev, float2 *grad_dev,
                          cudaStream_t s);
cudaError_t launch_grid_compose(const float2 *q1, const float2 *q2, int nx, int ny, int spacing,
                                float2 *out, cudaStream_t s);
cudaError_t launch_grid_dense(const float2 *grids, const int *nodes, int n, int nx, int ny,
                              int spacing, int W, int H, float *out, cudaStream_t s);
cudaError_t launch_grid_from_dense(const float *u, int W, int H, int nx, int ny, int spacing,
                                   float2 *out, cudaStream_t s);
// Set the calling thread's message returned by reg_last_error_message().
void set_last_error(const char *msg);
int max_cluster_size();

}  // namespace reg
