// Internal definitions shared by the host API and the kernels of libmsqoc.
#pragma once

#include <cuda_runtime.h>
#include <cmath>
#include <cstdint>

namespace msqoc {

constexpr int MAXQ = 6;       // subsystems
constexpr int MAXEX = 15;     // exchange-coupled pairs (q (q - 1) / 2)
constexpr int MAXNF = 64;     // carriers over all subsystems
constexpr int MAXL = 4;       // levels per subsystem handled by the sweep kernels
constexpr int MAX_TILE_THREADS = 256;       // threads of a one-thread-per-fiber tile (255 registers a thread)
constexpr int MAX_LEAN_TILE_THREADS = 384;  // the same family compiled for 168 registers a thread: tiles of
                                            // up to 12 warps, or two 6-warp tiles on an SM
constexpr int MAX_PAIR_TILE_THREADS = 384;  // threads of a lane-pair tile (168 registers a thread)
constexpr int MAX_QUAD_TILE_THREADS = 384;  // threads of a lane-quad tile (168 registers a thread)
constexpr int MAX_HDEPTH = 8;               // steps per history group at most
// threads of any tile (host arrays of a tile's lane map are sized by it)
constexpr int MAX_ANY_TILE_THREADS = 384;
static_assert(MAX_TILE_THREADS <= MAX_ANY_TILE_THREADS && MAX_LEAN_TILE_THREADS <= MAX_ANY_TILE_THREADS &&
                  MAX_PAIR_TILE_THREADS <= MAX_ANY_TILE_THREADS && MAX_QUAD_TILE_THREADS <= MAX_ANY_TILE_THREADS,
              "a tile limit exceeds MAX_ANY_TILE_THREADS");

enum Solver { SOLVER_FP64 = 1, SOLVER_MIXED = 2 };

// device status word bits
enum Status { ST_OK = 0, ST_TIMEOUT = 1, ST_SOLVER_RANGE = 4 };

// Index of the first of the three quadratic B-splines (spacing dtau, d1 of them) active at time
// t, clamped to the grid.  The controls kernel and the host take it from here.
__host__ __device__ inline int spline_index(double t, double dtau, int d1) {
    const int s0 = static_cast<int>(floor(t / dtau));
    return s0 < 0 ? 0 : (s0 > d1 - 3 ? d1 - 3 : s0);
}

// Per-step table: first active spline index, the step solver's iteration counts packed as
// j1 | j2 << 8 | passes << 16 | out-of-range << 24, and the three spline weights.
struct __align__(16) Spline4 {
    int s;
    int cnt;
    double w0, w1, w2;
};

// Everything a kernel needs about one problem.  The small kernels take it by value; the sweep
// kernels read it from a device copy (several problems share a batched sweep launch).
struct ProbDev {
    // shape
    int q, L, N, E, F, ness, d1, M, nfsum, d;
    int m_off;     // global index of the first window minus one (0 unless the problem is a shard)
    int M_glob;    // windows of the whole problem (M for a whole problem; windows are local
                   // 1..M, global m_off + 1 .. m_off + M, on the whole problem's time grid)
    int cb;        // columns of a full tile
    int nthreads;  // threads per tile (multiple of 32)
    int pair;      // kernel family: log2 of the threads per fiber (0: one thread, 1: a lane pair,
                   // the real and the imaginary part; 2: a lane quad, a pair per entry of a
                   // 2-level fiber)
    int lean;      // one thread per fiber compiled for 168 registers (more warps per SM), pair = 0
    int ntiles;    // tiles of the problem's sweeps
    int glocal;    // doubles of a window's part of the alpha-gradient (its active splines with a
                   // margin of two, every carrier): enters the admission of tiles only
    int solver;
    int C;         // slices per window (1: a window is swept as a whole; see k_compose)
    int kseg;      // steps per history segment (checkpoint interval; >= the longest window when
                   // every midpoint state is kept)
    int nseg;      // segments per window: ceil(longest window / kseg)
    int kadj;      // steps per adjoint launch (a chunk of a segment; kseg when it is not cut)
    int nsub;      // chunks per segment: ceil(kseg / kadj)
    int hdepth;    // steps per history synchronisation: midpoint states staged and stored in
                   // groups of hdepth steps, one wait per group
    int64_t nsteps;
    double T, h, mu, dtau;
    double lam;    // ||a + a^+|| on L levels (bound of the ladder-term norm per unit |d|)
    int nf[MAXQ];
    int cof[MAXQ + 1];           // carrier offsets
    double omega[MAXNF];
    double sc[2 * MAXL];         // (h/2) sqrt(l+1) [dir +] and (h/2) sqrt(l) [dir -], index 2l+dir
    // dipole exchange J_jk (a_k^+ a_j + a_k a_j^+), j < k, a constant part of the off-diagonal
    // operator of the step: pairs, (h/2) J_jk, and its contribution to the contraction bound
    int nex;
    int ex_j[MAXEX], ex_k[MAXEX];
    double ex_c[MAXEX];
    double rho_ex;
    double kap;                  // max |(h/2) D_i| over the rows: the largest diagonal rotation of a step
    // constant tables
    const double2* P;            // [N] (1 + i h/2 D_i)^-1
    const int* emb;              // [E] full row index of essential column e
    const double2* V;            // [E][N] target
    // inputs of this evaluation (device memory)
    const double* alpha;         // [d]
    const double2* W;            // [M-1][E][N]; W + (m - 2) E N is the initial state of local
                                 // window m (a shard that starts past the first window reads its
                                 // first window's initial state at index -1)
    // scratch
    double2* ctrl;               // [nsteps][q] d_k(t_{n+1/2})
    float4* coef;                // [nsteps][q][L-1] (h/2) sqrt(j) d_k split into two floats (hi.x, hi.y,
                                 // lo.x, lo.y), j = 1 .. L-1; nullptr: the sweeps form it from ctrl
    Spline4* spl;                // [nsteps] (first spline index, solver counts, w0, w1, w2)
    double2* phase;              // [nsteps][nfsum] exp(i Omega t_{n+1/2})
    // sliced problems (C > 1): slice i of window m is virtual window m C + i (0-based) and every per-
    // window history below is per virtual window
    double2* Phi;                // [M C][N][N] propagators, column-major
    double2* Ubeg;               // [M C][E][N] states at the slices' starts
    double2* Lend;               // [M C][E][N] adjoint states at the slices' ends
    double2* hist;               // [M][kseg][E][N] midpoint states Ubar of one segment of every window
                                 // (the mixed solver's one-thread families store each entry as the
                                 // two-float split of Ubar 2^-hsh, hsh the column's scale exponent)
    int* hsh;                    // [M][nseg][E] column scale exponent of each window segment's
                                 // history (mixed solver, one thread per fiber), after hist
    double2* lhist;              // [M][kadj][E][N] adjoint midpoint states Lbar of one chunk of every
                                 // window, in the form of hist
    int* lsh;                    // [M][E] their column scale exponents, after lhist
    double2* quad;               // [q][nsteps] the step's gradient products (A_k, B_k) of every step
                                 // (msqoc_quad.cuh)
    double2* ckpt;               // [M][nseg][E][N] states at the segment starts (kseg < longest window)
    double2* Uend;               // [M][E][N] U^m(t_m)
    double2* Lterm;              // [M][E][N] Lambda^m(t_m)
    double2* Lam0;               // [M][E][N] Lambda^m(t_{m-1})
    double2* Lstate;             // [M C][E][N] adjoint state between launches (chunks, segments)
    double* term;                // [M] pen_m (m < M), J (m = M)
    int* status;                 // status word (ST_* bits)
};

// One sweep tile (one CTA): `ncol` consecutive columns of problem `prob` in window-major column
// order, starting at column c0 of window m0 (1-based).  The first `ncol0` columns belong to
// window m0, the rest to window m0 + 1 (a tile covers at most two windows).  `map` selects the
// thread -> (column, fiber) assignment in the launch's lane maps.
struct Tile {
    int prob, m0, c0, ncol, ncol0, map, pad[2];
};

// What a sweep launch does.
enum SweepMode {
    SWEEP_OBJECTIVE = 0,  // forward over whole windows; end states U^m(t_m)
    SWEEP_HISTORY = 1,    // forward over whole windows for a gradient; also every midpoint state
                          // (a problem with one history segment) or the states at the segment
                          // starts (checkpoints, more segments)
    SWEEP_RECOMPUTE = 3,  // forward over segment `seg` from its checkpoint; midpoint states
                          // (no work for a problem with one segment)
    SWEEP_ADJOINT = 4,    // adjoint over chunk `sub` of segment `seg`; its midpoint states
    SWEEP_PROP = 5,       // forward over every slice from the N unit vectors: its propagator
                          // (one thread per fiber)
    SWEEP_BOTH = 6        // SWEEP_HISTORY and SWEEP_ADJOINT (chunk `sub`) of sliced problems in one
                          // launch (one thread per fiber, mixed solver)
};

// Arguments of one sweep launch (uniform over its tiles; problems share shape and solver).
struct SweepArgs {
    const ProbDev* pds;   // [problems] device copies
    const Tile* tiles;    // [tiles] one per CTA
    const int* lanemap;   // [maps][threads]: (column << 16 | fiber), ~value for idle lanes
    int cpt;              // columns of the widest tile (shared-memory sizing)
    int gmax;             // largest ProbDev::glocal over the problems (admission)
    int mode;             // SweepMode
    int seg;              // segment (SWEEP_RECOMPUTE, SWEEP_ADJOINT)
    int sub;              // chunk of the segment (SWEEP_ADJOINT)
    int L, q, solver, nthreads;
    int pair;             // kernel family: log2 of the threads per fiber (0, 1 or 2)
    int lean;             // pair = 0 with the 168-register build (ProbDev::lean)
    int hdepth;           // steps per history group (ProbDev::hdepth), >= 1
    int slices, voff;     // SWEEP_PROP with slices > 0: slices a window instead of ProbDev::C, the
                          // first virtual window of the launch (0-based), and
    double2* phi;         // its propagators [virtual windows of the launch][N][N]
};

// A launch that may begin while the kernel before it on the stream ends: its blocks are placed and
// run up to chain_wait() (msqoc_chain.cuh), which every kernel launched this way calls before it
// reads what an earlier kernel wrote and before it writes anything, in every block.  With the
// copies ahead of the first kernel left out (take_inputs), QFT-4's gradient of eight dependent
// launches 116 -> 104 us, QFT-8's 372 -> 347, three transmons' 1060 -> 992, QFT-8's roll-out
// 387 -> 323.  Captured launches are plain ones (a graph has its own edges).
// Blocks of two kernels share an SM only under one split of its L1, so every kernel asks for the most
// shared memory: QFT-4's gradient 104 -> 91 us, QFT-8's 304 -> 266.
// chained: false for a plain launch, whose blocks are placed when the kernel before has ended.
template <class... P, class... A>
cudaError_t launch_split(bool chained, void (*kern)(P...), dim3 grid, int threads, size_t smem, cudaStream_t s,
                          A... args) {
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(s, &cap) != cudaSuccess) {
        cudaGetLastError();
        cap = cudaStreamCaptureStatusActive;
    }
    cudaLaunchAttribute at[2] = {};
    int n = 0;
    at[n].id = cudaLaunchAttributePreferredSharedMemoryCarveout;
    at[n++].val.sharedMemCarveout = cudaSharedmemCarveoutMaxShared;
    if (chained && cap == cudaStreamCaptureStatusNone) {
        at[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        at[n++].val.programmaticStreamSerializationAllowed = 1;
    }
    cudaLaunchConfig_t c{};
    c.gridDim = grid;
    c.blockDim = dim3(threads);
    c.dynamicSmemBytes = smem;
    c.stream = s;
    c.attrs = at;
    c.numAttrs = n;
    const cudaError_t e = cudaLaunchKernelEx(&c, kern, P(args)...);
    if (e != cudaSuccess) cudaGetLastError();   // returned here, not to the next caller that asks
    return e;
}
template <class... P, class... A>
cudaError_t launch_chained(void (*kern)(P...), dim3 grid, int threads, size_t smem, cudaStream_t s, A... args) {
    return launch_split(true, kern, grid, threads, smem, s, args...);
}

// shared-memory bytes of a sweep launch
size_t sweep_smem_bytes(const SweepArgs& a);

// launcher (dispatches on L, q, solver, direction); returns cudaError_t
cudaError_t launch_sweep(const SweepArgs& a, int ntiles, cudaStream_t s);

// Arguments of one quadrature launch: the gradient products of chunk `sub` of segment `seg` of
// every problem listed (problems share shape, solver and kernel family).
struct QuadArgs {
    const ProbDev* pds;   // device copies
    const int* list;      // [blocks in y] problem of each row of blocks; nullptr: row y is problem y
    int L, q, mode;       // mode: k_quad's MODE
    int seg, sub;
};
// First global step of virtual window v (1-based) of a problem with C slices a window; the end of the
// grid beyond the last.
__host__ __device__ inline int64_t slice_start(const ProbDev& pd, int C, int v) {
    const int w = (v - 1) / C;
    const auto win = [&](int m) { return (static_cast<int64_t>(pd.m_off + m) * pd.nsteps) / pd.M_glob; };
    if (w >= pd.M) return win(pd.M);
    const int64_t n0 = win(w);
    return C == 1 ? n0 : n0 + ((v - 1 - w * C) * (win(w + 1) - n0)) / C;
}
// rows up to which the quadrature kernel stages 32 and 16 lanes (quad_lanes; more rows: 8)
constexpr int QUAD_ROWS_32 = 32, QUAD_ROWS_16 = 128;
// blocks a problem needs for its windows' chunks
int quad_blocks(const ProbDev& pd);
// nprob rows of `blocks` blocks each (0 blocks: only sets the kernel's attributes)
cudaError_t launch_quad(const QuadArgs& a, int blocks, int nprob, cudaStream_t s);

// resident CTAs per SM of a sweep kernel at this launch shape (0 on error)
int sweep_ctas_per_sm(const SweepArgs& a);

}  // namespace msqoc
