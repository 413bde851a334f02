// pgc_kernels.cuh -- the time-step kernels of the particle stochastic-Galerkin scheme
// (arXiv:2404.19602, Algorithm 1 for P = Q = 1, Algorithm 2 otherwise), templated on the gPC
// basis size P, the number of quadrature nodes Q and the arithmetic type R.
//
// One time step n is two launches:
//   k_phase1 (every particle, streaming): drift of the coefficients (Eq. (17), Sec. 4.1),
//       reconstruction at the Q nodes (Eq. (23)), first flight-time draw, and a conservative
//       rate bound that proves "no collision in this step" for most particles; those are
//       finished here (histogram f^{n+1} of Eq. (24), moments).  The rest are appended to a
//       collider queue.  It also clears the histogram buffer of step n+2 and the next queue
//       counter, so that no separate memset is needed.
//   k_phase2 (queued particles only): the exact collision loop of Algorithm 1 / 2 with the
//       Pauli test against f^n, then the histogram f^{n+1} and moments of the final state.
// On moment steps k_finalize_cols reduces the block partial sums in a fixed order, one block per
// column, and writes the node values, mean and variance of the record (Sec. 4.2).
//
// Pipelined form (several steps per call): k_phase2<EXT = true> of step n, after the collision
// loop of a queued particle, carries that particle on through the drift and the flight-time
// screen of step n + 1 (finishing it there, or queueing it for step n + 1), and k_phase1 of step
// n + 1 skips the particles queued at step n (a bitmap).  The two then touch disjoint particles and
// buffers and are the two roles of one launch, k_step; every particle undergoes the same arithmetic
// as in the two-launch form, so the trajectories are identical.
#pragma once

#include "pgc_device.cuh"
#include "pgc_fd.cuh"

namespace pgc {

constexpr int kPhase1Threads = 256;   // threads of a streaming block (P1Threads: 512 at 36 nodes in FP32)
constexpr int kPhase2Threads = 128;
constexpr int kClearBytes = 64 << 10;   // of the histogram to be cleared, per streaming block (see RunnerT)
constexpr int kMaxGrid1 = 4096;   // block partials sized for at most this many phase-1 blocks
constexpr int kGrid2 = 608;       // phase-2 blocks (grid-stride over the queue)
// Phase-2 blocks per SM the collider kernel is compiled for (four: no spills at 36 nodes; five
// were measured 1 % slower with the collider's rolled slot loops, six slower still).
template <int P, int Q> struct Phase2Blocks { static constexpr int per_sm = 4; };
constexpr int kGrid2Max = 5 * 152; // phase-2 partial sums are sized for this many blocks
// Block-private histogram window of the streaming kernels: W x W cells around the grid centre, in
// shared memory, flushed to the global histogram once per block.  Two nodes share a word per cell,
// node 2p in the low and node 2p + 1 in the high half, so that a node's increment is a constant
// (1 or 1 << 16) and a cell's byte offset within a node pair is one multiply-add of its row and
// column.  Cells outside the window go straight to the global histogram.
//   36 nodes, FP32: one block of 512 threads per SM owns one window of 48 x 48 cells (166 KB).  Two
//   blocks with 32 x 32 each (+-0.67 eV) left 2-4 % of the particles with a node outside (3/4 of
//   the warps had such a lane) once the field had heated the ensemble; 48 x 48 (+-1 eV): 0.1 %.
//   One-dimensional shapes: 48 x 48 up to 6 nodes (28 KB), 40 x 40 up to 26 (83 KB), 36 x 36 at 31 (83 KB: two
//   blocks per SM; 40 x 40, 102 KB, left one in FP32); 36 nodes FP64: 32 x 32.
template <int P, int Q, typename R> struct HistWin {
    static constexpr int pairs = (Q + 1) / 2;
    static constexpr int W = (Q == 36) ? (sizeof(R) == 4 ? 48 : 32) : (Q <= 6 ? 48 : Q <= 26 ? 40 : 36);
    static constexpr size_t bytes = (size_t)pairs * W * W * 4;
    // the batched kernel (blocks of up to 256 threads, two per SM at 36 nodes)
    static constexpr int batchW = (Q == 36) ? (sizeof(R) == 4 ? 36 : 32) : 56;
    static constexpr size_t batch_bytes = (size_t)pairs * batchW * batchW * 4;
};
// threads of a streaming block
template <int P, int Q, typename R> struct P1Threads {
    static constexpr int value = (Q == 36 && sizeof(R) == 4) ? 512 : kPhase1Threads;
};
// The window of the tensor-core streaming kernel: kWin x kWin cells per node, two columns per word.
constexpr int kWin = 32;
constexpr int kWinWords = kWin * kWin / 2;
// Rotating buffers.  Histogram f^n lives in buffer n % kHistBufs: while phase 2 of step n - 1
// (reading f^{n-1}, writing f^n and f^{n+1}) runs beside phase 1 of step n (writing f^{n+1},
// clearing f^{n+2}), four buffers are in use.  Collider counters: n % 3; queues and moment
// partials: n % 2; collider bitmaps: n % 3.
constexpr int kHistBufs = 4;
constexpr int kQSlots = 3;
// Moment partial sums of step n (streaming part1, collider part2, carried partN) live in slot
// n % kPartSlots: the record of step m is reduced beside the launches of steps m + 1 and m + 2,
// and step m + 3 is the first to overwrite its slot.
constexpr int kPartSlots = 3;
constexpr int kMarkSlots = 3;

// Basis of total degree <= 5 in two variables on 6 x 6 tensor nodes (the compiled 2-D shape):
// coefficient (h1, h2) sits at index t(t+1)/2 + h2 with t = h1 + h2.
template <int P, int Q> struct TensorShape { static constexpr bool value = (P == 21 && Q == 36); };
__host__ __device__ constexpr int hidx2(int h1, int h2) { return (h1 + h2) * (h1 + h2 + 1) / 2 + h2; }

// Quadrature / basis tables of one context (Sec. 4.1).
template <int P, int Q, typename R>
struct Nodes {
    R psi[Q * P];    // Psi_h(z_q), [q][h]
    R wpsi[Q * P];   // w_q Psi_h(z_q)
    R dhat[P];       // per-step drift of the x coefficients
    R eps0[Q];       // band minimum at the node
    R dq[Q];         // per-step drift (e/hbar) E(z_q) dt at the node
    R lkx[Q];        // x offset of the grid at the node: Lk, or Lk - dq/2 (Strang)
    R xs[Q];         // x shift from the stored state to the state at the step boundary: 0, or dq/2 (Strang)
    R eps0_max;
    uint32_t drift_mask;  // coefficients h with dhat[h] != 0
    // 2-D tensor nodes (P = 21, Q = 36): one-dimensional basis values for sum factorisation,
    // a1[q1][h1] = psi_h1(z1_q1), b2[q2][h2] = psi_h2(z2_q2)
    R a1[36], b2[36];
    // FP32: the same weights as pairs (w, w), the operand of the two-lane FMA that reconstructs
    // the x and y components together (one unused entry in FP64)
    unsigned long long psi2[(TensorShape<P, Q>::value || sizeof(R) == 8) ? 1 : Q * P];
    unsigned long long wpsi2[(TensorShape<P, Q>::value || sizeof(R) == 8) ? 1 : Q * P];
    unsigned long long a1_2[36], b2_2[36];
    unsigned long long lk2[Q];   // (lkx[q], Lk) in FP32
};

template <int P, int Q, typename R>
struct StepArgs {
    Phys<R> ph;
    Nodes<P, Q, R> nd;
    R *khat;                 // [2][P][ld]
    int64_t N, ld;
    const uint32_t *Hcur;    // f^n   [Q][Nk*Nk]
    uint32_t *Hnext;         // f^{n+1}
    uint32_t *Hclear;        // buffer of step n+2, cleared by phase 1
    int64_t hist_elems;      // Q*Nk*Nk
    const uint32_t *nmax;    // [Q]
    uint32_t *queue;         // [N]
    uint32_t *qcount;        // collider count of this step
    uint32_t *qcount_next;   // counter of the next step (zeroed by phase 1)
    uint32_t *tilectr;       // phase-1 tile counter of this step (nullptr: static tile assignment)
    uint32_t *tilectr_next;  // tile counter of the next step (zeroed by phase 1)
    double *part1;           // [gridDim(phase1)][Q*3]
    double *part2;           // [kGrid2Max][Q*3]
    unsigned long long *counters;
    uint32_t key0, key1, stream_id, step;
    int32_t out_step;        // 1: accumulate the moments of the post-step state
    int32_t win_r0;          // first row / column of the shared-memory window
    int32_t use_win;         // 1: phase 1 counts into the shared-memory window
    float kk_in;             // |k|^2 up to which a node value's cell lies in the window (< 0: none known to)
    // collider bitmaps (bit i of word i / 32), all optional (nullptr)
    const uint32_t *skip;    // phase 1: particles queued at step n - 1, owned by a concurrent phase 2
    uint32_t *mark;          // phase 1: set for every particle queued at step n
    uint32_t *mark_clear;    // phase 1: bitmap of step n + 1, cleared
    int64_t mark_words;      // words per bitmap (multiple of 4)
    // phase 2 continuation into step n + 1 (k_phase2<EXT = true>)
    uint32_t *Hnext2;        // f^{n+2}
    uint32_t *queue_next;    // collider queue of step n + 1 (its counter is qcount_next)
    uint32_t *mark_next;     // bitmap of step n + 1
    double *partN;           // [kGrid2Max][Q*3] moments of step n + 1 of the particles finished here
    int32_t out_next;        // 1: step n + 1 is a moment step
    const Nodes<P, Q, R> *nd_dev;  // device copy of nd (phase 2 stages it into shared memory)
};

template <typename T>
__device__ __forceinline__ T warp_sum(T v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Per-warp moment accumulators of the streaming kernels.  FP64 in the FP64 mode.  In the FP32
// mode a float-float pair (hi, lo) advanced by the error-free transformation TwoSum (Knuth,
// TAOCP vol. 2, 4.2.2): hi + lo carries ~48 significant bits, and no operation runs on the FP64
// pipe, which on this part issues a small fraction of the FP32 rate.  The block's partial sum
// is then formed in FP64 from hi + lo, in a fixed warp order.
template <typename R> struct MomAcc;
template <> struct MomAcc<double> { using T = double; };
template <> struct MomAcc<float> { using T = float2; };
__device__ __forceinline__ void acc_zero(double &a) { a = 0.0; }
__device__ __forceinline__ void acc_zero(float2 &a) { a = make_float2(0.0f, 0.0f); }
__device__ __forceinline__ void acc_add(double &a, double x) { a += x; }
__device__ __forceinline__ void acc_add(float2 &a, float x)
{
    const float s = a.x + x;
    const float bp = s - a.x;
    const float err = (a.x - (s - bp)) + (x - bp);
    a.x = s;
    a.y += err;
}
__device__ __forceinline__ double acc_value(double a) { return a; }
__device__ __forceinline__ double acc_value(float2 a) { return (double)a.x + (double)a.y; }

// Warp sums of 16 values at once (a reduce-scatter): lane l ends with the sum over the 32 lanes
// of v[(l >> 1) & 15] (lanes l and l ^ 1 hold the same sum), after 16 shuffles instead of the
// 80 of 16 separate butterflies.  The lanes with l even add their sum to the accumulator
// dst[(l >> 1)] when that index is below count.
__device__ __forceinline__ void warp_scatter16_add(const float v[16], float2 *dst, int count, int lane)
{
    float a[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        const bool up = lane & 16;
        const float send = up ? v[j] : v[j + 8], keep = up ? v[j + 8] : v[j];
        a[j] = keep + __shfl_xor_sync(0xffffffffu, send, 16);
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const bool up = lane & 8;
        const float send = up ? a[j] : a[j + 4], keep = up ? a[j + 4] : a[j];
        a[j] = keep + __shfl_xor_sync(0xffffffffu, send, 8);
    }
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        const bool up = lane & 4;
        const float send = up ? a[j] : a[j + 2], keep = up ? a[j + 2] : a[j];
        a[j] = keep + __shfl_xor_sync(0xffffffffu, send, 4);
    }
    {
        const bool up = lane & 2;
        const float send = up ? a[0] : a[1], keep = up ? a[1] : a[0];
        a[0] = keep + __shfl_xor_sync(0xffffffffu, send, 2);
    }
    a[0] += __shfl_xor_sync(0xffffffffu, a[0], 1);
    const int idx = (lane >> 1) & 15;
    if (!(lane & 1) && idx < count) acc_add(dst[idx], a[0]);
}

// s + p[b * n3 + col] summed over b = b0, b0 + step, ... < b1 in that order (the fixed-order
// reductions of the block partials).  The loads are issued eight at a time ahead of their adds,
// so a thread waits for one memory round trip per eight rows instead of one per row; the sum is
// the plain loop's, bit for bit.
__device__ __forceinline__ double strided_sum(const double *p, int64_t b0, int64_t b1, int step, int n3, int col, double s)
{
    for (int64_t b = b0; b < b1; b += 8 * (int64_t)step) {
        double v[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const int64_t bb = b + (int64_t)k * step;
            v[k] = bb < b1 ? p[bb * n3 + col] : 0.0;
        }
#pragma unroll
        for (int k = 0; k < 8; ++k)
            if (b + (int64_t)k * step < b1) s += v[k];
    }
    return s;
}

// The same for 4 values: lane l ends with the sum over the 32 lanes of v[(l >> 3) & 3]; lanes
// 0, 8, 16, 24 add their sum to the accumulator dst[l >> 3] when that index is below count.
template <typename T>
__device__ __forceinline__ void warp_scatter4_add(const float v[4], T *dst, int count, int lane)
{
    float a[2];
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        const bool up = lane & 16;
        const float send = up ? v[j] : v[j + 2], keep = up ? v[j + 2] : v[j];
        a[j] = keep + __shfl_xor_sync(0xffffffffu, send, 16);
    }
    {
        const bool up = lane & 8;
        const float send = up ? a[0] : a[1], keep = up ? a[1] : a[0];
        a[0] = keep + __shfl_xor_sync(0xffffffffu, send, 8);
    }
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) a[0] += __shfl_xor_sync(0xffffffffu, a[0], o);
    const int idx = (lane >> 3) & 3;
    if (!(lane & 7) && idx < count) acc_add(dst[idx], a[0]);
}

// |k|^2 and the screen of the first flight time with an explicit operation order, so that
// phase 1 and the continuation in phase 2 take bit-identical decisions.
template <typename R>
__device__ __forceinline__ R knorm2(R kx, R ky)
{
    if constexpr (sizeof(R) == 8) return __fma_rn(kx, kx, __dmul_rn(ky, ky));
    else return __fmaf_rn(kx, kx, __fmul_rn(ky, ky));
}

// Maxima of three: `max3` drops NaN as fmaxf does, `max3_nan` keeps it.  A particle with a NaN node value
// must not be taken for one inside the window (its cell codes are garbage), while the screen's
// maximum drops NaN: both maxima over pairs of nodes cost what one over single nodes does.
__device__ __forceinline__ float max3(float a, float b, float c)
{
    float r;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}
__device__ __forceinline__ float max3_nan(float a, float b, float c)
{
    float r;
    asm("max.NaN.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}
// max over the nodes of kk, taken in node order
struct KkMax {
    float m = 0.0f, n = 0.0f, prev = 0.0f;   // without and with NaN; the even node of a pair
    __device__ __forceinline__ void add(int q, int Q, float kk)
    {
        if (q & 1) { m = max3(m, prev, kk); n = max3_nan(n, prev, kk); }
        else if (q == Q - 1) { m = fmaxf(m, kk); n = max3_nan(n, kk, kk); }
        else prev = kk;
    }
};

template <int P, int Q, typename R>
__device__ __forceinline__ bool screen_maybe(const Phys<R> &ph, const Nodes<P, Q, R> &nd, R kkmax, uint32_t xi_bits)
{
    const R lnxi = -rlog<R>(u01<R>(xi_bits));
    const R emax = rsqrt_<R>(ph.hvF2 * kkmax + nd.eps0_max * nd.eps0_max);
    const R gub = ph.alpha1 * rate_bound(ph, emax, nd.eps0_max) * (R)1.0001;
    return lnxi < gub * ph.dt;
}

// The FP64 screen decided in FP32 where the two cannot differ: 1 collides or may, 0 does not, -1
// undecided (to be taken in FP64).  kkmax, the energy, each rate and the logarithm carry a few FP32
// roundings; 3e-5 of the bound plus 2e-6 of all rate prefactors times the energy (the emission terms
// subtract the phonon energy) is more than ten times their sum, and the undecided share is ~1e-6.
__device__ __forceinline__ int screen_f32(const ScreenF &f, float kkmax, float eps0_max, uint32_t xi_bits)
{
    const float lnxi = -logf(u01<float>(xi_bits));
    const float emax = sqrtf(f.hvF2 * kkmax + eps0_max * eps0_max);
    const float x = f.alpha1 * rate_bound(f, emax, eps0_max) * 1.0001f * f.dt;
    const float tol = 3e-5f * x + 2e-6f * f.Csum * emax;
    return lnxi > x + tol ? 0 : (lnxi < x - tol ? 1 : -1);
}

template <int P, int Q, typename R>
__device__ __forceinline__ void load_coeffs(const StepArgs<P, Q, R> &a, int64_t i, R cx[P], R cy[P])
{
#pragma unroll
    for (int h = 0; h < P; ++h) {
        cx[h] = a.khat[(int64_t)h * a.ld + i];
        cy[h] = a.khat[(int64_t)(P + h) * a.ld + i];
    }
}

// Two FP32 fused multiply-adds in one instruction (packed f32x2 of sm_100+; each lane rounds as
// a scalar fmaf, so results are those of the scalar code): (x, y) pairs share a weight (w, w).
struct F2 { unsigned long long v; };
__device__ __forceinline__ F2 f2_pack(float a, float b)
{
    F2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ void f2_unpack(F2 p, float &a, float &b) { asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(p.v)); }
__device__ __forceinline__ F2 f2_fma(F2 a, unsigned long long w2, F2 c)
{
    F2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(w2), "l"(c.v));
    return r;
}

__device__ __forceinline__ F2 f2_add(F2 a, unsigned long long b)
{
    F2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b));
    return r;
}
__device__ __forceinline__ F2 f2_mul(F2 a, F2 b)
{
    F2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ F2 f2_add_rd(F2 a, F2 b)
{
    F2 r;
    asm("add.rm.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}

// Byte offset, within a node pair's part of the window, of the cell of a node value inside the window
// (the bits above 15 and the low two are not meaningful: mask with 0xfffc).  The cell is that of
// cell_rl: the same addition and multiplication, and floor by an addition rounded down at a magnitude
// where a float's last bit is 1 (row, 2^23) or 1/4 (column, 2^21): the low bits of the sums are then
// row - r0 and 4 (column - r0) + fraction.  Three packed operations and a multiply-add where two
// additions, two multiplications, two conversions, the bounds checks and the word and shift
// arithmetic were ~20.  A particle whose |k| stays inside the window's circle at every node (kk_in, from
// the majorant's kkmax that the screen needs anyway) takes no per-node check at all.  Instructions
// issued bound the streaming kernel: at 4e6 particles x 36 nodes 468 us a launch with the checks, 250 without (481
// and 256 after 2000 steps; one step in ten with moments).
template <int W>
__device__ __forceinline__ uint32_t window_code(float kx, float ky, unsigned long long lk2, F2 inv2, F2 magic2)
{
    const F2 s = f2_add_rd(f2_mul(f2_add(f2_pack(kx, ky), lk2), inv2), magic2);
    return (uint32_t)s.v * (4u * W) + (uint32_t)(s.v >> 32);
}
// The FP64 mode's cell (row << 16 | column, 0xffffffff outside the grid) from the node value rounded to FP32; `near`
// is set where the FP32 coordinates lie within their rounding of a cell edge (also for NaN and infinities):
// elsewhere the FP64 cell is the same.
constexpr float kCellGuard = 4e-7f;   // of Nk cells: four roundings of 2^-24 of at most Nk cells (2.4e-7) and as much again
__device__ __forceinline__ uint32_t cell_code_f64(double kx, double ky, unsigned long long lk2, F2 inv2, int Nk, float guard, bool &near)
{
    float yx, yy;
    f2_unpack(f2_mul(f2_add(f2_pack((float)kx, (float)ky), lk2), inv2), yx, yy);
    const float fx = yx - floorf(yx), fy = yy - floorf(yy);
    near = !(fminf(fminf(fx, 1.0f - fx), fminf(fy, 1.0f - fy)) > guard);
    const int r = __float2int_rd(yx), l = __float2int_rd(yy);
    return (unsigned)r < (unsigned)Nk && (unsigned)l < (unsigned)Nk ? ((uint32_t)r << 16) | (uint32_t)l : 0xffffffffu;
}
__device__ __forceinline__ F2 window_magic(int r0) { return f2_pack(8388608.0f - (float)r0, 2097152.0f - (float)r0); }

template <int P, int Q, typename R>
__device__ __forceinline__ void recon_node(const Nodes<P, Q, R> &nd, int q, const R cx[P], const R cy[P],
                                           R &kx, R &ky)
{
    if constexpr (sizeof(R) == 4 && !TensorShape<P, Q>::value) {
        F2 s = f2_pack(0.f, 0.f);
#pragma unroll
        for (int h = 0; h < P; ++h) s = f2_fma(f2_pack(cx[h], cy[h]), nd.psi2[q * P + h], s);
        f2_unpack(s, kx, ky);
    } else {
        R sx = (R)0, sy = (R)0;
#pragma unroll
        for (int h = 0; h < P; ++h) {
            sx += cx[h] * nd.psi[q * P + h];
            sy += cy[h] * nd.psi[q * P + h];
        }
        kx = sx;
        ky = sy;
    }
}

// The node values of recon_all (same operations in the same order) by a rolled loop over the rows of
// nodes: for code that seldom runs.
template <int P, int Q, typename R, typename F>
__device__ __forceinline__ void recon_all_rolled(const Nodes<P, Q, R> &nd, const R cx[P], const R cy[P], F &&f)
{
    if constexpr (TensorShape<P, Q>::value && sizeof(R) == 4) {
#pragma unroll 1
        for (int q1 = 0; q1 < 6; ++q1) {
            F2 t2[6];
#pragma unroll
            for (int h2 = 0; h2 < 6; ++h2) {
                F2 s2 = f2_pack(0.f, 0.f);
#pragma unroll
                for (int h1 = 0; h1 + h2 <= 5; ++h1)
                    s2 = f2_fma(f2_pack(cx[hidx2(h1, h2)], cy[hidx2(h1, h2)]), nd.a1_2[q1 * 6 + h1], s2);
                t2[h2] = s2;
            }
#pragma unroll
            for (int q2 = 0; q2 < 6; ++q2) {
                F2 k2 = f2_pack(0.f, 0.f);
#pragma unroll
                for (int h2 = 0; h2 < 6; ++h2) k2 = f2_fma(t2[h2], nd.b2_2[q2 * 6 + h2], k2);
                R kx, ky;
                f2_unpack(k2, kx, ky);
                f(q1 * 6 + q2, kx, ky);
            }
        }
    } else if constexpr (TensorShape<P, Q>::value) {
#pragma unroll 1
        for (int q1 = 0; q1 < 6; ++q1) {
            R tx[6], ty[6];
#pragma unroll
            for (int h2 = 0; h2 < 6; ++h2) {
                R sx = (R)0, sy = (R)0;
#pragma unroll
                for (int h1 = 0; h1 + h2 <= 5; ++h1) {
                    sx += cx[hidx2(h1, h2)] * nd.a1[q1 * 6 + h1];
                    sy += cy[hidx2(h1, h2)] * nd.a1[q1 * 6 + h1];
                }
                tx[h2] = sx;
                ty[h2] = sy;
            }
#pragma unroll
            for (int q2 = 0; q2 < 6; ++q2) {
                R kx = (R)0, ky = (R)0;
#pragma unroll
                for (int h2 = 0; h2 < 6; ++h2) {
                    kx += tx[h2] * nd.b2[q2 * 6 + h2];
                    ky += ty[h2] * nd.b2[q2 * 6 + h2];
                }
                f(q1 * 6 + q2, kx, ky);
            }
        }
    } else {
#pragma unroll 1
        for (int q = 0; q < Q; ++q) {
            R kx, ky;
            recon_node(nd, q, cx, cy, kx, ky);
            f(q, kx, ky);
        }
    }
}

// Reconstruction at every node (Eq. 23), calling f(q, kx, ky) per node.  For the 2-D tensor
// shape the sum is factorised: t(q1, h2) = sum_h1 c(h1,h2) a_h1(q1), k(q1,q2) = sum_h2 t b_h2(q2)
// (2 x 342 instead of 2 x 756 multiply-adds per particle).
template <int P, int Q, typename R, typename F>
__device__ __forceinline__ void recon_all(const Nodes<P, Q, R> &nd, const R cx[P], const R cy[P], F &&f)
{
    if constexpr (TensorShape<P, Q>::value && sizeof(R) == 4) {
        F2 c2[P];
#pragma unroll
        for (int h = 0; h < P; ++h) c2[h] = f2_pack(cx[h], cy[h]);
#pragma unroll
        for (int q1 = 0; q1 < 6; ++q1) {
            F2 t2[6];
#pragma unroll
            for (int h2 = 0; h2 < 6; ++h2) {
                F2 s2 = f2_pack(0.f, 0.f);
#pragma unroll
                for (int h1 = 0; h1 + h2 <= 5; ++h1) s2 = f2_fma(c2[hidx2(h1, h2)], nd.a1_2[q1 * 6 + h1], s2);
                t2[h2] = s2;
            }
#pragma unroll
            for (int q2 = 0; q2 < 6; ++q2) {
                F2 k2 = f2_pack(0.f, 0.f);
#pragma unroll
                for (int h2 = 0; h2 < 6; ++h2) k2 = f2_fma(t2[h2], nd.b2_2[q2 * 6 + h2], k2);
                R kx, ky;
                f2_unpack(k2, kx, ky);
                f(q1 * 6 + q2, kx, ky);
            }
        }
    } else if constexpr (TensorShape<P, Q>::value) {
#pragma unroll
        for (int q1 = 0; q1 < 6; ++q1) {
            R tx[6], ty[6];
#pragma unroll
            for (int h2 = 0; h2 < 6; ++h2) {
                R sx = (R)0, sy = (R)0;
#pragma unroll
                for (int h1 = 0; h1 + h2 <= 5; ++h1) {
                    sx += cx[hidx2(h1, h2)] * nd.a1[q1 * 6 + h1];
                    sy += cy[hidx2(h1, h2)] * nd.a1[q1 * 6 + h1];
                }
                tx[h2] = sx;
                ty[h2] = sy;
            }
#pragma unroll
            for (int q2 = 0; q2 < 6; ++q2) {
                R kx = (R)0, ky = (R)0;
#pragma unroll
                for (int h2 = 0; h2 < 6; ++h2) {
                    kx += tx[h2] * nd.b2[q2 * 6 + h2];
                    ky += ty[h2] * nd.b2[q2 * 6 + h2];
                }
                f(q1 * 6 + q2, kx, ky);
            }
        }
    } else {
        // (large one-dimensional shapes: a rolled node loop keeps the code size in check)
#pragma unroll (P * Q <= 64 ? Q : 1)
        for (int q = 0; q < Q; ++q) {
            R kx, ky;
            recon_node(nd, q, cx, cy, kx, ky);
            f(q, kx, ky);
        }
    }
}

// The value recon_all produces at node q (same operations in the same order).
template <int P, int Q, typename R>
__device__ __forceinline__ void recon_at(const Nodes<P, Q, R> &nd, int q, const R cx[P], const R cy[P], R &kx, R &ky)
{
    if constexpr (TensorShape<P, Q>::value) {
        const int q1 = q / 6, q2 = q - 6 * (q / 6);
        R sx2 = (R)0, sy2 = (R)0;
#pragma unroll
        for (int h2 = 0; h2 < 6; ++h2) {
            R sx = (R)0, sy = (R)0;
#pragma unroll
            for (int h1 = 0; h1 + h2 <= 5; ++h1) {
                sx += cx[hidx2(h1, h2)] * nd.a1[q1 * 6 + h1];
                sy += cy[hidx2(h1, h2)] * nd.a1[q1 * 6 + h1];
            }
            sx2 += sx * nd.b2[q2 * 6 + h2];
            sy2 += sy * nd.b2[q2 * 6 + h2];
        }
        kx = sx2;
        ky = sy2;
    } else {
        recon_node(nd, q, cx, cy, kx, ky);
    }
}

// The same from a particle's stored coefficients (k: its column of [2P][ld]).
template <int P, int Q, typename R>
__device__ __forceinline__ void recon_stored(const Nodes<P, Q, R> &nd, int q, const R *k, int64_t ld, R &kx, R &ky)
{
    R sx2 = (R)0, sy2 = (R)0;
    if constexpr (TensorShape<P, Q>::value) {
        const int q1 = q / 6, q2 = q - 6 * (q / 6);
#pragma unroll 1
        for (int h2 = 0; h2 < 6; ++h2) {
            R sx = (R)0, sy = (R)0;
            for (int h1 = 0; h1 + h2 <= 5; ++h1) {
                const int h = hidx2(h1, h2);
                sx += k[(int64_t)h * ld] * nd.a1[q1 * 6 + h1];
                sy += k[(int64_t)(P + h) * ld] * nd.a1[q1 * 6 + h1];
            }
            sx2 += sx * nd.b2[q2 * 6 + h2];
            sy2 += sy * nd.b2[q2 * 6 + h2];
        }
    } else {
#pragma unroll 4
        for (int h = 0; h < P; ++h) {
            sx2 += k[(int64_t)h * ld] * nd.psi[q * P + h];
            sy2 += k[(int64_t)(P + h) * ld] * nd.psi[q * P + h];
        }
    }
    kx = sx2;
    ky = sy2;
}

// group velocity (units of vF) and energy at one node (Sec. 2).  The warp partial sums are
// taken in R (FP32 in the production mode, FP64 in the FP64 mode) and accumulated in FP64.
// In FP32 the contraction is written out (which products are rounded: left to the compiler it follows the
// surrounding code, and a record of a thousand particles moves by 1e-8); the one-node shape keeps the
// compiler's, which is another there.
template <int Q, typename R>
__device__ __forceinline__ void observe(const Phys<R> &ph, R kx, R ky, R eps0, R &vx, R &vy, R &e)
{
    R s2;
    if constexpr (sizeof(R) == 4 && Q > 1) s2 = fma_rn(eps0, eps0, mul_rn(ph.hvF2, fma_rn(ky, ky, mul_rn(kx, kx))));
    else s2 = ph.hvF2 * (kx * kx + ky * ky) + eps0 * eps0;
    const R eps = rsqrt_<R>(s2);
    vx = ph.hvF * kx / eps;
    vy = ph.hvF * ky / eps;
    e = eps;
}

// The same observables in FP32 from one reciprocal square root (rsqrtf, 2 ulp): 1/eps, eps and
// both velocity components (the 36-node moment steps, where the divisions were the cost).
__device__ __forceinline__ void observe_fast(const Phys<float> &ph, float kx, float ky, float eps0, float &vx, float &vy,
                                             float &e)
{
    const float s2 = ph.hvF2 * (kx * kx + ky * ky) + eps0 * eps0;
    const float inv = rsqrtf(s2);
    vx = ph.hvF * kx * inv;
    vy = ph.hvF * ky * inv;
    e = s2 * inv;
}

// ------------------------------------------------------------------------------------------
// Phase 1: every particle.  Each thread takes PPT consecutive particles and reads each
// coefficient plane with one 16-byte load (float4 / 2 x double2); the ensemble is streamed once.
// ------------------------------------------------------------------------------------------
template <int P> struct Phase1PPT { static constexpr int value = (P <= 8) ? 4 : 1; };
// resident blocks per SM the streaming kernels are compiled for: three for the small FP32
// shapes, two (more registers, fewer spills) for the large shapes and for FP64; one block of 512
// threads for 36 nodes in FP32 (the same 128 registers, one window per SM).  k_phase1 alone also three at 9
// nodes (it fits; 1e6 particles 59 us a launch with two, 55 with three).
template <int P, int Q, typename R> struct kPhase1MinBlocks {
    static constexpr int value = (Q == 36 && sizeof(R) == 4) ? 1 : (P * Q > 64 || sizeof(R) == 8) ? 2 : 3;
    static constexpr int phase1 = (sizeof(R) == 4 && P * Q <= 100) ? 3 : value;
};

template <typename R, int PPT>
__device__ __forceinline__ void load_vec(const R *p, R v[PPT])
{
    if constexpr (PPT == 4 && sizeof(R) == 4) {
        const float4 t = *reinterpret_cast<const float4 *>(p);
        v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
    } else if constexpr (PPT == 4 && sizeof(R) == 8) {
        const double2 a = reinterpret_cast<const double2 *>(p)[0];
        const double2 b = reinterpret_cast<const double2 *>(p)[1];
        v[0] = a.x; v[1] = a.y; v[2] = b.x; v[3] = b.y;
    } else if constexpr (PPT == 2 && sizeof(R) == 4) {
        const float2 t = *reinterpret_cast<const float2 *>(p);
        v[0] = t.x; v[1] = t.y;
    } else if constexpr (PPT == 2 && sizeof(R) == 8) {
        const double2 t = *reinterpret_cast<const double2 *>(p);
        v[0] = t.x; v[1] = t.y;
    } else {
#pragma unroll
        for (int e = 0; e < PPT; ++e) v[e] = p[e];
    }
}

template <typename R, int PPT>
__device__ __forceinline__ void store_vec(R *p, const R v[PPT])
{
    if constexpr (PPT == 4 && sizeof(R) == 4) {
        *reinterpret_cast<float4 *>(p) = make_float4(v[0], v[1], v[2], v[3]);
    } else if constexpr (PPT == 4 && sizeof(R) == 8) {
        reinterpret_cast<double2 *>(p)[0] = make_double2(v[0], v[1]);
        reinterpret_cast<double2 *>(p)[1] = make_double2(v[2], v[3]);
    } else if constexpr (PPT == 2 && sizeof(R) == 4) {
        *reinterpret_cast<float2 *>(p) = make_float2(v[0], v[1]);
    } else if constexpr (PPT == 2 && sizeof(R) == 8) {
        *reinterpret_cast<double2 *>(p) = make_double2(v[0], v[1]);
    } else {
#pragma unroll
        for (int e = 0; e < PPT; ++e) p[e] = v[e];
    }
}

// The rolled node loop of the large one-dimensional FP32 shapes reads its weights from a shared-memory copy
// (rows padded to 16 bytes, two weights per load, four nodes' sums in flight): indexed reads of the
// parameter bank, one weight each, and one dependent sum at a time bounded it (21 nodes, 1e4
// particles: 17.3 us a launch; 15.8 us).
template <int P, int Q, typename R> struct StagePsi {
    static constexpr bool value = P * Q > 64 && !TensorShape<P, Q>::value && sizeof(R) == 4;
    static constexpr int row = (P + 1) & ~1;
    static constexpr int elems = value ? Q * row : 2;
};

// Everything phase 1 needs about one ensemble (one case of a batch).
template <typename R>
struct P1Target {
    R *khat;
    int64_t N, ld;
    uint32_t *Hnext;          // f^{n+1} [Q][Nk*Nk]
    uint32_t *qcount;         // collider counter of this step
    uint32_t *queue;          // collider queue
    uint32_t qoffset;         // added to the particle index in queue entries
    uint32_t key0, key1, stream_id, step;
    const uint32_t *skip = nullptr;  // optional: particles left to a concurrent phase 2 (not touched here)
    uint32_t *mark = nullptr;        // optional: bitmap of the particles queued here
};

// The particles of a warp with a node value outside the circle of the window (kk_in), put aside in
// shared memory: a rolled pass over their nodes for one lane costs a warp as much as for 32, so they
// are taken 32 at a time (at most 31 stay between passes).  Not in FP64 and not at the large one-dimensional
// shapes: there the cells are a small part of a pass, and even the last incomplete list of a warp costs as much
// as the pass itself, so each node's cell is checked against the window by itself (FP32, us a launch with
// lists and one window per SM at 31 nodes / by node: 31 nodes 2e4 particles 33.5 / 23.6, 2e5 139 / 66;
// 21 nodes 1e6 174 / 140).
template <int P, int Q, typename R> struct PutsAside { static constexpr bool value = sizeof(R) == 4 && !StagePsi<P, Q, R>::value; };
template <int PPT> struct AsideList { static constexpr int cap = 32 * (PPT + 1); };

// The colliders a warp finds wait in a list of their own (also AsideList::cap entries) and reach the
// queue 32 at a time, the rest of a block's warps together at its end: every append is an atomic with
// a result on one address of the launch, which L2 serves about every 2 ns.  One per warp pass with a
// collider (a quarter of them) was the kernel's time in the small shapes: 64 cases of 5e4 particles,
// one node, 25000 appends a step, 50 -> 41.5 us.
__device__ __forceinline__ void queue_warp(uint32_t *qcount, uint32_t *queue, const uint32_t *list, int lane)
{
    __syncwarp();
    uint32_t pos = 0;
    if (lane == 0) pos = atomicAdd(qcount, 32u);
    pos = __shfl_sync(0xffffffffu, pos, 0);
    queue[pos + lane] = list[lane];
    __syncwarp();
}
// The remainders (n < 32 each) of a block's warps; s_base: nwarps + 1 words.  Synchronises the block.
__device__ __forceinline__ void queue_block(uint32_t *qcount, uint32_t *queue, const uint32_t *list, int n, uint32_t *s_base)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    if (lane == 0) s_base[warp] = (uint32_t)n;
    __syncthreads();
    if (threadIdx.x == 0) {
        uint32_t s = 0;
        for (int v = 0; v < nw; ++v) { const uint32_t c = s_base[v]; s_base[v] = s; s += c; }
        s_base[nw] = s ? atomicAdd(qcount, s) : 0u;
    }
    __syncthreads();
    if (lane < n) queue[s_base[nw] + s_base[warp] + lane] = list[lane];
}

// Counts the cell of node q's value in the window or in the global histogram; 1 if it is outside the grid.
template <int Q, int W, typename R>
__device__ __forceinline__ unsigned int count_cell(const Phys<R> &ph, R lkx, int q, R kx, R ky, uint32_t *swin, int win_r0, bool use_win,
                                                   uint32_t *Hnext)
{
    int r, l;
    if (!cell_rl(ph, lkx, kx, ky, r, l)) return 1u;
    const int rr = r - win_r0, ll = l - win_r0;
    if (use_win && (unsigned)rr < (unsigned)W && (unsigned)ll < (unsigned)W)
        atomicAdd(&swin[(q >> 1) * (W * W) + rr * W + ll], 1u << ((q & 1) << 4));
    else
        atomicAdd(&Hnext[((int64_t)q * ph.Nk + r) * ph.Nk + l], 1u);
    return 0u;
}

// FP64: counts the nodes in `nodes` of one particle from its stored coefficients (k: its column).  Not inlined and
// with no copy of the coefficients: it seldom runs, and the streaming pass has no registers for it.
template <int P, int Q, int W>
__device__ __noinline__ unsigned int count_nodes(const Phys<double> &ph, const Nodes<P, Q, double> &nd, const double *k, int64_t ld,
                                                 uint64_t nodes, uint32_t *swin, int win_r0, bool use_win, uint32_t *Hnext)
{
    unsigned int oog = 0u;
#pragma unroll 1
    for (; nodes; nodes &= nodes - 1) {
        const int q = __ffsll((long long)nodes) - 1;
        double kx, ky;
        recon_stored(nd, q, k, ld, kx, ky);
        oog += count_cell<Q, W, double>(ph, nd.lkx[q], q, kx, ky, swin, win_r0, use_win, Hnext);
    }
    return oog;
}

// Counts the histogram cells of n <= 32 such particles (one per lane) from their stored state.
template <int P, int Q, typename R, int W>
__device__ __forceinline__ void count_aside(const Phys<R> &ph, const Nodes<P, Q, R> &nd, const P1Target<R> &t, const uint32_t *list,
                                            int n, uint32_t *swin, int win_r0, bool use_win, unsigned int &oog)
{
    if constexpr (PutsAside<P, Q, R>::value) {
        const int lane = threadIdx.x & 31;
        __syncwarp();   // the list and the drifted coefficients, written by other lanes
        if (lane < n) {
            const int64_t i = list[lane];
            R cx[P], cy[P];
#pragma unroll
            for (int h = 0; h < P; ++h) {
                cx[h] = t.khat[(int64_t)h * t.ld + i];
                cy[h] = t.khat[(int64_t)(P + h) * t.ld + i];
            }
            recon_all_rolled(nd, cx, cy, [&](int q, R kx, R ky) {
                oog += count_cell<Q, W, R>(ph, nd.lkx[q], q, kx, ky, swin, win_r0, use_win, t.Hnext);
            });
        }
        __syncwarp();   // the list may be written again
    }
}

// One pass of a block over blockDim * PPT consecutive particles starting at i0 + threadIdx*PPT:
// drift, reconstruction, flight-time screen, histogram (window or global), queue, moments.
// (PPT particles per thread; i0 a multiple of PPT.)  ndb: the basis and the grid offsets, nd: what
// depends on the inputs (drift, band minima); a batch's cases share the former, which then stays in the
// parameter bank.
template <int P, int Q, typename R, int W = HistWin<P, Q, R>::W, int PPT = Phase1PPT<P>::value>
__device__ __forceinline__ void phase1_pass(const Phys<R> &ph, const Nodes<P, Q, R> &ndb, const Nodes<P, Q, R> &nd, const P1Target<R> &t,
                                            int64_t i0, uint32_t *swin, int win_r0, bool use_win, float kk_in, bool out_step,
                                            typename MomAcc<R>::T *smom_warp, uint32_t *aside, int &n_aside,
                                            uint32_t *qlist, int &n_q, unsigned int &oog,
                                            const unsigned long long *spsi = nullptr, const R *pre = nullptr)
{
    const int lane = threadIdx.x & 31;
    const int64_t NN = (int64_t)ph.Nk * ph.Nk;
    R cx[PPT][P], cy[PPT][P];
    bool finished[PPT];
    const bool any = i0 < t.N;
    // i0 is a multiple of PPT, so its PPT bits lie in one word
    const uint32_t skipbits = (t.skip && any) ? (t.skip[i0 >> 5] >> (i0 & 31)) & ((1u << PPT) - 1u) : 0u;
    if (any) {
        if (PPT == 1 && pre) {   // loaded by the caller
#pragma unroll
            for (int h = 0; h < P; ++h) { cx[0][h] = pre[h]; cy[0][h] = pre[P + h]; }
        } else
#pragma unroll
        for (int h = 0; h < P; ++h) {
            R vx[PPT], vy[PPT];
            load_vec<R, PPT>(t.khat + (int64_t)h * t.ld + i0, vx);
            load_vec<R, PPT>(t.khat + (int64_t)(P + h) * t.ld + i0, vy);
#pragma unroll
            for (int e = 0; e < PPT; ++e) { cx[e][h] = vx[e]; cy[e][h] = vy[e]; }
        }
        // drift (Eq. (17) / sG forcing term); the padding beyond N is left untouched
#pragma unroll
        for (int h = 0; h < P; ++h)
            if (nd.drift_mask & (1u << h)) {
                R v[PPT];
#pragma unroll
                for (int e = 0; e < PPT; ++e) {
                    if (i0 + e < t.N) cx[e][h] -= nd.dhat[h];
                    v[e] = cx[e][h];
                }
                if (skipbits == 0u) {
                    store_vec<R, PPT>(t.khat + (int64_t)h * t.ld + i0, v);
                } else {
                    // a skipped particle is being written by phase 2: element-wise stores
#pragma unroll
                    for (int e = 0; e < PPT; ++e)
                        if (!((skipbits >> e) & 1u) && i0 + e < t.N) t.khat[(int64_t)h * t.ld + i0 + e] = v[e];
                }
            }
    }
    constexpr bool kUnrollQ = P * Q <= 64 || (TensorShape<P, Q>::value && sizeof(R) == 4);
    constexpr bool kCells = !PutsAside<P, Q, R>::value;
#pragma unroll
    for (int e = 0; e < PPT; ++e) {
        const int64_t i = i0 + e;
        finished[e] = false;
        bool maybe = false, put_aside = false;
        if (any && i < t.N && !((skipbits >> e) & 1u)) {
            // reconstruction, cells and the bound on the majorant
            uint32_t cell[Q];   // window_code, or with kCells row << 16 | column (0xffffffff outside the grid)
            using NearMask = typename std::conditional<(Q > 32), uint64_t, uint32_t>::type;
            NearMask near = 0;   // FP64: nodes whose cell FP32 does not decide
            const F2 inv2 = sizeof(R) == 4 ? f2_pack((float)ph.inv_dk, (float)ph.inv_dk) : f2_pack(ph.f.inv_dk, ph.f.inv_dk);
            const U4 r = philox4x32_10((uint32_t)i, t.stream_id, t.step, 0u, t.key0, t.key1);
            bool in_window;
            if constexpr (sizeof(R) == 4) {
                const F2 magic2 = window_magic(win_r0);
                KkMax km;
                if constexpr (StagePsi<P, Q, R>::value) {
#pragma unroll 4
                    for (int q = 0; q < Q; ++q) {
                        const ulonglong2 *w = reinterpret_cast<const ulonglong2 *>(spsi + q * StagePsi<P, Q, R>::row);
                        F2 s2 = f2_pack(0.f, 0.f);
#pragma unroll
                        for (int h = 0; h < P; ++h) s2 = f2_fma(f2_pack(cx[e][h], cy[e][h]), (h & 1) ? w[h >> 1].y : w[h >> 1].x, s2);
                        float kx, ky;
                        f2_unpack(s2, kx, ky);
                        int rw, cl;
                        cell[q] = cell_rl(ph, ndb.lkx[q], kx, ky, rw, cl) ? ((uint32_t)rw << 16) | (uint32_t)cl : 0xffffffffu;
                        km.m = fmaxf(km.m, knorm2(kx, ky));
                    }
                } else {
                    recon_all(ndb, cx[e], cy[e], [&](int q, R kx, R ky) {
                        cell[q] = window_code<W>(kx, ky, ndb.lk2[q], inv2, magic2);
                        km.add(q, Q, knorm2(kx, ky));
                    });
                }
                in_window = kCells || km.n <= kk_in;   // (false for NaN)
                maybe = screen_maybe(ph, nd, km.m, r.x);
            } else {
                // FP64: cells and screen in FP32 where FP32 is certain of them (the FP64 pipe issues one warp
                // instruction per 16 clocks; the reconstruction is what it has to do), else in FP64: a node near a
                // cell edge (one in 2500 at 240 cells) by itself.  No particle is formed a second time: the
                // pipe is busy as long for one lane as for 32, and with the particles near an edge or outside
                // the window's circle put aside every warp had such a lane (us a launch, put aside / here: 31 nodes,
                // 1e4 particles 297 / 165; 36 nodes, 4e4 358 / 140; 6 nodes, 1e6 at 1000 cells, 1e5 79 / 48).
                KkMax km;
                const float guard = kCellGuard * (float)ph.Nk;
                auto node = [&](int q, R kx, R ky) {
                    bool nr;
                    cell[q] = cell_code_f64(kx, ky, ndb.lk2[q], inv2, ph.Nk, guard, nr);
                    near |= (NearMask)nr << q;
                    const float xf = (float)kx, yf = (float)ky;
                    km.add(q, Q, xf * xf + yf * yf);
                };
                // (36 nodes row by row: unrolled, the values of all nodes were held at once and 3 KB a thread spilled)
                if constexpr (TensorShape<P, Q>::value) recon_all_rolled(ndb, cx[e], cy[e], node);
                else recon_all(ndb, cx[e], cy[e], node);
                const int sc = screen_f32(ph.f, km.n, (float)nd.eps0_max, r.x);
                maybe = sc > 0;
                if (sc < 0) {
                    R kk = (R)0;
                    recon_all_rolled(ndb, cx[e], cy[e], [&](int, R kx, R ky) { kk = fmax(kk, knorm2(kx, ky)); });
                    maybe = screen_maybe(ph, nd, kk, r.x);
                }
                in_window = true;
            }
            if (!maybe) {
                finished[e] = true;
                if (in_window) {
#pragma unroll (kUnrollQ ? Q : 1)
                    for (int q = 0; q < Q; ++q) {
                        if constexpr (!kCells) {   // every node value lies in the window
                            atomicAdd(reinterpret_cast<uint32_t *>(reinterpret_cast<char *>(swin + (q >> 1) * (W * W)) + (cell[q] & 0xfffcu)),
                                      (q & 1) ? 0x10000u : 1u);
                        } else if (sizeof(R) == 4 || !((near >> q) & 1)) {
                            if (cell[q] == 0xffffffffu) { ++oog; continue; }
                            const int r = (int)(cell[q] >> 16), l = (int)(cell[q] & 0xffffu), rr = r - win_r0, ll = l - win_r0;
                            if (use_win && (unsigned)rr < (unsigned)W && (unsigned)ll < (unsigned)W)
                                atomicAdd(&swin[(q >> 1) * (W * W) + rr * W + ll], 1u << ((q & 1) << 4));
                            else
                                atomicAdd(&t.Hnext[((int64_t)q * ph.Nk + r) * ph.Nk + l], 1u);
                        }
                    }
                    if constexpr (sizeof(R) == 8)
                        if (near) oog += count_nodes<P, Q, W>(ph, ndb, t.khat + i, t.ld, near, swin, win_r0, use_win, t.Hnext);
                } else {
                    put_aside = true;
                }
            }
        }
        if (!kCells) {
            const unsigned int am = __ballot_sync(0xffffffffu, put_aside);
            if (am) {
                if (put_aside) aside[n_aside + __popc(am & ((1u << lane) - 1u))] = (uint32_t)i;
                n_aside += __popc(am);
            }
        }
        // colliders go to the warp's list for the queue
        const unsigned int mask = __ballot_sync(0xffffffffu, maybe);
        if (mask) {
            if (maybe) {
                qlist[n_q + __popc(mask & ((1u << lane) - 1u))] = t.qoffset + (uint32_t)i;
                if (t.mark) atomicOr(&t.mark[i >> 5], 1u << (i & 31));
            }
            n_q += __popc(mask);
        }
    }
    while (n_q >= 32) {
        n_q -= 32;
        queue_warp(t.qcount, t.queue, qlist + n_q, lane);
    }
    if (out_step) {
        if constexpr (TensorShape<P, Q>::value && sizeof(R) == 4 && PPT == 1) {
            // one particle per thread: the node values again by the (unrolled) sum factorisation,
            // their observables streamed 16 at a time into warp reduce-scatters (node q,
            // quantity j is value 3 q + j)
            float buf[16];
            const bool fin = finished[0];
            recon_all(ndb, cx[0], cy[0], [&](int q, R kx, R ky) {
                float o[3] = {0.0f, 0.0f, 0.0f};
                if (fin) observe_fast(ph, kx - nd.xs[q], ky, nd.eps0[q], o[0], o[1], o[2]);
#pragma unroll
                for (int j = 0; j < 3; ++j) {
                    const int idx = 3 * q + j;
                    buf[idx & 15] = o[j];
                    if ((idx & 15) == 15 || idx == 3 * Q - 1) {
                        for (int z = (idx & 15) + 1; z < 16; ++z) buf[z] = 0.0f;
                        warp_scatter16_add(buf, smom_warp + (idx & ~15), (idx & 15) + 1, lane);
                    }
                }
            });
        } else if constexpr (sizeof(R) == 4) {
            // per node: the three observables summed over the thread's particles, then one 4-value
            // warp reduce-scatter (6 shuffles instead of the 15 of three butterflies)
#pragma unroll 1
            for (int q = 0; q < Q; ++q) {
                float s[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
                for (int e = 0; e < PPT; ++e)
                    if (finished[e]) {
                        float kx, ky, a1, a2, a3;
                        recon_node(ndb, q, cx[e], cy[e], kx, ky);
                        observe<Q>(ph, kx - nd.xs[q], ky, nd.eps0[q], a1, a2, a3);
                        s[0] += a1; s[1] += a2; s[2] += a3;
                    }
                warp_scatter4_add(s, smom_warp + q * 3, 3, lane);
            }
        } else {
#pragma unroll 1
            for (int q = 0; q < Q; ++q) {
                R vx = (R)0, vy = (R)0, en = (R)0;
#pragma unroll
                for (int e = 0; e < PPT; ++e)
                    if (finished[e]) {
                        R kx, ky, a1, a2, a3;
                        recon_node(ndb, q, cx[e], cy[e], kx, ky);
                        observe<Q>(ph, kx - nd.xs[q], ky, nd.eps0[q], a1, a2, a3);
                        vx += a1; vy += a2; en += a3;
                    }
                vx = warp_sum(vx);
                vy = warp_sum(vy);
                en = warp_sum(en);
                if (lane == 0) {
                    acc_add(smom_warp[q * 3 + 0], vx);
                    acc_add(smom_warp[q * 3 + 1], vy);
                    acc_add(smom_warp[q * 3 + 2], en);
                }
            }
        }
    }
    while (n_aside >= 32) {
        n_aside -= 32;
        count_aside<P, Q, R, W>(ph, ndb, t, aside + n_aside, 32, swin, win_r0, use_win, oog);
    }
}

// PPT passes of one particle per thread over the PPT * blockDim particles from `base` (a step without
// moments), each pass's coefficients loaded behind the one before it.
template <int P, int Q, typename R, int W, int PPT>
__device__ __forceinline__ void phase1_rolled(const Phys<R> &ph, const Nodes<P, Q, R> &ndb, const Nodes<P, Q, R> &nd, const P1Target<R> &t,
                                              int64_t base, uint32_t *swin, int win_r0, bool use_win, float kk_in,
                                              typename MomAcc<R>::T *smom_warp, uint32_t *aside, int &n_aside, uint32_t *qlist,
                                              int &n_q, unsigned int &oog)
{
    R nx[2 * P];
    auto load = [&](int64_t i) {
        if (i < t.N) {
#pragma unroll
            for (int h = 0; h < 2 * P; ++h) nx[h] = t.khat[(int64_t)h * t.ld + i];
        }
    };
    int64_t i = base + threadIdx.x;
    load(i);
#pragma unroll 1
    for (int e = 0; e < PPT; ++e, i += blockDim.x) {
        R c[2 * P];
#pragma unroll
        for (int h = 0; h < 2 * P; ++h) c[h] = nx[h];
        if (e + 1 < PPT) load(i + blockDim.x);
        phase1_pass<P, Q, R, W, 1>(ph, ndb, nd, t, i, swin, win_r0, use_win, kk_in, false, smom_warp, aside, n_aside, qlist, n_q, oog,
                                   nullptr, c);
    }
}

// Clear a block's window (dynamic shared memory).
template <int Q, int W>
__device__ __forceinline__ void clear_window(uint32_t *swin)
{
    static_assert(W % 4 == 0, "four cells of a row per access");
    for (int j = threadIdx.x; j < (Q + 1) / 2 * (W * W / 4); j += blockDim.x)
        reinterpret_cast<uint4 *>(swin)[j] = make_uint4(0u, 0u, 0u, 0u);
}

// Add it to the global histogram, one add per non-empty cell and node; flush_quads with four cells a lane, which
// passes over empty words fastest, flush_window word by word, so that a warp's adds fall on 32 cells side
// by side, four sectors of L2 instead of sixteen.  The fuller the window the more the adds are the step (1e6 particles
// x 6 nodes, us a step, quads / words: 240 cells 33.5 / 32.4, after 3000 steps 38.4 / 36.0; 480 cells 48.2 /
// 36.4; 600 cells 57 / 41); a window that has counted fewer than kSparseWindow particles on a grid of fewer than
// kFineGrid cells is mostly empty (36 nodes, 2e5 particles, 1300 a block, us a launch: 240 cells 27.5 / 29.0;
// 6 nodes, 3e5 particles, 1024 a block, us a step: 480 cells 25.1 / 22.6), as are those of the batch's tiles.
// Not inlined: the streaming loop has no register to spare for it.
constexpr int kSparseWindow = 2000, kFineGrid = 400;
template <int Q, int W>
__device__ __forceinline__ void flush_quads(const uint32_t *swin, uint32_t *Hnext, int Nk, int win_r0)
{
    const int64_t NN = (int64_t)Nk * Nk;
    for (int j = threadIdx.x; j < (Q + 1) / 2 * (W * W / 4); j += blockDim.x) {
        const uint4 v4 = reinterpret_cast<const uint4 *>(swin)[j];
        if (!(v4.x | v4.y | v4.z | v4.w)) continue;
        const int p = j / (W * W / 4), w = j % (W * W / 4);
        uint32_t *base = Hnext + (int64_t)(2 * p) * NN + (int64_t)(w / (W / 4) + win_r0) * Nk + 4 * (w % (W / 4)) + win_r0;
        const uint32_t v[4] = {v4.x, v4.y, v4.z, v4.w};
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            if (v[c] & 0xffffu) atomicAdd(base + c, v[c] & 0xffffu);
            if (v[c] >> 16) atomicAdd(base + NN + c, v[c] >> 16);
        }
    }
}

template <int Q, int W>
__device__ __noinline__ void flush_window(uint32_t *Hnext, int Nk, int win_r0, int64_t counted)
{
    extern __shared__ __align__(16) uint32_t swin[];
    if (counted < kSparseWindow && Nk < kFineGrid) return flush_quads<Q, W>(swin, Hnext, Nk, win_r0);
    constexpr uint32_t n = (Q + 1) / 2 * W * W, U = Q > 6 ? 8 : 4;
    const uint32_t NN = (uint32_t)Nk * Nk, pair = 2 * NN - W * (uint32_t)Nk;   // (a histogram of all nodes has < 2^32 cells)
    uint32_t *base = Hnext + win_r0 * (Nk + 1);
    for (uint32_t j0 = threadIdx.x; j0 < n; j0 += U * blockDim.x) {
        uint32_t v[U];
#pragma unroll
        for (uint32_t u = 0; u < U; ++u) v[u] = j0 + u * blockDim.x < n ? swin[j0 + u * blockDim.x] : 0u;
#pragma unroll
        for (uint32_t u = 0; u < U; ++u) {
            if (!v[u]) continue;
            const uint32_t j = j0 + u * blockDim.x, r = j / W, p = r / W;   // row of all pairs' windows, node pair
            uint32_t *h = base + (size_t)(p * pair + r * (uint32_t)Nk + (j - r * W));
            if (v[u] & 0xffffu) atomicAdd(h, v[u] & 0xffffu);
            if (v[u] >> 16) atomicAdd(h + NN, v[u] >> 16);
        }
    }
}

// The window of the tensor-core streaming kernel.
template <int Q>
__device__ __forceinline__ void flush_window_tc(const uint32_t *swin, uint32_t *Hnext, int Nk, int win_r0)
{
    const int64_t NN = (int64_t)Nk * Nk;
    for (int j = threadIdx.x; j < Q * kWinWords; j += blockDim.x) {
        const uint32_t v = swin[j];
        if (!v) continue;
        const int q = j / kWinWords, w = j % kWinWords;
        const int rr = w / (kWin / 2) + win_r0, ll = 2 * (w % (kWin / 2)) + win_r0;
        uint32_t *base = Hnext + (int64_t)q * NN + (int64_t)rr * Nk + ll;
        if (v & 0xffffu) atomicAdd(base, v & 0xffffu);
        if (v >> 16) atomicAdd(base + 1, v >> 16);
    }
}

// Phase 1 of one block, block bid of the nb blocks doing phase 1.  Tiles of blockDim * PPT
// particles: taken from the step's tile counter when there is one (blocks that start late take
// fewer), else every nb-th tile.  swin: dynamic shared memory of the histogram window.
template <int P, int Q, typename R>
__device__ __forceinline__ void phase1_block(const StepArgs<P, Q, R> &a, int bid, int nb, uint32_t *swin)
{
    constexpr int PPT = Phase1PPT<P>::value;
    constexpr int NW = P1Threads<P, Q, R>::value / 32;
    __shared__ typename MomAcc<R>::T smom[NW][Q * 3];
    __shared__ uint32_t s_tile;
    __shared__ uint32_t s_aside[NW][AsideList<PPT>::cap];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    __shared__ uint32_t s_qlist[NW][AsideList<PPT>::cap], s_qbase[NW + 1];
    uint32_t *aside = s_aside[warp], *qlist = s_qlist[warp];
    int n_aside = 0, n_q = 0;
    using SP = StagePsi<P, Q, R>;
    __shared__ __align__(16) unsigned long long spsi[SP::elems];
    const int64_t tile = (int64_t)blockDim.x * PPT;
    if constexpr (SP::value)
        if (a.tilectr || (int64_t)bid * tile < a.N)   // (a block without particles only clears)
            for (int j = threadIdx.x; j < Q * P; j += blockDim.x) {
                const float w = a.nd_dev ? a.nd_dev->psi[j] : a.nd.psi[j];
                spsi[(j / P) * SP::row + j % P] = f2_pack(w, w).v;
            }
    if (a.out_step)
        for (int j = lane; j < Q * 3; j += 32) acc_zero(smom[warp][j]);
    __syncthreads();

    // housekeeping for the next steps
    if (bid == 0 && threadIdx.x == 0) {
        *a.qcount_next = 0u;
        if (a.tilectr_next) *a.tilectr_next = 0u;
    }
    {
        uint4 *hc = reinterpret_cast<uint4 *>(a.Hclear);
        const int64_t n4 = a.hist_elems >> 2;
        for (int64_t j = (int64_t)bid * blockDim.x + threadIdx.x; j < n4; j += (int64_t)nb * blockDim.x)
            hc[j] = make_uint4(0u, 0u, 0u, 0u);
        if (bid == 0)
            for (int64_t j = (n4 << 2) + threadIdx.x; j < a.hist_elems; j += blockDim.x) a.Hclear[j] = 0u;
        if (a.mark_clear) {
            uint4 *mc = reinterpret_cast<uint4 *>(a.mark_clear);
            for (int64_t j = (int64_t)bid * blockDim.x + threadIdx.x; j < (a.mark_words >> 2); j += (int64_t)nb * blockDim.x)
                mc[j] = make_uint4(0u, 0u, 0u, 0u);
        }
    }

    P1Target<R> t;
    t.khat = a.khat; t.N = a.N; t.ld = a.ld; t.Hnext = a.Hnext; t.qcount = a.qcount; t.queue = a.queue;
    t.qoffset = 0u; t.key0 = a.key0; t.key1 = a.key1; t.stream_id = a.stream_id; t.step = a.step;
    t.skip = a.skip; t.mark = a.mark;
    unsigned int oog = 0u;
    // A window cell holds 16 bits and a particle adds at most one count to a cell per node, so the
    // window is flushed to f^{n+1} before the block has counted 65535 particles since the last
    // flush (block-uniform; with the tile counter a block may take any number of tiles).  A block
    // without a tile has no window: it neither clears nor flushes one.
    int64_t since_flush = 0;
    auto guard_window = [&]() {
        if (a.use_win && (since_flush == 0 || since_flush + tile + blockDim.x > 65535)) {   // (blockDim.x: particles put aside before the flush)
            if (since_flush > 0) {
                __syncthreads();
                flush_window<Q, HistWin<P, Q, R>::W>(a.Hnext, a.ph.Nk, a.win_r0, since_flush);
                __syncthreads();
            }
            clear_window<Q, HistWin<P, Q, R>::W>(swin);
            __syncthreads();
            since_flush = 0;
        }
        since_flush += tile;
    };
    // One node: a step without moments takes the tile's particles one per thread at a time (coalesced 4-byte
    // loads, each pass's ahead of the one before).  64 cases of 5e4 particles: 41.5 -> 37.6 us a launch.  With
    // 6 nodes the rolled form is slower (1e6 particles 26 -> 32 us: its loads are waited for one by one).
    auto pass = [&](int64_t base) {
        constexpr int W = HistWin<P, Q, R>::W;
        if (PPT == 1 || P > 1 || sizeof(R) == 8 || a.out_step) {
            phase1_pass<P, Q, R, W, PPT>(a.ph, a.nd, a.nd, t, base + (int64_t)threadIdx.x * PPT, swin, a.win_r0, a.use_win != 0, a.kk_in,
                                         a.out_step != 0, smom[warp], aside, n_aside, qlist, n_q, oog, spsi);
        } else {
            phase1_rolled<P, Q, R, W, PPT>(a.ph, a.nd, a.nd, t, base, swin, a.win_r0, a.use_win != 0, a.kk_in, smom[warp], aside, n_aside,
                                           qlist, n_q, oog);
        }
    };
    if (a.tilectr) {
        const int64_t ntiles = (a.N + tile - 1) / tile;
        for (;;) {
            if (threadIdx.x == 0) s_tile = atomicAdd(a.tilectr, 1u);
            __syncthreads();
            const int64_t tl = s_tile;
            __syncthreads();   // every thread has read s_tile before it is overwritten
            if (tl >= ntiles) break;
            guard_window();
            pass(tl * tile);
        }
    } else {
        for (int64_t base = (int64_t)bid * tile; base < a.N; base += (int64_t)nb * tile) {
            guard_window();
            pass(base);
        }
    }
    if (n_aside > 0)
        count_aside<P, Q, R, HistWin<P, Q, R>::W>(a.ph, a.nd, t, aside, n_aside, swin, a.win_r0, a.use_win != 0, oog);
    oog = warp_sum(oog);
    if (lane == 0 && oog) atomicAdd(&a.counters[4], (unsigned long long)oog);
    queue_block(t.qcount, t.queue, qlist, n_q, s_qbase);   // (synchronises)
    if (a.use_win && since_flush > 0) flush_window<Q, HistWin<P, Q, R>::W>(a.Hnext, a.ph.Nk, a.win_r0, since_flush);
    if (a.out_step) {
        for (int j = threadIdx.x; j < Q * 3; j += blockDim.x) {
            double s = 0.0;
#pragma unroll
            for (int w = 0; w < NW; ++w) s += acc_value(smom[w][j]);
            a.part1[(int64_t)bid * (Q * 3) + j] = s;
        }
    }
}

template <int P, int Q, typename R>
__global__ void __launch_bounds__(P1Threads<P, Q, R>::value, kPhase1MinBlocks<P, Q, R>::phase1)
k_phase1(const __grid_constant__ StepArgs<P, Q, R> a)
{
    extern __shared__ __align__(16) uint32_t swin[];   // HistWin when a.use_win
    phase1_block<P, Q, R>(a, blockIdx.x, gridDim.x, swin);
}

// ------------------------------------------------------------------------------------------
// Phase 2: the collision loop of Algorithm 1 / 2 for the queued particles.  A group of G
// lanes carries one particle, lane r owning the nodes q = r, r + G, ... (lanes <-> quadrature
// nodes): the rates, the mechanism selection, the final states and the Pauli look-ups of the Q
// nodes run in parallel, and the projection of Eqs. (28)-(30) and the majorant of Eq. (25) are
// group reductions by shuffles.
// ------------------------------------------------------------------------------------------
#ifndef PGC_GROUP36
#define PGC_GROUP36 32
#endif
#ifndef PGC_GROUP8
#define PGC_GROUP8 8
#endif

template <int Q> struct GroupOf {
    static constexpr int G = (Q == 36) ? PGC_GROUP36
                           : (Q >= 32) ? 32 : (Q > 16 ? 32 : (Q > 8 ? 16 : (Q > 4 ? PGC_GROUP8 : (Q > 2 ? 4 : (Q > 1 ? 2 : 1)))));
    static constexpr int NPL = (Q + G - 1) / G;  // nodes per lane
};

// Node slots of a lane (s = 0 .. NPL - 1) read and written with a runtime slot index by selects,
// so that a rolled loop over the slots keeps the per-slot arrays in registers: the per-node code
// of the collision loop is emitted once instead of NPL times (instruction-cache footprint).
template <int N, typename T>
__device__ __forceinline__ T slot_get(const T (&a)[N], int s)
{
    T v = a[0];
#pragma unroll
    for (int k = 1; k < N; ++k)
        if (s == k) v = a[k];
    return v;
}
template <int N, typename T>
__device__ __forceinline__ void slot_set(T (&a)[N], int s, T v)
{
#pragma unroll
    for (int k = 0; k < N; ++k)
        if (s == k) a[k] = v;
}

template <int G, typename T>
__device__ __forceinline__ T group_sum(T v, unsigned mask)
{
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) v += __shfl_xor_sync(mask, v, o, G);
    return v;
}

template <int G, typename T>
__device__ __forceinline__ T group_max(T v, unsigned mask)
{
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(mask, v, o, G));
    return v;
}

template <int G>
__device__ __forceinline__ bool group_any(bool b, unsigned mask)
{
    return (__ballot_sync(mask, b) & mask) != 0u;
}

// Shared-memory transpose reduction of the projection for groups of a whole warp: per warp, 32
// rows of 2P partial sums (row stride 2P + 1, odd, so that the column reads are conflict-free)
// and the 2P totals.
template <int P, int Q, typename R> struct ProjRed {   // (its area fits the static shared memory up to P = 21)
    static constexpr bool value = GroupOf<Q>::G == 32 && sizeof(R) == 4 && P <= 21;
    static constexpr int stride = 2 * P + 1;
    static constexpr int warp_elems = 32 * stride + 2 * P;
};

// Projection of the node values onto the basis (the collisional matrices K1 + K2 of Eqs.
// (28)-(30)): cx_h = sum_q w_q Psi_h(z_q) kx_q, summed over the G lanes of the group (lane r holds
// nodes r, r + G, ...); every lane receives all 2P coefficients.  FP32 whole-warp groups: each
// lane writes its 2P partial sums to shared memory (red: this block's ProjRed area, one per warp),
// lane j adds column j over the 32 lanes in a fixed order, and every lane reads the 2P totals back
// (~2P shared stores and loads per lane instead of 2P five-level shuffle butterflies).  Otherwise
// butterfly shuffles.
template <int P, int Q, typename R>
__device__ __forceinline__ void project_group(const Nodes<P, Q, R> &nd, const R kx[GroupOf<Q>::NPL],
                                              const R ky[GroupOf<Q>::NPL], int r, unsigned gmask, R cx[P], R cy[P],
                                              R *red)
{
    constexpr int G = GroupOf<Q>::G, NPL = GroupOf<Q>::NPL;
    constexpr int S = ProjRed<P, Q, R>::stride;
    R *w = red + (threadIdx.x >> 5) * ProjRed<P, Q, R>::warp_elems;   // used by ProjRed shapes only
#pragma unroll (P * Q <= 64 ? P : 1)
    for (int h = 0; h < P; ++h) {
        R sx = (R)0, sy = (R)0;
        if constexpr (sizeof(R) == 4 && !TensorShape<P, Q>::value) {
            F2 s2 = f2_pack(0.f, 0.f);
#pragma unroll
            for (int s = 0; s < NPL; ++s) {
                const int q = r + s * G;
                if (q < Q) s2 = f2_fma(f2_pack(kx[s], ky[s]), nd.wpsi2[q * P + h], s2);
            }
            f2_unpack(s2, sx, sy);
        } else {
#pragma unroll
            for (int s = 0; s < NPL; ++s) {
                const int q = r + s * G;
                if (q < Q) {
                    sx += nd.wpsi[q * P + h] * kx[s];
                    sy += nd.wpsi[q * P + h] * ky[s];
                }
            }
        }
        if constexpr (ProjRed<P, Q, R>::value) {
            w[r * S + h] = sx;
            w[r * S + P + h] = sy;
        } else {
            cx[h] = group_sum<G>(sx, gmask);
            cy[h] = group_sum<G>(sy, gmask);
        }
    }
    if constexpr (ProjRed<P, Q, R>::value) {
        R *tot = w + 32 * S;
        __syncwarp(gmask);
        for (int v = r; v < 2 * P; v += 32) {
            R acc = (R)0;
#pragma unroll 8
            for (int l = 0; l < 32; ++l) acc += w[l * S + v];
            tot[v] = acc;
        }
        __syncwarp(gmask);
#pragma unroll
        for (int h = 0; h < P; ++h) {
            cx[h] = tot[h];
            cy[h] = tot[P + h];
        }
        __syncwarp(gmask);   // all lanes have read the totals before the next projection writes
    }
}

// Everything the collision loop of one particle needs about its ensemble.
template <typename R>
struct P2Target {
    R *khat;
    int64_t ld;
    const uint32_t *Hcur;     // f^n
    uint32_t *Hnext;          // f^{n+1}
    const uint32_t *nmax;
    double *mom;              // [Q*3] moment accumulators (shared or global), on moment steps
    uint32_t key0, key1, stream_id, step;
    bool out_step;
    // continuation into step n + 1 (EXT)
    uint32_t *Hnext2 = nullptr;      // f^{n+2}
    uint32_t *queue_next = nullptr, *qcount_next = nullptr, *mark_next = nullptr;
    double *momN = nullptr;          // [Q*3] moments of step n + 1
    bool out_next = false;
    R *red = nullptr;                // shared-memory area of project_group (ProjRed shapes)
};

struct P2Counts { unsigned long long att = 0, chg = 0, rej = 0, cap = 0, oog = 0; };

// The collision loop of Algorithm 1 / 2 for particle i, carried by the G lanes of a group (lane r
// owns nodes r, r + G, ...), then the histogram f^{n+1} and moments of its final state.  With
// EXT, the particle then goes through step n + 1 as far as phase 1 would take it: drift,
// reconstruction, flight-time screen, and either the histogram f^{n+2} and moments of step n + 1
// or a place in the collider queue of step n + 1.
template <int P, int Q, typename R, bool EXT = false>
__device__ __forceinline__ void collide_particle(const Phys<R> &ph, const Nodes<P, Q, R> &nd, const P2Target<R> &t,
                                                 int64_t i, int r, unsigned gmask, P2Counts &cnt)
{
    constexpr int G = GroupOf<Q>::G, NPL = GroupOf<Q>::NPL;
    const int64_t NN = (int64_t)ph.Nk * ph.Nk;
    R cx[P], cy[P], kx[NPL], ky[NPL];
#pragma unroll
    for (int h = 0; h < P; ++h) {
        cx[h] = t.khat[(int64_t)h * t.ld + i];
        cy[h] = t.khat[(int64_t)(P + h) * t.ld + i];
    }
    // the node values of the lane's slots from the coefficients
    // (NPL > 1: loops over the slots are rolled, see slot_get)
    auto recon_slots = [&](const R (&ccx)[P], const R (&ccy)[P], R (&x)[NPL], R (&y)[NPL]) {
        if constexpr (NPL > 1) {
#pragma unroll 1
            for (int s = 0; s < NPL; ++s) {
                const int q = r + s * G;
                if (q >= Q) break;
                R a, b;
                recon_node(nd, q, ccx, ccy, a, b);
                slot_set(x, s, a);
                slot_set(y, s, b);
            }
        } else {
            recon_node(nd, r, ccx, ccy, x[0], y[0]);
        }
    };
    recon_slots(cx, cy, kx, ky);
    R gc[NPL][6];  // rates of the current state at the lane's nodes (reused by the selection)
    R tc = (R)0, Gt = (R)0;
    uint32_t c = 0;
    bool touched = false, fresh = true;
    // One pass per free flight: majorant of the current state (Eq. (25)), flight time, and, if
    // the flight ends inside the step, a collision.  The rates and the random draw have one
    // call site each (instruction-cache footprint).  An event that changes no node (self
    // scattering or Pauli rejection everywhere) leaves the state, its rates and the majorant
    // as they were: the projection of unchanged node values returns the same coefficients, so
    // it, the reconstruction and the rates are not redone (fresh = false).
    for (;;) {
        if (fresh) {
            R gm = (R)0;
            if constexpr (NPL > 1) {
#pragma unroll 1
                for (int s = 0; s < NPL; ++s) {
                    const int q = r + s * G;
                    if (q >= Q) break;
                    R g[6];
                    gm = fmax(gm, rates6(ph, slot_get(kx, s), slot_get(ky, s), nd.eps0[q], g));
#pragma unroll
                    for (int m = 0; m < 6; ++m)
#pragma unroll
                        for (int k = 0; k < NPL; ++k)
                            if (s == k) gc[k][m] = g[m];
                }
            } else {
#pragma unroll
                for (int s = 0; s < NPL; ++s) {
                    const int q = r + s * G;
                    if (q < Q) gm = fmax(gm, rates6(ph, kx[s], ky[s], nd.eps0[q], gc[s]));
                }
            }
            Gt = ph.alpha1 * group_max<G>(gm, gmask);
        }
        const U4 rr = philox4x32_10((uint32_t)i, t.stream_id, t.step, c, t.key0, t.key1);
        const R dtc = (Gt > (R)0) ? -rlog<R>(u01<R>(rr.x)) / Gt : (R)INFINITY;
        if (!(tc + dtc < ph.dt)) break;             // group-uniform condition
        if ((int)c >= ph.max_coll) { if (r == 0) ++cnt.cap; break; }
        if (r == 0) ++cnt.att;
        EventAngles<R> ang;
        ang.reset(u01<R>(rr.w));
        const R target = u01<R>(rr.y) * Gt;
        bool changed = false;
        if constexpr (NPL > 1) {
#pragma unroll 1
            for (int s = 0; s < NPL; ++s) {
                const int q = r + s * G;
                if (q >= Q) break;
                int l = 6;
                R cum = (R)0;
#pragma unroll
                for (int m = 0; m < 6; ++m) {
                    R gsm = gc[0][m];
#pragma unroll
                    for (int k = 1; k < NPL; ++k)
                        if (s == k) gsm = gc[k][m];
                    cum += gsm;
                    if (l == 6 && target < cum) l = m;
                }
                if (l == 6) continue;  // self scattering: h^7 = identity
                R nkx, nky;
                final_state<EXT ? 1 : 8>(ph, l, slot_get(kx, s), slot_get(ky, s), nd.eps0[q], ang, &nkx, &nky);
                bool accept = true;
                if (ph.pauli_mode != 2) {
                    const int cl = cell_of(ph, nd.lkx[q], nkx + nd.dq[q], nky);
                    if (cl >= 0) accept = pauli_accept(t.Hcur[(int64_t)q * NN + cl], t.nmax[q], rr.z);
                }
                if (accept) {
                    slot_set(kx, s, nkx);
                    slot_set(ky, s, nky);
                    changed = true;
                } else {
                    ++cnt.rej;
                }
            }
        } else {
#pragma unroll
        for (int s = 0; s < NPL; ++s) {
            const int q = r + s * G;
            if (q >= Q) continue;
            int l = 6;
            R cum = (R)0;
#pragma unroll
            for (int m = 0; m < 6; ++m) {
                cum += gc[s][m];
                if (l == 6 && target < cum) l = m;
            }
            if (l == 6) continue;  // self scattering: h^7 = identity
            R nkx, nky;
            final_state<EXT ? 1 : 8>(ph, l, kx[s], ky[s], nd.eps0[q], ang, &nkx, &nky);
            bool accept = true;
            if (ph.pauli_mode != 2) {
                const int cl = cell_of(ph, nd.lkx[q], nkx + nd.dq[q], nky);
                if (cl >= 0) accept = pauli_accept(t.Hcur[(int64_t)q * NN + cl], t.nmax[q], rr.z);
            }
            if (accept) { kx[s] = nkx; ky[s] = nky; changed = true; }
            else ++cnt.rej;
        }
        }
        fresh = group_any<G>(changed, gmask);
        if (fresh && r == 0) ++cnt.chg;
        if (fresh) {
            touched = true;
            // collisional matrices K1 + K2 (Eqs. (28)-(30)): project the node values
            project_group<P, Q, R>(nd, kx, ky, r, gmask, cx, cy, t.red);
            recon_slots(cx, cy, kx, ky);
        }
        tc += dtc;
        ++c;
    }
    if constexpr (EXT) {
        // drift of step n + 1 (before the store: the stored state is the post-drift one, as phase 1 leaves it)
#pragma unroll
        for (int h = 0; h < P; ++h)
            if (nd.drift_mask & (1u << h)) cx[h] -= nd.dhat[h];
    }
    if (touched || (EXT && nd.drift_mask != 0u)) {
        // lane h of the group writes coefficient h (x and y planes)
        for (int h = r; h < P; h += G) {
            R vx = cx[0], vy = cy[0];
#pragma unroll
            for (int hh = 0; hh < P; ++hh) if (hh == h) { vx = cx[hh]; vy = cy[hh]; }
            t.khat[(int64_t)h * t.ld + i] = vx;
            t.khat[(int64_t)(P + h) * t.ld + i] = vy;
        }
    }
    auto finish_node = [&](int q, R x, R y) {
        const int cl = cell_of(ph, nd.lkx[q], x, y);
        if (cl >= 0) atomicAdd(&t.Hnext[(int64_t)q * NN + cl], 1u);
        else ++cnt.oog;
        if (t.out_step) {
            R vx, vy, e;
            observe<Q>(ph, x - nd.xs[q], y, nd.eps0[q], vx, vy, e);
            atomicAdd(&t.mom[q * 3 + 0], (double)vx);
            atomicAdd(&t.mom[q * 3 + 1], (double)vy);
            atomicAdd(&t.mom[q * 3 + 2], (double)e);
        }
    };
    if constexpr (NPL > 1) {
#pragma unroll 1
        for (int s = 0; s < NPL; ++s) {
            const int q = r + s * G;
            if (q >= Q) break;
            finish_node(q, slot_get(kx, s), slot_get(ky, s));
        }
    } else {
#pragma unroll
        for (int s = 0; s < NPL; ++s) {
            const int q = r + s * G;
            if (q < Q) finish_node(q, kx[s], ky[s]);
        }
    }
    if constexpr (EXT) {
        // step n + 1 up to the flight-time screen, with the operations of phase 1
        int cl2[NPL];
        R kk = (R)0;
#pragma unroll
        for (int s = 0; s < NPL; ++s) {
            const int q = r + s * G;
            cl2[s] = -1;
            if (q < Q) {
                R x, y;
                recon_at(nd, q, cx, cy, x, y);
                cl2[s] = cell_of(ph, nd.lkx[q], x, y);
                kk = fmax(kk, knorm2(x, y));
            }
        }
        const R kkmax = group_max<G>(kk, gmask);
        const U4 r1 = philox4x32_10((uint32_t)i, t.stream_id, t.step + 1u, 0u, t.key0, t.key1);
        if (!screen_maybe(ph, nd, kkmax, r1.x)) {
#pragma unroll
            for (int s = 0; s < NPL; ++s) {
                const int q = r + s * G;
                if (q >= Q) continue;
                if (cl2[s] >= 0) atomicAdd(&t.Hnext2[(int64_t)q * NN + cl2[s]], 1u);
                else ++cnt.oog;
                if (t.out_next) {
                    R x, y, vx, vy, e;
                    recon_node(nd, q, cx, cy, x, y);
                    observe<Q>(ph, x - nd.xs[q], y, nd.eps0[q], vx, vy, e);
                    atomicAdd(&t.momN[q * 3 + 0], (double)vx);
                    atomicAdd(&t.momN[q * 3 + 1], (double)vy);
                    atomicAdd(&t.momN[q * 3 + 2], (double)e);
                }
            }
        } else if (r == 0) {
            const uint32_t pos = atomicAdd(t.qcount_next, 1u);
            t.queue_next[pos] = (uint32_t)i;
            atomicOr(&t.mark_next[i >> 5], 1u << (i & 31));
        }
    }
}

// The queue entries of this thread's collider group among the nb blocks of a launch: entries first,
// first + stride, ... < count.  The groups of a warp take different mechanisms and numbers of events
// and the warp runs their union.  A queue of at most half as many entries as warps is spread one group
// per warp, over the blocks first: the chain of one particle is then the kernel's time
// (deterministic FP64 run of 1e4 particles, ~90 colliders a step: 99.6 us a step in three warps
// of one block, 77 us spread; 32 us with the edge table and the root starts as well).  A longer one
// fills whole warps: spread, 6 nodes, 5e5 particles took 25.0 instead of 22.0 us a fused step (every
// collider block then holds its place on an SM) and 43.8 instead of 37.7 us in the adjoint's collider
// kernel.
struct QueueShare { uint32_t first, stride; };
template <int G>
__device__ __forceinline__ QueueShare queue_share(uint32_t count, int bid, int nb)
{
    constexpr uint32_t W = 32 / G;
    const uint32_t nw = blockDim.x >> 5, warps = (uint32_t)nb * nw;
    const uint32_t sub = (threadIdx.x & 31) / G, warp = threadIdx.x >> 5;
    if (W > 1 && 2 * count <= warps) return QueueShare{sub == 0 ? warp * (uint32_t)nb + (uint32_t)bid : 0xffffffffu, warps};
    return QueueShare{((uint32_t)bid * nw + warp) * W + sub, warps * W};
}

// Copy a trivially-copyable table into shared memory (all threads; caller synchronises).
template <typename T>
__device__ __forceinline__ void stage(uint32_t *dst, const T &src)
{
    const uint32_t *s = reinterpret_cast<const uint32_t *>(&src);
    for (int j = threadIdx.x; j < (int)(sizeof(T) / 4); j += blockDim.x) dst[j] = s[j];
}

// The queue of a step and, if save is non-NULL, the queued particles' coefficients before their collisions
// (column j of [2P][ld] for queue entry j), for the adjoint's backward step.
template <int P, typename R>
__global__ void __launch_bounds__(256)
k_keep_colliders(const R *khat, int64_t ld, const uint32_t *queue, const uint32_t *qcount, R *save, uint32_t *save_queue,
                 uint32_t *save_count)
{
    const uint32_t count = *qcount;
    if (blockIdx.x == 0 && threadIdx.x == 0) *save_count = count;
    for (uint32_t j = blockIdx.x * blockDim.x + threadIdx.x; j < count; j += gridDim.x * blockDim.x) {
        const uint32_t i = queue[j];
        save_queue[j] = i;
        if (!save) continue;
#pragma unroll 6
        for (int h = 0; h < 2 * P; ++h) save[(int64_t)h * ld + j] = khat[(int64_t)h * ld + i];
    }
}

// Phase 2 of one block, block bid of the nb blocks doing phase 2 (any block size that is a
// multiple of the group size).
template <int P, int Q, typename R, bool EXT>
__device__ __forceinline__ void phase2_block(const StepArgs<P, Q, R> &a, int bid, int nb, R *red)
{
    constexpr int G = GroupOf<Q>::G;
    __shared__ double smom[Q * 3];
    __shared__ double smomN[EXT ? Q * 3 : 1];
    __shared__ unsigned long long scnt[5];
    // The lanes of a group read different nodes' entries of the node tables: staged in shared
    // memory from their device copy (divergent reads of the parameter bank serialise).  The
    // physics constants are read by all lanes alike and stay in the parameter bank.
    __shared__ __align__(16) uint32_t snd[(sizeof(Nodes<P, Q, R>) + 3) / 4];
    if (threadIdx.x < 5) scnt[threadIdx.x] = 0ull;
    for (int j = threadIdx.x; j < Q * 3; j += blockDim.x) smom[j] = 0.0;
    if constexpr (EXT)
        for (int j = threadIdx.x; j < Q * 3; j += blockDim.x) smomN[j] = 0.0;
    if (a.nd_dev) {
        const uint32_t *src = reinterpret_cast<const uint32_t *>(a.nd_dev);
        for (int j = threadIdx.x; j < (int)(sizeof(Nodes<P, Q, R>) / 4); j += blockDim.x) snd[j] = src[j];
    } else {
        stage(snd, a.nd);
    }
    __syncthreads();

    const Phys<R> &ph = a.ph;
    const Nodes<P, Q, R> &nd = *reinterpret_cast<const Nodes<P, Q, R> *>(snd);
    const uint32_t count = *a.qcount;
    P2Counts cnt;
    P2Target<R> t;
    t.khat = a.khat; t.ld = a.ld; t.Hcur = a.Hcur; t.Hnext = a.Hnext; t.nmax = a.nmax; t.mom = smom;
    t.key0 = a.key0; t.key1 = a.key1; t.stream_id = a.stream_id; t.step = a.step; t.out_step = a.out_step != 0;
    t.red = red;
    if constexpr (EXT) {
        t.Hnext2 = a.Hnext2; t.queue_next = a.queue_next; t.qcount_next = a.qcount_next; t.mark_next = a.mark_next;
        t.momN = smomN; t.out_next = a.out_next != 0;
    }

    const int lane = threadIdx.x & 31;
    const int r = lane % G;                                  // lane in the group
    const unsigned gmask = (G == 32) ? 0xffffffffu : (((1u << G) - 1u) << (lane - r));
    const QueueShare qs = queue_share<G>(count, bid, nb);
    for (uint32_t j = qs.first; j < count; j += qs.stride) collide_particle<P, Q, R, EXT>(ph, nd, t, a.queue[j], r, gmask, cnt);

    if (cnt.att) atomicAdd(&scnt[0], cnt.att);
    if (cnt.chg) atomicAdd(&scnt[1], cnt.chg);
    if (cnt.rej) atomicAdd(&scnt[2], cnt.rej);
    if (cnt.cap) atomicAdd(&scnt[3], cnt.cap);
    if (cnt.oog) atomicAdd(&scnt[4], cnt.oog);
    __syncthreads();
    if (threadIdx.x < 5 && scnt[threadIdx.x]) atomicAdd(&a.counters[threadIdx.x], scnt[threadIdx.x]);
    if (threadIdx.x == 0 && bid == 0) atomicAdd(&a.counters[5], (unsigned long long)count);
    if (a.out_step)
        for (int j = threadIdx.x; j < Q * 3; j += blockDim.x) a.part2[(int64_t)bid * (Q * 3) + j] = smom[j];
    if constexpr (EXT)
        if (a.out_next)
            for (int j = threadIdx.x; j < Q * 3; j += blockDim.x) a.partN[(int64_t)bid * (Q * 3) + j] = smomN[j];
}

template <int P, int Q, typename R, bool EXT>
__global__ void __launch_bounds__(kPhase2Threads, Phase2Blocks<P, Q>::per_sm)
k_phase2(const __grid_constant__ StepArgs<P, Q, R> a)
{
    __shared__ R sred[ProjRed<P, Q, R>::value ? (kPhase2Threads / 32) * ProjRed<P, Q, R>::warp_elems : 1];
    phase2_block<P, Q, R, EXT>(a, blockIdx.x, gridDim.x, sred);
}

// One launch per time step in the pipelined form: blocks [0, nb2) run phase 2 of step n - 1 with
// the continuation into step n (a2), the others phase 1 of step n (a1, tiles from the tile
// counter, skipping the particles queued at step n - 1).  The two roles touch disjoint particles;
// shared buffers are only added to (histograms, queue of step n, bitmap of step n).
template <int P, int Q, typename R>
__global__ void __launch_bounds__(P1Threads<P, Q, R>::value, kPhase1MinBlocks<P, Q, R>::value)
k_step(const __grid_constant__ StepArgs<P, Q, R> a1, const __grid_constant__ StepArgs<P, Q, R> a2, int nb2)
{
    extern __shared__ __align__(16) uint32_t swin[];   // phase 1: histogram window; phase 2: projection area
    if ((int)blockIdx.x < nb2) phase2_block<P, Q, R, true>(a2, blockIdx.x, nb2, reinterpret_cast<R *>(swin));
    else phase1_block<P, Q, R>(a1, blockIdx.x - nb2, gridDim.x - nb2, swin);
}

// ------------------------------------------------------------------------------------------
// Observation of a whole state: histogram into H and (optionally) moment partials into part1.
// Used after the initial sampling and after a state upload.
// ------------------------------------------------------------------------------------------
// Counts go to the block's window as in the streaming kernels (checked cell by cell: an uploaded state
// may hold anything), FP32 weights come from shared memory, and a node's three sums leave the warp in
// one reduce-scatter (the same tree as three butterflies) and are accumulated in FP64 in both
// precisions.  Counted in the global histogram cell by cell, with indexed parameter-bank weights: 5e5
// particles at 36 nodes 235 us; 161 us now.
template <int P, int Q, typename R>
__global__ void __launch_bounds__(P1Threads<P, Q, R>::value)
k_observe(const __grid_constant__ StepArgs<P, Q, R> a)
{
    constexpr int NW = P1Threads<P, Q, R>::value / 32, W = HistWin<P, Q, R>::W;
    constexpr int row = (P + 1) & ~1;
    __shared__ double smom[NW][Q * 3];
    __shared__ __align__(16) unsigned long long spsi[sizeof(R) == 4 ? Q * row : 2];
    extern __shared__ __align__(16) uint32_t swin[];   // HistWin when a.use_win
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int j = lane; j < Q * 3; j += 32) acc_zero(smom[warp][j]);
    const Phys<R> &ph = a.ph;
    const Nodes<P, Q, R> &nd = a.nd;
    if constexpr (sizeof(R) == 4)
        for (int j = threadIdx.x; j < Q * P; j += blockDim.x) {
            const float w = a.nd_dev ? a.nd_dev->psi[j] : nd.psi[j];
            spsi[(j / P) * row + j % P] = f2_pack(w, w).v;
        }
    if (a.use_win) clear_window<Q, W>(swin);
    __syncthreads();
    const int64_t NN = (int64_t)ph.Nk * ph.Nk;
    int64_t since_flush = 0;
    for (int64_t base = (int64_t)blockIdx.x * blockDim.x; base < a.N; base += (int64_t)gridDim.x * blockDim.x) {
        if (a.use_win && since_flush + blockDim.x > 65535) {   // 16-bit cells (see phase1_block)
            __syncthreads();
            flush_window<Q, W>(a.Hnext, ph.Nk, a.win_r0, since_flush);
            __syncthreads();
            clear_window<Q, W>(swin);
            __syncthreads();
            since_flush = 0;
        }
        since_flush += blockDim.x;
        const int64_t i = base + threadIdx.x;
        const bool valid = i < a.N;
        R cx[P], cy[P];
        if (valid) load_coeffs(a, i, cx, cy);
#pragma unroll 2
        for (int q = 0; q < Q; ++q) {
            R o[4] = {(R)0, (R)0, (R)0, (R)0};
            if (valid) {
                R kx, ky;
                if constexpr (sizeof(R) == 4) {
                    const ulonglong2 *w = reinterpret_cast<const ulonglong2 *>(spsi + q * row);
                    F2 s2 = f2_pack(0.f, 0.f);
#pragma unroll
                    for (int h = 0; h < P; ++h) s2 = f2_fma(f2_pack(cx[h], cy[h]), (h & 1) ? w[h >> 1].y : w[h >> 1].x, s2);
                    f2_unpack(s2, kx, ky);
                } else {
                    recon_node(nd, q, cx, cy, kx, ky);
                }
                int r, l;
                if (cell_rl(ph, nd.lkx[q], kx, ky, r, l)) {
                    const int rr = r - a.win_r0, ll = l - a.win_r0;
                    if (a.use_win && (unsigned)rr < (unsigned)W && (unsigned)ll < (unsigned)W)
                        atomicAdd(&swin[(q >> 1) * (W * W) + rr * W + ll], 1u << ((q & 1) << 4));
                    else
                        atomicAdd(&a.Hnext[(int64_t)q * NN + r * ph.Nk + l], 1u);
                }
                observe<Q>(ph, kx - nd.xs[q], ky, nd.eps0[q], o[0], o[1], o[2]);
            }
            if constexpr (sizeof(R) == 4) {
                warp_scatter4_add(o, smom[warp] + q * 3, 3, lane);
            } else {
#pragma unroll
                for (int m = 0; m < 3; ++m) {
                    const R v = warp_sum(o[m]);
                    if (lane == 0) acc_add(smom[warp][q * 3 + m], v);
                }
            }
        }
    }
    __syncthreads();
    if (a.use_win) flush_window<Q, W>(a.Hnext, ph.Nk, a.win_r0, since_flush);
    for (int j = threadIdx.x; j < Q * 3; j += blockDim.x) {
        double s = 0.0;
#pragma unroll
        for (int w = 0; w < NW; ++w) s += acc_value(smom[w][j]);
        a.part1[(int64_t)blockIdx.x * (Q * 3) + j] = s;
    }
}

// ------------------------------------------------------------------------------------------
// Initial state: Fermi-Dirac sampling at every node with shared uniforms, projection (FP64).
// ------------------------------------------------------------------------------------------
// The law depends on a node through its band minimum alone, and nodes that differ in the field share
// theirs (36 nodes of two inputs: 6 band minima; a random field: 1).  The sampler runs over the distinct
// band minima; wpsi holds the projection weights summed over the nodes of each.
// One band minimum common to several nodes (a random field alone) in FP64: the sampled state does not depend on z,
// and its higher coefficients and the record's variance over z are the rounding of this kernel and nothing
// else.  That rounding is part of the output, so it is kept: the energy by the iteration (fd_inverse), projected node
// by node (FdPerNode, k_init_nodes; wpsi holds the nodes' own weights).  3e5 particles x 6 nodes: the whole call 12.2 ms with every
// node inverted, 2.3 ms with one inversion per particle (0.6 ms from the table, with another rounding).
template <int Q, typename R> struct FdPerNode {
    static constexpr bool possible = Q > 1 && sizeof(R) == 8;
    static bool value(int ng) { return possible && ng == 1; }
};
template <int P, int Q>
struct InitArgs {
    int32_t ng;        // distinct band minima
    double wpsi[Q * P];
    double eps0[Q];
    double ratio[Q], y0[Q];   // G(w0_q) / Gmax and (eps0_q / kT)^2 (the table of pgc_fd.cuh)
    FdInv fd;
    double mu, kT, hvF;
    double dhalf[P];   // Strang: the stored state leads by half a drift (x coefficients)
    int32_t strang;
    int64_t N, ld;
    uint32_t key0, key1, stream_id;
};

// Every node's |k| lies along the particle's one angle, so |k| is projected and the coefficients are
// its projection times (cos, sin): P multiply-adds per node instead of 2P.  Bound by the FP64 pipe:
// 5e5 particles at 36 nodes 1.55 ms with every node inverted, 0.35 ms over the six band minima.
template <int P, int Q, typename R>
__global__ void __launch_bounds__(128)
k_init(const __grid_constant__ InitArgs<P, Q> ia, R *khat)
{
    const double kw = ia.kT / ia.hvF;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < ia.N; i += (int64_t)gridDim.x * blockDim.x) {
        const U4 r = philox4x32_10((uint32_t)i, ia.stream_id, 0u, 0x10000u, ia.key0, ia.key1);
        const double ue = u01<double>(r.x), uth = u01<double>(r.y);
        double s, c;
        sincos(2.0 * kPi * uth, &s, &c);
        double hk[P];
#pragma unroll
        for (int h = 0; h < P; ++h) hk[h] = 0.0;
#pragma unroll 1
        for (int q = 0; q < ia.ng; ++q) {
            double km;
            if (ia.fd.tab) {
                const double rr = fd_Y<false>(ia.fd, (1.0 - ue) * ia.ratio[q], nullptr) - ia.y0[q];
                km = (rr > 0.0) ? sqrt(rr) * kw : 0.0;
            } else {
                const double e0 = ia.eps0[q];
                const double eps = fd_inverse(e0, ia.mu, ia.kT, ue);
                const double rr = eps * eps - e0 * e0;
                km = (rr > 0.0) ? sqrt(rr) / ia.hvF : 0.0;
            }
#pragma unroll
            for (int h = 0; h < P; ++h) hk[h] += ia.wpsi[q * P + h] * km;
        }
#pragma unroll
        for (int h = 0; h < P; ++h) {
            const double hx = hk[h] * c, hy = hk[h] * s;
            khat[(int64_t)h * ia.ld + i] = (R)(ia.strang ? hx + ia.dhalf[h] : hx);
            khat[(int64_t)(P + h) * ia.ld + i] = (R)hy;
        }
    }
}

// The sampler of an FdPerNode ensemble (a kernel of its own: k_init has no registers for it).
template <int P, int Q, typename R>
__global__ void __launch_bounds__(128)
k_init_nodes(const __grid_constant__ InitArgs<P, Q> ia, R *khat)
{
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < ia.N; i += (int64_t)gridDim.x * blockDim.x) {
        const U4 r = philox4x32_10((uint32_t)i, ia.stream_id, 0u, 0x10000u, ia.key0, ia.key1);
        const double ue = u01<double>(r.x), uth = u01<double>(r.y);
        double s, c;
        sincos(2.0 * kPi * uth, &s, &c);
        const double e0 = ia.eps0[0], eps = fd_inverse(e0, ia.mu, ia.kT, ue), rr = eps * eps - e0 * e0;
        const double km = (rr > 0.0) ? sqrt(rr) / ia.hvF : 0.0;
        const double kx = km * c, ky = km * s;
        double hx[P], hy[P];
#pragma unroll
        for (int h = 0; h < P; ++h) { hx[h] = 0.0; hy[h] = 0.0; }
#pragma unroll 1
        for (int q = 0; q < Q; ++q) {
#pragma unroll
            for (int h = 0; h < P; ++h) {
                hx[h] += ia.wpsi[q * P + h] * kx;
                hy[h] += ia.wpsi[q * P + h] * ky;
            }
        }
#pragma unroll
        for (int h = 0; h < P; ++h) {
            khat[(int64_t)h * ia.ld + i] = (R)(ia.strang ? hx[h] + ia.dhalf[h] : hx[h]);
            khat[(int64_t)(P + h) * ia.ld + i] = (R)hy[h];
        }
    }
}

// Histogram of the particles reconstructed at one arbitrary z (Eq. (24)); psi given in FP64.
template <int P, int Q, typename R>
struct ReconArgs {
    double psi[P];
    R lkx;   // x offset of the grid at z (Lk, or Lk minus half the drift at z under Strang)
};

// Block-private window of kHistAtW x kHistAtW cells around the grid centre (32-bit counts), flushed once
// per block: the ~2000 occupied cells are hot, and counted one by one in the global histogram they
// bounded the kernel (1e6 particles x 6 coefficients: 34 us; 12 us with the window).
constexpr int kHistAtW = 64;
constexpr int kHistAtGrid = 304;

template <int P, int Q, typename R>
__global__ void __launch_bounds__(512)
k_hist_at(const __grid_constant__ StepArgs<P, Q, R> a, const __grid_constant__ ReconArgs<P, Q, R> z,
          uint32_t *out)
{
    __shared__ uint32_t win[kHistAtW * kHistAtW];
    const int Nk = a.ph.Nk, r0 = (Nk - kHistAtW) / 2;   // (< 0 on a smaller grid: the window covers it)
    for (int j = threadIdx.x; j < kHistAtW * kHistAtW; j += blockDim.x) win[j] = 0u;
    __syncthreads();
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < a.N; i += (int64_t)gridDim.x * blockDim.x) {
        R kx = (R)0, ky = (R)0;
#pragma unroll
        for (int h = 0; h < P; ++h) {
            kx += a.khat[(int64_t)h * a.ld + i] * (R)z.psi[h];
            ky += a.khat[(int64_t)(P + h) * a.ld + i] * (R)z.psi[h];
        }
        int r, l;
        if (!cell_rl(a.ph, z.lkx, kx, ky, r, l)) continue;
        const int rr = r - r0, ll = l - r0;
        if ((unsigned)rr < (unsigned)kHistAtW && (unsigned)ll < (unsigned)kHistAtW) atomicAdd(&win[rr * kHistAtW + ll], 1u);
        else atomicAdd(&out[r * Nk + l], 1u);
    }
    __syncthreads();
    for (int j = threadIdx.x; j < kHistAtW * kHistAtW; j += blockDim.x)
        if (win[j]) atomicAdd(&out[(j / kHistAtW + r0) * Nk + j % kHistAtW + r0], win[j]);
}

// ------------------------------------------------------------------------------------------
// Observables at arbitrary points z (Eqs. (35)-(37) of the state reconstructed by Eq. (23) off
// the nodes).  Lane l of every warp evaluates point z_l; a block stages a tile of particles in
// shared memory as (x, y) coefficient pairs and each warp walks a share of the tile, every lane
// reading the same particle (broadcast).  Sums: in R over the particles of one tile, then FP64;
// block partials [kObsGrid][kObsZ][3] = (sum kx/eps, sum ky/eps, sum eps), reduced over the
// blocks in a fixed order by k_obs_fin.
// Bound: instructions (~40 per particle and point, two of them the square root's and reciprocal's
// sequences); one particle at a time at two blocks per SM they were latency-bound, 91 us a pass of 32
// points at 1e6 x 6 coefficients; 60 us with four particles unrolled at four blocks per SM.
// ------------------------------------------------------------------------------------------
constexpr int kObsZ = 32;        // points per pass over the state (one per lane)
constexpr int kObsGrid = 608;    // blocks of one pass (4 per SM)
constexpr int kObsThreads = 256;
constexpr int kObsBatch = 64;    // passes whose results are kept on the device for one copy

template <int P, typename R>
struct ObsTile {   // particles per tile: the staged pairs take at most 32 KB
    static constexpr int value = (2 * P * (int)sizeof(R) * 256 <= 32768) ? 256
                               : (2 * P * (int)sizeof(R) * 128 <= 32768) ? 128 : 64;
};

template <int P, typename R>
struct ObsArgs {
    const R *khat;
    int64_t ld, N;
    R hvF2;
    R psi[kObsZ * P];   // basis at each point; zero rows for unused lanes
    R e0sq[kObsZ];      // eps0(z)^2; 1 for unused lanes
    R xs[kObsZ];        // x shift of the state at the point (Strang; else 0)
};

template <typename R> struct Pair;
template <> struct Pair<float> { using T = float2; };
template <> struct Pair<double> { using T = double2; };

template <int P, typename R>
__global__ void __launch_bounds__(kObsThreads)
k_obs_at(const __grid_constant__ ObsArgs<P, R> a, double *part)
{
    constexpr int T = ObsTile<P, R>::value;
    constexpr int kWarps = kObsThreads / 32;
    using R2 = typename Pair<R>::T;
    __shared__ R2 tile[P * T];
    __shared__ double red[kWarps][kObsZ * 3];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    R ps[P];
#pragma unroll
    for (int h = 0; h < P; ++h) ps[h] = a.psi[lane * P + h];
    const R e0sq = a.e0sq[lane];
    const R xs = a.xs[lane];
    double ax = 0.0, ay = 0.0, ae = 0.0;
    const int64_t ntiles = (a.N + T - 1) / T;
    for (int64_t t = blockIdx.x; t < ntiles; t += gridDim.x) {
        const int64_t base = t * T;
        const int nv = (a.N - base < (int64_t)T) ? (int)(a.N - base) : T;
        __syncthreads();   // the previous tile is consumed
        for (int idx = threadIdx.x; idx < P * T; idx += kObsThreads) {
            const int h = idx / T, j = idx - h * T;
            R2 v;
            v.x = (j < nv) ? a.khat[(int64_t)h * a.ld + base + j] : (R)0;
            v.y = (j < nv) ? a.khat[(int64_t)(P + h) * a.ld + base + j] : (R)0;
            tile[h * T + j] = v;
        }
        __syncthreads();
        R sx = (R)0, sy = (R)0, se = (R)0;
#pragma unroll 4
        for (int j = warp; j < nv; j += kWarps) {   // uniform over the warp; four particles' chains in flight
            R kx, ky;
            if constexpr (sizeof(R) == 4) {
                F2 s = f2_pack(0.f, 0.f);
#pragma unroll
                for (int h = 0; h < P; ++h) {
                    const float2 c = tile[h * T + j];
                    F2 w;
                    asm("mov.b64 %0, {%1, %1};" : "=l"(w.v) : "f"(ps[h]));
                    s = f2_fma(f2_pack(c.x, c.y), w.v, s);
                }
                f2_unpack(s, kx, ky);
                kx -= xs;
            } else {
                kx = (R)0;
                ky = (R)0;
#pragma unroll
                for (int h = 0; h < P; ++h) {
                    const R2 c = tile[h * T + j];
                    kx += c.x * ps[h];
                    ky += c.y * ps[h];
                }
                kx -= xs;
            }
            const R eps = rsqrt_<R>(a.hvF2 * (kx * kx + ky * ky) + e0sq);
            const R ie = (R)1 / eps;
            sx += kx * ie;
            sy += ky * ie;
            se += eps;
        }
        ax += (double)sx;
        ay += (double)sy;
        ae += (double)se;
    }
    red[warp][lane * 3 + 0] = ax;
    red[warp][lane * 3 + 1] = ay;
    red[warp][lane * 3 + 2] = ae;
    __syncthreads();
    if (threadIdx.x < kObsZ * 3) {
        double s = 0.0;
#pragma unroll
        for (int w = 0; w < kWarps; ++w) s += red[w][threadIdx.x];
        part[(int64_t)blockIdx.x * kObsZ * 3 + threadIdx.x] = s;
    }
}

}  // namespace pgc
