// Declarations of the screening path for D <= 128 (internal).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>
#include <stddef.h>

namespace fg {

constexpr int SCR_MAX_K = 4096;
// Points per round of launches: capacity of the per-point buffers.  Every launch has a tail and the sort by component a part that
// does not depend on the points: at D = 128, K = 1024 a step over 10M points took 13.9 ms with 2^18, 11.9 with 2^19, 10.9 with 2^20
// (and 18.3 with 2^17: that X stays in L2 between the kernels does not make up for it).
constexpr int64_t SCR_PIECE = 1 << 20;
constexpr int SCR_TILE = 256;                // points per tile of the sweep
constexpr int SCR_SLOTS = 16;                // room for marked pairs per point (on average over the 32 points of a warp)
constexpr int SCR_WORDS = 8;                 // room for words (32 positions, mask) per point, on average over the points of a warp
constexpr int SCR_EXTRA = 2;                 // and, per point of a piece, for the rows that do not fit there
constexpr int64_t SCR_PAIRS = SCR_PIECE * (SCR_SLOTS + SCR_EXTRA);
constexpr int SCR_SEG = 64;                  // pairs per work item of the statistics
constexpr int SCR_MARKS = 10;                // marked pairs of a piece, per point of a full one: beyond them the piece counts as dense
constexpr int ST_THREADS = 128, ST_CTAS = 3;  // of the statistics: threads per CTA, CTAs per SM
constexpr int SCR_STAT_WARPS = 148 * ST_CTAS * (ST_THREADS / 32);      // in one wave, each with a run of work items
constexpr int SCR_RANGES = 3 * 148;          // CTAs of the pair evaluation and of the sort by component (at most)
constexpr int SCR_LL = 4096;                 // log-likelihood partial sums (one per CTA of a launch), then one per component
constexpr int SCR_DIM_BLOCKS = 64;
constexpr int SCR_GROUP = 32768;             // points of a group that launch_screen_groups takes (16-bit cursors; one CTA sorts a group)
constexpr int PR_ROWS = 4, PR_GROUPS = 16, PR_CTAS = 16;     // rows that are looked at ahead of a call's sweep: see screen_probe
constexpr int SCR_SPILL = 25, SCR_MAX_SMS = 160;      // see screen_sweep_kernel

// Control words (in the context's result block, so that they travel to the host with the log-likelihood).
enum { SC_DENSE = 0,      // set when a piece marks too many pairs or is not finite, or a wait ran out: later kernels return at once, the caller takes the dense path
       SC_MARKS,          // pairs marked in the current piece
       SC_OVF,            // rows of the current piece that left the sweep without a list
       SC_EXTRA,          // pairs of those rows
       SC_TICKET_A, SC_TICKET_B,
       SC_PROBED,         // pairs of the rows that were looked at ahead of the sweep
       SC_ACTIVE,         // components with a weight
       SC_KEPT,           // kept pairs of all pieces (saturating)
       SC_DONE,           // pieces of the call that are done (SC_DENSE: the others are left to the dense kernels)
       SC_ILL, SC_FALLBACK,      // parameters or a piece of an assignment that the FP32 kernels have to take (see launch_screen_gate)
       SC_WORDS };

struct ScreenBuffers {
    float* sd;            // [128] power-of-two scale per dimension
    float* gd;            // [128] centre
    double* dimpart;      // [SCR_DIM_BLOCKS][4][128]
    float4* prm;          // [K] c, error allowance (constant, per unit of |u|^2), largest |nu|
    float* key;           // [K] the allowance of a typical point
    unsigned char* p;     // coefficients [Kpad / 128][screen_group_bytes]
    int4* blk;            // [SCR_MAX_K / 32] of 32 positions: largest allowances (as bits), whether one is capped
    int* comp_of;         // [Kpad]
    unsigned* probe;      // [PR_GROUPS][PR_ROWS + 1] of the probed rows: largest lower bound (see order_up); CTAs that are done
    unsigned char* y;     // rows of u [SCR_PIECE][16-byte chunks of 8 halves]
    float* n2;            // [SCR_PIECE] |u|^2
    unsigned* pt_off;     // [SCR_PIECE] where a point's pairs start
    int* pt_cnt;          // [SCR_PIECE] how many there are (until the evaluation also where the words are and how many)
    uint2* words;         // [SCR_PIECE][SCR_WORDS] the sweep's marks: a mask, the block of 32 positions it belongs to
    unsigned long long* spill;        // [SCR_MAX_SMS][SCR_SPILL][256]
    unsigned short* ids;  // [SCR_PAIRS] component of a kept pair
    float* val;           // [SCR_PAIRS] its responsibility (-1: the point's only pair)
    uint2* srt;           // [SCR_PAIRS] (row, responsibility) sorted by component
    int* counts;          // [SCR_RANGES][K]
    int* totals;          // [K]
    int* off;             // [K + 1] where a component's pairs start in srt
    int* segoff;          // [K + 1] where its work items start
    double* part;         // [SCR_STAT_WARPS + K][2 D + 2] (see screen_stats_kernel)
    double* ll;           // [SCR_LL + K]
    int* ovf;             // [SCR_PIECE]
    int* ctl;             // [SC_WORDS]
    int test_silent;      // (time-out test, see SweepParams)
};

bool screen_supports(int D, int K);
inline int screen_kpad(int K) { return (K + 127) / 128 * 128; }
// (unit: the linear terms alone, see em_screen.cu)
__host__ __device__ inline int screen_atoms(int D, bool unit) { return unit ? (D + 63) / 64 : (D + 31) / 32; }
__host__ __device__ inline size_t screen_group_bytes(int D, bool unit = false) { return 4096 + (size_t)screen_atoms(D, unit) * 16384; }

// A call's data X [n] (n = 0: none), of which some rows are looked at ahead of the sweep, and what the sweep will be asked (see launch_screen_sweep).
struct ScreenProbe { const float* X; int64_t n; float margin; int top; float max_marks; };
// Parameters -> w2, c2, c2d (as launch_prepare_fp32, with the same checks), coefficient plane and tables.  unit: k-means (mu =
// centroids; pi, var not read; log2 z = -F |x - mu|^2, F a power of two; one that is not finite or too far out sets SC_DENSE and no status).  SC_DENSE: 0, or 1
// where the probed rows have too many pairs.  Clears the partial log-likelihoods.
cudaError_t launch_screen_prepare(cudaStream_t s, int D, int K, const float* pi, const float* mu, const float* var, bool unit,
                                  const ScreenProbe& probe, const ScreenBuffers& b, float* w2, float* c2, double* c2d, int* status);
// One piece of n <= SCR_PIECE points: (plane,) sweep, rows without a list.  unit: as in launch_screen_prepare.  margin: log2 units below a point's best value down to
// which pairs are marked (40, or 0 for the arg-max alone); top: so many of its largest pairs are marked in any case (1 to 4).  max_marks: pairs per point up to which the screening pays; stats:
// statistics are to follow, which have room for SCR_MARKS of them.
cudaError_t launch_screen_sweep(cudaStream_t s, const float* X, int64_t n, int D, int K, bool unit, float margin, int top, float max_marks, bool stats,
                                const float* mu, const float* w2, const double* c2d, const ScreenBuffers& b, int* status, int sms,
                                int64_t* launches);
// SCREEN_ARGMAX: how near ties are decided.  g: NULL, or the centre of the FP32 tile kernel (then w = 1, c = 0); else weight and constant
// of the unit mixture that the tensor assignment is given.
struct ScreenTie { const float* g; float w, c; };
// Exact values of the marked pairs.  SCREEN_EM: responsibilities of the pairs within 2^-40 of their point's total, counted per
// component; SCREEN_LOGP: logp[i]; SCREEN_ARGMAX: idx[i], and the pair itself kept with weight 1 for the statistics.
// SCREEN_TOP: the m largest pairs of every point into idx [n][m] and (may be NULL) their responsibilities into resp [n][m].
enum { SCREEN_EM = 0, SCREEN_LOGP = 1, SCREEN_ARGMAX = 2, SCREEN_TOP = 3 };
cudaError_t launch_screen_eval(cudaStream_t s, int mode, const float* X, int64_t n, int D, int K, const float* mu, const float* w2,
                               const double* c2d, const ScreenBuffers& b, float* logp, int32_t* idx, bool count = true, int m = 1, float* resp = nullptr,
                               const ScreenTie* tie = nullptr);
// (count: leave the number of kept pairs per component and range for launch_screen_stats)
// Behind the last piece of an asynchronous assignment, for its piece p: *gate = 0 and *fallback = 0 if the tile kernels have to do it, 1
// and 1 if the FP32 kernels have to, 1 and 0 if it is done.  gate: the tile kernels' flag for parameters that are not for them, looked
// at when `first` (NULL: there are no tile kernels).
cudaError_t launch_screen_gate(cudaStream_t s, const ScreenBuffers& b, int* gate, int* fallback, int64_t p, bool first);
// Statistics of the kept pairs: sorted by component, summed in fixed segments, added to (Nk, S1, S2) in float64.
cudaError_t launch_screen_stats(cudaStream_t s, const float* X, int64_t n, int D, int K, const float* mu, const float* w2,
                                const double* c2d, const ScreenBuffers& b, double* Nk, double* S1, double* S2, int64_t* launches);

// After the evaluation (SCREEN_EM): Fisher vectors of `groups` groups of consecutive points (n in all) of the piece (group g =
// g_len[g] <= SCR_GROUP points from row g_start[g] on, in order) into fv [groups][2][K][D].  g_off: groups * (K + 1) ints of scratch.
cudaError_t launch_screen_groups(cudaStream_t s, const float* X, int64_t n, int groups, int D, int K, const int* g_start, const int* g_len, int* g_off,
                                 const float* pi, const float* mu, const float* var, const float* w2, const double* c2d,
                                 const ScreenBuffers& b, float* fv, int64_t* launches);
// k-means: new centroids from (Nk, S1) as launch_screen_stats left them (unit parameters), points and inertia per centroid.
cudaError_t launch_screen_centroids(cudaStream_t s, int D, int K, const float* cent_in, const double* Nk, const double* S1,
                                    const ScreenBuffers& b, float* cent_out, int64_t* counts, double* inertia_k);

}  // namespace fg
