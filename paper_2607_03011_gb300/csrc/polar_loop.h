// polar_loop.h -- the polar loop's tables and parameters (polar_loop.cu), built by the plan.
#pragma once
#include "types.h"  // ControlMat, GemmGroup, TileFlags

namespace isoloco {

// Phases of one iteration, in the order the tiles are handed out.
enum LoopKind : int { kLoopW = 0, kLoopGram = 1, kLoopGramGs = 2, kLoopPoly = 3, kLoopUpdate = 4 };
constexpr int kLoopPhases = 5;
// Arrival counters of a matrix (the two Gram kinds share one: a matrix has only one of them).
enum LoopArrival : int { kArrW = 0, kArrGram = 1, kArrPoly = 2, kArrUpdate = 3 };
constexpr int kArrKinds = 4;

// One shape bucket in one phase: its GEMM group and what the walk and the control step need.
struct LoopGroup {
    GemmGroup g;
    ControlMat cm;   // of the bucket's first matrix (the others follow at gpart_slot + b n_gtiles)
    int tiles;       // output tiles of a matrix in this phase
    int dep_tiles;   // output tiles of a matrix in the phase whose arrivals it waits for
};

struct LoopPhase {
    TileFlags f;
    int kind;
    int first;           // its first group
    int count;           // the matrices of its groups
    // order in which they come up (walk_matrix in polar_loop.cu): the first `regular` in rising
    // or falling order, the first `skip` of these after the next `skip`, the others (Gram-side)
    // at position side_at
    int regular, side_at, skip, falling;
};

// Everything the loop reads besides the matrices' states and counters is in its parameters:
// an acquire (each poll of a counter) empties L1, the constant bank keeps them at hand.
template <int NG>
struct LoopParams {
    LoopGroup groups[NG];
    LoopPhase phases[2 * kLoopPhases];  // odd and even iterations (ping-pong buffers)
    MatState* state;
    const float* fin_part;
    uint32_t* ctl;             // [matrices]
    uint32_t* arr;             // [matrices][kArrKinds]
    unsigned long long* prof;  // null, or [kLoopPhases] nanoseconds per phase (phases then run apart)
    uint32_t* err;
    int max_t;                 // iterations at most (every matrix is done before)
    int max_iter;
    float tol;
    int fast_steps;
    int4 gram_one, upd_one;
    int gs_on;
};
// Kernel parameters hold 32,764 bytes: plans whose two iterations need more than kLoopGroups
// groups (three per shape bucket and iteration, four for a Gram-side one) keep the graph of launches.
constexpr int kLoopGroupsSmall = 32, kLoopGroups = 96;
static_assert(sizeof(LoopParams<kLoopGroups>) <= 32764, "kernel parameter space");

// Shared memory: the ring and staging of the GEMM, then barriers and the tile queue.
constexpr int kLoopTailBytes = 2048;
constexpr int kLoopSmemBytes = kRingBytes + kEpiStagingBytes + 1024 /*align*/ + kLoopTailBytes;
static_assert(kLoopSmemBytes <= 232448, "227 KB of shared memory per CTA");

template <int NG>
cudaError_t launch_polar_loop(const LoopParams<NG>& p, int clusters, cudaStream_t stream);

}  // namespace isoloco
