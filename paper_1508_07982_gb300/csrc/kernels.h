// Structures shared between the host runtime (capi.cu) and the kernels, and the launchers that
// each per-precision translation unit provides.
#pragma once
#include <cuda_runtime.h>

#include <cstdint>

#include "lbm_internal.h"

namespace lbm {

// A factor c / 2^62, |c| < 2^62, as a signed high and a 31-bit low limb, for products of 64-bit integers.
struct Limb {
    int h;
    uint32_t l;
};

// Constants of the fixed-point collision with FP64 storage (collide64): populations in units of
// 2^(E0 - 60), with rho0 2^-E0 in [2/3, 4/3).
struct FixParams {
    uint32_t base;        // high word of 2^(E0 - 7)
    int top, on;          // 1014 + E0; 1: the fixed-point path may be taken
    double unit;          // 2^(E0 - 60)
    Limb leh, loh;        // le / 2, lo / 2
    Limb ca, cq, cg, third;   // le / 36, le / (8 rho0 2^-E0), lo / 12, 1/3
    long long g0[3];      // fa / 36
};

// Per-level parameters, device-resident so that captured graphs never need rebuilding.
struct LevelParams {
    double le, lo;        // lambda_e, lambda_o (omega, omega for SRT)
    double fa[3];         // 3 rho0 a_L: the body force term is F_a = w_a (e_a . fa), Sec. 2.1
    double acc[3];        // a_L
    float lef, lof;       // the same in FP32, for the FP32-arithmetic kernels
    float faf[3];
    FixParams fix;
};

struct DevLevel {
    void* f[2];           // two PDF grids, [19][ncells]
    const uint8_t* cell;  // [ncells] CK_*
    const int32_t* nbr;   // [nbricks][27], the centre entry holding the brick's BK_* bits
    const int32_t* parent;
    const int32_t* pos;   // [nbricks][3]
    const uint32_t* link;    // [nown * B^3] per owned cell: bit q set = link q needs the general
                             // pull; bits 25-27 and 29 bounce-back; bit 30 = a coupled cell;
                             // bit 31 = not a fluid cell
    const uint2* gcopy[2];     // ghost stream copies of sub-step 1 and 2: {source cell, ghost cell}
    const uint4* gseg[2];      // their segments: {direction + 32 (coarse source), first, count, 0}
    const uint2* gspec[2];     // ghost cells with values that are no copies: {cell, directions}
    int ngseg[2], ngspec[2];
    const uint2* ecopy;        // explosion copies and segments, likewise
    const uint4* eseg;
    int neseg;
    const uint4* cwork;        // coupled cells: {cell, marked links but the coalescing ones, coalescing
                               // links, first child in the finer level's grid}, or with LINK_FACES in the
                               // second word the wall face of direction q at bit 3 (q - 1) of the last two
    int ncwork;
    int nown, nbricks;
    int64_t ncells;
    int N[3];
    double u0[3];         // storage shift velocity: shifted layouts hold f - f^eq(rho0, u0); 0 for FP64
};

struct StepArgs {
    DevLevel lv, co, fi;  // this level, the next coarser, the next finer
    int cur, cur_c, cur_f;
    const void* sq[19];   // the 19 directions' planes of this level's current grid and of the other one
    void* dq[19];
    int substep;          // 1: ghost layers hold the exploded (coarse) values; 2: layers 1-2 hold
                          // their sub-step-1 stream
    int LB;
    int per;              // bit a set: axis a periodic
    int fslip;            // bit f set: face f (x-, x+, y-, y+, z-, z+) is free-slip
    const LevelParams* params;
    const float* wallf;   // `wall` in FP32 for the FP32-arithmetic walk, row 7 zero without a storage shift
    const double* wall;   // [8][19] bounce-back terms 6 w_a rho0 (e_a . (u_w - u0)): faces 0-5,
                          // row 7 obstacles (u_w = 0), row 6 unused
    int wall_terms;       // bit f set: row f of `wall` holds a nonzero term (row 7: and obstacle_term)
    double rho0, inv_rho0;
    double* totals;       // per-warp post-streaming moments of the owned cells, or NULL
    int obstacle_term;    // 1: obstacle bounce-backs add wall row 7 (a nonzero storage shift)
    float two_u0[3];      // 2 u0 and 2 e_a . u0 of the storage shift (FP32 arithmetic; 0 unshifted)
    float e_two_u0[19];
    int wwarps;           // the walk's warps (its totals entries)
};

// Bits of the per-cell link mask.
constexpr uint32_t LINK_NOT_FLUID = 1u << 31;
constexpr uint32_t LINK_COUPLED = 1u << 30;       // a coupled cell: the walk skips it
constexpr uint32_t LINK_FACES = 1u << 28;         // coupled cells' entries: bounce-backs with a face per direction
constexpr uint32_t LINK_BOUNCE_ONLY = 1u << 29;   // face of the wall term in bits 25-27
constexpr uint32_t LINK_ALL = 0x7FFFEu;   // directions 1..18

// Levels whose density and velocity one launch reads out: CTAs of 256 cells, level after level.
struct MacroLevel {
    const void* f;        // the current grid
    const uint8_t* cell;
    const LevelParams* params;
    int64_t cells, ncells;   // owned cells, cells of a direction's plane
    int64_t offset;       // first cell in the output
    int ctas;
};
struct MacroArgs {
    MacroLevel lv[LBM_MAX_LEVELS];
    double u0[3];         // storage shift velocity
};

// Warps per CTA of the FP32 / FP16 walk; each warp takes 128 consecutive cells of a brick.
constexpr int kWalkWarps = 2;
// Threads per CTA of the coupled cells' and the ghost work, and of the FP64 kernel (one cell each).
constexpr int kSideThreads = 128;

// Launchers (one set per storage precision: 0 FP64, 1 FP32S, 2 FP16S).
struct Launchers {
    void (*step)(const StepArgs& a, int collision, int grid, cudaStream_t s);
    void (*init)(const DevLevel& lv, int cur, int LB, const LevelParams* P, double rho0, const double* rho,
                 const double* u, int uniform, const double u_const[4], int collision, cudaStream_t s);
    void (*macro)(const MacroArgs& a, int ctas, double rho0, double* rho, double* u, int64_t ustride, cudaStream_t s);
    void (*get_pdfs)(const DevLevel& lv, int cur, int LB, double rho0, double* out, cudaStream_t s);
    void (*set_pdfs)(const DevLevel& lv, int cur, int LB, double rho0, const double* in, cudaStream_t s);
    void (*reduce)(const DevLevel& lv, int cur, int LB, const LevelParams* P, double rho0, double w, double* partial,
                   int grid, cudaStream_t s);
    void (*explode)(const DevLevel& lv, const DevLevel& co, int cur, int cur_c, cudaStream_t s);
    // One phase of a batch of forests: args[n] per forest, prefix[n+1] its first CTA of the phase's
    // `total`, owner[total] the forest of each CTA.
    void (*step_batch)(const StepArgs* args, const int* prefix, const int* owner, int total, int collision, int LB,
                       cudaStream_t s);
    void (*explode_batch)(const StepArgs* args, const int* prefix, const int* owner, int total, cudaStream_t s);
    // Whether the coupled cells and the ghost work run in kernels of their own (FP32/FP16 storage) beside the
    // walk of F_L(s), `grid` CTAs each; for a batch of forests, in one, as step_batch.
    bool split_side;
    void (*coupled)(const StepArgs& a, int collision, int grid, cudaStream_t s);
    void (*ghost)(const StepArgs& a, int grid, cudaStream_t s);
    void (*side_batch)(const StepArgs* args, const int* prefix, const int* owner, int total, int collision, int LB,
                       cudaStream_t s);
};
const Launchers& launchers_f64();
const Launchers& launchers_f32();
const Launchers& launchers_f16();

}  // namespace lbm
