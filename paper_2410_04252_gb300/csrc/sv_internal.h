// Internal structures shared by the planner, the kernels and the C ABI.
#pragma once

#include <cstdint>
#include <functional>
#include <string>
#include <vector>

#include "../../include/sv.h"

namespace sv {

constexpr int kMaxQubits = 40;
constexpr int kMaxSpan = 10;         // coset dimension limit of an EVC / H|psi> pass
constexpr int kMaxRunBits = 7;       // longest contiguous run of a coset pass (2^7 amplitudes)
constexpr int kMaxPassStrings = 384; // strings per EVC pass (shared-memory accumulators and constants)
constexpr int kMaxPassOps = 256;       // gates per shared-memory pass
constexpr int kMaxGroupStrings = 256; // distinct Z masks sharing one X/Y mask in one group

// ---------------------------------------------------------------- planning --

// One schedulable operator: a gate (QSU) or a Pauli string (EVC).
struct Op {
    int32_t kind = 0, nq = 0;
    int32_t q[4] = {-1, -1, -1, -1};
    int32_t param = -1, mat = -1;
    uint64_t tmask = 0;   // logical targets T(op)
};

// A tile of Sec. IV: operators applied under one qubit mapping.
struct Tile {
    int32_t begin = 0, end = 0;      // range of the schedule (order)
    uint64_t local_mask = 0;         // logical local set Q_L
    std::vector<int32_t> pairs;      // QR before the tile: (local phys, global phys) pairs
    std::vector<int32_t> l2p;        // layout in force during the tile
    uint64_t intra_mask = 0;         // hierarchical tiling: logical intra set Q_intra (Alg. 4/5)
};

// Device-side gate of a pass: kind, targets as TILE-LOCAL bit positions.  A
// target t >= kOutTarget is outside the staged tile (only diagonal gates on
// global qubits under the diagonal exemption): physical bit t - kOutTarget,
// constant over a tile.
constexpr int kOutTarget = 64;
struct DevOp {
    int32_t kind;
    int8_t t[4];
    int32_t gate;     // index in the caller's gate list (coefficient / gradient slot)
    int32_t mat;      // complex offset into the matrix array, or -1
    int32_t pm;       // register-blocked passes: complex offset of the prepared matrix (PrepMat), else -1
};

// A caller matrix of a register-blocked pass, prepared once per call: M'[u][w]
// = M[j(u)][j(w)] with u, w over the gate's register bits in ascending order
// and j the caller's index (bit t of j = bit perm[t] of u), followed by its
// conjugate transpose (dim * dim elements each).
struct PrepMat {
    int32_t nq, src, dst;    // targets; complex offsets into the caller's and the prepared array
    int8_t perm[4];
};

// One shared-memory pass of K-GATE / K-ADJ.
struct GatePass {
    int32_t tile = 0;
    int32_t k = 0, nlow = 0;          // staged bits, of which the nlow lowest are contiguous
    uint64_t bits = 0;                // physical staged bits
    int32_t op_begin = 0, op_end = 0; // into QsuPlan::ops
    int32_t ph_begin = -1, ph_end = -1;  // register phases (register-blocked passes), else -1
    int32_t pairs = 0;                   // the phases hold pair rotations (1: Givens, 2: double excitations)
    int32_t others = 0;                  // 1: the phases hold gates besides pair rotations
    int32_t mat1 = 0;                    // 1: the phases hold 1-qubit matrices
    int32_t dense = 0;                   // 1: the phases hold 2- or 4-qubit matrices (forward only)
    int32_t db_begin = 0, db_end = 0;    // diagonal blocks of the pass (register-blocked passes)
    int32_t st_begin = 0, st_end = 0;    // steps of the pass's phases
    int32_t area = 0;                    // bytes of the pass's diagonal-block data (shared memory)
    int32_t mem_begin = 0, mem_end = 0;  // the pass's diagonal-block members (QsuPlan::dmembers)
};

// A run of consecutive diagonal operations (RZ, CZ) inside one register
// phase, applied as one diagonal operator.  Two kinds:
//  * register block (kind 0): RZ / CZ on register bits and CZs between a
//    register and a thread bit; the factor of register amplitude v of a
//    thread is a table entry T[v][zm], zm = the register bits on which the
//    thread's register-thread CZs put a Z (a per-thread constant);
//  * thread block (kind 1): RZ / CZ on thread bits only; one complex factor
//    per thread for all its amplitudes.  Such gates commute with everything
//    else in the phase, so all of a phase's go into one thread block.
// Every member op carries mat = -2 - (block index).  smem: byte offset of
// the block's data in the kernels' block area (tables and per-thread data).
struct DiagBlock {
    int32_t op_begin, op_end;     // member ops (consecutive in QsuPlan::ops)
    int32_t m_begin, m_end;       // into QsuPlan::dmembers
    uint32_t rmask;               // register tile bits of the phase
    int32_t kind;                 // 0 register block, 1 thread block
    int32_t smem;
    uint32_t lanes;               // the phase's lane bits (Phase::lanes)
};
enum { SV_DM_REG_RZ = 0, SV_DM_THR_RZ = 1, SV_DM_REG_CZ = 2, SV_DM_THR_CZ = 3, SV_DM_MIX_CZ = 4 };
struct DiagMember {
    int32_t type;     // SV_DM_*
    int32_t a, b;     // register index (0..r-1) or tile bit, per type; MIX_CZ: a register, b tile bit
    int32_t op;       // index into QsuPlan::ops (coefficient and gradient slot)
};
constexpr int kMaxPassDiag = 24;       // diagonal blocks per register-blocked pass
// Register-blocked passes: each thread holds 2^kRegBits amplitudes of a tile,
// so a tile of 2^k amplitudes takes 2^(k - kRegBits) threads, at least a warp.
constexpr int kRegBits = 4;
constexpr int kRegMinTile = kRegBits + 5;
constexpr int kL2QubitsC128 = 22;    // complex128 states of 64 MB (half of L2)

// A register phase of a register-blocked pass: each thread holds the
// amplitudes spanned by the tile bits in rmask; ops [op_begin, op_end) are
// applied in registers (non-diagonal gates on rmask bits, diagonal gates on
// any bits).
struct Phase {
    uint32_t rmask;
    int32_t op_begin, op_end;
    int32_t st_begin, st_end;   // steps of the phase (QsuPlan::steps)
    uint32_t lanes;             // tile bits held by the lane bits of the thread index (phase_lanes)
};

// A step of a register phase, executed as one unit by the register-blocked
// kernels.  ROT: RY gates on distinct register bits (they commute), ops
// [op_begin, op_end) ordered by register bit, a = the register-bit mask.
// DIAG: a diagonal block (a = its index in QsuPlan::dblocks), ops = its
// members.  OP: one operation (a = op_begin), applied by the generic code.
// SCALE: no operation; the register kernels apply the RYs without their larger
// coefficient (each at least 2^-1/2) and the product of these factors at the
// store, so that amplitudes grow by up to 2^(1/2) an RY meanwhile: 2^128 over a
// full pass, past FP32.  A complex64 pass has a SCALE step after at most
// kScaleRYs RYs, which applies the product there unless it is above 2^-4 (then
// the next one does): what the registers hold stays within 2^52 of the
// amplitudes, the gradient sums, products of two, within 2^104.
enum { SV_STEP_ROT = 0, SV_STEP_DIAG = 1, SV_STEP_OP = 2, SV_STEP_SCALE = 3 };
constexpr int kScaleRYs = 96;
constexpr int kMaxScaleSteps = kMaxPassOps / (kScaleRYs - 3);   // (a ROT step holds up to four RYs)
// The shared-memory slot of tile index i in the register-blocked passes: a
// linear (XOR) swizzle, so that slot(a | b) = slot(a) ^ slot(b) for disjoint
// a, b.  It keeps bit 0 (an even index and its successor stay one 16-byte
// pair of complex64, so tiles move by 16-byte accesses and a phase that holds
// tile bit 0 gathers pairs) and XORs bits 1..3 with the bit triples 4..6 and
// 7..9 and with independent mixtures of bits 10..12: whatever 4 of 13 bits a
// phase holds in registers, the others still reach every value of the low
// bits (at most 7 of the 12 bits fall into any one plane of the three).
#ifdef __CUDACC__
#define SV_HD __host__ __device__
#else
#define SV_HD
#endif
SV_HD inline uint32_t swz_slot(uint32_t i) {
    const uint32_t y = (i >> 10) & 7u;
    return i ^ ((((i >> 4) ^ (i >> 7) ^ y ^ (y << 1) ^ (y >> 2)) & 7u) << 1);
}
// Shared memory of a register-blocked pass of k staged bits (amplitudes of
// amp bytes): the block area needs at most this much beyond the tiles, tables
// and accumulators, and each block takes diag_block_bytes() of it.
constexpr int kRegSmemLimit = 226 * 1024;
constexpr int kAdjSlotStride = 17;   // adjoint gradient slots per op (one per warp, padded)
inline int diag_block_bytes(int kind, int k, int amp) {
    const int V = 1 << kRegBits, NT = 1 << (k - kRegBits);
    return kind == 0 ? V * V * amp + NT : NT * amp;
}
inline int reg_pass_fixed_bytes(int k, int nlow, int nops, int nsteps, int nphases, int amp, bool pairs) {
    // adjoint (the larger): psi and lambda tiles, high offsets, chunk offsets,
    // (c, s) per op, steps, block headers and members, phases with their
    // thread bases and register offsets, per-warp gradient slots, the RY
    // factor per step, pair rotations' coefficients, alignment
    return 2 * (1 << k) * amp + 8 * (1 << (k - nlow)) + 256 + nops * amp + 16 * nsteps + 32 * kMaxPassDiag +
           16 * nops + nphases * (2 * (1 << (k - kRegBits)) + 16 + 16) + nops * kAdjSlotStride * 8 +
           8 * (nsteps + 1) + (pairs ? 4 * amp * nops : 0) + 320;
}
struct RegStep {
    int32_t type, a;
    int32_t op_begin, op_end;
};

struct QsuPlan {
    int n = 0, g = 0, nL = 0;
    std::vector<int32_t> order;       // schedule g at tile granularity
    std::vector<Tile> tiles;
    std::vector<GatePass> passes;
    std::vector<DevOp> ops;           // pass operations, pass by pass, in execution order
    std::vector<Phase> phases;        // register phases of register-blocked passes
    std::vector<RegStep> steps;       // steps of the register phases
    std::vector<DiagBlock> dblocks;   // diagonal blocks of register phases
    std::vector<DiagMember> dmembers;
    std::vector<PrepMat> prep;        // caller matrices of register phases
    int32_t prep_elems = 0;           // complex elements of the prepared array
    std::vector<int32_t> init_l2p, final_l2p;
    int32_t nqr() const {
        int32_t c = 0;
        for (auto &t : tiles) c += t.pairs.empty() ? 0 : 1;
        return c;
    }
};

// Few-string expectation passes (every group one string): at most this many groups.
constexpr int kEvcFew = 8;

// EVC / H|psi>: strings grouped by physical X/Y mask, groups packed into
// coset passes (see kernels).
struct EvcString {
    uint64_t z;        // physical Z/Y mask
    int32_t nY;        // |x & z| mod 4
    uint32_t bz;       // bit j = parity(basis_j & z) for the pass's span basis
    double coef;       // summed coefficient of the merged terms
};
struct EvcGroup {
    uint64_t x;        // physical X/Y mask
    uint32_t X;        // partner offset inside the coset tile: (c << kl) | (x & (2^kl - 1))
    int32_t s_begin, s_end;   // strings (slots)
};
// Expectation passes over many X/Y masks of one or two staged bits (a
// Jordan-Wigner Hamiltonian's): register phases.  In a phase a thread holds
// the 2^r amplitudes spanned by r staged-index bits (rmask), so the pairs of
// every group whose mask lies in them are pairs of its own registers.
// A group's pair index p (element v with bit h = 0, partner v ^ x): its top
// bit is register bit l, the others the remaining register bits ascending.
// An item is one or two strings (the sum and the difference over the top bit)
// that share everything else: the part, the frequency w over the other bits,
// the thread's frequency tau and z on the coset representatives.
constexpr int kEvcRegPhases = 12;    // phases of one pass (shared-memory tables)
constexpr int kEvcRegItems = 16;     // items of one phase (two bits each in the thread's sign word)
struct EvcRegPhase {
    uint32_t rmask, lanes;           // staged-index bits in registers and in the lane bits (phase_lanes)
    int32_t i_begin, i_end;
};
struct EvcRegItem {                  // an item of the Re part and one of the Im part of a group
    uint64_t z[2];
    uint32_t tau[2], w[2];
    int32_t slot_sum[2], slot_dif[2];   // strings of the pass (relative), or -1
    uint32_t ctl;                    // bits 0..3: signs (Re sum, difference, Im sum, difference); bits 8..15: place
                                     // of (h, l); bits 16, 17: the part is there; bit 18: another item of the group
                                     // came before without an Im part, its Re products are still held
    uint32_t pad;
};

// Passes of few strings, one per X/Y mask (random strings), whose span basis
// is the masks themselves: a string then flips one span bit (and perhaps bit
// 0) of the staged index.  Half of the warps hold bit 0 and the first four
// span bits in registers, half bit 0 and the other four, and every string
// goes to the half that holds its pairs; the strings that neither half holds
// (masks inside the span of the others) read their partners.
constexpr int kEvcUnitSpan = 8, kEvcUnitRun = 5, kEvcUnitMax = 8;   // span bits, run bits, strings per half
struct EvcUnitItem {
    uint64_t z;                      // on the coset representatives
    uint32_t tau;                    // staged-index frequency
    uint32_t w;                      // of it, the four register bits besides the flipped span bit (all five: code 16)
    uint32_t X;
    uint32_t code;                   // 4 * (register bit h - 1) + 2 * (bit 0 flips) + (Im: 1); 16, 17: partners read
    uint32_t neg;
    int32_t slot;                    // string of the pass (relative)
};

struct CosetPass {
    int32_t kl = 0, m = 0;
    uint64_t basis[kMaxSpan] = {};    // span vectors over bits >= kl, reduced
    int32_t pivot[kMaxSpan] = {};
    int32_t g_begin = 0, g_end = 0;   // groups
    int32_t s_begin = 0, s_end = 0;   // strings (slots), contiguous
    // register phases (k_evc_reg): they take the groups before g_reg
    // (half of the warps run phases [rp_begin, rp_begin + rp_first), the others the rest)
    int32_t rp_begin = 0, rp_end = 0, rp_first = 0, g_reg = 0, s_reg = 0;
    int32_t ri_begin = 0, ri_end = 0;
    // k_evc_unit: strings of the first and of the second half of the warps
    int32_t u_begin = 0, u_mid = 0, u_end = 0;
};

struct EvcPlan {
    int n = 0, g = 0, nL = 0;
    std::vector<int32_t> order;       // term order at tile granularity
    std::vector<Tile> tiles;
    std::vector<int32_t> tile_pass_begin, tile_pass_end;
    std::vector<char> tile_wide;      // 1: strings wider than n_L, pairs cross chunks
    std::vector<CosetPass> passes;
    std::vector<EvcGroup> groups;
    std::vector<EvcString> strings;   // slots
    std::vector<EvcRegPhase> rphases;
    std::vector<EvcRegItem> ritems;
    std::vector<EvcUnitItem> uitems;
    std::vector<int32_t> term_slot;   // per input term
    std::vector<int32_t> init_l2p, final_l2p;
    int32_t nqr() const {
        int32_t c = 0;
        for (auto &t : tiles) c += t.pairs.empty() ? 0 : 1;
        return c;
    }
};

struct PlanOptions {
    int tile_bits = 12, low_bits = 5;
    int evc_low_bits = 7, evc_span = 6;
    bool pad_highest = true;
    int fuse_max = 0;            // gate operations per gate pass (0 = as many as fit)
    int hier_intra = -1;         // >= 0: hierarchical tiling (Alg. 4/5) with this many intra qubits
    int max_diag = kMaxPassDiag; // diagonal blocks per register-blocked pass (shared-memory budget)
    int amp_bytes = 8;           // 8 complex64, 16 complex128 (shared-memory budget of the blocks)
    bool reg_pairs = true;       // Givens, double excitations and dense matrices may run in register phases
    int image_limit = 0;         // bytes for a pass's tables when it is less than the shared memory leaves (0)
    int reg_threads = 0;         // register phases on CTAs of this size (the batched kernel), 0 = 2^(k - kRegBits)
    bool diag_exempt = false;    // QSU: diagonal gates (RZ, CZ) never ask for a QR (per-chunk phases)
    // One greedy step of Alg. 6 done elsewhere (on the device): given the
    // distinct X/Y supports xs with remaining weights w, return the rank of
    // the first global set (lexicographic order) of maximal count and that
    // count.  Empty: the host search with incrementally maintained counts.
    std::function<std::string(const std::vector<uint64_t> &xs, const std::vector<int32_t> &w, int n, int nG,
                              int64_t &rank, int64_t &count)>
        alg6_step;
};

// Returns an empty string on success, else the error message.
std::string validate_gates(int n, const sv_gate *gates, size_t m, size_t np, size_t nmats);
std::string plan_qsu(int n, int g, const sv_gate *gates, size_t m, bool lazy,
                     const PlanOptions &o, const std::vector<int32_t> &l2p_init, QsuPlan &out);
std::string plan_evc(int n, int g, const sv_pauli *p, const double *coeffs, size_t nterms,
                     bool lazy, const PlanOptions &o, const std::vector<int32_t> &l2p_init,
                     EvcPlan &out);
// H|psi> grouping: one tile, no QR, cosets over all n bits.
std::string plan_hpsi(int n, const sv_pauli *p, const double *coeffs, size_t nterms,
                      const PlanOptions &o, const std::vector<int32_t> &l2p, EvcPlan &out);
// The kernels of the expectation passes that differ from the general ones:
// few strings by k_evc_unit, else masks of one or two staged bits by k_evc_reg.
void plan_evc_kernels(EvcPlan &P, sv_dtype dt);
constexpr int kXformMinStrings = 16;  // groups with at least this many strings take the transform path
constexpr int kEvcRegMinGroups = 6;
// Write a bit permutation from layout `from` to layout `to` as at most two
// sets of disjoint physical bit swaps (every permutation is a product of two
// involutions).
void permutation_swaps(const std::vector<int32_t> &from, const std::vector<int32_t> &to,
                       std::vector<std::vector<int32_t>> &swap_sets);

uint64_t hash_bytes(const void *p, size_t n, uint64_t h = 1469598103934665603ull);

// Thread-local message returned by sv_last_error().
void set_last_error(const std::string &m);

}  // namespace sv
