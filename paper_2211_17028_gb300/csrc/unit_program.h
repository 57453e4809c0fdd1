// Programs of the unit sweep kernel (kernels_units.cu): the operations of one
// pass, assembled on the host for one 12-qubit tile of one state.
//
// A program is an array of 16-byte words: a header, the phases, one record
// per operation, then the matrices.  The assembler (unit_program.cpp) decides
// everything that does not depend on the tile: which diagonal factors are
// pending at each operation, where they have to be multiplied into the
// amplitudes, and which constants fold into a matrix.  The kernel keeps no
// flags of its own.
#pragma once

#include <cstdint>
#include <vector>

#include "sweep_types.h"

namespace nqs {

constexpr int kUnitRB = 4;                      // register qubits: 16 amplitudes per thread
constexpr int kUnitThreads = 1 << (kMaxTileQ - kUnitRB);
constexpr int kUnitSlots = 8;                   // checkpoint pointers of a pass (reductions, saves)
constexpr int kNoLoc = 31;                      // location of an absent bit (always 0)

// How a program keeps pending diagonals:
//   UM_PAIRS   a scalar and a pair of factors per register bit, taken by gates
//              and multiplied into the amplitudes in a fixed order.  States
//              swept alone (backward and main sweeps, from which levels 0 and 1
//              come) through circuits with phases use it: the order of an
//              amplitude's products, and so its rounding, is fixed by the order
//              of the operations, whichever kernel sweeps it.  (Reductions add
//              the amplitudes up in an order of their own.)
//   UM_RATIOS  a scalar and one ratio per register bit: half the products.
//              Branch groups use it, and every program whose diagonals are
//              signs, which are exact either way.
enum UnitMode : int { UM_RATIOS = 0, UM_PAIRS = 1 };

// Operation codes; a code in a family of four is FAMILY + register bit, in a
// family of six FAMILY + pair of register bits.
enum UnitOp : int {
    UO_G1 = 0,      // dense one-qubit matrices of register bits, ascending, after UO_DN of the pairs in a:
                    // mask = their flags (8 bits each), off[i] = {sign mask}, 0, matrix of bit i
    UO_GK = 4,      // dense factor K_0 of a site
    UO_KD = 8,      // diagonal factor K_0 of a site; UF_REAL: real entries
    UO_FLB = 12,    // pairs: the scalar and the pair of one register bit into the amplitudes; ratios: the ratio
    UO_FLR = 16,    // multiply the sign of one register bit into the amplitudes
    UO_HP = 20,     // c = the bit at location a; pairs: pair of the bit *= m[2c], m[2c + 1]; ratios: ratio *= m[c]
    UO_SITE = 24,   // noise site
    UO_DN = 28,     // negate the amplitudes with both register bits, for every pair in a
    UO_DG = 34,     // pairs: amplitudes *= m[2 * (low bit) + (high bit)]; ratios: those with both bits *= m[0]
    UO_G2 = 40,     // dense two-qubit matrix, its first qubit on the low bit (+ 6: on the high bit)
    UO_SC = 52,     // scalar *= m[c], c = the bits at locations a, b
    UO_FLS = 53,    // multiply the scalar into the amplitudes; UF_REAL: a real one
    UO_FLA = 54     // multiply the scalar and all four pairs or ratios into the amplitudes
};
// A gate takes the pending pair or ratio of its bit, its pending sign (parity
// of the bits `mask`), the pending scalar; the scalar is real.
enum : int { UF_DIAG = 1, UF_SIGN = 2, UF_SCALAR = 4, UF_REAL = 8, UF_HERE = 64 };

// pairs of register bits (i < j) in the order 01 02 03 12 13 23
inline int unit_pair(int i, int j) { return i == 0 ? j - 1 : i == 1 ? j + 1 : 5; }

struct UnitRec {               // 16 bytes
    unsigned char code, a, b, flags;
    union {
        struct {
            unsigned char ev, nspawn, sp, pad0;   // reduction / checkpoint slot, spawned factors, spawn slot
            unsigned short mat, pad1;
        };
        unsigned short off[4];                    // UO_G1: matrices of the register bits
    };
    unsigned int mask;
};

struct UnitPhase {             // 96 bytes
    unsigned short lane_j[32]; // tile index bits of a lane
    unsigned short warp_j[8];  // tile index bits of a warp
    unsigned short reg_j[4];   // tile index bit of each register bit
    unsigned short op_begin, op_end;
    unsigned short pad[2];
};

struct UnitHeader {            // 64 bytes
    unsigned int n_phases, n_ops, ops_word, mats_word;
    unsigned long long nl_mask;             // qubits outside the tile
    unsigned int n_events, words;
    unsigned char local[12];                // tile qubits, ascending
    unsigned char n_slots, pad[3];
    unsigned short slot_site[kUnitSlots];   // site of each checkpoint slot from site_base on (bit 15: forward table)
};

struct UnitProgram {
    UnitMode mode = UM_RATIOS;
    int word = 0, words = 0, n_phases = 0, n_events = 0;
    int site_base = 0;           // the units' checkpoint tables start at this site
};

// Assemble dops[off .. off + n) (execution order) on the tile qubits `local`
// of an n_qubits-wide state, appending to `out`; mats is the float2 table the
// operations index; single: for a state swept alone.
UnitProgram assemble_unit(bool single, const std::vector<DevOp>& dops, int off, int n, const int* local, int n_qubits,
                          const std::vector<float2>& mats, std::vector<uint4>& out);

// One state swept through one pass: `ctas` consecutive blocks share its tiles.
struct SweepUnit {
    const float2* in;
    float2* out;               // null: the swept state is not kept
    float2* spawn;             // spawned state (slot k, factor i) at spawn + ((3 k + i) << n)
    const uint4* prog;
    float2* const* ckpt;       // phi_s, s from the program's site_base on
    float2* const* ckpt_fwd;   // chi_s
    double* partials;          // [event][cta][8]
    int* err;
    int n_tiles, n, cta_begin, ctas;
};

// kernel of a launch: states swept alone or of branch groups, and the mode
inline int unit_kind(bool single, UnitMode mode) { return 2 * (int)single + (int)mode; }
constexpr int kUnitKinds = 4;
size_t unit_smem_bytes(int max_words, int max_events);
int unit_blocks_per_sm(int kind, size_t smem);
// whether a launch of such programs can use the form with three blocks per SM
bool unit_three_blocks(int kind, size_t smem);
// blk: unit of every block, or null when every unit has `ctas` blocks
// kind: unit_kind of the units' programs
cudaError_t launch_units(int kind, const SweepUnit* units, const int* blk, int ctas, int total_ctas, size_t smem,
                         cudaStream_t st);
// Blocks per unit of a launch of n_units units of n_tiles tiles each.
int unit_ctas(int n_units, long long n_tiles, int slots);

}  // namespace nqs
