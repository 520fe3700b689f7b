// Evolution in the Pauli basis: the state as the real vector v_P = Tr[P rho], one FP32 number per
// Pauli string P on the register (4^n of them, rho = 2^-n sum_P v_P P; Sec. 5.2's form
// rho = (1 + P . sigma) / 2 for every qubit at once).
//
// rho is Hermitian (Sec. 5.2), so the 2^n x 2^n complex matrix has 4^n real degrees of freedom
// and v holds exactly those: half the bytes of complex64 rho with no mirrored half to skip or
// complete, every operation a real matrix on the labels of its qubits.  A one-qubit operation is
// a real 4 x 4 map (its first row is (1, 0, 0, 0) when it keeps the trace: 12 multiply-adds per
// four elements), CNOT and CZ are signed permutations of the labels (no arithmetic), any other
// two-qubit operation is a real 16 x 16 map.
//
// Label of one qubit: p = 2 x + z, i.e. I = 0, Z = 1, X = 2, Y = 3 (P = i^{xz} X^x Z^z).  Index
// of a string: qubit q's label is base-4 digit n - 1 - q, so qubit n - 1 is the lowest digit.
#pragma once
#include <stdint.h>

#include <vector>

#include "planner.h"

namespace qcw {

// A pass brings tiles of kPTile digits (4^7 floats = 64 KiB) into shared memory: the qubits it
// works on, always with the two lowest digits so that a tile's contiguous runs are 64 bytes.
constexpr int kPTile = 7;
constexpr int kPMinDigits = 3;  // a round holds three digits in registers: smaller registers are padded

// One round of a pass: each thread holds the 64 elements of three digits (tile digit 0, db and
// dc) in registers and applies the round's operations to them.  Positions are byte offsets of
// 16-byte chunks (the four labels of digit 0) in the swizzled tile, and combine by XOR.  A CNOT or
// CZ between db and dc is linear on the label bits, so the round that starts with one just reads its
// chunks in the permuted order (ld != st) and flips the signs it brings.
struct PRound {
    uint8_t db, dc;    // tile digits beside digit 0, 1 <= db < dc < t
    uint8_t nob;       // bits of the group index: 2 (t - 3)
    uint8_t nop;
    uint16_t op0;      // first operation in the pass's list
    uint8_t perm;      // PP_*
    uint8_t direct;    // last round of a pass on full tiles, leaving tile digit 1 alone: results go straight to v
    uint16_t ld[4];    // contribution of the label bits z, x of db and z, x of dc when reading
    uint16_t st[4];    // and when writing
    uint16_t pad2[4];
    uint16_t lo[16], hi[16];  // position of group g: lo[g & 15] ^ hi[g >> 4]
};
enum : int { PP_NONE = 0, PP_CX_BC = 1, PP_CX_CB = 2, PP_CZ = 3 };  // CX_BC: db controls dc

// Operation kinds; register digits 0, 1, 2 are tile digits 0, db, dc.
enum : int {
    PO_ONE = 0,   // + d: general 4 x 4 map of digit d, 16 coefficients
    PO_CX = 3,    // + pair (control, target) of (0,1) (0,2) (1,0) (1,2) (2,0) (2,1), then a trace-
                  // preserving map of the control and one of the target: 12 + 12 coefficients
    PO_CZ = 9,    // + pair (0,1) (0,2) (1,2), then a trace-preserving map of each: 12 + 12
    PO_TWO = 12,  // + pair (high, low) of (1,0) (2,0) (2,1): general 16 x 16 map, 256 coefficients
    PO_MM = 15,   // trace-preserving maps of digits 1 and 2 (after the round's own permutation): 12 + 12
    PO_KINDS = 16
};
struct POp {
    uint16_t kind;
    uint16_t coef;  // first coefficient, in units of 4
};

// Limits of one pass (it is cut before it exceeds any): its program travels as a kernel parameter
// (below 32 KiB), each coefficient twice.
constexpr int kPMaxCoef = 3072;
constexpr int kPMaxRounds = 60;
constexpr int kPMaxOps = 60;

struct PPass {
    int t = 0;
    std::vector<int> td, od;  // register digits inside the tile and outside it, ascending
    std::vector<PRound> rounds;
    std::vector<POp> ops;
    std::vector<float> coefs;
};

struct PauliPlan {
    int n = 0, nd = 0;  // qubits; digits (n, at least kPMinDigits)
    std::vector<PPass> passes;
    // zero start: what the one-qubit operations before any two-qubit operation make of |0..0>, a product
    // state, v_P = prod_d w[d][label of digit d]; the first pass starts from it.  (1, 1, 0, 0) else.
    std::vector<float> w;
};

// Plan ops[begin, end) (k <= 2, no controls) for an n-qubit register.  kmax = 0: a pass works on
// every qubit of its tile; else on at most kmax qubits.  beam: pass sets by the beam search.  zero:
// the state before is |0..0><0..0| (there is then at least one pass).
PauliPlan plan_pauli(const std::vector<QOp> &ops, size_t begin, size_t end, int n, int kmax, bool beam,
                     bool zero = false);

// The same for a caller's checked operation list (gates and channels on one and two qubits), from
// |0..0>.
PauliPlan plan_pauli_list(const qcw_op *ops, int nops, const double *matrices, int n, int kmax);

// One pass of the plain path over rho (plain_list.cu): a run of a list's operations that stays on two
// qubits, as maps of either and permutations; or one dense two-qubit map (T); or a map left over on
// one qubit (b = -1).
enum : int {
    PK_MAP = 0,   // + 0, 1: trace-preserving map of a, of b; 12 coefficients (rows 1..3)
    PK_GEN = 2,   // + 0, 1: general map, 16
    PK_CX = 4,    // + 0: a controls; + 1: b controls
    PK_CZ = 6
};
constexpr int kPairMaxOps = 16;  // a longer run is cut: the program travels as a kernel parameter
struct PairProg {
    int a = 0, b = -1;
    std::vector<uint8_t> kind;
    std::vector<float> coefs;
    std::vector<double> T;  // index 4 p_a + p_b, labels as everywhere here
    double one[16];         // b = -1
};

// Plan ops[begin, end) (k <= 2, no controls) as passes over rho, to be run in order.
std::vector<PairProg> plan_pairs(const std::vector<QOp> &ops, size_t begin, size_t end, int n);

// Position of 16-byte chunk c of a tile in shared memory: bits 0..2 (which 16 of 128 bytes) are
// mixed with the bits above so that digits 1..6 of the tile each contribute a different plane of
// GF(2)^3 there; any two digits then reach all eight positions, and a quarter-warp whose lanes
// enumerate two digits outside the round reads without bank conflicts.  Linear in the bits of c.
#ifdef __CUDACC__
__host__ __device__
#endif
inline unsigned pauli_swz(unsigned c)
{
    const unsigned t = c >> 3;
    const unsigned s0 = t ^ (t >> 3) ^ (t >> 6) ^ (t >> 8);
    const unsigned s1 = (t >> 1) ^ (t >> 4) ^ (t >> 5) ^ (t >> 8);
    const unsigned s2 = (t >> 2) ^ (t >> 4) ^ (t >> 6) ^ (t >> 7);
    return c ^ ((s0 & 1u) | ((s1 & 1u) << 1) | ((s2 & 1u) << 2));
}

}  // namespace qcw
