// Work-item engine shared by the batched runner (qcw_batch_*) and the serving loop
// (qcw_server_*): circuits are planned into tile programs, programs into work items, and one
// persistent kernel drains the item list.
#pragma once
#include <stdint.h>

#include <vector>

#include "pauli_run.h"

namespace qcw {

// Kinds of work item.
enum : int {
    WI_TILES = 0,   // one tile of one pass of a multi-tile program
    WI_REDUCE = 1,  // FP64 readouts over a run of elements (trace and P(q = 1) with the first)
    WI_WHOLE = 2,   // a whole program whose state fits one tile: all passes, readouts, store
};
enum : int { WF_INIT = 1 };  // the item's tiles start as |0..0><0..0| instead of being loaded

struct WItem {
    float *v;                // the state's Pauli coefficients
    const char *pass;        // description of the (first) pass
    unsigned *dep;           // wait until *dep >= dep_target (nullptr: no dependency)
    unsigned *done;          // incremented once the item's stores are complete (nullptr: none)
    double *red;             // readout output (kinds 1, 2): trace re, trace im, purity, p1[n]
    unsigned long long e0, ecount;  // kind 1: elements [e0, e0 + ecount)
    unsigned dep_target;
    unsigned tile;
    int npass;
    int kind;
    int flags;
    int n;
};

// A pass in a descriptor buffer: this header, then PRound[nround], POp[nop] (padded to 16 bytes) and
// float[ncoef] (padded); `bytes` from one pass to the next.
struct PassDesc {
    PauliHdr h;
    int bytes;
};
static_assert(sizeof(PassDesc) % 16 == 0, "16-byte sections");

constexpr int kRedVals = 3 + QCW_MAX_QUBITS;  // values per readout block

// Launch state of the persistent kernel.
struct EngineLaunch {
    const WItem *items;
    const int *nitems;
    int *next;
    int *err;
    long long spin_limit;
};

// dense: some pass has dense two-qubit maps.
void engine_launch(const EngineLaunch &L, bool dense, int grid, size_t smem, cudaStream_t s);
qcw_status engine_prepare(int dev, bool dense, size_t smem, int *grid);

// A circuit turned into device-ready descriptors.  Registers below kPMinDigits qubits are padded with
// qubits in |0> above them.
struct Program {
    int n = 0;
    bool whole = false;      // the state fits one tile: one WI_WHOLE item
    bool dense = false;
    std::vector<char> desc;  // the passes, PassDesc after PassDesc
    std::vector<size_t> pass_off;
    std::vector<unsigned> tiles;  // per pass
    size_t smem = 0;         // largest need of a pass
    long long rounds = 0;
    double cost = 0;         // modeled SM-seconds
    size_t off = 0;          // offset inside a descriptor buffer
};

// Plan a checked op list for an n-qubit register; fuse_k (0: no bound) bounds the qubits of a pass.
Program make_program(const qcw_op *ops, int nops, const double *matrices, int n, int fuse_k);

// Elements of an n-qubit program's state.
inline size_t program_elems(int n) { return (size_t)1 << (2 * (n < kPMinDigits ? kPMinDigits : n)); }
// Bytes of a program's descriptors in a descriptor buffer.
inline size_t program_desc_bytes(const Program &p) { return (p.desc.size() + 255) & ~(size_t)255; }

// Readout chunks of a multi-tile program: 2^17 elements each.
constexpr unsigned long long kReduceElems = 1ull << 17;
inline int program_chunks(const Program &p)
{
    return p.whole ? 1 : (int)((program_elems(p.n) + kReduceElems - 1) / kReduceElems);
}

// Shared memory of the engine kernel for any pass a planner can produce.
size_t engine_max_smem();

// Items of passes [pass_begin, pass_end) of one program.  Appends to `levels[l]` (level = pass
// index - pass_begin; readouts on the level after the last pass).  desc: device base of the
// descriptor buffer holding the program; counters: (pass_end - pass_begin) zeroed device
// counters, one per pass of the range; red: its readout blocks (chunk count in *nchunks).
void program_items(const Program &p, float *v, const char *desc, unsigned *counters, double *red, int pass_begin,
                   int pass_end, bool init, bool readout, std::vector<std::vector<WItem>> &levels, int *nchunks);

// rho of a program's state on the host (2^n x 2^n, complex128); v is left as it is.  copy: program_elems(n)
// floats of device scratch (if program_copies(n)); rho goes in pieces of whole rows through stage
// (program_stage(n) elements on the device) and from there through host (program_pinned(n), pinned).
size_t program_stage(int n);
size_t program_pinned(int n);
bool program_copies(int n);
cudaError_t program_rho(const float *v, int n, float *copy, float2 *stage, float2 *host, double *out, cudaStream_t s);

}  // namespace qcw
