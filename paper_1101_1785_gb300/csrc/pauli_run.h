// Launchers of the Pauli-basis path (pauli.cu), for the context layer and the work-item engine.
#pragma once
#include <vector>

#include "pauli.h"
#include "qcw_internal.h"

namespace qcw {

struct PauliHdr {
    int t, nod, nround, nop, ncoef;
    int8_t td[8], od[16];
    float w[4 * QCW_MAX_QUBITS];  // PauliPlan::w, for the pass that starts from it
};

// A pass in the form the kernels take: header, then rounds | operations | coefficients.
struct PauliBlob {
    PauliHdr h;
    bool dense = false;  // has dense two-qubit maps
    std::vector<unsigned> words;
};
PauliBlob pauli_blob(const PPass &p, const std::vector<float> &w);
PauliHdr pauli_header(const PPass &p, const std::vector<float> &w);
bool pass_dense(const PPass &p);  // has dense two-qubit maps
unsigned pauli_grid(const PauliHdr &h, int nsm);

// One pass over v (nd digits).  init: v is the header's product state and not read.  ppart (2 pauli_grid values):
// also leave per-team partial sums of the purity.
cudaError_t launch_pauli_pass(const PauliBlob &B, float *v, int nd, int nsm, bool init, unsigned long long *err,
                              unsigned wait_limit, int stall_tile, double *ppart, cudaStream_t s);
cudaError_t launch_pauli_to_rho(float *v, float2 *rho, int n, cudaStream_t s);
cudaError_t launch_rho_to_pauli(const float2 *rho, float *v, int n, cudaStream_t s);
int pauli_convert_launches(int n);
// The same in pieces: launch_pauli_unfold once (v is used up; up to seven qubits it is left alone), then
// rows [row, row + count) of rho, both multiples of pauli_row_block(n).
cudaError_t launch_pauli_unfold(float *v, int n, cudaStream_t s);
int pauli_row_block(int n);
cudaError_t launch_pauli_rows(const float *v, float2 *rows, int n, int row, int count, cudaStream_t s);
cudaError_t launch_pauli_zero(float *v, int n, int nsm, cudaStream_t s);
void launch_pauli_diag(const float *v, int n, double *out, cudaStream_t s);
void launch_pauli_terms(const float *v, const PauliTerms &T, double *out, cudaStream_t s);
void launch_pauli_project(float *v, int n, int qubit, int m, double scale, int nsm, cudaStream_t s);
int launch_pauli_purity(const float *v, int n, double *partials, double *out, int nblocks, cudaStream_t s);
constexpr int kPauliPtMax = 6;  // most kept qubits of launch_pauli_ptrace
void launch_pauli_ptrace(const float *v, const PTParams &p, double2 *out, cudaStream_t s);

}  // namespace qcw
