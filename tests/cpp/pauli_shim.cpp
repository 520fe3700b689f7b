// Test-only C shim around the Pauli-basis planner (host code of the library): plans an op list
// and replays the passes on a vector of Pauli coefficients the way the kernel walks them (tile by
// tile, group by group through the swizzled chunk positions), in double.
#include <cstring>
#include <vector>

#include "pauli.h"

using namespace qcw;

static void map4(std::vector<double *> &x, int stride, const float *m, bool tp)
{
    for (size_t i = 0; i < x.size(); i++) {
        if ((i / stride) % 4) continue;
        double v[4], y[4];
        for (int k = 0; k < 4; k++) v[k] = *x[i + k * stride];
        for (int r = 0; r < 4; r++) {
            y[r] = 0;
            if (tp && r == 0) y[0] = v[0];
            else
                for (int k = 0; k < 4; k++) y[r] += (double)m[4 * (tp ? r - 1 : r) + k] * v[k];
        }
        for (int k = 0; k < 4; k++) *x[i + k * stride] = y[k];
    }
}

static std::vector<QOp> op_list(int nops, const int *kind, const int *k, const int *qubits, const double *mats,
                                const long long *mat_off)
{
    std::vector<QOp> ops(nops);
    for (int i = 0; i < nops; i++) {
        QOp &o = ops[i];
        o.kind = kind[i];
        o.k = k[i];
        o.ncontrols = 0;
        for (int j = 0; j < o.k; j++) o.qubits[j] = qubits[2 * i + j];
        const int dim = o.kind == 0 ? (1 << o.k) : (1 << (2 * o.k));
        o.m.resize((size_t)dim * dim);
        for (int t = 0; t < dim * dim; t++)
            o.m[t] = c128(mats[2 * (mat_off[i] + t)], mats[2 * (mat_off[i] + t) + 1]);
    }
    return ops;
}

// Returns the number of passes; *bad counts positions a round visits not exactly once.
extern "C" int pauli_replay(int n, int kmax, int beam, int zero, int nops, const int *kind, const int *k, const int *qubits,
                            const double *mats, const long long *mat_off, double *v, int *nrounds, int *bad)
{
    const std::vector<QOp> ops = op_list(nops, kind, k, qubits, mats, mat_off);
    const PauliPlan plan = plan_pauli(ops, 0, ops.size(), n, kmax, beam != 0, zero != 0);
    if (zero)
        for (size_t i = 0; i < (size_t)1 << (2 * plan.nd); i++) {
            v[i] = 1;
            for (int d = 0; d < plan.nd; d++) v[i] *= plan.w[4 * d + ((i >> (2 * d)) & 3)];
        }
    *nrounds = *bad = 0;
    for (const PPass &P : plan.passes) {
        *nrounds += (int)P.rounds.size();
        if ((int)P.coefs.size() > kPMaxCoef || (int)P.rounds.size() > kPMaxRounds || (int)P.ops.size() > kPMaxOps ||
            (int)P.td.size() != P.t || P.td[0] != 0 || P.td[1] != 1)
            return -1;
        const size_t tiles = (size_t)1 << (2 * P.od.size()), nchunk = (size_t)1 << (2 * (P.t - 1));
        for (size_t tile = 0; tile < tiles; tile++) {
            size_t base = 0;
            for (size_t j = 0; j < P.od.size(); j++) base |= ((tile >> (2 * j)) & 3) << (2 * P.od[j]);
            // shared-memory image: position of chunk c holds global elements
            std::vector<size_t> at(4 * nchunk);
            std::vector<int> filled(nchunk, 0);
            for (size_t c = 0; c < nchunk; c++) {
                size_t g = base;
                for (int d = 1; d < P.t; d++) g |= ((c >> (2 * (d - 1))) & 3) << (2 * P.td[d]);
                const unsigned pc = pauli_swz((unsigned)c);
                if (pc >= nchunk) return -2;
                filled[pc]++;
                for (int e = 0; e < 4; e++) at[4 * pc + e] = g + e;
            }
            for (int f : filled) *bad += f != 1;
            for (const PRound &r : P.rounds) {
                std::vector<int> seen(nchunk, 0);
                std::vector<double> in(v, v + ((size_t)1 << (2 * (P.t + P.od.size()))));
                for (unsigned g = 0; g < (1u << r.nob); g++) {
                    const unsigned b = r.lo[g & 15u] ^ r.hi[g >> 4];
                    std::vector<double *> x(64);
                    for (unsigned kk = 0; kk < 4; kk++)
                        for (unsigned jj = 0; jj < 4; jj++) {
                            auto pos = [&](const uint16_t *m) {
                                return (b ^ ((jj & 1) ? m[0] : 0u) ^ ((jj & 2) ? m[1] : 0u) ^ ((kk & 1) ? m[2] : 0u) ^
                                        ((kk & 2) ? m[3] : 0u)) / 16u;
                            };
                            const unsigned pl = pos(r.ld), pc = pos(r.st);
                            if (pc >= nchunk || pl >= nchunk) return -3;
                            seen[pc]++;
                            const int za = jj & 1, xa = jj >> 1, zb = kk & 1, xb = kk >> 1;
                            const bool neg = r.perm == PP_CX_BC ? (xa & zb & (xb ^ za ^ 1)) : r.perm == PP_CX_CB ? (xb & za & (xa ^ zb ^ 1))
                                             : r.perm == PP_CZ ? (xa & xb & (za ^ zb)) : 0;
                            for (int e = 0; e < 4; e++) {
                                x[e + 4 * jj + 16 * kk] = v + at[4 * pc + e];
                                v[at[4 * pc + e]] = neg ? -in[at[4 * pl + e]] : in[at[4 * pl + e]];
                            }
                        }
                    for (int o = r.op0; o < r.op0 + r.nop; o++) {
                        const POp &op = P.ops[o];
                        const float *m = &P.coefs[4 * (size_t)op.coef];
                        const int st[3] = {1, 4, 16};
                        if (op.kind == PO_MM) {
                            map4(x, 4, m, true);
                            map4(x, 16, m + 12, true);
                            continue;
                        }
                        if (op.kind < PO_CX) {
                            map4(x, st[op.kind], m, false);
                            continue;
                        }
                        static const int cx[6][2] = {{0, 1}, {0, 2}, {1, 0}, {1, 2}, {2, 0}, {2, 1}};
                        static const int cz[3][2] = {{0, 1}, {0, 2}, {1, 2}}, tw[3][2] = {{1, 0}, {2, 0}, {2, 1}};
                        const int kd = op.kind < PO_CZ ? 0 : op.kind < PO_TWO ? 1 : 2;
                        const int *pr = kd == 0 ? cx[op.kind - PO_CX] : kd == 1 ? cz[op.kind - PO_CZ] : tw[op.kind - PO_TWO];
                        const int sa = st[pr[0]], sb = st[pr[1]];
                        for (int i = 0; i < 64; i++) {
                            if ((i / sa) % 4 || (i / sb) % 4) continue;
                            double in[16], out[16];
                            for (int e = 0; e < 16; e++) in[e] = *x[i + (e >> 2) * sa + (e & 3) * sb];
                            for (int e = 0; e < 16; e++) {
                                int xa = (e >> 3) & 1, za = (e >> 2) & 1, xb = (e >> 1) & 1, zb = e & 1;
                                if (kd == 0) {
                                    const double s = (xa & zb & (xb ^ za ^ 1)) ? -1 : 1;
                                    out[e] = s * in[8 * xa + 4 * (za ^ zb) + 2 * (xb ^ xa) + zb];
                                } else if (kd == 1) {
                                    const double s = (xa & xb & (za ^ zb)) ? -1 : 1;
                                    out[e] = s * in[8 * xa + 4 * (za ^ xb) + 2 * xb + (zb ^ xa)];
                                } else {
                                    out[e] = 0;
                                    for (int f = 0; f < 16; f++) out[e] += (double)m[16 * e + f] * in[f];
                                }
                            }
                            for (int e = 0; e < 16; e++) *x[i + (e >> 2) * sa + (e & 3) * sb] = out[e];
                        }
                        if (kd < 2) {
                            map4(x, sa, m, true);
                            map4(x, sb, m + 12, true);
                        }
                    }
                }
                for (int s : seen) *bad += s != 1;
                // eight consecutive lanes reach eight different 16-byte bank positions
                if (r.nob >= 3) {
                    unsigned hit = 0;
                    for (unsigned g = 0; g < 8; g++) {
                        hit |= 1u << ((r.lo[g] / 16u) & 7u);
                    }
                    *bad += hit != 255u && P.t == kPTile;
                }
            }
        }
    }
    return (int)plan.passes.size();
}

// The plain path's passes over a list, on the coefficients v; returns their number.
extern "C" int pairs_replay(int n, int nops, const int *kind, const int *k, const int *qubits, const double *mats,
                            const long long *mat_off, double *v)
{
    const std::vector<QOp> ops = op_list(nops, kind, k, qubits, mats, mat_off);
    const std::vector<PairProg> progs = plan_pairs(ops, 0, ops.size(), n);
    const size_t N = (size_t)1 << (2 * n);
    std::vector<double *> x(N);
    for (size_t i = 0; i < N; i++) x[i] = v + i;
    for (const PairProg &p : progs) {
        const int da = n - 1 - p.a, db = n - 1 - p.b;
        if (p.b < 0) {
            float m[16];
            for (int i = 0; i < 16; i++) m[i] = (float)p.one[i];
            map4(x, 1 << (2 * da), m, false);
            continue;
        }
        if (p.kind.size() > (size_t)kPairMaxOps || (p.T.empty() && p.kind.empty())) return -1;
        size_t c = 0;
        for (uint8_t kd : p.kind) {
            if (kd < PK_CX) {
                const bool tp = kd < PK_GEN;
                map4(x, 1 << (2 * ((kd & 1) ? db : da)), &p.coefs[c], tp);
                c += tp ? 12 : 16;
                continue;
            }
            const std::vector<double> in(v, v + N);
            for (size_t i = 0; i < N; i++) {
                const int s = kd == PK_CX + 1 ? db : da, t = kd == PK_CX + 1 ? da : db;  // control, target
                int pc = (i >> (2 * s)) & 3, pt = (i >> (2 * t)) & 3;
                const int xa = pc >> 1, za = pc & 1, xb = pt >> 1, zb = pt & 1;
                const bool cz = kd == PK_CZ;
                const double sg = (cz ? xa & xb & (za ^ zb) : xa & zb & (xb ^ za ^ 1)) ? -1 : 1;
                const int fc = cz ? 2 * xa + (za ^ xb) : 2 * xa + (za ^ zb), ft = cz ? 2 * xb + (zb ^ xa) : 2 * (xb ^ xa) + zb;
                const size_t from = (i & ~(((size_t)3 << (2 * s)) | ((size_t)3 << (2 * t)))) | ((size_t)fc << (2 * s)) | ((size_t)ft << (2 * t));
                v[i] = sg * in[from];
            }
        }
        if (c != p.coefs.size()) return -2;
        if (!p.T.empty()) {
            const std::vector<double> in(v, v + N);
            for (size_t i = 0; i < N; i++) {
                const size_t base = i & ~(((size_t)3 << (2 * da)) | ((size_t)3 << (2 * db)));
                const int e = 4 * ((i >> (2 * da)) & 3) + ((i >> (2 * db)) & 3);
                v[i] = 0;
                for (int f = 0; f < 16; f++) v[i] += p.T[16 * e + f] * in[base | ((size_t)(f >> 2) << (2 * da)) | ((size_t)(f & 3) << (2 * db))];
            }
        }
    }
    return (int)progs.size();
}

// The start factors and passes of plan_pauli_list (a caller's list, from |0..0>) against plan_pauli's on
// the same operations: 0 if alike.
extern "C" int list_plan_differs(int n, int nops, const int *kind, const int *k, const int *qubits, const double *mats,
                                 const long long *mat_off, const double *raw, const int *nkraus, const long long *raw_off)
{
    const std::vector<QOp> ops = op_list(nops, kind, k, qubits, mats, mat_off);
    std::vector<qcw_op> list(nops);
    for (int i = 0; i < nops; i++) {
        list[i].kind = kind[i] == 0 ? QCW_OP_GATE : QCW_OP_KRAUS;
        list[i].k = k[i];
        for (int j = 0; j < k[i]; j++) list[i].qubits[j] = qubits[2 * i + j];
        list[i].nkraus = nkraus[i];
        list[i].offset = 2 * raw_off[i];
    }
    const PauliPlan a = plan_pauli(ops, 0, ops.size(), n, 0, false, true);
    const PauliPlan b = plan_pauli_list(list.data(), nops, raw, n, 0);
    if (a.passes.size() != b.passes.size() || a.w.size() != b.w.size()) return 1;
    auto differ = [](float x, float y) { return !(x - y <= 1e-6f && y - x <= 1e-6f); };
    for (size_t i = 0; i < a.w.size(); i++)
        if (differ(a.w[i], b.w[i])) return 2;
    for (size_t p = 0; p < a.passes.size(); p++) {
        const PPass &x = a.passes[p], &y = b.passes[p];
        if (x.ops.size() != y.ops.size() || x.coefs.size() != y.coefs.size()) return 3;
        for (size_t i = 0; i < x.coefs.size(); i++)
            if (differ(x.coefs[i], y.coefs[i])) return 4;
    }
    return 0;
}

// Passes of a plan that have no operation; *npass: all of them.
extern "C" int pauli_empty_passes(int n, int kmax, int beam, int nops, const int *kind, const int *k, const int *qubits,
                                  const double *mats, const long long *mat_off, int *npass)
{
    const std::vector<QOp> ops = op_list(nops, kind, k, qubits, mats, mat_off);
    const PauliPlan plan = plan_pauli(ops, 0, ops.size(), n, kmax, beam != 0, false);
    int empty = 0;
    for (const PPass &p : plan.passes) empty += p.ops.empty() ? 1 : 0;
    *npass = (int)plan.passes.size();
    return empty;
}
