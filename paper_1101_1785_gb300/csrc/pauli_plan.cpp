// Planner of the Pauli-basis path: operations -> merged nodes -> passes -> rounds.
//
// Nodes.  Every one-qubit operation is multiplied into the map that follows the last two-qubit
// operation on its qubit (they commute past everything else), so between two two-qubit operations
// a qubit has exactly one real 4 x 4 map.  CNOT and CZ nodes carry the maps of their two qubits
// that follow; any other two-qubit operation is a dense 16 x 16 node into which such maps, and a
// directly following two-qubit operation on the same pair, are multiplied.
#include "pauli.h"

#include <algorithm>
#include <cmath>
#include <cstring>

#include "tile.h"

namespace qcw {

namespace {

// label of member index 2 r + c of pauli_transfer's basis (I, X, Y, Z)
const int kLab[4] = {0, 2, 3, 1};

struct M4 {
    double m[16];
    bool id;
};

M4 m4_identity()
{
    M4 r{};
    for (int i = 0; i < 4; i++) r.m[5 * i] = 1.0;
    r.id = true;
    return r;
}

// a <- b a
void m4_lmul(M4 &a, const M4 &b)
{
    if (b.id) return;
    if (a.id) {
        a = b;
        return;
    }
    M4 r;
    for (int i = 0; i < 4; i++)
        for (int j = 0; j < 4; j++) {
            double s = 0;
            for (int k = 0; k < 4; k++) s += b.m[4 * i + k] * a.m[4 * k + j];
            r.m[4 * i + j] = s;
        }
    r.id = false;
    a = r;
}

bool m4_tp(const M4 &a)  // first row (1, 0, 0, 0): keeps the trace
{
    return std::fabs(a.m[0] - 1.0) < 1e-12 && std::fabs(a.m[1]) < 1e-13 && std::fabs(a.m[2]) < 1e-13 &&
           std::fabs(a.m[3]) < 1e-13;
}

// Real map of a one-qubit superoperator S (S[2 r' + c'][2 r + c]) on the labels:
// T_ij = Tr[P_i S(P_j)] / 2, with P = I, Z, X, Y read off rows and columns of S directly.
// Entries below 1e-14 of the largest are rounding residue of exact zeros; the largest is T_00, half the
// trace of what S makes of the identity (|Tr[P S(P')]| <= Tr[S(1)] for S = sum_j K_j . K_j^dagger).
M4 super_map(const c128 *S)
{
    double cr[4][4], ci[4][4];  // S applied to P_j, element e (for Y: to Y / -i)
    for (int e = 0; e < 4; e++) {
        const c128 *r = S + 4 * e;
        cr[e][0] = r[0].real() + r[3].real(), ci[e][0] = r[0].imag() + r[3].imag();
        cr[e][1] = r[0].real() - r[3].real(), ci[e][1] = r[0].imag() - r[3].imag();
        cr[e][2] = r[1].real() + r[2].real(), ci[e][2] = r[1].imag() + r[2].imag();
        // Y = -i (b01 - b10): real part of -i z is Im z, imaginary part -Re z
        cr[e][3] = r[1].imag() - r[2].imag(), ci[e][3] = r[2].real() - r[1].real();
    }
    M4 t;
    t.id = false;
    for (int j = 0; j < 4; j++) {
        t.m[j] = 0.5 * (cr[0][j] + cr[3][j]);
        t.m[4 + j] = 0.5 * (cr[0][j] - cr[3][j]);
        t.m[8 + j] = 0.5 * (cr[1][j] + cr[2][j]);
        t.m[12 + j] = 0.5 * (ci[2][j] - ci[1][j]);  // Re of i (s01 - s10)
    }
    const double tiny = 1e-14 * t.m[0];
    for (double &x : t.m)
        if (std::fabs(x) < tiny) x = 0.0;
    return t;
}

// A queued operation or one of a caller's list: kind 0 with U, 1 with its superoperator.
struct OpView {
    int kind, k;
    const int *qubits;
    const c128 *m;
};

M4 one_map(const OpView &op)
{
    if (op.kind != 0) return super_map(op.m);
    c128 S[16];
    const c128 *u = op.m;
    for (int r2 = 0; r2 < 2; r2++)
        for (int c2 = 0; c2 < 2; c2++)
            for (int r = 0; r < 2; r++)
                for (int c = 0; c < 2; c++) S[(2 * r2 + c2) * 4 + 2 * r + c] = u[2 * r2 + r] * std::conj(u[2 * c2 + c]);
    return super_map(S);
}

// Real 16 x 16 map of a two-qubit operation, index 4 p_first + p_second.
void two_map(const OpView &op, double *T)
{
    std::vector<c128> S(256);
    if (op.kind != 0) {
        for (int i = 0; i < 256; i++) S[i] = op.m[i];
    } else {
        const c128 *u = op.m;
        for (int r2 = 0; r2 < 4; r2++)
            for (int c2 = 0; c2 < 4; c2++)
                for (int r = 0; r < 4; r++)
                    for (int c = 0; c < 4; c++)
                        S[(size_t)(r2 * 4 + c2) * 16 + r * 4 + c] = u[r2 * 4 + r] * std::conj(u[c2 * 4 + c]);
    }
    double R[16][16];
    pauli_transfer(S, R);
    auto lab = [](int e) {  // member 8 r_a + 4 r_b + 2 c_a + c_b
        const int a = 2 * ((e >> 3) & 1) + ((e >> 1) & 1), b = 2 * ((e >> 2) & 1) + (e & 1);
        return 4 * kLab[a] + kLab[b];
    };
    // pauli_transfer's basis has D = -i Y per qubit with i where their number is odd, so its
    // member with two D is -(Y Y)
    auto sg = [](int e) { return (e & 12) == 12 && (e & 3) == 0 ? -1.0 : 1.0; };
    for (int i = 0; i < 16; i++)
        for (int j = 0; j < 16; j++) T[16 * lab(i) + lab(j)] = 4.0 * R[i][j] * sg(i) * sg(j);
}

struct Node {
    int kind;   // PO_ONE, PO_CX, PO_CZ, PO_TWO
    int a, b;   // qubits (b = -1 for PO_ONE); PO_CX: a controls
    M4 A, B;    // maps that follow on a and b (PO_ONE: A is the map)
    std::vector<double> T;  // PO_TWO
};

// Image of label pair (pa, pb) under the conjugation by CNOT (a controls) or CZ, and its sign.
int conj_label(bool cz, int e, double *sgn)
{
    int xa = (e >> 3) & 1, za = (e >> 2) & 1, xb = (e >> 1) & 1, zb = e & 1;
    if (!cz) {
        *sgn = (xa & zb & (xb ^ za ^ 1)) ? -1.0 : 1.0;
        xb ^= xa;
        za ^= zb;
    } else {
        *sgn = (xa & xb & (za ^ zb)) ? -1.0 : 1.0;
        za ^= xb;
        zb ^= xa;
    }
    return 8 * xa + 4 * za + 2 * xb + zb;
}

// T <- (A (x) B) T
void kron_lmul(std::vector<double> &T, const M4 &A, const M4 &B)
{
    if (A.id && B.id) return;
    std::vector<double> R(256, 0.0);
    for (int ia = 0; ia < 4; ia++)
        for (int ib = 0; ib < 4; ib++)
            for (int ka = 0; ka < 4; ka++)
                for (int kb = 0; kb < 4; kb++) {
                    const double w = A.m[4 * ia + ka] * B.m[4 * ib + kb];
                    if (w == 0) continue;
                    for (int j = 0; j < 16; j++) R[16 * (4 * ia + ib) + j] += w * T[16 * (4 * ka + kb) + j];
                }
    T.swap(R);
}

std::vector<double> node_matrix(const Node &nd)  // its two-qubit operation and following maps
{
    std::vector<double> T(256, 0.0);
    if (nd.kind == PO_TWO) T = nd.T;
    else
        for (int e = 0; e < 16; e++) {
            double s;
            const int f = conj_label(nd.kind == PO_CZ, e, &s);
            T[16 * e + f] = s;
        }
    kron_lmul(T, nd.A, nd.B);
    return T;
}

// The same map with the two qubits exchanged.
std::vector<double> exchanged(const std::vector<double> &T)
{
    std::vector<double> R(256);
    auto x = [](int e) { return 4 * (e & 3) + (e >> 2); };
    for (int i = 0; i < 16; i++)
        for (int j = 0; j < 16; j++) R[16 * x(i) + x(j)] = T[16 * i + j];
    return R;
}

std::vector<double> matmul16(const std::vector<double> &A, const std::vector<double> &B)
{
    std::vector<double> R(256, 0.0);
    for (int i = 0; i < 16; i++)
        for (int k = 0; k < 16; k++) {
            const double w = A[16 * i + k];
            if (w == 0) continue;
            for (int j = 0; j < 16; j++) R[16 * i + j] += w * B[16 * k + j];
        }
    return R;
}

// Exactly CNOT (*a, *b in order control, target) or CZ.
int classify(const OpView &op, int *a, int *b)
{
    *a = op.qubits[0];
    *b = op.qubits[1];
    if (op.kind != 0) return PO_TWO;
    const c128 *u = op.m;
    auto is = [&](const int *col, const double *val) {
        for (int i = 0; i < 4; i++)
            for (int j = 0; j < 4; j++)
                if (u[4 * i + j] != (j == col[i] ? c128(val[i], 0) : c128(0, 0))) return false;
        return true;
    };
    const double one[4] = {1, 1, 1, 1}, cz[4] = {1, 1, 1, -1};
    const int id[4] = {0, 1, 2, 3}, cx[4] = {0, 1, 3, 2}, xc[4] = {0, 3, 2, 1};
    if (is(cx, one)) return PO_CX;
    if (is(xc, one)) {
        std::swap(*a, *b);
        return PO_CX;
    }
    return is(id, cz) ? PO_CZ : PO_TWO;
}

// FP32 rounding of a map's coefficients with feedback.  A channel repeated after every gate (a
// depolarising factor 1 - 4 p / 3, say) rounds the same way each time, so the coefficients it
// shrinks would drift by up to 3e-8 per application, all in one direction.  c: the scale error the
// qubit's maps have collected so far; the next map's linear part is scaled by 1 - c before it is
// rounded, and c becomes what its own rounding adds, so the sum stays within one rounding.  Only where
// the map's largest entry is well inside FP32's normal range: below it the relative rounding is as
// large as 1 (a run of channels that takes a qubit's polarisation to nothing, say), above it infinite,
// and neither says anything about the scale of the maps that follow.
void round_map(M4 &a, double &c)
{
    if (a.id) return;
    double f[9], num = 0, den = 0;
    for (int i = 0; i < 9; i++) {
        const double x = a.m[4 * (i / 3 + 1) + i % 3 + 1];
        f[i] = (double)(float)(x * (1.0 - c));
        num += f[i] * x;
        den += x * x;
    }
    if (!(den >= 1e-60 && den <= 1e60)) return;
    for (int i = 0; i < 9; i++) a.m[4 * (i / 3 + 1) + i % 3 + 1] = f[i];
    c += num / den - 1.0;
}

class NodeBuilder {
  public:
    // zero: one-qubit operations before any two-qubit one on their qubit act on (1, 1, 0, 0) of the
    // product state |0..0>, not as maps of their own
    NodeBuilder(int n, bool zero) : n(n), zero(zero), last(n, -1), pre(n, m4_identity()), start(n, m4_identity()) {}
    void add(const OpView &op);
    std::vector<float> product(int nd) const;
    std::vector<Node> finish();

  private:
    int n;
    bool zero;
    std::vector<Node> out;
    std::vector<int> last;
    std::vector<M4> pre, start;
};

std::vector<float> NodeBuilder::product(int nd) const
{
    std::vector<float> w(4 * (size_t)nd, 0.f);
    for (int d = 0; d < nd; d++)
        for (int p = 0; p < 4; p++) {
            const double *m = d < n ? start[n - 1 - d].m : nullptr;
            w[4 * d + p] = m ? (float)(m[4 * p] + m[4 * p + 1]) : p < 2 ? 1.f : 0.f;
        }
    return w;
}

void NodeBuilder::add(const OpView &op)
{
    {
        if (op.k == 1) {
            const int q = op.qubits[0];
            const M4 m = one_map(op);
            if (last[q] < 0) m4_lmul(zero ? start[q] : pre[q], m);
            else m4_lmul(out[last[q]].a == q ? out[last[q]].A : out[last[q]].B, m);
            return;
        }
        int a, b;
        const int kind = classify(op, &a, &b);
        const bool same = last[a] >= 0 && last[a] == last[b];
        if (same && (kind == PO_TWO || out[last[a]].kind == PO_TWO)) {  // one dense map for both
            Node &nd = out[last[a]];
            Node nw{kind, a, b, m4_identity(), m4_identity(), {}};
            if (kind == PO_TWO) {
                nw.T.resize(256);
                two_map(op, nw.T.data());
            }
            std::vector<double> T2 = node_matrix(nw);
            if (nd.a != a) T2 = exchanged(T2);
            nd.T = matmul16(T2, node_matrix(nd));
            nd.kind = PO_TWO;
            nd.A = nd.B = m4_identity();
            return;
        }
        Node nd{kind, a, b, m4_identity(), m4_identity(), {}};
        if (kind == PO_TWO) {
            nd.T.resize(256);
            two_map(op, nd.T.data());
            if (!pre[a].id || !pre[b].id) {
                std::vector<double> P(256, 0.0);
                for (int e = 0; e < 16; e++) P[17 * e] = 1.0;
                kron_lmul(P, pre[a], pre[b]);
                nd.T = matmul16(nd.T, P);
            }
        } else {
            for (int q : {a, b})
                if (!pre[q].id) out.push_back(Node{PO_ONE, q, -1, pre[q], m4_identity(), {}});
        }
        pre[a] = pre[b] = m4_identity();
        last[a] = last[b] = (int)out.size();
        out.push_back(std::move(nd));
    }
}

std::vector<Node> NodeBuilder::finish()
{
    std::vector<Node> fin;
    for (int q = 0; q < n; q++)
        if (!pre[q].id) fin.push_back(Node{PO_ONE, q, -1, pre[q], m4_identity(), {}});
    for (Node &nd : out) {
        if (nd.kind == PO_TWO) {
            nd.T = node_matrix(nd);
            nd.A = nd.B = m4_identity();
            fin.push_back(std::move(nd));
        } else if (nd.kind == PO_ONE) {
            fin.push_back(std::move(nd));
        } else {
            // maps that do not keep the trace follow as general one-qubit maps
            const Node g = nd;
            if (!m4_tp(nd.A)) nd.A = m4_identity();
            if (!m4_tp(nd.B)) nd.B = m4_identity();
            fin.push_back(std::move(nd));
            if (!m4_tp(g.A)) fin.push_back(Node{PO_ONE, g.a, -1, g.A, m4_identity(), {}});
            if (!m4_tp(g.B)) fin.push_back(Node{PO_ONE, g.b, -1, g.B, m4_identity(), {}});
        }
    }
    std::vector<double> err(n, 0.0);
    for (Node &nd : fin) {
        if (nd.kind == PO_TWO) continue;
        round_map(nd.A, err[nd.a]);
        if (nd.b >= 0) round_map(nd.B, err[nd.b]);
    }
    return fin;
}

std::vector<unsigned> pass_candidates(int nd, int t, int kmax)
{
    std::vector<unsigned> out;
    const unsigned all = (1u << nd) - 1u;
    const int k = kmax ? std::min(kmax, t) : t;
    const unsigned low = 3u;  // the two lowest digits are in every tile
    for (unsigned s = 0; s <= all; s++) {
        if (__builtin_popcount(s) != k) continue;
        if (!kmax && (s & low) != low) continue;
        if (kmax && __builtin_popcount(s | low) > t) continue;
        out.push_back(s);
    }
    return out;
}

// Positions of the round: the group-index bits go to the chunk-index bits outside digits db and dc,
// the first three to bits with independent contributions to the bank position (see pauli_swz).
void round_positions(int t, PRound &r)
{
    std::vector<int> order;
    bool taken[12] = {};
    unsigned basis[3];
    int nb = 0;
    auto inside = [&](int bit) { return bit / 2 + 1 == r.db || bit / 2 + 1 == r.dc; };
    for (int bit = 0; bit < 2 * (t - 1) && nb < 3; bit++) {
        if (inside(bit)) continue;
        unsigned v = pauli_swz(1u << bit) & 7u;
        for (int i = 0; i < nb; i++) v = std::min(v, v ^ basis[i]);
        if (!v) continue;
        basis[nb++] = v;
        order.push_back(bit);
        taken[bit] = true;
    }
    for (int bit = 0; bit < 2 * (t - 1); bit++)
        if (!inside(bit) && !taken[bit]) order.push_back(bit);
    r.nob = (uint8_t)order.size();
    auto at = [&](int bit) { return (uint16_t)(16u * pauli_swz(1u << bit)); };
    for (unsigned g = 0; g < 16; g++)
        for (int i = 0; i < 4; i++) {
            if (!((g >> i) & 1u)) continue;
            if (i < (int)order.size()) r.lo[g] ^= at(order[i]);
            if (4 + i < (int)order.size()) r.hi[g] ^= at(order[4 + i]);
        }
    uint16_t *m = r.st;
    m[0] = at(2 * (r.db - 1)), m[1] = at(2 * (r.db - 1) + 1);
    m[2] = at(2 * (r.dc - 1)), m[3] = at(2 * (r.dc - 1) + 1);
    for (int i = 0; i < 4; i++) r.ld[i] = m[i];
    // the label pair that moves to (p_b, p_c): x_t ^= x_c, z_c ^= z_t (CNOT); z ^= the other x (CZ)
    if (r.perm == PP_CX_BC) r.ld[1] ^= m[3], r.ld[2] ^= m[0];
    if (r.perm == PP_CX_CB) r.ld[3] ^= m[1], r.ld[0] ^= m[2];
    if (r.perm == PP_CZ) r.ld[1] ^= m[2], r.ld[3] ^= m[0];
}

void push_tp(std::vector<float> &c, const M4 &m)  // rows 1..3
{
    for (int i = 4; i < 16; i++) c.push_back((float)m.m[i]);
}

int node_coefs(const Node &nd) { return nd.kind == PO_TWO ? 256 : nd.kind == PO_ONE ? 16 : 24; }

// Append node nd to a pass; dig(q) = 0, 1, 2: the register digit of its qubits.  maps_only: its
// permutation is the round's own.
template <typename F>
void emit(PPass &ps, const Node &nd, bool maps_only, F dig)
{
    POp op{};
    op.coef = (uint16_t)(ps.coefs.size() / 4);
    const int da = dig(nd.a), db = nd.b >= 0 ? dig(nd.b) : -1;
    if (maps_only) {
        op.kind = PO_MM;
        push_tp(ps.coefs, da == 1 ? nd.A : nd.B);
        push_tp(ps.coefs, da == 1 ? nd.B : nd.A);
    } else if (nd.kind == PO_ONE) {
        op.kind = (uint16_t)(PO_ONE + da);
        for (int i = 0; i < 16; i++) ps.coefs.push_back((float)nd.A.m[i]);
    } else if (nd.kind == PO_CX) {
        op.kind = (uint16_t)(PO_CX + 2 * da + (db > da ? db - 1 : db));
        push_tp(ps.coefs, nd.A);
        push_tp(ps.coefs, nd.B);
    } else if (nd.kind == PO_CZ) {
        const int lo = std::min(da, db), hi = std::max(da, db);
        op.kind = (uint16_t)(PO_CZ + lo + hi - 1);  // (0,1) (0,2) (1,2)
        push_tp(ps.coefs, da < db ? nd.A : nd.B);
        push_tp(ps.coefs, da < db ? nd.B : nd.A);
    } else {
        const int lo = std::min(da, db), hi = std::max(da, db);
        op.kind = (uint16_t)(PO_TWO + lo + hi - 1);  // (1,0) (2,0) (2,1)
        const std::vector<double> T = da > db ? nd.T : exchanged(nd.T);
        for (double x : T) ps.coefs.push_back((float)x);
    }
    ps.ops.push_back(op);
}

}  // namespace

static PauliPlan plan_nodes(NodeBuilder &nb, int n, int kmax, bool beam, bool zero)
{
    std::vector<Node> nodes = nb.finish();
    PauliPlan plan;
    plan.n = n;
    plan.nd = std::max(n, kPMinDigits);
    const int nd = plan.nd, t = std::min(nd, kPTile);
    auto digit = [&](int q) { return n - 1 - q; };
    std::vector<unsigned> mask(nodes.size());
    for (size_t i = 0; i < nodes.size(); i++) {
        mask[i] = 1u << digit(nodes[i].a);
        if (nodes[i].b >= 0) mask[i] |= 1u << digit(nodes[i].b);
    }
    const bool whole = nd <= t && !kmax;
    std::vector<unsigned> cand;
    if (whole) cand.push_back((1u << nd) - 1u);
    else cand = pass_candidates(nd, t, kmax);
    std::vector<unsigned> seq;
    if (beam && cand.size() > 1) seq = beam_pass_sets(mask, cand);
    std::vector<size_t> rem(nodes.size());
    for (size_t i = 0; i < rem.size(); i++) rem[i] = i;
    size_t nseq = 0;
    while (!rem.empty()) {
        std::vector<unsigned> rm;
        for (size_t i : rem) rm.push_back(mask[i]);
        unsigned Q = 0;
        if (nseq < seq.size()) {
            Q = seq[nseq++];
        } else {
            size_t best = 0;
            for (unsigned C : cand) {
                const size_t a = cand.size() == 1 ? 1 : absorbable(rm, C);
                if (a > best) best = a, Q = C;
            }
        }
        // the tile: Q, the two lowest digits, then the lowest others
        unsigned T = Q | 3u;
        for (int d = 0; d < nd && __builtin_popcount(T) < t; d++) T |= 1u << d;
        PPass ps;
        ps.t = t;
        int tile_of[32];
        for (int d = 0; d < nd; d++) {
            tile_of[d] = -1;
            if (T & (1u << d)) tile_of[d] = (int)ps.td.size(), ps.td.push_back(d);
            else ps.od.push_back(d);
        }
        std::vector<size_t> chosen, rest;
        unsigned blocked = 0;
        size_t ncoef = 0;
        for (size_t j = 0; j < rem.size(); j++) {
            const int nc = node_coefs(nodes[rem[j]]);
            if ((rm[j] & ~Q) || (rm[j] & blocked) || ncoef + nc > (size_t)kPMaxCoef || (int)chosen.size() >= kPMaxRounds) {
                rest.push_back(rem[j]);
                blocked |= rm[j];
            } else {
                chosen.push_back(rem[j]);
                ncoef += nc;
            }
        }
        if (chosen.empty()) continue;  // a set of the sequence whose operations wait for ones a full pass left
        // rounds: of all pairs of tile digits beside digit 0, the one that takes most of what is left
        auto tmask = [&](size_t i) {
            unsigned m = 1u << tile_of[digit(nodes[i].a)];
            if (nodes[i].b >= 0) m |= 1u << tile_of[digit(nodes[i].b)];
            return m;
        };
        while (!chosen.empty()) {
            std::vector<unsigned> cm;
            for (size_t i : chosen) cm.push_back(tmask(i));
            PRound r{};
            size_t best = 0;
            for (int b = 1; b < t; b++)
                for (int c = b + 1; c < t; c++) {
                    const size_t a = absorbable(cm, 1u | (1u << b) | (1u << c));
                    if (a > best) best = a, r.db = (uint8_t)b, r.dc = (uint8_t)c;
                }
            const unsigned R = 1u | (1u << r.db) | (1u << r.dc);
            r.op0 = (uint16_t)ps.ops.size();
            std::vector<size_t> left, take;
            unsigned bl = 0;
            for (size_t j = 0; j < chosen.size(); j++) {
                if ((cm[j] & ~R) || (cm[j] & bl)) {
                    left.push_back(chosen[j]);
                    bl |= cm[j];
                } else {
                    take.push_back(chosen[j]);
                }
            }
            // a CNOT / CZ of db and dc that nothing but digit-0 maps precede starts the round
            for (size_t j = 0; j < take.size(); j++) {
                const Node &nd2 = nodes[take[j]];
                const unsigned m = tmask(take[j]);
                if (m == 1u) continue;
                if (!(m & 1u) && (nd2.kind == PO_CX || nd2.kind == PO_CZ)) {
                    r.perm = nd2.kind == PO_CZ ? PP_CZ : tile_of[digit(nd2.a)] == r.db ? PP_CX_BC : PP_CX_CB;
                    std::rotate(take.begin(), take.begin() + j, take.begin() + j + 1);
                }
                break;
            }
            round_positions(t, r);
            auto lone = [&](size_t j) {  // trace-preserving one-qubit map of db or dc
                return j < take.size() && nodes[take[j]].kind == PO_ONE && tmask(take[j]) != 1u && m4_tp(nodes[take[j]].A);
            };
            for (size_t j = 0; j < take.size(); j++) {
                if (lone(j) && lone(j + 1) && tmask(take[j]) != tmask(take[j + 1])) {  // one of each: both at once
                    const bool first = tmask(take[j]) == 1u << r.db;
                    POp op{PO_MM, (uint16_t)(ps.coefs.size() / 4)};
                    push_tp(ps.coefs, nodes[take[first ? j : j + 1]].A);
                    push_tp(ps.coefs, nodes[take[first ? j + 1 : j]].A);
                    ps.ops.push_back(op);
                    j++;
                    continue;
                }
                emit(ps, nodes[take[j]], j == 0 && r.perm, [&](int q) {
                    const int d = tile_of[digit(q)];
                    return d == 0 ? 0 : d == r.db ? 1 : 2;
                });
            }
            r.nop = (uint8_t)(ps.ops.size() - r.op0);
            ps.rounds.push_back(r);
            chosen.swap(left);
        }
        plan.passes.push_back(std::move(ps));
        rem.swap(rest);
    }
    plan.w = nb.product(nd);
    if (zero && plan.passes.empty()) {  // the product state still has to be written
        PPass ps;
        ps.t = t;
        for (int d = 0; d < nd; d++) (d < t ? ps.td : ps.od).push_back(d);
        plan.passes.push_back(std::move(ps));
    }
    return plan;
}

PauliPlan plan_pauli(const std::vector<QOp> &ops, size_t begin, size_t end, int n, int kmax, bool beam, bool zero)
{
    NodeBuilder nb(n, zero);
    for (size_t i = begin; i < end; i++) nb.add(OpView{ops[i].kind, ops[i].k, ops[i].qubits, ops[i].m.data()});
    return plan_nodes(nb, n, kmax, beam, zero);
}

PauliPlan plan_pauli_list(const qcw_op *ops, int nops, const double *matrices, int n, int kmax)
{
    NodeBuilder nb(n, true);
    c128 S[256];
    for (int i = 0; i < nops; i++) {
        const qcw_op &o = ops[i];
        const c128 *m = reinterpret_cast<const c128 *>(matrices + o.offset);
        if (o.kind != QCW_OP_KRAUS) {
            nb.add(OpView{0, o.k, o.qubits, m});
            continue;
        }
        const int d = 1 << o.k, D = d * d;  // sum_j K_j (x) conj K_j
        for (int e = 0; e < D * D; e++) S[e] = 0;
        for (int j = 0; j < o.nkraus; j++, m += D)
            for (int r2 = 0; r2 < d; r2++)
                for (int c2 = 0; c2 < d; c2++)
                    for (int r = 0; r < d; r++) {
                        const double a = m[r2 * d + r].real(), b = m[r2 * d + r].imag();
                        if (a == 0 && b == 0) continue;
                        c128 *row = S + (r2 * d + c2) * D + r * d;
                        for (int c = 0; c < d; c++) {
                            const double x = m[c2 * d + c].real(), y = m[c2 * d + c].imag();
                            row[c] += c128(a * x + b * y, b * x - a * y);
                        }
                    }
        nb.add(OpView{1, o.k, o.qubits, S});
    }
    return plan_nodes(nb, n, kmax, false, true);
}

// Runs on pairs.  A node joins the pass of its qubits while no later pass holds one of them (so the
// passes can run in the order they were opened); maps of a qubit that is in no open pass wait for its
// next one, and the qubits left over at the end share passes two by two.
std::vector<PairProg> plan_pairs(const std::vector<QOp> &ops, size_t begin, size_t end, int n)
{
    NodeBuilder nb(n, false);
    for (size_t i = begin; i < end; i++) nb.add(OpView{ops[i].kind, ops[i].k, ops[i].qubits, ops[i].m.data()});
    std::vector<PairProg> out;
    std::vector<int> open(n, -1);
    std::vector<M4> wait(n, m4_identity());
    auto map = [&](PairProg &p, int q, const M4 &m) {
        if (m.id) return;
        const bool tp = m4_tp(m);
        p.kind.push_back((uint8_t)((tp ? PK_MAP : PK_GEN) + (q == p.a ? 0 : 1)));
        for (int i = tp ? 4 : 0; i < 16; i++) p.coefs.push_back((float)m.m[i]);
    };
    auto close = [&](int q) {
        const int j = open[q];
        if (j >= 0) open[out[j].a] = -1, open[out[j].b] = -1;
    };
    auto fresh = [&](int a, int b) -> PairProg & {
        close(a), close(b);
        open[a] = open[b] = (int)out.size();
        PairProg p;
        p.a = a, p.b = b;
        for (int q : {a, b}) {
            map(p, q, wait[q]);
            wait[q] = m4_identity();
        }
        out.push_back(std::move(p));
        return out.back();
    };
    for (const Node &nd : nb.finish()) {
        if (nd.kind == PO_ONE) {
            if (open[nd.a] >= 0 && (int)out[open[nd.a]].kind.size() < kPairMaxOps) map(out[open[nd.a]], nd.a, nd.A);
            else {
                close(nd.a);
                m4_lmul(wait[nd.a], nd.A);
            }
            continue;
        }
        const bool same = open[nd.a] >= 0 && open[nd.a] == open[nd.b];
        if (nd.kind == PO_TWO) {
            PairProg &p = fresh(nd.a, nd.b);
            p.T = nd.T;
            if (!p.kind.empty()) {  // maps that waited: a pass of their own before
                PairProg t;
                t.a = nd.a, t.b = nd.b;
                t.T.swap(p.T);
                out.push_back(std::move(t));
            }
            open[nd.a] = open[nd.b] = -1;
            continue;
        }
        PairProg &p = same && (int)out[open[nd.a]].kind.size() + 3 <= kPairMaxOps ? out[open[nd.a]] : fresh(nd.a, nd.b);
        p.kind.push_back((uint8_t)(nd.kind == PO_CZ ? PK_CZ : nd.a == p.a ? PK_CX : PK_CX + 1));
        map(p, nd.a, nd.A);
        map(p, nd.b, nd.B);
    }
    std::vector<int> left;
    for (int q = 0; q < n; q++)
        if (!wait[q].id) left.push_back(q);
    for (size_t i = 0; i + 1 < left.size(); i += 2) fresh(left[i], left[i + 1]);
    if (left.size() % 2) {
        PairProg p;
        p.a = left.back();
        std::copy(wait[p.a].m, wait[p.a].m + 16, p.one);
        out.push_back(std::move(p));
    }
    return out;
}

}  // namespace qcw
