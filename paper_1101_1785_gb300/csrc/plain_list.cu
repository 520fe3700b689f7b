// Operation lists on the plain path: the operations of one call, merged into fewer passes over rho.
// Applied one by one, every operation is a launch of its own and, from ten qubits up, a read and a write
// of rho.  In a list the one-qubit operations between two two-qubit ones are multiplied (in double)
// into one map per qubit, and what stays on two qubits runs in one pass.  12 qubits, 30 gates with
// depolarising noise: 8 passes of 39 us (269 MB each: 6.8 TB/s, as k_super1 and k_mono2) where there
// were 69; 2.95 -> 0.61 ms with the readouts.  4 qubits, 40 gates with amplitude and phase damping:
// one launch of 9 us where there were about 120; 485 -> 120 us.  The errors against 64 bits shrink
// with the number of roundings (1.4e-6 -> 2.6e-7 and 9.7e-7 -> 1.3e-7 relative).
// Lists of one operation, controlled, wider and exactly permuting operations (SWAP, iSWAP) run as they
// do one by one.
#include <algorithm>
#include <cstddef>
#include <cstring>

#include "pauli.cuh"
#include "qcw_internal.h"

namespace qcw {

// ------------------------------------------------------------------ a run on two qubits
// 16-member groups as in k_super2: member e = 8 r_a + 4 r_b + 2 c_a + c_b, row and column bits of both
// qubits.  rho is a complex combination of Hermitian matrices, so every map is real on the Pauli
// coefficients of its qubit's quartets: as in k_super1 a quartet goes to them, through the map and back.
// The other qubit's members stay as they are and CNOT and CZ rename them (CZ with signs), so what they
// hold keeps its own relative precision: a population of 1e-9 beside one of 1 survives operations on
// other qubits and its own as a control.  (Members kept as coefficients of both qubits across the run
// need fewer operations, but lose whatever lies below 2^-24 of the group; the 12-qubit circuit takes
// 698 us with its readouts that way and 702 us this way.)
__device__ __forceinline__ pu64 padd2(pu64 a, pu64 b)
{
    pu64 d;
    asm("add.rn.f32x2 %0, %1, %2;\n" : "=l"(d) : "l"(a), "l"(b));
    return d;
}

// Map of a (B = false) or b, coefficients halved (from twice the inverse of the change of basis); TP:
// rows 1..3.  The fence keeps the coefficients from being loaded before the quartets are changed (spills).
template <bool B, bool TP, int V, class P>
__device__ __forceinline__ void pair_map(pu64 (&x)[V][16], const P &p, unsigned k)
{
    constexpr int N = TP ? 12 : 16, SR = B ? 4 : 8, SC = B ? 1 : 2, O1 = B ? 2 : 1, O2 = B ? 8 : 4;
#pragma unroll
    for (int v = 0; v < V; v++)
#pragma unroll
        for (int l = 0; l < 4; l++) {  // elements 00, 11, 01, 10 -> I, Z, X, Y = i (e01 - e10)
            const int o = (l & 1) * O1 + (l >> 1) * O2;
            const pu64 a = x[v][o], d = x[v][o + SR + SC], s = x[v][o + SC], t = x[v][o + SR];
            const float2 b = unpack2(s), c = unpack2(t);
            x[v][o] = padd2(a, d);
            x[v][o + SR + SC] = padd2(a, fneg2(d));
            x[v][o + SC] = padd2(s, t);
            x[v][o + SR] = pack2(c.y - b.y, b.x - c.x);
        }
    __syncwarp(__activemask());
    pu64 c[N];
    p_coefs(p, k, c);
#pragma unroll
    for (int v = 0; v < V; v++)
#pragma unroll
        for (int l = 0; l < 4; l++) {
            const int o = (l & 1) * O1 + (l >> 1) * O2;
            const pu64 in[4] = {x[v][o], x[v][o + SR + SC], x[v][o + SC], x[v][o + SR]};
            pu64 out[4];
            if (TP) out[0] = fmul2(pack2(0.5f, 0.5f), in[0]);
#pragma unroll
            for (int r = TP ? 1 : 0; r < 4; r++) {
                const pu64 *w = c + 4 * (TP ? r - 1 : r);
                out[r] = ffma2(w[3], in[3], ffma2(w[2], in[2], ffma2(w[1], in[1], fmul2(w[0], in[0]))));
            }
            const float2 u = unpack2(out[2]), y = unpack2(out[3]);
            x[v][o] = padd2(out[0], out[1]);
            x[v][o + SR + SC] = padd2(out[0], fneg2(out[1]));
            x[v][o + SC] = pack2(u.x + y.y, u.y - y.x);
            x[v][o + SR] = pack2(u.x - y.y, u.y + y.x);
        }
}

// CNOT (SWAP = false: a controls) or CZ.
template <bool CZ, bool SWAP, int V>
__device__ __forceinline__ void pair_perm(pu64 (&x)[V][16])
{
#pragma unroll
    for (int v = 0; v < V; v++) {
        pu64 y[16];
#pragma unroll
        for (int e = 0; e < 16; e++) {
            const int ra = e >> 3, rb = (e >> 2) & 1, ca = (e >> 1) & 1, cb = e & 1;
            if (CZ) y[e] = (ra & rb) != (ca & cb) ? fneg2(x[v][e]) : x[v][e];
            else y[e] = x[v][SWAP ? e ^ (8 * rb + 2 * cb) : e ^ (4 * ra + ca)];
        }
#pragma unroll
        for (int e = 0; e < 16; e++) x[v][e] = y[e];
    }
}

// Operation word: PK_* kind, first coefficient pair from bit 8.
template <int V, class P>
__device__ __forceinline__ void pair_run(pu64 (&x)[V][16], const P &p, unsigned op0, unsigned nop)
{
#pragma unroll 1
    for (unsigned o = op0; o < op0 + nop; o++) {
        const unsigned w = p.op(o), k = w >> 8;
        switch (w & 255u) {
        case PK_MAP: pair_map<false, true>(x, p, k); break;
        case PK_MAP + 1: pair_map<true, true>(x, p, k); break;
        case PK_GEN: pair_map<false, false>(x, p, k); break;
        case PK_GEN + 1: pair_map<true, false>(x, p, k); break;
        case PK_CX: pair_perm<false, false>(x); break;
        case PK_CX + 1: pair_perm<false, true>(x); break;
        case PK_CZ: pair_perm<true, false>(x); break;
        }
    }
}

struct PairHead {
    uint8_t bit[4];  // of the flat index of rho: row of a, of b, column of a, of b
    uint8_t pos[4];  // the same, ascending
    uint16_t op0, nop;
    uint32_t pad;
};

template <int W>
struct PairParams {
    int nprog, ops, coef, n;  // ops, coef: word offsets; n: words in use
    unsigned w[W];            // PairHead[nprog], operation words, coefficient pairs
};
static_assert(offsetof(PairParams<4>, w) % 16 == 0, "vector loads from the parameter block");

__device__ __forceinline__ uint64_t pair_base(uint64_t t, const PairHead &h)
{
    return insert0(insert0(insert0(insert0(t, h.pos[0]), h.pos[1]), h.pos[2]), h.pos[3]);
}

constexpr int kPairWords = 4 + kPairMaxOps + 2 * 16 * kPairMaxOps;
constexpr int kPairThreads = 128;

// One read and one write of rho per run.  Bound by HBM: a run of four maps and a CNOT adds about 50
// issue slots per element, 22 us at 12 qubits where the traffic takes 39.  Two neighbouring groups per
// thread (float4) unless column bit 0 is struck; four blocks of 128 threads per SM keep 16 loads in
// flight each, and the 64 values of two groups with a map's coefficients fit 128 registers.
template <int V>
__global__ void __launch_bounds__(kPairThreads, 4)
    k_pair(float2 *__restrict__ rho, uint64_t nitems, const __grid_constant__ PairParams<kPairWords> prm)
{
    const PairHead h = *reinterpret_cast<const PairHead *>(prm.w);
    const ProgParam prog{prm.w, prm.ops, prm.coef};
    for (uint64_t s = blockIdx.x * (uint64_t)kPairThreads + threadIdx.x; s < nitems; s += (uint64_t)gridDim.x * kPairThreads) {
        float2 *g = rho + pair_base(V * s, h);
        auto at = [&](int e) {
            return g + ((uint64_t)((e >> 3) & 1) << h.bit[0]) + ((uint64_t)((e >> 2) & 1) << h.bit[1]) +
                   ((uint64_t)((e >> 1) & 1) << h.bit[2]) + ((uint64_t)(e & 1) << h.bit[3]);
        };
        pu64 x[V][16];
#pragma unroll
        for (int e = 0; e < 16; e++) {
            if constexpr (V == 2) {
                const ulonglong2 a = *reinterpret_cast<const ulonglong2 *>(at(e));
                x[0][e] = a.x, x[V - 1][e] = a.y;
            } else {
                x[0][e] = *reinterpret_cast<const pu64 *>(at(e));
            }
        }
        pair_run(x, prog, 0, h.nop);
#pragma unroll
        for (int e = 0; e < 16; e++) {
            if constexpr (V == 2) *reinterpret_cast<ulonglong2 *>(at(e)) = make_ulonglong2(x[0][e], x[V - 1][e]);
            else *reinterpret_cast<pu64 *>(at(e)) = x[0][e];
        }
    }
}

// ------------------------------------------------------------------ registers of 2 to 6 qubits
// rho (at most 32 KiB) in the shared memory of one block, all runs of the list in one launch, a group
// per thread, against a launch per run: circuits of 40 and 400 gates with readouts 154 and
// 381 against 168 and 527 us (4 qubits), 175 and 424 against 181 and 585 us (6 qubits); of 5 gates alike.
// The line is where a block of 256 threads holds every group and the tile fits static shared memory;
// seven qubits would need 128 KiB and four groups per thread.
constexpr int kSmallList = 6;
constexpr int kSmallWords = 1920;  // 7.5 KiB of parameters: a longer list takes several launches

__global__ void __launch_bounds__(256)
    k_pair_small(float2 *__restrict__ rho, int n, const __grid_constant__ PairParams<kSmallWords> prm)
{
    __shared__ __align__(16) pu64 tile[1 << (2 * kSmallList)];
    __shared__ __align__(16) unsigned prog[kSmallWords];
    const unsigned ngroup = 1u << (2 * n - 4), nelem = 1u << (2 * n);
    for (unsigned i = threadIdx.x; i < (unsigned)prm.n; i += blockDim.x) prog[i] = prm.w[i];
    for (unsigned i = threadIdx.x; i < nelem; i += blockDim.x) tile[i] = reinterpret_cast<const pu64 *>(rho)[i];
    __syncthreads();
    const ProgShared p{nullptr, reinterpret_cast<const POp *>(prog + prm.ops), smem_u32(prog + prm.coef)};
    const int nprog = prm.nprog;
#pragma unroll 1
    for (int r = 0; r < nprog; r++) {
        if (threadIdx.x < ngroup) {
            const PairHead h = reinterpret_cast<const PairHead *>(prog)[r];
            const unsigned g = (unsigned)pair_base(threadIdx.x, h);
            pu64 x[1][16];
#pragma unroll
            for (int e = 0; e < 16; e++)
                x[0][e] = tile[g + (((e >> 3) & 1u) << h.bit[0]) + (((e >> 2) & 1u) << h.bit[1]) +
                               (((e >> 1) & 1u) << h.bit[2]) + ((e & 1u) << h.bit[3])];
            pair_run(x, p, h.op0, h.nop);
#pragma unroll
            for (int e = 0; e < 16; e++)
                tile[g + (((e >> 3) & 1u) << h.bit[0]) + (((e >> 2) & 1u) << h.bit[1]) + (((e >> 1) & 1u) << h.bit[2]) +
                     ((e & 1u) << h.bit[3])] = x[0][e];
        }
        __syncthreads();
    }
    for (unsigned i = threadIdx.x; i < nelem; i += blockDim.x) reinterpret_cast<pu64 *>(rho)[i] = tile[i];
}

// ------------------------------------------------------------------ host
namespace {

qcw_status launched(qcw_ctx *c)
{
    c->launches++;
    const cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? QCW_OK : cuda_error(e, "kernel launch");
}

int words_of(const PairProg &p) { return 4 + (int)p.kind.size() + 2 * (int)p.coefs.size(); }

// progs[0, cnt) as one parameter block of prm.w's size.
template <int W>
void encode(const PairProg *progs, int cnt, int n, PairParams<W> &prm)
{
    int nop = 0;
    for (int i = 0; i < cnt; i++) nop += (int)progs[i].kind.size();
    prm.nprog = cnt;
    prm.ops = 4 * cnt;
    prm.coef = prm.ops + ((nop + 3) & ~3);
    unsigned *ops = prm.w + prm.ops, *coef = prm.w + prm.coef;
    int o = 0, k = 0;
    for (int i = 0; i < cnt; i++) {
        const PairProg &p = progs[i];
        PairHead h{};
        h.bit[0] = (uint8_t)(2 * n - 1 - p.a), h.bit[1] = (uint8_t)(2 * n - 1 - p.b);
        h.bit[2] = (uint8_t)(n - 1 - p.a), h.bit[3] = (uint8_t)(n - 1 - p.b);
        std::copy(h.bit, h.bit + 4, h.pos);
        std::sort(h.pos, h.pos + 4);
        h.op0 = (uint16_t)o, h.nop = (uint16_t)p.kind.size();
        memcpy(prm.w + 4 * i, &h, sizeof h);
        size_t c = 0;
        for (uint8_t kind : p.kind) {
            ops[o++] = kind | (unsigned)k << 8;
            const int m = kind < PK_GEN ? 12 : kind < PK_CX ? 16 : 0;
            for (int j = 0; j < m; j++, k++, c++) {
                const float half = 0.5f * p.coefs[c];
                memcpy(coef + 2 * k, &half, 4), memcpy(coef + 2 * k + 1, &half, 4);
            }
        }
    }
    prm.n = prm.coef + 2 * k;
}

bool has_map(const PairProg &p)
{
    for (uint8_t k : p.kind)
        if (k < PK_CX) return true;
    return false;
}

// A 4 x 4 (or 16 x 16) matrix on the labels as the transfer matrix of k_super1 (k_super2).
const int kMemberLab[4] = {0, 2, 3, 1};

qcw_status run_one(qcw_ctx *c, const PairProg &p)
{
    Super1Params s{};
    for (int i = 0; i < 4; i++)
        for (int j = 0; j < 4; j++) s.r[4 * i + j] = (float)(0.5 * p.one[4 * kMemberLab[i] + kMemberLab[j]]);
    s.pc = c->n - 1 - p.a;
    s.pr = 2 * c->n - 1 - p.a;
    launch_super1(s, c->rho, c->n, c->nsm, c->stream);
    return launched(c);
}

qcw_status run_dense(qcw_ctx *c, const PairProg &p)
{
    Super2Params s{};
    auto lab = [](int e) {
        return 4 * kMemberLab[2 * ((e >> 3) & 1) + ((e >> 1) & 1)] + kMemberLab[2 * ((e >> 2) & 1) + (e & 1)];
    };
    auto sg = [](int e) { return (e & 12) == 12 && (e & 3) == 0 ? -1.0 : 1.0; };  // D D = -(Y Y)
    for (int i = 0; i < 16; i++)
        for (int j = 0; j < 16; j++) s.r[16 * i + j] = (float)(0.25 * p.T[16 * lab(i) + lab(j)] * sg(i) * sg(j));
    quartet_layout(c->n, p.a, p.b, s.pos, s.off_r, s.off_c);
    launch_super2(s, c->rho, c->n, c->nsm, c->stream);
    return launched(c);
}

qcw_status run_perms(qcw_ctx *c, const PairProg &p)
{
    const c128 cx[16] = {1, 0, 0, 0, 0, 1, 0, 0, 0, 0, 0, 1, 0, 0, 1, 0}, cz[16] = {1, 0, 0, 0, 0, 1, 0, 0, 0, 0, 1, 0, 0, 0, 0, -1};
    for (uint8_t k : p.kind) {
        const bool rev = k == PK_CX + 1;
        const qcw_status st = plain_gate2(c, k == PK_CZ ? cz : cx, rev ? p.b : p.a, rev ? p.a : p.b, nullptr, 0);
        if (st) return st;
    }
    return QCW_OK;
}

qcw_status run_pairs(qcw_ctx *c, const std::vector<PairProg> &progs)
{
    const int n = c->n;
    for (size_t i = 0; i < progs.size();) {
        const PairProg &p = progs[i];
        if (p.b >= 0 && p.T.empty() && n <= kSmallList) {
            size_t e = i, words = 4;
            while (e < progs.size() && progs[e].b >= 0 && progs[e].T.empty() && words + words_of(progs[e]) <= kSmallWords)
                words += words_of(progs[e++]);
            bool maps = false;
            for (size_t j = i; j < e; j++) maps |= has_map(progs[j]);
            if (maps) {
                PairParams<kSmallWords> prm;
                encode(&progs[i], (int)(e - i), n, prm);
                k_pair_small<<<1, n == kSmallList ? 256 : 64, 0, c->stream>>>(c->rho, n, prm);
                const qcw_status st = launched(c);
                if (st) return st;
                i = e;
                continue;
            }
        }
        qcw_status st = QCW_OK;
        if (p.b < 0) st = run_one(c, p);
        else if (!p.T.empty()) st = run_dense(c, p);
        else if (!has_map(p)) st = run_perms(c, p);
        else {
            PairParams<kPairWords> prm;
            encode(&p, 1, n, prm);
            const uint64_t ng = 1ull << (2 * n - 4);
            const bool one = (p.a == n - 1 || p.b == n - 1);  // a struck bit 0: no neighbouring groups
            const uint64_t items = one ? ng : ng / 2;
            const unsigned grid = (unsigned)std::min<uint64_t>((items + kPairThreads - 1) / kPairThreads, 1u << 20);
            if (one) k_pair<1><<<grid, kPairThreads, 0, c->stream>>>(c->rho, items, prm);
            else k_pair<2><<<grid, kPairThreads, 0, c->stream>>>(c->rho, items, prm);
            st = launched(c);
        }
        if (st) return st;
        i++;
    }
    return QCW_OK;
}

// Gates and channels on one and two qubits join; not the exact permutations other than CNOT and CZ
// (SWAP, iSWAP, Pauli products), which k_mono2 moves without rounding and a dense map would not.
bool joins(const QOp &op)
{
    if (op.k > 2 || op.ncontrols > 0 || op.kind == 2) return false;
    if (op.k == 1 || op.kind == 1) return true;
    int sigma[4];
    c128 v[4];
    if (!monomial4(op.m.data(), sigma, v)) return true;
    const bool ones = v[0] == c128(1) && v[1] == c128(1) && v[2] == c128(1);
    const bool cx = sigma[0] == 0 && ((sigma[1] == 1 && sigma[2] == 3) || (sigma[1] == 3 && sigma[2] == 2));
    const bool id = sigma[0] == 0 && sigma[1] == 1 && sigma[2] == 2;
    return ones && ((cx && v[3] == c128(1)) || (id && v[3] == c128(-1)));
}

}  // namespace

qcw_status plain_list(qcw_ctx *c, const std::vector<QOp> &ops)
{
    for (size_t i = 0; i < ops.size();) {
        size_t e = i;
        while (e < ops.size() && joins(ops[e])) e++;
        qcw_status st;
        if (e - i < 2) {
            st = plain_apply(c, ops[i]);
            e = i + 1;
        } else {
            c->state_ver++;
            st = ensure_full(c);
            if (!st) st = run_pairs(c, plan_pairs(ops, i, e, c->n));
        }
        if (st) return st;
        i = e;
    }
    return QCW_OK;
}

}  // namespace qcw
