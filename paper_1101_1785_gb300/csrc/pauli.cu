// Pauli-basis path (see pauli.h): the pass kernel, the changes of basis to and from rho, and the
// readouts, all on the real vector v_P = Tr[P rho].
#include <algorithm>
#include <cstddef>
#include <cstring>
#include <type_traits>

#include "pauli.cuh"
#include "pauli_run.h"
#include "qcw_internal.h"

namespace qcw {

// ------------------------------------------------------------------ pass kernel
// Persistent, one CTA per SM: two teams of 256 threads work on alternate tiles of the CTA's list
// out of three tile buffers, so one buffer's loads (cp.async, released through an mbarrier) are in
// flight while the two teams evolve theirs.  Each buffer has one mbarrier per team: a buffer's tiles
// go to the two teams in turn, and a team that waited on the other's phases by parity could take an
// earlier one for its own.  A thread stores and reloads the same chunks of a
// buffer, so the write-back of tile i and the load of tile i + 3 need no barrier between them.
// Traffic: one read and one write of v, 8 * 4^n bytes.  Measured at n = 14 (2.15 GB): 0.56 ms per
// pass of four rounds and six operations, 3.8 TB/s (k_fused_herm_ws, on rho: 1.10 ms per pass, and a
// third more passes), 0.51 ms with the operations left out, 0.34 ms (6.2 TB/s) with the rounds left
// out: the rounds' trips through shared memory are what it waits for.  Hence the last round's results
// go from the registers straight to v (StoreDirect), one trip less: 0.61 before.  Each wait is
// bounded: the team that gives up sets the error word and stops, the other runs out of tiles or gives
// up in turn.
constexpr int kPBuf = 3;
constexpr int kPThreads = 512;
constexpr unsigned kPWaitLimit = 1u << 21;

template <int BYTES>
struct PauliParams {
    PauliHdr h;
    int pad[1];
    unsigned blob[BYTES / 4];  // PRound[nround], POp[nop], coefficient pairs float2[ncoef]
};
static_assert(offsetof(PauliParams<16>, blob) % 16 == 0, "vector loads from the parameter block");

// offsets in the blob (4-byte units)
__host__ __device__ inline int pb_ops(const PauliHdr &h) { return (int)(sizeof(PRound) / 4) * h.nround; }
__host__ __device__ inline int pb_coef(const PauliHdr &h) { return pb_ops(h) + ((h.nop + 3) & ~3); }

size_t pauli_pass_smem(const PauliHdr &h, bool dense)
{
    const size_t prog = dense ? 4 * (size_t)pb_coef(h) + sizeof(float2) * (size_t)h.ncoef : sizeof(PRound) * (size_t)h.nround;
    return (size_t)kPBuf * (sizeof(float) << (2 * h.t)) + prog + 16 * sizeof(double) + 2 * kPBuf * sizeof(uint64_t) + 32;
}

// The last round's elements straight from the registers to v: the lanes of a quarter-warp hold the
// labels of tile digit 1 (which the round does not touch), so they fill 64-byte runs.  A round that
// does touch digit 1 would scatter 16-byte pieces; there, and for dense maps and small tiles, the
// results go through the tile.  Per pass, through the tile / direct: n = 9 13.2 / 12.8 us, n = 13
// 170 / 156 us, n = 14 610 / 562 us.
template <bool PUR>
struct StoreDirect {
    static constexpr bool kDirect = true, kFull = true;
    float *v;
    const volatile int8_t *td;  // tile digits, then (8 on) the outside ones, in shared memory: see Walk
    int nod;
    unsigned tid, tile;
    float &ps;
    __device__ __forceinline__ void store(const PRound &R, const pu64 (&x)[32], unsigned db, unsigned dc) const
    {
        const unsigned c = pauli_swz(((unsigned)R.lo[tid & 15u] ^ (unsigned)R.hi[tid >> 4]) >> 4);  // its own inverse
        uint64_t g = 0;
        for (int d = 0; d < nod; d++) g += (uint64_t)((tile >> (2 * d)) & 3u) << (2 * td[8 + d]);
#pragma unroll
        for (int d = 1; d < kPTile; d++) g += (uint64_t)((c >> (2 * (d - 1))) & 3u) << (2 * td[d]);
        const uint64_t sb = 1ull << (2 * td[db]), sc = 1ull << (2 * td[dc]);
        float *pj = v + g;
#pragma unroll
        for (int j = 0; j < 4; j++) {
            float *pi = pj;
#pragma unroll
            for (int i = 0; i < 4; i++) {
                const float2 a = unpack2(x[px(0, i, j)]), b = unpack2(x[px(1, i, j)]);
                *reinterpret_cast<float4 *>(pi) = make_float4(a.x, a.y, b.x, b.y);
                if (PUR) ps = fmaf(a.x, a.x, fmaf(a.y, a.y, fmaf(b.x, b.x, fmaf(b.y, b.y, ps))));
                pi += sb;
            }
            pj += sc;
        }
    }
};

// INIT: start from the header's product state.  FULL: tiles of kPTile digits (every register from
// seven qubits up) and no dense maps.  Both are fixed at compile time because the registers are all
// in use: either one as a run-time branch spilled part of the 64 elements.
template <int BYTES, bool DENSE, bool FULL, bool INIT, bool PUR>
__global__ void __launch_bounds__(kPThreads, 1)
    k_pauli_pass(float *__restrict__ v, unsigned ntiles, unsigned long long *__restrict__ err,
                 unsigned wait_limit, int stall_tile, double *__restrict__ ppart, double pscale,
                 const __grid_constant__ PauliParams<BYTES> prm)
{
    extern __shared__ __align__(16) unsigned char smem[];
    const PauliHdr &H = prm.h;
    const int t = FULL ? kPTile : H.t;
    const unsigned nchunk = 1u << (2 * (t - 1));
    const size_t tbytes = sizeof(float) << (2 * t);
    unsigned char *p = smem + kPBuf * tbytes;
    PRound *rounds = reinterpret_cast<PRound *>(p);
    const int nword = DENSE ? pb_coef(H) + 2 * H.ncoef : pb_ops(H);  // of the program kept in shared memory
    double *red = reinterpret_cast<double *>(reinterpret_cast<unsigned *>(rounds) + nword);
    uint64_t *full = reinterpret_cast<uint64_t *>(red + 16);
    volatile int8_t *td = reinterpret_cast<volatile int8_t *>(full + 2 * kPBuf);
    if (threadIdx.x < 24) td[threadIdx.x] = threadIdx.x < 8 ? H.td[threadIdx.x] : H.od[threadIdx.x - 8];
    const unsigned tid = threadIdx.x & 255u, team = threadIdx.x >> 8;
    for (int i = threadIdx.x; i < nword; i += kPThreads) reinterpret_cast<unsigned *>(rounds)[i] = prm.blob[i];
    if (threadIdx.x < 2 * kPBuf) mbar_init(&full[threadIdx.x], 256);
    __syncthreads();
    const unsigned ntile = blockIdx.x < ntiles ? (ntiles - 1 - blockIdx.x) / gridDim.x + 1 : 0;
    // A thread's chunks are tid + 256 k: offsets split into a part of the tile and of tid (tile digits
    // 1..4) and a part of k (digits 5, 6).  Worked out again for every copy, from digits read from
    // shared memory each time: kept across the rounds they would take registers from the 64 elements.
    struct Walk {
        uint64_t base, step5, step6;
        unsigned plo, mine;
        __device__ __forceinline__ uint64_t at(unsigned k) const { return (k & 3u) * step5 + (k >> 2) * step6; }
    };
    auto walk = [&](unsigned i) {
        unsigned id;
        asm volatile("mov.u32 %0, %1;\n" : "=r"(id) : "r"(tid));
        Walk w;
        const unsigned tile = blockIdx.x + i * gridDim.x;
        w.base = 0;
        for (int d = 1; d < t && d < 5; d++) w.base += (uint64_t)((id >> (2 * (d - 1))) & 3u) << (2 * td[d]);
        for (int d = 0; d < H.nod; d++) w.base += (uint64_t)((tile >> (2 * d)) & 3u) << (2 * td[8 + d]);
        w.step5 = t > 5 ? 1ull << (2 * td[5]) : 0;
        w.step6 = t > 6 ? 1ull << (2 * td[6]) : 0;
        w.plo = pauli_swz(id);
        w.mine = id < nchunk ? (nchunk + 255u) >> 8 : 0u;
        return w;
    };
    auto load = [&](unsigned i) {
        if (blockIdx.x == 0 && (int)i == stall_tile) return;
        const unsigned b = i % kPBuf;
        float4 *buf = reinterpret_cast<float4 *>(smem + b * tbytes);
        uint64_t *bar = &full[2 * b + (i & 1u)];
        const Walk w = walk(i);
        if (INIT) {  // the product state
            const unsigned tile = blockIdx.x + i * gridDim.x;
            const float f0 = p_factor(H.w, H.od, H.nod, tile);
            const float w0 = H.w[0], w1 = H.w[1], w2 = H.w[2], w3 = H.w[3];
            for (unsigned k = 0; k < w.mine; k++) {
                const float f = f0 * p_factor(H.w, H.td + 1, t - 1, tid + 256u * k);
                buf[w.plo ^ pauli_swz(256u * k)] = make_float4(f * w0, f * w1, f * w2, f * w3);
            }
            mbar_arrive(bar);
        } else {
            const float *src = v + w.base;
            if (t == kPTile) {
#pragma unroll
                for (unsigned k = 0; k < 16; k++) {
                    cp_async16(buf + (w.plo ^ pauli_swz(256u * k)), src);
                    src += (k & 3u) == 3u ? w.step6 - 3 * w.step5 : w.step5;
                }
            } else {
                for (unsigned k = 0; k < w.mine; k++) cp_async16(buf + (w.plo ^ pauli_swz(256u * k)), src + w.at(k));
            }
            cp_async_mbar_arrive(bar);
        }
    };
    if (team == 0) {
        if (ntile > 0) load(0);
        if (ntile > 2) load(2);
    } else if (ntile > 1) {
        load(1);
    }
    const bool direct = FULL && H.nround > 0 && rounds[H.nround - 1].direct;
    double pacc = 0.0;
    for (unsigned i = team; i < ntile; i += 2) {
        const unsigned b = i % kPBuf;
        const bool ok = bar_and(1 + team, 256, mbar_wait(&full[2 * b + team], (i / (2 * kPBuf)) & 1u, wait_limit));
        if (!ok) {
            if (tid == 0) atomicOr(err, 1ull);
            break;
        }
        float ps = 0.f;
        const unsigned ba = smem_u32(smem) + (unsigned)(b * tbytes);
        if constexpr (DENSE) {
            const unsigned *w = reinterpret_cast<const unsigned *>(rounds);
            const ProgShared prog{rounds, reinterpret_cast<const POp *>(w + pb_ops(H)), smem_u32(w + pb_coef(H))};
            pauli_rounds<true>(ba, rounds, H.nround, prog, tid, 1 + team);
        } else {
            const ProgParam prog{prm.blob, pb_ops(H), pb_coef(H)};
            if constexpr (FULL) {
                const StoreDirect<PUR> last{v, td, H.nod, tid, blockIdx.x + i * gridDim.x, ps};
                pauli_rounds<false>(ba, rounds, H.nround, prog, tid, 1 + team, last);
                if (direct) {
                    if (PUR) pacc += (double)ps;
                    if (i + kPBuf < ntile) load(i + kPBuf);
                    continue;
                }
            } else {
                pauli_rounds<false>(ba, rounds, H.nround, prog, tid, 1 + team);
            }
        }
        const Walk w = walk(i);
        float *dst = v + w.base;
        auto put = [&](unsigned k, float *to) {
            const float4 x = p_lds4(ba + 16u * (w.plo ^ pauli_swz(256u * k)));
            *reinterpret_cast<float4 *>(to) = x;
            if (PUR) ps = fmaf(x.x, x.x, fmaf(x.y, x.y, fmaf(x.z, x.z, fmaf(x.w, x.w, ps))));
        };
        if (t == kPTile) {
#pragma unroll
            for (unsigned k = 0; k < 16; k++) {
                put(k, dst);
                dst += (k & 3u) == 3u ? w.step6 - 3 * w.step5 : w.step5;
            }
        } else {
            for (unsigned k = 0; k < w.mine; k++) put(k, dst + w.at(k));
        }
        if (PUR) pacc += (double)ps;
        if (i + kPBuf < ntile) load(i + kPBuf);
    }
    cp_async_wait_all();
    if (PUR) {  // one partial per team, fixed order: shuffle tree per warp, then the warps in turn
        pacc = warp_sum(pacc);
        if ((threadIdx.x & 31u) == 0) red[threadIdx.x >> 5] = pacc;
        bar_sync(1 + team, 256);
        if (tid == 0) {
            double s = 0;
            for (int w = 0; w < 8; w++) s += red[8 * team + w];
            ppart[2 * blockIdx.x + team] = s * pscale;
        }
    }
}

template <int BYTES, bool DENSE, bool FULL>
static cudaError_t launch_pass(const PauliBlob &B, float *v, unsigned ntiles, unsigned grid, bool init,
                               unsigned long long *err, unsigned wait_limit, int stall_tile, double *ppart, double pscale,
                               cudaStream_t s)
{
    PauliParams<BYTES> prm;
    prm.h = B.h;
    memcpy(prm.blob, B.words.data(), 4 * B.words.size());
    auto kern = ppart ? (init ? k_pauli_pass<BYTES, DENSE, FULL, true, true> : k_pauli_pass<BYTES, DENSE, FULL, false, true>)
                      : (init ? k_pauli_pass<BYTES, DENSE, FULL, true, false> : k_pauli_pass<BYTES, DENSE, FULL, false, false>);
    const size_t sm = pauli_pass_smem(B.h, DENSE);
    if (ensure_smem_attr(reinterpret_cast<const void *>(kern), sm)) return cudaErrorInvalidValue;
    kern<<<grid, kPThreads, sm, s>>>(v, ntiles, err, wait_limit ? wait_limit : kPWaitLimit, stall_tile, ppart,
                                     pscale, prm);
    return cudaGetLastError();
}

bool pass_dense(const PPass &p)
{
    for (const POp &o : p.ops)
        if (o.kind >= PO_TWO && o.kind < PO_TWO + 3) return true;
    return false;
}

PauliHdr pauli_header(const PPass &p, const std::vector<float> &w)
{
    PauliHdr h;
    memset(&h, 0, sizeof h);
    h.t = p.t;
    h.nod = (int)p.od.size();
    h.nround = (int)p.rounds.size();
    h.nop = (int)p.ops.size();
    h.ncoef = (int)p.coefs.size();
    for (size_t i = 0; i < p.td.size(); i++) h.td[i] = (int8_t)p.td[i];
    for (size_t i = 0; i < p.od.size(); i++) h.od[i] = (int8_t)p.od[i];
    std::copy(w.begin(), w.end(), h.w);
    return h;
}

PauliBlob pauli_blob(const PPass &p, const std::vector<float> &w)
{
    PauliBlob B;
    B.h = pauli_header(p, w);
    B.dense = pass_dense(p);
    const PauliHdr &h = B.h;
    static_assert(sizeof(PRound) == 96 && sizeof(POp) == 4, "blob layout");
    B.words.assign((size_t)pb_coef(h) + 2 * h.ncoef, 0u);
    memcpy(B.words.data(), p.rounds.data(), sizeof(PRound) * p.rounds.size());
    if (h.nround && h.t == kPTile && !B.dense && p.rounds.back().db > 1)
        reinterpret_cast<PRound *>(B.words.data())[h.nround - 1].direct = 1;
    if (h.nop) memcpy(B.words.data() + pb_ops(h), p.ops.data(), sizeof(POp) * p.ops.size());
    for (size_t i = 0; i < p.coefs.size(); i++)
        for (int j = 0; j < 2; j++) memcpy(B.words.data() + pb_coef(h) + 2 * i + j, &p.coefs[i], sizeof(float));
    return B;
}

// A launch copies its whole parameter block, so the usual pass (no dense two-qubit map, a few
// rounds) has a small one.  Longer programs without dense maps, from deep circuits on up to about ten
// qubits, still read their coefficients through the constant cache, not from shared memory: 7 qubits,
// one pass of 21 rounds 55 -> 38 us, of 37 rounds 90 -> 63 us; 10 qubits, seven passes 17.1 -> 15.2 us
// each.
cudaError_t launch_pauli_pass(const PauliBlob &B, float *v, int nd, int nsm, bool init, unsigned long long *err,
                              unsigned wait_limit, int stall_tile, double *ppart, cudaStream_t s)
{
    const unsigned ntiles = 1u << (2 * B.h.nod), grid = pauli_grid(B.h, nsm);
    double pscale = 1.0;
    for (int i = 0; i < nd; i++) pscale *= 0.5;
    constexpr int kSmall = 3584;
    constexpr int kLarge = 8 * kPMaxCoef + (int)sizeof(PRound) * kPMaxRounds + 4 * kPMaxOps;
    if (!B.dense && 4 * B.words.size() <= kSmall)
        return B.h.t == kPTile
                   ? launch_pass<kSmall, false, true>(B, v, ntiles, grid, init, err, wait_limit, stall_tile, ppart, pscale, s)
                   : launch_pass<kSmall, false, false>(B, v, ntiles, grid, init, err, wait_limit, stall_tile, ppart, pscale, s);
    if (!B.dense && B.h.t == kPTile)
        return launch_pass<kLarge, false, true>(B, v, ntiles, grid, init, err, wait_limit, stall_tile, ppart, pscale, s);
    return launch_pass<kLarge, true, false>(B, v, ntiles, grid, init, err, wait_limit, stall_tile, ppart, pscale, s);
}

unsigned pauli_grid(const PauliHdr &h, int nsm)
{
    return std::min(1u << (2 * h.nod), (unsigned)nsm);
}

// ------------------------------------------------------------------ change of basis
// rho[r][c], c = r ^ x: 2^-n sum_z (-1)^{z.r} (-i)^{|x & z|} v_{x,z}.  With the signs u = s v
// (s = -1 where |x & z| mod 4 is 1 or 2) the terms with even |x & z| are real, the odd ones
// imaginary, and since flipping r by x changes the sign of exactly the odd ones, one real
// Walsh-Hadamard transform W_{x,r} = sum_z (-1)^{z.r} u_{x,z} holds both parts:
//   2^n rho[r][r ^ x] = (W_{x,r} + W_{x,r^x}) / 2 + i (W_{x,r} - W_{x,r^x}) / 2.
// Conversely W = 2^n (Re + Im) rho[r][r ^ x] and v = s 2^-n WHT(W).  The transform is separable over
// the qubits: k_pauli_high runs it in place over the z bits of all but the seven lowest qubits,
// k_pauli_emit / k_pauli_absorb over those and between v and rho, in 16 KiB tiles: everything is
// real and each stage reads and writes its data once.
// Applied to a chunk (labels I, Z, X, Y of the lowest qubit, idx a multiple of 4): Y adds one.
template <typename V>
__device__ __forceinline__ void p_signs4(V &a, uint64_t idx)
{
    const int k = __popcll(idx & (idx >> 1) & 0x5555555555555555ull);
    if ((k + 1) & 2) a.x = -a.x, a.y = -a.y, a.z = -a.z;
    if ((k + 2) & 2) a.w = -a.w;
}

// Bits of v to the even positions.
__device__ __forceinline__ uint64_t p_spread(unsigned v)
{
    uint64_t x = v;
    x = (x | (x << 16)) & 0x0000FFFF0000FFFFull;
    x = (x | (x << 8)) & 0x00FF00FF00FF00FFull;
    x = (x | (x << 4)) & 0x0F0F0F0F0F0F0F0Full;
    x = (x | (x << 2)) & 0x3333333333333333ull;
    x = (x | (x << 1)) & 0x5555555555555555ull;
    return x;
}

template <int NB, typename T, typename F, typename G>
__device__ __forceinline__ void p_wht(F ld, G st)
{
    T e[1 << NB];
#pragma unroll
    for (int j = 0; j < (1 << NB); j++) e[j] = ld(j);
#pragma unroll
    for (int b = 0; b < NB; b++)
#pragma unroll
        for (int j = 0; j < (1 << NB); j++)
            if (!(j & (1 << b))) {
                const T a = e[j], c = e[j | (1 << b)];
                e[j] = a + c;
                e[j | (1 << b)] = a - c;
            }
#pragma unroll
    for (int j = 0; j < (1 << NB); j++) st(j, e[j]);
}

struct alignas(16) F4 {
    float x, y, z, w;
};
__device__ __forceinline__ F4 operator+(F4 a, F4 b) { return F4{a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w}; }
__device__ __forceinline__ F4 operator-(F4 a, F4 b) { return F4{a.x - b.x, a.y - b.y, a.z - b.z, a.w - b.w}; }

constexpr int kCvLow = 7;  // qubits transformed by the emit / absorb stage

// In place over the z bits of the `hi` high qubits.  A CTA owns one x of them and a run of 4 * 2^rb
// low elements: 2^hi rows of that run, 2048 chunks (4096 at hi = 10) in shared memory.  A thread
// loads 16 chunks and transforms them in registers (the top row bits), then the rest takes one trip
// through shared memory (two from hi = 8 up).  Bound by HBM if the integer work per chunk is small,
// hence the offsets split into a thread's and a chunk number's part: n = 14 (2.15 GB) 0.57 ms with
// the general index arithmetic for every chunk and radix-8 steps all through shared memory.
constexpr int kHiThreads = 128;
__global__ void __launch_bounds__(kHiThreads) k_pauli_high(float *__restrict__ v, int hi, int low, int rb, int sign_in,
                                                           int sign_out)
{
    extern __shared__ __align__(16) unsigned char smem[];
    F4 *sm = reinterpret_cast<F4 *>(smem);
    const unsigned nrun = 1u << (2 * low - 2 - rb);  // runs of a row
    const unsigned run = blockIdx.x % nrun, xa = blockIdx.x / nrun, rmask = (1u << rb) - 1u;
    const int ebits = hi + rb;                       // chunk index e: row above rb bits of the run
    const uint64_t xo = p_spread(xa) << (2 * low + 1);
    auto at = [&](unsigned e) {
        return xo + (p_spread(e >> rb) << (2 * low)) + 4ull * (((uint64_t)run << rb) + (e & rmask));
    };
    auto low_count = [&](unsigned e) {  // |x & z| of the low qubits
        const unsigned l = 4u * ((run << rb) + (e & rmask));
        return __popc(l & (l >> 1) & 0x55555555u);
    };
    auto signs = [&](F4 &a, unsigned k) {
        if ((k + 1) & 2) a.x = -a.x, a.y = -a.y, a.z = -a.z;
        if ((k + 2) & 2) a.w = -a.w;
    };
    const int top = hi < 4 ? hi : 4;  // row bits among the four highest bits of e
    for (unsigned b0 = 0; b0 < (1u << (ebits - 11)); b0++) {
        // chunks e = u 2^(ebits - 4) + b0 128 + tid
        const unsigned e0 = b0 * kHiThreads + threadIdx.x;
        const int us = ebits - 4 - rb;  // u shifts the row by this (hi >= 4), else the run and the row
        const uint64_t g0 = at(e0);
        const unsigned k0 = low_count(e0) + __popc(xa & (e0 >> rb));
        F4 a[16];
        if (hi >= 4) {
            const uint64_t step = 1ull << (2 * us + 2 * low);
#pragma unroll
            for (int u = 0; u < 16; u++)
                a[u] = *reinterpret_cast<const F4 *>(v + g0 + ((u & 1) + 4 * ((u >> 1) & 1) + 16 * ((u >> 2) & 1) + 64 * (u >> 3)) * step);
            if (sign_in) {
                const unsigned xu = xa >> us;
#pragma unroll
                for (int u = 0; u < 16; u++) signs(a[u], k0 + __popc(xu & u));
            }
        } else {
#pragma unroll
            for (int u = 0; u < 16; u++) {
                const unsigned e = ((unsigned)u << (ebits - 4)) + e0;
                a[u] = *reinterpret_cast<const F4 *>(v + at(e));
                if (sign_in) signs(a[u], low_count(e) + __popc(xa & (e >> rb)));
            }
        }
#pragma unroll
        for (int b = 3; b >= 0; b--)
            if (3 - b < top)
#pragma unroll
                for (int u = 0; u < 16; u++)
                    if (!(u & (1 << b))) {
                        const F4 x = a[u], y = a[u | (1 << b)];
                        a[u] = x + y;
                        a[u | (1 << b)] = x - y;
                    }
#pragma unroll
        for (int u = 0; u < 16; u++) sm[((unsigned)u << (ebits - 4)) + e0] = a[u];
    }
    __syncthreads();
    // the lower row bits: three at a time, the last three on the way out
    int rem = hi - top;
    for (; rem > 3; rem -= rem - 3 < 3 ? rem - 3 : 3) {
        const int nb = rem - 3 < 3 ? rem - 3 : 3, sh = rb + rem - nb;
        for (unsigned i = threadIdx.x; i < (1u << (ebits - nb)); i += kHiThreads) {
            const unsigned lo = i & ((1u << sh) - 1u), base = ((i >> sh) << (sh + nb)) | lo;
            auto ld = [&](int j) { return sm[base + ((unsigned)j << sh)]; };
            auto st = [&](int j, F4 x) { sm[base + ((unsigned)j << sh)] = x; };
            if (nb == 3) p_wht<3, F4>(ld, st);
            else if (nb == 2) p_wht<2, F4>(ld, st);
            else p_wht<1, F4>(ld, st);
        }
        __syncthreads();
    }
    auto out = [&](auto nbc) {
        constexpr int NB = decltype(nbc)::value;
        for (unsigned i = threadIdx.x; i < (1u << (ebits - NB)); i += kHiThreads) {
            const unsigned e0 = ((i >> rb) << (rb + NB)) | (i & rmask);
            const uint64_t g0 = at(e0);
            const unsigned k0 = sign_out ? low_count(e0) + __popc(xa & (e0 >> rb)) : 0u;
            auto ld = [&](int j) { return sm[e0 + ((unsigned)j << rb)]; };
            auto st = [&](int j, F4 x) {
                if (sign_out) signs(x, k0 + __popc(xa & j));
                *reinterpret_cast<F4 *>(v + g0 + ((uint64_t)((j & 1) + 4 * ((j >> 1) & 1) + 16 * (j >> 2)) << (2 * low))) = x;
            };
            p_wht<NB, F4>(ld, st);
        }
    };
    if (rem == 3) out(std::integral_constant<int, 3>());
    else if (rem == 2) out(std::integral_constant<int, 2>());
    else if (rem == 1) out(std::integral_constant<int, 1>());
    else out(std::integral_constant<int, 0>());
}

// The low stage on M = min(n, 7) qubits.  Tile: high qubits' labels (ra, ca) with ca <= ra (x = ra ^
// ca), one value xh of the x bits of the low qubits above the four lowest; it holds, for the two rows
// ra and ca of the transform, W over all z / r bits of the low qubits and all x bits of the ML lowest.
constexpr int kCvThreads = 256;
constexpr int kCvPitch = 17;  // floats per r_L (16 x values + 1)

template <int M>
struct CvTile {
    static constexpr int ML = M < 4 ? M : 4, MH = M - ML;
    static constexpr int kArray = (1 << M) * kCvPitch;            // floats of one of the two arrays
    static constexpr int kChunks = 1 << (MH + 2 * ML - 2);        // 4-element chunks of one array
    static constexpr int kPairs = 1 << (M + ML - 1);              // element pairs of one block of rho
    static constexpr int U = (kChunks + kCvThreads - 1) / kCvThreads, UP = (kPairs + kCvThreads - 1) / kCvThreads;
    unsigned ra, ca, xh;
    int narr;
    uint64_t off[2];  // element offset of the arrays' low part in v
    unsigned pos0;    // this thread's first chunk: position in an array (labels I, Z, X, Y: + 0, pitch, 1, pitch + 1)
    unsigned loff0;   // and element offset in v's low part; chunk + u 256 adds cpos(u), coff(u)

    // Tile blk of all pairs ca <= ra.
    __device__ __forceinline__ explicit CvTile(unsigned blk)
    {
        const unsigned long long p = blk >> MH;
        unsigned long long c = (unsigned long long)((sqrtf(8.0f * (float)p + 1.0f) - 1.0f) * 0.5f);
        while ((c + 1) * (c + 2) / 2 <= p) c++;
        while (c * (c + 1) / 2 > p) c--;
        init((unsigned)c, (unsigned)(p - c * (c + 1) / 2), blk & ((1u << MH) - 1u));
    }
    // Tile blk of the pairs that hold row block r.
    __device__ __forceinline__ CvTile(unsigned blk, unsigned r)
    {
        const unsigned c = blk >> MH;
        init(r > c ? r : c, r > c ? c : r, blk & ((1u << MH) - 1u));
    }
    __device__ __forceinline__ void init(unsigned r, unsigned c, unsigned x_high)
    {
        ra = r, ca = c, xh = x_high;
        narr = ra == ca ? 1 : 2;
        const uint64_t x = p_spread(ra ^ ca) << 1;
        off[0] = (x | p_spread(ra)) << (2 * M);
        off[1] = (x | p_spread(ca)) << (2 * M);
        const unsigned k = threadIdx.x & (kChunks - 1), lowc = k & ((1u << (2 * ML - 2)) - 1u), zh = k >> (2 * ML - 2);
        loff0 = (((unsigned)p_spread(zh) | ((unsigned)p_spread(xh) << 1)) << (2 * ML)) + 4u * lowc;
        unsigned z = 0, xx = 0;
#pragma unroll
        for (int d = 0; d < ML - 1; d++) {
            z |= ((lowc >> (2 * d)) & 1u) << (d + 1);
            xx |= ((lowc >> (2 * d + 1)) & 1u) << (d + 1);
        }
        pos0 = ((zh << ML) | z) * kCvPitch + xx;
    }
    // u-th chunk of this thread (U = 2: the second half of the z bits above)
    static __device__ __forceinline__ unsigned cpos(int u) { return u * (((256u >> (2 * ML - 2)) << ML) * kCvPitch); }
    static __device__ __forceinline__ unsigned coff(int u) { return u * ((16u) << (2 * ML)); }
    __device__ __forceinline__ bool has(int u) const { return threadIdx.x + u * kCvThreads < kChunks; }
};

// WHT over the z bits of the low qubits, both arrays.
template <int M>
__device__ __forceinline__ void cv_transform(const CvTile<M> &T, float *sm)
{
    constexpr int ML = CvTile<M>::ML;
    auto step = [&](auto bc, auto nbc) {
        constexpr int B = decltype(bc)::value, NB = decltype(nbc)::value;
        constexpr unsigned per = 1u << (M - NB + ML);
        for (unsigned i = threadIdx.x; i < per * (unsigned)T.narr; i += kCvThreads) {
            const unsigned a = i / per, k = i % per, xl = k & ((1u << ML) - 1u), q = k >> ML;
            const unsigned z0 = ((q >> B) << (B + NB)) | (q & ((1u << B) - 1u));
            float *p = sm + a * CvTile<M>::kArray + z0 * kCvPitch + xl;
            constexpr unsigned stp = (unsigned)kCvPitch << B;
            auto ld = [&](int j) { return p[j * stp]; };
            auto st = [&](int j, float x) { p[j * stp] = x; };
            p_wht<NB, float>(ld, st);
        }
        __syncthreads();
    };
    step(std::integral_constant<int, 0>(), std::integral_constant<int, ML>());
    if constexpr (M > 4) step(std::integral_constant<int, 4>(), std::integral_constant<int, M - 4>());
}

// ROWS: only the blocks of row block r0 + blockIdx.y, from rho on; else all of rho.
template <int M, bool ROWS>
__global__ void __launch_bounds__(kCvThreads)
    k_pauli_emit(const float *__restrict__ v, float2 *__restrict__ rho, int n, float scale, int sign, unsigned r0)
{
    using C = CvTile<M>;
    constexpr int ML = C::ML;
    __shared__ float sm[2 * C::kArray];
    const unsigned row_block = r0 + blockIdx.y;
    const C T = ROWS ? C(blockIdx.x, row_block) : C(blockIdx.x);
    const float h = 0.5f * scale;
    {
        float4 x[2][C::U];  // all loads in flight
#pragma unroll
        for (int a = 0; a < 2; a++)
#pragma unroll
            for (int u = 0; u < C::U; u++)
                if (a < T.narr && T.has(u)) x[a][u] = *reinterpret_cast<const float4 *>(v + T.off[a] + T.loff0 + C::coff(u));
#pragma unroll
        for (int a = 0; a < 2; a++)
#pragma unroll
            for (int u = 0; u < C::U; u++)
                if (a < T.narr && T.has(u)) {
                    float4 y = x[a][u];
                    if (sign) p_signs4(y, T.off[a] + T.loff0 + C::coff(u));
                    float *p = sm + a * C::kArray + T.pos0 + C::cpos(u);
                    p[0] = h * y.x, p[kCvPitch] = h * y.y, p[1] = h * y.z, p[kCvPitch + 1] = h * y.w;
                }
    }
    __syncthreads();
    cv_transform<M>(T, sm);
    // block (ra, ca), then its mirror (ca, ra): rows in turn, two columns per thread; the x bits
    // row ^ column of a thread's elements are the same in all its rows
    constexpr unsigned half = 1u << (ML - 1), lmask = (1u << ML) - 1u, rstep = kCvThreads / half;
    const unsigned row0 = threadIdx.x / half, c0 = 2 * (threadIdx.x % half);
    const unsigned x0 = (row0 & lmask) ^ c0, x1 = x0 ^ 1u;
    const uint64_t dim = 1ull << n;
#pragma unroll
    for (int blkm = 0; blkm < 2; blkm++) {
        if (blkm == T.narr) break;
        if (ROWS && row_block != (blkm ? T.ca : T.ra)) continue;
        const float *wr = blkm ? sm + C::kArray : sm, *wc = T.narr == 2 && !blkm ? sm + C::kArray : sm;  // by row, by column
        const unsigned rb = ROWS ? blockIdx.y : blkm ? T.ca : T.ra;
        float2 *dst = rho + (((uint64_t)rb << M) + row0) * dim + ((uint64_t)(blkm ? T.ra : T.ca) << M) + c0;
        wr += row0 * kCvPitch;
        wc += c0 * kCvPitch;
#pragma unroll
        for (int u = 0; u < C::UP; u++) {
            const unsigned row = row0 + u * rstep;
            if (row >= (1u << M)) break;
            const unsigned colh = ((row >> ML) ^ T.xh) << ML;
            const float A0 = wr[u * rstep * kCvPitch + x0], A1 = wr[u * rstep * kCvPitch + x1];
            const float B0 = wc[colh * kCvPitch + x0], B1 = wc[(colh + 1) * kCvPitch + x1];
            // the imaginary part is (W at the row - W at the column) in block and mirror alike
            *reinterpret_cast<float4 *>(dst + u * rstep * dim + colh) = make_float4(A0 + B0, A0 - B0, A1 + B1, A1 - B1);
        }
    }
}

// The lower triangle of rho (r >= c; the diagonal's real part) -> W, transformed over the low qubits.
__global__ void __launch_bounds__(kCvThreads) k_pauli_absorb(const float2 *__restrict__ rho, float *__restrict__ v, int n)
{
    constexpr int M = kCvLow;
    using C = CvTile<M>;
    constexpr int ML = C::ML;
    __shared__ float sm[2 * C::kArray];
    const C T(blockIdx.x);
    constexpr unsigned half = 1u << (ML - 1), lmask = (1u << ML) - 1u, rstep = kCvThreads / half;
    const unsigned row0 = threadIdx.x / half, c0 = 2 * (threadIdx.x % half);
    const unsigned x0 = (row0 & lmask) ^ c0, x1 = x0 ^ 1u;
    const uint64_t dim = 1ull << n;
    const float2 *src = rho + (((uint64_t)T.ra << M) + row0) * dim + ((uint64_t)T.ca << M) + c0;
    const bool two = T.narr == 2;
    float *wr = sm + row0 * kCvPitch, *wc = (two ? sm + C::kArray : sm) + c0 * kCvPitch;
    float4 in[C::UP];  // all loads in flight
#pragma unroll
    for (int u = 0; u < C::UP; u++) {
        const unsigned row = row0 + u * rstep, colh = ((row >> ML) ^ T.xh) << ML;
        if (row < (1u << M) && (two || row >= (colh | c0))) in[u] = *reinterpret_cast<const float4 *>(src + u * rstep * dim + colh);
    }
#pragma unroll
    for (int u = 0; u < C::UP; u++) {
        const unsigned row = row0 + u * rstep, colh = ((row >> ML) ^ T.xh) << ML, col = colh | c0;
        if (row >= (1u << M) || (!two && row < col)) continue;
        const float4 x = in[u];
        if (!two && row == col) {
            wr[u * rstep * kCvPitch + x0] = x.x;
            continue;  // column c0 + 1 lies above the diagonal
        }
        wr[u * rstep * kCvPitch + x0] = x.x + x.y;
        wc[colh * kCvPitch + x0] = x.x - x.y;
        if (!two && row == col + 1) {
            wr[u * rstep * kCvPitch + x1] = x.z;
            continue;
        }
        wr[u * rstep * kCvPitch + x1] = x.z + x.w;
        wc[(colh + 1) * kCvPitch + x1] = x.z - x.w;
    }
    __syncthreads();
    cv_transform<M>(T, sm);
#pragma unroll
    for (int a = 0; a < 2; a++)
#pragma unroll
        for (int u = 0; u < C::U; u++)
            if (a < T.narr && T.has(u)) {
                const float *p = sm + a * C::kArray + T.pos0 + C::cpos(u);
                *reinterpret_cast<float4 *>(v + T.off[a] + T.loff0 + C::coff(u)) =
                    make_float4(p[0], p[kCvPitch], p[1], p[kCvPitch + 1]);
            }
}

static cudaError_t launch_high(float *v, int n, int sign_in, int sign_out, cudaStream_t s)
{
    const int hi = n - kCvLow, low = kCvLow;
    const int rb = std::max(2, 11 - hi);  // runs of 64 bytes and more
    const size_t sm = sizeof(F4) << (hi + rb);
    if (ensure_smem_attr(reinterpret_cast<const void *>(k_pauli_high), sm)) return cudaErrorInvalidValue;
    const unsigned blocks = 1u << (hi + 2 * low - 2 - rb);
    k_pauli_high<<<blocks, kHiThreads, sm, s>>>(v, hi, low, rb, sign_in, sign_out);
    return cudaGetLastError();
}

static unsigned cv_blocks(int n)
{
    const int m = std::min(n, kCvLow), mh = m - std::min(m, 4);
    const unsigned long long M = 1ull << (n - m);
    return (unsigned)((M * (M + 1) / 2) << mh);
}

int pauli_convert_launches(int n) { return n > kCvLow ? 2 : 1; }

cudaError_t launch_pauli_unfold(float *v, int n, cudaStream_t s) { return n > kCvLow ? launch_high(v, n, 1, 0, s) : cudaSuccess; }

template <int M, bool ROWS>
static void emit_m(const float *v, float2 *rho, int n, int r0, int nr, cudaStream_t s)
{
    float scale = 1.f;
    for (int i = 0; i < n; i++) scale *= 0.5f;
    const dim3 grid = ROWS ? dim3(1u << (n - M + CvTile<M>::MH), nr) : dim3(cv_blocks(n));
    k_pauli_emit<M, ROWS><<<grid, kCvThreads, 0, s>>>(v, rho, n, scale, n > kCvLow ? 0 : 1, (unsigned)r0);
}

template <bool ROWS>
static cudaError_t emit(const float *v, float2 *rho, int n, int r0, int nr, cudaStream_t s)
{
    switch (n) {
    case 3: emit_m<3, ROWS>(v, rho, n, r0, nr, s); break;
    case 4: emit_m<4, ROWS>(v, rho, n, r0, nr, s); break;
    case 5: emit_m<5, ROWS>(v, rho, n, r0, nr, s); break;
    case 6: emit_m<6, ROWS>(v, rho, n, r0, nr, s); break;
    default: emit_m<kCvLow, ROWS>(v, rho, n, r0, nr, s); break;
    }
    return cudaGetLastError();
}

// rho <- v (v is used up: the high stage works in place).  n >= 3.
cudaError_t launch_pauli_to_rho(float *v, float2 *rho, int n, cudaStream_t s)
{
    const cudaError_t e = launch_pauli_unfold(v, n, s);
    return e != cudaSuccess ? e : emit<false>(v, rho, n, 0, 0, s);
}

int pauli_row_block(int n) { return 1 << std::min(n, kCvLow); }

cudaError_t launch_pauli_rows(const float *v, float2 *rows, int n, int row, int count, cudaStream_t s)
{
    const int block = pauli_row_block(n);
    return emit<true>(v, rows, n, row / block, count / block, s);
}

// v <- rho, from its lower triangle.  n > kCvLow (a state of fewer qubits held as rho stays there).
cudaError_t launch_rho_to_pauli(const float2 *rho, float *v, int n, cudaStream_t s)
{
    k_pauli_absorb<<<cv_blocks(n), kCvThreads, 0, s>>>(rho, v, n);
    const cudaError_t e = cudaGetLastError();
    return e != cudaSuccess ? e : launch_high(v, n, 0, 1, s);
}

// ------------------------------------------------------------------ readouts
__global__ void k_pauli_zero(float4 *__restrict__ v, uint64_t nchunk)
{
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < nchunk; i += (uint64_t)gridDim.x * blockDim.x)
        v[i] = (i & 0xAAAAAAAAAAAAAAAAull) == 0 ? make_float4(1.f, 1.f, 0.f, 0.f) : make_float4(0.f, 0.f, 0.f, 0.f);
}

cudaError_t launch_pauli_zero(float *v, int n, int nsm, cudaStream_t s)
{
    const uint64_t nchunk = 1ull << (2 * n - 2);
    const uint64_t g = (nchunk + 255) / 256, cap = (uint64_t)nsm * 32;
    k_pauli_zero<<<(unsigned)(g < cap ? g : cap), 256, 0, s>>>(reinterpret_cast<float4 *>(v), nchunk);
    return cudaGetLastError();
}

// out[0], out[1] = trace; out[2 + q] = P(qubit q = 1) = (v_I - v_{Z_q}) / 2.
__global__ void k_pauli_diag(const float *__restrict__ v, int n, double *__restrict__ out)
{
    const int q = threadIdx.x;
    const double v0 = v[0];
    if (q == 0) out[0] = v0, out[1] = 0.0;
    if (q < n) out[2 + q] = 0.5 * (v0 - (double)v[1ull << (2 * (n - 1 - q))]);
}

void launch_pauli_diag(const float *v, int n, double *out, cudaStream_t s) { k_pauli_diag<<<1, 32, 0, s>>>(v, n, out); }

// out[s] = Tr[P_s rho]: the string's own coefficient.
__global__ void k_pauli_terms(const float *__restrict__ v, const __grid_constant__ PauliTerms T, double *__restrict__ out)
{
    const int s = threadIdx.x;
    if (s < T.count) out[s] = v[(p_spread(T.flip[s]) << 1) | p_spread(T.ym[s] | T.zm[s])];
}

void launch_pauli_terms(const float *v, const PauliTerms &T, double *out, cudaStream_t s)
{
    k_pauli_terms<<<1, 64, 0, s>>>(v, T, out);
}

// Projection on outcome m of a qubit, times scale: (I, Z, X, Y) -> ((I + s Z) / 2, s (I + s Z) / 2, 0, 0).
__global__ void k_pauli_project(float *__restrict__ v, uint64_t items, int d, float sgn, float h)
{
    float4 *v4 = reinterpret_cast<float4 *>(v);
    const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < items; i += (uint64_t)gridDim.x * blockDim.x) {
        if (d == 0) {
            const float4 x = v4[i];
            const float a = h * fmaf(sgn, x.y, x.x);
            v4[i] = make_float4(a, sgn * a, 0.f, 0.f);
        } else {
            const int sh = 2 * (d - 1);
            const uint64_t b = ((i >> sh) << (sh + 2)) | (i & ((1ull << sh) - 1)), st = 1ull << sh;
            const float4 x = v4[b], z = v4[b + st];
            const float4 a = make_float4(h * fmaf(sgn, z.x, x.x), h * fmaf(sgn, z.y, x.y), h * fmaf(sgn, z.z, x.z),
                                         h * fmaf(sgn, z.w, x.w));
            v4[b] = a;
            v4[b + st] = make_float4(sgn * a.x, sgn * a.y, sgn * a.z, sgn * a.w);
            v4[b + 2 * st] = zero;
            v4[b + 3 * st] = zero;
        }
    }
}

void launch_pauli_project(float *v, int n, int qubit, int m, double scale, int nsm, cudaStream_t s)
{
    const int d = n - 1 - qubit;
    const uint64_t items = d == 0 ? 1ull << (2 * n - 2) : 1ull << (2 * n - 4);
    const uint64_t g = (items + 255) / 256, cap = (uint64_t)nsm * 32;
    k_pauli_project<<<(unsigned)(g < cap ? g : cap), 256, 0, s>>>(v, items, d, m ? -1.f : 1.f, (float)(0.5 * scale));
}

// Purity 2^-n sum v^2: squares in FP32 over 16 elements, totals in FP64, fixed tree.
constexpr int kPpThreads = 256;
__global__ void __launch_bounds__(kPpThreads) k_pauli_purity(const float4 *__restrict__ v, uint64_t n4, double scale,
                                                             double *__restrict__ part)
{
    double acc = 0;
    const uint64_t stride = (uint64_t)gridDim.x * kPpThreads;
    for (uint64_t i = blockIdx.x * (uint64_t)kPpThreads + threadIdx.x; i < n4; i += 4 * stride) {
        float s = 0.f;
#pragma unroll
        for (int u = 0; u < 4; u++)
            if (i + u * stride < n4) {
                const float4 a = v[i + u * stride];
                s = fmaf(a.x, a.x, fmaf(a.y, a.y, fmaf(a.z, a.z, fmaf(a.w, a.w, s))));
            }
        acc += (double)s;
    }
    __shared__ double sh[kPpThreads / 32];
    acc = warp_sum(acc);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0;
        for (int w = 0; w < kPpThreads / 32; w++) t += sh[w];
        part[blockIdx.x] = t * scale;
    }
}

int launch_pauli_purity(const float *v, int n, double *partials, double *out, int nblocks, cudaStream_t s)
{
    const uint64_t n4 = 1ull << (2 * n - 2), need = (n4 + 4 * kPpThreads - 1) / (4 * kPpThreads);
    const int nb = (int)(need < (uint64_t)nblocks ? need : (uint64_t)nblocks);
    double scale = 1.0;
    for (int i = 0; i < n; i++) scale *= 0.5;
    k_pauli_purity<<<nb, kPpThreads, 0, s>>>(reinterpret_cast<const float4 *>(v), n4, scale, nb == 1 ? out : partials);
    if (nb > 1) launch_fold(partials, nb, out, s);
    return nb > 1 ? 2 : 1;
}

// Reduced state of the kept qubits (k <= 6): their strings' coefficients, changed to rho_A in FP64.
__global__ void __launch_bounds__(256) k_pauli_ptrace(const float *__restrict__ v, PTParams p, double2 *__restrict__ out)
{
    __shared__ double w[4096];
    const int k = p.nkeep;
    const unsigned N = 1u << (2 * k), dim = 1u << k;
    for (unsigned e = threadIdx.x; e < N; e += 256) {  // e = x * dim + z
        const unsigned x = e >> k, z = e & (dim - 1);
        uint64_t idx = 0;
        for (int j = 0; j < k; j++)
            idx |= ((uint64_t)((x >> (k - 1 - j)) & 1u) << (2 * p.kpos[j] + 1)) |
                   ((uint64_t)((z >> (k - 1 - j)) & 1u) << (2 * p.kpos[j]));
        const int c = __popc(x & z);
        w[e] = ((c + 1) & 2) ? -(double)v[idx] : (double)v[idx];
    }
    __syncthreads();
    for (int b = 0; b < k; b++) {
        for (unsigned i = threadIdx.x; i < N / 2; i += 256) {
            const unsigned e = ((i >> b) << (b + 1)) | (i & ((1u << b) - 1u));
            const double a = w[e], c = w[e | (1u << b)];
            w[e] = a + c;
            w[e | (1u << b)] = a - c;
        }
        __syncthreads();
    }
    const double h = 0.5 / (double)dim;
    for (unsigned e = threadIdx.x; e < N; e += 256) {
        const unsigned r = e >> k, c = e & (dim - 1), x = r ^ c;
        const double a = w[x * dim + r], b = w[x * dim + c];
        out[e] = make_double2(h * (a + b), h * (a - b));
    }
}

void launch_pauli_ptrace(const float *v, const PTParams &p, double2 *out, cudaStream_t s)
{
    k_pauli_ptrace<<<1, 256, 0, s>>>(v, p, out);
}

}  // namespace qcw
