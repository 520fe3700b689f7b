// Persistent work-item kernel shared by the batched runner and the serving loop, and the
// host code that turns circuits into programs and programs into work items.
//
// Every CTA repeatedly takes the next item from a global counter.  Items are listed in an
// order where an item's dependency (the previous pass of the same circuit) always comes
// earlier in the list, so a CTA only ever waits for items that running CTAs already hold;
// every wait is bounded (spin_limit polls) and a wait that runs out sets *err instead of
// hanging.  States are kept as Pauli coefficients (pauli.h) from |0..0> to the readouts, which are
// coefficients themselves (trace, probabilities) or their sum of squares (purity).  A circuit
// whose state fits one tile (up to seven qubits) is one item: it starts, runs through every round
// and is read out in shared memory.  Larger circuits are split into one item per tile and pass,
// chained by per-pass counters, followed by readout chunks.  Each circuit is processed by a fixed
// item decomposition with a fixed thread-to-data mapping, so its result does not depend on what
// else is in the batch.
//
// Two CTAs per SM (64 KiB tile and the pass's program each) overlap one's loads with the other's
// rounds.  64 circuits of 4 to 10 qubits, 50 to 400 gates deep: 0.40 ms per launch (on complex tiles
// without symmetry 1.01 ms); the passes of the deepest ten-qubit circuit, one after the other, are the
// longest chain.
#include <algorithm>
#include <cstring>

#include "engine.h"
#include "pauli.cuh"
#include "qcw_internal.h"

namespace qcw {

constexpr int kEngThreads = 256;

__device__ __forceinline__ unsigned ld_acquire(const unsigned *p)
{
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];\n" : "=r"(v) : "l"(p) : "memory");
    return v;
}

using RedShared = double[kEngThreads / 32][kRedVals];

// Fold per-thread accumulators (first nv used) into out[0..nv) with a fixed tree.
__device__ __forceinline__ void red_store(double (&acc)[kRedVals], int nv, double *out, RedShared &sh)
{
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
    for (int v = 0; v < kRedVals; v++) {
        if (v < nv) {
            double s = warp_sum(acc[v]);
            if (lane == 0) sh[w][v] = s;
        }
    }
    __syncthreads();
    if ((int)threadIdx.x < nv) {
        double t = 0;
        for (int j = 0; j < kEngThreads / 32; j++) t += sh[j][threadIdx.x];
        out[threadIdx.x] = t;
    }
    __syncthreads();
}

// Shared memory of an item: the tile, then the pass's program (rounds, operations, coefficient pairs).
struct EngSmem {
    unsigned char *base;
    __device__ __forceinline__ float4 *tile() const { return reinterpret_cast<float4 *>(base); }
    __device__ __forceinline__ unsigned *prog(int t) const { return reinterpret_cast<unsigned *>(base + (sizeof(float) << (2 * t))); }
};

// Bring a pass's program to shared memory.
__device__ __forceinline__ ProgShared eng_stage(const PassDesc &D, const EngSmem &sm)
{
    const int nr = D.h.nround * (int)(sizeof(PRound) / 4), no = (D.h.nop + 3) & ~3;
    const unsigned *src = reinterpret_cast<const unsigned *>(&D + 1);
    unsigned *dst = sm.prog(D.h.t);
    for (int i = threadIdx.x; i < nr + no; i += kEngThreads) dst[i] = src[i];
    for (int i = threadIdx.x; i < D.h.ncoef; i += kEngThreads) dst[nr + no + 2 * i] = dst[nr + no + 2 * i + 1] = src[nr + no + i];
    const PRound *r = reinterpret_cast<const PRound *>(dst);
    return ProgShared{r, reinterpret_cast<const POp *>(dst + nr), smem_u32(dst + nr + no)};
}

// The product state a program starts from (PauliPlan::w).
__device__ __forceinline__ void eng_init(const EngSmem &sm, const PauliHdr &h, unsigned tile)
{
    const float f0 = p_factor(h.w, h.od, h.nod, tile);
    for (unsigned k = threadIdx.x; k < (1u << (2 * (h.t - 1))); k += kEngThreads) {
        const float f = f0 * p_factor(h.w, h.td + 1, h.t - 1, k);
        sm.tile()[pauli_swz(k)] = make_float4(f * h.w[0], f * h.w[1], f * h.w[2], f * h.w[3]);
    }
}

__device__ __forceinline__ uint64_t eng_base(const PauliHdr &h, unsigned tile)
{
    uint64_t b = 0;
    for (int d = 0; d < h.nod; d++) b += (uint64_t)((tile >> (2 * d)) & 3u) << (2 * h.od[d]);
    return b;
}

__device__ __forceinline__ uint64_t eng_chunk(const PauliHdr &h, unsigned k)
{
    uint64_t b = 0;
    for (int d = 1; d < h.t; d++) b += (uint64_t)((k >> (2 * (d - 1))) & 3u) << (2 * h.td[d]);
    return b;
}

// Out of line: the rounds need nearly all 128 registers, so nothing of the item loop lives across them.
template <bool DENSE, bool FULL>
__device__ __noinline__ void eng_rounds(unsigned tile, const PRound *rounds, int nround, const POp *ops, unsigned coef)
{
    const ProgShared prog{rounds, ops, coef};
    pauli_rounds<DENSE>(tile, rounds, nround, prog, threadIdx.x, 0, KeepTile<FULL>());
}

template <bool DENSE>
__device__ __forceinline__ void eng_evolve(const PauliHdr &h, const EngSmem &sm, const ProgShared &prog)
{
    if (h.t == kPTile) eng_rounds<DENSE, true>(smem_u32(sm.base), prog.rounds, h.nround, prog.ops, prog.coef);
    else eng_rounds<DENSE, false>(smem_u32(sm.base), prog.rounds, h.nround, prog.ops, prog.coef);
}

template <bool DENSE>
__device__ void run_tile(const WItem &W, const EngSmem &sm)
{
    const PassDesc &D = *reinterpret_cast<const PassDesc *>(W.pass);
    const unsigned nch = 1u << (2 * (D.h.t - 1));
    float *g = W.v + eng_base(D.h, W.tile);
    if (W.flags & WF_INIT) {
        eng_init(sm, D.h, W.tile);
    } else {
        for (unsigned k = threadIdx.x; k < nch; k += kEngThreads) cp_async16(sm.tile() + pauli_swz(k), g + eng_chunk(D.h, k));
    }
    const ProgShared prog = eng_stage(D, sm);
    cp_async_wait_all();
    __syncthreads();
    eng_evolve<DENSE>(D.h, sm, prog);
    for (unsigned k = threadIdx.x; k < nch; k += kEngThreads)
        *reinterpret_cast<float4 *>(g + eng_chunk(D.h, k)) = p_lds4(smem_u32(sm.base) + 16u * pauli_swz(k));
}

// Trace (2 values), purity and P(q = 1): v0 and vz(q), the strings I..I and Z_q, by thread; s the
// thread's share of the sum of squares.
template <typename F>
__device__ __forceinline__ void eng_readout(double s, bool first, int n, float v0, F vz, double *out, RedShared &sh)
{
    double acc[kRedVals];
#pragma unroll
    for (int i = 0; i < kRedVals; i++) acc[i] = 0;
    const int nd = n < kPMinDigits ? kPMinDigits : n;
    double scale = 1.0;
    for (int i = 0; i < nd; i++) scale *= 0.5;
    acc[2] = s * scale;
    if (first) {
        if (threadIdx.x == 0) acc[0] = v0;
#pragma unroll
        for (int q = 0; q < QCW_MAX_QUBITS; q++)
            if (q < n && (int)threadIdx.x == q) acc[3 + q] = 0.5 * ((double)v0 - (double)vz(q));
    }
    red_store(acc, n + 3, out, sh);
}

__device__ __forceinline__ float sq4(float4 a, float s)
{
    return fmaf(a.x, a.x, fmaf(a.y, a.y, fmaf(a.z, a.z, fmaf(a.w, a.w, s))));
}

template <bool DENSE>
__device__ void run_whole(const WItem &W, const EngSmem &sm, RedShared &sh)
{
    const PauliHdr &h = reinterpret_cast<const PassDesc *>(W.pass)->h;
    const int t = h.t;
    const unsigned nch = 1u << (2 * (t - 1));
    eng_init(sm, h, 0);
    const char *p = W.pass;
    for (int i = 0; i < W.npass; i++) {
        const PassDesc &D = *reinterpret_cast<const PassDesc *>(p);
        const ProgShared prog = eng_stage(D, sm);
        __syncthreads();
        eng_evolve<DENSE>(D.h, sm, prog);
        __syncthreads();
        p += D.bytes;
    }
    double acc = 0;
    const float4 *tile = sm.tile();
    for (unsigned k = threadIdx.x; k < nch; k += kEngThreads) {
        const float4 x = tile[pauli_swz(k)];
        acc += (double)sq4(x, 0.f);
        *reinterpret_cast<float4 *>(W.v + 4 * (size_t)k) = x;
    }
    if (W.red) {
        auto vz = [&](int q) {
            const unsigned e = 1u << (2 * (W.n - 1 - q));
            return reinterpret_cast<const float *>(tile)[4 * pauli_swz(e >> 2) + (e & 3u)];
        };
        eng_readout(acc, true, W.n, reinterpret_cast<const float *>(tile)[0], vz, W.red, sh);
    }
}

__device__ void run_reduce(const WItem &W, RedShared &sh)
{
    double acc = 0;
    const float4 *v4 = reinterpret_cast<const float4 *>(W.v + W.e0);
    const unsigned long long n4 = W.ecount / 4;
    for (unsigned long long i = threadIdx.x; i < n4; i += 4 * kEngThreads) {
        float s = 0.f;
#pragma unroll
        for (int u = 0; u < 4; u++)
            if (i + u * kEngThreads < n4) s = sq4(__ldcg(v4 + i + u * kEngThreads), s);
        acc += (double)s;
    }
    auto vz = [&](int q) { return __ldcg(W.v + (1ull << (2 * (W.n - 1 - q)))); };
    eng_readout(acc, W.e0 == 0, W.n, __ldcg(W.v), vz, W.red, sh);
}

template <bool DENSE>
__global__ void __launch_bounds__(kEngThreads, 2) k_engine(EngineLaunch L)
{
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int s_item;
    __shared__ RedShared s_red;
    const int nitems = *L.nitems;
    for (;;) {
        if (threadIdx.x == 0) s_item = atomicAdd(L.next, 1);
        __syncthreads();
        const int it = s_item;
        __syncthreads();
        if (it >= nitems) return;
        const WItem W = L.items[it];
        if (W.dep) {
            if (threadIdx.x == 0) {
                long long spins = 0;
                while (ld_acquire(W.dep) < W.dep_target) {
                    if (++spins > L.spin_limit) {
                        atomicOr(L.err, 1);
                        break;
                    }
                    __nanosleep(128);
                }
            }
            __syncthreads();
        }
        const EngSmem sm{smem};
        if (W.kind == WI_TILES) run_tile<DENSE>(W, sm);
        else if (W.kind == WI_WHOLE) run_whole<DENSE>(W, sm, s_red);
        else run_reduce(W, s_red);
        __syncthreads();
        if (W.done && threadIdx.x == 0) {
            __threadfence();
            atomicAdd(W.done, 1u);
        }
    }
}

void engine_launch(const EngineLaunch &L, bool dense, int grid, size_t smem, cudaStream_t s)
{
    if (dense) k_engine<true><<<grid, kEngThreads, smem, s>>>(L);
    else k_engine<false><<<grid, kEngThreads, smem, s>>>(L);
}

qcw_status engine_prepare(int dev, bool dense, size_t smem, int *grid)
{
    const void *k = dense ? reinterpret_cast<const void *>(k_engine<true>) : reinterpret_cast<const void *>(k_engine<false>);
    qcw_status st = ensure_smem_attr(k, smem);
    if (st) return st;
    int occ = 0, nsm = 0;
    cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k, kEngThreads, smem);
    if (e != cudaSuccess) return cuda_error(e, "engine occupancy");
    e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return cuda_error(e, "SM count");
    if (occ < 1) return set_error(QCW_ENOTSUP, "engine kernel does not fit on an SM");
    *grid = occ * nsm;
    return QCW_OK;
}

// ------------------------------------------------------------------ host: programs
// Cost model (SM-seconds per coefficient), from the pass kernel at 14 qubits: 344 us for a pass's one
// read and one write of 2^28 coefficients on 152 SMs, 68 us per round with its operations.
static const double kCostPass = 0.195e-9;
static const double kCostRound = 0.038e-9;

static size_t pass_smem(int t, int nround, int nop, int ncoef)
{
    return (sizeof(float) << (2 * t)) + sizeof(PRound) * nround + 4 * (size_t)((nop + 3) & ~3) + sizeof(float2) * ncoef;
}

size_t engine_max_smem() { return pass_smem(kPTile, kPMaxRounds, kPMaxOps, kPMaxCoef); }

Program make_program(const qcw_op *ops, int nops, const double *matrices, int n, int fuse_k)
{
    Program p;
    PauliPlan plan = plan_pauli_list(ops, nops, matrices, n, fuse_k);
    p.n = n;
    p.whole = plan.nd <= kPTile;
    for (const PPass &ps : plan.passes) {
        PassDesc D;
        D.h = pauli_header(ps, plan.w);
        const size_t nr = sizeof(PRound) * ps.rounds.size(), no = 4 * (size_t)((ps.ops.size() + 3) & ~(size_t)3);
        const size_t nc = sizeof(float) * ((ps.coefs.size() + 3) & ~(size_t)3);
        D.bytes = (int)(sizeof D + nr + no + nc);
        const size_t at = p.desc.size();
        p.pass_off.push_back(at);
        p.desc.resize(at + D.bytes, 0);
        char *w = p.desc.data() + at;
        memcpy(w, &D, sizeof D);
        if (nr) memcpy(w + sizeof D, ps.rounds.data(), nr);
        if (!ps.ops.empty()) memcpy(w + sizeof D + nr, ps.ops.data(), sizeof(POp) * ps.ops.size());
        if (!ps.coefs.empty()) memcpy(w + sizeof D + nr + no, ps.coefs.data(), sizeof(float) * ps.coefs.size());
        p.tiles.push_back(1u << (2 * ps.od.size()));
        p.smem = std::max(p.smem, pass_smem(ps.t, (int)ps.rounds.size(), (int)ps.ops.size(), (int)ps.coefs.size()));
        p.dense |= pass_dense(ps);
        p.rounds += (long long)ps.rounds.size();
        p.cost += (double)program_elems(n) * (kCostPass + kCostRound * (double)ps.rounds.size());
    }
    return p;
}

void program_items(const Program &p, float *v, const char *desc, unsigned *counters, double *red, int pass_begin,
                   int pass_end, bool init, bool readout, std::vector<std::vector<WItem>> &levels, int *nchunks)
{
    const char *base = desc + p.off;
    *nchunks = 0;
    auto level = [&](size_t l) -> std::vector<WItem> & {
        if (levels.size() <= l) levels.resize(l + 1);
        return levels[l];
    };
    if (p.whole) {
        WItem w{};
        w.v = v;
        w.pass = base;
        w.npass = (int)p.tiles.size();
        w.kind = WI_WHOLE;
        w.n = p.n;
        w.red = readout ? red : nullptr;
        level(0).push_back(w);
        *nchunks = readout ? 1 : 0;
        return;
    }
    for (int ps = pass_begin; ps < pass_end; ps++) {
        for (unsigned t = 0; t < p.tiles[ps]; t++) {
            WItem w{};
            w.v = v;
            w.pass = base + p.pass_off[ps];
            w.tile = t;
            w.npass = 1;
            w.kind = WI_TILES;
            w.flags = (init && ps == 0) ? WF_INIT : 0;
            w.n = p.n;
            if (ps > pass_begin) {
                w.dep = counters + (ps - 1 - pass_begin);
                w.dep_target = p.tiles[ps - 1];
            }
            w.done = counters + (ps - pass_begin);
            level(ps - pass_begin).push_back(w);
        }
    }
    if (readout && pass_end == (int)p.tiles.size()) {
        const unsigned long long total = program_elems(p.n);
        int c = 0;
        for (unsigned long long e0 = 0; e0 < total; e0 += kReduceElems, c++) {
            WItem w{};
            w.v = v;
            w.kind = WI_REDUCE;
            w.n = p.n;
            w.red = red + (size_t)c * kRedVals;
            w.e0 = e0;
            w.ecount = std::min(kReduceElems, total - e0);
            if (pass_end > pass_begin) {
                w.dep = counters + (pass_end - 1 - pass_begin);
                w.dep_target = p.tiles[pass_end - 1];
            }
            level(pass_end - pass_begin).push_back(w);
        }
        *nchunks = c;
    }
}

// Rows of a piece: 2^17 elements (1 MiB), at least a row block (134 MB at 17 qubits).
constexpr size_t kPiece = (size_t)1 << 17;
static int stage_rows(int nd)
{
    return std::max(pauli_row_block(nd), (int)std::min<size_t>((size_t)1 << nd, kPiece >> nd));
}

size_t program_stage(int n)
{
    const int nd = std::max(n, kPMinDigits);
    return (size_t)stage_rows(nd) << nd;
}

size_t program_pinned(int n) { return std::min(program_elems(n), kPiece); }

bool program_copies(int n) { return n > kPTile; }

// Through a pinned buffer of at most 1 MiB, which the conversion to double finds in the cache: 12
// qubits (134 MB) 20 ms, 13 qubits 78 ms (copied whole to pageable memory 29 and 109 ms; as complex128
// from the device to the caller's pageable memory 43 and 107 ms).
cudaError_t program_rho(const float *v, int n, float *copy, float2 *stage, float2 *host, double *out, cudaStream_t s)
{
    const int nd = std::max(n, kPMinDigits), rows = stage_rows(nd);
    cudaError_t e = cudaSuccess;
    if (program_copies(n)) {
        e = cudaMemcpyAsync(copy, v, sizeof(float) * program_elems(n), cudaMemcpyDeviceToDevice, s);
        if (e == cudaSuccess) e = launch_pauli_unfold(copy, nd, s);
        v = copy;
    }
    const size_t dim = (size_t)1 << n, piece = program_pinned(n);
    for (size_t r = 0; r < dim && e == cudaSuccess; r += rows) {
        e = launch_pauli_rows(v, stage, nd, (int)r, rows, s);
        const size_t el = (size_t)rows << nd;
        for (size_t f = 0; f < el && e == cudaSuccess; f += piece) {
            const size_t cnt = std::min(piece, el - f);
            e = cudaMemcpyAsync(host, stage + f, sizeof(float2) * cnt, cudaMemcpyDeviceToHost, s);
            if (e == cudaSuccess) e = cudaStreamSynchronize(s);
            if (e != cudaSuccess) break;
            if (n == nd) {
                double *to = out + 2 * (r * dim + f);
                for (size_t i = 0; i < cnt; i++) to[2 * i] = host[i].x, to[2 * i + 1] = host[i].y;
                continue;
            }
            // a padded register's own qubits are the lowest: its rho is the corner where the others are |0>
            for (size_t i = 0; i < dim * dim; i++) {
                const float2 z = host[((i >> n) << nd) + (i & (dim - 1))];
                out[2 * i] = z.x, out[2 * i + 1] = z.y;
            }
        }
    }
    return e;
}

}  // namespace qcw
