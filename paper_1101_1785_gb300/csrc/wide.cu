// Dense operations on three to five qubits: rho <- sum_j K_j rho K_j^dagger (Eq. rhoE2; a gate is
// one K), both sides and the whole sum in one pass over rho.
//
// For every setting of the other qubits' row and column labels the operation acts on a d x d
// complex tile of rho, d = 2^k: T <- sum_j K_j T K_j^dagger.  A warp owns 32 / d tiles (neighbouring
// columns where the struck bits allow, so that its loads fill whole sectors) and a lane one column
// of a tile: Y = K T comes from the lane's own column with K broadcast from shared memory, Z = Y
// K^dagger takes the other lanes' columns of Y from shared memory and the lane's own row of K.
// Complex products run as two packed FMAs, (k_r, k_r) (x_r, x_i) and (k_i, k_i) (x_r, x_i) summed
// apart and combined once per output, 2 d per element and operator: the arithmetic bounds k = 4
// and 5 and channels of several operators, HBM a three-qubit gate.  Measured at 12 qubits (rho =
// 128 MiB) against two side passes and, per operator, a copy and an accumulation: five-qubit gate
// 395 -> 253 us, channel of three three-qubit operators 570 -> 178 us; the 17-operator channel on all
// of a 5-qubit register (one tile) 420 us -> 25 us with an operator per block.
#include "qcw_device.cuh"
#include "qcw_internal.h"
#include "tile.cuh"

namespace qcw {

constexpr int kWideThreads = 128;

template <int ENT>
struct WideParams {
    int nk;           // operators in m
    int pos[10];      // ascending struck bits of the flat index (row and column)
    int cbit[5], rbit[5];  // column / row bit of local bit j (bit 0 = the last listed qubit)
    const float2 *g;  // ENT = 0: the operators in device memory
    float2 m[ENT > 0 ? ENT : 1];    // operators one after another, row-major d x d
};

// Y's layout per warp: element (r, c) of a tile at c * wide_py + r (float2, rows in 16-byte pairs), the
// tiles wide_ty apart so that a read of one element per tile falls on different banks.
__host__ __device__ constexpr int wide_py(int k) { return (1 << k) + 2; }
__host__ __device__ constexpr int wide_ty(int k) { return (1 << k) * wide_py(k) + 4; }

// add: also add what it holds at the same places (may be out).  grid.y > 1: block row y runs operator y alone and writes its own
// copy out + y * 4^n (few tiles: the operators spread over the chip, k_wide_sum adds the copies).
// ALL: the operators of the launch stay in shared memory (48 of k = 3 take 54 KiB), so that the loop
// over them has no barriers and a tile's column is read once; else each operator is staged for each
// tile.  12 qubits, k = 3, staged / ALL: 3 operators 225 / 178 us, 8 540 / 391, 17 906 / 779, 48 2519 /
// 2405.  For k = 4 the columns kept cost 40 registers more and a quarter of the warps: 2 operators 239 /
// 258 us, 4 406 / 472; there and for k = 5 each operator is staged.
template <int K, int ENT, bool ALL>
__global__ void __launch_bounds__(kWideThreads) k_wide(const float2 *rho, float2 *out, const float2 *add,
                                                       uint64_t ntiles, uint64_t elems, const __grid_constant__ WideParams<ENT> p)
{
    constexpr int D = 1 << K, TP = 32 / D, PK = D + 1, PY = wide_py(K), RB = K == 5 ? 16 : 8;
    extern __shared__ __align__(16) unsigned char smem[];
    float4 *Ks = reinterpret_cast<float4 *>(smem);                      // (k_r, k_r, k_i, k_i), pitch PK
    float2 *Ys = reinterpret_cast<float2 *>(Ks + (ALL ? p.nk : 1) * D * PK);  // per warp TP tiles
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, c = lane & (D - 1), t = lane >> K;
    float2 *Y = Ys + (w * TP + t) * wide_ty(K);
    const int j0 = gridDim.y > 1 ? blockIdx.y : 0, j1 = gridDim.y > 1 ? j0 + 1 : p.nk;
    float2 *dst = out + (gridDim.y > 1 ? blockIdx.y * elems : 0);
    if constexpr (ALL) {
        for (int e = threadIdx.x; e < p.nk * D * D; e += kWideThreads) {
            const float2 m = p.m[e];
            Ks[(e >> K) * PK + (e & (D - 1))] = make_float4(m.x, m.x, m.y, m.y);
        }
        __syncthreads();
    }
    uint64_t coff = 0;
#pragma unroll
    for (int b = 0; b < K; b++) coff |= (uint64_t)((c >> b) & 1) << p.cbit[b];
    const uint64_t per = (uint64_t)(kWideThreads / 32) * TP;
    for (uint64_t first = blockIdx.x * per; first < ntiles; first += gridDim.x * per) {
        const uint64_t tile = first + w * TP + t;
        const bool on = tile < ntiles;
        uint64_t g = tile;
#pragma unroll
        for (int b = 0; b < 2 * K; b++) g = insert0(g, p.pos[b]);
        const float2 *src = rho + g + coff;
        auto roff = [&](int r) {
            uint64_t o = 0;
#pragma unroll
            for (int b = 0; b < K; b++) o |= (uint64_t)((r >> b) & 1) << p.rbit[b];
            return o;
        };
        float2 res[D];
#pragma unroll
        for (int r = 0; r < D; r++) res[r] = make_float2(0.f, 0.f);
        float2 x[D];
        if constexpr (ALL) {
#pragma unroll
            for (int r = 0; r < D; r++) x[r] = on ? src[roff(r)] : make_float2(0.f, 0.f);
        }
        for (int j = j0; j < j1; j++) {
            if constexpr (!ALL) {
                if (first != blockIdx.x * per || j != j0 || j1 - j0 > 1) __syncthreads();  // the last readers of Ks are done
                if (j1 - j0 > 1 || first == blockIdx.x * per)
                    for (int e = threadIdx.x; e < D * D; e += kWideThreads) {
                        const float2 m = ENT > 0 ? p.m[j * D * D + e] : p.g[j * D * D + e];
                        Ks[(e >> K) * PK + (e & (D - 1))] = make_float4(m.x, m.x, m.y, m.y);
                    }
#pragma unroll
                for (int r = 0; r < D; r++) x[r] = on ? src[roff(r)] : make_float2(0.f, 0.f);
                __syncthreads();
            }
            const float4 *Kj = Ks + (ALL ? j * D * PK : 0);
            if constexpr (K == 5 || ENT == 0) {  // Y = K T, K broadcast from shared memory
#pragma unroll 4
                for (int r = 0; r < D; r++) {
                    unsigned long long a = 0ull, b = 0ull;
#pragma unroll
                    for (int l = 0; l < D; l++) {
                        const ulonglong2 k = *reinterpret_cast<const ulonglong2 *>(Kj + r * PK + l);
                        const unsigned long long xl = pack2(x[l].x, x[l].y);
                        a = ffma2(k.x, xl, a);
                        b = ffma2(k.y, xl, b);
                    }
                    const float2 ya = unpack2(a), yb = unpack2(b);
                    Y[c * PY + r] = make_float2(ya.x - yb.y, ya.y + yb.x);
                }
            } else {  // small K: from the parameter block, which leaves shared memory to the second side
                const float2 *kj = p.m + j * D * D;
#pragma unroll 2
                for (int r = 0; r < D; r++) {
                    float2 y = make_float2(0.f, 0.f);
#pragma unroll
                    for (int l = 0; l < D; l++) cfma(y, kj[r * D + l], x[l]);
                    Y[c * PY + r] = y;
                }
            }
            __syncwarp();
#pragma unroll
            for (int rb = 0; rb < D; rb += RB) {  // column c of Z = Y K^dagger
                unsigned long long a[RB], b[RB];
#pragma unroll
                for (int i = 0; i < RB; i++) a[i] = b[i] = 0ull;
#pragma unroll 4
                for (int l = 0; l < D; l++) {
                    const ulonglong2 k = *reinterpret_cast<const ulonglong2 *>(Kj + c * PK + l);
#pragma unroll
                    for (int i = 0; i < RB; i += 2) {
                        const ulonglong2 y = *reinterpret_cast<const ulonglong2 *>(Y + l * PY + rb + i);
                        a[i] = ffma2(k.x, y.x, a[i]);
                        b[i] = ffma2(k.y, y.x, b[i]);
                        a[i + 1] = ffma2(k.x, y.y, a[i + 1]);
                        b[i + 1] = ffma2(k.y, y.y, b[i + 1]);
                    }
                }
#pragma unroll
                for (int i = 0; i < RB; i++) {
                    const float2 za = unpack2(a[i]), zb = unpack2(b[i]);
                    res[rb + i].x += za.x + zb.y;
                    res[rb + i].y += za.y - zb.x;
                }
            }
            __syncwarp();
        }
        if (on) {
            float2 *to = dst + g + coff;
#pragma unroll
            for (int r = 0; r < D; r++) {
                float2 v = res[r];
                if (add) {
                    const float2 o = add[g + coff + roff(r)];
                    v.x += o.x, v.y += o.y;
                }
                to[roff(r)] = v;
            }
        }
    }
}

// rho = the sum of nk copies, in order.
__global__ void k_wide_sum(const float4 *__restrict__ part, float4 *__restrict__ rho, uint64_t n4, int nk)
{
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < n4; i += (uint64_t)gridDim.x * blockDim.x) {
        float4 s = part[i];
        for (int j = 1; j < nk; j++) {
            const float4 a = part[j * n4 + i];
            s.x += a.x, s.y += a.y, s.z += a.z, s.w += a.w;
        }
        rho[i] = s;
    }
}

// Operators in separate blocks when the tiles alone leave most of the chip idle.
bool wide_splits(int n, int k, int nk, int nsm)
{
    const uint64_t warps = (1ull << (2 * (n - k))) * (1u << k) / 32;
    return nk > 1 && warps < (uint64_t)nsm * 4;
}

template <int K, int ENT>
static cudaError_t run_wide(const WideOp &op, int first, int count, const float2 *in, float2 *out, bool split,
                            const float2 *add, int n, int nsm, cudaStream_t s)
{
    constexpr int D = 1 << K, TP = 32 / D;
    WideParams<ENT> p;
    p.nk = count;
    int v[10];
    for (int j = 0; j < K; j++) {
        p.cbit[j] = n - 1 - op.qubits[K - 1 - j];
        p.rbit[j] = 2 * n - 1 - op.qubits[K - 1 - j];
        v[j] = p.cbit[j], v[K + j] = p.rbit[j];
    }
    for (int a = 0; a < 2 * K; a++)
        for (int b = a + 1; b < 2 * K; b++)
            if (v[b] < v[a]) { const int x = v[a]; v[a] = v[b]; v[b] = x; }
    for (int a = 0; a < 2 * K; a++) p.pos[a] = v[a];
    p.g = op.dev;
    for (int i = 0; ENT > 0 && i < count * D * D; i++) {
        const c128 z = op.m[(size_t)first * D * D + i];
        p.m[i] = make_float2((float)z.real(), (float)z.imag());
    }
    const size_t ks = sizeof(float4) * D * (D + 1);
    auto kern = k_wide<K, ENT, false>;
    bool all = false;
    if constexpr (K == 3 && ENT == kWideEntries) {
        all = !split;
        if (all) kern = k_wide<K, ENT, true>;
    }
    const size_t sm = (all ? count : 1) * ks + sizeof(float2) * (kWideThreads / 32) * TP * wide_ty(K);
    if (ensure_smem_attr(reinterpret_cast<const void *>(kern), sm)) return cudaErrorInvalidValue;
    const uint64_t ntiles = 1ull << (2 * (n - K)), per = (uint64_t)(kWideThreads / 32) * TP;
    const uint64_t need = (ntiles + per - 1) / per, cap = (uint64_t)nsm * 16;
    kern<<<dim3((unsigned)(need < cap ? need : cap), split ? count : 1), kWideThreads, sm, s>>>(in, out, add, ntiles, 1ull << (2 * n),
                                                                                              p);
    return cudaGetLastError();
}

template <int K>
static cudaError_t wide_k(const WideOp &op, float2 *rho, float2 *scratch, int n, int nsm, cudaStream_t s, int *launches)
{
    constexpr int E1 = 1 << (2 * K), CH = kWideEntries / E1;  // operators a launch carries
    const bool split = wide_splits(n, K, op.nk, nsm);
    *launches = 0;
    if (split && op.dev) {  // every operator in one launch
        const cudaError_t e = run_wide<K, 0>(op, 0, op.nk, rho, scratch, true, nullptr, n, nsm, s);
        if (e != cudaSuccess) return e;
        ++*launches;
    }
    for (int f = split && op.dev ? op.nk : 0; f < op.nk; f += CH) {
        const int cnt = op.nk - f < CH ? op.nk - f : CH;
        const bool last = f + cnt == op.nk;
        // split: copies of their own; else the sum over the launches collects in scratch and the
        // last one writes rho (each tile is read and written by one warp)
        float2 *out = split ? scratch + ((size_t)f << (2 * n)) : last ? rho : scratch;
        const float2 *add = !split && f > 0 ? scratch : nullptr;
        cudaError_t e = cnt == 1 ? run_wide<K, E1>(op, f, cnt, rho, out, split, add, n, nsm, s)
                                 : run_wide<K, kWideEntries>(op, f, cnt, rho, out, split, add, n, nsm, s);
        if (e != cudaSuccess) return e;
        ++*launches;
    }
    if (split) {
        const uint64_t n4 = (1ull << (2 * n)) / 2, g = (n4 + 255) / 256;
        k_wide_sum<<<(unsigned)(g < 1024 ? g : 1024), 256, 0, s>>>(reinterpret_cast<const float4 *>(scratch),
                                                                   reinterpret_cast<float4 *>(rho), n4, op.nk);
        ++*launches;
        return cudaGetLastError();
    }
    return cudaSuccess;
}

// Copies of rho that launch_wide needs as scratch.
int wide_scratch(int n, int k, int nk, int nsm)
{
    if (wide_splits(n, k, nk, nsm)) return nk;
    return nk * (1 << (2 * k)) > kWideEntries ? 1 : 0;
}

cudaError_t launch_wide(const WideOp &op, float2 *rho, float2 *scratch, int n, int nsm, cudaStream_t s, int *launches)
{
    switch (op.k) {
    case 3: return wide_k<3>(op, rho, scratch, n, nsm, s, launches);
    case 4: return wide_k<4>(op, rho, scratch, n, nsm, s, launches);
    default: return wide_k<5>(op, rho, scratch, n, nsm, s, launches);
    }
}

}  // namespace qcw
