// Multiverse ensemble (Sec. 5.2.1, Eq. rhoE1): nvec state vectors evolved by the one- and
// two-qubit operators of Sec. 3, per-vector noise operators chosen by the caller, and the
// density matrix rho = sum_v w_v |psi_v><psi_v| formed on the GPU.
#include "qcw_device.cuh"
#include "qcw_internal.h"

#include <algorithm>
#include <cmath>
#include <utility>
#include <vector>

struct qcw_ensemble {
    int n = 0, nvec = 0, dev = 0, nsm = 0;
    float2 *psi = nullptr;  // nvec x 2^n
    int *d_choice = nullptr;
    float *d_w = nullptr;
    // pinned copies of the caller's draws and weights on their way to the device, kEnsSlots in turn,
    // each with the event after its copy; scratch for densities split over the vectors
    int *h_choice = nullptr;
    float *h_w = nullptr;
    cudaEvent_t slot_ev[2][4] = {};
    int slot_next[2] = {0, 0};
    cudaEvent_t ready = nullptr, taken = nullptr;  // vectors ready for a density; density done with them
    float2 *d_part = nullptr;
    size_t part_elems = 0;
    void *d_stage = nullptr;  // complex128 staging, one vector
    cudaStream_t stream = nullptr;
};

namespace qcw {

constexpr int kEnsThreads = 256;
constexpr int kEnsMaxOmega = 16;
constexpr int kEnsSlots = 4;

struct EnsGate {
    float2 u[16];    // 2^k x 2^k, k <= 2
    int k;
    int pos[2];      // ascending label bits of the struck qubits
    uint64_t off[4]; // offset of local index a (first qubit = most significant bit of a)
};

struct EnsNoise {
    float2 om[kEnsMaxOmega][4];
    int pos;
};

static unsigned ens_grid(uint64_t items, int nsm)
{
    uint64_t g = (items + kEnsThreads - 1) / kEnsThreads;
    const uint64_t cap = (uint64_t)nsm * 16;
    return (unsigned)(g < 1 ? 1 : g > cap ? cap : g);
}

// One thread per (vector, group of 2^k amplitudes differing in the struck bits): the pair /
// quartet update of Eqs. resmat1 / resmat2.
template <int K>
__global__ void k_ens_gate(float2 *__restrict__ psi, int n, uint64_t items, const __grid_constant__ EnsGate p)
{
    constexpr int M = 1 << K;
    const int sh = n - K;
    for (uint64_t t = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; t < items;
         t += (uint64_t)gridDim.x * blockDim.x) {
        const uint64_t v = t >> sh;
        uint64_t g = t & ((1ull << sh) - 1);
#pragma unroll
        for (int j = 0; j < K; j++) g = insert0(g, p.pos[j]);
        float2 *b = psi + (v << n) + g;
        float2 x[M];
#pragma unroll
        for (int a = 0; a < M; a++) x[a] = b[p.off[a]];
#pragma unroll
        for (int a = 0; a < M; a++) {
            float2 y = make_float2(0.f, 0.f);
#pragma unroll
            for (int c = 0; c < M; c++) cfma(y, p.u[M * a + c], x[c]);
            b[p.off[a]] = y;
        }
    }
}

__global__ void k_ens_noise(float2 *__restrict__ psi, int n, uint64_t items, const int *__restrict__ choice,
                            const __grid_constant__ EnsNoise p)
{
    const int sh = n - 1;
    const uint64_t bit = 1ull << p.pos;
    for (uint64_t t = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; t < items;
         t += (uint64_t)gridDim.x * blockDim.x) {
        const uint64_t v = t >> sh;
        const uint64_t g = insert0(t & ((1ull << sh) - 1), p.pos);
        const float2 *u = p.om[choice[v]];
        float2 *b = psi + (v << n) + g;
        const float2 x0 = b[0], x1 = b[bit];
        float2 y0 = make_float2(0.f, 0.f), y1 = make_float2(0.f, 0.f);
        cfma(y0, u[0], x0), cfma(y0, u[1], x1);
        cfma(y1, u[2], x0), cfma(y1, u[3], x1);
        b[0] = y0, b[bit] = y1;
    }
}

// Registers below 6 qubits: a block sums its share of the vectors (staged through shared memory, 16
// at a time) for every element of rho into its own copy; k_ens_sum adds the copies.  (One thread per
// element over all vectors left the chip idle: 530 us for 2048 vectors of 5 qubits.)
constexpr int kSmV = 16;
__global__ void __launch_bounds__(kEnsThreads) k_ens_density_small(const float2 *__restrict__ psi, int nvec, int n,
                                                                   const float *__restrict__ w, float2 *__restrict__ part)
{
    __shared__ float2 a[kSmV][32], b[kSmV][32];
    const int dim = 1 << n, el = dim * dim;
    float2 acc[4];
#pragma unroll
    for (int k = 0; k < 4; k++) acc[k] = make_float2(0.f, 0.f);
    for (int v0 = blockIdx.x * kSmV; v0 < nvec; v0 += gridDim.x * kSmV) {
        __syncthreads();
        for (int e = threadIdx.x; e < (kSmV << n); e += kEnsThreads) {
            const int v = e >> n, i = e & (dim - 1);
            const float2 x = v0 + v < nvec ? psi[((uint64_t)(v0 + v) << n) + i] : make_float2(0.f, 0.f);
            const float wv = v0 + v < nvec ? w[v0 + v] : 0.f;
            b[v][i] = x;
            a[v][i] = make_float2(wv * x.x, wv * x.y);
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < 4; k++) {
            const int e = threadIdx.x + k * kEnsThreads;
            if (e >= el) break;
            const int r = e >> n, c = e & (dim - 1);
#pragma unroll
            for (int v = 0; v < kSmV; v++) cfmac(acc[k], b[v][c], a[v][r]);
        }
    }
#pragma unroll
    for (int k = 0; k < 4; k++) {
        const int e = threadIdx.x + k * kEnsThreads;
        if (e < el) part[(uint64_t)blockIdx.x * el + e] = acc[k];
    }
}

// rho = the sum of np copies of el elements, one after the other: a warp per element when there are
// few of them (lanes take copies in turn, fixed shuffle tree), else a thread.  FP64 sums.
template <bool WARP>
__global__ void k_ens_sum(const float2 *__restrict__ part, int np, uint64_t el, float2 *__restrict__ rho)
{
    const uint64_t t0 = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x, nt = (uint64_t)gridDim.x * blockDim.x;
    const int lane = WARP ? threadIdx.x & 31 : 0;
    for (uint64_t e = WARP ? t0 >> 5 : t0; e < el; e += WARP ? nt >> 5 : nt) {
        double x = 0, y = 0;
        for (int j = lane; j < np; j += WARP ? 32 : 1) {
            const float2 v = part[(uint64_t)j * el + e];
            x += v.x, y += v.y;
        }
        if (WARP) x = warp_sum(x), y = warp_sum(y);
        if (lane == 0) rho[e] = make_float2((float)x, (float)y);
    }
}

// Tiled form of the same rank-nvec update for n >= 6: rho = Psi^T diag(w) conj(Psi) is an outer
// product summed over the vectors, so a CTA owns a 64 x 64 tile of rho, stages 16 vectors' 64
// row amplitudes (times w_v) and 64 column amplitudes in shared memory at a time, and each thread
// accumulates a 4 x 4 block of the tile in registers: 64 FMAs per 8 shared-memory loads instead of
// two global loads per 4 FMAs.  rho is Hermitian, so only tiles on or below the diagonal are
// computed; the one above is written as the conjugate transpose through shared memory.  Tile
// pairs in the order of pair_blocked's triangle, one per CTA in a grid-stride loop.
constexpr int kDenT = 64;   // tile edge
constexpr int kDenV = 16;   // vectors staged per round
constexpr int kDenThreads = 256;
constexpr int kEnsSplitMax = 9;  // qubits up to which the vectors are shared out instead of the tiles

// gridDim.y > 1: grid row y takes its share of the vectors and writes its own copy of rho (rho + y *
// 4^n), for registers with fewer tiles than the chip has SMs.
// diag_blocks: only the 64 x 64 tiles inside the 128 x 128 blocks on the diagonal (three lower
// tiles per block; the tensor-core kernel does the rest).
__global__ void __launch_bounds__(kDenThreads) k_ens_density_tiled(const float2 *__restrict__ psi, int nvec, int n,
                                                                   const float *__restrict__ w,
                                                                   float2 *__restrict__ rho, int diag_blocks)
{
    // one buffer: the staged vectors (As, Bs) while a tile accumulates, then the finished tile
    // (Tt, padded rows) for its mirrored write
    __shared__ __align__(16) float2 sbuf[kDenT * (kDenT + 1)];
    float2(*As)[kDenT] = reinterpret_cast<float2(*)[kDenT]>(sbuf);
    float2(*Bs)[kDenT] = reinterpret_cast<float2(*)[kDenT]>(sbuf + kDenV * kDenT);
    float2(*Tt)[kDenT + 1] = reinterpret_cast<float2(*)[kDenT + 1]>(sbuf);
    const uint64_t dim = 1ull << n;
    const int share = ((nvec + (int)gridDim.y - 1) / (int)gridDim.y + kDenV - 1) / kDenV * kDenV;
    const int vbeg = (int)blockIdx.y * share, vend = nvec < vbeg + share ? nvec : vbeg + share;
    rho += (uint64_t)blockIdx.y * dim * dim;
    const unsigned M = (unsigned)(dim / kDenT);
    const unsigned npairs = diag_blocks ? 3 * (M / 2) : M * (M + 1) / 2;
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    for (unsigned pr = blockIdx.x; pr < npairs; pr += gridDim.x) {
        unsigned R, C;  // row-tile R >= column-tile C
        if (diag_blocks) {  // block b: (2b, 2b), (2b + 1, 2b), (2b + 1, 2b + 1)
            const unsigned b = pr / 3, j = pr % 3;
            R = 2 * b + (j > 0 ? 1u : 0u);
            C = 2 * b + (j == 2 ? 1u : 0u);
        } else {  // pr = R (R + 1) / 2 + C
            R = (unsigned)((sqrt(8.0 * pr + 1.0) - 1.0) / 2.0);
            while (R * (R + 1) / 2 > pr) R--;
            while ((R + 1) * (R + 2) / 2 <= pr) R++;
            C = pr - R * (R + 1) / 2;
        }
        const uint64_t r0 = (uint64_t)R * kDenT, c0 = (uint64_t)C * kDenT;
        float2 acc[4][4];
#pragma unroll
        for (int i = 0; i < 4; i++)
#pragma unroll
            for (int j = 0; j < 4; j++) acc[i][j] = make_float2(0.f, 0.f);
        for (int v0 = vbeg; v0 < vend; v0 += kDenV) {
            __syncthreads();  // the previous round's (or tile's) reads of As / Bs are done
            for (int e = tid; e < kDenV * kDenT; e += kDenThreads) {
                const int v = e / kDenT, i = e % kDenT;
                float2 a = make_float2(0.f, 0.f), b = a;
                if (v0 + v < vend) {
                    const float2 *pv = psi + ((uint64_t)(v0 + v) << n);
                    const float wv = w[v0 + v];
                    a = pv[r0 + i];
                    a = make_float2(wv * a.x, wv * a.y);
                    b = pv[c0 + i];
                }
                As[v][i] = a;
                Bs[v][i] = b;
            }
            __syncthreads();
#pragma unroll 4
            for (int v = 0; v < kDenV; v++) {
                const float4 a01 = *reinterpret_cast<const float4 *>(&As[v][4 * ty]);
                const float4 a23 = *reinterpret_cast<const float4 *>(&As[v][4 * ty + 2]);
                const float4 b01 = *reinterpret_cast<const float4 *>(&Bs[v][4 * tx]);
                const float4 b23 = *reinterpret_cast<const float4 *>(&Bs[v][4 * tx + 2]);
                const float2 a[4] = {make_float2(a01.x, a01.y), make_float2(a01.z, a01.w), make_float2(a23.x, a23.y),
                                     make_float2(a23.z, a23.w)};
                const float2 b[4] = {make_float2(b01.x, b01.y), make_float2(b01.z, b01.w), make_float2(b23.x, b23.y),
                                     make_float2(b23.z, b23.w)};
#pragma unroll
                for (int i = 0; i < 4; i++)
#pragma unroll
                    for (int j = 0; j < 4; j++) {  // acc += a_i conj(b_j)
                        acc[i][j].x = fmaf(a[i].x, b[j].x, fmaf(a[i].y, b[j].y, acc[i][j].x));
                        acc[i][j].y = fmaf(a[i].y, b[j].x, fmaf(-a[i].x, b[j].y, acc[i][j].y));
                    }
            }
        }
#pragma unroll
        for (int i = 0; i < 4; i++) {
            float2 *row = rho + (r0 + 4 * ty + i) * dim + c0 + 4 * tx;
            *reinterpret_cast<float4 *>(row) = make_float4(acc[i][0].x, acc[i][0].y, acc[i][1].x, acc[i][1].y);
            *reinterpret_cast<float4 *>(row + 2) = make_float4(acc[i][2].x, acc[i][2].y, acc[i][3].x, acc[i][3].y);
        }
        if (R == C) continue;
        __syncthreads();  // every thread is done reading As / Bs
#pragma unroll
        for (int i = 0; i < 4; i++)
#pragma unroll
            for (int j = 0; j < 4; j++) Tt[4 * ty + i][4 * tx + j] = acc[i][j];
        __syncthreads();
        // mirror tile (C, R): element (jj, ii) = conj(tile (ii, jj)); consecutive threads take
        // consecutive columns ii of a mirror row jj
        for (int e = tid; e < kDenT * kDenT; e += kDenThreads) {
            const int jj = e / kDenT, ii = e % kDenT;
            const float2 t = Tt[ii][jj];
            rho[(c0 + jj) * dim + r0 + ii] = make_float2(t.x, -t.y);
        }
    }
}

__global__ void k_ens_zero(float2 *__restrict__ psi, int n, uint64_t items)
{
    for (uint64_t t = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; t < items;
         t += (uint64_t)gridDim.x * blockDim.x)
        psi[t] = make_float2((t & ((1ull << n) - 1)) == 0 ? 1.f : 0.f, 0.f);
}

__global__ void k_ens_c128_to_c64(const double2 *__restrict__ src, float2 *__restrict__ dst, uint64_t cnt)
{
    for (uint64_t t = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; t < cnt; t += (uint64_t)gridDim.x * blockDim.x)
        dst[t] = make_float2((float)src[t].x, (float)src[t].y);
}

__global__ void k_ens_c64_to_c128(const float2 *__restrict__ src, double2 *__restrict__ dst, uint64_t cnt)
{
    for (uint64_t t = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; t < cnt; t += (uint64_t)gridDim.x * blockDim.x)
        dst[t] = make_double2(src[t].x, src[t].y);
}

static float2 to_f2(const double *z) { return make_float2((float)z[0], (float)z[1]); }

static bool finite_all(const double *a, size_t cnt)
{
    for (size_t i = 0; i < cnt; i++)
        if (!std::isfinite(a[i])) return false;
    return true;
}

}  // namespace qcw

using namespace qcw;

#define ENS_CK(call)                                               \
    do {                                                           \
        cudaError_t e_ = (call);                                   \
        if (e_ != cudaSuccess) return cuda_error(e_, #call);       \
    } while (0)

static void ens_free(qcw_ensemble *e)
{
    if (!e) return;
    if (e->stream) cudaStreamSynchronize(e->stream);  // also behind the last density (taken)
    if (e->h_choice) cudaFreeHost(e->h_choice);
    if (e->h_w) cudaFreeHost(e->h_w);
    for (auto &k : e->slot_ev)
        for (cudaEvent_t ev : k)
            if (ev) cudaEventDestroy(ev);
    if (e->ready) cudaEventDestroy(e->ready);
    if (e->taken) cudaEventDestroy(e->taken);
    if (e->d_part) cudaFree(e->d_part);
    if (e->psi) cudaFree(e->psi);
    if (e->d_choice) cudaFree(e->d_choice);
    if (e->d_w) cudaFree(e->d_w);
    if (e->d_stage) cudaFree(e->d_stage);
    if (e->stream) cudaStreamDestroy(e->stream);
    delete e;
}

extern "C" qcw_status qcw_ensemble_create(int nqubits, int nvec, qcw_ensemble **out)
{
    if (!out) return set_error(QCW_EINVAL, "null output");
    *out = nullptr;
    if (nqubits < 1 || nqubits > QCW_MAX_QUBITS || nvec < 1 || nvec > 65536)
        return set_error(QCW_EINVAL, "ensemble size out of range");
    qcw_ensemble *e = new qcw_ensemble();
    e->n = nqubits;
    e->nvec = nvec;
    cudaError_t er = cudaGetDevice(&e->dev);
    if (er == cudaSuccess) er = cudaDeviceGetAttribute(&e->nsm, cudaDevAttrMultiProcessorCount, e->dev);
    if (er == cudaSuccess) er = cudaStreamCreateWithFlags(&e->stream, cudaStreamNonBlocking);
    const uint64_t items = (uint64_t)nvec << nqubits;
    if (er == cudaSuccess) er = cudaMalloc(&e->psi, sizeof(float2) * items);
    if (er == cudaSuccess) er = cudaMalloc(&e->d_choice, sizeof(int) * (size_t)nvec);
    if (er == cudaSuccess) er = cudaMalloc(&e->d_w, sizeof(float) * (size_t)nvec);
    if (er == cudaSuccess) er = cudaMallocHost(&e->h_choice, sizeof(int) * (size_t)nvec * kEnsSlots);
    if (er == cudaSuccess) er = cudaMallocHost(&e->h_w, sizeof(float) * (size_t)nvec * kEnsSlots);
    for (auto &k : e->slot_ev)
        for (cudaEvent_t &ev : k)
            if (er == cudaSuccess) er = cudaEventCreateWithFlags(&ev, cudaEventDisableTiming);
    if (er == cudaSuccess) er = cudaEventCreateWithFlags(&e->ready, cudaEventDisableTiming);
    if (er == cudaSuccess) er = cudaEventCreateWithFlags(&e->taken, cudaEventDisableTiming);
    if (er == cudaSuccess) er = cudaMalloc(&e->d_stage, sizeof(double2) << nqubits);
    if (er != cudaSuccess) {
        cudaGetLastError();
        ens_free(e);
        return set_error(QCW_ENOMEM, "ensemble buffers");
    }
    k_ens_zero<<<ens_grid(items, e->nsm), kEnsThreads, 0, e->stream>>>(e->psi, nqubits, items);
    er = cudaGetLastError();
    if (er != cudaSuccess) {
        ens_free(e);
        return cuda_error(er, "ensemble init");
    }
    *out = e;
    return QCW_OK;
}

extern "C" qcw_status qcw_ensemble_destroy(qcw_ensemble *e)
{
    if (!e) return set_error(QCW_EINVAL, "null ensemble");
    ens_free(e);
    return QCW_OK;
}

extern "C" qcw_status qcw_ensemble_set(qcw_ensemble *e, const double *psi_c128)
{
    if (!e || !psi_c128) return set_error(QCW_EINVAL, "null argument");
    const uint64_t dim = 1ull << e->n;
    for (int v = 0; v < e->nvec; v++) {  // one vector at a time through the staging buffer
        ENS_CK(cudaMemcpyAsync(e->d_stage, psi_c128 + 2 * dim * v, sizeof(double2) * dim, cudaMemcpyHostToDevice,
                               e->stream));
        k_ens_c128_to_c64<<<ens_grid(dim, e->nsm), kEnsThreads, 0, e->stream>>>(
            static_cast<const double2 *>(e->d_stage), e->psi + dim * v, dim);
        ENS_CK(cudaGetLastError());
    }
    ENS_CK(cudaStreamSynchronize(e->stream));
    return QCW_OK;
}

extern "C" qcw_status qcw_ensemble_get(qcw_ensemble *e, double *psi_c128)
{
    if (!e || !psi_c128) return set_error(QCW_EINVAL, "null argument");
    const uint64_t dim = 1ull << e->n;
    for (int v = 0; v < e->nvec; v++) {
        k_ens_c64_to_c128<<<ens_grid(dim, e->nsm), kEnsThreads, 0, e->stream>>>(
            e->psi + dim * v, static_cast<double2 *>(e->d_stage), dim);
        ENS_CK(cudaGetLastError());
        ENS_CK(cudaMemcpyAsync(psi_c128 + 2 * dim * v, e->d_stage, sizeof(double2) * dim, cudaMemcpyDeviceToHost,
                               e->stream));
        ENS_CK(cudaStreamSynchronize(e->stream));
    }
    return QCW_OK;
}

// The next pinned slot of a kind (0 draws, 1 weights), once its last copy has left it.
static cudaError_t ens_slot(qcw_ensemble *e, int kind, int *slot)
{
    *slot = e->slot_next[kind]++ % kEnsSlots;
    return cudaEventSynchronize(e->slot_ev[kind][*slot]);
}

static qcw_status ens_gate(qcw_ensemble *e, const double *u, const int *qs, int k)
{
    if (!e || !u) return set_error(QCW_EINVAL, "null argument");
    for (int j = 0; j < k; j++) {
        if (qs[j] < 0 || qs[j] >= e->n) return set_error(QCW_EINVAL, "qubit index out of range");
        for (int i = 0; i < j; i++)
            if (qs[i] == qs[j]) return set_error(QCW_EINVAL, "repeated qubit");
    }
    const int m = 1 << k;
    if (!finite_all(u, 2 * (size_t)m * m)) return set_error(QCW_EINVAL, "non-finite matrix entry");
    EnsGate p{};
    p.k = k;
    for (int i = 0; i < m * m; i++) p.u[i] = to_f2(u + 2 * i);
    int v[2];
    for (int j = 0; j < k; j++) v[j] = e->n - 1 - qs[j];
    for (int a = 0; a < m; a++) {
        uint64_t o = 0;
        for (int j = 0; j < k; j++)
            if ((a >> (k - 1 - j)) & 1) o |= 1ull << v[j];
        p.off[a] = o;
    }
    if (k == 2 && v[1] < v[0]) std::swap(v[0], v[1]);
    for (int j = 0; j < k; j++) p.pos[j] = v[j];
    const uint64_t items = (uint64_t)e->nvec << (e->n - k);
    if (k == 1) k_ens_gate<1><<<ens_grid(items, e->nsm), kEnsThreads, 0, e->stream>>>(e->psi, e->n, items, p);
    else k_ens_gate<2><<<ens_grid(items, e->nsm), kEnsThreads, 0, e->stream>>>(e->psi, e->n, items, p);
    ENS_CK(cudaGetLastError());
    return QCW_OK;
}

extern "C" qcw_status qcw_ensemble_apply_gate1(qcw_ensemble *e, const double u[8], int target)
{
    return ens_gate(e, u, &target, 1);
}

extern "C" qcw_status qcw_ensemble_apply_gate2(qcw_ensemble *e, const double u[32], int q1, int q2)
{
    if (e && e->n < 2) return set_error(QCW_EINVAL, "two-qubit gate on one qubit");
    const int qs[2] = {q1, q2};
    return ens_gate(e, u, qs, 2);
}

extern "C" qcw_status qcw_ensemble_apply_noise1(qcw_ensemble *e, const double *omegas, int nomega, int target,
                                              const int *choice)
{
    if (!e || !omegas || !choice) return set_error(QCW_EINVAL, "null argument");
    if (nomega < 1 || nomega > kEnsMaxOmega) return set_error(QCW_EINVAL, "1 to 16 noise operators");
    if (target < 0 || target >= e->n) return set_error(QCW_EINVAL, "qubit index out of range");
    if (!finite_all(omegas, 8 * (size_t)nomega)) return set_error(QCW_EINVAL, "non-finite matrix entry");
    for (int v = 0; v < e->nvec; v++)
        if (choice[v] < 0 || choice[v] >= nomega) return set_error(QCW_EINVAL, "noise choice out of range");
    EnsNoise p{};
    for (int k = 0; k < nomega; k++)
        for (int i = 0; i < 4; i++) p.om[k][i] = to_f2(omegas + 8 * k + 2 * i);
    p.pos = e->n - 1 - target;
    // through a pinned slot: the caller's array is free when the call returns, without a wait
    int slot = 0;
    ENS_CK(ens_slot(e, 0, &slot));
    int *h = e->h_choice + (size_t)slot * e->nvec;
    std::copy(choice, choice + e->nvec, h);
    ENS_CK(cudaMemcpyAsync(e->d_choice, h, sizeof(int) * (size_t)e->nvec, cudaMemcpyHostToDevice, e->stream));
    ENS_CK(cudaEventRecord(e->slot_ev[0][slot], e->stream));
    const uint64_t items = (uint64_t)e->nvec << (e->n - 1);
    k_ens_noise<<<ens_grid(items, e->nsm), kEnsThreads, 0, e->stream>>>(e->psi, e->n, items, e->d_choice, p);
    ENS_CK(cudaGetLastError());
    return QCW_OK;
}

// Scratch for np copies of rho.
static qcw_status ens_scratch(qcw_ensemble *e, size_t elems)
{
    if (elems <= e->part_elems) return QCW_OK;
    float2 *b = nullptr;
    if (cudaMalloc(&b, sizeof(float2) * elems) != cudaSuccess) {
        cudaGetLastError();
        return set_error(QCW_ENOMEM, "ensemble density scratch");
    }
    if (e->d_part) cudaFree(e->d_part);  // waits for the work that uses it
    e->d_part = b;
    e->part_elems = elems;
    return QCW_OK;
}

extern "C" qcw_status qcw_ensemble_density(qcw_ensemble *e, const double *weights, qcw_ctx *ctx)
{
    if (!e || !weights || !ctx) return set_error(QCW_EINVAL, "null argument");
    if (qcw_nqubits(ctx) != e->n) return set_error(QCW_EINVAL, "qubit counts differ");
    if (!finite_all(weights, (size_t)e->nvec)) return set_error(QCW_EINVAL, "non-finite weight");
    const uint64_t dim = 1ull << e->n, el = dim * dim;
    // copies of rho, each from a share of the vectors, where the tiles alone leave SMs idle (up to 9
    // qubits there are 45 tiles or fewer)
    int split = 1;
    if (dim < (uint64_t)kDenT) {
        split = std::min((e->nvec + kSmV - 1) / kSmV, e->nsm);
    } else if (e->n <= kEnsSplitMax) {
        const int m = (int)(dim / kDenT), tiles = m * (m + 1) / 2;
        split = std::max(1, std::min((e->nvec + 2 * kDenV - 1) / (2 * kDenV), 2 * e->nsm / tiles));
    }
    if (split > 1) {
        qcw_status es = ens_scratch(e, (size_t)split * el);
        if (es) return es;
    }
    int slot = 0;
    ENS_CK(ens_slot(e, 1, &slot));
    float *h = e->h_w + (size_t)slot * e->nvec;
    for (int v = 0; v < e->nvec; v++) h[v] = (float)weights[v];
    ENS_CK(cudaMemcpyAsync(e->d_w, h, sizeof(float) * (size_t)e->nvec, cudaMemcpyHostToDevice, e->stream));
    ENS_CK(cudaEventRecord(e->slot_ev[1][slot], e->stream));
    qcw_status st = begin_state_replace(ctx);
    if (st) return st;
    // ctx's stream takes over from the ensemble's, and back: the vectors, weights and scratch are not
    // touched again before the density is done with them
    ENS_CK(cudaEventRecord(e->ready, e->stream));
    ENS_CK(cudaStreamWaitEvent(ctx->stream, e->ready, 0));
    float2 *out = split > 1 ? e->d_part : ctx->rho;
    if (e->n > kEnsSplitMax) {
        // tiles strictly below the 128 x 128 diagonal blocks on the tensor cores, the diagonal
        // blocks (trace, probabilities) in FP32
        const uint64_t blocks = dim / (2 * kDenT), pairs = 3 * blocks;
        const uint64_t cap = (uint64_t)e->nsm * 8;
        k_ens_density_tiled<<<(unsigned)(pairs < cap ? pairs : cap), kDenThreads, 0, ctx->stream>>>(
            e->psi, e->nvec, e->n, e->d_w, ctx->rho, 1);
        ENS_CK(cudaGetLastError());
        ctx->launches++;
        if (!launch_ens_density_tc(e->psi, e->nvec, e->n, e->d_w, ctx->rho,
                                   reinterpret_cast<unsigned *>(device_error_word(ctx)), ctx->wait_limit, ctx->stall_tile,
                                   e->nsm, ctx->stream))
            return set_error(QCW_ECUDA, "tensor-core density kernel could not be configured");
    } else if (dim >= (uint64_t)kDenT) {
        const uint64_t m = dim / kDenT, pairs = m * (m + 1) / 2;
        k_ens_density_tiled<<<dim3((unsigned)pairs, split), kDenThreads, 0, ctx->stream>>>(e->psi, e->nvec, e->n, e->d_w,
                                                                                          out, 0);
    } else {
        k_ens_density_small<<<split, kEnsThreads, 0, ctx->stream>>>(e->psi, e->nvec, e->n, e->d_w, out);
    }
    ENS_CK(cudaGetLastError());
    ctx->launches++;
    if (split > 1) {
        if (el <= 4096) k_ens_sum<true><<<(unsigned)((el * 32 + 255) / 256), 256, 0, ctx->stream>>>(out, split, el, ctx->rho);
        else k_ens_sum<false><<<(unsigned)((el + 255) / 256), 256, 0, ctx->stream>>>(out, split, el, ctx->rho);
        ENS_CK(cudaGetLastError());
        ctx->launches++;
    }
    ENS_CK(cudaEventRecord(e->taken, ctx->stream));
    ENS_CK(cudaStreamWaitEvent(e->stream, e->taken, 0));
    // the tensor-core kernel's waits are bounded: the call that reads the matrix or hands it out looks whether
    // one ran out (a wait here took 16 us more: two steps, density and purity at 13 qubits 347 -> 363 us)
    ctx->unchecked = e->n > kEnsSplitMax;
    return QCW_OK;
}
