// Device side of a Pauli-basis pass over one tile (see pauli.h): 256 threads hold 64 elements
// each -- the label combinations of three digits -- and apply a round's operations in registers.
//
// Elements are kept as packed pairs along digit 0 (one 64-bit register pair), so that maps on the
// two other digits run as fma.rn.f32x2 with a coefficient duplicated in both halves; maps on digit
// 0 use the halves.  CNOT and CZ are renamings of registers at compile time: their cost is that of
// the two maps that follow, 24 multiply-adds per four-by-four group of elements against 256 for a
// dense two-qubit map.
#pragma once
#include "pauli.h"
#include "qcw_device.cuh"
#include "tile.cuh"

namespace qcw {

using pu64 = unsigned long long;

__device__ __forceinline__ pu64 fmul2(pu64 a, pu64 b)
{
    pu64 d;
    asm("mul.rn.f32x2 %0, %1, %2;\n" : "=l"(d) : "l"(a), "l"(b));
    return d;
}

__device__ __forceinline__ pu64 fneg2(pu64 a) { return a ^ 0x8000000080000000ull; }

// Where a pass's program is read from.  Every coefficient is stored twice, as the pair (c, c) that a
// packed multiply-add takes; an operation's coefficients start at pair 4 op.coef.
// In shared memory (passes with dense maps, programs of the work-item engine): volatile, so that an
// operation reads its coefficients again instead of the compiler keeping them in registers across
// it; the fence between two maps keeps the second one's coefficients from being loaded early (24
// more registers, spills).
struct ProgShared {
    static constexpr bool kFence = true;
    const PRound *rounds;
    const POp *ops;
    unsigned coef;  // shared address
    __device__ __forceinline__ uint4 head(int r) const { return *reinterpret_cast<const uint4 *>(rounds + r); }
    __device__ __forceinline__ uint2 store(int r) const { return *reinterpret_cast<const uint2 *>(rounds[r].st); }
    __device__ __forceinline__ unsigned op(unsigned o) const { return *reinterpret_cast<const unsigned *>(ops + o); }
    __device__ __forceinline__ void pair2(unsigned k, pu64 &a, pu64 &b) const
    {
        asm volatile("ld.shared.v2.b64 {%0, %1}, [%2];\n" : "=l"(a), "=l"(b) : "r"(coef + 8u * k));
    }
};

// In the kernel's parameter block (passes of one context): read through the constant cache with
// warp-uniform addresses, off the shared-memory pipe that the tiles keep busy.
struct ProgParam {
    static constexpr bool kFence = false;
    const unsigned *blob;  // PRound[], POp[] (padded to 16 bytes), coefficient pairs
    int ops, coef;         // word offsets
    __device__ __forceinline__ uint4 head(int r) const { return *reinterpret_cast<const uint4 *>(blob + 24 * r); }
    __device__ __forceinline__ uint2 store(int r) const { return *reinterpret_cast<const uint2 *>(blob + 24 * r + 4); }
    __device__ __forceinline__ unsigned op(unsigned o) const { return blob[ops + o]; }
    __device__ __forceinline__ void pair2(unsigned k, pu64 &a, pu64 &b) const
    {
        const ulonglong2 v = *reinterpret_cast<const ulonglong2 *>(blob + coef + 2 * k);
        a = v.x, b = v.y;
    }
};

template <int N, class P>
__device__ __forceinline__ void p_coefs(const P &p, unsigned k, pu64 (&c)[N])
{
#pragma unroll
    for (int i = 0; i < N; i += 2) p.pair2(k + i, c[i], c[i + 1]);
}

// Index of the pair (digit-0 labels 2h, 2h + 1; digit-1 label i; digit-2 label j).
__host__ __device__ constexpr int px(int h, int i, int j) { return h + 2 * i + 8 * j; }

// Trace-preserving one-qubit map of digit D: y_0 = v_0, y_r = sum_k c[4 (r - 1) + k] v_k.
template <int D, class P>
__device__ __forceinline__ void p_map_tp(pu64 (&x)[32], const P &p, unsigned k)
{
    pu64 c[12];
    p_coefs(p, k, c);
    if constexpr (D == 0) {
        float s[12];
#pragma unroll
        for (int i = 0; i < 12; i++) s[i] = unpack2(c[i]).x;
#pragma unroll
        for (int q = 0; q < 16; q++) {
            const float2 a = unpack2(x[2 * q]), b = unpack2(x[2 * q + 1]);
            float y[4];
            y[0] = a.x;
#pragma unroll
            for (int r = 1; r < 4; r++)
                y[r] = fmaf(s[4 * r - 1], b.y, fmaf(s[4 * r - 2], b.x, fmaf(s[4 * r - 3], a.y, s[4 * r - 4] * a.x)));
            x[2 * q] = pack2(y[0], y[1]);
            x[2 * q + 1] = pack2(y[2], y[3]);
        }
    } else {
#pragma unroll
        for (int q = 0; q < 8; q++) {
            const int o = D == 1 ? px(q & 1, 0, q >> 1) : px(q & 1, q >> 1, 0), st = D == 1 ? 2 : 8;
            const pu64 v0 = x[o], v1 = x[o + st], v2 = x[o + 2 * st], v3 = x[o + 3 * st];
#pragma unroll
            for (int r = 1; r < 4; r++)
                x[o + r * st] = ffma2(c[4 * r - 1], v3, ffma2(c[4 * r - 2], v2, ffma2(c[4 * r - 3], v1, fmul2(c[4 * r - 4], v0))));
        }
    }
}

// General one-qubit map of digit D (16 coefficients).
template <int D, class P>
__device__ __forceinline__ void p_map(pu64 (&x)[32], const P &p, unsigned k)
{
    pu64 c[16];
    p_coefs(p, k, c);
    if constexpr (D == 0) {
#pragma unroll
        for (int q = 0; q < 16; q++) {
            const float2 a = unpack2(x[2 * q]), b = unpack2(x[2 * q + 1]);
            float y[4];
#pragma unroll
            for (int r = 0; r < 4; r++)
                y[r] = fmaf(unpack2(c[4 * r + 3]).x, b.y,
                            fmaf(unpack2(c[4 * r + 2]).x, b.x, fmaf(unpack2(c[4 * r + 1]).x, a.y, unpack2(c[4 * r]).x * a.x)));
            x[2 * q] = pack2(y[0], y[1]);
            x[2 * q + 1] = pack2(y[2], y[3]);
        }
    } else {
#pragma unroll
        for (int q = 0; q < 8; q++) {
            const int o = D == 1 ? px(q & 1, 0, q >> 1) : px(q & 1, q >> 1, 0), st = D == 1 ? 2 : 8;
            const pu64 v0 = x[o], v1 = x[o + st], v2 = x[o + 2 * st], v3 = x[o + 3 * st];
#pragma unroll
            for (int r = 0; r < 4; r++)
                x[o + r * st] = ffma2(c[4 * r + 3], v3, ffma2(c[4 * r + 2], v2, ffma2(c[4 * r + 1], v1, fmul2(c[4 * r], v0))));
        }
    }
}

// Label pair whose coefficient CNOT (first qubit controls) or CZ moves to label pair e = 4 p_first +
// p_second, and whether its sign flips: x_t ^= x_c, z_c ^= z_t (CNOT); z_c ^= x_t, z_t ^= x_c (CZ).
template <bool CZ>
__host__ __device__ constexpr int p_src(int e)
{
    const int xa = (e >> 3) & 1, za = (e >> 2) & 1, xb = (e >> 1) & 1, zb = e & 1;
    return CZ ? 8 * xa + 4 * (za ^ xb) + 2 * xb + (zb ^ xa) : 8 * xa + 4 * (za ^ zb) + 2 * (xb ^ xa) + zb;
}
template <bool CZ>
__host__ __device__ constexpr bool p_neg(int e)
{
    const int xa = (e >> 3) & 1, za = (e >> 2) & 1, xb = (e >> 1) & 1, zb = e & 1;
    return CZ ? (xa & xb & (za ^ zb)) != 0 : (xa & zb & (xb ^ za ^ 1)) != 0;
}

// The permutation on digits (A, B).
template <bool CZ, int A, int B>
__device__ __forceinline__ void p_permute(pu64 (&x)[32])
{
    if constexpr (A != 0 && B != 0) {
#pragma unroll
        for (int h = 0; h < 2; h++) {
            pu64 in[16];
#pragma unroll
            for (int e = 0; e < 16; e++) in[e] = x[A == 1 ? px(h, e >> 2, e & 3) : px(h, e & 3, e >> 2)];
#pragma unroll
            for (int e = 0; e < 16; e++) {
                const pu64 v = in[p_src<CZ>(e)];
                x[A == 1 ? px(h, e >> 2, e & 3) : px(h, e & 3, e >> 2)] = p_neg<CZ>(e) ? fneg2(v) : v;
            }
        }
    } else {
        constexpr int O = A + B;         // the digit that is not digit 0 (1 or 2)
        constexpr int N = O == 1 ? 2 : 1;  // the digit not involved
#pragma unroll
        for (int k = 0; k < 4; k++) {
            float in[4][4];  // [digit 0][digit O]
#pragma unroll
            for (int i = 0; i < 4; i++)
#pragma unroll
                for (int h = 0; h < 2; h++) {
                    const float2 v = unpack2(x[N == 2 ? px(h, i, k) : px(h, k, i)]);
                    in[2 * h][i] = v.x;
                    in[2 * h + 1][i] = v.y;
                }
            float out[4][4];
#pragma unroll
            for (int e = 0; e < 16; e++) {
                const int s = p_src<CZ>(e);
                const float v = A == 0 ? in[s >> 2][s & 3] : in[s & 3][s >> 2];
                (A == 0 ? out[e >> 2][e & 3] : out[e & 3][e >> 2]) = p_neg<CZ>(e) ? -v : v;
            }
#pragma unroll
            for (int i = 0; i < 4; i++)
#pragma unroll
                for (int h = 0; h < 2; h++)
                    x[N == 2 ? px(h, i, k) : px(h, k, i)] = pack2(out[2 * h][i], out[2 * h + 1][i]);
        }
    }
}

// CNOT / CZ on digits (A, B), then the maps of A and of B (digit 0 first: it reads single halves, so
// the renaming costs no moves there).
template <bool CZ, int A, int B, class P>
__device__ __forceinline__ void p_pair(pu64 (&x)[32], const P &p, unsigned k)
{
    p_permute<CZ, A, B>(x);
    if constexpr (B == 0) {
        p_map_tp<B>(x, p, k + 12);
        if constexpr (P::kFence) __syncwarp(__activemask());
        p_map_tp<A>(x, p, k);
    } else {
        p_map_tp<A>(x, p, k);
        if constexpr (P::kFence) __syncwarp(__activemask());
        p_map_tp<B>(x, p, k + 12);
    }
}

// Dense 16 x 16 map on digits (H, L), label pair index 4 p_H + p_L.
template <int H, int L, class P>
__device__ __forceinline__ void p_two(pu64 (&x)[32], const P &p, unsigned k0)
{
    if constexpr (L != 0) {  // (2, 1): packed along digit 0
#pragma unroll
        for (int h = 0; h < 2; h++) {
            pu64 y[16];
#pragma unroll
            for (int e = 0; e < 16; e++) {
#pragma unroll
                for (int f = 0; f < 16; f += 2) {
                    pu64 c0, c1;
                    p.pair2(k0 + 16 * e + f, c0, c1);
                    const pu64 a = x[px(h, f & 3, f >> 2)], b = x[px(h, (f + 1) & 3, f >> 2)];
                    y[e] = f ? ffma2(c0, a, y[e]) : fmul2(c0, a);
                    y[e] = ffma2(c1, b, y[e]);
                }
            }
#pragma unroll
            for (int e = 0; e < 16; e++) x[px(h, e & 3, e >> 2)] = y[e];
        }
    } else {
#pragma unroll
        for (int k = 0; k < 4; k++) {  // the digit not involved
            float v[16], y[16];
#pragma unroll
            for (int i = 0; i < 4; i++)
#pragma unroll
                for (int h = 0; h < 2; h++) {
                    const float2 a = unpack2(x[H == 1 ? px(h, i, k) : px(h, k, i)]);
                    v[4 * i + 2 * h] = a.x;
                    v[4 * i + 2 * h + 1] = a.y;
                }
#pragma unroll
            for (int e = 0; e < 16; e++) {
#pragma unroll
                for (int f = 0; f < 16; f += 2) {
                    pu64 c0, c1;
                    p.pair2(k0 + 16 * e + f, c0, c1);
                    y[e] = f ? fmaf(unpack2(c0).x, v[f], y[e]) : unpack2(c0).x * v[f];
                    y[e] = fmaf(unpack2(c1).x, v[f + 1], y[e]);
                }
            }
#pragma unroll
            for (int i = 0; i < 4; i++)
#pragma unroll
                for (int h = 0; h < 2; h++)
                    x[H == 1 ? px(h, i, k) : px(h, k, i)] = pack2(y[4 * i + 2 * h], y[4 * i + 2 * h + 1]);
        }
    }
}

// DENSE: with the dense two-qubit maps (left out of the kernel that most passes take: they are two
// thirds of the code).
template <bool DENSE, class P>
__device__ __forceinline__ void p_op(pu64 (&x)[32], int kind, const P &p, unsigned k)
{
    if (DENSE && kind >= PO_TWO && kind < PO_TWO + 3) {
        if (kind == PO_TWO) p_two<1, 0>(x, p, k);
        else if (kind == PO_TWO + 1) p_two<2, 0>(x, p, k);
        else p_two<2, 1>(x, p, k);
        return;
    }
    switch (kind) {
    case PO_ONE: p_map<0>(x, p, k); break;
    case PO_ONE + 1: p_map<1>(x, p, k); break;
    case PO_ONE + 2: p_map<2>(x, p, k); break;
    case PO_CX: p_pair<false, 0, 1>(x, p, k); break;
    case PO_CX + 1: p_pair<false, 0, 2>(x, p, k); break;
    case PO_CX + 2: p_pair<false, 1, 0>(x, p, k); break;
    case PO_CX + 3: p_pair<false, 1, 2>(x, p, k); break;
    case PO_CX + 4: p_pair<false, 2, 0>(x, p, k); break;
    case PO_CX + 5: p_pair<false, 2, 1>(x, p, k); break;
    case PO_CZ: p_pair<true, 0, 1>(x, p, k); break;
    case PO_CZ + 1: p_pair<true, 0, 2>(x, p, k); break;
    case PO_CZ + 2: p_pair<true, 1, 2>(x, p, k); break;
    default:
        p_map_tp<1>(x, p, k);
        if constexpr (P::kFence) __syncwarp(__activemask());
        p_map_tp<2>(x, p, k + 12);
        break;
    }
}

__device__ __forceinline__ float4 p_lds4(unsigned addr)
{
    float4 v;
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];\n" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr) : "memory");
    return v;
}
__device__ __forceinline__ void p_sts2(unsigned addr, pu64 a, pu64 b)
{
    asm volatile("st.shared.v2.b64 [%0], {%1, %2};\n" ::"r"(addr), "l"(a), "l"(b) : "memory");
}
__device__ __forceinline__ void p_lds2(unsigned addr, pu64 &a, pu64 &b)
{
    asm volatile("ld.shared.v2.b64 {%0, %1}, [%2];\n" : "=l"(a), "=l"(b) : "r"(addr) : "memory");
}

// Signs that the round's own permutation brings, on digits 1 and 2.
template <bool CZ, bool BC>
__device__ __forceinline__ void p_signs(pu64 (&x)[32])
{
#pragma unroll
    for (int e = 0; e < 16; e++)
        if (p_neg<CZ>(e))
#pragma unroll
            for (int h = 0; h < 2; h++) {
                const int k = BC ? px(h, e >> 2, e & 3) : px(h, e & 3, e >> 2);
                x[k] = fneg2(x[k]);
            }
}

// Product of the start factors (PauliHdr::w) of the digits dig[0..nd) at the labels in lab.
template <class D>
__device__ __forceinline__ float p_factor(const float *w, const D *dig, int nd, unsigned lab)
{
    float f = 1.f;
    for (int d = 0; d < nd; d++) f *= w[4 * dig[d] + ((lab >> (2 * d)) & 3u)];
    return f;
}

// What the last round does with its results: back to the tile in shared memory.
template <bool FULL = false>
struct KeepTile {
    static constexpr bool kDirect = false, kFull = FULL;
    __device__ __forceinline__ void store(const PRound &, const pu64 (&)[32], unsigned, unsigned) const {}
};

// The rounds of a pass on the tile at shared address `tile`, by 256 threads (tid) that meet at
// named barrier `bar`.  tab: the rounds in shared memory (their position tables are read per thread).
// T::kFull: the tile has kPTile digits.  T::kDirect: the elements of a round marked direct (the last one of a pass) go to T::store from the registers instead of back to the
// tile, which is free for its next contents once the call returns (every thread has read its own).
template <bool DENSE, class P, class T = KeepTile<>>
__device__ __forceinline__ void pauli_rounds(unsigned tile, const PRound *__restrict__ tab, int nround, const P &p,
                                             unsigned tid, int bar, const T &last = T())
{
    for (int r = 0; r < nround; r++) {
        const uint4 w = p.head(r);  // db dc nob nop | op0 perm | ld
        if (T::kFull || tid < (1u << ((w.x >> 16) & 255u))) {  // full tiles: every thread has a group
            const unsigned base = (unsigned)tab[r].lo[tid & 15u] ^ (unsigned)tab[r].hi[tid >> 4];
            pu64 x[32];
            {
                const unsigned b[4] = {0u, w.z & 0xFFFFu, w.z >> 16, (w.z & 0xFFFFu) ^ (w.z >> 16)};
                const unsigned c[4] = {0u, w.w & 0xFFFFu, w.w >> 16, (w.w & 0xFFFFu) ^ (w.w >> 16)};
#pragma unroll
                for (int j = 0; j < 4; j++)
#pragma unroll
                    for (int i = 0; i < 4; i++) p_lds2(tile + (base ^ b[i] ^ c[j]), x[px(0, i, j)], x[px(1, i, j)]);
            }
            if (T::kDirect && (w.y >> 24)) {  // full tiles only: every thread is here
                bar_sync(bar, 256);
            }
            const unsigned perm = (w.y >> 16) & 255u;
            if (perm == PP_CX_BC) p_signs<false, true>(x);
            else if (perm == PP_CX_CB) p_signs<false, false>(x);
            else if (perm == PP_CZ) p_signs<true, true>(x);
            const unsigned o1 = (w.y & 65535u) + (w.x >> 24);
            for (unsigned o = w.y & 65535u; o < o1; o++) {
                const unsigned op = p.op(o);
                p_op<DENSE>(x, (int)(op & 65535u), p, 4u * (op >> 16));
            }
            if (T::kDirect && (w.y >> 24)) {
                last.store(tab[r], x, w.x & 255u, (w.x >> 8) & 255u);
                return;
            }
            {
                const uint2 s = p.store(r);
                const unsigned b[4] = {0u, s.x & 0xFFFFu, s.x >> 16, (s.x & 0xFFFFu) ^ (s.x >> 16)};
                const unsigned c[4] = {0u, s.y & 0xFFFFu, s.y >> 16, (s.y & 0xFFFFu) ^ (s.y >> 16)};
#pragma unroll
                for (int j = 0; j < 4; j++)
#pragma unroll
                    for (int i = 0; i < 4; i++) p_sts2(tile + (base ^ b[i] ^ c[j]), x[px(0, i, j)], x[px(1, i, j)]);
            }
        }
        bar_sync(bar, 256);
    }
}

}  // namespace qcw
