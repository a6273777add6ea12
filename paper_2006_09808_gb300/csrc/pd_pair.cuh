// pd_pair.cuh -- the fused primal-dual iteration with one complex 2-D transform pair per
// iteration and the slice's state on chip for all iterations.
//
// The two dipole convolutions of one iteration of the Sec. II.A pseudocode, v = D W p and the next
// u = D chibar, travel as the two real channels of one complex field.  With d = G^T M q,
//     chi_n     = chi_{n-1} - tau (v + d)                 (primal step)
//     chibar_n  = 2 chi_n - chi_{n-1} = b - 2 tau v,      b = chi_{n-1} - 2 tau d
//     u         = D chibar_n = D b - 2 tau D^2 (W p),
// so the forward transform Z of z = s W p + i b holds everything both need, and with
// P = (Z(k) + conj Z(-k)) / 2 = s F(W p) one pointwise product gives both at once:
//     out(k) = D(k) Z(k) - i (2 tau / s) D(k)^2 P(k),     F^-1 out = s v + i u.
// b is formed from the stored chi in every iteration (nothing is accumulated in the spectrum).  The
// power of two s ~ 1/lambda (pair_scale) brings W p to the size of b: the rounding that leaks
// between the channels then stays below that of the separate transforms.  Against FP64, 300 iterations
// of 64 x 64 emulated in FP32: the same error as with separate transforms for lambda up to 1e-2 (2.5e-7
// at 5e-4), 5e-7 instead of 1.5e-7 from lambda = 1 on, whatever the scale: u is the transform of chibar
// before its rounding, which reaches the data term one iteration later.
//
// One iteration of a cluster of C CTAs (CTA c owns rows [cR, (c+1)R); column kx is kept together
// with column W - kx, as the pair of the product above):
//   phase A  gather rows, inverse row FFT -> v, u; chi, chibar; p (dual data prox)
//   phase B  q (dual TV prox) from chibar of this row and the next
//   phase C  b, forward row FFT of s W p + i b, scatter
//   columns  forward FFTs of a pair, the product, inverse FFTs
// against two gathers, scatters, column passes and real-row splits per iteration in
// pd_cluster.cuh.
//
// A group of T lanes carries rows a = 2j, b = 2j + 1 of the slice for the whole solve, so every thread
// owns the same 2E pixels throughout and their chi, p, qx, qy never leave the SM: in tensor memory
// (StTmem: 512 threads x 8E words, 256 KB for E = 16; these CTAs take more than half of the SM's
// shared memory each, so no two of them share an SM and the allocation never waits for a peer) or, for
// small CTAs, in shared memory (StShared).  Neighbouring rows of other groups pass through one row
// slot per group boundary, which carries chibar of the lower group's row a up and then q_y of the
// upper group's row b down.
//
// Both rows (in the column pass both columns of a pair) go through every transform together, one in
// each half of 64-bit registers (F2): one packed instruction for both, half the issue slots.
//
// Spectrum layout of a CTA: row pair j is a line of 2 PC 16-byte units (re a, re b, im a, im b), unit k
// of column kx = k, then of the mirror columns, the index XORed with j & 7.  A lane gathers and
// scatters both rows with one 16-byte access; the 16 lanes of a group cover whole 128-byte lines of
// one CTA, and the strided accesses of the column pass spread over the banks.
//
// What bounds it (256 x 256, 4 CTAs of 512 threads): 64 slices x 500 iterations take 19.9 ms, 31.1
// for pd_cluster.cuh's kernel in the same geometry.  On the way there: scalar transforms of one row
// after the other, state in tensor memory 35.9 ms (280 bytes of spills, whose reloads miss the small
// L1); both rows packed f32x2 26.0; whole lines per gather instead of 32-byte sectors (column-major
// units) 21.8; barriers split around independent work, D(k) in flight during one, the field in thread
// order 19.9.  What is left is the exchange through distributed shared memory (gather, scatter and the
// barrier behind it, a quarter of an iteration), packed FP32 issue (a third), the shared-memory
// wavefronts of the column pass and the skew at the barriers.
#pragma once

#include <type_traits>

#include "pd_cluster.cuh"

namespace pcs {

// ------------------------------------------------------------------ geometry

// N x N slices, clusters of C CTAs of NT threads (two rows per lane group).
// TMEM: state in tensor memory (CTAs that fill an SM), else in shared memory.
template <int N_, int C_, int NT_, bool TMEM_, int E_ = 0>
struct GeoPair {
    static constexpr int N = N_, H = N_, W = N_, C = C_, NT = NT_;
    static constexpr bool TMEM = TMEM_;
    static constexpr int E = E_ ? E_ : default_elems(N), T = N / E;  // elements per lane, lanes per transform
    static constexpr int M = N / 2;
    static constexpr int R = N / C;      // rows per CTA
    static constexpr int NG = NT / T;    // lane groups = row pairs = column pairs of the CTA
    static constexpr int PC = M / C;     // column pairs per CTA
    static constexpr int NCH = E / 2;    // chunks of two elements of both rows
    static constexpr int MINB = (NT >= 512) ? 1 : 512 / NT;
    static constexpr int TW = StageTw<N, E>::SIZE;
    // bytes
    static constexpr size_t SPEC_BYTES = sizeof(float2) * 2 * PC * N;
    static constexpr size_t ROWS_BYTES = sizeof(float2) * NG * N;
    // (the last slot is written by the slice's last rows and read by none)
    static constexpr size_t SLOT_BYTES = sizeof(float) * (NG + 1) * N;
    static constexpr size_t STATE_BYTES = TMEM ? 0 : sizeof(float) * 4 * 2 * E * NT;
    // row slots in shared memory where they fit, else in the chibar scratch rows (global)
    static constexpr size_t BASE_BYTES = SPEC_BYTES + ROWS_BYTES + sizeof(float2) * TW + STATE_BYTES + 16;
    static constexpr bool SLOT_GLOBAL = BASE_BYTES + SLOT_BYTES > 232448;
    static constexpr size_t SMEM_BYTES = BASE_BYTES + (SLOT_GLOBAL ? 0 : SLOT_BYTES);
    static_assert(NG * 2 == R && NG == PC, "two rows and one column pair per lane group");
    static_assert(T >= 8 && T <= 32 && (T & (T - 1)) == 0 && E % 4 == 0, "lane groups");
    // p in global scratch (thread order) when four arrays exceed the tensor memory
    static constexpr bool P_GLOBAL = TMEM && (NT / 128) * 8 * E > 512;
    static constexpr int TM_WORDS = (P_GLOBAL ? 6 : 8) * E;  // tensor-memory words per thread
    static_assert(!TMEM || (NT > 256 && (NT / 128) * TM_WORDS <= 512), "tensor-memory state: one CTA per SM");
    static_assert(E <= 32, "mask bits");
    static_assert(SMEM_BYTES <= 232448, "shared memory");
    static_assert(!TMEM || 2 * (SMEM_BYTES + 1024) > 233472, "one tensor-memory CTA per SM");
    static constexpr int TMEM_COLS = 512;
};

// ------------------------------------------------------------------ small PTX helpers

// Hides where a value comes from, so that what is derived from it is recomputed where it is used
// and not kept in registers across the phases of an iteration.
template <class I>
__device__ __forceinline__ I fresh(I v) {
    asm volatile("" : "+r"(v));
    return v;
}
template <class X>
__device__ __forceinline__ X* fresh(X* v) {
    asm volatile("" : "+l"(v));
    return v;
}

__device__ __forceinline__ unsigned smem_u32(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }

// shared::cluster address of `addr` in CTA `rank` of the cluster
template <int C>
__device__ __forceinline__ unsigned map_rank(unsigned addr, int rank) {
    if constexpr (C == 1) {
        return addr;
    } else {
        unsigned r;
        asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
        return r;
    }
}
// Remote addresses are complete before the access (fresh): no part of them becomes an immediate
// offset (see PairLane).
template <int C>
__device__ __forceinline__ ulonglong2 ld_cluster_pair(unsigned a) {
    ulonglong2 v;
    if constexpr (C == 1) {
        asm volatile("ld.shared.v2.b64 {%0,%1}, [%2];" : "=l"(v.x), "=l"(v.y) : "r"(a) : "memory");
    } else {
        asm volatile("ld.shared::cluster.v2.b64 {%0,%1}, [%2];" : "=l"(v.x), "=l"(v.y) : "r"(fresh(a)) : "memory");
    }
    return v;
}
template <int C>
__device__ __forceinline__ void st_cluster_pair(unsigned a, ulonglong2 v) {
    if constexpr (C == 1) {
        asm volatile("st.shared.v2.b64 [%0], {%1,%2};" ::"r"(a), "l"(v.x), "l"(v.y) : "memory");
    } else {
        asm volatile("st.shared::cluster.v2.b64 [%0], {%1,%2};" ::"r"(fresh(a)), "l"(v.x), "l"(v.y) : "memory");
    }
}
template <int C>
__device__ __forceinline__ float2 ld_cluster2(unsigned a) {
    float2 v;
    if constexpr (C == 1) {
        asm volatile("ld.shared.v2.f32 {%0,%1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(a) : "memory");
    } else {
        asm volatile("ld.shared::cluster.v2.f32 {%0,%1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(fresh(a)) : "memory");
    }
    return v;
}
template <int C>
__device__ __forceinline__ void st_cluster2(unsigned a, float2 v) {
    if constexpr (C == 1) {
        asm volatile("st.shared.v2.f32 [%0], {%1,%2};" ::"r"(a), "f"(v.x), "f"(v.y) : "memory");
    } else {
        asm volatile("st.shared::cluster.v2.f32 [%0], {%1,%2};" ::"r"(fresh(a)), "f"(v.x), "f"(v.y) : "memory");
    }
}

// ------------------------------------------------------------------ two transforms at a time

// A pair of FP32 values (one of each of two transforms) in a 64-bit register: add, subtract,
// multiply and fused multiply-add of both in one instruction, each rounded as the scalar one.
struct F2 {
    unsigned long long v;
    F2() = default;
    __device__ __forceinline__ explicit F2(unsigned long long w) : v(w) {}
    __device__ __forceinline__ F2(float a, float b) { asm("mov.b64 %0, {%1, %2};" : "=l"(v) : "f"(a), "f"(b)); }
    __device__ __forceinline__ explicit F2(double c) : F2((float)c, (float)c) {}
    __device__ __forceinline__ float lo() const {
        float a, b;
        asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
        return a;
    }
    __device__ __forceinline__ float hi() const {
        float a, b;
        asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
        return b;
    }
};
__device__ __forceinline__ F2 operator+(F2 a, F2 b) {
    F2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ F2 operator-(F2 a, F2 b) {
    F2 r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ F2 operator*(F2 a, F2 b) {
    F2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ F2 fma2(F2 a, F2 b, F2 c) {
    F2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
    return r;
}

// A complex element of both transforms.
struct C2 {
    F2 x, y;
};
__device__ __forceinline__ C2 cadd(C2 a, C2 b) { return C2{a.x + b.x, a.y + b.y}; }
__device__ __forceinline__ C2 csub(C2 a, C2 b) { return C2{a.x - b.x, a.y - b.y}; }
// a +- (-i) b forward, a +- (+i) b inverse
template <bool INV>
__device__ __forceinline__ C2 cadd_mi(C2 a, C2 b) {
    return INV ? C2{a.x - b.y, a.y + b.x} : C2{a.x + b.y, a.y - b.x};
}
template <bool INV>
__device__ __forceinline__ C2 csub_mi(C2 a, C2 b) {
    return INV ? C2{a.x + b.y, a.y - b.x} : C2{a.x - b.y, a.y + b.x};
}
// multiply by the constant (c, s), s for the forward sign (mul_const of fft_core.cuh, pairwise)
template <bool INV>
__device__ __forceinline__ C2 cmulc(C2 a, double c, double s) {
    const double ss = INV ? -s : s;
    return C2{fma2(a.x, F2(c), a.y * F2(-ss)), fma2(a.x, F2(ss), a.y * F2(c))};
}

template <bool INV>
__device__ __forceinline__ void dft4p(C2& v0, C2& v1, C2& v2, C2& v3) {
    const C2 t0 = cadd(v0, v2), t1 = csub(v0, v2), t2 = cadd(v1, v3), t3 = csub(v1, v3);
    v0 = cadd(t0, t2);
    v2 = csub(t0, t2);
    v1 = cadd_mi<INV>(t1, t3);
    v3 = csub_mi<INV>(t1, t3);
}
template <bool INV>
__device__ __forceinline__ void dft8p(C2 (&v)[8]) {
    C2 e0 = v[0], e1 = v[2], e2 = v[4], e3 = v[6];
    C2 o0 = v[1], o1 = v[3], o2 = v[5], o3 = v[7];
    dft4p<INV>(e0, e1, e2, e3);
    dft4p<INV>(o0, o1, o2, o3);
    o1 = cmulc<INV>(o1, kR2, -kR2);
    o3 = cmulc<INV>(o3, -kR2, -kR2);
    v[0] = cadd(e0, o0);
    v[4] = csub(e0, o0);
    v[1] = cadd(e1, o1);
    v[5] = csub(e1, o1);
    v[2] = cadd_mi<INV>(e2, o2);
    v[6] = csub_mi<INV>(e2, o2);
    v[3] = cadd(e3, o3);
    v[7] = csub(e3, o3);
}
template <bool INV>
__device__ __forceinline__ void dft16p(C2 (&v)[16]) {
    C2 e[8], o[8];
#pragma unroll
    for (int t = 0; t < 8; ++t) {
        e[t] = v[2 * t];
        o[t] = v[2 * t + 1];
    }
    dft8p<INV>(e);
    dft8p<INV>(o);
    o[1] = cmulc<INV>(o[1], kC1, -kS1);
    o[2] = cmulc<INV>(o[2], kR2, -kR2);
    o[3] = cmulc<INV>(o[3], kS1, -kC1);
    o[5] = cmulc<INV>(o[5], -kS1, -kC1);
    o[6] = cmulc<INV>(o[6], -kR2, -kR2);
    o[7] = cmulc<INV>(o[7], -kC1, -kS1);
#pragma unroll
    for (int t = 0; t < 8; ++t) {
        if (t == 4) {
            v[4] = cadd_mi<INV>(e[4], o[4]);
            v[12] = csub_mi<INV>(e[4], o[4]);
        } else {
            v[t] = cadd(e[t], o[t]);
            v[t + 8] = csub(e[t], o[t]);
        }
    }
}
template <bool INV>
__device__ __forceinline__ void dft3p(C2& a, C2& b, C2& c) {
    const C2 t1 = cadd(b, c), d = csub(b, c);
    const C2 t2 = C2{fma2(F2(-0.5), t1.x, a.x), fma2(F2(-0.5), t1.y, a.y)};
    const C2 t3 = C2{d.x * F2(kH3), d.y * F2(kH3)};
    a = cadd(a, t1);
    b = cadd_mi<INV>(t2, t3);
    c = csub_mi<INV>(t2, t3);
}
template <int R, bool INV>
__device__ __forceinline__ void dftRp(C2 (&v)[R]) {
    if constexpr (R == 2) {
        const C2 t = v[0];
        v[0] = cadd(t, v[1]);
        v[1] = csub(t, v[1]);
    } else if constexpr (R == 4) {
        dft4p<INV>(v[0], v[1], v[2], v[3]);
    } else if constexpr (R == 6) {
        // n = 3 n1 + n2, k = k1 + 2 k2 (dft_composite of fft_core.cuh)
        C2 y[3][2];
#pragma unroll
        for (int n2 = 0; n2 < 3; ++n2) {
            y[n2][0] = cadd(v[n2], v[3 + n2]);
            const C2 t = csub(v[n2], v[3 + n2]);
            y[n2][1] = (n2 == 0) ? t : cmulc<INV>(t, cos24(4 * n2), -sin24(4 * n2));
        }
#pragma unroll
        for (int k1 = 0; k1 < 2; ++k1) {
            dft3p<INV>(y[0][k1], y[1][k1], y[2][k1]);
#pragma unroll
            for (int k2 = 0; k2 < 3; ++k2) v[k1 + 2 * k2] = y[k2][k1];
        }
    } else if constexpr (R == 8) {
        dft8p<INV>(v);
    } else if constexpr (R == 12) {
        // n = 3 n1 + n2, k = k1 + 4 k2 (dft_composite of fft_core.cuh)
        C2 y[3][4];
#pragma unroll
        for (int n2 = 0; n2 < 3; ++n2) {
            C2 t0 = v[n2], t1 = v[3 + n2], t2 = v[6 + n2], t3 = v[9 + n2];
            dft4p<INV>(t0, t1, t2, t3);
            const C2 t[4] = {t0, t1, t2, t3};
#pragma unroll
            for (int k1 = 0; k1 < 4; ++k1) {
                const int m = n2 * k1 * 2;  // multiples of 15 degrees
                y[n2][k1] = (m == 0) ? t[k1] : cmulc<INV>(t[k1], cos24(m), -sin24(m));
            }
        }
#pragma unroll
        for (int k1 = 0; k1 < 4; ++k1) {
            dft3p<INV>(y[0][k1], y[1][k1], y[2][k1]);
#pragma unroll
            for (int k2 = 0; k2 < 3; ++k2) v[k1 + 4 * k2] = y[k2][k1];
        }
    } else {
        static_assert(R == 16, "radix");
        dft16p<INV>(v);
    }
}

// Twiddle one element of both transforms (scalar products: both halves by the same factor).
template <bool INV>
__device__ __forceinline__ C2 ctw(C2 a, float2 w) {
    if (INV) w.y = -w.y;
    const float ax = a.x.lo(), ay = a.y.lo(), bx = a.x.hi(), by = a.y.hi();
    return C2{F2(fmaf(ax, w.x, -ay * w.y), fmaf(bx, w.x, -by * w.y)), F2(fmaf(ax, w.y, ay * w.x), fmaf(bx, w.y, by * w.x))};
}

// Buffers of the exchange between two stages: element i of a stage's output goes to position i.
// RowBuf: N 8-byte positions, used for the real and then for the imaginary parts.
struct RowBuf {
    unsigned char* b;
    template <int E, class FS, class FL>
    __device__ __forceinline__ void exchange(C2 (&x)[E], FS store_at, FL load_at) const {
        unsigned long long* u = reinterpret_cast<unsigned long long*>(b);
        auto at = [](int i) { return i ^ ((i >> 4) & 15); };
        __syncwarp();
#pragma unroll
        for (int e = 0; e < E; ++e) u[at(store_at(e))] = x[e].x.v;
        __syncwarp();
#pragma unroll
        for (int e = 0; e < E; ++e) x[e].x = F2(u[at(load_at(e))]);
        __syncwarp();
#pragma unroll
        for (int e = 0; e < E; ++e) u[at(store_at(e))] = x[e].y.v;
        __syncwarp();
#pragma unroll
        for (int e = 0; e < E; ++e) x[e].y = F2(u[at(load_at(e))]);
    }
};
// ColBuf: the 2 x N/2 16-byte units of a column pair in the spectrum (both components at once).
// Position 16 a + b is half b & 1 of row pair 8 a + ((b >> 1) ^ (a & 7)): the stage-1 stores (a over
// the lanes) and the loads in natural order (b over the lanes) of 8 lanes touch every bank once.
template <int PC>
struct ColBuf {
    unsigned char* spec;
    int cl;
    __device__ __forceinline__ unsigned char* unit(int i) const {
        const int a = i >> 4, b = i & 15;
        const int j = 8 * a + ((b >> 1) ^ (a & 7));
        return spec + j * (32 * PC) + 16 * ((((b & 1) ? PC + (cl ^ 4) : cl)) ^ (j & 7));
    }
    template <int E, class FS, class FL>
    __device__ __forceinline__ void exchange(C2 (&x)[E], FS store_at, FL load_at) const {
        __syncwarp();
#pragma unroll
        for (int e = 0; e < E; ++e)
            *reinterpret_cast<ulonglong2*>(unit(store_at(e))) = make_ulonglong2(x[e].x.v, x[e].y.v);
        __syncwarp();
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const ulonglong2 t = *reinterpret_cast<const ulonglong2*>(unit(load_at(e)));
            x[e] = C2{F2(t.x), F2(t.y)};
        }
    }
};

// fft<N, T, INV> of fft_core.cuh on two transforms at a time (same factorisation, element order
// and twiddles): the whole warp calls it.
template <int N, int T, bool INV, class Buf>
__device__ __forceinline__ void fft_pair(C2 (&x)[N / T], const Buf& buf, const float2* __restrict__ stw, int g) {
    constexpr int E = N / T;
    using PL = Plan<N, E>;
    constexpr int R1 = PL::R1, RM = PL::RM, RL = PL::RL;
    constexpr int B1 = E / R1, BL = E / RL;
    // stage 1: butterfly b takes x[b + r B1]; output r of butterfly j = g + b T to position j R1 + r
#pragma unroll
    for (int b = 0; b < B1; ++b) {
        C2 v[R1];
#pragma unroll
        for (int r = 0; r < R1; ++r) v[r] = x[b + r * B1];
        dftRp<R1, INV>(v);
#pragma unroll
        for (int r = 0; r < R1; ++r) x[b + r * B1] = v[r];
    }
    auto at1 = [g](int e) { return (g + (e % B1) * T) * R1 + e / B1; };
    if constexpr (RM != 0) {
        constexpr int BM = E / RM, NS = R1;
        buf.exchange(x, at1, [g](int e) { return g + (e % BM) * T + (e / BM) * (N / RM); });
#pragma unroll
        for (int b = 0; b < BM; ++b) {
            C2 v[RM];
            const int k = (g + b * T) % NS;
#pragma unroll
            for (int r = 0; r < RM; ++r) v[r] = (r == 0) ? x[b] : ctw<INV>(x[b + r * BM], stw[(r - 1) * NS + k]);
            dftRp<RM, INV>(v);
#pragma unroll
            for (int r = 0; r < RM; ++r) x[b + r * BM] = v[r];
        }
        buf.exchange(
            x,
            [g](int e) {
                const int j = g + (e % BM) * T, k = j % NS;
                return (j / NS) * NS * RM + k + (e / BM) * NS;
            },
            [g](int e) { return g + (e % BL) * T + (e / BL) * (N / RL); });
    } else {
        buf.exchange(x, at1, [g](int e) { return g + (e % BL) * T + (e / BL) * (N / RL); });
    }
    constexpr int NS = N / RL;
    const float2* tl = stw + StageTw<N, E>::MID;
#pragma unroll
    for (int b = 0; b < BL; ++b) {
        C2 v[RL];
        const int k = (g + b * T) % NS;
#pragma unroll
        for (int r = 0; r < RL; ++r) v[r] = (r == 0) ? x[b] : ctw<INV>(x[b + r * BL], tl[(r - 1) * NS + k]);
        dftRp<RL, INV>(v);
#pragma unroll
        for (int r = 0; r < RL; ++r) x[b + r * BL] = v[r];
    }
}

// ------------------------------------------------------------------ per-thread state

enum { kChi = 0, kP = 1, kQx = 2, kQy = 3 };

// Chunk q of array a of this thread: elements 2q, 2q + 1 as (row a, row b, row a, row b).  load() returns
// K chunks; in tensor memory the loads and the wait for them are one asm block, since nothing may
// touch the destination registers in between.
struct ChunkId {
    int a, q;
};

#define PCS_TMEM_LD "tcgen05.ld.sync.aligned.32x32b.x4.b32 "
#define PCS_TMEM_WAIT "tcgen05.wait::ld.sync.aligned;"
#define PCS_OUT4(k) "=&r"(w[4 * (k)]), "=&r"(w[4 * (k) + 1]), "=&r"(w[4 * (k) + 2]), "=&r"(w[4 * (k) + 3])

template <class G>
struct StTmem {
    unsigned base;
    float4* gp;  // P_GLOBAL: this thread's p chunks, [NCH][NT]
    __device__ __forceinline__ void init(unsigned taddr, float*) {
        const int warp = threadIdx.x >> 5;
        base = taddr + ((unsigned)(warp & 3) << 21) + (unsigned)((warp >> 2) * G::TM_WORDS);
    }
    __device__ __forceinline__ unsigned addr(ChunkId c) const {
        const int a = (G::P_GLOBAL && c.a > kP) ? c.a - 1 : c.a;
        return base + (unsigned)(2 * G::E * a + 4 * c.q);
    }
    // the four arrays' chunk q, in the order q_x, q_y, chi, p.  with_p false: p is not used, and not read
    // from global memory
    __device__ __forceinline__ void load_all(float4 (&v)[4], int q, bool with_p = true) const {
        if constexpr (G::P_GLOBAL) {
            v[3] = with_p ? __ldcg(gp + q * G::NT) : make_float4(0.f, 0.f, 0.f, 0.f);
            float4 t[3];
            load(t, {{kQx, q}, {kQy, q}, {kChi, q}});
            v[0] = t[0], v[1] = t[1], v[2] = t[2];
        } else {
            load(v, {{kQx, q}, {kQy, q}, {kChi, q}, {kP, q}});
        }
    }
    template <int K>
    __device__ __forceinline__ void load(float4 (&v)[K], const ChunkId (&c)[K]) const {
        unsigned w[4 * K];
        static_assert(K >= 1 && K <= 4, "compiled block sizes");
        if constexpr (K == 1) {
            asm volatile("{\n\t" PCS_TMEM_LD "{%0,%1,%2,%3}, [%4];\n\t" PCS_TMEM_WAIT "\n\t}"
                         : PCS_OUT4(0)
                         : "r"(addr(c[0])));
        } else if constexpr (K == 2) {
            asm volatile("{\n\t" PCS_TMEM_LD "{%0,%1,%2,%3}, [%8];\n\t" PCS_TMEM_LD "{%4,%5,%6,%7}, [%9];\n\t" PCS_TMEM_WAIT
                         "\n\t}"
                         : PCS_OUT4(0), PCS_OUT4(1)
                         : "r"(addr(c[0])), "r"(addr(c[1])));
        } else if constexpr (K == 3) {
            asm volatile("{\n\t" PCS_TMEM_LD "{%0,%1,%2,%3}, [%12];\n\t" PCS_TMEM_LD "{%4,%5,%6,%7}, [%13];\n\t" PCS_TMEM_LD
                         "{%8,%9,%10,%11}, [%14];\n\t" PCS_TMEM_WAIT "\n\t}"
                         : PCS_OUT4(0), PCS_OUT4(1), PCS_OUT4(2)
                         : "r"(addr(c[0])), "r"(addr(c[1])), "r"(addr(c[2])));
        } else {
            asm volatile("{\n\t" PCS_TMEM_LD "{%0,%1,%2,%3}, [%16];\n\t" PCS_TMEM_LD "{%4,%5,%6,%7}, [%17];\n\t" PCS_TMEM_LD
                         "{%8,%9,%10,%11}, [%18];\n\t" PCS_TMEM_LD "{%12,%13,%14,%15}, [%19];\n\t" PCS_TMEM_WAIT "\n\t}"
                         : PCS_OUT4(0), PCS_OUT4(1), PCS_OUT4(2), PCS_OUT4(3)
                         : "r"(addr(c[0])), "r"(addr(c[1])), "r"(addr(c[2])), "r"(addr(c[3])));
        }
#pragma unroll
        for (int k = 0; k < K; ++k)
            v[k] = make_float4(__uint_as_float(w[4 * k]), __uint_as_float(w[4 * k + 1]), __uint_as_float(w[4 * k + 2]),
                               __uint_as_float(w[4 * k + 3]));
    }
    __device__ __forceinline__ void st(int a, int q, float4 v) const {
        if (G::P_GLOBAL && a == kP) {
            __stcg(gp + q * G::NT, v);
            return;
        }
        asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1,%2,%3,%4};" ::"r"(addr({a, q})),
                     "r"(__float_as_uint(v.x)), "r"(__float_as_uint(v.y)), "r"(__float_as_uint(v.z)),
                     "r"(__float_as_uint(v.w)));
    }
    __device__ __forceinline__ void wait_st() const { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
};

template <class G>
struct StShared {
    float4* base;  // [4 arrays x NCH][NT]
    float4* gp;    // unused
    __device__ __forceinline__ void init(unsigned, float* mem) {
        base = reinterpret_cast<float4*>(mem) + threadIdx.x;
    }
    __device__ __forceinline__ void load_all(float4 (&v)[4], int q, bool = true) const {
        load(v, {{kQx, q}, {kQy, q}, {kChi, q}, {kP, q}});
    }
    template <int K>
    __device__ __forceinline__ void load(float4 (&v)[K], const ChunkId (&c)[K]) const {
#pragma unroll
        for (int k = 0; k < K; ++k) v[k] = base[(c[k].a * G::NCH + c[k].q) * G::NT];
    }
    __device__ __forceinline__ void st(int a, int q, float4 v) const { base[(a * G::NCH + q) * G::NT] = v; }
    __device__ __forceinline__ void wait_st() const {}
};

// ------------------------------------------------------------------ kernel body

// Scale of the W p channel: the power of two at or below 1/lambda, in [16, 65536].
__device__ __forceinline__ float pair_scale(float sigma, float inv_den) {
    const float r = (1.0f - inv_den) / (sigma * inv_den);  // 1 / lambda
    const float p2 = __uint_as_float(__float_as_uint(r) & 0x7f800000u);
    return fminf(65536.0f, fmaxf(16.0f, p2));
}

template <class G>
struct PairCtx {
    using State = typename std::conditional<G::TMEM, StTmem<G>, StShared<G>>::type;
    unsigned char* spec;  // [N/2 row pairs][2 PC units]
    unsigned char* rows;  // row-transform scratch, 8 N bytes per group
    float2* stw;          // stage twiddles
    float* slots;         // [NG + 1][N] (not with SLOT_GLOBAL)
    int* word;            // 16 bytes: tensor-memory address / schedule decision
    State st;
    int crank;
};

template <class G>
__device__ __forceinline__ void pair_ctx_init(PairCtx<G>& cx, unsigned char* smem_raw, const float2* __restrict__ twid) {
    cx.spec = smem_raw;
    cx.rows = cx.spec + G::SPEC_BYTES;
    cx.stw = reinterpret_cast<float2*>(cx.rows + G::ROWS_BYTES);
    float* f = reinterpret_cast<float*>(cx.stw + G::TW);
    float* state = f;
    f += G::STATE_BYTES / sizeof(float);
    cx.slots = f;
    if (!G::SLOT_GLOBAL) f += (G::NG + 1) * G::N;
    cx.word = reinterpret_cast<int*>(f);
    StageTw<G::N, G::E>::fill(cx.stw, twid, 1, threadIdx.x, G::NT);
    cx.crank = (G::C == 1) ? 0 : (int)cg::this_cluster().block_rank();
    unsigned taddr = 0;
    if constexpr (G::TMEM) {
        if (threadIdx.x < 32) {
            asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(cx.word)),
                         "n"(G::TMEM_COLS)
                         : "memory");
            asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
        }
        __syncthreads();
        taddr = *reinterpret_cast<volatile unsigned*>(cx.word);
    }
    cx.st.init(taddr, state);
    __syncthreads();  // twiddles; the word may be reused
}

template <class G>
__device__ __forceinline__ void pair_ctx_release(const PairCtx<G>& cx) {
    if constexpr (G::TMEM) {
        __syncthreads();
        if (threadIdx.x < 32)  // warp 0: its base is the allocation's address
            asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(cx.st.base), "n"(G::TMEM_COLS));
    }
}

// Byte offset of the 16-byte unit (re, re, im, im) of row pair j in column kx (mirror 0) or W - kx (1)
// of pair cl.
template <int PC>
__device__ __forceinline__ int pair_unit(int j, int cl, int mirror) {
    return j * (32 * PC) + 16 * ((mirror ? PC + (cl ^ 4) : cl) ^ (j & 7));
}

// Lane indices of a gather or scatter: g and T - g as values of their own.  The mirror columns'
// addresses must not be formed as (base - g ...) + constant: the constant would become the
// instruction's immediate offset, and a shared::cluster address below zero before that addition
// does not wrap (an illegal address).
struct PairLane {
    int g, m;
};
template <class G>
__device__ __forceinline__ PairLane pair_lane(int g) {
    return PairLane{fresh(g), fresh(G::T - g)};
}

// shared::cluster address of row pair j of the slice in spectrum column k = g + T e.
template <class G>
__device__ __forceinline__ unsigned pair_addr(unsigned spec, int j, PairLane ln, int e) {
    constexpr int T = G::T, PC = G::PC, N = G::N, M = G::M;
    const bool mirror = (e >= G::E / 2);
    if constexpr (PC % T == 0) {
        if (!mirror) {
            const int q = (T * e) / PC, cl = T * e - q * PC;
            return map_rank<G::C>(spec, q) + 16u * cl + (unsigned)pair_unit<PC>(j, ln.g, 0);
        }
        // columns W - kx of lanes g >= 1 share an owner; lane 0 (kx a multiple of T) may start the next
        const int k1 = N - T * e;                       // kx of lane 0 (M: the pair of column 0)
        const int q1 = (k1 - 1) / PC, cl1 = k1 - q1 * PC - T;  // cl of lane g: cl1 + (T - g)
        const int k0 = (k1 == M) ? 0 : k1;
        const int q0 = k0 / PC, cl0 = k0 - q0 * PC;
        unsigned a = map_rank<G::C>(spec, q1) + 16u * cl1 + (unsigned)pair_unit<PC>(j, ln.m, 1);
        if (q0 != q1 || k1 == M) {
            const unsigned a0 = map_rank<G::C>(spec, q0) + 16u * cl0 + (unsigned)pair_unit<PC>(j, 0, 1);
            a = (ln.g == 0) ? a0 : a;
        }
        return a;
    } else {
        const int k = ln.g + T * e;
        const int kx = !mirror ? k : (k == M ? 0 : ln.m + (N - T - T * e));
        const int q = kx / PC, cl = fresh(kx - q * PC);
        return map_rank<G::C>(spec, q) + (unsigned)pair_unit<PC>(j, cl, mirror ? 1 : 0);
    }
}

// Column pass of the group's pair: column kx in the low halves and, with its components swapped
// (swap(z) = i conj z), column W - kx in the high halves.  With Y(ky) = conj Z(-kx, -ky) the high
// transform is Y' = i Y, and the product of the file comment is pointwise per lane:
//   S = c2 D^2 (Z + Y),  out(kx) = D Z - i S,  i conj out(-kx, -ky) = D Y' - S,  c2 = tau H W / s
// (dtab holds D / (H W)); the inverse transform of the latter is swapped back at the store.  Odd pairs
// exchange the roles of the halves (low: kx swapped, high: W - kx plain), which only moves their
// 4-byte accesses to the other words of a unit: the two groups of a warp then share no bank.
// dk: D of this lane's elements, loaded by the caller.
// Pair 0 holds columns 0 and W/2, each its own mirror image.
template <class G>
__device__ __forceinline__ void pair_columns(const PairCtx<G>& cx, const float* __restrict__ dtab,
                                             const float* __restrict__ ddtab, float c2, float (&dk)[G::E]) {
    constexpr int N = G::N, T = G::T, E = G::E;
    const int tid = fresh((int)threadIdx.x);
    const int g = tid % T, cl = tid / T;
    const int kx = cx.crank * G::PC + cl;
    const ColBuf<G::PC> buf{cx.spec, cl};
    const int w0 = (cl & 1) * 2, w1 = 2 - w0;  // words of a unit: re, im (odd pairs: im, re)
    C2 x[E];
#pragma unroll
    for (int e = 0; e < E; ++e) {
        const int i = g + T * e;
        const float* a = reinterpret_cast<const float*>(cx.spec + pair_unit<G::PC>(i >> 1, cl, 0)) + (i & 1);
        const float* b = reinterpret_cast<const float*>(cx.spec + pair_unit<G::PC>(i >> 1, cl, 1)) + (i & 1);
        x[e] = C2{F2(a[w0], b[w1]), F2(a[w1], b[w0])};
    }
    fft_pair<N, T, false>(x, buf, cx.stw, g);
    if (kx != 0) {
        const float sg = (cl & 1) ? -1.0f : 1.0f;
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const float c = c2 * dk[e] * dk[e], cs = sg * c;
            const float lx = x[e].x.lo(), hx = x[e].x.hi(), ly = x[e].y.lo(), hy = x[e].y.hi();
            const float A = fmaf(-sg, hx, ly), B = fmaf(sg, hy, lx);
            x[e] = C2{F2(fmaf(dk[e], lx, cs * A), fmaf(dk[e], hx, -c * B)), F2(fmaf(dk[e], ly, -cs * B), fmaf(dk[e], hy, -c * A))};
        }
    } else {
        // through the pair's buffer, so that nothing of this rare path adds to the registers of the
        // other: a lane takes ky and -ky together (in place), D(-ky) = D(ky)
        const unsigned gm = group_mask<T>(tid & 31);
        auto b = [buf](int i) -> float4& { return *reinterpret_cast<float4*>(buf.unit(i)); };  // (Z re, Y' re, Z im, Y' im)
        __syncwarp(gm);
#pragma unroll
        for (int e = 0; e < E; ++e) b(g + T * e) = make_float4(x[e].x.lo(), x[e].x.hi(), x[e].y.lo(), x[e].y.hi());
        __syncwarp(gm);
#pragma unroll 2
        for (int ky = g; ky <= N / 2; ky += T) {
            const int km = (N - ky) % N;
            const float4 u = b(ky), v = b(km);
            const float dm0 = __ldg(dtab + ky), dd = __ldg(ddtab + ky);
            const float d0 = dm0 + dd, dm = dm0 - dd;  // D(ky, 0), D(ky, W/2)
            const float c0 = c2 * d0 * d0, cm = c2 * dm * dm;
            const float s0r = c0 * (u.x + v.x), s0i = c0 * (u.z - v.z);  // of ky; of -ky: (s0r, -s0i)
            const float smr = cm * (u.w + v.w), smi = cm * (v.y - u.y);  // of ky; of -ky: (smr, -smi)
            b(ky) = make_float4(fmaf(d0, u.x, s0i), fmaf(dm, u.y, -smr), fmaf(d0, u.z, -s0r), fmaf(dm, u.w, -smi));
            if (km != ky)
                b(km) = make_float4(fmaf(d0, v.x, -s0i), fmaf(dm, v.y, -smr), fmaf(d0, v.z, -s0r), fmaf(dm, v.w, smi));
        }
        __syncwarp(gm);
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const float4 u = b(g + T * e);
            x[e] = C2{F2(u.x, u.y), F2(u.z, u.w)};
        }
    }
    __syncwarp();
    fft_pair<N, T, true>(x, buf, cx.stw, fresh(g));
    __syncwarp();
    const int g2 = fresh(g), cl2 = fresh(cl);
#pragma unroll
    for (int e = 0; e < E; ++e) {
        const int i = g2 + T * e;
        float* a = reinterpret_cast<float*>(cx.spec + pair_unit<G::PC>(i >> 1, cl2, 0)) + (i & 1);
        float* b = reinterpret_cast<float*>(cx.spec + pair_unit<G::PC>(i >> 1, cl2, 1)) + (i & 1);
        a[w0] = x[e].x.lo();
        a[w1] = x[e].y.lo();
        b[w0] = x[e].y.hi();
        b[w1] = x[e].x.hi();
    }
}

// Row slots: elements 2q, 2q + 1 of this lane (8 bytes per lane, a group's lanes contiguous).
template <class G>
struct PairSlots {
    unsigned up, dn;   // own slot (boundary above the group's rows); the next group's (shared::cluster)
    float *gup, *gdn;  // SLOT_GLOBAL: the same as global rows
    int g;
    __device__ __forceinline__ float2 ld_up(int q) const {
        if constexpr (G::SLOT_GLOBAL) {
            return __ldcg(reinterpret_cast<const float2*>(gup) + q * G::T + g);
        } else {
            return ld_cluster2<1>(up + (unsigned)(q * G::T * 8));
        }
    }
    __device__ __forceinline__ float2 ld_dn(int q) const {
        if constexpr (G::SLOT_GLOBAL) {
            return __ldcg(reinterpret_cast<const float2*>(gdn) + q * G::T + g);
        } else {
            return ld_cluster2<G::C>(dn + (unsigned)(q * G::T * 8));
        }
    }
    __device__ __forceinline__ void st_up(int q, float2 v) const {
        if constexpr (G::SLOT_GLOBAL) {
            __stcg(reinterpret_cast<float2*>(gup) + q * G::T + g, v);
        } else {
            st_cluster2<1>(up + (unsigned)(q * G::T * 8), v);
        }
    }
    __device__ __forceinline__ void st_dn(int q, float2 v) const {
        if constexpr (G::SLOT_GLOBAL) {
            __stcg(reinterpret_cast<float2*>(gdn) + q * G::T + g, v);
        } else {
            st_cluster2<G::C>(dn + (unsigned)(q * G::T * 8), v);
        }
    }
};

// p in thread order (P_GLOBAL) to its rows.
template <class G>
__device__ __forceinline__ void pair_save_p(const PairCtx<G>& cx, float* p) {
#pragma unroll 1
    for (int q = 0; q < G::NCH; ++q) {
        const float4 v = __ldcg(cx.st.gp + q * G::NT);
        float* o = p + G::T * 2 * q;
        __stcg(o, v.x);
        __stcg(o + G::N, v.y);
        __stcg(o + G::T, v.z);
        __stcg(o + G::T + G::N, v.w);
    }
}

// Bit e of the mask as 0.0f or the value v.
__device__ __forceinline__ float bit_sel(unsigned bits, int e, float v) { return ((bits >> e) & 1u) ? v : 0.0f; }

// Iterations [it_b, it_e) of slice s: a zero start when it_b = 0 (and no resume), else a
// continuation from the stored state: chi_{n-1} (in the chibar scratch), p_n, q_n.
// P_GLOBAL: in the last pass chi goes where other threads' p lies.  Plain launches load p as ever and store
// chi after a CTA barrier; scheduled ones do not load it.  Each way is the one that costs its kernel
// nothing (15 slices of 384 x 384, us per iteration: 48.5 with the two racing on values that nobody uses,
// 48.3 and 49.4 the two ways; 32 slices, isotropic, on the schedule: 113.7, 114.7 and 113.8).
template <class G, bool SCHED>
__device__ __forceinline__ void pair_run_slice(PairCtx<G>& cx, const PDParams& prm, int s, int it_b, int it_e) {
    constexpr int N = G::N, T = G::T, E = G::E, NCH = G::NCH, C = G::C;
    constexpr unsigned gm = 0xffffffffu;  // the groups of a warp run in step
    constexpr bool CHI_LATE = G::P_GLOBAL && !SCHED;
    const int lane = threadIdx.x & 31;
    const int grp = threadIdx.x / T;
    const int g = lane % T;
    const int src_left = (g == 0) ? lane + (T - 1) : lane - 1;
    const int src_right = (g == T - 1) ? lane - (T - 1) : lane + 1;
    const int i0 = cx.crank * G::R + 2 * grp;  // the group's rows i0 (a), i0 + 1 (b)
    const bool has_up = i0 > 0, has_down = i0 + 2 < N;
    const size_t row0 = (size_t)s * (N * N) + (size_t)i0 * N + g;  // element e of row a at row0 + T e
    const float sigma = prm.sigma, tau = prm.tau;
    const float inv_den = slice_inv_den(prm, s);
    const float scale = pair_scale(sigma, inv_den);
    const float tau_s = tau / scale;
    const float c2 = tau_s * (float)(N * N);
    const unsigned spec = smem_u32(cx.spec);
    PairSlots<G> slot;
    slot.g = g;
    if constexpr (G::SLOT_GLOBAL) {
        slot.gup = prm.chibar + row0 - g;
        slot.gdn = prm.chibar + row0 - g + (has_down ? 2 * N : N);  // spare: an odd row
    } else {
        const unsigned s0 = smem_u32(cx.slots) + (unsigned)(g * 8);
        const bool own = grp + 1 < G::NG || cx.crank + 1 == C;  // the slice's last group: the spare slot
        slot.up = s0 + (unsigned)(grp * N * 4);
        slot.dn = map_rank<C>(s0 + (unsigned)((own ? grp + 1 : 0) * N * 4), own ? cx.crank : cx.crank + 1);
    }
    const bool cont = prm.resume || it_b > 0;
    const int count = it_e - it_b;

    // ---- mask bits of rows a and b, and state
    unsigned mbit_a = 0, mbit_b = 0;
#pragma unroll 1
    for (int e = 0; e < E; ++e) {
        mbit_a |= (__ldg(prm.mask + row0 + T * e) ? 1u : 0u) << e;
        mbit_b |= (__ldg(prm.mask + row0 + N + T * e) ? 1u : 0u) << e;
    }
    if (E <= 16) mbit_a |= mbit_b << 16;  // one register for both
    // P_GLOBAL: p in the threads' order in chi_out's rows of the CTA (chi is on chip until the end)
    cx.st.gp = reinterpret_cast<float4*>(prm.chi + (size_t)s * (N * N) + (size_t)cx.crank * G::R * N) + threadIdx.x;
#pragma unroll 1
    for (int a = 0; a < 4; ++a) {
        const float* src = (a == kChi ? prm.chibar : a == kP ? prm.p : a == kQx ? prm.qx : prm.qy) + row0;
#pragma unroll 1
        for (int q = 0; q < NCH; ++q) {
            float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
            const float* o = src + T * 2 * q;
            if (cont) v = make_float4(__ldcg(o), __ldcg(o + N), __ldcg(o + T), __ldcg(o + T + N));
            cx.st.st(a, q, v);
        }
    }
    cx.st.wait_st();
    if constexpr (G::SLOT_GLOBAL) {
        // the chibar rows become slots: every thread of the cluster has read its chi first
        if (cont) cluster_barrier<C>();
    }
#pragma unroll 1
    for (int q = 0; q < NCH; ++q) {  // q_y of the row above (row 0 has none: phases A and C take zero there)
        float2 v = make_float2(0.f, 0.f);
        const float* o = prm.qy + row0 - (has_up ? N : 0) + T * 2 * q;
        if (cont) v = make_float2(__ldcg(o), __ldcg(o + T));
        slot.st_up(q, v);
    }

    // the field in the threads' own order, in the q_x scratch of the CTA's rows (its values are on
    // chip until the end): one 16-byte load per chunk
    __syncthreads();  // every q_x of the CTA read
    float4* fpk = reinterpret_cast<float4*>(prm.qx + (size_t)s * (N * N) + (size_t)cx.crank * G::R * N) + threadIdx.x;
#pragma unroll 1
    for (int q = 0; q < NCH; ++q) {
        const float* o = prm.field + row0 + T * 2 * q;
        __stcg(fpk + q * G::NT, make_float4(__ldg(o), __ldg(o + N), __ldg(o + T), __ldg(o + T + N)));
    }

    bool skip = cont;           // a continuation starts with phase C of its last stored p, q
    bool zero = !cont;          // v = u = 0 (zero start)
    int n = cont ? -1 : 0;
    if (count > 0) {
#pragma unroll 1
        while (true) {
            const bool last = (n == count);
            if (G::P_GLOBAL && last) {  // chi_out is about to be written
                pair_save_p<G>(cx, prm.p + row0);
                __syncthreads();
            }
            C2 x[E];
            if (!skip) {
                // ================= phase A: chi, chibar, p of both rows
                if (!zero) {
                    const unsigned spec_a = fresh(spec);
                    const PairLane ln = pair_lane<G>(g);
                    const int j = i0 >> 1;
#pragma unroll
                    for (int e = 0; e < E; ++e) {
                        const ulonglong2 t = ld_cluster_pair<C>(pair_addr<G>(spec_a, j, ln, e));
                        x[e] = C2{F2(t.x), F2(t.y)};
                    }
                } else {
#pragma unroll
                    for (int e = 0; e < E; ++e) x[e] = C2{F2(0.f, 0.f), F2(0.f, 0.f)};
                }
                fft_pair<N, T, true>(x, RowBuf{cx.rows + fresh(grp) * (8 * N)}, cx.stw, fresh(g));  // x = (s v, u)
                {
                    const F2 m_tau(-tau, -tau), m_tau_s(-tau_s, -tau_s), inv(inv_den, inv_den);
                    const unsigned ma = fresh(mbit_a), mb = (E <= 16) ? ma >> 16 : fresh(mbit_b);
                    const float4* fp = fresh(fpk);
                    float4 f0 = __ldcg(fp), f1 = __ldcg(fp + G::NT);  // two chunks ahead
                    float2 u0{}, u1{};
                    if (G::SLOT_GLOBAL) u0 = slot.ld_up(0), u1 = slot.ld_up(1);
                    float pla = 0.f, plb = 0.f;
#pragma unroll
                    for (int q = 0; q < NCH; ++q) {
                        float4 v[4];
                        cx.st.load_all(v, q, CHI_LATE || !last);
                        const float2 qu = G::SLOT_GLOBAL ? u0 : slot.ld_up(q);  // q_y of the row above row a
                        u0 = u1;
                        if (G::SLOT_GLOBAL && q + 2 < NCH) u1 = slot.ld_up(q + 2);
                        const float4 f = f0;
                        f0 = f1;
                        if (q + 2 < NCH) f1 = __ldcg(fp + (q + 2) * G::NT);
                        F2 cn[2], pn[2];
                        float2 slot_v;
#pragma unroll
                        for (int c = 0; c < 2; ++c) {
                            const int e = 2 * q + c;
                            const float qxa = c ? v[0].z : v[0].x, qxb = c ? v[0].w : v[0].y;
                            const float qya = c ? v[1].z : v[1].x, qyb = c ? v[1].w : v[1].y;
                            const F2 c0(c ? v[2].z : v[2].x, c ? v[2].w : v[2].y), p0(c ? v[3].z : v[3].x, c ? v[3].w : v[3].y);
                            const float sha = __shfl_sync(gm, qxa, src_left), shb = __shfl_sync(gm, qxb, src_left);
                            // q_x of the pixel to the left (the first column has none)
                            const F2 ql(g == 0 ? pla : sha, g == 0 ? plb : shb);
                            pla = sha;
                            plb = shb;
                            const float up = has_up ? (c ? qu.y : qu.x) : 0.f;
                            const F2 d2 = (ql - F2(qxa, qxb)) + (F2(up, qya) - F2(qya, qyb));
                            cn[c] = fma2(m_tau, d2, fma2(m_tau_s, x[e].x, c0));
                            const F2 bar = (cn[c] + cn[c]) - c0;
                            F2 sw(bit_sel(ma, e, sigma), bit_sel(mb, e, sigma));
                            if (prm.weight) {
                                const float* w = prm.weight + row0 + T * e;
                                sw = F2(sigma * __ldg(w), sigma * __ldg(w + N));
                            }
                            pn[c] = fma2(sw, x[e].y - F2(c ? f.z : f.x, c ? f.w : f.y), p0) * inv;
                            x[e].x = bar;
                            if (c == 0)
                                slot_v.x = bar.lo();
                            else
                                slot_v.y = bar.lo();
                        }
                        if (!last) {
                            cx.st.st(kChi, q, make_float4(cn[0].lo(), cn[0].hi(), cn[1].lo(), cn[1].hi()));
                            cx.st.st(kP, q, make_float4(pn[0].lo(), pn[0].hi(), pn[1].lo(), pn[1].hi()));
                            slot.st_up(q, slot_v);
                        } else if (!CHI_LATE) {
                            float* o = prm.chi + row0 + T * 2 * q;
                            __stcg(o, cn[0].lo());
                            __stcg(o + N, cn[0].hi());
                            __stcg(o + T, cn[1].lo());
                            __stcg(o + T + N, cn[1].hi());
                        }
                        if (CHI_LATE) x[2 * q].y = cn[0], x[2 * q + 1].y = cn[1];  // u is used up
                    }
                    if (CHI_LATE && last) {
                        __syncthreads();  // every thread has loaded its p
#pragma unroll
                        for (int e = 0; e < E; ++e) {
                            __stcg(prm.chi + row0 + T * e, x[e].y.lo());
                            __stcg(prm.chi + row0 + T * e + N, x[e].y.hi());
                        }
                    }
                }
                cluster_arrive<C>();
                if (last) {
                    cluster_wait<C>();
                    break;
                }
                cx.st.wait_st();
                // ================= phase B: q of both rows; q_y of row b after the wait for chibar of
                // the next group's row a (isotropic TV: the projection of row b too)
                {
                    const unsigned ma = fresh(mbit_a), mb = (E <= 16) ? ma >> 16 : fresh(mbit_b);
                    const int iso = prm.tv_iso;
                    // chibar of the pixel to the right, one element ahead
                    float na = __shfl_sync(gm, x[0].x.lo(), src_right), nb = __shfl_sync(gm, x[0].x.hi(), src_right);
#pragma unroll
                    for (int q = 0; q < NCH; ++q) {
                        float4 v[2];
                        cx.st.load(v, {{kQx, q}, {kQy, q}});
                        float vx[4], vy[4] = {v[1].x, v[1].y, v[1].z, v[1].w};
#pragma unroll
                        for (int c = 0; c < 2; ++c) {
                            const int e = 2 * q + c;
                            const float ca = x[e].x.lo(), cb = x[e].x.hi();
                            float ra = na, rb = nb;
                            if (e + 1 < E) {
                                na = __shfl_sync(gm, x[e + 1 < E ? e + 1 : e].x.lo(), src_right);
                                nb = __shfl_sync(gm, x[e + 1 < E ? e + 1 : e].x.hi(), src_right);
                            }
                            // past the last column the difference is zero (Neumann)
                            if (g == T - 1) {
                                ra = (e + 1 < E) ? na : ca;
                                rb = (e + 1 < E) ? nb : cb;
                            }
                            const float sma = bit_sel(ma, e, sigma), smb = bit_sel(mb, e, sigma);
                            const F2 bx = fma2(F2(sma, smb), F2(ra, rb) - x[e].x, F2(c ? v[0].z : v[0].x, c ? v[0].w : v[0].y));
                            vx[2 * c] = bx.lo(), vx[2 * c + 1] = bx.hi();
                            vy[2 * c] = fmaf(sma, cb - ca, vy[2 * c]);
                            tv_prox(vx[2 * c], vy[2 * c], iso);
                            if (!iso) vx[2 * c + 1] = fmin(1.0f, fmax(-1.0f, vx[2 * c + 1]));
                        }
                        cx.st.st(kQx, q, make_float4(vx[0], vx[1], vx[2], vx[3]));
                        cx.st.st(kQy, q, make_float4(vy[0], vy[1], vy[2], vy[3]));
                    }
                    cx.st.wait_st();
                    cluster_wait<C>();  // every gather of this iteration is done, too
                    float2 below[NCH];  // slots in global memory: all loads in flight at once
                    if constexpr (G::SLOT_GLOBAL) {
#pragma unroll
                        for (int q = 0; q < NCH; ++q) below[q] = slot.ld_dn(q);
                    }
#pragma unroll
                    for (int q = 0; q < NCH; ++q) {
                        const float2 dn = G::SLOT_GLOBAL ? below[q] : slot.ld_dn(q);
                        float4 v[2];
                        cx.st.load(v, {{kQx, q}, {kQy, q}});
                        const float cb0 = x[2 * q].x.hi(), cb1 = x[2 * q + 1].x.hi();
                        // below the last row the difference is zero (Neumann)
                        v[1].y = fmaf(bit_sel(mb, 2 * q, sigma), (has_down ? dn.x : cb0) - cb0, v[1].y);
                        v[1].w = fmaf(bit_sel(mb, 2 * q + 1, sigma), (has_down ? dn.y : cb1) - cb1, v[1].w);
                        tv_prox(v[0].y, v[1].y, iso);
                        tv_prox(v[0].w, v[1].w, iso);
                        if (iso) cx.st.st(kQx, q, v[0]);
                        cx.st.st(kQy, q, v[1]);
                        slot.st_dn(q, make_float2(v[1].y, v[1].w));
                    }
                    cx.st.wait_st();
                }
            }
            cluster_arrive<C>();
            // ================= phase C: forward transform of s W p + i b
            {
                const F2 m_2tau(-2.0f * tau, -2.0f * tau);
                const unsigned ma = fresh(mbit_a), mb = (E <= 16) ? ma >> 16 : fresh(mbit_b);
                float pla = 0.f, plb = 0.f;
#pragma unroll
                for (int q = 0; q < NCH; ++q) {
                    float4 v[4];
                    cx.st.load_all(v, q);
#pragma unroll
                    for (int c = 0; c < 2; ++c) {
                        const int e = 2 * q + c;
                        const float qxa = c ? v[0].z : v[0].x, qxb = c ? v[0].w : v[0].y;
                        const float qya = c ? v[1].z : v[1].x, qyb = c ? v[1].w : v[1].y;
                        const float sha = __shfl_sync(gm, qxa, src_left), shb = __shfl_sync(gm, qxb, src_left);
                        const F2 ql(g == 0 ? pla : sha, g == 0 ? plb : shb);
                        pla = sha;
                        plb = shb;
                        // row a's q_y from above follows after the wait
                        const F2 d2 = (ql - F2(qxa, qxb)) + (F2(0.f, qya) - F2(qya, qyb));
                        F2 sw(bit_sel(ma, e, scale), bit_sel(mb, e, scale));
                        if (prm.weight) {
                            const float* w = prm.weight + row0 + T * e;
                            sw = F2(scale * __ldg(w), scale * __ldg(w + N));
                        }
                        x[e].x = sw * F2(c ? v[3].z : v[3].x, c ? v[3].w : v[3].y);
                        x[e].y = fma2(m_2tau, d2, F2(c ? v[2].z : v[2].x, c ? v[2].w : v[2].y));
                    }
                }
                cluster_wait<C>();  // q_y of the row above row a
                const float up2 = has_up ? -2.0f * tau : 0.f;
                float2 above[NCH];
                if constexpr (G::SLOT_GLOBAL) {
#pragma unroll
                    for (int q = 0; q < NCH; ++q) above[q] = slot.ld_up(q);
                }
#pragma unroll
                for (int q = 0; q < NCH; ++q) {
                    const float2 qu = G::SLOT_GLOBAL ? above[q] : slot.ld_up(q);
                    x[2 * q].y = F2(fmaf(up2, qu.x, x[2 * q].y.lo()), x[2 * q].y.hi());
                    x[2 * q + 1].y = F2(fmaf(up2, qu.y, x[2 * q + 1].y.lo()), x[2 * q + 1].y.hi());
                }
                fft_pair<N, T, false>(x, RowBuf{cx.rows + fresh(grp) * (8 * N)}, cx.stw, fresh(g));
                const unsigned spec_c = fresh(spec);
                const PairLane ln = pair_lane<G>(g);
                const int j = i0 >> 1;
#pragma unroll
                for (int e = 0; e < E; ++e)
                    st_cluster_pair<C>(pair_addr<G>(spec_c, j, ln, e), make_ulonglong2(x[e].x.v, x[e].y.v));
            }
            cluster_arrive<C>();
            {
                // D of this lane's column elements, in flight during the barrier
                float dk[E];
                const float* d = fresh(prm.dtab) + (size_t)(cx.crank * G::PC + grp) * N + g;
#pragma unroll
                for (int e = 0; e < E; ++e) dk[e] = __ldg(d + T * e);
                cluster_wait<C>();
                pair_columns<G>(cx, prm.dtab, prm.ddtab, c2, dk);
            }
            cluster_barrier<C>();
            skip = false;
            zero = false;
            ++n;
        }
    } else {
        // no iterations: chi = 0 (the zero start)
        if (G::P_GLOBAL) {
            pair_save_p<G>(cx, prm.p + row0);
            __syncthreads();
        }
#pragma unroll 1
        for (int t = 0; t < 2 * E; ++t) __stcg(prm.chi + row0 + (t / E) * N + T * (t % E), 0.f);
        cluster_barrier<C>();
    }
    // ---- the state, for diagnostics and continuations: chi_{N-1} (chibar scratch), p, q
#pragma unroll 1
    for (int a = 0; a < 4; ++a) {
        if (G::P_GLOBAL && a == kP) continue;  // saved before chi_out was written
        float* dst = (a == kChi ? prm.chibar : a == kP ? prm.p : a == kQx ? prm.qx : prm.qy) + row0;
#pragma unroll 1
        for (int q = 0; q < NCH; ++q) {
            float4 v[1];
            cx.st.load(v, {{a, q}});
            float* o = dst + T * 2 * q;
            __stcg(o, v[0].x);
            __stcg(o + N, v[0].y);
            __stcg(o + T, v[0].z);
            __stcg(o + T + N, v[0].w);
        }
    }
}

// SCHED: run the balanced schedule's segments (pd_cluster_kernel).
template <class G, bool SCHED = false>
__global__ void __launch_bounds__(G::NT, G::MINB) pd_pair_kernel(PDParams prm) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    PairCtx<G> cx;
    pair_ctx_init<G>(cx, smem_raw, prm.twid);
    const int cid = blockIdx.x / G::C;
    if constexpr (!SCHED) {
#pragma unroll 1
        for (int s = cid; s < prm.S; s += gridDim.x / G::C) {
            if (prm.active && __ldg(prm.active + s) == 0) continue;  // same decision in every CTA of the cluster
            pair_run_slice<G, false>(cx, prm, s, 0, prm.n_iter);
        }
    } else {
#pragma unroll 1
        for (int k = __ldg(prm.sched_off + cid); k < __ldg(prm.sched_off + cid + 1); ++k) {
            const int4 sg = __ldg(prm.sched + k);
            if (sg.w & 1) {
                // the slice's first part runs on another cluster: CTA 0 waits (bounded) and the
                // cluster follows its decision, so that every CTA proceeds or every CTA returns
                if (cx.crank == 0 && threadIdx.x == 0)
                    *cx.word = wait_flag(prm.seg_flags + sg.x, prm.wait_limit) ? 1 : 0;
                cluster_barrier<G::C>();
                int ok;
                if constexpr (G::C == 1) {
                    ok = *cx.word;
                } else {
                    ok = *cg::this_cluster().map_shared_rank(cx.word, 0);
                }
                cluster_barrier<G::C>();  // every CTA has read CTA 0's decision
                if (!ok) {
                    if (cx.crank == 0 && threadIdx.x == 0) atomicExch(prm.err, 1);
                    break;
                }
                if (threadIdx.x == 0) (void)wait_flag(prm.seg_flags + sg.x, prm.wait_limit);  // this CTA's acquire
                __syncthreads();
            }
            pair_run_slice<G, true>(cx, prm, sg.x, sg.y, sg.z);
            const int4 done = __ldg(prm.sched + k);
            if (done.w & 2) {
                cluster_barrier<G::C>();  // every CTA's state is written
                if (cx.crank == 0 && threadIdx.x == 0) set_flag(prm.seg_flags + done.x);
            }
        }
    }
    cluster_barrier<G::C>();  // no CTA leaves while a peer may still gather from it
    pair_ctx_release<G>(cx);
}

}  // namespace pcs
