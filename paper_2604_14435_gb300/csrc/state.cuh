// Shared-memory state vector of the Ry + CZ-ring ansatz, used by the term
// kernels, the fidelity and the optimizer.  Ansatz (Sec. 2.3 / Sec. 3, Ry + CZ
// form): Ry layer alpha[0..n), then d times { CZ ring ; Ry layer
// alpha[l*n .. l*n+n) }, with Ry(t) = [[cos t/2, -sin t/2], [sin t/2, cos t/2]]
// and the CZ ring CZ(q,q+1), q < n-1, plus CZ(n-1,0) when n >= 3.
#pragma once

#include <cuda_fp16.h>

#include <cuda_runtime.h>

namespace dvqls {

template <typename R>
struct V2;
template <>
struct V2<float> {
    using t = float2;
};
template <>
struct V2<double> {
    using t = double2;
};

__device__ __forceinline__ int czring_parity(int i, int n) {
    int p = __popc(i & (i >> 1) & ((1 << (n - 1)) - 1));
    if (n >= 3) p += (i >> (n - 1)) & i & 1;
    return p & 1;
}

// The state builders below form psi = V(alpha_s)|0> and end with a barrier.  cs
// holds (cos, sin) of the half angles: [0, P) at alpha, [P, 2P) at alpha + pi/2,
// [2P, 3P) at alpha - pi/2; shift s selects alpha (s = 0), alpha + pi/2 e_k
// (s = 2k+1) or alpha - pi/2 e_k (s = 2k+2).  scs receives the P (cos, sin) pairs
// used.
// Barrier over the threads that build a state: the whole block (bar = 0) or
// the NTH threads that share named barrier `bar`.
__device__ __forceinline__ void group_sync(int bar, int NTH) {
    if (bar == 0) __syncthreads();
    else asm volatile("bar.sync %0, %1;" ::"r"(bar), "r"(NTH) : "memory");
}

// Shifted state s in precision R, real (every gate of the ansatz is), multiplied
// by `scale`, by threads t = 0 .. NTH-1 of a group: psi[0 .. 2^n), scs[0 .. P) as
// (cos, sin).  The CZ ring (diagonal) is applied while loading a layer's first
// pass; the Ry rotations of qubits q and q+1 are fused into one pass over groups
// of four amplitudes, so a layer takes ceil(n/2) passes and barriers.
template <typename R>
__device__ inline void build_state_real(R* psi, typename V2<R>::t* scs, int n, int d, int P, const double2* cs, int s,
                                        int t, int NTH, int bar, R scale) {
    using R2 = typename V2<R>::t;
    const int N = 1 << n;
    int k = -1, which = 0;
    if (s > 0) {
        k = (s - 1) >> 1;
        which = ((s - 1) & 1) ? 2 : 1;
    }
    for (int a = t; a < P; a += NTH) {
        const double2 v = cs[(a == k ? which : 0) * P + a];
        R2 r;
        r.x = (R)v.x;
        r.y = (R)v.y;
        scs[a] = r;
    }
    group_sync(bar, NTH);
    for (int i = t; i < N; i += NTH) {  // initial Ry layer on |0>: a product state
        R v = scale;
        for (int q = 0; q < n; ++q) v *= ((i >> q) & 1) ? scs[q].y : scs[q].x;
        psi[i] = v;
    }
    group_sync(bar, NTH);
    for (int layer = 1; layer <= d; ++layer) {
        for (int q = 0; q < n; q += 2) {
            const R c0 = scs[layer * n + q].x, s0 = scs[layer * n + q].y;
            if (q + 1 < n) {
                const R c1 = scs[layer * n + q + 1].x, s1 = scs[layer * n + q + 1].y;
                for (int p = t; p < N / 4; p += NTH) {
                    const int i00 = ((p >> q) << (q + 2)) | (p & ((1 << q) - 1));
                    const int i01 = i00 | (1 << q), i10 = i00 | (2 << q), i11 = i00 | (3 << q);
                    R a = psi[i00], b = psi[i01], c = psi[i10], e = psi[i11];
                    if (q == 0) {  // the CZ ring, applied while loading the layer's first pass
                        if (czring_parity(i00, n)) a = -a;
                        if (czring_parity(i01, n)) b = -b;
                        if (czring_parity(i10, n)) c = -c;
                        if (czring_parity(i11, n)) e = -e;
                    }
                    const R a1 = c0 * a - s0 * b, b1 = s0 * a + c0 * b;  // Ry on qubit q
                    const R c2 = c0 * c - s0 * e, e1 = s0 * c + c0 * e;
                    psi[i00] = c1 * a1 - s1 * c2;  // Ry on qubit q + 1
                    psi[i10] = s1 * a1 + c1 * c2;
                    psi[i01] = c1 * b1 - s1 * e1;
                    psi[i11] = s1 * b1 + c1 * e1;
                }
            } else {
                for (int p = t; p < N / 2; p += NTH) {
                    const int i0 = ((p >> q) << (q + 1)) | (p & ((1 << q) - 1)), i1 = i0 | (1 << q);
                    R a = psi[i0], b = psi[i1];
                    if (q == 0) {
                        if (czring_parity(i0, n)) a = -a;
                        if (czring_parity(i1, n)) b = -b;
                    }
                    psi[i0] = c0 * a - s0 * b;
                    psi[i1] = s0 * a + c0 * b;
                }
            }
            group_sync(bar, NTH);
        }
    }
}

// ---- Register-resident real state build for a group of 256 threads.
//
// The group holds 2^n = 256 A amplitudes with A per thread.  Mapping M1:
// i = (r << 8) | (warp << 5) | lane (qubits 0-4 on lanes, 5-7 on warps, 8+ on
// registers); mapping M2: i = (r << 8) | (lane << 3) | warp (qubits 3-7 on
// lanes, 0-2 on warps).  A qubit on a lane bit rotates with one shuffle, on a
// register bit in place; the warp-bit qubits of a layer are reached by one
// transpose through shared memory (padded by one word per 32, conflict-free),
// alternating M1 and M2 from layer to layer.  Ry gates of a layer commute, so
// the layer splits across the transpose; the CZ ring is a sign per amplitude.

// The tensor-core operand pair of x: hi = RN_fp16(x) in the low half-word and
// RN_fp16(2 (x - hi)) -- the low part, doubled -- in the high one (x - hi is
// exact in FP32).  x ~ hi + (high half) / 2.
__device__ __forceinline__ uint32_t split_h2l(float x) {
    const __half h = __float2half_rn(x);
    const __half l = __float2half_rn(2.f * (x - __half2float(h)));
    return (uint32_t)__half_as_ushort(h) | ((uint32_t)__half_as_ushort(l) << 16);
}

__device__ __forceinline__ int st_index(int M, int r, int w, int lane) {
    return M == 0 ? (r << 8) | (w << 5) | lane : (r << 8) | (lane << 3) | w;
}
__device__ __forceinline__ int st_pad(int i) { return i + (i >> 5); }

// Ry(theta) on a register bit in scaled form.  With c = cos(theta/2) and
// s = sin(theta/2), Ry = c [[1, -t], [t, 1]] (t = s/c) when |c| >= |s|, else
// s [[u, -1], [1, u]] (u = c/s): the bracketed matrix takes one FMA per
// amplitude (two per pair instead of four), and the factor (c or s) is
// applied once for all the rotations of a pass.  |t|, |u| <= 1 keeps every
// step as well conditioned as the plain rotation.
struct RyScaled {
    float r, fac;
    int sform;
};
__device__ __forceinline__ RyScaled ry_scaled(float c, float s) {
    RyScaled q;
    if (fabsf(c) >= fabsf(s)) {
        q.r = s / c;
        q.fac = c;
        q.sform = 0;
    } else {
        q.r = c / s;
        q.fac = s;
        q.sform = 1;
    }
    return q;
}
// The bracketed matrix on register bit kb (a compile-time constant in the
// unrolled callers) of the A amplitudes v.
template <int A>
__device__ __forceinline__ void ry_regs_scaled(float (&v)[A], int kb, float r, int sform) {
    if (sform) {
#pragma unroll
        for (int i = 0; i < A; ++i)
            if (!((i >> kb) & 1)) {
                const float a0 = v[i], a1 = v[i | (1 << kb)];
                v[i] = fmaf(r, a0, -a1);
                v[i | (1 << kb)] = fmaf(r, a1, a0);
            }
    } else {
#pragma unroll
        for (int i = 0; i < A; ++i)
            if (!((i >> kb) & 1)) {
                const float a0 = v[i], a1 = v[i | (1 << kb)];
                v[i] = fmaf(-r, a1, a0);
                v[i | (1 << kb)] = fmaf(r, a0, a1);
            }
    }
}

// Ry(theta) on the qubit of lane bit b: v' = c v -+ s v_partner.
__device__ __forceinline__ float ry_lane(float v, int lane, int b, float c, float s) {
    const float p = __shfl_xor_sync(0xffffffffu, v, 1 << b);
    return fmaf(c, v, ((lane >> b) & 1) ? s * p : -s * p);
}

// Final store of an amplitude: packed FP16 (hi, 2 lo) (PACK) or FP32.
template <bool PACK>
__device__ __forceinline__ void st_out(void* psi, int i, float v) {
    if (PACK) reinterpret_cast<uint32_t*>(psi)[i] = split_h2l(v);
    else reinterpret_cast<float*>(psi)[i] = v;
}

template <int A, int LOGA, bool PACK>
__device__ void state_regs_multiwarp(void* psi, float* scr0, float* scr1, const float2* scs, int n, int d, int t,
                                     int bar, float scale) {
    const int lane = t & 31, w = t >> 5;
    float v[A];
#pragma unroll
    for (int r = 0; r < A; ++r) {  // initial Ry layer on |0>: a product state
        const int i = st_index(0, r, w, lane);
        float x = scale;
        for (int q = 0; q < n; ++q) x *= ((i >> q) & 1) ? scs[q].y : scs[q].x;
        v[r] = x;
    }
    int M = 0, k = 0;
    for (int layer = 1; layer <= d; ++layer) {
        const float2* ang = scs + layer * n;
#pragma unroll
        for (int r = 0; r < A; ++r)
            if (czring_parity(st_index(M, r, w, lane), n)) v[r] = -v[r];
        const int qlane = M == 0 ? 0 : 3;  // qubit of lane bit 0
#pragma unroll
        for (int b = 0; b < 5; ++b) {
            const float c = ang[qlane + b].x, sn = ang[qlane + b].y;
#pragma unroll
            for (int r = 0; r < A; ++r) v[r] = ry_lane(v[r], lane, b, c, sn);
        }
#pragma unroll
        for (int kb = 0; kb < LOGA; ++kb) {  // register-bit qubits 8 + kb
            const float c = ang[8 + kb].x, sn = ang[8 + kb].y;
#pragma unroll
            for (int r = 0; r < A; ++r)
                if (!((r >> kb) & 1)) {
                    const float a0 = v[r], a1 = v[r | (1 << kb)];
                    v[r] = c * a0 - sn * a1;
                    v[r | (1 << kb)] = sn * a0 + c * a1;
                }
        }
        // transpose to the other mapping through scratch buffer k
        float* scr = k ? scr1 : scr0;
#pragma unroll
        for (int r = 0; r < A; ++r) scr[st_pad(st_index(M, r, w, lane))] = v[r];
        group_sync(bar, 256);
        M ^= 1;
        k ^= 1;
#pragma unroll
        for (int r = 0; r < A; ++r) v[r] = scr[st_pad(st_index(M, r, w, lane))];
        // the qubits that were on warp bits are now on lanes: M1 lanes 0-2 = qubits 0-2,
        // M2 lanes 2-4 = qubits 5-7
        const int b0 = M == 0 ? 0 : 2, q0 = M == 0 ? 0 : 5;
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            const float c = ang[q0 + j].x, sn = ang[q0 + j].y;
#pragma unroll
            for (int r = 0; r < A; ++r) v[r] = ry_lane(v[r], lane, b0 + j, c, sn);
        }
    }
#pragma unroll
    for (int r = 0; r < A; ++r) st_out<PACK>(psi, st_index(M, r, w, lane), v[r]);
    group_sync(bar, 256);
}

// n <= 10: one warp holds the whole state (i = (r << 5) | lane; for n < 5 lane
// i is lane mod 2^n), no barrier inside.  The initial Ry layer on |0> is a
// product state: a lane factor (qubits on lane bits) times register factors
// built by doubling (qubits on register bits).  The CZ-ring signs depend only
// on the amplitude index, so they are one bit mask per lane for every layer.
template <int A, int LOGA, bool PACK>
__device__ void state_regs_warp(void* psi, const float2* scs, int n, int d, int lane, float scale) {
    const int N = 1 << n, lmask = N < 32 ? N - 1 : 31, nl = n < 5 ? n : 5, li = lane & lmask;
    float v[A];
    {
        float f = scale;  // qubits 0 .. nl - 1 on the lane bits
        for (int q = 0; q < nl; ++q) f *= ((li >> q) & 1) ? scs[q].y : scs[q].x;
        v[0] = f;
#pragma unroll
        for (int kb = 0; kb < LOGA; ++kb) {  // qubit 5 + kb on register bit kb
            const float c = scs[5 + kb].x, sn = scs[5 + kb].y;
#pragma unroll
            for (int r = 0; r < (1 << kb); ++r) {
                v[r + (1 << kb)] = v[r] * sn;
                v[r] *= c;
            }
        }
    }
    uint32_t czm = 0u;  // bit r: the CZ ring flips the sign of amplitude (r << 5) | lane
#pragma unroll
    for (int r = 0; r < A; ++r) czm |= uint32_t(czring_parity((r << 5) | li, n)) << r;
    for (int layer = 1; layer <= d; ++layer) {
        const float2* ang = scs + layer * n;
#pragma unroll
        for (int r = 0; r < A; ++r)
            v[r] = __uint_as_float(__float_as_uint(v[r]) ^ (((czm >> r) & 1u) << 31));
        for (int b = 0; b < nl; ++b) {
            const float c = ang[b].x, sb = ((lane >> b) & 1) ? ang[b].y : -ang[b].y;
#pragma unroll
            for (int r = 0; r < A; ++r) v[r] = fmaf(c, v[r], sb * __shfl_xor_sync(0xffffffffu, v[r], 1 << b));
        }
#pragma unroll
        for (int kb = 0; kb < LOGA; ++kb) {  // register-bit qubits 5 + kb
            const float c = ang[5 + kb].x, sn = ang[5 + kb].y;
#pragma unroll
            for (int r = 0; r < A; ++r)
                if (!((r >> kb) & 1)) {
                    const float a0 = v[r], a1 = v[r | (1 << kb)];
                    v[r] = c * a0 - sn * a1;
                    v[r | (1 << kb)] = sn * a0 + c * a1;
                }
        }
    }
    if (lane < N || N >= 32) {
#pragma unroll
        for (int r = 0; r < A; ++r) st_out<PACK>(psi, (r << 5) | lane, v[r]);
    }
}

// The real state of shift s, times `scale`, for a group of 256 threads (ids t,
// named barrier `bar`) into psi[0 .. 2^n), as packed FP16 (hi, 2 lo) pairs
// (split_h2l; PACK) or as FP32; n <= 12.  scratch: 2 x (2^n + 2^n / 32) floats
// of shared memory that nothing else uses meanwhile.
template <bool PACK>
__device__ inline void build_state_regs(void* psi, float* scratch, float2* scs, int n, int d, int P,
                                        const double2* cs, int s, int t, int bar, float scale) {
    int k = -1, which = 0;
    if (s > 0) {
        k = (s - 1) >> 1;
        which = ((s - 1) & 1) ? 2 : 1;
    }
    for (int a = t; a < P; a += 256) {
        const double2 v = cs[(a == k ? which : 0) * P + a];
        scs[a] = make_float2((float)v.x, (float)v.y);
    }
    group_sync(bar, 256);
    const int N = 1 << n;
    float* scr1 = scratch + N + N / 32;
    switch (n) {
        case 9: state_regs_multiwarp<2, 1, PACK>(psi, scratch, scr1, scs, n, d, t, bar, scale); return;
        case 10: state_regs_multiwarp<4, 2, PACK>(psi, scratch, scr1, scs, n, d, t, bar, scale); return;
        case 11: state_regs_multiwarp<8, 3, PACK>(psi, scratch, scr1, scs, n, d, t, bar, scale); return;
        case 12: {  // 16 amplitudes per thread would crowd the registers: gate passes in shared memory
            float* f = reinterpret_cast<float*>(psi);
            build_state_real<float>(f, scs, n, d, P, cs, s, t, 256, bar, scale);  // ends with a barrier
            if (PACK) {
                for (int i = t; i < N; i += 256) st_out<true>(psi, i, f[i]);  // in place, one word each
                group_sync(bar, 256);
            }
            return;
        }
        default: break;
    }
    if ((t >> 5) == 0) {
        const int lane = t & 31;
        switch (n) {
            case 6: state_regs_warp<2, 1, PACK>(psi, scs, n, d, lane, scale); break;
            case 7: state_regs_warp<4, 2, PACK>(psi, scs, n, d, lane, scale); break;
            case 8: state_regs_warp<8, 3, PACK>(psi, scs, n, d, lane, scale); break;
            default: state_regs_warp<1, 0, PACK>(psi, scs, n, d, lane, scale); break;  // n <= 5
        }
    }
    group_sync(bar, 256);
}

// ---- The state in 64-bit fixed point, for 256 threads, n <= 10 (FP64 precision).
//
// FP64 instructions issue at 1/64 of the FP32 rate, six integer multiply-adds
// and a shift in less time than one of them.  The state has norm
// one, so every amplitude and every cos and sin is h 2^30 + l in units of 2^-60
// (|h| <= 2^30, l in [-2^29, 2^29)), and c a + t b is six multiply-adds and a
// shift.  It is rounded at 2^-60 and leaves out the two products of low parts, a
// quarter of that unit each at most: an error of one unit at most.  An FP64 rotation
// rounds an amplitude near 2^-5 (the mean at n = 10) at 2^-58, so this is no less exact
// for amplitudes of that size; small ones lose relative accuracy, and whoever sums up
// products of them takes the FP64 state instead (build_state_f64).
// n = 10, depth 4: 18 k cycles of an SM for a state, 60 k in FP64 with the state in
// shared memory.
constexpr int FX_BITS = 60;
struct Fx {
    int h, l;
};
__device__ __forceinline__ Fx fx_split(long long y) {  // y: the value + 2^29
    Fx r;
    r.h = int(y >> 30);
    r.l = int(uint32_t(y) & 0x3FFFFFFFu) - (1 << 29);
    return r;
}
__device__ __forceinline__ Fx fx_from(double v) { return fx_split(__double2ll_rn(v * 0x1p60) + (1LL << 29)); }
__device__ __forceinline__ Fx fx_neg(Fx a) { return Fx{-a.h, -a.l}; }  // l = -2^29 gives 2^29, which the products take
// a b in units of 2^-60, rounded to nearest.
__device__ __forceinline__ long long fx_mul(Fx a, Fx b) {
    const long long x = (1LL << 29) + (long long)a.h * b.l + (long long)a.l * b.h;
    return (x >> 30) + (long long)a.h * b.h;
}
// c a + t b, rounded; |c a + t b| <= 1.
__device__ __forceinline__ Fx fx_rot(Fx a, Fx b, Fx c, Fx t) {
    // 2^59 carries the 2^29 that fx_split wants
    const long long x = ((1LL << 29) + (1LL << 59)) + (long long)a.h * c.l + (long long)a.l * c.h + (long long)b.h * t.l +
                        (long long)b.l * t.h;
    return fx_split((x >> 30) + (long long)a.h * c.h + (long long)b.h * t.h);
}

// Ry of the qubits on lane bits 0 .. nb - 1 (first qubit q0) and register bits.
template <int A>
__device__ __forceinline__ void fx_lanes(Fx (&v)[A], int lane, int b0, int nb, const int4* ang) {
    for (int j = 0; j < nb; ++j) {
        const int4 q = ang[j];
        const Fx c{q.x, q.y}, sn{q.z, q.w}, t = (lane >> (b0 + j)) & 1 ? sn : fx_neg(sn);
#pragma unroll
        for (int r = 0; r < A; ++r) {
            Fx p;
            p.h = __shfl_xor_sync(0xffffffffu, v[r].h, 1 << (b0 + j));
            p.l = __shfl_xor_sync(0xffffffffu, v[r].l, 1 << (b0 + j));
            v[r] = fx_rot(v[r], p, c, t);
        }
    }
}
template <int A, int LOGA>
__device__ __forceinline__ void fx_regs(Fx (&v)[A], const int4* ang) {
#pragma unroll
    for (int kb = 0; kb < LOGA; ++kb) {
        const int4 q = ang[kb];
        const Fx c{q.x, q.y}, sn{q.z, q.w}, ns = fx_neg(sn);
#pragma unroll
        for (int r = 0; r < A; ++r)
            if (!((r >> kb) & 1)) {
                const Fx a0 = v[r], a1 = v[r | (1 << kb)];
                v[r] = fx_rot(a0, a1, c, ns);
                v[r | (1 << kb)] = fx_rot(a1, a0, c, sn);
            }
    }
}
__device__ __forceinline__ Fx fx_sign(Fx a, int flip) { return flip ? fx_neg(a) : a; }

// Place of element i in a transpose buffer: both mappings below take a
// half-warp's 16 elements to 16 different bank pairs.
__device__ __forceinline__ int fx_at(int i) { return i ^ ((i >> 4) & 15); }
// Shared memory of build_state_fx, in bytes: P angles of 16 bytes and two buffers
// of 2^n amplitudes.
__host__ __device__ inline size_t fx_smem(int n, int P) { return 16 * (size_t(P) + (size_t(1) << n)); }

// n >= 8: A = 2^n / 256 amplitudes per thread.  Mapping 0: i = (r << 8) | (w << 5) |
// lane (qubits 0..4 on lanes, 5..7 on warps), mapping 1: i = (r << 8) | (lane << 3) | w
// (3..7 on lanes, 0..2 on warps); one transpose per layer brings the three
// qubits of the warp bits onto lanes, alternating the mappings, as
// state_regs_multiwarp.
template <int A, int LOGA>
__device__ void fx_multiwarp(Fx* out, Fx* scr, const int4* ang, const Fx* lowt, const Fx* hight, int n, int d, int t) {
    const int lane = t & 31, w = t >> 5, N = 1 << n;
    auto index = [&](int M, int r) { return M == 0 ? (r << 8) | (w << 5) | lane : (r << 8) | (lane << 3) | w; };
    Fx v[A];
#pragma unroll
    for (int r = 0; r < A; ++r) {
        const int i = index(0, r);
        v[r] = fx_split(fx_mul(lowt[i & 31], hight[i >> 5]) + (1LL << 29));
    }
    int M = 0;
    for (int layer = 1; layer <= d; ++layer) {
        const int4* la = ang + layer * n;
#pragma unroll
        for (int r = 0; r < A; ++r) v[r] = fx_sign(v[r], czring_parity(index(M, r), n));
        fx_lanes<A>(v, lane, 0, 5, la + (M == 0 ? 0 : 3));
        fx_regs<A, LOGA>(v, la + 8);
        Fx* buf = scr + (layer & 1) * N;
#pragma unroll
        for (int r = 0; r < A; ++r) buf[fx_at(index(M, r))] = v[r];
        __syncthreads();
        M ^= 1;
#pragma unroll
        for (int r = 0; r < A; ++r) v[r] = buf[fx_at(index(M, r))];
        // mapping 0: lanes 0..2 hold qubits 0..2; mapping 1: lanes 2..4 hold qubits 5..7
        fx_lanes<A>(v, lane, M == 0 ? 0 : 2, 3, la + (M == 0 ? 0 : 5));
    }
#pragma unroll
    for (int r = 0; r < A; ++r) out[index(M, r)] = v[r];
}

// n <= 7: one warp holds the state, A = max(1, 2^n / 32) amplitudes per lane.
template <int A, int LOGA>
__device__ void fx_warp(Fx* out, const int4* ang, const Fx* lowt, const Fx* hight, int n, int d, int lane) {
    const int N = 1 << n, li = N < 32 ? lane & (N - 1) : lane, nl = n < 5 ? n : 5;
    Fx v[A];
#pragma unroll
    for (int r = 0; r < A; ++r) v[r] = fx_split(fx_mul(lowt[li], hight[r]) + (1LL << 29));
    for (int layer = 1; layer <= d; ++layer) {
        const int4* la = ang + layer * n;
#pragma unroll
        for (int r = 0; r < A; ++r) v[r] = fx_sign(v[r], czring_parity((r << 5) | li, n));
        fx_lanes<A>(v, lane, 0, nl, la);
        fx_regs<A, LOGA>(v, la + 5);
    }
    __syncwarp();  // the tables are read: out may lie over their end
    if (lane < N || N >= 32) {
#pragma unroll
        for (int r = 0; r < A; ++r) out[(r << 5) | lane] = v[r];
    }
}

// psi(alpha_s), n <= 10: returns where its 2^n amplitudes lie in smem (fx_smem(n, P)
// bytes).  cs as for build_state_real.  Whole CTA of 256 threads; ends with a
// barrier.
__device__ inline Fx* build_state_fx(unsigned char* smem, int n, int d, int P, const double2* cs, int s) {
    const int N = 1 << n, t = threadIdx.x;
    int4* angw = reinterpret_cast<int4*>(smem);
    Fx* scr = reinterpret_cast<Fx*>(angw + P);  // two buffers; the factor tables start in the one first written at layer 2
    Fx* lowt = scr;
    Fx* hight = lowt + (N < 32 ? N : 32);
    // the result: not the buffer of the last transpose, whose reads may still go on
    Fx* out = scr + (n < 8 ? 1 : (d + 1) & 1) * N;
    int k = -1, which = 0;
    if (s > 0) {
        k = (s - 1) >> 1;
        which = ((s - 1) & 1) ? 2 : 1;
    }
    auto angle = [&](int a) { return cs[(a == k ? which : 0) * P + a]; };
    for (int a = n + t; a < P; a += 256) {
        const double2 v = angle(a);
        const Fx c = fx_from(v.x), sn = fx_from(v.y);
        angw[a] = make_int4(c.h, c.l, sn.h, sn.l);
    }
    // the initial Ry layer on |0> is a product state: factors of qubits 0..4 and of the others
    const int nl = n < 5 ? n : 5, nh = N >> nl;
    const int nlow = 1 << nl;
    for (int e = t ^ 255; e < nlow + nh; e += 256) {
        const bool lo = e < nlow;
        const int i = lo ? e : e - nlow, q0 = lo ? 0 : nl, q1 = lo ? nl : n;
        // in fixed point: a table entry is shared by 32 amplitudes, whose sums would show FP64
        // roundings of it (2^-53 of itself) where roundings of each amplitude average out
        Fx v{1 << 30, 0};
        for (int q = q0; q < q1; ++q) {
            const double2 c = angle(q);
            v = fx_split(fx_mul(v, fx_from(((i >> (q - q0)) & 1) ? c.y : c.x)) + (1LL << 29));
        }
        (lo ? lowt : hight)[i] = v;
    }
    __syncthreads();
    switch (n) {
        case 8: fx_multiwarp<1, 0>(out, scr, angw, lowt, hight, n, d, t); break;
        case 9: fx_multiwarp<2, 1>(out, scr, angw, lowt, hight, n, d, t); break;
        case 10: fx_multiwarp<4, 2>(out, scr, angw, lowt, hight, n, d, t); break;
        default:
            if (t < 32) {
                if (n == 7) fx_warp<4, 2>(out, angw, lowt, hight, n, d, t);
                else if (n == 6) fx_warp<2, 1>(out, angw, lowt, hight, n, d, t);
                else fx_warp<1, 0>(out, angw, lowt, hight, n, d, t);
            }
            break;
    }
    __syncthreads();
    return out;
}

// ---- The state in FP64 registers, for 256 threads, n <= 12.
//
// FP64 instructions issue at 1/64 of the FP32 rate and bound this, so a rotation runs
// in scaled form (ry_scaled): one FMA per amplitude, and the factors, multiplied
// together by a warp, once per group of layers.  Every amplitude keeps its relative
// accuracy, whatever its size.  n = 10, depth 4: 31 k cycles of an SM per state (40 k
// FMAs are 20 k), the fixed-point state above 18 k.

// Ratio of an Ry in scaled form: |ratio| <= 1 leaves bit 62 clear, it is set for the
// sine form.  (A NaN is reported by whoever formed the angles' table.)
__device__ __forceinline__ long long ry64_pack(double2 v) {  // v: (cos, sin)
    const bool sf = fabs(v.y) > fabs(v.x);
    return __double_as_longlong(sf ? v.x / v.y : v.y / v.x) | (long long)sf << 62;
}
__device__ __forceinline__ double flip_sign(double v, int flip) {  // flip: 0 or the sign bit
    return __hiloint2double(__double2hiint(v) ^ flip, __double2loint(v));
}

// Layers whose factors are applied together: at most 64 rotations, each of which lets
// the amplitudes grow by sqrt(2) at most.
__host__ __device__ inline int ry64_group(int n) { return 64 / n; }
__host__ __device__ inline int ry64_groups(int n, int P) { return (P / n - 1 + ry64_group(n) - 1) / ry64_group(n); }

// The product of the factors of rotations first .. first + count - 1 (count <= 64), by
// a warp; angle(a) is (cos, sin).  Formed as 64-bit significands (2^-63 relative per
// product, as FP64 products would not be) and rounded once.
template <class Angle>
__device__ __forceinline__ double ry64_factor(int first, int count, int lane, const Angle& angle) {
    unsigned long long m = 1ull << 63;  // m 2^(e - 63)
    int e = 0, neg = 0;
    auto times = [&](unsigned long long m2, int e2, int neg2) {
        m = __umul64hi(m, m2);
        e += e2 + 1;
        if (!(m >> 63)) {
            m <<= 1;
            --e;
        }
        neg ^= neg2;
    };
    for (int k = lane; k < count; k += 32) {
        const double2 v = angle(first + k);
        const unsigned long long f = (unsigned long long)__double_as_longlong(fabs(v.y) > fabs(v.x) ? v.y : v.x);
        times((f | 1ull << 52) << 11, int((f >> 52) & 0x7ff) - 1023, int(f >> 63));
    }
    for (int o = 16; o; o >>= 1) {
        const unsigned long long m2 = __shfl_xor_sync(0xffffffffu, m, o);
        const int e2 = __shfl_xor_sync(0xffffffffu, e, o), neg2 = __shfl_xor_sync(0xffffffffu, neg, o);
        times(m2, e2, neg2);
    }
    const double f = scalbn((double)m, e - 63);
    return neg ? -f : f;
}

// Ry of the qubits on lane bits b0 .. b0 + nb - 1 and on the register bits.
template <int A>
__device__ __forceinline__ void ry64_lanes(double (&v)[A], int lane, int b0, int nb, const long long* ang) {
    for (int j = 0; j < nb; ++j) {
        const long long q = ang[j];
        const double r = __longlong_as_double(q & ~(1LL << 62));
        const bool sf = (q >> 62) & 1;
        const int flip = (lane >> (b0 + j)) & 1 ? 0 : int(0x80000000u);
#pragma unroll
        for (int k = 0; k < A; ++k) {
            const double p = flip_sign(__shfl_xor_sync(0xffffffffu, v[k], 1 << (b0 + j)), flip);
            v[k] = fma(r, sf ? v[k] : p, sf ? p : v[k]);
        }
    }
}
template <int A, int LOGA>
__device__ __forceinline__ void ry64_regs(double (&v)[A], const long long* ang) {
#pragma unroll
    for (int kb = 0; kb < LOGA; ++kb) {
        const long long q = ang[kb];
        const double r = __longlong_as_double(q & ~(1LL << 62));
        const bool sf = (q >> 62) & 1;
#pragma unroll
        for (int k = 0; k < A; ++k)
            if (!((k >> kb) & 1)) {
                const double a0 = v[k], a1 = v[k | (1 << kb)];
                v[k] = fma(r, sf ? a0 : -a1, sf ? -a1 : a0);
                v[k | (1 << kb)] = fma(r, sf ? a1 : a0, sf ? a0 : a1);
            }
    }
}

// The first layer on |0>, a product state: the factors of the qubits below nt, by the bits of i,
// then those of the register bits.
template <int A, int LOGA>
__device__ __forceinline__ void ry64_product(double (&v)[A], int i, int nt, const double2* c0) {
    v[0] = 1.0;
    for (int q = 0; q < nt; ++q) v[0] *= ((i >> q) & 1) ? c0[q].y : c0[q].x;
#pragma unroll
    for (int kb = 0; kb < LOGA; ++kb)
#pragma unroll
        for (int r = 0; r < (1 << kb); ++r) {
            v[r | (1 << kb)] = v[r] * c0[nt + kb].y;
            v[r] *= c0[nt + kb].x;
        }
}
// Shared memory of build_state_f64, in bytes: the ratios and the groups' factors, two
// buffers of 2^n amplitudes.
__host__ __device__ inline size_t f64_angle_bytes(int n, int P) {
    return (8 * size_t(P + ry64_groups(n, P)) + 15) & ~size_t(15);
}
__host__ __device__ inline size_t f64_smem(int n, int P) { return f64_angle_bytes(n, P) + (size_t(16) << n); }

// n >= 8: A = 2^n / 256 amplitudes per thread.  Mapping 0: i = (r << 8) | (w << 5) |
// lane (qubits 0..4 on lanes, 5..7 on warps), mapping 1: i = (r << 8) | (lane << 3) | w
// (3..7 on lanes, 0..2 on warps); one transpose per layer brings the three
// qubits of the warp bits onto lanes, alternating the mappings, as
// state_regs_multiwarp.
template <int A, int LOGA>
__device__ void f64_multiwarp(double* out, double* scr, const long long* ang, const double* fac, const double2* c0, int n,
                              int d, int t) {
    const int lane = t & 31, w = t >> 5, N = 1 << n, G = ry64_group(n);
    auto index = [&](int M, int r) { return M == 0 ? (r << 8) | (w << 5) | lane : (r << 8) | (lane << 3) | w; };
    double v[A];
    ry64_product<A, LOGA>(v, (w << 5) | lane, 8, c0);
    int M = 0, g = 0;
    for (int layer = 1; layer <= d; ++layer) {
        const long long* la = ang + layer * n;
#pragma unroll
        for (int r = 0; r < A; ++r) v[r] = flip_sign(v[r], czring_parity(index(M, r), n) << 31);
        ry64_lanes<A>(v, lane, 0, 5, la + (M == 0 ? 0 : 3));
        ry64_regs<A, LOGA>(v, la + 8);
        double* buf = scr + (layer & 1) * N;
#pragma unroll
        for (int r = 0; r < A; ++r) buf[fx_at(index(M, r))] = v[r];
        __syncthreads();
        M ^= 1;
#pragma unroll
        for (int r = 0; r < A; ++r) v[r] = buf[fx_at(index(M, r))];
        // mapping 0: lanes 0..2 hold qubits 0..2; mapping 1: lanes 2..4 hold qubits 5..7
        ry64_lanes<A>(v, lane, M == 0 ? 0 : 2, 3, la + (M == 0 ? 0 : 5));
        if (layer == d || layer == (g + 1) * G) {
            const double f = fac[g++];
#pragma unroll
            for (int r = 0; r < A; ++r) v[r] *= f;
        }
    }
#pragma unroll
    for (int r = 0; r < A; ++r) out[index(M, r)] = v[r];
}

// n <= 7: one warp holds the state, A = max(1, 2^n / 32) amplitudes per lane.
template <int A, int LOGA>
__device__ void f64_warp(double* out, const long long* ang, const double* fac, const double2* c0, int n, int d, int lane) {
    const int N = 1 << n, li = N < 32 ? lane & (N - 1) : lane, nl = n < 5 ? n : 5, G = ry64_group(n);
    double v[A];
    ry64_product<A, LOGA>(v, li, nl, c0);
    int g = 0;
    for (int layer = 1; layer <= d; ++layer) {
        const long long* la = ang + layer * n;
#pragma unroll
        for (int r = 0; r < A; ++r) v[r] = flip_sign(v[r], czring_parity((r << 5) | li, n) << 31);
        ry64_lanes<A>(v, lane, 0, nl, la);
        ry64_regs<A, LOGA>(v, la + 5);
        if (layer == d || layer == (g + 1) * G) {
            const double f = fac[g++];
#pragma unroll
            for (int r = 0; r < A; ++r) v[r] *= f;
        }
    }
    if (lane < N || N >= 32) {
#pragma unroll
        for (int r = 0; r < A; ++r) out[(r << 5) | lane] = v[r];
    }
}

// psi(alpha_s) in `out`, 2^n doubles of smem (f64_smem(n, P) bytes); as many in `other`
// are free afterwards.  cs as for build_state_real; n <= NMAX.  Whole CTA of 256
// threads; ends with a barrier.
template <int NMAX>
__device__ inline void build_state_f64(unsigned char* smem, int n, int d, int P, const double2* cs, int s, double*& out,
                                       double*& other) {
    const int N = 1 << n, t = threadIdx.x, lane = t & 31, w = t >> 5;
    long long* ang = reinterpret_cast<long long*>(smem);
    double* fac = reinterpret_cast<double*>(ang + P);
    double* scr = reinterpret_cast<double*>(smem + f64_angle_bytes(n, P));  // two buffers; the first layer's (cos, sin)
    double2* c0 = reinterpret_cast<double2*>(scr);                          // start in the one first written at layer 2
    // the result: not the buffer of the last transpose, whose reads may still go on
    out = scr + (n < 8 ? 1 : (d + 1) & 1) * N;
    other = out == scr ? scr + N : scr;
    int k = -1, which = 0;
    if (s > 0) {
        k = (s - 1) >> 1;
        which = ((s - 1) & 1) ? 2 : 1;
    }
    auto angle = [&](int a) { return cs[(a == k ? which : 0) * P + a]; };
    const int G = ry64_group(n), groups = ry64_groups(n, P);
    for (int g = w; g < groups; g += 8) {
        const int first = n * (1 + g * G);
        const double f = ry64_factor(first, min(n * G, P - first), lane, angle);
        if (lane == 0) fac[g] = f;
    }
    for (int a = n + (t ^ 128); a < P; a += 256) ang[a] = ry64_pack(angle(a));
    if (t < n) c0[t] = angle(t);  // on |0>: a product state
    __syncthreads();
    switch (n) {
        case 8: f64_multiwarp<1, 0>(out, scr, ang, fac, c0, n, d, t); break;
        case 9: f64_multiwarp<2, 1>(out, scr, ang, fac, c0, n, d, t); break;
        case 10: f64_multiwarp<4, 2>(out, scr, ang, fac, c0, n, d, t); break;
        case 11:
            if constexpr (NMAX >= 11) f64_multiwarp<8, 3>(out, scr, ang, fac, c0, n, d, t);
            break;
        case 12:
            if constexpr (NMAX >= 12) f64_multiwarp<16, 4>(out, scr, ang, fac, c0, n, d, t);
            break;
        default:
            if (t < 32) {
                if (n == 7) f64_warp<4, 2>(out, ang, fac, c0, n, d, t);
                else if (n == 6) f64_warp<2, 1>(out, ang, fac, c0, n, d, t);
                else f64_warp<1, 0>(out, ang, fac, c0, n, d, t);
            }
            break;
    }
    __syncthreads();
}

}  // namespace dvqls
