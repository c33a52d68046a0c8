// FWHT-based Pauli decomposition with tau pruning and top-L selection
// (Sec. 2.2, Eq. 5; Algorithm 1, Steps 1-2).
//
// Pipeline (all on the device; the host only reads three counts back):
//   1. X-mask scan: every nonzero A[r, c] marks mask r ^ c;  compaction gives
//      the present masks in ascending order.
//   2. Per mask x: gather d_x(i) = A[i ^ x, i], Walsh-Hadamard transform with
//      the radix-2 butterfly at strides 1, 2, ..., N/2 (u, v) -> (u+v, u-v),
//      then c(x,z) = (-i)^popc(x&z) W_x(z) / N and key = re*re + im*im.
//      n <= 12: one CTA per mask, the whole diagonal in shared memory.
//      n > 12: strides < 4096 in shared-memory chunks, the remaining strides
//      in a second pass over column tiles, in place; the butterfly graph (and
//      so every rounding) is the same as a stride-by-stride transform.  One
//      FP64 value per coefficient is kept (its other component is zero).
//   3. max key, the counts L_pre (key > 0) and L_post (key > thr) with
//      thr = (tau*tau) * max key, and the top-L_max select ordered by key
//      descending then (x << n) | z ascending: a radix selection of the
//      candidates, then one sort of those.
//
// Add/sub, power-of-two scaling and the phase are exact or correctly
// rounded, and the key is formed with explicit _rn intrinsics (no fused
// multiply-add), so coefficients, masks, order and counts are bit-identical to
// any implementation that follows the same butterfly order.
#include <algorithm>

#include "internal.cuh"

namespace {

constexpr int MAX_TERMS = 2048;  // largest L_max
constexpr int MAX_BANDS = 64;

struct Band {
    int nbands;
    int off[MAX_BANDS];
};

__device__ __forceinline__ double band_entry(const Band& bd, const double* vals, int n, long long row,
                                             long long col) {
    const long long o = col - row;
    for (int k = 0; k < bd.nbands; ++k)
        if (bd.off[k] == o) return vals[(long long)k << n | row];
    return 0.0;
}

__device__ __forceinline__ double entry(const double* A, const Band& bd, const double* vals, int n,
                                        long long row, long long col) {
    return A ? A[(row << n) | col] : band_entry(bd, vals, n, row, col);
}

__device__ __forceinline__ bool zero_bits(double v) { return ((unsigned long long)__double_as_longlong(v) << 1) == 0ull; }
__device__ __forceinline__ bool finite_bits(double v) {
    return (__double2hiint(v) & 0x7ff00000) != 0x7ff00000;
}
// A mask is marked at most once per reader that still sees it unmarked: most
// entries of a banded matrix share a few masks, and a store per entry would
// queue up on their bytes (n = 20 tridiagonal: 111 us with a store per entry,
// 22 us with the test).  The tests are on bits: FP64 compares issue at 1/64 of
// the FP32 rate.
__device__ __forceinline__ void mark(unsigned char* flags, long long x) {
    if (!flags[x]) flags[x] = 1;
}

__global__ void k_flags_dense(const double* __restrict__ A, int n, unsigned char* flags, int* status) {
    const long long N = 1LL << n, NN = N * N;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < NN;
         e += (long long)gridDim.x * blockDim.x) {
        const double v = A[e];
        if (zero_bits(v)) continue;
        if (!finite_bits(v)) atomicCAS(status, 0, dvqls::DEV_NONFINITE_INPUT);
        mark(flags, (e >> n) ^ (e & (N - 1)));
    }
}

__global__ void k_flags_banded(int n, Band bd, const double* __restrict__ vals, unsigned char* flags,
                               int* status) {
    const long long N = 1LL << n, tot = (long long)bd.nbands * N;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < tot;
         e += (long long)gridDim.x * blockDim.x) {
        const int k = int(e >> n);
        const long long r = e & (N - 1), c = r + bd.off[k];
        if (c < 0 || c >= N) continue;
        const double v = vals[e];
        if (zero_bits(v)) continue;
        if (!finite_bits(v)) atomicCAS(status, 0, dvqls::DEV_NONFINITE_INPUT);
        mark(flags, r ^ c);
    }
}

// Present masks in ascending order.  A CTA takes CMP_CHUNK flags (32 bytes per
// thread, two 16-byte loads); with more than one chunk k_mask_count runs first
// and each CTA of k_mask_write adds up the counts before its own.  (One CTA over
// all 2^20 flags, byte by byte, took 1,043 us; the two kernels take 6.)
constexpr int CMP_T = 256, CMP_CHUNK = 32 * CMP_T;

__device__ __forceinline__ int flag_count(const uint4& v) {  // bytes are 0 or 1
    return __popc(v.x) + __popc(v.y) + __popc(v.z) + __popc(v.w);
}

__global__ void __launch_bounds__(CMP_T) k_mask_count(const unsigned char* __restrict__ flags, int* cnt) {
    const uint4* f = reinterpret_cast<const uint4*>(flags) + (size_t)blockIdx.x * (CMP_CHUNK / 16) + 2 * threadIdx.x;
    int c = flag_count(f[0]) + flag_count(f[1]);
    for (int o = 16; o; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
    __shared__ int part[CMP_T / 32];
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = c;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int k = 1; k < CMP_T / 32; ++k) c += part[k];
        cnt[blockIdx.x] = c;
    }
}

__global__ void __launch_bounds__(CMP_T) k_mask_write(const unsigned char* __restrict__ flags, const int* cnt,
                                                      uint32_t* masks, int* count) {
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    const uint4* f = reinterpret_cast<const uint4*>(flags) + (size_t)blockIdx.x * (CMP_CHUNK / 16) + 2 * t;
    const uint4 v[2] = {f[0], f[1]};
    const int c = flag_count(v[0]) + flag_count(v[1]);
    __shared__ int part[CMP_T / 32], before[CMP_T / 32];
    int pre = 0;
    for (int k = t; k < int(blockIdx.x); k += CMP_T) pre += cnt[k];
    int incl = c;
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
    }
    for (int o = 16; o; o >>= 1) pre += __shfl_xor_sync(0xffffffffu, pre, o);
    if (lane == 31) part[w] = incl;
    if (lane == 0) before[w] = pre;
    __syncthreads();
    int o = incl - c, total = 0;
    for (int k = 0; k < CMP_T / 32; ++k) {
        o += before[k] + (k < w ? part[k] : 0);
        total += before[k] + part[k];
    }
    const uint32_t i0 = blockIdx.x * uint32_t(CMP_CHUNK) + 32u * t;
    const uint32_t wd[8] = {v[0].x, v[0].y, v[0].z, v[0].w, v[1].x, v[1].y, v[1].z, v[1].w};
    if (c)
#pragma unroll
        for (int k = 0; k < 32; ++k)
            if ((wd[k >> 2] >> (8 * (k & 3))) & 1u) masks[o++] = i0 + k;
    if (blockIdx.x == gridDim.x - 1 && t == 0) *count = total;
}

// ------------------------------------------------------------- transform
// Walsh-Hadamard butterflies at the strides of bits b .. b + NB - 1 of the
// element index (within a row of `per` interleaved columns), 2^NB elements per
// thread in registers: the same butterfly graph as one stride at a time, so
// the same roundings, with one shared-memory round trip and one barrier for
// four strides.  A group whose elements are all zero stays zero and is passed
// over (a banded matrix's diagonal at a large mask is zero over most of its
// blocks).  FP64 adds bound the transform (they issue at 1/64 of the FP32
// rate): n = 20 tridiagonal, 440 M adds are 700 us of the FP64 pipe; one stride
// per pass and no test took 1,156 us, this 511.  Element e sits at word e + (e >> 4): the strides of bit 0 would put
// all 16 lanes of a half-warp in one bank.
__device__ __forceinline__ int fw_pad(int e) { return e + (e >> 4); }

template <int NB>
__device__ __forceinline__ void fwht_groups(double* w, int elems, int b) {
    for (int g = threadIdx.x; g < (elems >> NB); g += blockDim.x) {
        const int i0 = ((g >> b) << (b + NB)) | (g & ((1 << b) - 1));
        double v[1 << NB];
        unsigned long long any = 0ull;
#pragma unroll
        for (int r = 0; r < (1 << NB); ++r) {
            v[r] = w[fw_pad(i0 | (r << b))];
            any |= (unsigned long long)__double_as_longlong(v[r]) << 1;
        }
        if (any == 0ull) continue;
#pragma unroll
        for (int k = 0; k < NB; ++k)
#pragma unroll
            for (int r = 0; r < (1 << NB); ++r)
                if (!((r >> k) & 1)) {
                    const double x = v[r], y = v[r | (1 << k)];
                    v[r] = __dadd_rn(x, y);
                    v[r | (1 << k)] = __dsub_rn(x, y);
                }
#pragma unroll
        for (int r = 0; r < (1 << NB); ++r) w[fw_pad(i0 | (r << b))] = v[r];
    }
    __syncthreads();
}

// Strides of bits b0 .. b0 + bits - 1, ascending.
__device__ __forceinline__ void fwht_bits(double* w, int elems, int b0, int bits) {
    int b = b0;
    const int end = b0 + bits;
    for (; b + 4 <= end; b += 4) fwht_groups<4>(w, elems, b);
    switch (end - b) {
        case 3: fwht_groups<3>(w, elems, b); break;
        case 2: fwht_groups<2>(w, elems, b); break;
        case 1: fwht_groups<1>(w, elems, b); break;
        default: break;
    }
}

// -------------------------------------------------------------- selection
// Top L_max of the keys above the threshold, ordered by key descending then
// position ascending, by radix selection: the transform's last kernel counts
// its keys into SEL_BINS bins of their leading bits (exponent and one mantissa
// bit), k_sel_pick finds the lowest bin that is needed, k_sel_collect copies
// the keys from it on into a candidate list, and one CTA sorts that list and
// writes the terms.  The list nearly always fits (SEL_CAP candidates); when it
// does not (a mass of nearly or exactly equal keys at the cut), the host launches
// rounds over the next SEL_BITS bits of the keys and, at equal keys, of their
// positions, after which exactly L_max candidates are left.  A sort of every
// 4,096-key block took 2,154 us of the n = 20 tridiagonal decomposition (22 M
// coefficients) with its counting passes, the selection takes 66.
constexpr int SEL_BITS = 12, SEL_BINS = 1 << SEL_BITS, SEL_CAP = 4096, SEL_T = 1024;
constexpr int SEL_ROUNDS = 10;
constexpr int SEL_POS_BITS = 40;  // positions below 2^40 (n <= 20 masks x 2^20 entries)
// Low bit and width of the digit of each round: key bits 62 .. 0, then position bits.
__device__ __constant__ const int SEL_SHIFT[SEL_ROUNDS] = {51, 39, 27, 15, 3, 0, 28, 16, 4, 0};
__device__ __constant__ const int SEL_WIDTH[SEL_ROUNDS] = {12, 12, 12, 12, 12, 3, 12, 12, 12, 4};
constexpr int SEL_KEY_ROUNDS = 6;

struct Misc {  // counters of a call; cleared before it
    int masks, l_pre, l_post, l_out;
    unsigned long long kmax;  // largest key (ordered bits of a non-negative double)
    unsigned long long lb_key, lb_pos;  // candidates are the entries with (key, ~position) >= this
    long long need;           // entries still wanted inside the current bin
    int done, cands;          // the candidates fit SEL_CAP; candidates collected
};

constexpr unsigned long long INF_BITS = 0x7ff0000000000000ull;

// Key of a coefficient of magnitude |v| (its other component is zero): re*re +
// im*im without a fused multiply-add.
__device__ __forceinline__ unsigned long long key_bits(double v) {
    return (unsigned long long)__double_as_longlong(__dmul_rn(v, v));
}
__device__ __forceinline__ bool key_counts(unsigned long long kb) { return kb - 1ull < INF_BITS; }  // > 0, no NaN
__device__ __forceinline__ unsigned long long sel_pos(long long e) { return ((1ull << SEL_POS_BITS) - 1) - e; }

// Largest bits that do not pass the tau filter (all ones when nothing passes).
__device__ __forceinline__ unsigned long long threshold_bits(double tau, unsigned long long kmax) {
    const double thr = tau > 0.0 ? __dmul_rn(__dmul_rn(tau, tau), __longlong_as_double((long long)kmax)) : 0.0;
    const unsigned long long b = (unsigned long long)__double_as_longlong(thr);
    return b > INF_BITS ? ~0ull : b;
}

// A transform CTA's keys: the maximum, the number above zero and the first
// digits' counts, gathered in shared memory and added to the call's.
struct KeyStats {
    uint32_t* hist;  // SEL_BINS, cleared by start()
    unsigned long long m = 0;
    int c = 0;
    __device__ explicit KeyStats(uint32_t* h) : hist(h) {}
    __device__ void start() {
        for (int k = threadIdx.x; k < SEL_BINS; k += blockDim.x) hist[k] = 0u;
    }
    __device__ void add(double v) {
        const unsigned long long kb = key_bits(v);
        m = kb > m ? kb : m;
        if (key_counts(kb)) {
            ++c;
            atomicAdd(&hist[kb >> 51], 1u);
        }
    }
    __device__ void finish(Misc* misc, uint32_t* ghist) {
        for (int o = 16; o; o >>= 1) {
            const unsigned long long m2 = __shfl_xor_sync(0xffffffffu, m, o);
            m = m2 > m ? m2 : m;
            c += __shfl_xor_sync(0xffffffffu, c, o);
        }
        __shared__ unsigned long long sm;
        __shared__ int sc;
        if (threadIdx.x == 0) {
            sm = 0ull;
            sc = 0;
        }
        __syncthreads();
        if ((threadIdx.x & 31) == 0 && m) {
            atomicMax(&sm, m);
            atomicAdd(&sc, c);
        }
        __syncthreads();
        if (threadIdx.x == 0 && sm) {
            atomicMax(&misc->kmax, sm);
            if (sc) atomicAdd(&misc->l_pre, sc);
        }
        if (sc)
            for (int k = threadIdx.x; k < SEL_BINS; k += blockDim.x)
                if (hist[k]) atomicAdd(&ghist[k], hist[k]);
    }
};

constexpr int FW_T = 256;

// n <= 12: one CTA per mask, the whole transform in shared memory.
__global__ void __launch_bounds__(FW_T) k_fwht_smem(const double* __restrict__ A, Band bd, const double* __restrict__ vals,
                                                    int n, const uint32_t* __restrict__ masks, double* val, Misc* misc,
                                                    uint32_t* ghist) {
    extern __shared__ __align__(16) unsigned char sm_raw[];
    uint32_t* hist = reinterpret_cast<uint32_t*>(sm_raw);
    double* w = reinterpret_cast<double*>(sm_raw + SEL_BINS * 4);
    KeyStats ks(hist);
    ks.start();
    const int r = blockIdx.x, N = 1 << n;
    const uint32_t x = masks[r];
    for (int i = threadIdx.x; i < N; i += FW_T) w[fw_pad(i)] = entry(A, bd, vals, n, i ^ x, i);
    __syncthreads();
    fwht_bits(w, N, 0, n);
    const double scale = ldexp(1.0, -n);
    for (int z = threadIdx.x; z < N; z += FW_T) {
        double v = w[fw_pad(z)];
        if (!zero_bits(v)) {
            v *= scale;
            ks.add(v);
        }
        val[((long long)r << n) + z] = v;
    }
    ks.finish(misc, ghist);
}

constexpr int LO_BITS = 12, LO = 1 << LO_BITS, HI_TILE = 16;

// n > 12, pass 1: gather and strides 1 .. 2048 inside 4096-element chunks (a
// chunk without a nonzero entry is written as zeros).
__global__ void __launch_bounds__(FW_T) k_fwht_lo(const double* __restrict__ A, Band bd, const double* __restrict__ vals,
                                                  int n, const uint32_t* __restrict__ masks, double* val) {
    __shared__ double w[LO + LO / 16];
    const long long N = 1LL << n;
    const int chunks = int(N >> LO_BITS);
    const int r = blockIdx.x / chunks, ch = blockIdx.x % chunks;
    const uint32_t x = masks[r];
    const long long base = (long long)ch << LO_BITS;
    bool any = false;
#pragma unroll 4
    for (int i = threadIdx.x; i < LO; i += FW_T) {
        const double v = entry(A, bd, vals, n, (base + i) ^ x, base + i);
        any |= !zero_bits(v);
        w[fw_pad(i)] = v;
    }
    if (__syncthreads_or(any)) fwht_bits(w, LO, 0, LO_BITS);
    double* out = val + ((long long)r << n) + base;
    for (int i = threadIdx.x; i < LO; i += FW_T) out[i] = w[fw_pad(i)];
}

// n > 12, pass 2, in place: strides 4096 .. N/2 on tiles of HI_TILE consecutive
// low indices (element (hi, lo) of the tile at hi HI_TILE + lo), then the scale
// and the keys.
__global__ void __launch_bounds__(FW_T) k_fwht_hi(int n, double* val, Misc* misc, uint32_t* ghist) {
    extern __shared__ __align__(16) unsigned char sm_raw[];
    uint32_t* hist = reinterpret_cast<uint32_t*>(sm_raw);
    double* w = reinterpret_cast<double*>(sm_raw + SEL_BINS * 4);
    KeyStats ks(hist);
    ks.start();
    const int hb = n - LO_BITS, elems = HI_TILE << hb;
    const int tiles = LO / HI_TILE;
    const int r = blockIdx.x / tiles, lo0 = (blockIdx.x % tiles) * HI_TILE;
    double* src = val + ((long long)r << n) + lo0;
#pragma unroll 4
    for (int e = threadIdx.x; e < elems; e += FW_T) w[fw_pad(e)] = src[((long long)(e / HI_TILE) << LO_BITS) + e % HI_TILE];
    __syncthreads();
    fwht_bits(w, elems, 4, hb);  // HI_TILE = 2^4 columns
    const double scale = ldexp(1.0, -n);
    for (int e = threadIdx.x; e < elems; e += FW_T) {
        double v = w[fw_pad(e)];
        if (!zero_bits(v)) {
            v *= scale;
            ks.add(v);
        }
        src[((long long)(e / HI_TILE) << LO_BITS) + e % HI_TILE] = v;
    }
    ks.finish(misc, ghist);
}

// The digit of round `round` (one CTA): the highest digit value whose suffix
// count reaches what is needed (0 when the counts fall short: then every entry
// that is left is wanted), from the counts of the entries that share the digits
// found so far.  Clears the counts for the next round.
__global__ void __launch_bounds__(SEL_T) k_sel_pick(int round, double tau, int L_max, Misc* misc, uint32_t* ghist) {
    constexpr int PER = SEL_BINS / SEL_T;
    if (misc->done) return;  // an earlier round was enough
    __shared__ long long part[SEL_T / 32];
    __shared__ long long s_at, s_above;
    __shared__ int s_bin;
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    const long long need = round == 0 ? L_max : misc->need;
    // thread t holds bins SEL_BINS - 1 - PER t downwards, so prefix sums over threads are suffix counts
    uint32_t h[PER];
    long long run = 0;
#pragma unroll
    for (int k = 0; k < PER; ++k) {
        h[k] = ghist[SEL_BINS - 1 - (PER * t + k)];
        ghist[SEL_BINS - 1 - (PER * t + k)] = 0u;
        run += h[k];
    }
    long long incl = run;
    for (int o = 1; o < 32; o <<= 1) {
        const long long y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
    }
    if (lane == 31) part[w] = incl;
    if (t == 0) s_bin = -1;
    __syncthreads();
    for (int k = 0; k < w; ++k) incl += part[k];
    const int low = round == 0 ? int(min(threshold_bits(tau, misc->kmax) >> 51, (unsigned long long)(SEL_BINS - 1))) : 0;
    long long above = incl - run;
#pragma unroll
    for (int k = 0; k < PER; ++k) {
        const int bin = SEL_BINS - 1 - (PER * t + k);
        // the bin that reaches the need, or the lowest one asked for
        if ((above < need && above + h[k] >= need && bin >= low) || (bin == low && above + h[k] < need)) {
            s_bin = bin;
            s_above = above;
            s_at = h[k];
        }
        above += h[k];
    }
    __syncthreads();
    if (t == 0 && s_bin >= 0) {
        const unsigned long long digit = (unsigned long long)s_bin << SEL_SHIFT[round];
        if (round < SEL_KEY_ROUNDS) misc->lb_key |= digit;
        else misc->lb_pos |= digit;
        misc->need = need - s_above;
        misc->done = (L_max - need) + s_above + s_at <= SEL_CAP;
    }
}

// Counts of round `round`'s digits over the entries that share the earlier ones.
__global__ void __launch_bounds__(256) k_sel_hist(int round, const double* __restrict__ val, long long E, double tau,
                                                  const Misc* misc, uint32_t* ghist) {
    __shared__ uint32_t hist[SEL_BINS];
    if (misc->done) return;  // an earlier round was enough
    for (int k = threadIdx.x; k < SEL_BINS; k += blockDim.x) hist[k] = 0u;
    __syncthreads();
    const unsigned long long thr = threshold_bits(tau, misc->kmax), lk = misc->lb_key, lp = misc->lb_pos;
    const int sh = SEL_SHIFT[round], up = sh + SEL_WIDTH[round];
    const uint32_t mask = (1u << SEL_WIDTH[round]) - 1u;
    for (long long e = blockIdx.x * 256LL + threadIdx.x; e < E; e += gridDim.x * 256LL) {
        const double v = val[e];
        if (zero_bits(v)) continue;
        const unsigned long long kb = key_bits(v);
        if (!key_counts(kb) || kb <= thr) continue;
        if (round < SEL_KEY_ROUNDS) {
            if ((kb >> up) == (lk >> up)) atomicAdd(&hist[uint32_t(kb >> sh) & mask], 1u);
        } else if (kb == lk) {
            const unsigned long long pc = sel_pos(e);
            if (round == SEL_KEY_ROUNDS || (pc >> up) == (lp >> up)) atomicAdd(&hist[uint32_t(pc >> sh) & mask], 1u);
        }
    }
    __syncthreads();
    for (int k = threadIdx.x; k < SEL_BINS; k += blockDim.x)
        if (hist[k]) atomicAdd(&ghist[k], hist[k]);
}

// Entries that pass the tau filter are counted (`count`), and those at or above
// the bound join the candidates, in any order (they are sorted afterwards).
__global__ void __launch_bounds__(256) k_sel_collect(const double* __restrict__ val, long long E, double tau, int count,
                                                     Misc* misc, unsigned long long* cand_k, unsigned long long* cand_p) {
    const unsigned long long thr = threshold_bits(tau, misc->kmax), lk = misc->lb_key, lp = misc->lb_pos;
    const bool done = misc->done;
    int c = 0;
#pragma unroll 4
    for (long long e = blockIdx.x * 256LL + threadIdx.x; e < E; e += gridDim.x * 256LL) {
        const double v = val[e];
        if (zero_bits(v)) continue;
        const unsigned long long kb = key_bits(v);
        if (!key_counts(kb) || kb <= thr) continue;
        ++c;
        if (done && (kb > lk || (kb == lk && sel_pos(e) >= lp))) {
            const int at = atomicAdd(&misc->cands, 1);
            if (at < SEL_CAP) {
                cand_k[at] = kb;
                cand_p[at] = (unsigned long long)e;
            }
        }
    }
    if (!count) return;
    for (int o = 16; o; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
    if ((threadIdx.x & 31) == 0 && c) atomicAdd(&misc->l_post, c);
}

// Sorts the candidates (key descending, position ascending; one CTA, bitonic
// over the next power of two) and writes the first min(l_post, L_max) terms.
__global__ void __launch_bounds__(SEL_T) k_sel_emit(Misc* misc, const unsigned long long* __restrict__ cand_k,
                                                    const unsigned long long* __restrict__ cand_p,
                                                    const double* __restrict__ val, const uint32_t* __restrict__ masks,
                                                    int n, int L_max, double* out_c, uint32_t* out_x, uint32_t* out_z) {
    extern __shared__ __align__(16) unsigned char sm_raw[];
    if (!misc->done) return;
    unsigned long long* k = reinterpret_cast<unsigned long long*>(sm_raw);
    unsigned long long* p = k + SEL_CAP;
    const int t = threadIdx.x, C = min(misc->cands, SEL_CAP), L = min(misc->l_post, L_max);
    int P2 = 1;
    while (P2 < C) P2 <<= 1;
    for (int i = t; i < P2; i += SEL_T) {
        k[i] = i < C ? ~cand_k[i] : ~0ull;
        p[i] = i < C ? cand_p[i] : ~0ull;
    }
    __syncthreads();
    for (int q = 2; q <= P2; q <<= 1)
        for (int j = q >> 1; j > 0; j >>= 1) {
            for (int h = t; h < P2 / 2; h += SEL_T) {
                const int i = ((h & ~(j - 1)) << 1) | (h & (j - 1)), m = i | j;
                const unsigned long long ka = k[i], kb = k[m], pa = p[i], pb = p[m];
                const bool less = kb < ka || (kb == ka && pb < pa);
                if (less == ((i & q) == 0)) {
                    k[i] = kb;
                    k[m] = ka;
                    p[i] = pb;
                    p[m] = pa;
                }
            }
            __syncthreads();
        }
    if (t == 0) misc->l_out = L;
    for (int i = t; i < L; i += SEL_T) {
        const unsigned long long e = p[i];
        const uint32_t x = masks[e >> n], z = uint32_t(e & ((1ull << n) - 1));
        const double v = val[e];
        double re = 0.0, im = 0.0;
        switch (__popc(x & z) & 3) {  // (-i)^popc(x & z)
            case 0: re = v; break;
            case 1: im = -v; break;
            case 2: re = -v; break;
            default: im = v; break;
        }
        out_c[2 * i] = re;
        out_c[2 * i + 1] = im;
        out_x[i] = x;
        out_z[i] = z;
    }
}

int decompose_common(dvqls_ctx* ctx, const double* A_in, int n, int nbands, const int* offsets,
                     const double* bands_in, double tau, int L_max, double* coef_out, uint32_t* x_out,
                     uint32_t* z_out, int* L_out, int* L_pre, int* L_post) {
    using namespace dvqls;
    if (!ctx) return DVQLS_ERR_INVALID_ARG;
    ctx->err.clear();
    const bool dense = A_in != nullptr;
    if (n < 1 || n > (dense ? DVQLS_MAX_DENSE_QUBITS : DVQLS_MAX_QUBITS))
        return set_error(ctx, DVQLS_ERR_INVALID_ARG, "n = %d out of range", n);
    if (L_max < 1) return set_error(ctx, DVQLS_ERR_INVALID_ARG, "L_max must be >= 1");
    if (L_max > MAX_TERMS)
        return set_error(ctx, DVQLS_ERR_UNSUPPORTED, "L_max = %d above the supported %d", L_max, MAX_TERMS);
    if (tau != tau || tau == -INFINITY) return set_error(ctx, DVQLS_ERR_INVALID_ARG, "tau is NaN");
    if (!coef_out || !x_out || !z_out || !L_out || !L_pre || !L_post)
        return set_error(ctx, DVQLS_ERR_INVALID_ARG, "NULL output");
    Band bd{};
    const long long N = 1LL << n;
    if (!dense) {
        if (nbands < 1 || nbands > MAX_BANDS || !offsets || !bands_in)
            return set_error(ctx, DVQLS_ERR_INVALID_ARG, "need 1..%d bands", MAX_BANDS);
        if (is_device_ptr(ctx, offsets)) return set_error(ctx, DVQLS_ERR_INVALID_ARG, "offsets must be host memory");
        bd.nbands = nbands;
        for (int k = 0; k < nbands; ++k) {
            if (offsets[k] <= -N || offsets[k] >= N)
                return set_error(ctx, DVQLS_ERR_INVALID_ARG, "band offset %d out of range", offsets[k]);
            for (int j = 0; j < k; ++j)
                if (offsets[j] == offsets[k]) return set_error(ctx, DVQLS_ERR_INVALID_ARG, "repeated band offset");
            bd.off[k] = offsets[k];
        }
    }
    cudaSetDevice(ctx->device);

    // Plan: the input, the counters, the selection's bins and the flags (one
    // clear), the masks, the candidates and the results; then, once the number
    // of masks is known, one FP64 value per coefficient.
    const size_t in_bytes = dense ? size_t(N) * N * 8 : size_t(nbands) * N * 8;
    const int chunks = ceil_div(N, CMP_CHUNK);
    Arena ar;
    const size_t o_in = ar.reserve(in_bytes);
    const size_t o_misc = ar.reserve(sizeof(Misc));
    const size_t o_hist = ar.reserve(SEL_BINS * 4);
    const size_t o_flags = ar.reserve(size_t(chunks) * CMP_CHUNK);
    const size_t clear = ar.total() - o_misc;
    const size_t o_cnt = ar.reserve(size_t(chunks) * 4);
    const size_t o_masks = ar.reserve(N * 4);
    const size_t o_cand = ar.reserve(size_t(SEL_CAP) * 16);
    const size_t o_out = ar.reserve(size_t(L_max) * 24);
    int rc = ensure_workspace(ctx, ar.total());
    if (rc) return rc;
    rc = ensure_pinned(ctx, in_bytes + 4096 + size_t(L_max) * 24);
    if (!rc) rc = pin_acquire(ctx);
    if (rc) return rc;
    const size_t p_misc = (in_bytes + 255) & ~size_t(255), p_out = p_misc + 256;
    Misc* hm = reinterpret_cast<Misc*>(ctx->pin + p_misc);
    const double* dA = (const double*)stage_in(ctx, dense ? A_in : bands_in, in_bytes, 0, o_in);
    DVQLS_CUDA_TRY(ctx, cudaMemsetAsync(ctx->ws + o_misc, 0, clear, ctx->stream));
    auto misc_dev = [&]() { return reinterpret_cast<Misc*>(ctx->ws + o_misc); };
    auto masks_dev = [&]() { return reinterpret_cast<uint32_t*>(ctx->ws + o_masks); };
    auto hist_dev = [&]() { return reinterpret_cast<uint32_t*>(ctx->ws + o_hist); };
    unsigned char* flags = (unsigned char*)(ctx->ws + o_flags);
    int* cnt = (int*)(ctx->ws + o_cnt);
    const int grid = ctx->num_sms * 8;
    if (dense) k_flags_dense<<<grid, 256, 0, ctx->stream>>>(dA, n, flags, ctx->d_status);
    else k_flags_banded<<<grid, 256, 0, ctx->stream>>>(n, bd, dA, flags, ctx->d_status);
    if (chunks > 1) k_mask_count<<<chunks, CMP_T, 0, ctx->stream>>>(flags, cnt);
    k_mask_write<<<chunks, CMP_T, 0, ctx->stream>>>(flags, cnt, masks_dev(), &misc_dev()->masks);
    DVQLS_CUDA_TRY(ctx, cudaGetLastError());
    auto read_misc = [&]() -> int {
        DVQLS_CUDA_TRY(ctx, cudaMemcpyAsync(hm, misc_dev(), sizeof(Misc), cudaMemcpyDeviceToHost, ctx->stream));
        return sync_and_check(ctx);
    };
    rc = read_misc();
    if (rc) return rc;
    const int M = hm->masks;
    if (M == 0) {
        *L_out = *L_pre = *L_post = 0;
        return DVQLS_OK;
    }

    // Second plan: everything above stays in place (same offsets), append
    // the M x N values.
    const long long E = (long long)M * N;
    const size_t o_val = ar.reserve(size_t(E) * 8);
    if (ar.total() > ctx->ws_cap) {
        // Growing reallocates: the staged input, the masks and the cleared
        // counters must be rebuilt, so copy the small mask list out and back.
        std::vector<uint32_t> hmask(M);
        DVQLS_CUDA_TRY(ctx, cudaMemcpy(hmask.data(), masks_dev(), size_t(M) * 4, cudaMemcpyDeviceToHost));
        rc = ensure_workspace(ctx, ar.total());
        if (rc) return rc;
        dA = (const double*)stage_in(ctx, dense ? A_in : bands_in, in_bytes, 0, o_in);
        DVQLS_CUDA_TRY(ctx, cudaMemcpyAsync(masks_dev(), hmask.data(), size_t(M) * 4, cudaMemcpyHostToDevice, ctx->stream));
        DVQLS_CUDA_TRY(ctx, cudaStreamSynchronize(ctx->stream));
        DVQLS_CUDA_TRY(ctx, cudaMemsetAsync(ctx->ws + o_misc, 0, clear, ctx->stream));
    }
    char* ws = ctx->ws;
    Misc* misc = misc_dev();
    uint32_t* masks = masks_dev();
    uint32_t* hist = hist_dev();
    double* val = (double*)(ws + o_val);
    const double* dense_in = dense ? dA : nullptr;
    const double* band_in = dense ? nullptr : dA;
    if (n <= LO_BITS) {
        const size_t smem = SEL_BINS * 4 + size_t(N + N / 16) * 8;
        DVQLS_CUDA_TRY(ctx, allow_dynamic_smem((const void*)k_fwht_smem));
        k_fwht_smem<<<M, FW_T, smem, ctx->stream>>>(dense_in, bd, band_in, n, masks, val, misc, hist);
    } else {
        k_fwht_lo<<<M * int(N >> LO_BITS), FW_T, 0, ctx->stream>>>(dense_in, bd, band_in, n, masks, val);
        const size_t elems = size_t(N >> LO_BITS) * HI_TILE, smem = SEL_BINS * 4 + (elems + elems / 16) * 8;
        DVQLS_CUDA_TRY(ctx, allow_dynamic_smem((const void*)k_fwht_hi));
        k_fwht_hi<<<M * (LO / HI_TILE), FW_T, smem, ctx->stream>>>(n, val, misc, hist);
    }
    unsigned long long* cand_k = (unsigned long long*)(ws + o_cand);
    unsigned long long* cand_p = cand_k + SEL_CAP;
    // Results go straight to device outputs of natural alignment, else
    // through the workspace.
    auto direct = [&](const void* p, size_t align) {
        return is_device_ptr(ctx, p) && reinterpret_cast<uintptr_t>(p) % align == 0;
    };
    const bool d_c = direct(coef_out, 8), d_x = direct(x_out, 4), d_z = direct(z_out, 4);
    double* oc = d_c ? coef_out : (double*)(ws + o_out);
    uint32_t* ox = d_x ? x_out : (uint32_t*)(ws + o_out + size_t(L_max) * 16);
    uint32_t* oz = d_z ? z_out : (uint32_t*)(ws + o_out + size_t(L_max) * 20);
    const bool host_out = !is_device_ptr(ctx, coef_out) || !is_device_ptr(ctx, x_out) || !is_device_ptr(ctx, z_out);
    DVQLS_CUDA_TRY(ctx, allow_dynamic_smem((const void*)k_sel_emit));
    const int egrid = (int)std::min<long long>(grid, ceil_div(E, 1024));
    auto collect = [&](int count) -> int {
        k_sel_collect<<<egrid, 256, 0, ctx->stream>>>(val, E, tau, count, misc, cand_k, cand_p);
        k_sel_emit<<<1, SEL_T, size_t(SEL_CAP) * 16, ctx->stream>>>(misc, cand_k, cand_p, val, masks, n, L_max, oc, ox, oz);
        DVQLS_CUDA_TRY(ctx, cudaGetLastError());
        if (host_out)  // with the counters in one synchronisation
            DVQLS_CUDA_TRY(ctx, cudaMemcpyAsync(ctx->pin + p_out, ws + o_out, size_t(L_max) * 24, cudaMemcpyDeviceToHost,
                                                ctx->stream));
        return read_misc();
    };
    k_sel_pick<<<1, SEL_T, 0, ctx->stream>>>(0, tau, L_max, misc, hist);
    rc = collect(1);
    if (!rc && !hm->done) {
        // All rounds without a look from the host (a round after the last one needed ends at once):
        // with a synchronisation each, 65,536 equal keys took 323 us in all.
        for (int round = 1; round < SEL_ROUNDS; ++round) {
            k_sel_hist<<<egrid, 256, 0, ctx->stream>>>(round, val, E, tau, misc, hist);
            k_sel_pick<<<1, SEL_T, 0, ctx->stream>>>(round, tau, L_max, misc, hist);
        }
        DVQLS_CUDA_TRY(ctx, cudaGetLastError());
        rc = collect(0);
    }
    if (rc) return rc;
    const int L = hm->l_out;
    auto give = [&](void* dst, bool straight, const void* dev, size_t pin_off, size_t bytes) -> int {
        if (straight || bytes == 0) return DVQLS_OK;
        if (!is_device_ptr(ctx, dst)) {
            memcpy(dst, ctx->pin + pin_off, bytes);
            return DVQLS_OK;
        }
        DVQLS_CUDA_TRY(ctx, cudaMemcpyAsync(dst, dev, bytes, cudaMemcpyDeviceToDevice, ctx->stream));
        DVQLS_CUDA_TRY(ctx, cudaStreamSynchronize(ctx->stream));
        return DVQLS_OK;
    };
    rc = give(coef_out, d_c, oc, p_out, size_t(L) * 16);
    if (!rc) rc = give(x_out, d_x, ox, p_out + size_t(L_max) * 16, size_t(L) * 4);
    if (!rc) rc = give(z_out, d_z, oz, p_out + size_t(L_max) * 20, size_t(L) * 4);
    if (rc) return rc;
    *L_out = L;
    *L_pre = hm->l_pre;
    *L_post = hm->l_post;
    return DVQLS_OK;
}

}  // namespace

extern "C" int dvqls_pauli_decompose(dvqls_ctx* ctx, const double* A, int n, double tau, int L_max, double* coef,
                                     uint32_t* xmask, uint32_t* zmask, int* L_out, int* L_pre, int* L_post) {
    DVQLS_NVTX("dvqls_pauli_decompose");
    if (!A) return ctx ? dvqls::set_error(ctx, DVQLS_ERR_INVALID_ARG, "A is NULL") : DVQLS_ERR_INVALID_ARG;
    return decompose_common(ctx, A, n, 0, nullptr, nullptr, tau, L_max, coef, xmask, zmask, L_out, L_pre, L_post);
}

extern "C" int dvqls_pauli_decompose_banded(dvqls_ctx* ctx, int n, int nbands, const int* offsets,
                                            const double* band_values, double tau, int L_max, double* coef,
                                            uint32_t* xmask, uint32_t* zmask, int* L_out, int* L_pre, int* L_post) {
    DVQLS_NVTX("dvqls_pauli_decompose_banded");
    return decompose_common(ctx, nullptr, n, nbands, offsets, band_values, tau, L_max, coef, xmask, zmask, L_out,
                            L_pre, L_post);
}
