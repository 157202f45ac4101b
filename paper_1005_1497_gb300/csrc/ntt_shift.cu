// ntt_shift.cu -- the strict bit-shift form of the transform (Sec. I, Eq. 2
// and 3 "only bit-shifting, modulo and addition"; Sec. III-A, Prop. 2) for
// the regime where it is literal: a Rader prime m dividing a Fermat number
// F_t = 2^(2^t) + 1 with ord_m(2) = 2^(t+1), so every twiddle is 2^e with
// e < 2^t and N <= 2^(t+1) (t = 4: m = 65537, N <= 32; t = 5: m = 641 or
// 6700417, N <= 64).
//
// SHIFT mode computes the convolution modulo F_t (a multiple of m) and
// reduces modulo m at the end:
//   * a twiddle product b 2^e (b <= 2^(2^t), e < 2^t) is the shift b << e
//     followed by the reduction lo - hi modulo F_t (2^(2^t) = -1): no
//     multiply in any butterfly;
//   * N^-1 = 2^-L = -2^(2^t - L) modulo F_t is a shift and a negation;
//   * the N pointwise products F G are genuine products (the convolution
//     theorem needs them), reduced the same way;
//   * the final residue modulo m uses one Shoup product per output.
// SHOUP mode is the same kernel with every twiddle applied as a Shoup
// product modulo m (the multiply form of the main path), for comparison.
//
// Layout.  E = min(8, N) elements per thread, T = N / E threads per pair.
// Pass 1: a thread holds x = q + T k (k < E, q its place among the T), so
// the three top levels act inside it and their shift amounts are compile-time constants.
// Pass 2 (N > 8): after an exchange through the warp's shared memory it
// holds x = E q + k, and the remaining levels' amounts are one exponent of q
// and constants.  Forward: the node tree of the main path (node i = x >> (L -
// d), twiddle w^brv(i)); inverse: its transpose, output at <-x>_N.  Every
// pair's words move as whole 32-byte sectors.
//
// SHIFT mode keeps values lazily, as signed words (64 bits for F_5, 32 for
// F_4): a twiddle product leaves lo - hi without a fix-up and sums are never
// reduced.  |x| < 2^36 after the forward levels and < 2^40 after the inverse ones
// for F_5 (inputs < 2^23, each level adds at most 2^32 + half the bound),
// < 2^21 and < 2^24 for F_4 (K = 16).
//
// What bounds it: integer instructions (five for a twiddle product, four for
// a butterfly's sums; the schedulers issue in 77% of cycles, the ALU pipe is
// 76% busy).  Measured on GB300 at 1000003 x 64, m = 641: 252 us, 3.0 TB/s
// (0.45 of the copy rate); one or two elements per lane, with shuffles at
// every level and each sum reduced to [0, F_t], took 1772 us.
#include <cuda_runtime.h>

#include <cstring>

#include "../../include/ntt_gb300.h"
#include "ntt_count.h"
#include "ntt_internal.h"
#include "nt_host.h"

namespace {

constexpr int BLK = 256;

struct ShiftArgs {
    const uint32_t *f;
    const uint32_t *g;
    uint32_t *h;
    long long batch;
    uint64_t m;              // the Rader prime (result modulus)
    uint64_t onep;           // floor(2^64 / m)
    // SHOUP mode: twiddles z_i = w^brv(i) mod m and Shoup quotients, i < N/2
    uint32_t z[32];
    uint32_t zp[32];
    uint32_t ninv, ninvp;    // N^-1 mod m, Shoup quotient (SHOUP mode)
    uint32_t onep32;         // floor(2^32 / m)
    uint32_t big;            // the largest multiple of m below 2^31
};

// Exponent of the twiddle of node i at length 2^L: w = 2^(2K/N), z_i = w^brv_{L-1}(i).
template <int K, int L>
__device__ __forceinline__ uint32_t tw_exp(uint32_t i)
{
    return (2u * K >> L) * (__brev(i) >> (32 - (L - 1 > 0 ? L - 1 : 1))) * (L > 1 ? 1u : 0u);
}

// Values, twiddles and reductions of the two modes.
//   Tw: a node's twiddle (an exponent e < K, or a factor and its quotient);
//   mul(b, t): b times it; lift(v): a word in [0, 2^32) equal to v modulo m;
//   point(F, G): F G N^-1; out(v): the canonical residue modulo m.
// Inverse level j (0 the first): sub(x, y, j) is x - y.
template <int K, int L, bool SHIFT> struct Ops;

// ---- modulo F_5 = 2^32 + 1, signed 64-bit words ----
template <int L> struct Ops<32, L, true> {
    using V = int64_t;
    using Tw = uint32_t;
    __device__ __forceinline__ static V load(uint32_t x) { return (V)x; }
    __device__ __forceinline__ static Tw node(uint32_t i, const ShiftArgs &) { return tw_exp<32, L>(i); }
    // b 2^e = B1 2^32 + B0 2^e, B0 the low 32 - e bits of b: 2^32 = -1
    __device__ __forceinline__ static V mul(V b, Tw e, const ShiftArgs &)
    {
        return (V)(uint32_t)((uint32_t)b << e) - (b >> (32u - e));
    }
    __device__ __forceinline__ static V add(V x, V y) { return x + y; }
    __device__ __forceinline__ static V sub(V x, V y, int, const ShiftArgs &) { return x - y; }
    __device__ __forceinline__ static V sub_fwd(V x, V y, const ShiftArgs &) { return x - y; }
    // lo - hi + m with |hi| < 2^8 <= m; past 2^32 a large multiple of m is taken away
    __device__ __forceinline__ static uint32_t lift(V v, const ShiftArgs &a)
    {
        const uint32_t lo = (uint32_t)v, t = (uint32_t)a.m - (uint32_t)(v >> 32);
        const uint32_t r = lo + t;
        return r < lo ? r - a.big : r;
    }
    __device__ __forceinline__ static V point(V F, V G, const ShiftArgs &a)
    {
        const uint64_t p = (uint64_t)lift(F, a) * lift(G, a);
        const V v = (V)(uint32_t)p - (V)(p >> 32);                       // modulo F_5
        return (v >> L) - (V)(uint32_t)((uint32_t)v << (32 - L));        // N^-1 = 2^-L = -2^(32 - L)
    }
    __device__ __forceinline__ static uint32_t out(V v, const ShiftArgs &a)
    {
        const uint32_t r = lift(v, a), s = r - __umulhi(r, a.onep32) * (uint32_t)a.m;
        return min(s, s - (uint32_t)a.m);
    }
};

// ---- modulo F_4 = 2^16 + 1 = m, signed 32-bit words ----
template <int L> struct Ops<16, L, true> {
    using V = int32_t;
    using Tw = uint32_t;
    __device__ __forceinline__ static V load(uint32_t x) { return (V)x; }
    __device__ __forceinline__ static Tw node(uint32_t i, const ShiftArgs &) { return tw_exp<16, L>(i); }
    __device__ __forceinline__ static V mul(V b, Tw e, const ShiftArgs &)
    {
        return (V)(((uint32_t)b << e) & 0xffffu) - (b >> (16u - e));
    }
    __device__ __forceinline__ static V add(V x, V y) { return x + y; }
    __device__ __forceinline__ static V sub(V x, V y, int, const ShiftArgs &) { return x - y; }
    __device__ __forceinline__ static V sub_fwd(V x, V y, const ShiftArgs &) { return x - y; }
    __device__ __forceinline__ static uint32_t canon16(V v)             // |v >> 16| < 2^8: [0, 2^16]
    {
        V r = (V)((uint32_t)v & 0xffffu) - (v >> 16);
        r = r < 0 ? r + 65537 : r;
        return (uint32_t)(r > 65536 ? r - 65537 : r);
    }
    __device__ __forceinline__ static V point(V F, V G, const ShiftArgs &)
    {
        const uint64_t p = (uint64_t)canon16(F) * canon16(G);             // <= 2^32
        const V v = (V)((uint32_t)p & 0xffffu) - (V)(uint32_t)(p >> 16);
        return (v >> L) - (V)(((uint32_t)v << (16 - L)) & 0xffffu);       // N^-1 = -2^(16 - L)
    }
    __device__ __forceinline__ static uint32_t out(V v, const ShiftArgs &) { return canon16(v); }
};

// ---- modulo m with Shoup products (SHOUP mode): forward below 25 m (a unit
// butterfly of levels 0..2 takes y < 4m, every level adds at most 4m),
// inverse below 128 m < 2^30 ----
template <int K, int L> struct Ops<K, L, false> {
    using V = uint32_t;
    struct Tw { uint32_t z, zp; };
    __device__ __forceinline__ static V load(uint32_t x) { return x; }
    __device__ __forceinline__ static Tw node(uint32_t i, const ShiftArgs &a) { return Tw{a.z[i], a.zp[i]}; }
    __device__ __forceinline__ static V mul(V b, Tw t, const ShiftArgs &a) { return b * t.z - __umulhi(b, t.zp) * (uint32_t)a.m; }
    __device__ __forceinline__ static V add(V x, V y) { return x + y; }
    // products are below 2m; the inputs of inverse level j below 2^(j+1) m
    __device__ __forceinline__ static V sub(V x, V y, int j, const ShiftArgs &a) { return x - y + ((uint32_t)a.m << (j + 1)); }
    __device__ __forceinline__ static V sub_fwd(V x, V y, const ShiftArgs &a) { return x - y + 4 * (uint32_t)a.m; }   // y < 4m
    __device__ __forceinline__ static V point(V F, V G, const ShiftArgs &a)
    {
        const uint64_t p = (uint64_t)F * G;
        const uint64_t r = p - __umul64hi(p, a.onep) * a.m;               // [0, 2m)
        return mul((uint32_t)r, Tw{a.ninv, a.ninvp}, a);                  // [0, 2m)
    }
    __device__ __forceinline__ static uint32_t out(V v, const ShiftArgs &a)
    {
        const uint32_t m = (uint32_t)a.m, s = v - __umulhi(v, a.onep32) * m;
        return min(s, s - m);
    }
};

// Levels of one pass over the thread's E elements: register bits HI - 1
// (forward first) down to 0.  tw holds the nodes level by level, the top
// level's E >> HI first; tw_at is the place of the node of element k at
// register bit j.
template <int E, int HI> __device__ __forceinline__ constexpr int tw_at(int k, int j)
{
    return (k >> (j + 1)) + (E >> (j + 1)) - (E >> HI);
}

template <class O, int E, int HI>
__device__ __forceinline__ void fwd(typename O::V (&v)[E], const typename O::Tw *tw, bool first, const ShiftArgs &a)
{
#pragma unroll
    for (int j = HI - 1; j >= 0; --j)
#pragma unroll
        for (int k = 0; k < E; ++k) {
            if (k & (1 << j)) continue;
            const bool one = first && (k >> (j + 1)) == 0;                // node 0: twiddle 1
            const typename O::V x = v[k];
            const typename O::V t = one ? v[k | (1 << j)] : O::mul(v[k | (1 << j)], tw[tw_at<E, HI>(k, j)], a);
            v[k] = O::add(x, t);
            v[k | (1 << j)] = O::sub_fwd(x, t, a);
        }
}

template <class O, int E, int HI>
__device__ __forceinline__ void inv(typename O::V (&v)[E], const typename O::Tw *tw, bool first, int j0, const ShiftArgs &a)
{
#pragma unroll
    for (int j = 0; j < HI; ++j)
#pragma unroll
        for (int k = 0; k < E; ++k) {
            if (k & (1 << j)) continue;
            const bool one = first && (k >> (j + 1)) == 0;
            const typename O::V x = v[k], y = v[k | (1 << j)], d = O::sub(x, y, j0 + j, a);
            v[k] = O::add(x, y);
            v[k | (1 << j)] = one ? d : O::mul(d, tw[tw_at<E, HI>(k, j)], a);
        }
}

template <int K, int L, bool SHIFT>
__global__ void __launch_bounds__(BLK) k_conv_shift(const __grid_constant__ ShiftArgs a)
{
    using O = Ops<K, L, SHIFT>;
    using V = typename O::V;
    using Tw = typename O::Tw;
    constexpr int N = 1 << L, E = N < 8 ? N : 8, T = N / E, LE = L < 3 ? L : 3, L2 = L - LE;
    constexpr int PPW = 32 / T;                            // pairs per warp
    constexpr int PST = N + N / 8;                         // words of a pair's exchange region: x at x + x / 8
    __shared__ V ex[L2 > 0 ? (BLK / 32) * PPW * PST : 1];
    const int lane = threadIdx.x & 31, q = lane & (T - 1);
    V *S = ex + (L2 > 0 ? ((threadIdx.x >> 5) * PPW + lane / T) * PST : 0);
    // pass 1: nodes of the top levels, the same for every thread; pass 2: this thread's
    Tw t1[E], t2[E];
#pragma unroll
    for (int j = LE - 1, n = 0; j >= 0; --j)
#pragma unroll
        for (int i = 0; i < (E >> (j + 1)); ++i, ++n) t1[n] = O::node((uint32_t)i, a);
    if constexpr (L2 > 0) {
#pragma unroll
        for (int j = L2 - 1, n = 0; j >= 0; --j)
#pragma unroll
            for (int i = 0; i < (E >> (j + 1)); ++i, ++n) t2[n] = O::node((uint32_t)(q * (E >> (j + 1)) + i), a);
    }
    auto to_rows = [&](V (&v)[E]) {                        // pass 1 layout -> pass 2 layout
        __syncwarp();
#pragma unroll
        for (int k = 0; k < E; ++k) S[(q + T * k) + (q + T * k) / 8] = v[k];
        __syncwarp();
#pragma unroll
        for (int k = 0; k < E; ++k) v[k] = S[9 * q + k];
    };
    const long long gwarp = ((long long)blockIdx.x * BLK + threadIdx.x) >> 5;
    const long long nwarp = ((long long)gridDim.x * BLK) >> 5;
    for (long long base = gwarp * PPW; base < a.batch; base += nwarp * PPW) {
        const long long pair = base + lane / T;
        const bool live = pair < a.batch;
        const uint32_t *f = a.f + pair * N + q, *g = a.g + pair * N + q;
        V v[E], w[E];
#pragma unroll
        for (int k = 0; k < E; ++k) {
            v[k] = O::load(live ? f[T * k] : 0u);
            w[k] = O::load(live ? g[T * k] : 0u);
        }
        fwd<O, E, LE>(v, t1, true, a);
        fwd<O, E, LE>(w, t1, true, a);
        if constexpr (L2 > 0) {
            to_rows(v);
            fwd<O, E, L2>(v, t2, false, a);
            to_rows(w);
            fwd<O, E, L2>(w, t2, false, a);
        }
#pragma unroll
        for (int k = 0; k < E; ++k) v[k] = O::point(v[k], w[k], a);
        if constexpr (L2 > 0) {
            inv<O, E, L2>(v, t2, false, 0, a);
            __syncwarp();
#pragma unroll
            for (int k = 0; k < E; ++k) S[9 * q + k] = v[k];
            __syncwarp();
#pragma unroll
            for (int k = 0; k < E; ++k) v[k] = S[(q + T * k) + (q + T * k) / 8];
        }
        inv<O, E, LE>(v, t1, true, L2, a);
        if (live) {
#pragma unroll
            for (int k = 0; k < E; ++k) {
                const uint32_t x = (uint32_t)(q + T * k);
                a.h[pair * N + ((N - x) & (N - 1))] = O::out(v[k], a);
            }
        }
    }
}

template <int K, bool SHIFT>
cudaError_t launch(int L, const ShiftArgs &a, int grid, cudaStream_t st)
{
    switch (L) {
#define C(X) case X: if constexpr ((2 * K >> X) >= 1) { k_conv_shift<K, X, SHIFT><<<grid, BLK, 0, st>>>(a); return ntt::launched(); } break;
    C(1) C(2) C(3) C(4) C(5) C(6)
#undef C
    default: break;
    }
    return cudaErrorInvalidValue;
}

}  // namespace

extern "C" ntt_status conv_circular_shift(uint64_t m, uint32_t N, const uint32_t *f, const uint32_t *g, uint32_t *h,
                                          size_t batch, int mode, ntt_stream_t stream)
{
    if (!f || !g || !h || batch == 0 || (mode != NTT_SHIFT_STRICT && mode != NTT_SHIFT_SHOUP))
        return ntt_fail(NTT_ERR_ARG, "conv_circular_shift: invalid argument");
    int t = 0;
    if (m > 2 && ((1ull << 32) + 1) % m == 0) t = 5;
    else if (m > 2 && ((1ull << 16) + 1) % m == 0) t = 4;
    if (t == 0 || !nt::is_prime(m))
        return ntt_fail(NTT_ERR_MODULUS, "conv_circular_shift: m=%llu is not a prime factor of F_4 or F_5",
                        (unsigned long long)m);
    const uint32_t nmax = 2u << t;                       // ord_m(2) = 2^(t+1)
    if (nt::order_of_two_pow2(m) != nmax)
        return ntt_fail(NTT_ERR_MODULUS, "conv_circular_shift: ord_m(2) != 2^%d", t + 1);
    if (N < 2 || (N & (N - 1)) || N > nmax)
        return ntt_fail(NTT_ERR_LENGTH, "conv_circular_shift: N=%u must be a power of two in 2..%u", N, nmax);
    int L = 0;
    while ((1u << L) < N) ++L;
    ShiftArgs a{};
    a.f = f; a.g = g; a.h = h; a.batch = (long long)batch; a.m = m;
    a.onep = (uint64_t)(((unsigned __int128)1 << 64) / m);
    a.onep32 = (uint32_t)((1ull << 32) / m);
    a.big = (uint32_t)((1ull << 31) / m * m);
    const uint64_t w = nt::pow_mod(2, nmax / N, m);
    for (uint32_t i = 0; i < N / 2; ++i) {
        uint32_t r = 0;
        for (int k = 0; k < L - 1; ++k) r |= ((i >> k) & 1u) << (L - 2 - k);
        a.z[i] = (uint32_t)nt::pow_mod(w, r, m);
        a.zp[i] = (uint32_t)(((uint64_t)a.z[i] << 32) / m);
    }
    a.ninv = (uint32_t)nt::pow_mod(N % m, m - 2, m);
    a.ninvp = (uint32_t)(((uint64_t)a.ninv << 32) / m);
    int dev = 0, nsm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    const long long pairs_per_block = (long long)BLK / (N < 8 ? 1 : N / 8);
    const long long need = ((long long)batch + pairs_per_block - 1) / pairs_per_block;
    const int grid = (int)(need < (long long)nsm * 8 ? need : (long long)nsm * 8);
    cudaStream_t st = (cudaStream_t)stream;
    cudaError_t e;
    if (t == 5) e = mode == NTT_SHIFT_STRICT ? launch<32, true>(L, a, grid, st) : launch<32, false>(L, a, grid, st);
    else e = mode == NTT_SHIFT_STRICT ? launch<16, true>(L, a, grid, st) : launch<16, false>(L, a, grid, st);
    if (e != cudaSuccess) return ntt_fail(NTT_ERR_CUDA, "conv_circular_shift: %s", cudaGetErrorString(e));
    return NTT_OK;
}
