// Device-side building blocks shared by the spinmc kernels (sm_103a):
// Philox4x32-10, the device control block, and the fixed-order reduction of
// per-block partial sums that finishes every sweep's observables.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace spinmc {

// Philox4x32-10 (Salmon, Moraes, Dror & Shaw, SC'11).  The ten round keys are
// precomputed on the host (key + r * Weyl constant) so that a kernel reads
// them straight from its parameter bank.
struct RoundKeys {
    uint32_t k0[10];
    uint32_t k1[10];
};

__host__ inline RoundKeys make_round_keys(uint64_t seed)
{
    RoundKeys rk;
    uint32_t k0 = (uint32_t)(seed & 0xffffffffu), k1 = (uint32_t)(seed >> 32);
    for (int r = 0; r < 10; ++r) {
        rk.k0[r] = k0;
        rk.k1[r] = k1;
        k0 += 0x9E3779B9u;
        k1 += 0xBB67AE85u;
    }
    return rk;
}

__device__ __forceinline__ uint4 philox4x32_10(uint4 c, const RoundKeys& rk)
{
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        const uint32_t lo0 = c.x * 0xD2511F53u;
        const uint32_t hi0 = __umulhi(c.x, 0xD2511F53u);
        const uint32_t lo1 = c.z * 0xCD9E8D57u;
        const uint32_t hi1 = __umulhi(c.z, 0xCD9E8D57u);
        c = make_uint4(hi1 ^ c.y ^ rk.k0[r], lo1, hi0 ^ c.w ^ rk.k1[r], lo0);
    }
    return c;
}

// Philox4x32-10 of counters (g, t, replica, w) that differ only in g: what the
// first two rounds make of the other three words is worked out once (2 of the
// 20 wide multiplies, and the XORs around them).
struct PhiloxGroups {
    uint32_t z1, x2, z2, w2;
};

__device__ __forceinline__ PhiloxGroups philox_groups(uint32_t t, uint32_t replica, uint32_t w,
                                                      const RoundKeys& rk)
{
    const uint64_t p = (uint64_t)replica * 0xCD9E8D57u;
    const uint32_t x1 = (uint32_t)(p >> 32) ^ t ^ rk.k0[0];
    const uint64_t q = (uint64_t)x1 * 0xD2511F53u;
    PhiloxGroups c;
    c.z1 = w ^ rk.k1[0];
    c.x2 = (uint32_t)p ^ rk.k0[1];
    c.z2 = (uint32_t)(q >> 32) ^ rk.k1[1];
    c.w2 = (uint32_t)q;
    return c;
}

// What the first two rounds make of g alone, for one z1 (a colour's w).
struct PhiloxHead {
    uint32_t x, y, z;
};

__device__ __forceinline__ PhiloxHead philox_head(uint32_t g, uint32_t z1)
{
    const uint64_t p0 = (uint64_t)g * 0xD2511F53u;
    const uint64_t p1 = (uint64_t)((uint32_t)(p0 >> 32) ^ z1) * 0xCD9E8D57u;
    PhiloxHead h;
    h.x = (uint32_t)(p1 >> 32);
    h.y = (uint32_t)p1;
    h.z = (uint32_t)p0;
    return h;
}

// Both parts and the other eight rounds.
__device__ __forceinline__ uint4 philox_tail(const PhiloxHead& h, uint32_t x2, uint32_t z2,
                                             uint32_t w2, const RoundKeys& rk)
{
    uint4 c = make_uint4(h.x ^ x2, h.y, h.z ^ z2, w2);
#pragma unroll
    for (int r = 2; r < 10; ++r) {
        const uint64_t a = (uint64_t)c.x * 0xD2511F53u;
        const uint64_t b = (uint64_t)c.z * 0xCD9E8D57u;
        c = make_uint4((uint32_t)(b >> 32) ^ c.y ^ rk.k0[r], (uint32_t)b,
                       (uint32_t)(a >> 32) ^ c.w ^ rk.k1[r], (uint32_t)a);
    }
    return c;
}

__device__ __forceinline__ uint4 philox_at(const PhiloxGroups& pg, uint32_t g, const RoundKeys& rk)
{
    return philox_tail(philox_head(g, pg.z1), pg.x2, pg.z2, pg.w2, rk);
}

enum Purpose : uint32_t { kSweep = 0, kInit = 1, kCoupling = 2, kExchange = 3 };

// Device control block: one per lattice, inside the caller's buffer.
struct Ctrl {
    unsigned long long t;      // index of the sweep in progress
    long long series_base;     // sweep index written to series[0]; -1: that of the next one closed
    double* series_E;          // per-sweep energy, or null
    double* series_absm;       // per-sweep |m|, or null
    unsigned int done;         // blocks finished in the measuring pass
    unsigned int error;        // bit 0: a bounded device-side wait ran out (sticky)
    double obs[4];             // E, Mx, My, Mz after the last measured pass
};

// Place in the series of the sweep with index t, which the caller closes.  A call's first
// is its place 0 whatever its index, which runs ahead of the host's count where captured
// calls were replayed and behind it where a launch failed.  (Read here, beside the next
// sweep, and not when the series is set, where the read took up to 2 us of a short call.)
__device__ __forceinline__ long long series_place(Ctrl* c, unsigned long long t)
{
    if (c->series_base < 0) c->series_base = (long long)t;
    return (long long)t - c->series_base;
}

// Partial sums one block contributes to a measured pass.  Ising passes use
// the integer members (exact), continuous spins the double members.
struct Partial {
    long long i0, i1;
    double f[4];
};

// Division of n < 2^31 by a divisor fixed for a launch: a multiply-high and a
// shift in place of the some 20 instructions of a 32-bit division (and 70 of a
// 64-bit one).  With 2^(s-1) < d <= 2^s and m = ceil(2^(31+s) / d) < 2^32 the
// error m d - 2^(31+s) is below 2^s, so n m >> (31 + s) is exact for n < 2^31;
// the shift beyond the high word is kept (d = 1, whose s = 0, is let through).
struct FastDiv {
    uint32_t d, m, s;
    __device__ __forceinline__ uint32_t div(uint32_t n) const
    {
        return d == 1u ? n : __umulhi(n, m) >> s;
    }
};

__host__ inline FastDiv make_fast_div(uint32_t d)
{
    FastDiv f;
    int s = 0;
    while (((uint64_t)1 << s) < d) ++s;
    f.d = d;
    f.m = (uint32_t)((((uint64_t)1 << (31 + s)) + d - 1) / d);
    f.s = (uint32_t)(s > 0 ? s - 1 : 0);
    return f;
}

// Fold one value across a warp (any type with operator+).
template <typename T>
__device__ __forceinline__ T warp_sum(T v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Block-wide sum, result valid in thread 0.  `scratch` holds >= 32 T.
template <typename T>
__device__ __forceinline__ T block_sum(T v, T* scratch)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    v = warp_sum(v);
    __syncthreads();
    if (lane == 0) scratch[warp] = v;
    __syncthreads();
    T r = T(0);
    if (warp == 0) {
        const int nw = (blockDim.x + 31) >> 5;
        r = lane < nw ? scratch[lane] : T(0);
        r = warp_sum(r);
    }
    return r;
}

// Block-wide sums of four doubles, valid in thread 0.  FP64 adds run at two
// lanes per clock and multiprocessor, so a warp's butterfly over each value (20
// warp adds, 180 for a block of 256 threads with the second stage) took 7 to
// 12 us of a measuring pass of 1024 blocks.  Here the lanes split the values
// between them as they fold: after two exchanges each quarter of the warp
// holds one value, 6 warp adds in all, and one warp folds the warps' sums of
// all four values together (51 adds for the block).  `scratch` holds 4 doubles
// per warp; the order of the additions is fixed.
__device__ __forceinline__ void block_sum4(double (&v)[4], double* scratch)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const bool up = (lane & 16) != 0, odd = (lane & 8) != 0;
    // lanes 0-15 keep values 0 and 1, lanes 16-31 values 2 and 3
    double a = up ? v[2] : v[0], b = up ? v[3] : v[1];
    a += __shfl_xor_sync(0xffffffffu, up ? v[0] : v[2], 16);
    b += __shfl_xor_sync(0xffffffffu, up ? v[1] : v[3], 16);
    double x = (odd ? b : a) + __shfl_xor_sync(0xffffffffu, odd ? a : b, 8);
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    __syncthreads();
    if ((lane & 7) == 0) scratch[4 * warp + (lane >> 3)] = x;
    __syncthreads();
    if (warp == 0) {
        // lane (value, slot): the sums of warps slot, slot + 8, ...
        const int nw = (blockDim.x + 31) >> 5;
        x = 0.0;
        for (int w = lane & 7; w < nw; w += 8) x += scratch[4 * w + (lane >> 3)];
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
#pragma unroll
        for (int k = 0; k < 4; ++k) v[k] = __shfl_sync(0xffffffffu, x, 8 * k);
    }
}

// Called by every thread of every block at the end of a measured pass with
// the block's partial (valid in thread 0).  The last block to arrive adds all
// partials: thread k takes blocks k, k + blockDim, ... in order and the block
// tree-sums the threads, a fixed order for a given grid, so FP64 totals are
// reproducible.  Thread 0 of that block passes the totals to `finish` and
// resets the arrival count.  FP: the totals are the double members, else the
// integer ones.
template <bool FP, typename Finish>
__device__ __forceinline__ void finish_pass(Ctrl* ctrl, Partial* partials, const Partial& mine,
                                            Finish finish)
{
    __shared__ bool last;
    __shared__ long long red_i[FP ? 1 : 32];
    __shared__ double red_f[FP ? 128 : 1];
    if (threadIdx.x == 0) {
        partials[blockIdx.x] = mine;
        __threadfence();
        const unsigned prev = atomicAdd(&ctrl->done, 1u);
        last = (prev == gridDim.x - 1);
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    long long i0 = 0, i1 = 0;
    double f[4] = {0.0, 0.0, 0.0, 0.0};
    for (unsigned b = threadIdx.x; b < gridDim.x; b += blockDim.x) {
        const Partial* p = partials + b;
        if (FP) {
#pragma unroll
            for (int k = 0; k < 4; ++k) f[k] += __ldcg(&p->f[k]);
        } else {
            i0 += __ldcg(&p->i0);
            i1 += __ldcg(&p->i1);
        }
    }
    Partial tot;
    if (FP) {
        block_sum4(f, red_f);
    } else {
        i0 = block_sum(i0, red_i);
        i1 = block_sum(i1, red_i);
    }
    tot.i0 = i0;
    tot.i1 = i1;
#pragma unroll
    for (int k = 0; k < 4; ++k) tot.f[k] = f[k];
    if (threadIdx.x == 0) {
        finish(tot);
        ctrl->done = 0;
        __threadfence();
    }
}

// Deferred finishing.  A measuring pass of thousands of short blocks loses
// several percent of its time if every block ends with the fence and the
// arrival atomic above while its SM slot waits.  Instead each block stores
// its partial (no fence, no atomic) and a one-block kernel launched right
// after the pass on the same stream adds them; the kernel boundary orders the
// stores before the loads.  Thread k adds blocks k, k + kFinishThreads, ...
// in order and the block tree-sums the threads: a fixed order for a given
// grid, so FP64 totals stay reproducible.
constexpr int kFinishThreads = 256;

// A continuous-spin block's FP32 sums of a measuring pass, added in FP64;
// scratch holds 4 doubles per warp.
__device__ __forceinline__ Partial fp_partial(float e, float mx, float my, float mz,
                                              double* scratch)
{
    double v[4] = {(double)e, (double)mx, (double)my, (double)mz};
    block_sum4(v, scratch);
    Partial p;
    p.i0 = p.i1 = 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) p.f[k] = v[k];
    return p;
}

// FP32 sum of a thread over a segment of any length, with what the additions round off
// added up beside it, so that it errs by some 2^-40 of the terms' sizes however many there
// are; a plain sum's error grows with them, over 512 rows to 4e-6 of a uniform lattice's M.
// The sum starts at a bias above all it can reach: what x - (t - s) gives is then exactly
// what was lost, as s is the larger one (without it that takes six additions for three).
// (Per sweep, plain sums and these: 3D Heisenberg L = 256 143.8 and 145.1 us, on single
// columns 179.2 and 183.4, L = 128 24.0 and 23.8, 2D L = 2048 35.4 and 35.9; 2D XY L =
// 4096 91.9 and 92.9, L = 1408 20.0 and 19.9.)
struct __align__(8) LongSum {
    float s, lost;
    __device__ __forceinline__ void add(float x)
    {
        const float t = __fadd_rn(s, x);
        lost = __fadd_rn(lost, __fsub_rn(x, __fsub_rn(t, s)));
        s = t;
    }
};

// the exponent of J, between those of 2^-127 and 2^100
__device__ __forceinline__ int coupling_exponent(float J)
{
    return min((int)(__float_as_uint(J) >> 23 & 255u), 227) - 127;
}

// the biases of the energy (k = 0; terms up to 24 |J|) and of M's components (up to 4)
__device__ __forceinline__ float sum_bias(int k, float J)
{
    return __uint_as_float((uint32_t)(127 + (k == 0 ? 17 + coupling_exponent(J) : 14)) << 23);
}

template <int N>
__device__ __forceinline__ void start_sums(LongSum (&v)[N], float J)
{
#pragma unroll
    for (int k = 0; k < N; ++k) {
        v[k].s = sum_bias(k, J);
        v[k].lost = 0.f;
    }
}

// (sum, what rounding took from it) of two such pairs
__device__ __forceinline__ float2 add_pairs(float2 a, float2 b)
{
    const float s = __fadd_rn(a.x, b.x), t = __fsub_rn(s, a.x);
    const float lost = __fadd_rn(__fsub_rn(a.x, __fsub_rn(s, t)), __fsub_rn(b.x, t));
    return make_float2(s, __fadd_rn(lost, __fadd_rn(a.y, b.y)));
}

__device__ __forceinline__ float2 shfl_xor_pair(float2 a, int o)
{
    return make_float2(__shfl_xor_sync(0xffffffffu, a.x, o), __shfl_xor_sync(0xffffffffu, a.y, o));
}

// Totals of a block of 256 threads from such sums, valid in thread 0.  The pairs are added
// up as pairs over the warp, the lanes splitting the values between them as in
// block_sum4; FP64 adds are left to one warp of the block (a warp's own took 1 to 2 us of
// a pass).  The energy is kept in units
// of J's power of two meanwhile, so that no sum of a warp leaves FP32's range whatever J.
template <int N>
__device__ __forceinline__ Partial long_partial(const LongSum (&v)[N], float J)
{
    __shared__ float2 warps[8][4];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const bool up = (lane & 16) != 0, odd = (lane & 8) != 0;
    const int ej = coupling_exponent(J);
    const float scale = __uint_as_float((uint32_t)(127 - ej) << 23);
    float2 f[4];
#pragma unroll
    for (int k = 0; k < 4; ++k)
        f[k] = k < N ? make_float2(v[k % N].s - sum_bias(k, J), v[k % N].lost)
                     : make_float2(0.f, 0.f);
    f[0].x *= scale;
    f[0].y *= scale;
    const float2 a = add_pairs(up ? f[2] : f[0], shfl_xor_pair(up ? f[0] : f[2], 16));
    const float2 b = add_pairs(up ? f[3] : f[1], shfl_xor_pair(up ? f[1] : f[3], 16));
    float2 p = add_pairs(odd ? b : a, shfl_xor_pair(odd ? a : b, 8));
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) p = add_pairs(p, shfl_xor_pair(p, o));
    if ((lane & 7) == 0) warps[warp][lane >> 3] = p;
    __syncthreads();
    Partial tot;
    tot.i0 = tot.i1 = 0;
    if (warp == 0) {
        // lane (value, warp); a sum that is infinite lost nothing
        p = warps[lane & 7][lane >> 3];
        double x = isfinite(p.x) ? (double)p.x + (double)p.y : (double)p.x;
        if (lane < 8) x *= __hiloint2double((1023 + ej) << 20, 0);
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
#pragma unroll
        for (int k = 0; k < 4; ++k) tot.f[k] = __shfl_sync(0xffffffffu, x, 8 * k);
    }
    return tot;
}

__device__ __forceinline__ void store_partial(Partial* partials, const Partial& mine)
{
    if (threadIdx.x == 0) partials[blockIdx.x] = mine;
}

// FP64 totals of the first nblocks partials, valid in thread 0 of a block of
// kFinishThreads.
__device__ __forceinline__ Partial sum_partials(const Partial* partials, unsigned nblocks)
{
    __shared__ double red[4 * (kFinishThreads / 32)];
    double f[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll 4
    for (unsigned b = threadIdx.x; b < nblocks; b += blockDim.x) {
#pragma unroll
        for (int k = 0; k < 4; ++k) f[k] += partials[b].f[k];
    }
    block_sum4(f, red);
    Partial tot;
    tot.i0 = tot.i1 = 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) tot.f[k] = f[k];
    return tot;
}

}  // namespace spinmc
