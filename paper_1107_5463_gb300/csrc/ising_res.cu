// Byte-Ising sweeps of lattices that fit the chip's shared memory: one launch
// runs many checkerboard sweeps (Metropolis or heat-bath, uniform or +-1
// couplings) with the spins resident in shared memory, so a sweep costs no
// launches and no trips to L2 for its neighbours.
//
// The lattice is split along its slowest axis (y in 2D, z in 3D) over G
// blocks, one per multiprocessor; block r owns planes z0 .. z0 + n - 1 of both
// colours.  A pass updates the block's groups of one colour; one block barrier
// separates the passes.
//   One block (MULTI = false) keeps a copy of the last plane before the first
//          one and of the first behind the last; the threads that update those
//          planes write the copies too.
//   Several blocks write their first and last planes to the lattice's arrays
//          in global memory, each word of four spins tagged in the spare upper
//          bits of its bytes with the number of the pass; a thread that needs
//          such a word polls it for the tag of the pass before its own.  Data
//          and flag are one 32-bit word, so no fence, flag or second trip to L2
//          stands between a pass and the next, and only the warps of the
//          boundary planes wait for it while the others go on.
// A boundary word is written again two passes later, by a thread that has by
// then read its neighbours' words of the pass between, and those were written
// by threads that had read this one.  The tags are gone from the
// arrays when the launch ends: a block writes its spins back once both
// neighbours have said (a flag) that they have read its last tagged plane.
// Blocks that wait for one another are launched cooperatively; every wait is
// bounded (the error word's bit 0, reported as SL_ETIMEOUT).  The last block
// to finish turns the summed counts into the E and |m| series, advances the
// sweep counter and clears the flags and sums, so a launch can be captured
// and replayed.
//
// Why: a small lattice spent its time in launches (three graph nodes a sweep,
// 6.2 us at L = 64, whose two passes are 0.3 us of Philox on one
// multiprocessor), and row lengths that are no multiple of 16 bytes ran one
// site at a time with 64-bit index arithmetic (48 flips/ns at L = 1000).
#include <cstring>

#include "ising_group.cuh"

namespace spinmc {
namespace {

constexpr int kResSweeps = 1024;   // sweeps per launch
constexpr int kResMaxBlocks = 256;
constexpr int kResThreads = 1024;
constexpr int kFlagStride = 8;     // flags 32 bytes apart: one L2 sector each
constexpr int kResSmem = 216 * 1024;  // a block's dynamic part; its static arrays take 8.3 KB of 227
constexpr unsigned kResWaitLimit = 1u << 21;  // polls of one word: about a second

// In the upper half of the block partials (which the byte kernels' grids leave alone).
struct ResCtl {
    unsigned flags[kResMaxBlocks * kFlagStride];
    unsigned done;
    unsigned pad;
    unsigned long long sums[2 * kResSweeps];  // unsatisfied bonds, down spins per sweep
};
static_assert(sizeof(ResCtl) <= sizeof(Partial) * (kMaxBlocks - kI8Blocks), "control area");

struct ResArgs {
    int8_t* s[2];
    const int8_t* jb[2][3];
    GroupGeo geo;        // P: entries per plane
    FastDiv Wd, Ld;
    long long N;
    int G, unit, nunits; // planes are dealt out in units (unit * P a multiple of 4)
    int oown, cstride;   // shared memory: first own entry of a colour, bytes per colour
    int jstride;         // bytes of one direction's couplings
    int nsweeps;
    uint32_t replica;
    IsingTable tab;
    RoundKeys rk;
    Ctrl* ctrl;
    ResCtl* ctl;
    double J;
};

// the tag of a pass (1 .. 2 kResSweeps) in the upper bits of a word's bytes
__device__ __forceinline__ uint32_t pass_tag(unsigned pass)
{
    return (pass & 0x7Fu) << 1 | (pass >> 7 & 0x7Fu) << 9;
}

__device__ __forceinline__ uint32_t ld_word(const void* p)
{
    uint32_t v;
    asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ void st_word(void* p, uint32_t v)
{
    asm volatile("st.relaxed.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// the spins of a word once it carries `tag` (0: at once); false if it never did
__device__ __forceinline__ bool wait_word(const void* p, uint32_t tag, uint32_t& v)
{
    unsigned it = 0;
    do {
        v = ld_word(p);
    } while (tag != 0u && (v & 0xFEFEFEFEu) != tag && ++it < kResWaitLimit);
    v &= 0x01010101u;
    return it < kResWaitLimit;
}

// first plane of block r
__device__ __forceinline__ int first_plane(const ResArgs& a, int r)
{
    const int z = (int)((long long)r * a.nunits / a.G) * a.unit;
    return z < a.geo.L ? z : a.geo.L;
}

template <int C>
struct Int {
    static constexpr int value = C;
};

template <int D, bool ALIGNED, bool BONDS, bool HB, bool MULTI>
__global__ void __launch_bounds__(kResThreads, 1) i8_resident(const ResArgs a)
{
    extern __shared__ __align__(16) uint8_t rsm[];
    __shared__ uint32_t s_hb[16];
    __shared__ unsigned s_sum[2 * kResSweeps];
    __shared__ bool s_last;
    const int T = blockDim.x, tid = threadIdx.x, r = blockIdx.x, G = a.G;
    const int z0 = first_plane(a, r);
    const int np = (r + 1 == G ? a.geo.L : first_plane(a, r + 1)) - z0;
    const int P = a.geo.P, W = a.geo.W, L = a.geo.L, H = a.geo.H;
    const int base = z0 * P, nown = np * P;  // base is a multiple of 4
    uint8_t* const jsm = rsm + 2 * a.cstride;
    const unsigned long long t0 = a.ctrl->t;

    for (int q = tid; q < 2 * a.nsweeps; q += T) s_sum[q] = 0u;
    if (HB && tid < 13) s_hb[tid] = a.tab.hb[tid];
    // own planes
    for (int c = 0; c < 2; ++c) {
        uint32_t* d = reinterpret_cast<uint32_t*>(rsm + c * a.cstride + a.oown);
        const uint32_t* g = reinterpret_cast<const uint32_t*>(a.s[c] + base);
        if (ALIGNED) {
            for (int q = tid; q < nown / 4; q += T) d[q] = __ldcg(g + q);
        } else {
            for (int q = tid; q < nown; q += T)
                reinterpret_cast<uint8_t*>(d)[q] = (uint8_t)__ldcg(a.s[c] + base + q);
        }
    }
    if (!MULTI) {
        // the copies of the last and first plane
        for (int c = 0; c < 2; ++c) {
            uint8_t* d = rsm + c * a.cstride + a.oown;
            for (int q = tid; q < P; q += T) {
                d[q - P] = (uint8_t)__ldcg(a.s[c] + H - P + q);
                d[nown + q] = (uint8_t)__ldcg(a.s[c] + q);
            }
        }
    }
    if (BONDS) {
        // per colour and direction the sign (0 = +1, 1 = -1) of every own site's bond
        for (int c = 0; c < 2; ++c)
            for (int l = tid; l < nown; l += T) {
                const GroupPos g = group_at<D, false>(l, a.geo, a.Wd, a.Ld, z0 + c);
                const int j = base + l;
                uint8_t* d = jsm + c * 2 * D * a.jstride + l;
                auto put = [&](int dir, int8_t v) { d[dir * a.jstride] = (uint8_t)v; };
                // the x bonds in the order of the neighbour words: parity 0 has its
                // +x neighbour in its own column, parity 1 its -x neighbour
                const int8_t back =
                    a.jb[1 - c][0][g.p ? j : (g.k == 0 ? j + W - 1 : j - 1)];
                const int8_t forth = a.jb[c][0][j];
                put(0, g.p ? back : forth);
                put(1, g.p ? forth : back);
                if (D == 3) {
                    put(2, a.jb[1 - c][1][g.y == 0 ? j + (L - 1) * W : j - W]);
                    put(3, a.jb[c][1][j]);
                }
                put(2 * D - 2, a.jb[1 - c][D - 1][j < P ? j + H - P : j - P]);
                put(2 * D - 1, a.jb[c][D - 1][j]);
            }
    }
    __syncthreads();

    // The random numbers do not depend on the spins: every thread draws those of
    // its first group of the next pass ahead of the barrier.  The place of that group is worked out once for the launch.
    const GroupSign sg = group_sign<D>(a.tab);
    const int l0 = 4 * tid;
    const GroupPos g0 = group_at<D, ALIGNED>(l0, a.geo, a.Wd, a.Ld, z0);
    const bool edge0 = l0 < P || l0 + 4 > nown - P;
    // the planes below the first and above the last own one
    const int jlo = base == 0 ? H - P : base - P, jhi = base + nown == H ? 0 : base + nown;
    bool ok = true;  // no wait has run out
    PhiloxGroups pg = philox_groups((uint32_t)t0, a.replica, kSweep << 1, a.rk);
    uint4 rnd0 = philox_at(pg, (uint32_t)(base + l0) >> 2, a.rk);
    GroupCounts m = {0u, 0u, 0u, 0u};

    // one group of a pass of colour C; edge: it holds sites of the first or last plane
    auto update = [&](auto C, int s, const GroupPos& g, bool edge, const uint4& rnd) {
        constexpr int c = decltype(C)::value;
        // tags of the words this pass reads and writes (the arrays start without)
        const uint32_t waited = pass_tag(2u * (unsigned)s + c);
        const uint32_t tag = pass_tag(2u * (unsigned)s + c + 1u);
        const uint8_t* o = rsm + (1 - c) * a.cstride + a.oown;
        uint8_t* own = rsm + c * a.cstride + a.oown;
        const int l = g.l;
        uint32_t nw[2 * D];
        group_neighbours<D, ALIGNED, true>(o, g, a.geo, c, nw, [&](int e, bool up) {
            const int z = up ? e + P : e - P;
            if (!MULTI || !edge || !(up ? e + 4 > nown - P : e < P))
                return ALIGNED ? *reinterpret_cast<const uint32_t*>(o + z) : read4(o, z);
            if (ALIGNED) {
                uint32_t v;
                if (!wait_word(a.s[1 - c] + (up ? jhi + e - (nown - P) : jlo + e), waited, v))
                    ok = false;
                return v;
            }
            // bytes b0 .. b1 - 1 of the group have their neighbours in the other
            // block's plane, at entries j on: in one of its words or in two
            const int b0 = up ? max(0, nown - P - e) : 0;
            const int b1 = up ? min(4, nown - e) : min(4, P - e);
            const int j = up ? jhi + e + b0 - (nown - P) : jlo + e;
            const int8_t* w = a.s[1 - c] + (j & ~3);
            const bool two = (j & 3) + b1 - b0 > 4;
            uint32_t v0, v1 = waited;
            unsigned it = 0;
            do {
                v0 = ld_word(w);
                if (two) v1 = ld_word(w + 4);
            } while (waited != 0u && ((v0 & 0xFEFEFEFEu) != waited || (v1 & 0xFEFEFEFEu) != waited) &&
                     ++it < kResWaitLimit);
            if (it == kResWaitLimit) ok = false;
            const uint32_t far = __funnelshift_r(v0, v1, 8 * (j & 3)) & 0x01010101u;
            if (b0 == 0 && b1 == 4) return far;
            const uint32_t mask = low_bytes(b1) & ~low_bytes(b0);
            return ((far << (8 * b0)) & mask) | (read4(o, z) & ~mask);
        });
        const uint32_t cur = nw[0];
        const uint32_t av = *reinterpret_cast<const uint32_t*>(own + l);
        // the last group of an odd-sized colour array is not full
        const bool full = ALIGNED || l + 4 <= nown;
        const uint32_t valid =
            full ? 0x01010101u : 0x01010101u & ((1u << (8 * (nown - l))) - 1u);
        if (BONDS) {
#pragma unroll
            for (int q = 0; q < 2 * D; ++q)
                nw[q] ^= *reinterpret_cast<const uint32_t*>(jsm + (c * 2 * D + q) * a.jstride + l);
        }
        const uint32_t an =
            group_update<D, HB, c == 1>(av, nw, cur, rnd, a.tab, sg, s_hb, valid, m);
        if (full) {
            *reinterpret_cast<uint32_t*>(own + l) = an;
        } else {  // the copy of the first plane begins inside the last word
            for (int b = 0; l + b < nown; ++b) own[l + b] = (uint8_t)(an >> (8 * b));
        }
        if (!edge) return;
        if (MULTI) {
            st_word(a.s[c] + base + l, (an & valid) | tag);
        } else if (ALIGNED) {
            if (l < P) *reinterpret_cast<uint32_t*>(own + nown + l) = an;
            if (l >= nown - P) *reinterpret_cast<uint32_t*>(own + l - nown) = an;
        } else {
            for (int b = 0; b < 4 && l + b < nown; ++b) {
                const uint8_t x = (uint8_t)(an >> (8 * b));
                if (l + b < P) own[nown + l + b] = x;
                if (l + b >= nown - P) own[l + b - nown] = x;
            }
        }
    };
    // one pass; false if a wait ran out
    auto run_pass = [&](auto C, int s) {
        constexpr int c = decltype(C)::value;
        if (l0 < nown) update(C, s, g0, edge0, rnd0);
        for (int l = l0 + 4 * T; l < nown; l += 4 * T)
            update(C, s, group_at<D, ALIGNED>(l, a.geo, a.Wd, a.Ld, z0),
                   l < P || l + 4 > nown - P, philox_at(pg, (uint32_t)(base + l) >> 2, a.rk));
        pg = philox_groups((uint32_t)t0 + (uint32_t)s + c, a.replica, (kSweep << 1) | (1 - c), a.rk);
        rnd0 = philox_at(pg, (uint32_t)(base + l0) >> 2, a.rk);
        if (c == 1) {
            const uint32_t v = __reduce_add_sync(0xFFFFFFFFu, unsatisfied_after<D>(m));
            const uint32_t down = __reduce_add_sync(0xFFFFFFFFu, m.down);
            m.na = m.flips = m.flipna = m.down = 0u;
            if ((tid & 31) == 0) {
                atomicAdd(&s_sum[2 * s], v);
                atomicAdd(&s_sum[2 * s + 1], down);
            }
        }
        if (MULTI) return !__syncthreads_or(!ok);
        __syncthreads();
        return true;
    };
    for (int s = 0; s < a.nsweeps; ++s)
        if (!run_pass(Int<0>(), s) || !run_pass(Int<1>(), s)) break;
    if (MULTI) {
        // this block has read its neighbours' last tagged planes (colour 0 of the
        // last sweep) and says so
        if (tid == 0) {
            __threadfence();
            st_word(&a.ctl->flags[r * kFlagStride], 1u);
        }
        if (tid < 2) {
            const int nb = tid ? (r + 1 == G ? 0 : r + 1) : (r == 0 ? G - 1 : r - 1);
            unsigned it = 0;
            while (ld_word(&a.ctl->flags[nb * kFlagStride]) == 0u && ++it < kResWaitLimit) {
            }
            if (it == kResWaitLimit) ok = false;
            __threadfence();
        }
        if (__syncthreads_or(!ok) && tid == 0) atomicOr(&a.ctrl->error, 1u);
    }
    // the spins go back to the lattice, without tags
    for (int c = 0; c < 2; ++c) {
        const uint8_t* d = rsm + c * a.cstride + a.oown;
        if (ALIGNED) {
            for (int q = tid; q < nown / 4; q += T)
                reinterpret_cast<uint32_t*>(a.s[c] + base)[q] = reinterpret_cast<const uint32_t*>(d)[q];
        } else {
            // (with the padding of the lattice's last word, which a tag reaches too)
            for (int q = tid; q < (nown + 3) / 4 * 4; q += T)
                a.s[c][base + q] = q < nown ? (int8_t)d[q] : (int8_t)0;
        }
    }
    if (MULTI) {
        for (int q = tid; q < 2 * a.nsweeps; q += T)
            atomicAdd(&a.ctl->sums[q], (unsigned long long)s_sum[q]);
        __threadfence();
        __syncthreads();
        if (tid == 0) {
            s_last = atomicAdd(&a.ctl->done, 1u) == (unsigned)G - 1;
            __threadfence();
        }
        __syncthreads();
        if (!s_last) return;
    }
    // close the launch's sweeps: E = -J (2d H - 2 v) over the H colour-1 sites
    const bool flipsign = a.tab.sigma_neg && !HB;
    // (series_place; a thread that reads it after the last sweep's has set it finds the same)
    const long long set = a.ctrl->series_base, first = set < 0 ? (long long)t0 : set;
    for (int s = tid; s < a.nsweeps; s += T) {
        long long v, dn;
        if (MULTI) {
            v = (long long)__ldcg(&a.ctl->sums[2 * s]);
            dn = (long long)__ldcg(&a.ctl->sums[2 * s + 1]);
            a.ctl->sums[2 * s] = 0ull;
            a.ctl->sums[2 * s + 1] = 0ull;
        } else {
            v = s_sum[2 * s];
            dn = s_sum[2 * s + 1];
        }
        long long bond = 2LL * D * H - 2 * v;
        if (flipsign) bond = -bond;
        const double E = -a.J * (double)bond;
        const double M = (double)(a.N - 2 * dn);
        const long long k = (long long)t0 + s - first;
        if (a.ctrl->series_E) a.ctrl->series_E[k] = E;
        if (a.ctrl->series_absm) a.ctrl->series_absm[k] = fabs(M) / (double)a.N;
        if (s + 1 == a.nsweeps) {
            a.ctrl->series_base = first;
            a.ctrl->obs[0] = E;
            a.ctrl->obs[1] = M;
            a.ctrl->obs[2] = 0.0;
            a.ctrl->obs[3] = 0.0;
            a.ctrl->t = t0 + (unsigned long long)a.nsweeps;
        }
    }
    if (MULTI) {
        for (int q = tid; q < G; q += T) a.ctl->flags[q * kFlagStride] = 0u;
        if (tid == 0) a.ctl->done = 0u;
    }
}

using ResKernel = void (*)(const ResArgs);

template <int D, bool BONDS, bool HB>
ResKernel res_kernel(bool aligned, bool multi)
{
    if (multi)
        return aligned ? i8_resident<D, true, BONDS, HB, true> : i8_resident<D, false, BONDS, HB, true>;
    return aligned ? i8_resident<D, true, BONDS, HB, false> : i8_resident<D, false, BONDS, HB, false>;
}

ResKernel pick_kernel(const sl_lattice* h, bool multi)
{
    const bool al = h->W % 4 == 0, bonds = h->j_layout == SL_J_BONDS;
    const bool hb = h->update == SL_UPDATE_HEATBATH;
    if (h->d == 2) {
        if (bonds)
            return hb ? res_kernel<2, true, true>(al, multi) : res_kernel<2, true, false>(al, multi);
        return hb ? res_kernel<2, false, true>(al, multi) : res_kernel<2, false, false>(al, multi);
    }
    if (bonds)
        return hb ? res_kernel<3, true, true>(al, multi) : res_kernel<3, true, false>(al, multi);
    return hb ? res_kernel<3, false, true>(al, multi) : res_kernel<3, false, false>(al, multi);
}

struct ResShape {
    int G, unit, nunits, threads, oown, cstride, jstride;
    size_t smem;
};

int up16(long long x) { return (int)((x + 15) / 16 * 16); }

// The split of a lattice over the multiprocessors for calls of `sweeps` sweeps, or false
// if it does not fit or the other kernels are faster.
bool res_shape(const sl_lattice* h, int64_t sweeps, ResShape* y)
{
    if (h->N > (1LL << 28)) return false;  // offsets are 32-bit; far above the capacity
    const int P = (int)h->P;
    y->unit = P % 4 == 0 ? 1 : (P % 2 == 0 ? 2 : 4);
    y->nunits = (h->L + y->unit - 1) / y->unit;
    const int most = h->sms < kResMaxBlocks ? h->sms : kResMaxBlocks;
    // One block, whose passes are a barrier apart, for small lattices; beyond,
    // about 256 groups of each colour per block.
    long long G = h->N <= (P % 4 == 0 ? 5000 : 10000) ? 1 : (h->N + 2047) / 2048;
    if (G > most) G = most;
    if (G > y->nunits) G = y->nunits;
    y->G = (int)G;
    const long long np = (long long)((y->nunits + G - 1) / G) * y->unit;
    const long long nown = np * P;
    y->oown = G == 1 ? up16(P) : 16;  // (a few bytes before the first entry may be read)
    y->cstride = y->oown + up16(nown + P + 12);
    y->jstride = h->j_layout == SL_J_BONDS ? up16(nown) : 0;
    y->smem = 2 * (size_t)y->cstride + 4 * (size_t)h->d * y->jstride;
    const long long groups = (nown + 3) / 4;
    y->threads = groups >= kResThreads ? kResThreads : (int)((groups + 31) / 32 * 32);
    if (y->smem > (size_t)kResSmem) return false;
    if (G == 1) return true;
    // Several blocks finish with the one that owns most sites; the kernels in
    // global memory spread evenly but pay launches.  Microseconds a sweep, fitted to
    // both sides measured at L = 50 to 5120 (2D L = 2048: 6.3 against 10.4 streaming,
    // 4096: 22.0 and 22.5, 5120: 34.2 and 33.3; 3D L = 128: 6.2 and 7.8, 160: 15.0
    // and 11.9; ragged 2D L = 1002: 3.1 and 6.5 flat; 3D L = 102: 10.9 and 8.4).
    const bool al = h->W % 4 == 0, d3 = h->d == 3;
    const double own = 2.0 * (double)nown;
    const double site = d3 ? (al ? (np == 1 ? 0.37e-3 : 0.29e-3) : (np == 1 ? 0.95e-3 : 0.43e-3))
                           : (al ? 0.20e-3 : 0.27e-3);
    const bool bonds = h->j_layout == SL_J_BONDS;
    const bool stream = h->W % 16 == 0;  // else i8_flat, or with bonds i8_generic
    const double other = stream  ? (d3 ? 1.4e-6 : (bonds ? 1.2e-6 : 1.05e-6))
                         : bonds ? 9.2e-6
                                 : (d3 ? (al ? 1.9e-6 : 2.5e-6) : (al ? 1.4e-6 : 1.85e-6));
    const double here = 1.2 + own * site;
    const double there = (bonds && !stream ? 10.2 : 4.6) + (double)h->N * other;
    if (here >= there) return false;
    // A call also moves the spins to shared memory and back and meets its neighbours'
    // blocks at the end (4.4 us more than a graph, 1.2 more than the launches of a single
    // sweep), and puts the signs of its couplings together, so that short calls of large
    // lattices are faster on the other kernels.  (+-1 bonds, 3D L = 128: 24.7 us for one
    // sweep and 18.6, 68.9 and 67.7 for eight, 82.0 and 86.2 for ten; 2D L = 2048: 24.8
    // and 20.6 for one, 38.8 and 43.1 for three; without bonds 3D L = 128 24.4 and 22.5
    // for two, 35.2 and 36.9 for four.  `here` is some 13% above what such lattices take.)
    const double load = bonds ? own * 2 * h->d * 0.055e-3 : 0.0;
    return (double)sweeps * (there - 0.87 * here) > (sweeps == 1 ? 1.2 : 4.4) + load;
}

}  // namespace

bool i8_resident_ok(const sl_lattice* h, int64_t sweeps)
{
    if (h->storage != SL_STORE_I8 || h->slab || h->multihit > 0 || h->kernel != 0 ||
        h->update == SL_UPDATE_SW || h->bonds_have_zero || h->z0 != 0)
        return false;
    // rows and grid caps given by the user shape the streaming kernel
    if ((h->rows > 0 || h->blocks_per_sm > 0) && !h->shape_tuned) return false;
    ResShape y;
    return res_shape(h, sweeps, &y);
}

cudaError_t i8_resident_sweeps(const sl_lattice* h, const SweepParams& p, int64_t* left,
                               cudaStream_t s)
{
    ResShape y;
    if (!res_shape(h, *left, &y)) return cudaSuccess;
    ResArgs a;
    for (int c = 0; c < 2; ++c) {
        a.s[c] = (int8_t*)h->spins[c];
        for (int mu = 0; mu < 3; ++mu) a.jb[c][mu] = (const int8_t*)h->bonds[c][mu];
    }
    a.geo.W = h->W;
    a.geo.L = h->L;
    a.geo.P = (int)h->P;
    a.geo.H = (int)h->H;
    a.Wd = make_fast_div((uint32_t)h->W);
    a.Ld = make_fast_div((uint32_t)h->L);
    a.N = h->N;
    a.G = y.G;
    a.unit = y.unit;
    a.nunits = y.nunits;
    a.oown = y.oown;
    a.cstride = y.cstride;
    a.jstride = y.jstride;
    a.replica = h->replica;
    a.tab = p.tab;
    a.rk = p.rk;
    a.ctrl = h->ctrl;
    a.ctl = (ResCtl*)(h->partials + kI8Blocks);
    a.J = h->J;
    ResKernel k = pick_kernel(h, y.G > 1);
    // (one limit for every lattice: it is the kernel's, and another thread may launch it
    // with another size between this call and the launch)
    cudaError_t e =
        cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, kResSmem);
    while (e == cudaSuccess && *left > 0) {
        a.nsweeps = (int)(*left < kResSweeps ? *left : kResSweeps);
        void* args[] = {&a};
        if (y.G > 1)
            e = cudaLaunchCooperativeKernel((const void*)k, dim3(y.G), dim3(y.threads), args, y.smem,
                                            s);
        else
            e = cudaLaunchKernel((const void*)k, dim3(1), dim3(y.threads), args, y.smem, s);
        if (e == cudaSuccess) *left -= a.nsweeps;
    }
    // Where the context has fewer multiprocessors than the device (a partition of it) the
    // blocks do not all fit, and nothing was launched.
    if (e == cudaErrorCooperativeLaunchTooLarge || e == cudaErrorNotSupported) {
        cudaGetLastError();
        e = cudaSuccess;
    }
    return e;
}

cudaError_t i8_resident_clear(const sl_lattice* h, cudaStream_t s)
{
    return cudaMemsetAsync(h->partials + kI8Blocks, 0, sizeof(ResCtl), s);
}

}  // namespace spinmc
