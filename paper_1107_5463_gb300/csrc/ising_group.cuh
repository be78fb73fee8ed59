// Byte-Ising building blocks of the kernels that give a thread one Philox
// group (4 consecutive colour entries) at a time: i8_flat (ising_i8.cu) reads
// the colour arrays in global memory, i8_resident (ising_res.cu) keeps them in
// shared memory.  Decisions are those of i8_generic and i8_stream bit for bit.
#pragma once

#include "internal.h"

namespace spinmc {

// Per byte: 0x80 minus the number of thresholds below u, i.e. 0x80 - q(u)
// for the four sites of one Philox block (byte b <- output b).
template <int NCMP>
__device__ __forceinline__ uint32_t q_bias(const uint4& r, const IsingTable& tab)
{
    uint32_t acc = 0x80808080u;
    const uint32_t u[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
    for (int b = 0; b < 4; ++b)
#pragma unroll
        for (int k = 0; k < NCMP; ++k) acc -= (u[b] > tab.thr[k]) ? (1u << (8 * b)) : 0u;
    return acc;
}

// Extents: W columns, L rows per plane (3D), P entries per plane along the
// slowest axis, H entries.
struct GroupGeo {
    int W, L, P, H;
};

// Where a group sits, for the pass of colour 0 (the parity of its row is the
// other one in the pass of colour 1): flat colour entry l of the arrays, and
//   ALIGNED (W % 4 == 0, so the group lies in one row and every row neighbour is
//   an aligned word): the entry beside the group that the row's parity calls
//   for in each colour's pass, the byte selector that shifts it in, and the
//   offsets of the rows y -/+ 1;
//   otherwise the column k, row y and parity p of its first site (2D: y is not
//   used).
struct GroupPos {
    int l;
    int edge[2];
    uint32_t sel[2];
    int ym, yp;
    int k, y, p;
};

// par: parity added to that of the row and plane (a block's first plane)
template <int D, bool ALIGNED>
__device__ __forceinline__ GroupPos group_at(int l, const GroupGeo& e, const FastDiv& Wd,
                                             const FastDiv& Ld, int par)
{
    GroupPos g;
    const int row = (int)Wd.div((uint32_t)l);
    const int z = D == 3 ? (int)Ld.div((uint32_t)row) : 0;
    g.l = l;
    g.k = l - row * e.W;
    g.y = D == 3 ? row - z * e.L : row;
    g.p = (g.y + z + par) & 1;
    if (ALIGNED) {
        // parity 0 takes the byte before the word, parity 1 the one after it
        const int before = g.k == 0 ? l + e.W - 1 : l - 1;
        const int after = g.k + 4 == e.W ? l + 4 - e.W : l + 4;
        g.edge[0] = g.p ? after : before;
        g.edge[1] = g.p ? before : after;
        g.sel[0] = g.p ? 0x4321u : 0x2104u;
        g.sel[1] = g.p ? 0x2104u : 0x4321u;
        g.ym = g.y == 0 ? l + (e.L - 1) * e.W : l - e.W;
        g.yp = g.y == e.L - 1 ? l - (e.L - 1) * e.W : l + e.W;
    }
    return g;
}

// The four bytes at o + a (a of any alignment and sign): two words and a shift.
// Reads up to 3 bytes before them and 7 after.
__device__ __forceinline__ uint32_t read4(const uint8_t* o, int a)
{
    const uint32_t* w = reinterpret_cast<const uint32_t*>(o + (a & ~3));
    return __funnelshift_r(w[0], w[1], 8 * (a & 3));
}

// the low n bytes (0 <= n <= 4)
__device__ __forceinline__ uint32_t low_bytes(int n)
{
    return n <= 0 ? 0u : 0xFFFFFFFFu >> (32 - 8 * n);
}

// w with byte b replaced by v
__device__ __forceinline__ uint32_t put_byte(uint32_t w, int b, uint32_t v)
{
    return (w & ~(0xFFu << (8 * b))) | v << (8 * b);
}

// The other colour's bytes beside the group's four sites in the pass of colour
// c, one word per direction: [0] the x neighbour with the site's own column
// (the word at l), [1] the other x neighbour, then -y, +y (3D only), then the
// slowest axis -, +.  slow(l, up) gives the word of the plane before (up =
// false) or after the one that holds entry l.  SLACK: 16 bytes before and after
// the array may be read (shared memory), so short rows are put together without
// branches.
template <int D, bool ALIGNED, bool SLACK, typename Slow>
__device__ __forceinline__ void group_neighbours(const uint8_t* o, const GroupPos& g,
                                                 const GroupGeo& e, int c, uint32_t (&nw)[2 * D],
                                                 Slow slow)
{
    const int l = g.l;
    const uint32_t* ow = reinterpret_cast<const uint32_t*>(o + l);
    const uint32_t cur = ow[0];
    nw[0] = cur;
    nw[2 * D - 2] = slow(l, false);
    nw[2 * D - 1] = slow(l, true);
    if (ALIGNED) {
        nw[1] = __byte_perm(cur, (uint32_t)o[c ? g.edge[1] : g.edge[0]], c ? g.sel[1] : g.sel[0]);
        if (D == 3) {
            nw[2] = *reinterpret_cast<const uint32_t*>(o + g.ym);
            nw[3] = *reinterpret_cast<const uint32_t*>(o + g.yp);
        }
    } else if (e.W >= (SLACK ? 8 : 4)) {
        // the group holds n1 sites of one row and 4 - n1 of the next
        const int p = g.p ^ c, n1 = min(4, e.W - g.k);
        const bool two = n1 < 4, plane = D == 3 && g.y == e.L - 1;  // next row in the next plane
        const int p2 = plane ? p : p ^ 1;
        const uint32_t m1 = low_bytes(n1);
        const uint32_t before = __funnelshift_l(l > 0 ? ow[-1] : 0u, cur, 8);
        const uint32_t after = __funnelshift_r(cur, ow[1], 8);
        uint32_t x = ((p ? after : before) & m1) | ((p2 ? after : before) & ~m1);
        // the bytes that come from the other end of a row: rare on long rows, where
        // most warps skip them, a chain of divergent branches on short ones
        auto edge = [&](bool cond, int b, int i) {
            if (SLACK && e.W < 64) {
                const uint32_t y = put_byte(x, b, o[cond ? i : l]);
                x = cond ? y : x;
            } else if (cond) {
                x = put_byte(x, b, o[i]);
            }
        };
        edge(!p && g.k == 0, 0, l + e.W - 1);
        edge(p && g.k + n1 == e.W, n1 - 1, l + n1 - e.W);
        edge(two && !p2, n1 & 3, l + n1 + e.W - 1);
        nw[1] = x;
        if (D == 3) {
            const int wrap = (e.L - 1) * e.W;
            uint32_t ym = read4(o, g.y == 0 ? l + wrap : l - e.W);
            uint32_t yp = read4(o, plane ? l - wrap : l + e.W);
            // the second row's neighbours where they wrap differently from the first's
            auto second = [&](uint32_t w, int off) {
                if (SLACK) return (w & m1) | (read4(o, l + off) & ~m1);
                for (int b = n1; b < 4; ++b) w = put_byte(w, b, o[l + b + off]);
                return w;
            };
            if (two && plane) {  // row L - 1, then row 0
                ym = second(ym, wrap);
                yp = second(yp, e.W);
            } else if (two && g.y == 0) {
                ym = second(ym, -e.W);
            } else if (two && g.y == e.L - 2) {
                yp = second(yp, -wrap);
            }
            nw[2] = ym;
            nw[3] = yp;
        }
    } else {
        // rows shorter than a group (in shared memory also rows hardly longer): every
        // site finds its own neighbours
        int k = g.k, y = g.y, p = g.p ^ c;
#pragma unroll
        for (int q = 1; q < 2 * D - 2; ++q) nw[q] = 0u;
        uint32_t x = 0u;
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            const int lb = l + b;
            const int xo = p ? (k + 1 == e.W ? lb + 1 - e.W : lb + 1)
                             : (k == 0 ? lb + e.W - 1 : lb - 1);
            x |= (uint32_t)o[xo] << (8 * b);
            if (D == 3) {
                const int ym = y == 0 ? lb + (e.L - 1) * e.W : lb - e.W;
                const int yp = y == e.L - 1 ? lb - (e.L - 1) * e.W : lb + e.W;
                nw[2] |= (uint32_t)o[ym] << (8 * b);
                nw[3] |= (uint32_t)o[yp] << (8 * b);
            }
            if (++k == e.W) {  // next row; a new plane keeps the alternation (L is even)
                k = 0;
                if (D == 2) {
                    p ^= 1;
                } else if (++y == e.L) {
                    y = 0;      // y + z: -(L - 1) + 1, parity unchanged
                } else {
                    p ^= 1;
                }
            }
        }
        nw[1] = x;
    }
}

// What the sign of J does to the number na of unsatisfied bonds: as it is, or
// 2d - na (per byte; both forms one multiply-add).
struct GroupSign {
    uint32_t mul, add;
};

template <int D>
__device__ __forceinline__ GroupSign group_sign(const IsingTable& tab)
{
    GroupSign s;
    s.mul = tab.sigma_neg ? 0xFFFFFFFFu : 1u;
    s.add = tab.sigma_neg ? 0x01010101u * (uint32_t)(2 * D) : 0u;
    return s;
}

template <int D>
__device__ __forceinline__ uint32_t neighbour_sum(const uint32_t (&nw)[2 * D])
{
    uint32_t nd = nw[0] + nw[1] + nw[2] + nw[3];
    if (D == 3) nd += nw[2 * D - 2] + nw[2 * D - 1];
    return nd;
}

// Unsatisfied bonds (in the sense of J > 0) of the group's sites av.
template <int D>
__device__ __forceinline__ uint32_t group_unsatisfied(uint32_t av, const uint32_t (&nw)[2 * D],
                                                      uint32_t valid)
{
    const uint32_t na = (neighbour_sum<D>(nw) ^ (av * 7u)) - av * (uint32_t)(7 - 2 * D);
    return __dp4a(na & (valid * 0xFFu), 0x01010101u, 0u);
}

// Counts of a measuring pass: the unsatisfied bonds after the move (in the
// sense J's sign gives them), na' = na + flip (2d - 2 na), and the down spins.
struct GroupCounts {
    uint32_t na, flips, flipna, down;
};

template <int D>
__device__ __forceinline__ uint32_t unsatisfied_after(const GroupCounts& m)
{
    return m.na + 2 * D * m.flips - 2 * m.flipna;
}

// The new word of the group's sites av from the neighbour words (couplings
// already folded in as sign flips where there are any), and its counts over
// the bytes of `valid`.
template <int D, bool HB, bool MEAS>
__device__ __forceinline__ uint32_t group_update(uint32_t av, const uint32_t (&nw)[2 * D],
                                                 uint32_t cur, const uint4& rnd,
                                                 const IsingTable& tab, const GroupSign& sg,
                                                 const uint32_t* s_hb, uint32_t valid,
                                                 GroupCounts& m)
{
    uint32_t nd = neighbour_sum<D>(nw);
    uint32_t na, flip, an;
    if (HB) {
        // h = 2d - 2 nd; the new spin is down iff u > hb[h + 2d].  (Bytes past the
        // lattice's end hold anything, and they index the table: cleared.)
        nd &= valid * 0xFFu;
        const uint32_t u[4] = {rnd.x, rnd.y, rnd.z, rnd.w};
        flip = 0u;
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            const uint32_t nb = (nd >> (8 * b)) & 0xFFu;
            if (u[b] > s_hb[4 * D - 2 * nb]) flip |= 1u << (8 * b);
        }
        flip &= valid;
        an = flip;
        na = nd;
    } else {
        // own spin down: na = 2d - nd = (nd ^ 7) - (7 - 2d)
        na = (nd ^ (av * 7u)) * sg.mul + sg.add;
        na -= av * (sg.mul * (uint32_t)(7 - 2 * D));
        // byte bit 7 set iff na >= q(u): accept
        flip = ((na + q_bias<D>(rnd, tab)) >> 7) & valid;
        an = av ^ flip;
    }
    if (MEAS) {
        m.na = __dp4a(na, valid, m.na);
        m.flips = __dp4a(flip, valid, m.flips);
        m.flipna = __dp4a(flip, na, m.flipna);
        m.down = __dp4a(an, valid, __dp4a(cur, valid, m.down));
    }
    return an;
}

}  // namespace spinmc
