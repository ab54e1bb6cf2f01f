// ea_bits.cuh -- resident tile of the EA p-bit update for +-1 couplings
// (arXiv 2510.23419: Eqs. 2-3, update groups of Sec. 1.2.2, classical
// annealing of Sec. 1.3.1), one bit per spin.
//
// A tile is 4 WT replicas of one job (WT Philox quads).  A word holds 4
// replicas x G sites of one colour class, G = gcd(L, 8) (2, 4 or 8): with
// Z = L / G, bit 8 b + g of word (q, y, zb, w) is the spin (1 <=> m = -1) of
// replica 4 w + b at z = zb + g Z.  A class rank is k = q + (L/2)(y + L z), so
// word index wi = q + (L/2)(y + L zb) holds the ranks wi + g nw, nw words per
// class and quad.  Neighbour words are whole words: +-z of the edge planes
// zb = 0 and zb = Z - 1 is the same word of the opposite plane with the group
// bits of every byte rotated by one; +-x is the same word of the other class
// and the one at q + 1 or q - 1, chosen per group by the parity of z.
//
// What bounds it: the decisions, one 32-bit Philox word each.  Philox4x32-10 is
// 19 32x32->64 multiplies and 19 three-input logic operations per 4 updates;
// the byte-per-spin tile that this one replaces spent two thirds of its
// instructions on the rest (a neighbour word carried 4 spins).  Here the field
// of 32 updates is 6 loads, 12 sign operations and an 8-operation bit-sliced
// adder (F = 6 - 2 n, n in the three planes p0, p1, p2), the energy one more
// bit-sliced count; per update what is left beside Philox is a byte extraction,
// a threshold load, a compare and a predicated or.
#pragma once

#include "ea_kernels.cuh"
#include "ea_launch.h"
#include "ea_philox.cuh"

namespace pb {

// Flags of a word's position, kept in the top byte of its bond word.
enum : uint32_t {
    kBitQ0 = 1u << 24,
    kBitQL = 1u << 25,
    kBitY0 = 1u << 26,
    kBitYL = 1u << 27,
    kBitZ0 = 1u << 28,
    kBitZL = 1u << 29,
    kBitPar = 1u << 30,  // (y + zb) odd
};

__device__ __forceinline__ uint32_t bytes4(uint32_t v) { return v * 0x01010101u; }

template <int G, int CPT, bool COL, bool HH>
struct EaBitTile {
    static constexpr int LPW = G / CPT;  // lanes that share a word, CPT of its G Philox calls each
    // one Philox call per thread and class: few warps, so a half-sweep is one chain of latencies; the words
    // of the next half-sweep (their counters depend on no spin) are drawn beside it
    static constexpr bool kAhead = CPT == 1;
    static constexpr uint32_t kGroups = (1u << G) - 1u;
    static constexpr uint32_t kLive = kGroups * 0x01010101u;  // bits that hold spins

    // offsets (words) of the neighbours of a word of the tile
    struct Geo {
        int lin;  // own index: wi WT + w
        int qp, qm, yp, ym, zp, zm;
        uint32_t f;  // position flags
        bool live;
    };

    const EaJob& job;
    int tile, t, T, lane, L, h2, Z, nw, half, WT, wsh, nlin, step, lin0, W, w, sub, nrep;
    bool quad_live;
    uint32_t tq;
    uint32_t *c0, *c1, *best;
    uint32_t* bonds;
    int8_t* sh8;
    unsigned char* tab;   // without fields: three tables of two rows (sweep parities), at a fixed address
    unsigned char* htab;  // with fields: two rows
    int htab_bytes;
    Geo col;  // COL: the x and y neighbours of the thread's words, all in one column
    int32_t* eacc;
    uint8_t* sflag;
    RoundKeys rk;
    U4 ahead;  // kAhead: the words of the coming half-sweep

    __device__ __forceinline__ EaBitTile(const EaJob& j, int tile_, unsigned char* smem, unsigned char* tab_)
        : job(j), tile(tile_), tab(tab_)
    {
        t = threadIdx.x;
        T = blockDim.x;
        lane = t & 31;
        L = job.inst.L;
        h2 = L >> 1;
        Z = L / G;
        half = job.inst.half;
        nw = h2 * L * Z;
        WT = job.WT;
        wsh = __ffs(WT) - 1;
        nlin = nw << wsh;
        step = job.threads / LPW;  // of the tile's own thread count: the CTA may have more, for other jobs
        lin0 = t < job.threads ? t / LPW : nlin;
        W = (nlin + step - 1) / step;
        sub = t % LPW;
        w = (t / LPW) & (WT - 1);
        nrep = 4 * WT;
        tq = (uint32_t)(tile * WT + w);
        quad_live = (int)tq < (job.R + 3) / 4;  // the padding quads of the last tile hold nothing
        const EaBitsLayout lo = ea_bits_layout(L, WT, HH ? 1 : 0, job.nF);
        c0 = reinterpret_cast<uint32_t*>(smem);
        c1 = c0 + 2 * nlin;
        best = reinterpret_cast<uint32_t*>(smem + lo.best);
        bonds = reinterpret_cast<uint32_t*>(smem + lo.bonds);
        sh8 = reinterpret_cast<int8_t*>(smem + lo.h);
        htab = smem + lo.tab;
        htab_bytes = lo.tab_bytes;
        eacc = reinterpret_cast<int32_t*>(smem + lo.eacc);
        sflag = smem + lo.flags;
        rk = round_keys(job.key0, job.key1);
    }

    static constexpr int BW = G == 8 ? 2 : 1;  // 32-bit bond words per spin word

    // Bond-sign groups and position flags of every word of both classes.  G = 8: byte
    // 0 same-q, 1 other-q, 2 +y, 3 -y of the first word, byte 0 +z, 1 -z of the second,
    // flags in its top byte.  G < 8: one word, byte 0 same-q | other-q << 4, byte 1
    // +y | -y << 4, byte 2 +z | -z << 4, flags on top.  "Same q" is the +x neighbour of
    // an even-x site and the -x neighbour of an odd-x site.
    __device__ __forceinline__ void build_bonds()
    {
        for (int i = t; i < 2 * nw; i += T) {
            const int c = i >= nw ? 1 : 0, wi = i - c * nw;
            const int q = wi % h2, y = (wi / h2) % L, zb = wi / (h2 * L);
            uint32_t v[6] = {0, 0, 0, 0, 0, 0};
            for (int g = 0; g < G; ++g) {
                const uint32_t jb = (uint32_t)job.inst.jbits[c * half + wi + g * nw] >> 2;
                const int px = (c + y + zb + g * Z) & 1;
                v[0] |= ((jb >> (px ? 1 : 0)) & 1u) << g;
                v[1] |= ((jb >> (px ? 0 : 1)) & 1u) << g;
                for (int b = 2; b < 6; ++b) v[b] |= ((jb >> b) & 1u) << g;
            }
            const uint32_t f = (q == 0 ? kBitQ0 : 0u) | (q == h2 - 1 ? kBitQL : 0u) | (y == 0 ? kBitY0 : 0u) |
                               (y == L - 1 ? kBitYL : 0u) | (zb == 0 ? kBitZ0 : 0u) | (zb == Z - 1 ? kBitZL : 0u) |
                               (((y + zb) & 1) ? kBitPar : 0u);
            if constexpr (G == 8) {
                bonds[2 * i] = v[0] | (v[1] << 8) | (v[2] << 16) | (v[3] << 24);
                bonds[2 * i + 1] = v[4] | (v[5] << 8) | f;
            } else {
                bonds[i] = v[0] | (v[1] << 4) | (v[2] << 8) | (v[3] << 12) | (v[4] << 16) | (v[5] << 20) | f;
            }
        }
    }

    __device__ __forceinline__ void geometry_z(Geo& g, int lin, uint32_t f) const
    {
        const int plane = (h2 << wsh) * L;
        g.lin = lin;
        g.f = f;
        g.zp = (f & kBitZL) ? -(Z - 1) * plane : plane;
        g.zm = (f & kBitZ0) ? (Z - 1) * plane : -plane;
    }
    __device__ __forceinline__ Geo geometry(int lin, uint32_t f) const
    {
        Geo g;
        const int row = h2 << wsh;
        geometry_z(g, lin, f);
        g.qp = (f & kBitQL) ? -((h2 - 1) << wsh) : WT;
        g.qm = (f & kBitQ0) ? ((h2 - 1) << wsh) : -WT;
        g.yp = (f & kBitYL) ? -(L - 1) * row : row;
        g.ym = (f & kBitY0) ? (L - 1) * row : -row;
        g.live = true;
        return g;
    }

    __device__ __forceinline__ void init_state(uint32_t* dst0)
    {
        for (int i = t; i < 2 * nlin; i += T) {
            const int c = i >= nlin ? 1 : 0, lin = i - c * nlin;
            const int wi = lin >> wsh;
            const uint32_t q4 = (uint32_t)(tile * WT + (lin & (WT - 1)));
            uint32_t v = 0;
            if (job.resume) {  // resumed run: the given state
                v = job.final_words[(size_t)tile * 2 * nlin + i];
            } else if ((int)q4 < (job.R + 3) / 4) {
#pragma unroll 1
                for (int g = 0; g < G; ++g) {
                    const U4 r = philox10((uint32_t)(wi + g * nw), 0u, q4, (kTagInit << 24) | (uint32_t)c, job.key0,
                                          job.key1);
                    v |= ((r.x >> 31) | ((r.y >> 31) << 8) | ((r.z >> 31) << 16) | ((r.w >> 31) << 24)) << g;
                }
            }
            (c ? c1 : dst0)[lin] = v;
            best[i] = job.resume ? job.best_words[(size_t)tile * 2 * nlin + i] : v;
        }
    }

    // Threshold row of sweep s into the buffer of its parity.  Without fields: T[n],
    // n = 0..6 (F = 6 - 2 n), at strides 4, 8 and 16 bytes in three tables of 256 bytes, so a
    // count found at bits 2, 3 or 4 of a byte is an offset as it stands; bit 7 of the
    // offset is the sweep's parity.  The tables sit at a fixed address, so a lookup needs no
    // address arithmetic.  With fields: the whole row reversed, so that the address grows
    // with n.
    __device__ __forceinline__ uint32_t row_entry(int level) const
    {
        return job.table[(size_t)level * job.nF + (6 - 2 * (T - 1 - t) - job.fmin)];
    }
    __device__ __forceinline__ void put_entry(int s, uint32_t v) const
    {
        const int n = T - 1 - t;
        unsigned char* dst = tab + (s & 1) * 128;
        *reinterpret_cast<uint32_t*>(dst + 4 * n) = v;
        *reinterpret_cast<uint32_t*>(dst + 256 + 8 * n) = v;
        *reinterpret_cast<uint32_t*>(dst + 512 + 16 * n) = v;
    }
    __device__ __forceinline__ void put_row(int s, int level) const
    {
        const uint32_t* row = job.table + (size_t)level * job.nF;
        uint32_t* dst = reinterpret_cast<uint32_t*>(htab + (s & 1) * htab_bytes);
        for (int f = t; f < job.nF; f += T) dst[job.nF - 1 - f] = row[f];
    }

    // Counts of call J (bit J of every byte of the planes) as table offsets in the bytes
    // of the result: n << 2, 3 or 4, with the parity bits `par` (0x80 per byte) set.
    template <int J>
    static __device__ __forceinline__ uint32_t offsets(uint32_t p0, uint32_t p1, uint32_t p2, uint32_t par)
    {
        constexpr uint32_t m = 0x01010101u;
        if constexpr (HH) {
            return (((p0 >> J) & m) | (((p1 >> J) & m) << 1) | (((p2 >> J) & m) << 2)) << 3;
        } else if constexpr (J == 0) {
            return ((p0 & m) | ((p1 << 1) & (m << 1)) | ((p2 << 2) & (m << 2)) | (par >> 2)) << 2;
        } else if constexpr (J == 1) {
            return ((p0 & (m << 1)) | ((p1 << 1) & (m << 2)) | ((p2 << 2) & (m << 3)) | (par >> 1)) << 1;
        } else if constexpr (J <= 4) {
            return (p0 & (m << J)) | ((p1 << 1) & (m << (J + 1))) | ((p2 << 2) & (m << (J + 2))) | par;
        } else if constexpr (J <= 6) {
            return ((p0 >> 2) & (m << (J - 2))) | ((p1 >> 1) & (m << (J - 1))) | (p2 & (m << J)) | par;
        } else {
            return ((((p0 >> 2) & (m << 5)) | ((p1 >> 1) & (m << 6)) | (p2 & (m << 7))) >> 1) | par;
        }
    }
    template <int J>
    static constexpr int table_offset()
    {
        // J: 0 1 2 3 4 5 6 7 -> count at bit 2 2 2 3 4 3 4 4
        return (J <= 2) ? 0 : (J == 3 || J == 5) ? 256 : 512;
    }

    // The decisions of one Philox call: 4 replicas of the site of class rank k.
    template <int J>
    __device__ __forceinline__ void call(const U4& r, uint32_t k, int s, const int8_t* h, uint32_t p0, uint32_t p1,
                                         uint32_t p2, uint32_t par, uint32_t& res, int (&hm)[5]) const
    {
        const uint32_t X = offsets<J>(p0, p1, p2, par);
        const unsigned char* tb = tab + table_offset<J>();
        if constexpr (HH) {
            const int hv = h[k];
            tb = htab + (s & 1) * htab_bytes + 4 * (job.nF - 1 - (6 + hv - job.fmin));
            hm[4] += hv;
            uint32_t m[4] = {0, 0, 0, 0};
            or_if_ge(r.x, *reinterpret_cast<const uint32_t*>(tb + (X & 0xFFu)), 1u, m[0]);
            or_if_ge(r.y, *reinterpret_cast<const uint32_t*>(tb + __byte_perm(X, 0u, 0x4441u)), 1u, m[1]);
            or_if_ge(r.z, *reinterpret_cast<const uint32_t*>(tb + __byte_perm(X, 0u, 0x4442u)), 1u, m[2]);
            or_if_ge(r.w, *reinterpret_cast<const uint32_t*>(tb + (X >> 24)), 1u, m[3]);
#pragma unroll
            for (int b = 0; b < 4; ++b) {
                res |= m[b] << (8 * b + J);
                hm[b] += m[b] ? hv : 0;
            }
        } else {
            or_if_ge(r.x, *reinterpret_cast<const uint32_t*>(tb + (X & 0xFFu)), 1u << J, res);
            or_if_ge(r.y, *reinterpret_cast<const uint32_t*>(tb + __byte_perm(X, 0u, 0x4441u)), 0x100u << J, res);
            or_if_ge(r.z, *reinterpret_cast<const uint32_t*>(tb + __byte_perm(X, 0u, 0x4442u)), 0x10000u << J, res);
            or_if_ge(r.w, *reinterpret_cast<const uint32_t*>(tb + (X >> 24)), 0x1000000u << J, res);
        }
    }

    template <int J>
    __device__ __forceinline__ void calls(uint32_t k, const PhiloxPre& pre, int s, const int8_t* h, uint32_t p0,
                                          uint32_t p1, uint32_t p2, uint32_t par, uint32_t& res, int (&hm)[5]) const
    {
        if constexpr (J < CPT) {
            const uint32_t kj = k + (uint32_t)(J * nw);
            call<J>(philox_c0(kj, pre, rk), kj, s, h, p0, p1, p2, par, res, hm);
            calls<J + 1>(k, pre, s, h, p0, p1, p2, par, res, hm);
        }
    }

    // Count of negative terms J m < 0 of every spin of a word, in bit planes.
    template <int C>
    __device__ __forceinline__ void planes(const Geo& g, const uint32_t* o, uint32_t j0, uint32_t j1, uint32_t& p0,
                                           uint32_t& p1, uint32_t& p2) const
    {
        const uint32_t* at = o + g.lin;
        const uint32_t same = at[0], qp = at[g.qp], qm = at[g.qm], yp = at[g.yp], ym = at[g.ym];
        uint32_t zp = at[g.zp], zm = at[g.zm];
        // groups at odd x take q + 1 as their other x neighbour: x parity (C + y + zb + g Z) & 1
        const uint32_t alt = (Z & 1) ? (0xAAAAAAAAu & kLive) : 0u;
        const uint32_t odd = alt ^ ((((g.f & kBitPar) != 0u) != (C == 1)) ? kLive : 0u);
        const uint32_t other = (qp & odd) | (qm & ~odd);
        constexpr uint32_t hi = (1u << (G - 1)) * 0x01010101u;
        if (g.f & kBitZL) zp = ((zp >> 1) & (kLive ^ hi)) | ((zp << (G - 1)) & hi);
        if (g.f & kBitZ0) zm = ((zm << 1) & (kLive & ~0x01010101u)) | ((zm >> (G - 1)) & 0x01010101u);
        uint32_t y0, y1, y2, y3, y4, y5;
        if constexpr (G == 8) {
            y0 = same ^ __byte_perm(j0, 0u, 0x0000u);
            y1 = other ^ __byte_perm(j0, 0u, 0x1111u);
            y2 = yp ^ __byte_perm(j0, 0u, 0x2222u);
            y3 = ym ^ __byte_perm(j0, 0u, 0x3333u);
            y4 = zp ^ __byte_perm(j1, 0u, 0x0000u);
            y5 = zm ^ __byte_perm(j1, 0u, 0x1111u);
        } else {
            // bits past the groups of a byte are left dirty: nothing reads them
            const uint32_t b0 = __byte_perm(j0, 0u, 0x0000u), b1 = __byte_perm(j0, 0u, 0x1111u),
                           b2 = __byte_perm(j0, 0u, 0x2222u);
            y0 = same ^ b0;
            y1 = other ^ (b0 >> 4);
            y2 = yp ^ b1;
            y3 = ym ^ (b1 >> 4);
            y4 = zp ^ b2;
            y5 = zm ^ (b2 >> 4);
        }
        const uint32_t s0 = y0 ^ y1 ^ y2, k0 = (y0 & y1) | (y2 & (y0 | y1));
        const uint32_t s1 = y3 ^ y4 ^ y5, k1 = (y3 & y4) | (y5 & (y3 | y4));
        const uint32_t k2 = s0 & s1;
        p0 = s0 ^ s1;
        p1 = k0 ^ k1 ^ k2;
        p2 = (k0 & k1) | (k2 & (k0 | k1));
    }

    // Unsatisfied bonds of a word's spins m, summed over the groups of each byte (replica):
    // a spin has u = n (m = +1) or 6 - n (m = -1) of them, formed plane by plane.
    static __device__ __forceinline__ uint32_t unsatisfied(uint32_t p0, uint32_t p1, uint32_t p2, uint32_t m)
    {
        const uint32_t u0 = p0 & kLive;
        const uint32_t u1 = ((m & ~(p1 ^ p0)) | (~m & p1)) & kLive;
        const uint32_t q = p1 & p0;
        const uint32_t u2 = ((m & ~(p2 | q)) | (~m & p2)) & kLive;
        const uint32_t a = (u0 & 0x55555555u) + ((u0 >> 1) & 0x55555555u);
        const uint32_t b = (u1 & 0x55555555u) + ((u1 >> 1) & 0x55555555u);
        const uint32_t c = (u2 & 0x55555555u) + ((u2 >> 1) & 0x55555555u);
        const uint32_t a4 = (a & 0x33333333u) + ((a >> 2) & 0x33333333u);
        const uint32_t b4 = (b & 0x33333333u) + ((b >> 2) & 0x33333333u);
        const uint32_t c4 = (c & 0x33333333u) + ((c >> 2) & 0x33333333u);
        const uint32_t ab = a4 + 2u * b4;  // at most 4 + 2 * 4 per nibble
        return (ab & 0x0F0F0F0Fu) + ((ab >> 4) & 0x0F0F0F0Fu) + 4u * ((c4 + (c4 >> 4)) & 0x0F0F0F0Fu);
    }

    // One colour class of sweep s: update (DECIDE) or only the energy terms of the state
    // in place.  ulo / uhi: unsatisfied bonds of class 1, replicas 0, 2 / 1, 3 in 16-bit
    // lanes; hm: sums of h over the spins that are -1 ([b]) and over all spins ([4]).
    template <int C, bool DECIDE>
    __device__ __forceinline__ void word(const Geo& g, uint32_t j0, uint32_t j1, const uint32_t* o, uint32_t* own,
                                         const PhiloxPre& pre, int s, uint32_t& ulo, uint32_t& uhi, int (&hm)[5])
    {
        uint32_t p0 = 0, p1 = 0, p2 = 0, res = 0;
        const bool live = g.live && quad_live;
        const uint32_t wi = (uint32_t)(g.lin >> wsh);
        const uint32_t k = wi + (uint32_t)(sub * CPT * nw);
        const uint32_t par = (s & 1) ? 0x80808080u : 0u;
        const int8_t* h = HH ? sh8 + C * half : nullptr;
        if constexpr (DECIDE && kAhead) {
            // no branch: threads without a word work on word 0 and store nothing
            planes<C>(g, o, j0, j1, p0, p1, p2);
            const U4 r = ahead;
            ahead = philox_c0(k, pre, rk);
            int hx[5] = {0, 0, 0, 0, 0};
            call<0>(r, k, s, h, p0 >> sub, p1 >> sub, p2 >> sub, par, res, hx);
            res <<= sub;
            if constexpr (HH)
                if (live)
                    for (int b = 0; b < 5; ++b) hm[b] += hx[b];
        } else if (live) {
            planes<C>(g, o, j0, j1, p0, p1, p2);
            if constexpr (DECIDE) {
                if constexpr (LPW > 1) {
                    const int sft = sub * CPT;
                    calls<0>(k, pre, s, h, p0 >> sft, p1 >> sft, p2 >> sft, par, res, hm);
                    res <<= sft;
                } else {
                    calls<0>(k, pre, s, h, p0, p1, p2, par, res, hm);
                }
            }
        }
        if constexpr (DECIDE) {
#pragma unroll
            for (int d = 1; d < LPW; d <<= 1) res |= __shfl_xor_sync(0xFFFFFFFFu, res, d);
            if (live && sub == 0) own[g.lin] = res;
        } else if (live) {
            res = own[g.lin];
            if constexpr (HH) {
                if (sub == 0)
                    for (int gg = 0; gg < G; ++gg) {
                        const int hv = sh8[C * half + (int)wi + gg * nw];
                        hm[4] += hv;
                        for (int b = 0; b < 4; ++b)
                            if ((res >> (8 * b + gg)) & 1u) hm[b] += hv;
                    }
            }
        }
        if constexpr (C == 1) {
            if (live && sub == 0) {
                const uint32_t u = unsatisfied(p0, p1, p2, res);
                ulo += u & 0x00FF00FFu;
                uhi += (u >> 8) & 0x00FF00FFu;
            }
        }
    }

    template <int C, bool DECIDE>
    __device__ __forceinline__ void half_sweep(int s, const uint32_t* o, uint32_t* own, uint32_t& ulo, uint32_t& uhi,
                                               int (&hm)[5])
    {
        // kAhead: the words drawn in this half-sweep are those of the next one
        const PhiloxPre pre = kAhead ? philox_pre((uint32_t)(s + C), tq, (kTagDecision << 24) | (uint32_t)(1 - C), rk)
                                     : philox_pre((uint32_t)s, tq, (kTagDecision << 24) | (uint32_t)C, rk);
#pragma unroll 1
        for (int n = 0; n < (kAhead ? 1 : W); ++n) {
            const int lin = lin0 + n * step;
            const bool live = lin < nlin;
            const uint32_t* b = bonds + BW * (C * nw + ((live ? lin : 0) >> wsh));
            uint2 bw;
            if constexpr (BW == 2)
                bw = *reinterpret_cast<const uint2*>(b);
            else
                bw = make_uint2(*b, 0u);
            Geo g;
            if constexpr (COL) {
                g = col;
                geometry_z(g, live ? lin : 0, BW == 2 ? bw.y : bw.x);
            } else {
                g = geometry(live ? lin : 0, BW == 2 ? bw.y : bw.x);
            }
            g.live = live;
            word<C, DECIDE>(g, bw.x, bw.y, o, own, pre, s, ulo, uhi, hm);
        }
    }

    // Sum over the tile: lanes that hold the same quad, then one shared-memory add per
    // warp and replica (integers, so any order gives the same sum).
    __device__ __forceinline__ void accumulate(uint32_t ulo, uint32_t uhi, const int (&hm)[5], int32_t* acc)
    {
        if (WT == 1) {
            ulo = __reduce_add_sync(0xFFFFFFFFu, ulo);
            uhi = __reduce_add_sync(0xFFFFFFFFu, uhi);
        } else {
            for (int d = 1; d < 32; d <<= 1) {
                if (d >= LPW && d < LPW * WT) continue;  // lanes of other quads
                ulo += __shfl_xor_sync(0xFFFFFFFFu, ulo, d);
                uhi += __shfl_xor_sync(0xFFFFFFFFu, uhi, d);
            }
        }
        // E = -(3 N - 2 U) - sum h m = -3 N + 2 U - sum h + 2 sum_{m = -1} h
        int v[4] = {2 * (int)(ulo & 0xFFFFu), 2 * (int)(uhi & 0xFFFFu), 2 * (int)(ulo >> 16), 2 * (int)(uhi >> 16)};
        if constexpr (HH) {
            int x[5] = {hm[0], hm[1], hm[2], hm[3], hm[4]};
            for (int d = 1; d < 32; d <<= 1) {
                if (d >= LPW && d < LPW * WT) continue;
#pragma unroll
                for (int b = 0; b < 5; ++b) x[b] += __shfl_xor_sync(0xFFFFFFFFu, x[b], d);
            }
#pragma unroll
            for (int b = 0; b < 4; ++b) v[b] += 2 * x[b] - x[4];
        }
        if (sub == 0 && lane < LPW * WT) {
#pragma unroll
            for (int b = 0; b < 4; ++b) atomicAdd(acc + 4 * w + b, v[b]);
        }
    }

    // Merge the state (c0 words of parity buffer src0, c1) into the best for the quad's
    // improved replicas (byte b of f set: replica b).
    __device__ __forceinline__ void snapshot(const uint32_t* src0)
    {
        if (sub != 0) return;
        const uint32_t f = reinterpret_cast<const uint32_t*>(sflag)[w];
        if (f == 0u) return;
        const uint32_t mask = f * 0xFFu;
        for (int lin = lin0; lin < nlin; lin += step) {
            best[lin] = (best[lin] & ~mask) | (src0[lin] & mask);
            best[nlin + lin] = (best[nlin + lin] & ~mask) | (c1[lin] & mask);
        }
    }

    __device__ __forceinline__ void run()
    {
        build_bonds();
        if constexpr (HH)
            for (int i = t; i < 2 * half; i += T) sh8[i] = job.inst.h8[i];
        const int first = job.s0;
        init_state(c0 + ((first - 1) & 1) * nlin);
        // the last seven threads hold the threshold of n = 0..6 of the sweep after next, so the
        // load of a row from global memory is never waited for inside a sweep
        const int S = job.S, step_s = job.step;
        const bool tab_thread = !HH && t >= T - 7;
        int level = first < S ? first / step_s : 0, in_level = first < S ? first - level * step_s : 0;
        const int levels = S > 0 ? (S - 1) / step_s + 1 : 1;
        uint32_t entry = 0;
        if constexpr (HH) {
            put_row(first, level);
        } else if (tab_thread) {
            put_entry(first, row_entry(level));
        }
        auto next_level = [&]() {
            if (++in_level == step_s) {
                in_level = 0;
                if (level + 1 < levels) ++level;
            }
        };
        next_level();
        if (tab_thread) entry = row_entry(level);
        for (int i = t; i < 2 * nrep; i += T) eacc[i] = 0;
        __syncthreads();
        if constexpr (COL) {
            const int lin = lin0 < nlin ? lin0 : 0;
            col = geometry(lin, bonds[BW * (lin >> wsh) + BW - 1]);
        }
        const int N = job.inst.N;
        {
            uint32_t ulo = 0, uhi = 0;
            int hm[5] = {0, 0, 0, 0, 0};
            uint32_t* s0 = c0 + ((first - 1) & 1) * nlin;
            if constexpr (HH) half_sweep<0, false>(first, c1, s0, ulo, uhi, hm);
            half_sweep<1, false>(first, s0, c1, ulo, uhi, hm);
            accumulate(ulo, uhi, hm, eacc + ((first - 1) & 1) * nrep);
        }
        __syncthreads();
        int32_t bestE = 0, hit = -1, bsweep = -1;
        if (t < nrep) {
            int32_t* e = eacc + ((first - 1) & 1) * nrep + t;
            bestE = -3 * N + *e;
            *e = 0;
            if (job.resume) {  // the running best carried over
                bestE = job.E_best_i[tile * nrep + t];
                bsweep = job.best_sweep[tile * nrep + t];
            }
        }
        const int has_target = job.has_target, target = job.target_i;
        // Energy, running best and target of sweep s for the tile's replicas (one thread each).
        auto finish = [&](int s) {
            if (t >= nrep) return;
            int32_t* e = eacc + (s & 1) * nrep + t;
            const int32_t E = -3 * N + *e;
            *e = 0;
            const bool live = has_target != 2 || hit < 0;  // stop mode: the best is frozen at the target
            const bool imp = live && E < bestE;
            if (imp) {
                bestE = E;
                bsweep = s;
            }
            if (has_target && hit < 0 && E <= target) hit = s;
            sflag[t] = imp ? 1 : 0;
        };

        // Two barriers per sweep.  The energy of sweep s - 1 is taken while class 0 of
        // sweep s is updated into its other buffer, and the improved replicas' state of sweep
        // s - 1 is copied just before class 1 of sweep s is updated in place.
        if constexpr (kAhead)
            ahead = philox_c0((uint32_t)(((lin0 < nlin ? lin0 : 0) >> wsh) + sub * nw),
                              philox_pre((uint32_t)first, tq, kTagDecision << 24, rk), rk);
        int last = S - 1;
        bool flags_ready = false;
        const bool stop_mode = has_target == 2;
        for (int s = first; s < S; ++s) {
            uint32_t ulo = 0, uhi = 0;
            int hm[5] = {0, 0, 0, 0, 0};
            uint32_t* cur0 = c0 + (s & 1) * nlin;
            half_sweep<0, true>(s, c1, cur0, ulo, uhi, hm);
            if (s > first) finish(s - 1);
            if (s + 1 < S) {  // row s + 1; its buffer was last read in sweep s - 1
                if constexpr (HH) {
                    put_row(s + 1, level);
                    next_level();
                } else if (tab_thread) {
                    put_entry(s + 1, entry);
                    next_level();
                    entry = row_entry(level);
                }
            }
            if (stop_mode && s > first) {
                // stop mode: the tile ends once all its replicas (padding included) have reached the target
                if (__syncthreads_and(t >= nrep || hit >= 0 || tile * nrep + t >= job.R)) {
                    last = s - 1;
                    flags_ready = true;
                    break;
                }
            } else {
                __syncthreads();
            }
            if (s > first) snapshot(c0 + ((s - 1) & 1) * nlin);
            half_sweep<1, true>(s, cur0, c1, ulo, uhi, hm);
            accumulate(ulo, uhi, hm, eacc + (s & 1) * nrep);
            __syncthreads();
        }
        if (S > first) {
            if (!flags_ready) {
                finish(S - 1);
                __syncthreads();
            }
            snapshot(c0 + (last & 1) * nlin);
        } else {  // no sweep: the state before sweep `first` is the result
            last = first - 1;
        }
        __syncthreads();
        // the returned states, and their energies counted anew from them
        uint32_t* fin0 = c0 + (last & 1) * nlin;
#pragma unroll 1
        for (int k = 0; k < 2; ++k) {
            uint32_t* s0 = k ? best : fin0;
            uint32_t* s1 = k ? best + nlin : c1;
            uint32_t ulo = 0, uhi = 0;
            int hm[5] = {0, 0, 0, 0, 0};
            if constexpr (HH) half_sweep<0, false>(0, s1, s0, ulo, uhi, hm);
            half_sweep<1, false>(0, s0, s1, ulo, uhi, hm);
            accumulate(ulo, uhi, hm, eacc + k * nrep);
        }
        __syncthreads();
        for (int i = t; i < 2 * nlin; i += T) {
            const size_t d = (size_t)tile * 2 * nlin + i;
            job.final_words[d] = i < nlin ? fin0[i] : c1[i - nlin];
            job.best_words[d] = best[i];
        }
        if (t < nrep) {
            const int r = tile * nrep + t;
            job.E_best_i[r] = bestE;
            job.best_sweep[r] = bsweep;
            job.hit_sweep[r] = hit;
            if (r < job.R) {
                job.E_out[0][r] = (double)(-3 * N + eacc[t]);
                job.E_out[1][r] = (double)(-3 * N + eacc[nrep + t]);
            }
        }
        __syncthreads();
    }
};

template <int G, int CPT, bool COL, bool HH>
__device__ __forceinline__ void ea_tile_bits(const EaJob& job, int tile, unsigned char* smem, unsigned char* s_tab)
{
    EaBitTile<G, CPT, COL, HH> tl(job, tile, smem, s_tab);
    tl.run();
}

}  // namespace pb
