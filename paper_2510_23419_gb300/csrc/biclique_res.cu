// biclique_res.cu -- resident form of the biclique p-bit anneal for small
// instances (arXiv 2510.23419, Sec. 3; update groups of Sec. 1.2.2: the two
// sides of K_{n,n}).  One CTA anneals `groups` quads of 4 replicas (the four
// words of one Philox call) from the initial state to the last sweep without
// leaving the SM: couplings and spins stay in registers and shared memory, the
// two half-sweeps are separated by CTA barriers, and the energy, running best
// and best-state copies happen in the same launch.
//
//  +-1 couplings (n <= 512): one bit per spin and per coupling.  A thread owns row
//      i of both sides and keeps their coupling signs in registers (16 + 16
//      words at most); F = n - 2 popc(J ^ m) over the row, carry-save
//      compressed before the population counts; the 32 decisions of a warp are
//      one ballot, which is the spin word the other side reads.
//  real couplings (n <= 128): J once in shared memory (zero rows and columns up to a
//      multiple of 4), read without bank conflicts from both sides; a spin's four
//      replicas are one word of top bytes of +-1.0f, so the broadcast read of
//      a column is one wavefront a warp instead of the four of a float4 (which
//      bound the sweep: 20 cycles per column on 4 warps); fields by FFMA in the
//      order j = 0 .. n - 1, the FP32 rule.
//
// What bounds it: latency.  A half-sweep is one chain -- read the other side, sum
// n terms in order, draw, decide, barrier -- whatever the replica count, so a CTA
// takes as few replicas as fill the SMs (one quad up to 4 x SMs replicas), and
// everything that is not on that chain is done by a service warp beside it: the
// energy of sweep s - 1 (FP64 sums for real couplings), its running best and
// the copy of improved states while sweep s runs on the other parity of the
// state buffers, and the next level's threshold window.  Against one CTA per 32
// replicas that did all this in turn, us per sweep: real couplings n = 100, 100
// replicas 22.0 -> 2.2; n = 128, 256 replicas 31.0 -> 2.6; 1024 replicas 31.6
// -> 4.6; +-1 n = 128, 128 replicas 8.5 -> 0.83; n = 256, 512 replicas 26.0 -> 1.4.
//
// Random words, thresholds and the energy convention are those of the other
// forms, so the trajectories are the same as theirs (bit-exact for +-1).
#include <cuda_runtime.h>

#include <algorithm>
#include <mutex>
#include <type_traits>

#include "biclique_launch.h"
#include "bit_count.cuh"
#include "ea_kernels.cuh"
#include "ea_philox.cuh"

namespace pb {

namespace {

constexpr int kLdJ = kBqResMaxNf32 + 4;  // row stride of J in shared memory (real couplings): 16-byte rows whose
                                         // vector loads and columns both fall on distinct banks
// Threads of a CTA at most (the rest of the register file goes to the rows: 120 a thread).
constexpr int kResThreads = 544;

struct ResLayout {
    size_t J, st, best, eterm, eacc, tab, total;  // byte offsets of the parts, and the size
    int tab_stride;                               // entries of one window buffer
};

__host__ __device__ inline ResLayout res_layout(int jtype, int n, int groups, int tab_cap)
{
    ResLayout L{};
    size_t b = 0;
    if (jtype == PB_J_PM1_I8) {
        const int W = (n + 31) / 32;
        L.J = b;
        b += (size_t)32 * W * W * 4;  // row words of side A during set-up: [32 W][W]
        L.st = b;
        b += (size_t)2 * 2 * groups * W * 16;  // [parity][side][group][word] uint4 (4 replicas)
        L.best = b;
        b += (size_t)2 * groups * W * 16;
        L.eterm = b;
        L.eacc = b;
        b += (size_t)2 * groups * 4 * 4;  // [parity][group][4] int
        b = (b + 15) & ~(size_t)15;
        L.tab = b;
        L.tab_stride = (tab_cap + 3) / 4 * 4;
        b += (size_t)2 * L.tab_stride * 4;
    } else {
        L.J = b;
        const int n4 = (n + 3) / 4 * 4;
        b += (size_t)n4 * kLdJ * 4;
        L.st = b;
        b += (size_t)2 * 2 * groups * n4 * 4;  // [parity][side][group][spin] word (4 replicas)
        L.best = b;
        b += (size_t)2 * groups * n4 * 4;
        L.eterm = b;
        b += (size_t)2 * groups * n * 16;  // [parity][group][row of side B] float4: -m F
        L.eacc = b;
        L.tab = b;
    }
    L.total = (b + 15) & ~(size_t)15;
    return L;
}

__device__ __forceinline__ uint8_t enc_byte(bool minus) { return minus ? kE4m3Minus : kE4m3Plus; }
__device__ __forceinline__ uint16_t enc_half(bool minus) { return minus ? kBf16Minus : kBf16Plus; }

__device__ __forceinline__ void main_barrier(int threads) { asm volatile("bar.sync 1, %0;" ::"r"(threads) : "memory"); }

// Threads [0, rows * tg) own rows, rows = n rounded up to whole warps, thread group
// grp of tg the quads grp, grp + tg, ... of the CTA's `groups`; the last warp is the
// service warp.  NW: spin words per side (+-1: 1, 2, 4, 8 or 16; real couplings: unused).
template <int JT, int NW>
__global__ void __launch_bounds__(kResThreads, 1) bq_res_kernel(BqJob job, int groups, int tg, int tab_cap)
{
    extern __shared__ __align__(16) unsigned char sm[];
    // by parity of the sweep that sets and reads it: a thread late in reading it after a barrier must not see
    // the next sweep's value, or it alone would leave the loop
    __shared__ int s_stop[2];
    __shared__ int2 s_win[2];  // window of the sweep of each parity: first index, last entry
    constexpr bool PM1 = JT == PB_J_PM1_I8;
    const int n = job.inst.n, t = threadIdx.x, lane = t & 31;
    const int mainT = (int)blockDim.x - 32, rows = mainT / tg;
    const bool service = t >= mainT;
    const int grp = t / rows, i = t - grp * rows;  // main threads
    const bool live = !service && i < n;
    const int q0 = blockIdx.x * groups;  // first quad of the CTA
    const ResLayout Lo = res_layout(JT, n, groups, tab_cap);
    const int W = (n + 31) / 32;
    const RoundKeys rk = round_keys(job.key0, job.key1);
    const int S = job.S;

    // state of one side and parity: PM1 [group][word of 32 spins] uint4 (a word per replica), F32
    // [group][spin] words (a byte per replica, 0x3F / 0xBF)
    using ST = std::conditional_t<PM1, uint4, uint32_t>;
    const int n4 = (n + 3) / 4 * 4, len = PM1 ? W : n4;
    const int side_len = groups * len;
    auto state = [&](int par, int side) {
        return reinterpret_cast<ST*>(sm + Lo.st) + (size_t)(2 * par + side) * side_len;
    };
    ST* const best = reinterpret_cast<ST*>(sm + Lo.best);
    uint32_t* const stab = reinterpret_cast<uint32_t*>(sm + Lo.tab);
    float* const sJ = reinterpret_cast<float*>(sm + Lo.J);
    int32_t* const eacc = reinterpret_cast<int32_t*>(sm + Lo.eacc);
    float4* const eterm = reinterpret_cast<float4*>(sm + Lo.eterm);

    // ---- couplings
    uint32_t jA[NW], jB[NW];  // PM1: signs (1 <=> J = -1) of row i of J, of column i
    if constexpr (PM1) {
        // thread j of the first group reads column j (coalesced across the warp); a warp's ballot
        // over its 32 columns is a word of row r
        uint32_t* rowA = reinterpret_cast<uint32_t*>(sm + Lo.J);
#pragma unroll
        for (int w = 0; w < NW; ++w) jB[w] = 0;
        if (!service) {
            const int8_t* J = static_cast<const int8_t*>(job.inst.Jraw);
#pragma unroll
            for (int w = 0; w < NW; ++w) {
                uint32_t v = 0;
#pragma unroll 8
                for (int b = 0; b < 32; ++b) {
                    const int r = 32 * w + b;
                    const bool neg = r < n && live && J[(size_t)r * n + i] < 0;
                    const uint32_t m = __ballot_sync(0xFFFFFFFFu, neg);
                    if (grp == 0 && lane == 0 && r < 32 * W) rowA[r * W + (i >> 5)] = m;
                    v |= (neg ? 1u : 0u) << b;
                }
                jB[w] = v;
            }
        }
        __syncthreads();
#pragma unroll
        for (int w = 0; w < NW; ++w) jA[w] = (!service && w < W) ? rowA[i * W + w] : 0u;
        if (t < 2 * groups * 4) eacc[t] = 0;
    } else {
        for (int idx = t; idx < n4 * n4; idx += blockDim.x) {
            const int r = idx / n4, c = idx - r * n4;
            sJ[r * kLdJ + c] = r < n && c < n ? job.inst.Jf[(size_t)r * n + c] : 0.0f;
        }
        for (int idx = t; idx < 4 * side_len; idx += blockDim.x) state(0, 0)[idx] = 0x3F3F3F3Fu;  // incl. the padding
        __syncthreads();  // before the initial states go on top of it
    }
    if (t < 2) s_stop[t] = 0;

    const float hA = PM1 ? 0.0f : (live ? job.inst.hf[i] : 0.0f), hB = PM1 ? 0.0f : (live ? job.inst.hf[n + i] : 0.0f);
    const int iA = PM1 && live && job.inst.h8 ? job.inst.h8[i] : 0, iB = PM1 && live && job.inst.h8 ? job.inst.h8[n + i] : 0;

    // The quad's four spins of row i, as a word (PM1: one bit per row of the warp and replica) or floats.
    auto put = [&](int par, int side, int g, const bool (&mn)[4]) {
        if constexpr (PM1) {
            uint32_t m[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) m[k] = __ballot_sync(0xFFFFFFFFu, mn[k] && live);
            if (lane == 0) state(par, side)[g * W + (i >> 5)] = make_uint4(m[0], m[1], m[2], m[3]);
        } else if (live) {
            state(par, side)[g * len + i] = f32_word(mn[0], mn[1], mn[2], mn[3]);
        }
    };
    // Fields of row i of `side` from the other side's state of parity `par`, in the quad's four replicas.
    auto fields = [&](int side, int par, int g, int (&Fi)[4], float (&Ff)[4]) {
        if constexpr (PM1) {
            const uint4* o = state(par, 1 - side) + g * W;
            const int h = side == 0 ? iA : iB;
            if constexpr (NW <= 8) {
                uint32_t x[4][NW];
#pragma unroll
                for (int w = 0; w < NW; ++w) {
                    const uint4 v = w < W ? o[w] : make_uint4(0u, 0u, 0u, 0u);
                    const uint32_t j = side == 0 ? jA[w] : jB[w];
                    x[0][w] = v.x ^ j;
                    x[1][w] = v.y ^ j;
                    x[2][w] = v.z ^ j;
                    x[3][w] = v.w ^ j;
                }
#pragma unroll
                for (int k = 0; k < 4; ++k) Fi[k] = n - 2 * popc_words<NW>(x[k]) + h;
            } else {
                // two replicas at a time: four would take 64 registers
#pragma unroll
                for (int k = 0; k < 4; k += 2) {
                    uint32_t x[2][NW];
#pragma unroll
                    for (int w = 0; w < NW; ++w) {
                        const uint2 v = w < W ? reinterpret_cast<const uint2*>(o + w)[k >> 1] : make_uint2(0u, 0u);
                        const uint32_t j = side == 0 ? jA[w] : jB[w];
                        x[0][w] = v.x ^ j;
                        x[1][w] = v.y ^ j;
                    }
                    Fi[k] = n - 2 * popc_words<NW>(x[0]) + h;
                    Fi[k + 1] = n - 2 * popc_words<NW>(x[1]) + h;
                }
            }
        } else {
            const uint4* o = reinterpret_cast<const uint4*>(state(par, 1 - side) + g * len);
            const float* Jp = side == 0 ? sJ + (live ? i : 0) * kLdJ : sJ + (live ? i : 0);
            float a0 = 0.f, a1 = 0.f, a2 = 0.f, a3 = 0.f;
#pragma unroll 8
            for (int j = 0; j < n4; j += 4) {
                const uint4 b = o[j >> 2];
                float Jv[4];
                if (side == 0) {
                    const float4 v = *reinterpret_cast<const float4*>(Jp + j);
                    Jv[0] = v.x;
                    Jv[1] = v.y;
                    Jv[2] = v.z;
                    Jv[3] = v.w;
                } else {
#pragma unroll
                    for (int u = 0; u < 4; ++u) Jv[u] = Jp[(j + u) * kLdJ];
                }
                const uint32_t bw[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    a0 = fmaf(Jv[u], f32_sign(bw[u], 0), a0);
                    a1 = fmaf(Jv[u], f32_sign(bw[u], 1), a1);
                    a2 = fmaf(Jv[u], f32_sign(bw[u], 2), a2);
                    a3 = fmaf(Jv[u], f32_sign(bw[u], 3), a3);
                }
            }
            const float h = side == 0 ? hA : hB;
            Ff[0] = a0 + h;
            Ff[1] = a1 + h;
            Ff[2] = a2 + h;
            Ff[3] = a3 + h;
        }
    };
    // Energy terms of a side whose spins are mn: side 1 contributes -m F (F includes h), side 0 -h m.
    auto energy = [&](int side, int par, int g, const bool (&mn)[4], const int (&Fi)[4], const float (&Ff)[4]) {
        if constexpr (PM1) {
            if (side == 0 && !job.inst.has_h) return;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int x = side == 1 ? Fi[k] : iA;
                const int v = __reduce_add_sync(0xFFFFFFFFu, live ? (mn[k] ? x : -x) : 0);
                if (lane == 0) atomicAdd(eacc + (par * groups + g) * 4 + k, v);
            }
        } else if (side == 1 && live) {
            eterm[(size_t)(par * groups + g) * n + i] = make_float4(mn[0] ? Ff[0] : -Ff[0], mn[1] ? Ff[1] : -Ff[1],
                                                                     mn[2] ? Ff[2] : -Ff[2], mn[3] ? Ff[3] : -Ff[3]);
        }
    };
    // One side of sweep s (its state goes to parity s & 1).
    auto half = [&](int side, int s, int wlo, int wtop, float cexp) {
        const int par = s & 1;
#pragma unroll 1
        for (int g = grp; g < groups; g += tg) {
            const PhiloxPre pre = philox_pre((uint32_t)s, (uint32_t)(q0 + g), (kTagDecision << 24) | (uint32_t)side, rk);
            const U4 r = philox_c0((uint32_t)i, pre, rk);
            const uint32_t ws[4] = {r.x, r.y, r.z, r.w};
            int Fi[4];
            float Ff[4];
            fields(side, side == 0 ? 1 - par : par, g, Fi, Ff);  // side 0 reads side 1 of the previous sweep
            bool mn[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                if constexpr (PM1) {
                    const int f = min(max(Fi[k] - job.fmin - wlo, 0), wtop);
                    mn[k] = ws[k] >= stab[par * Lo.tab_stride + f];
                } else {
                    mn[k] = decide_f32(ws[k], Ff[k], cexp) != 0u;
                }
            }
            put(par, side, g, mn);
            energy(side, par, g, mn, Fi, Ff);
        }
    };

    // ---- initial state (tag 1): "sweep -1", parity 1, and its energy terms
    if (!service) {
#pragma unroll 1
        for (int side = 0; side < 2; ++side)
            for (int g = grp; g < groups; g += tg) {
                const U4 r = philox10((uint32_t)i, 0u, (uint32_t)(q0 + g), (kTagInit << 24) | (uint32_t)side, job.key0,
                                      job.key1);
                const bool mn[4] = {r.x >= 0x80000000u, r.y >= 0x80000000u, r.z >= 0x80000000u, r.w >= 0x80000000u};
                put(1, side, g, mn);
            }
    }
    // Threshold windows (service warp): the window of sweep s + 1 is fetched while sweep s runs, its
    // position one sweep earlier still, so neither load is waited for.
    int nlo = 0, nwidth = 0, noff = 0;  // window of the next sweep to fetch
    int flev = 0, fin = 0;              // its level and the sweep inside the level
    auto next_window = [&]() {
        nlo = job.win[3 * flev];
        nwidth = job.win[3 * flev + 1];
        noff = job.win[3 * flev + 2];
    };
    auto advance = [&](int s) {  // to the level of sweep s
        if (s >= S) return;
        if (++fin == job.step) {
            fin = 0;
            ++flev;
        }
        next_window();
    };
    constexpr int kFetch = 8;  // entries per lane in flight; a wider window's rest is copied directly
    if (PM1 && service && S > 0) {
        next_window();
        for (int f = lane; f < nwidth; f += 32) stab[f] = job.table[noff + f];
        if (lane == 0) s_win[0] = make_int2(nlo, nwidth - 1);
        advance(1);
    }
    __syncthreads();
    if (!service) {
#pragma unroll 1
        for (int side = 0; side < 2; ++side)
            for (int g = grp; g < groups; g += tg) {
                int Fi[4];
                float Ff[4];
                bool mn[4];
                fields(side, 1, g, Fi, Ff);
                if constexpr (PM1) {
                    const uint4 v = state(1, side)[g * W + (i >> 5)];
                    mn[0] = (v.x >> (i & 31)) & 1u;
                    mn[1] = (v.y >> (i & 31)) & 1u;
                    mn[2] = (v.z >> (i & 31)) & 1u;
                    mn[3] = (v.w >> (i & 31)) & 1u;
                } else {
                    const uint32_t v = state(1, side)[live ? g * len + i : 0];
#pragma unroll
                    for (int k = 0; k < 4; ++k) mn[k] = f32_minus(v, k) != 0u;
                }
                energy(side, 1, g, mn, Fi, Ff);
            }
    }
    __syncthreads();

    // Service warp: lane r < 4 groups keeps replica r's running best.  finish(s): energy of sweep
    // s (s = -1: the initial state, the first best), best, target, and the improved states' copy.
    double Ebest = 0.0;
    int bsweep = -1, hit = -1;
    auto finish = [&](int s) {
        const int par = s & 1;
        double E = 0.0;
        if constexpr (PM1) {
            if (lane < 4 * groups) {
                int32_t* e = eacc + par * groups * 4 + lane;
                E = (double)*e;
                *e = 0;
            }
        } else {
            // 8 lanes per replica of the quad sum the rows in FP64, then a fixed tree
            const float* h = job.inst.hf;
            for (int g = 0; g < groups; ++g) {
                const float* et = reinterpret_cast<const float*>(eterm + (size_t)(par * groups + g) * n);
                const uint32_t* a = state(par, 0) + (size_t)g * len;
                double e = 0.0;
                for (int r = lane >> 2; r < n; r += 8) {
                    if (job.inst.has_h) e -= (double)h[r] * (f32_minus(a[r], lane & 3) ? -1.0 : 1.0);
                    e += (double)et[4 * r + (lane & 3)];
                }
#pragma unroll
                for (int o = 4; o < 32; o <<= 1) e += __shfl_xor_sync(0xFFFFFFFFu, e, o);
                const double mine = __shfl_sync(0xFFFFFFFFu, e, lane & 3);
                if ((lane >> 2) == g) E = mine;
            }
        }
        const bool own = lane < 4 * groups;
        const bool alive = job.has_target != 2 || hit < 0;  // stop mode: the best is frozen at the target
        const bool imp = own && (s < 0 || (alive && E < Ebest));
        if (imp) {
            Ebest = E;
            bsweep = s;
        }
        if (own && s >= 0 && job.has_target && hit < 0 && E <= (PM1 ? (double)job.target_i : (double)job.target_f)) hit = s;
        const uint32_t im = __ballot_sync(0xFFFFFFFFu, imp);
        for (int g = 0; g < groups; ++g) {
            const uint32_t f = (im >> (4 * g)) & 0xFu;
            if (!f) continue;
            const uint32_t bytes = ((f & 1u) | ((f & 2u) << 7) | ((f & 4u) << 14) | ((f & 8u) << 21)) * 0xFFu;
            for (int side = 0; side < 2; ++side) {
                const ST* src = state(par, side) + (size_t)g * len;
                ST* dst = best + (size_t)side * side_len + (size_t)g * len;
                for (int x = lane; x < len; x += 32) {
                    const ST v = src[x];
                    ST d = dst[x];
                    if constexpr (PM1) {
                        if (f & 1u) d.x = v.x;
                        if (f & 2u) d.y = v.y;
                        if (f & 4u) d.z = v.z;
                        if (f & 8u) d.w = v.w;
                    } else {
                        d = (d & ~bytes) | (v & bytes);
                    }
                    dst[x] = d;
                }
            }
        }
        // stop mode: the block ends once all its replicas (padding included) have reached the target
        if (job.has_target == 2 && s >= 0 && __all_sync(0xFFFFFFFFu, !own || hit >= 0 || 4 * q0 + lane >= job.R))
            s_stop[(s + 1) & 1] = 1;
    };

    int last = S - 1;
    bool stopped = false;
    int lev = 0, in_lev = 0;
    for (int s = 0; s < S; ++s) {
        if (service) {
            uint32_t v[kFetch];
            const bool fetch = PM1 && s + 1 < S;
            uint32_t* const dst = stab + ((s + 1) & 1) * Lo.tab_stride;
            if (fetch) {
#pragma unroll
                for (int u = 0; u < kFetch; ++u) v[u] = lane + 32 * u < nwidth ? job.table[noff + lane + 32 * u] : 0u;
            }
            finish(s - 1);
            if (fetch) {
#pragma unroll
                for (int u = 0; u < kFetch; ++u)
                    if (lane + 32 * u < nwidth) dst[lane + 32 * u] = v[u];
                for (int f = lane + 32 * kFetch; f < nwidth; f += 32) dst[f] = job.table[noff + f];
                if (lane == 0) s_win[(s + 1) & 1] = make_int2(nlo, nwidth - 1);
                advance(s + 2);
            }
        } else {
            int2 w = make_int2(0, 0);
            float cexp = 0.0f;
            if constexpr (PM1)
                w = s_win[s & 1];
            else
                cexp = f32_cexp(job.betaf[lev]);
            half(0, s, w.x, w.y, cexp);
            main_barrier(mainT);
            half(1, s, w.x, w.y, cexp);
            if (++in_lev == job.step) {
                in_lev = 0;
                ++lev;
            }
        }
        __syncthreads();
        if (job.has_target == 2 && s_stop[s & 1]) {  // the state of sweep s - 1 is the result; sweep s is dropped
            last = s - 1;
            stopped = true;
            break;
        }
    }
    if (service && !stopped) finish(S - 1);
    __syncthreads();

    // ---- outputs: final state (in the buffers of the last sweep's parity, where the readout looks), best
    // state, best energies and sweeps
    const int outp = (S - 1) & 1;
    for (int idx = t; idx < 2 * groups * 4 * n; idx += blockDim.x) {
        const int x = idx % n, rest = idx / n, k = rest & 3, g = (rest >> 2) % groups, side = (rest >> 2) / groups;
        const int r = 4 * (q0 + g) + k;
        if (r >= job.Rpad) continue;
        const size_t off = (size_t)r * job.ld + x;
        if constexpr (PM1) {
            const uint32_t f = reinterpret_cast<const uint32_t*>(state(last & 1, side) + g * W + (x >> 5))[k];
            const uint32_t b = reinterpret_cast<const uint32_t*>(best + side * side_len + g * W + (x >> 5))[k];
            static_cast<uint8_t*>(job.buf[side][outp])[off] = enc_byte((f >> (x & 31)) & 1u);
            static_cast<uint8_t*>(job.best[side])[off] = enc_byte((b >> (x & 31)) & 1u);
        } else {
            static_cast<uint16_t*>(job.buf[side][outp])[off] = enc_half(f32_minus(state(last & 1, side)[g * len + x], k));
            static_cast<uint16_t*>(job.best[side])[off] = enc_half(f32_minus(best[side * side_len + g * len + x], k));
        }
    }
    if (service && lane < 4 * groups && 4 * q0 + lane < job.Rpad) {
        const int r = 4 * q0 + lane;
        if (PM1) job.E_best_i[r] = (int32_t)Ebest;
        else job.E_best_f[r] = (float)Ebest;
        job.best_sweep[r] = bsweep;
        job.hit_sweep[r] = hit;
    }
}

int res_rows(int n) { return (n + 31) / 32 * 32; }

template <int JT, int NW>
cudaError_t res_attr(size_t bytes)
{
    return cudaFuncSetAttribute(bq_res_kernel<JT, NW>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

int res_words(int n) { return n <= 32 ? 1 : n <= 64 ? 2 : n <= 128 ? 4 : n <= 256 ? 8 : 16; }

}  // namespace

size_t bq_res_smem_bytes(int jtype, int n, int groups, int tab_cap) { return res_layout(jtype, n, groups, tab_cap).total; }

// Quads per CTA: the fewest of 1, 2, 4, 8 whose CTAs fit the SMs in one wave, else 8.  Stop
// mode always takes 8: a run's final states are then those of blocks of 32 replicas.
int bq_res_groups(int R, bool stop_mode, int sms)
{
    const int quads = (R + 3) / 4;
    int g = 1;
    while (g < 8 && (stop_mode || (quads + g - 1) / g > sms)) g *= 2;
    return g;
}

// The limit belongs to the kernel and is shared by every run of the process:
// it only grows, so preparing a smaller run never breaks a larger prepared one.
cudaError_t bq_res_set_smem(int jtype, int n, size_t bytes)
{
    static std::mutex mu;
    static size_t current[64][6] = {};
    const int nw = res_words(n);
    const int k = jtype != PB_J_PM1_I8 ? 0 : nw == 1 ? 1 : nw == 2 ? 2 : nw == 4 ? 3 : nw == 8 ? 4 : 5;
    int dev = 0;
    cudaGetDevice(&dev);
    std::lock_guard<std::mutex> lock(mu);
    size_t* cur = (dev >= 0 && dev < 64) ? &current[dev][k] : nullptr;
    if (cur && bytes <= *cur) return cudaSuccess;
    const cudaError_t e = k == 0   ? res_attr<PB_J_F32, 1>(bytes)
                          : k == 1 ? res_attr<PB_J_PM1_I8, 1>(bytes)
                          : k == 2 ? res_attr<PB_J_PM1_I8, 2>(bytes)
                          : k == 3 ? res_attr<PB_J_PM1_I8, 4>(bytes)
                          : k == 4 ? res_attr<PB_J_PM1_I8, 8>(bytes)
                                   : res_attr<PB_J_PM1_I8, 16>(bytes);
    if (e == cudaSuccess && cur) *cur = bytes;
    return e;
}

cudaError_t bq_launch_res(const BqJob& job, int groups, int tab_cap, size_t smem, cudaStream_t st)
{
    const int n = job.inst.n;
    int tg = groups;
    while (res_rows(n) * tg + 32 > kResThreads) tg /= 2;
    const unsigned grid = (unsigned)(((job.R + 3) / 4 + groups - 1) / groups), threads = (unsigned)(res_rows(n) * tg + 32);
    if (job.inst.jtype != PB_J_PM1_I8)
        bq_res_kernel<PB_J_F32, 1><<<grid, threads, smem, st>>>(job, groups, tg, tab_cap);
    else if (res_words(n) == 1)
        bq_res_kernel<PB_J_PM1_I8, 1><<<grid, threads, smem, st>>>(job, groups, tg, tab_cap);
    else if (res_words(n) == 2)
        bq_res_kernel<PB_J_PM1_I8, 2><<<grid, threads, smem, st>>>(job, groups, tg, tab_cap);
    else if (res_words(n) == 4)
        bq_res_kernel<PB_J_PM1_I8, 4><<<grid, threads, smem, st>>>(job, groups, tg, tab_cap);
    else if (res_words(n) == 8)
        bq_res_kernel<PB_J_PM1_I8, 8><<<grid, threads, smem, st>>>(job, groups, tg, tab_cap);
    else
        bq_res_kernel<PB_J_PM1_I8, 16><<<grid, threads, smem, st>>>(job, groups, tg, tab_cap);
    return cudaGetLastError();
}

}  // namespace pb
