// ea_fast.cuh -- compile-time-shaped resident tile of the EA p-bit update for
// real (FP32) couplings (arXiv 2510.23419: Eqs. 2-3, update groups of Sec.
// 1.2.2, classical annealing of Sec. 1.3.1; the +-1 tile is ea_bits.cuh) for
// cubes whose colour-class columns make whole warps.  Summation lane (cw, zp)
// is the column (q, y, w) for z = zp mod 2 of both colours, i.e. the sites x =
// 2q + parity, fixed y, every other z, for 4 replicas: its energy terms are added
// in order of z, then over the lanes in a fixed order, so the sum does not
// depend on the threads.  A thread takes one lane (L = 24: 576) or the two
// of a column (L = 32, 16, 8: 1024 lanes on 512 threads).
//
// Same arithmetic, random words and outputs as the generic tile; what changes
// is only the instruction budget:
//  * x and y neighbours (and their periodic wrap) are per-thread bases, the
//    two z-wrapping sites are peeled out of the z loop;
//  * the Philox round keys live in registers, and the first round's products
//    of counter words 1..3 (sweep, replica quad, colour) are hoisted.
#pragma once

#include "ea_kernels.cuh"
#include "ea_launch.h"
#include "ea_philox.cuh"

namespace pb {

constexpr int kResidentWarps = kResidentThreads / 32;

template <int L, int WT>
struct EaFastTile {
    static constexpr int h2 = L / 2;
    static constexpr int CWN = h2 * L * WT;  // column-words: two summation lanes (z parities) per column
    static constexpr int TB = 2 * CWN;       // summation lanes
    static constexpr int T = ea_f32_threads(TB, 576);
    static constexpr int NV = TB / T;        // lanes per thread: t and t + T, the two z parities of one column
    static constexpr int half = h2 * L * L;
    static constexpr int N = 2 * half;
    static_assert(TB % 32 == 0 && L % 8 == 0 && TB == NV * T && (NV == 1 || CWN == T), "fast tile: whole warps of columns");
    static constexpr int SZ = L * h2 * WT;  // words between z planes of a class array
    static constexpr int CLS = half * WT;   // words of one class array
    static constexpr int NREP = 4 * WT;
    static constexpr int NW = TB / 32;

    const EaJob& job;
    int tile, t, lane, warp, w, q, y, zp0, base0, oyp, oym;
    const float4* j6;
    bool has_h;
    bool busy;  // the thread owns a column-word (the CTA may have more threads, for other jobs)
    uint32_t tq;
    uint32_t* sp;
    float* spart;
    uint8_t* sflag;
    RoundKeys rk;

    __device__ __forceinline__ EaFastTile(const EaJob& j, int tile_, unsigned char* smem) : job(j), tile(tile_)
    {
        t = threadIdx.x;
        lane = t & 31;
        warp = t >> 5;
        busy = t < T;
        const int cw = t % CWN;
        zp0 = NV == 1 ? t / CWN : 0;
        w = cw % WT;
        q = (cw / WT) % h2;
        y = cw / (WT * h2);
        sp = reinterpret_cast<uint32_t*>(smem);
        spart = reinterpret_cast<float*>(sp + N * WT);
        sflag = reinterpret_cast<uint8_t*>(spart + kResidentWarps * NREP);
        j6 = reinterpret_cast<const float4*>(job.inst.j6);
        has_h = job.inst.has_h != 0;
        rk = round_keys(job.key0, job.key1);
        tq = (uint32_t)(tile * WT + w);
        base0 = (q + h2 * y) * WT + w;
        oyp = ((y + 1 == L) ? -(L - 1) * h2 : h2) * WT;
        oym = ((y == 0) ? (L - 1) * h2 : -h2) * WT;
    }

    __device__ __forceinline__ void init_state()
    {
        if (!busy) return;
#pragma unroll 1
        for (int c = 0; c < 2; ++c)
            for (int z = NV == 1 ? zp0 : 0; z < L; z += NV == 1 ? 2 : 1) {
                const int k = q + h2 * (y + L * z), at = c * CLS + base0 + z * SZ;
                if (job.resume) {  // resumed run: the given state, in the tile layout of final_words
                    sp[at] = job.final_words[(size_t)tile * 2 * CLS + at];
                    continue;
                }
                const U4 r = philox10((uint32_t)k, 0u, tq, (kTagInit << 24) | (uint32_t)c, job.key0, job.key1);
                sp[at] = f32_word(r.x >> 31, r.y >> 31, r.z >> 31, r.w >> 31);
            }
    }

    // One colour class: update (DECIDE) or only accumulate the energy terms of
    // the current state: -m F over class 1 and -h m over class 0.
    template <int C, bool DECIDE>
    __device__ __forceinline__ void half_sweep(int s, float cexp, float (&ef)[NV][4])
    {
        if (!busy) return;
        const uint32_t* o = sp + (1 - C) * CLS;
        uint32_t* own = sp + C * CLS;
        const PhiloxPre pre = philox_pre((uint32_t)s, tq, (kTagDecision << 24) | (uint32_t)C, rk);
#pragma unroll
        for (int n = 0; n < NV; ++n) {
            const int zp = NV == 1 ? zp0 : n;
            const int px = (C + y + zp) & 1;
            const int oxp = (px ? ((q + 1 == h2) ? -(h2 - 1) : 1) : 0) * WT;
            const int oxm = (px ? 0 : ((q == 0) ? (h2 - 1) : -1)) * WT;
            const uint32_t* bxp = o + base0 + oxp;
            const uint32_t* bxm = o + base0 + oxm;
            const uint32_t* byp = o + base0 + oyp;
            const uint32_t* bym = o + base0 + oym;
            const uint32_t* bz = o + base0;
            // the wrapping sites (z = 0 for the even pass, z = L-1 for the odd pass) are
            // peeled; the others take their z neighbours at z +- 1.  Two sites per
            // iteration overlap their Philox chains and coupling loads; the terms still
            // enter the lane's energy in order of z.
            if (zp == 0) site<C, DECIDE>(0, 1, L - 1, couplings<C>(0), bxp, bxm, byp, bym, bz, own, pre, cexp, ef[n]);
#pragma unroll 2
            for (int z = 2 - zp; z < L - 1 - zp; z += 2)
                site<C, DECIDE>(z, z + 1, z - 1, couplings<C>(z), bxp, bxm, byp, bym, bz, own, pre, cexp, ef[n]);
            if (zp == 1) site<C, DECIDE>(L - 1, 0, L - 2, couplings<C>(L - 1), bxp, bxm, byp, bym, bz, own, pre, cexp, ef[n]);
        }
    }

    // six couplings and the field of the column's site at z
    struct Couplings {
        float4 a, b;
    };
    template <int C>
    __device__ __forceinline__ Couplings couplings(int z) const
    {
        const float4* j = j6 + 2 * (C * half + q + h2 * (y + L * z));
        return {__ldg(j), __ldg(j + 1)};
    }

    template <int C, bool DECIDE>
    __device__ __forceinline__ void site(int z, int zup, int zdn, const Couplings& j, const uint32_t* bxp, const uint32_t* bxm,
                                         const uint32_t* byp, const uint32_t* bym, const uint32_t* bz, uint32_t* own,
                                         const PhiloxPre& pre, float cexp, float (&ef)[4])
    {
        const int k = q + h2 * (y + L * z);
        const uint32_t n0 = bxp[z * SZ], n1 = bxm[z * SZ], n2 = byp[z * SZ], n3 = bym[z * SZ];
        const uint32_t n4 = bz[zup * SZ], n5 = bz[zdn * SZ];
        uint32_t snew;
        const float jv[6] = {j.a.x, j.a.y, j.a.z, j.a.w, j.b.x, j.b.y};
        const float hv = j.b.z;  // the site's field rides in the coupling vector
        const uint32_t nb[6] = {n0, n1, n2, n3, n4, n5};
        float F[4];
#pragma unroll
        for (int b = 0; b < 4; ++b) F[b] = ea_field_f32(jv, hv, nb, b);
        if constexpr (DECIDE) {
            const U4 r = philox_c0((uint32_t)k, pre, rk);
            snew = decide_f32_word(r.x, r.y, r.z, r.w, F[0], F[1], F[2], F[3], cexp);
            own[base0 + z * SZ] = snew;
        } else {
            snew = own[base0 + z * SZ];
        }
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            const float m = f32_sign(snew, b);  // -m F (class 1), -h m (class 0)
            if (C == 1)
                ef[b] = fmaf(-m, F[b], ef[b]);
            else if (has_h)
                ef[b] = fmaf(-m, hv, ef[b]);
        }
    }

    __device__ __forceinline__ void partials(const float (&ef)[NV][4])
    {
        if (warp >= T / 32) return;  // whole warps
#pragma unroll
        for (int n = 0; n < NV; ++n) {
            float v0 = ef[n][0], v1 = ef[n][1], v2 = ef[n][2], v3 = ef[n][3];
#pragma unroll
            for (int o2 = WT; o2 < 32; o2 <<= 1) {
                v0 += __shfl_xor_sync(0xFFFFFFFFu, v0, o2);
                v1 += __shfl_xor_sync(0xFFFFFFFFu, v1, o2);
                v2 += __shfl_xor_sync(0xFFFFFFFFu, v2, o2);
                v3 += __shfl_xor_sync(0xFFFFFFFFu, v3, o2);
            }
            if (lane < WT) {
                float* p = spart + (warp + n * (T / 32)) * NREP + 4 * lane;
                p[0] = v0;
                p[1] = v1;
                p[2] = v2;
                p[3] = v3;
            }
        }
    }

    __device__ __forceinline__ float energy_of(int r) const
    {
        float E = 0.0f;
#pragma unroll
        for (int v = 0; v < NW; ++v) E += spart[v * NREP + r];
        return E;
    }

    // the thread's words of both colours into a global state buffer, the replicas
    // that `flags` selects (byte b = 1: replica 4w + b; 0x01010101: all four)
    __device__ __forceinline__ void store_words(uint32_t* gdst, uint32_t flags) const
    {
        if (flags == 0u || !busy) return;
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            uint32_t* dst = gdst + ((size_t)tile * 2 + c) * CLS + base0;
            const uint32_t* src = sp + c * CLS + base0;
            const int z0 = NV == 1 ? zp0 * SZ : 0;
            constexpr int dz = NV == 1 ? 2 * SZ : SZ;
            snapshot_words<WT == 1, WT == 1 ? 2 : 8>(dst + z0, dz, src + z0, dz, NV == 1 ? L / 2 : L, flags);
        }
    }

    __device__ __forceinline__ void run()
    {
        init_state();
        __syncthreads();
        {
            float ef[NV][4] = {};
            half_sweep<0, false>(0, 0.0f, ef);
            half_sweep<1, false>(0, 0.0f, ef);
            partials(ef);
        }
        __syncthreads();
        int32_t hit = -1, bsweep = -1;
        float bestE = 0.0f;
        if (t < NREP) bestE = energy_of(t);
        if (job.resume) {  // the running best carried over
            if (t < NREP) {
                const int r = tile * NREP + t;
                bestE = job.E_best_f[r];
                bsweep = job.best_sweep[r];
            }
        } else {
            store_words(job.best_words, 0x01010101u);
        }

        const bool stop_mode = job.has_target == 2;
        for (int s = job.s0; s < job.S; ++s) {
            float ef[NV][4] = {};
            const float cexp = f32_cexp(job.betaf[s / job.step]);
            half_sweep<0, true>(s, cexp, ef);
            __syncthreads();
            half_sweep<1, true>(s, cexp, ef);
            partials(ef);
            __syncthreads();
            if (t < NREP) {
                const float E = energy_of(t);
                const bool live = job.has_target != 2 || hit < 0;  // stop mode: the best is frozen at the target
                const bool imp = live && E < bestE;
                if (imp) bestE = E;
                if (job.has_target && hit < 0 && E <= job.target_f) hit = s;
                if (imp) bsweep = s;
                sflag[t] = imp ? 1 : 0;
            }
            __syncthreads();
            const uint32_t f = reinterpret_cast<const uint32_t*>(sflag)[w];
            store_words(job.best_words, f);
            // stop mode: the tile ends once all its replicas (padding included) have reached the target
            if (stop_mode && __syncthreads_and(t >= NREP || hit >= 0 || tile * NREP + t >= job.R)) break;
        }

        store_words(job.final_words, 0x01010101u);
        if (t < NREP) {
            const int r = tile * NREP + t;
            job.E_best_f[r] = bestE;
            job.best_sweep[r] = bsweep;
            job.hit_sweep[r] = hit;
        }
        __syncthreads();
    }
};

template <int L, int WT>
__device__ __forceinline__ void ea_tile_fast(const EaJob& job, int tile, unsigned char* smem)
{
    EaFastTile<L, WT> tl(job, tile, smem);
    tl.run();
}

}  // namespace pb
