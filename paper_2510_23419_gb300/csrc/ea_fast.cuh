// ea_fast.cuh -- compile-time-shaped resident tile of the EA p-bit update for
// real (FP32) couplings (arXiv 2510.23419: Eqs. 2-3, update groups of Sec.
// 1.2.2, classical annealing of Sec. 1.3.1; the +-1 tile is ea_bits.cuh) for
// cubes whose colour-class columns exactly fill
// half the CTA: thread (cw, zp) owns the column (q, y, w) for z = zp mod 2 of
// both colours, i.e. the sites x = 2q + parity, fixed y, every other z, for 4
// replicas.
//
// Shapes whose columns fill fewer than half the CTA (L = 24: 288 column-words,
// 576 of the 1024 threads) leave the remaining warps without sites: they take
// part in the barriers and add zero energy partials.
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
    static constexpr int T = kResidentThreads;
    static constexpr int h2 = L / 2;
    static constexpr int CWN = h2 * L * WT;  // column-words: two threads (z parities) per column
    static constexpr int TB = 2 * CWN;       // threads with sites; the others only join the barriers
    static constexpr bool kAllBusy = TB == kResidentThreads;
    static constexpr int half = h2 * L * L;
    static constexpr int N = 2 * half;
    static_assert(TB <= T && TB % 32 == 0 && L % 8 == 0, "fast tile: whole warps of column-word pairs");
    static constexpr int SZ = L * h2 * WT;  // words between z planes of a class array
    static constexpr int CLS = half * WT;   // words of one class array
    static constexpr int NREP = 4 * WT;
    static constexpr int NW = kResidentWarps;

    const EaJob& job;
    int tile, t, lane, warp, w, q, y, zp, base0, oyp, oym;
    bool busy;  // the thread owns a column-word (always, when the columns fill the CTA)
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
        busy = kAllBusy || t < TB;
        const int cw = t % CWN;
        zp = t / CWN;
        w = cw % WT;
        q = (cw / WT) % h2;
        y = cw / (WT * h2);
        sp = reinterpret_cast<uint32_t*>(smem);
        spart = reinterpret_cast<float*>(sp + N * WT);
        sflag = reinterpret_cast<uint8_t*>(spart + NW * NREP);
        rk = round_keys(job.key0, job.key1);
        tq = (uint32_t)(tile * WT + w);
        base0 = (q + h2 * y) * WT + w;
        oyp = ((y + 1 == L) ? -(L - 1) * h2 : h2) * WT;
        oym = ((y == 0) ? (L - 1) * h2 : -h2) * WT;
    }

    __device__ __forceinline__ void init_state()
    {
        if constexpr (!kAllBusy)
            if (!busy) return;
        if (job.resume) {  // resumed run: the given state, in the tile layout of final_words
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                const uint32_t* src = job.final_words + ((size_t)tile * 2 + c) * CLS + base0;
                for (int z = zp; z < L; z += 2) sp[c * CLS + base0 + z * SZ] = src[z * SZ];
            }
            return;
        }
#pragma unroll
        for (int c = 0; c < 2; ++c)
#pragma unroll 4
            for (int z = zp; z < L; z += 2) {
                const int k = q + h2 * (y + L * z);
                const U4 r = philox10((uint32_t)k, 0u, tq, (kTagInit << 24) | (uint32_t)c, job.key0, job.key1);
                sp[c * CLS + base0 + z * SZ] = f32_word(r.x >> 31, r.y >> 31, r.z >> 31, r.w >> 31);
            }
    }

    // One colour class: update (DECIDE) or only accumulate the energy terms of
    // the current state: -m F over class 1 and -h m over class 0.
    template <int C, bool DECIDE>
    __device__ __forceinline__ void half_sweep(int s, float (&ef)[4])
    {
        if constexpr (!kAllBusy)
            if (!busy) return;
        const uint32_t* o = sp + (1 - C) * CLS;
        uint32_t* own = sp + C * CLS;
        const int zp = this->zp;
        const PhiloxPre pre = philox_pre((uint32_t)s, tq, (kTagDecision << 24) | (uint32_t)C, rk);
        const float cexp = f32_cexp(job.betaf[s / job.step]);
        {
            const int px = (C + y + zp) & 1;
            const int oxp = (px ? ((q + 1 == h2) ? -(h2 - 1) : 1) : 0) * WT;
            const int oxm = (px ? 0 : ((q == 0) ? (h2 - 1) : -1)) * WT;
            const uint32_t* bxp = o + base0 + oxp;
            const uint32_t* bxm = o + base0 + oxm;
            const uint32_t* byp = o + base0 + oyp;
            const uint32_t* bym = o + base0 + oym;
            const uint32_t* bz = o + base0;
            // the wrapping sites (z = 0 for the even pass, z = L-1 for the odd pass) are
            // peeled; the others take their z neighbours at z +- 1.  One site per
            // iteration: two would hold two sites' couplings and spill.
            if (zp == 0) site<C, DECIDE>(0, 1, L - 1, bxp, bxm, byp, bym, bz, own, pre, cexp, ef);
#pragma unroll 1
            for (int z = 2 - zp; z < L - 1 - zp; z += 2)
                site<C, DECIDE>(z, z + 1, z - 1, bxp, bxm, byp, bym, bz, own, pre, cexp, ef);
            if (zp == 1) site<C, DECIDE>(L - 1, 0, L - 2, bxp, bxm, byp, bym, bz, own, pre, cexp, ef);
        }
    }

    template <int C, bool DECIDE>
    __device__ __forceinline__ void site(int z, int zup, int zdn, const uint32_t* bxp, const uint32_t* bxm,
                                         const uint32_t* byp, const uint32_t* bym, const uint32_t* bz, uint32_t* own,
                                         const PhiloxPre& pre, float cexp, float (&ef)[4])
    {
        const int k = q + h2 * (y + L * z);
        const uint32_t n0 = bxp[z * SZ], n1 = bxm[z * SZ], n2 = byp[z * SZ], n3 = bym[z * SZ];
        const uint32_t n4 = bz[zup * SZ], n5 = bz[zdn * SZ];
        uint32_t snew;
        const size_t site_i = (size_t)C * half + k;
        const float4 ja = __ldg(reinterpret_cast<const float4*>(job.inst.j6) + 2 * site_i);
        const float4 jb = __ldg(reinterpret_cast<const float4*>(job.inst.j6) + 2 * site_i + 1);
        const float jv[6] = {ja.x, ja.y, ja.z, ja.w, jb.x, jb.y};
        const float hv = jb.z;  // the site's field rides in the coupling vector
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
            else if (job.inst.has_h)
                ef[b] = fmaf(-m, hv, ef[b]);
        }
    }

    __device__ __forceinline__ void partials(const float (&ef)[4])
    {
        float v0 = ef[0], v1 = ef[1], v2 = ef[2], v3 = ef[3];
#pragma unroll
        for (int o2 = WT; o2 < 32; o2 <<= 1) {
            v0 += __shfl_xor_sync(0xFFFFFFFFu, v0, o2);
            v1 += __shfl_xor_sync(0xFFFFFFFFu, v1, o2);
            v2 += __shfl_xor_sync(0xFFFFFFFFu, v2, o2);
            v3 += __shfl_xor_sync(0xFFFFFFFFu, v3, o2);
        }
        if (lane < WT) {
            float* p = spart + warp * NREP + 4 * lane;
            p[0] = v0;
            p[1] = v1;
            p[2] = v2;
            p[3] = v3;
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
        if (flags == 0u || (!kAllBusy && !busy)) return;
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            uint32_t* dst = gdst + ((size_t)tile * 2 + c) * CLS + base0;
            const uint32_t* src = sp + c * CLS + base0;
#pragma unroll 4
            for (int z = zp; z < L; z += 2) snapshot_word<WT == 1>(dst + z * SZ, src[z * SZ], flags);
        }
    }

    __device__ __forceinline__ void run()
    {
        init_state();
        __syncthreads();
        {
            float ef[4] = {0.f, 0.f, 0.f, 0.f};
            half_sweep<0, false>(0, ef);
            half_sweep<1, false>(0, ef);
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
            float ef[4] = {0.f, 0.f, 0.f, 0.f};
            half_sweep<0, true>(s, ef);
            __syncthreads();
            half_sweep<1, true>(s, ef);
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
