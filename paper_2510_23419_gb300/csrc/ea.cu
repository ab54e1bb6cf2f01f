// ea.cu -- sm_103a kernels of the graph-coloured p-bit update on the periodic
// 3D Edwards-Anderson cube (arXiv 2510.23419, Sec. 2; update groups Sec. 1.2.2;
// p-bit Eqs. 2-3; classical annealing Sec. 1.3.1).
//
// Two forms compute identical trajectories (same random words, same fields,
// same thresholds):
//  * resident: one persistent kernel per coupling type; a CTA takes a tile (one job, 4*WT
//    replicas), keeps that tile's whole lattice in shared memory for all
//    sweeps, and only touches global memory for best-state snapshots and the
//    final state.  The shared-neighbour reuse of Sec. 1.2.2 is total: every
//    neighbour word is read from shared memory.
//  * plain: spins in global memory, one launch per colour class and sweep,
//    plus one energy/best launch per sweep.
#include "ea_bits.cuh"
#include "ea_fast.cuh"
#include "ea_kernels.cuh"
#include "exact_split.cuh"

#include <mutex>
#include <type_traits>

#include "ea_launch.h"

namespace pb {

namespace {

// ---------------------------------------------------------------------------
// Resident form
// ---------------------------------------------------------------------------
struct TileCtx {
    int L, WT, h2, half, N, CW, V;
    int t, T, lane, warp;
    int K, part;   // K > 1: K threads share a summation lane, taking every K-th of its sites
};

// A column's place: summation lane v < V = 2 CW is (column cw, z parity zp).
struct Column {
    int w, q, y, zp;
};

__device__ __forceinline__ TileCtx tile_ctx(const EaJob& job)
{
    TileCtx g;
    g.L = job.inst.L;
    g.WT = job.WT;
    g.h2 = g.L >> 1;
    g.half = g.h2 * g.L * g.L;
    g.N = 2 * g.half;
    g.CW = g.h2 * g.L * g.WT;
    g.V = 2 * g.CW;
    g.t = threadIdx.x;
    g.T = job.threads;
    g.lane = g.t & 31;
    g.warp = g.t >> 5;
    g.K = job.split;
    g.part = g.t / g.V;
    return g;
}

__device__ __forceinline__ Column column_of(const TileCtx& g, int v)
{
    Column c;
    const int cw = v % g.CW;
    c.zp = v / g.CW;
    c.w = cw % g.WT;
    c.q = (cw / g.WT) % g.h2;
    c.y = cw / (g.WT * g.h2);
    return c;
}

// Sum 4 values per summation lane over the lanes of a warp that hold the same w, then
// store the warp's sums in part[vwarp][4w + b].
__device__ __forceinline__ void warp_partials(const TileCtx& g, int vwarp, float v0, float v1, float v2, float v3, float* part)
{
    for (int o = g.WT; o < 32; o <<= 1) {
        v0 += __shfl_xor_sync(0xFFFFFFFFu, v0, o);
        v1 += __shfl_xor_sync(0xFFFFFFFFu, v1, o);
        v2 += __shfl_xor_sync(0xFFFFFFFFu, v2, o);
        v3 += __shfl_xor_sync(0xFFFFFFFFu, v3, o);
    }
    if (g.lane < g.WT) {
        float* p = part + vwarp * 4 * g.WT + 4 * g.lane;
        p[0] = v0; p[1] = v1; p[2] = v2; p[3] = v3;
    }
}

// Generic tile of real couplings: any even L <= 32 without a compile-time tile.  The
// energy is summed over V = 2 CW summation lanes as in the compile-time tiles.  With
// fewer lanes than threads (lone small jobs), K threads share a lane: each
// updates every K-th of its sites and leaves the class-1 terms in shared memory, where
// the lane's first thread adds them in order of z -- the same sum.
__device__ void ea_tile(const EaJob& job, int tile, unsigned char* smem)
{
    const TileCtx g = tile_ctx(job);
    const int L = g.L, WT = g.WT;
    const int h2 = g.h2, half = g.half, N = g.N;
    const int nrep = 4 * WT, vwarps = (g.V + 31) / 32;

    // ---- shared memory carve-up (must match ea_resident_smem) ----
    uint32_t* sp = reinterpret_cast<uint32_t*>(smem);
    float* spart = reinterpret_cast<float*>(sp + (size_t)N * WT);
    uint8_t* sflag = reinterpret_cast<uint8_t*>(spart + kResidentWarps * nrep);
    float4* const terms = reinterpret_cast<float4*>(sflag + (nrep + 15) / 16 * 16);  // [L / 2][V], K > 1 only

    const int t = g.t;
    const RoundKeys rk = round_keys(job.key0, job.key1);

    // ---- initial state (tag 1) ----
    for (int j = t; j < N * WT; j += blockDim.x) {
        if (job.resume) {  // resumed run: the given state, in the tile layout of final_words
            sp[j] = job.final_words[(size_t)tile * N * WT + j];
            continue;
        }
        const int w2 = j % WT;
        const int ck = j / WT;
        const int c = ck >= half ? 1 : 0;
        const int k = ck - c * half;
        const U4 r = philox10((uint32_t)k, 0u, (uint32_t)(tile * WT + w2), (kTagInit << 24) | (uint32_t)c, job.key0, job.key1);
        sp[j] = f32_word(r.x >> 31, r.y >> 31, r.z >> 31, r.w >> 31);
    }

    // One colour class over the sites of one summation lane (K > 1: this thread's part of them):
    // update (DECIDE) or only the energy terms of the state, -m F (class 1) and -h m (class 0).
    const float4* const j6 = reinterpret_cast<const float4*>(job.inst.j6);
    const bool has_h = job.inst.has_h != 0;
    auto lane_sweep = [&](auto decide, int c, int s, float cexp, int v, const Column& col, float (&ef)[4]) {
        constexpr bool DECIDE = decltype(decide)::value;
        const uint32_t* o = sp + (size_t)(1 - c) * half * WT;
        uint32_t* own = sp + (size_t)c * half * WT;
        const int px = (c + col.y + col.zp) & 1;
        const EaColumn nbr = ea_column(L, h2, col.q, col.y, px);
        const int oxp = nbr.dxp * WT, oxm = nbr.dxm * WT, oyp = nbr.dyp * WT, oym = nbr.dym * WT;
        const int sz = L * h2 * WT;
        const PhiloxPre pre = philox_pre((uint32_t)s, (uint32_t)(tile * WT + col.w), (kTagDecision << 24) | (uint32_t)c, rk);
#pragma unroll 2
        for (int j = g.part; j < h2; j += g.K) {
            const int z = col.zp + 2 * j;
            const int k = col.q + h2 * (col.y + L * z);
            const int kw = k * WT + col.w;
            const int ozp = (z + 1 == L) ? -(L - 1) * sz : sz;
            const int ozm = (z == 0) ? (L - 1) * sz : -sz;
            const uint32_t nb[6] = {o[kw + oxp], o[kw + oxm], o[kw + oyp], o[kw + oym], o[kw + ozp], o[kw + ozm]};
            const size_t site = (size_t)c * half + k;
            const float4 ja = __ldg(j6 + 2 * site);
            const float4 jb = __ldg(j6 + 2 * site + 1);
            const float jv[6] = {ja.x, ja.y, ja.z, ja.w, jb.x, jb.y};
            const float hv = jb.z;  // the site's field rides in the coupling vector
            uint32_t snew;
            float F[4];
#pragma unroll
            for (int b = 0; b < 4; ++b) F[b] = ea_field_f32(jv, hv, nb, b);
            if constexpr (DECIDE) {
                const U4 r = philox_c0((uint32_t)k, pre, rk);
                snew = decide_f32_word(r.x, r.y, r.z, r.w, F[0], F[1], F[2], F[3], cexp);
                own[kw] = snew;
            } else {
                snew = own[kw];
            }
            float e[4];
#pragma unroll
            for (int b = 0; b < 4; ++b) {
                const float x = c == 1 ? F[b] : hv;  // -m F; -h m
                e[b] = f32_minus(snew, b) ? x : -x;
            }
            if (g.K > 1) {
                // class 0 terms (fields only) come first in a lane's sum: they take the first h2 rows
                if (c == 1 || has_h)
                    terms[(size_t)((c == 1 && has_h ? h2 : 0) + j) * g.V + v] = make_float4(e[0], e[1], e[2], e[3]);
            } else if (c == 1 || has_h) {
#pragma unroll
                for (int b = 0; b < 4; ++b) ef[b] += e[b];
            }
        }
    };
    constexpr int kMaxV = 2;  // summation lanes per thread
    const int lane0 = t % g.V;
    const Column col0 = column_of(g, lane0), col1 = column_of(g, (t + g.T) % g.V);
    auto half_sweep = [&](auto decide, int c, int s, float cexp, float (&ef)[kMaxV][4]) {
        if (g.K > 1) {
            if (t < g.K * g.V) lane_sweep(decide, c, s, cexp, lane0, col0, ef[0]);
            return;
        }
        if (t >= g.T) return;
        if (t < g.V) lane_sweep(decide, c, s, cexp, t, col0, ef[0]);
        if (t + g.T < g.V) lane_sweep(decide, c, s, cexp, t + g.T, col1, ef[1]);
    };
    // The lanes' sums into the warp partials (every thread calls it).
    auto partials = [&](float (&ef)[kMaxV][4]) {
        if (g.K > 1) {
            __syncthreads();  // the terms of class 1
            if (t < g.V)
                for (int j = 0; j < (has_h ? 2 : 1) * h2; ++j) {
                    const float4 e = terms[(size_t)j * g.V + t];
                    ef[0][0] += e.x;
                    ef[0][1] += e.y;
                    ef[0][2] += e.z;
                    ef[0][3] += e.w;
                }
            if (g.warp < vwarps) warp_partials(g, g.warp, ef[0][0], ef[0][1], ef[0][2], ef[0][3], spart);
            return;
        }
#pragma unroll
        for (int n = 0; n < kMaxV; ++n) {
            const int vw = g.warp + n * (g.T / 32);
            if (t < g.T && vw < vwarps) warp_partials(g, vw, ef[n][0], ef[n][1], ef[n][2], ef[n][3], spart);
        }
    };
    // Merge the lattice into a global state buffer for the replicas that the flags of a word's quad
    // select (byte b = 1: replica 4w + b; all = 0x01010101).
    auto store = [&](uint32_t* gdst, bool all) {
        // a thread's words share w: blockDim and WT are powers of two apart, rows are whole
        const uint32_t* flags = reinterpret_cast<const uint32_t*>(sflag);
        uint32_t* dst = gdst + (size_t)tile * N * WT;
        if (WT == 1) {
            const uint32_t f = all ? 0x01010101u : flags[0];
            if (f == 0u) return;
            if (t < N) snapshot_words<true, 1>(dst + t, blockDim.x, sp + t, blockDim.x, (N - t + blockDim.x - 1) / blockDim.x, f);
        } else {
            const int step = (int)blockDim.x / WT * WT;  // a multiple of WT, so that w = t % WT stays
            if (t >= step) return;
            const uint32_t f = all ? 0x01010101u : flags[t % WT];
            if (f == 0u) return;
            if (t < N * WT) snapshot_words<false, 2>(dst + t, step, sp + t, step, (N * WT - t + step - 1) / step, f);
        }
    };

    // Thread r < nrep: energy of replica r from the warp partials (fixed order; warps past the lanes hold none).
    auto energy_of = [&](int r) {
        float E = 0.0f;
#pragma unroll 8
        for (int v = 0; v < vwarps; ++v) E += spart[v * nrep + r];
        return E;
    };

    // ---- initial energy; the initial state is the first best state (unless resumed) ----
    __syncthreads();
    {
        float ef[kMaxV][4] = {};
        half_sweep(std::false_type{}, 0, 0, 0.0f, ef);
        half_sweep(std::false_type{}, 1, 0, 0.0f, ef);
        partials(ef);
    }
    __syncthreads();
    int32_t hit = -1, bsweep = -1;
    float bestE = 0.0f;
    if (t < nrep) bestE = energy_of(t);
    if (job.resume) {  // the running best carried over
        if (t < nrep) {
            const int r = tile * nrep + t;
            bestE = job.E_best_f[r];
            bsweep = job.best_sweep[r];
        }
    } else {
        store(job.best_words, true);
    }

    // ---- sweeps ----
    const bool stop_mode = job.has_target == 2;
    for (int s = job.s0; s < job.S; ++s) {
        float ef[kMaxV][4] = {};
        const float cexp = f32_cexp(job.betaf[s / job.step]);
        half_sweep(std::true_type{}, 0, s, cexp, ef);
        __syncthreads();
        half_sweep(std::true_type{}, 1, s, cexp, ef);
        partials(ef);
        __syncthreads();
        bool imp = false;
        if (t < nrep) {
            const float E = energy_of(t);
            const bool live = job.has_target != 2 || hit < 0;  // stop mode: the best is frozen at the target
            imp = live && E < bestE;
            if (imp) bestE = E;
            if (job.has_target && hit < 0 && E <= job.target_f) hit = s;
            if (imp) bsweep = s;
            sflag[t] = imp ? 1 : 0;
        }
        if (__syncthreads_or(imp)) {
            store(job.best_words, false);
            __syncthreads();  // the copies are read before the next sweep's class 0 changes under them
        }
        // stop mode: the tile ends once all its replicas (padding included) have reached the target
        if (stop_mode && __syncthreads_and(t >= nrep || hit >= 0 || tile * nrep + t >= job.R)) break;
    }

    // ---- results ----
    __syncthreads();
    store(job.final_words, true);
    if (t < nrep) {
        const int r = tile * nrep + t;
        job.E_best_f[r] = bestE;
        job.best_sweep[r] = bsweep;
        job.hit_sweep[r] = hit;
    }
    __syncthreads();
}

// One persistent kernel per coupling type in a batch (for FP32, one of two
// variants, EaKernel): a kernel holding both types' tiles gets one register
// allocation for all of them, and the FP32 tiles' pressure then costs the +-1
// tiles spill traffic.  The tile code comes with the work
// item (a branch on the job's own fields also led the compiler to spill).
// Every CTA lets a programmatically dependent launch (the other type's kernel
// of the same batch) start at once, so that kernel's CTAs take the SMs this
// one leaves as its list runs out.
template <int K>
__global__ void __launch_bounds__(ea_kernel_threads(K), 1)
    ea_resident_kernel(const EaJob* __restrict__ jobs, const EaWork* __restrict__ work, int n_work, int* counter)
{
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ int s_item;
    for (;;) {
        if (threadIdx.x == 0) s_item = atomicAdd(counter, 1);
        __syncthreads();
        const int item = s_item;
        __syncthreads();
        if (item >= n_work) break;
        const EaWork wk = work[item];
        const EaJob& job = jobs[wk.job];
        if constexpr (K == kEaKernelPm1 || K == kEaKernelPm1Split) {
            __shared__ __align__(256) unsigned char s_tab[768];  // threshold rows (EaBitTile::put_entry)
#define PB_BITS(G, CPT, COL, HH)                                  \
    case ea_bits_path(G, CPT, COL, HH):                           \
        ea_tile_bits<G, CPT, COL, HH>(job, wk.tile, smem, s_tab); \
        break
            if constexpr (K == kEaKernelPm1) {
                switch (wk.path) {
                    PB_BITS(8, 8, true, false);
                    PB_BITS(8, 8, false, false);
                    PB_BITS(4, 4, true, false);
                    PB_BITS(4, 4, false, false);
                    PB_BITS(2, 2, true, false);
                    PB_BITS(2, 2, false, false);
                    PB_BITS(8, 8, false, true);
                    PB_BITS(4, 4, false, true);
                    PB_BITS(2, 2, false, true);
                }
            } else {
                switch (wk.path) {
                    PB_BITS(8, 4, true, false);
                    PB_BITS(8, 2, true, false);
                    PB_BITS(8, 1, true, false);
                    PB_BITS(4, 2, true, false);
                    PB_BITS(4, 1, true, false);
                    PB_BITS(2, 1, true, false);
                    PB_BITS(8, 1, true, true);
                    PB_BITS(4, 1, true, true);
                    PB_BITS(2, 1, true, true);
                }
            }
#undef PB_BITS
        } else {
            // L = 24 tiles in the first kernel run the generic tile
            if (K == kEaKernelF32 && wk.path == kEaPathFast32)
                ea_tile_fast<32, 1>(job, wk.tile, smem);
            else if (K == kEaKernelF32L24 && wk.path == kEaPathFast24)
                ea_tile_fast<24, 1>(job, wk.tile, smem);
            else if (wk.path == kEaPathFast16)
                ea_tile_fast<16, 4>(job, wk.tile, smem);
            else if (wk.path == kEaPathFast8)
                ea_tile_fast<8, 16>(job, wk.tile, smem);
            else
                ea_tile(job, wk.tile, smem);
        }
    }
}

// ---------------------------------------------------------------------------
// Random-word ceiling of the EA update: the decision words of an L = 32 tile
// (same counters, round keys and first-round hoisting as the fast tile: one
// Philox4x32-10 call per site and 4 replicas, i.e. one word per update) and
// nothing else -- no field, no threshold, no state.  Each thread takes the
// sites of one column of both colours, two sites per iteration as the +-1
// tile does; the words are folded into one xor per thread so none is dead.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(kResidentThreads, 1)
    ea_philox_ceiling_kernel(uint32_t key0, uint32_t key1, int sweeps, uint32_t* __restrict__ sink)
{
    constexpr int L = 32, h2 = L / 2;
    const RoundKeys rk = round_keys(key0, key1);
    const int t = threadIdx.x;
    const int cw = t % (kResidentThreads / 2), zp = t / (kResidentThreads / 2);
    const int q = cw % h2, y = cw / h2;
    const uint32_t tq = blockIdx.x;
    uint32_t acc = 0;
    for (int s = 0; s < sweeps; ++s) {
#pragma unroll 1
        for (int c = 0; c < 2; ++c) {
            const PhiloxPre pre = philox_pre((uint32_t)s, tq, (kTagDecision << 24) | (uint32_t)c, rk);
#pragma unroll 2
            for (int z = zp; z < L; z += 2) {
                const U4 r = philox_c0((uint32_t)(q + h2 * (y + L * z)), pre, rk);
                acc ^= r.x ^ r.y ^ r.z ^ r.w;
            }
        }
    }
    sink[(size_t)blockIdx.x * kResidentThreads + t] = acc;
}

// ---------------------------------------------------------------------------
// Plain form (global memory state, one tile with WT = Rw)
// ---------------------------------------------------------------------------
struct SiteGeom {
    int x, y, z, q, row;
};

__device__ __forceinline__ SiteGeom site_of_rank(int L, int c, int k)
{
    SiteGeom s;
    const int h2 = L >> 1;
    s.row = k / h2;
    s.q = k - s.row * h2;
    s.y = s.row % L;
    s.z = s.row / L;
    s.x = 2 * s.q + ((c + s.y + s.z) & 1);
    return s;
}

// Class ranks of the 6 neighbours (+x, -x, +y, -y, +z, -z) of a site.
__device__ __forceinline__ void neighbour_ranks(int L, const SiteGeom& s, int (&kn)[6])
{
    const int h2 = L >> 1;
    const int xp = (s.x + 1 == L) ? 0 : s.x + 1, xm = (s.x == 0) ? L - 1 : s.x - 1;
    const int yp = (s.y + 1 == L) ? 0 : s.y + 1, ym = (s.y == 0) ? L - 1 : s.y - 1;
    const int zp = (s.z + 1 == L) ? 0 : s.z + 1, zm = (s.z == 0) ? L - 1 : s.z - 1;
    kn[0] = (xp >> 1) + h2 * (s.y + L * s.z);
    kn[1] = (xm >> 1) + h2 * (s.y + L * s.z);
    kn[2] = s.q + h2 * (yp + L * s.z);
    kn[3] = s.q + h2 * (ym + L * s.z);
    kn[4] = s.q + h2 * (s.y + L * zp);
    kn[5] = s.q + h2 * (s.y + L * zm);
}

// Plain form in stop mode: every replica has reached the target, the launches
// of the remaining sweeps return at once.
__device__ __forceinline__ bool ea_plain_stopped(const EaJob& job)
{
    return job.has_target == 2 && *reinterpret_cast<const volatile int32_t*>(job.n_hit) >= job.R;
}

template <int JT, bool HH>
__global__ void __launch_bounds__(256) ea_plain_half_kernel(EaJob job, int c, int s)
{
    if (ea_plain_stopped(job)) return;
    __shared__ uint32_t stab[256];
    const int L = job.inst.L;
    const int half = job.inst.half;
    const int WT = job.WT;
    if (JT == PB_J_PM1_I8) {
        const uint32_t* row = job.table + (size_t)(s / job.step) * job.nF;
        if (!HH) {
            if (threadIdx.x < 64) stab[threadIdx.x] = row[6 - 2 * __popc(threadIdx.x) - job.fmin];
        } else {
            for (int f = threadIdx.x; f < job.nF; f += blockDim.x) stab[f] = row[f];
        }
        __syncthreads();
    }
    const long long j = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= (long long)half * WT) return;
    const int k = (int)(j / WT);
    const int w = (int)(j - (long long)k * WT);
    const SiteGeom sg = site_of_rank(L, c, k);
    int kn[6];
    neighbour_ranks(L, sg, kn);
    const uint32_t* o = job.final_words + (size_t)(1 - c) * half * WT;
    uint32_t nb[6];
#pragma unroll
    for (int b = 0; b < 6; ++b) nb[b] = o[(size_t)kn[b] * WT + w];
    const U4 r = philox10((uint32_t)k, (uint32_t)s, (uint32_t)w, (kTagDecision << 24) | (uint32_t)c, job.key0, job.key1);
    uint32_t snew;
    if (JT == PB_J_PM1_I8) {
        const uint32_t X = ea_pattern(nb[0], nb[1], nb[2], nb[3], nb[4], nb[5], job.inst.jbits[c * half + k]);
        if (!HH) {
            const unsigned char* tb = reinterpret_cast<const unsigned char*>(stab);
            snew = decide_bit(r.x, *reinterpret_cast<const uint32_t*>(tb + (X & 0xFFu))) |
                   (decide_bit(r.y, *reinterpret_cast<const uint32_t*>(tb + ((X >> 8) & 0xFFu))) << 8) |
                   (decide_bit(r.z, *reinterpret_cast<const uint32_t*>(tb + ((X >> 16) & 0xFFu))) << 16) |
                   (decide_bit(r.w, *reinterpret_cast<const uint32_t*>(tb + (X >> 24))) << 24);
        } else {
            const int base = 6 + job.inst.h8[c * half + k] - job.fmin;
            snew = decide_bit(r.x, stab[base - 2 * __popc(X & 0xFCu)]) |
                   (decide_bit(r.y, stab[base - 2 * __popc((X >> 8) & 0xFCu)]) << 8) |
                   (decide_bit(r.z, stab[base - 2 * __popc((X >> 16) & 0xFCu)]) << 16) |
                   (decide_bit(r.w, stab[base - 2 * __popc((X >> 24) & 0xFCu)]) << 24);
        }
    } else {
        const size_t site = (size_t)c * half + k;
        const float4 ja = __ldg(reinterpret_cast<const float4*>(job.inst.j6) + 2 * site);
        const float4 jb = __ldg(reinterpret_cast<const float4*>(job.inst.j6) + 2 * site + 1);
        const float jv[6] = {ja.x, ja.y, ja.z, ja.w, jb.x, jb.y};
        const float hv = __ldg(job.inst.hf + site);
        const float cexp = f32_cexp(job.betaf[s / job.step]);
        snew = decide_f32_word(r.x, r.y, r.z, r.w, ea_field_f32(jv, hv, nb, 0), ea_field_f32(jv, hv, nb, 1),
                               ea_field_f32(jv, hv, nb, 2), ea_field_f32(jv, hv, nb, 3), cexp);
    }
    job.final_words[(size_t)c * half * WT + j] = snew;
}

__global__ void __launch_bounds__(256) ea_plain_init_kernel(EaJob job)
{
    const int half = job.inst.half;
    const int WT = job.WT;
    const long long j = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= 2LL * half * WT) return;
    const int w = (int)(j % WT);
    const long long ck = j / WT;
    const int c = ck >= half ? 1 : 0;
    const int k = (int)(ck - (long long)c * half);
    const U4 r = philox10((uint32_t)k, 0u, (uint32_t)w, (kTagInit << 24) | (uint32_t)c, job.key0, job.key1);
    job.final_words[j] = (job.inst.jtype == PB_J_PM1_I8)
                             ? ((r.x >> 31) | ((r.y >> 31) << 8) | ((r.z >> 31) << 16) | ((r.w >> 31) << 24))
                             : f32_word(r.x >> 31, r.y >> 31, r.z >> 31, r.w >> 31);
}

// One block per word column w (4 replicas): energy of the current state, best
// update, best snapshot.  init: the current state is the initial state.
template <int JT, bool HH>
__global__ void __launch_bounds__(256) ea_plain_energy_kernel(EaJob job, int s, int init)
{
    if (!init && ea_plain_stopped(job)) return;
    __shared__ int32_t red_i[8][256 / 32];
    __shared__ float red_f[4][256 / 32];
    __shared__ uint32_t s_mask;
    const int L = job.inst.L;
    const int half = job.inst.half;
    const int N = job.inst.N;
    const int WT = job.WT;
    const int w = blockIdx.x;
    const int t = threadIdx.x;
    uint32_t lo = 0, hi = 0;
    int32_t hm[4] = {0, 0, 0, 0};
    float ef[4] = {0.f, 0.f, 0.f, 0.f};
    for (int c = 0; c < 2; ++c) {
        const uint32_t* own = job.final_words + (size_t)c * half * WT;
        const uint32_t* o = job.final_words + (size_t)(1 - c) * half * WT;
        for (int k = t; k < half; k += blockDim.x) {
            const uint32_t sv = own[(size_t)k * WT + w];
            if (JT == PB_J_PM1_I8) {
                if (c == 1) {
                    const SiteGeom sg = site_of_rank(L, c, k);
                    int kn[6];
                    neighbour_ranks(L, sg, kn);
                    uint32_t nb[6];
#pragma unroll
                    for (int b = 0; b < 6; ++b) nb[b] = o[(size_t)kn[b] * WT + w];
                    const uint32_t X = ea_pattern(nb[0], nb[1], nb[2], nb[3], nb[4], nb[5], job.inst.jbits[c * half + k]);
                    const uint32_t u = ea_popc6_bytes(X ^ (sv * 0xFCu));
                    lo += u & 0x00FF00FFu;
                    hi += (u >> 8) & 0x00FF00FFu;
                }
                if (HH) {
                    const int hv = job.inst.h8[c * half + k];
#pragma unroll
                    for (int b = 0; b < 4; ++b) hm[b] += ((sv >> (8 * b)) & 1u) ? -hv : hv;
                }
            } else {
                const size_t site = (size_t)c * half + k;
                const float hv = job.inst.hf[site];
                if (c == 1) {
                    const SiteGeom sg = site_of_rank(L, c, k);
                    int kn[6];
                    neighbour_ranks(L, sg, kn);
                    uint32_t nb[6];
#pragma unroll
                    for (int b = 0; b < 6; ++b) nb[b] = o[(size_t)kn[b] * WT + w];
                    const float4 ja = reinterpret_cast<const float4*>(job.inst.j6)[2 * site];
                    const float4 jb = reinterpret_cast<const float4*>(job.inst.j6)[2 * site + 1];
                    const float jv[6] = {ja.x, ja.y, ja.z, ja.w, jb.x, jb.y};
#pragma unroll
                    for (int b = 0; b < 4; ++b) {
                        const float F = ea_field_f32(jv, hv, nb, b);
                        ef[b] += f32_minus(sv, b) ? F : -F;
                    }
                } else if (job.inst.has_h) {
#pragma unroll
                    for (int b = 0; b < 4; ++b) ef[b] += f32_minus(sv, b) ? hv : -hv;
                }
            }
        }
    }
    // deterministic block reduction
    const int lane = t & 31, warp = t >> 5;
    int32_t v[8] = {(int32_t)(lo & 0xFFFFu), (int32_t)(hi & 0xFFFFu), (int32_t)(lo >> 16), (int32_t)(hi >> 16),
                    hm[0], hm[1], hm[2], hm[3]};
#pragma unroll
    for (int a = 0; a < 8; ++a)
        for (int o = 16; o > 0; o >>= 1) v[a] += __shfl_xor_sync(0xFFFFFFFFu, v[a], o);
#pragma unroll
    for (int a = 0; a < 4; ++a)
        for (int o = 16; o > 0; o >>= 1) ef[a] += __shfl_xor_sync(0xFFFFFFFFu, ef[a], o);
    if (lane == 0) {
        for (int a = 0; a < 8; ++a) red_i[a][warp] = v[a];
        for (int a = 0; a < 4; ++a) red_f[a][warp] = ef[a];
    }
    __syncthreads();
    if (t < 4) {
        const int r = 4 * w + t;
        bool imp;
        if (JT == PB_J_PM1_I8) {
            int32_t U = 0, H = 0;
            for (int q = 0; q < 8; ++q) {
                U += red_i[t][q];
                H += red_i[4 + t][q];
            }
            const int32_t E = -(3 * N - 2 * U) - H;
            imp = init || ((job.has_target != 2 || job.hit_sweep[r] < 0) && E < job.E_best_i[r]);
            if (imp) job.E_best_i[r] = E;
            if (!init && job.has_target && job.hit_sweep[r] < 0 && E <= job.target_i) {
                job.hit_sweep[r] = s;
                if (job.has_target == 2 && r < job.R) atomicAdd(job.n_hit, 1);
            }
        } else {
            float E = 0.0f;
            for (int q = 0; q < 8; ++q) E += red_f[t][q];
            imp = init || ((job.has_target != 2 || job.hit_sweep[r] < 0) && E < job.E_best_f[r]);
            if (imp) job.E_best_f[r] = E;
            if (!init && job.has_target && job.hit_sweep[r] < 0 && E <= job.target_f) {
                job.hit_sweep[r] = s;
                if (job.has_target == 2 && r < job.R) atomicAdd(job.n_hit, 1);
            }
        }
        if (init) job.hit_sweep[r] = -1;
        if (imp) job.best_sweep[r] = init ? -1 : s;
        const uint32_t m = imp ? (0xFFu << (8 * t)) : 0u;
        if (t == 0) s_mask = 0u;
        __syncwarp(0xFu);
        atomicOr(&s_mask, m);
    }
    __syncthreads();
    const uint32_t mask = s_mask;
    if (mask == 0u) return;
    for (int j = t; j < N; j += blockDim.x) {
        const size_t idx = (size_t)j * WT + w;
        const uint32_t v2 = job.final_words[idx];
        if (mask == 0xFFFFFFFFu)
            job.best_words[idx] = v2;
        else
            job.best_words[idx] = (job.best_words[idx] & ~mask) | (v2 & mask);
    }
}

// ---------------------------------------------------------------------------
// Readout and exact energies
// ---------------------------------------------------------------------------
// State buffer -> [R][N] int8 +-1.  A thread writes 2 V consecutive sites of one
// replica, i.e. V words of both classes give a bit each: reads are whole words and writes
// whole rows.  (A byte per thread, with a 64-bit division each, took 0.4 ms per state
// set at L = 32 and 1024 replicas.)  The widest V that L and the output's address allow
// (ea_readout_sites); an odd address takes V = 0: one word of both classes, byte stores.
template <int V0>
__global__ void __launch_bounds__(256) ea_readout_kernel(EaJob job, const uint32_t* __restrict__ words,
                                                         int8_t* __restrict__ out, int blocks_per_replica)
{
    constexpr int V = V0 ? V0 : 1;
    const int L = job.inst.L, h2 = L >> 1, hv = h2 / V, WT = job.WT;
    const int r = blockIdx.x / blocks_per_replica;
    const int j = (blockIdx.x - r * blocks_per_replica) * 256 + threadIdx.x;
    if (j >= hv * L * L) return;
    const int row = j / hv, q0 = (j - row * hv) * V;
    const int z = row / L, y = row - z * L;
    const int Z = job.groups ? L / job.groups : L, nw = h2 * L * Z;  // words per class and quad
    const int g = z / Z, wi = q0 + h2 * (y + L * (z - g * Z));
    const int quad = r >> 2, tile = quad / WT, w = quad - tile * WT;
    // the spin's bit in its word: bit g of the replica's byte, or bit 7 (sign) of an FP32 run's byte
    const int sh = 8 * (r & 3) + (job.inst.jtype == PB_J_F32 ? 7 : g);
    const int even = (y + z) & 1;  // the class whose sites of this row have an even x
    const uint32_t* p0 = words + (((size_t)tile * 2 + even) * nw + wi) * WT + w;
    const uint32_t* p1 = words + (((size_t)tile * 2 + 1 - even) * nw + wi) * WT + w;
    uint16_t v[V];
#pragma unroll
    for (int k = 0; k < V; ++k) {
        const uint32_t a = (p0[(size_t)k * WT] >> sh) & 1u, b = (p1[(size_t)k * WT] >> sh) & 1u;
        v[k] = (uint16_t)(0x0101u + a * 0x00FEu + b * 0xFE00u);  // 0x01 = +1, 0xFF = -1
    }
    int8_t* dst = out + (size_t)r * job.inst.N + (size_t)row * L + 2 * q0;
    if constexpr (V0 == 4) {
        *reinterpret_cast<uint2*>(dst) = make_uint2(v[0] | ((uint32_t)v[1] << 16), v[2] | ((uint32_t)v[3] << 16));
    } else if constexpr (V0 == 2) {
        *reinterpret_cast<uint32_t*>(dst) = v[0] | ((uint32_t)v[1] << 16);
    } else if constexpr (V0 == 1) {
        *reinterpret_cast<uint16_t*>(dst) = v[0];
    } else {
        dst[0] = (int8_t)v[0];
        dst[1] = (int8_t)(v[0] >> 8);
    }
}

// E = -sum_{d,i} J[d][i] m_i m_{i+d} - sum_i h_i m_i, one block per replica;
// int64 for PM1.  F32: a term's coupling is split into three FP32 parts whose sums over 64 terms are exact
// (exact_split.cuh) and go to FP64, the third to a sum of its own, so that small terms meet the rest
// once; a term without a split (rare) goes there whole, in FP64.  A warp takes
// whole rows of the cube (several when they are short), so the site's coordinates cost one division per row
// and every load is a row's: with six divisions and three FP64 terms per site this took 0.66 ms per state set
// at L = 32 and 1024 replicas, now 0.42 ms.
template <int JT>
__global__ void __launch_bounds__(256) ea_energy_kernel(EaJob job, const int8_t* __restrict__ m, double* __restrict__ E)
{
    __shared__ long long red_i[8];
    __shared__ double red_f[8], red_d[8];
    const int L = job.inst.L, N = job.inst.N;
    const int r = blockIdx.x;
    const int8_t* mr = m + (size_t)r * N;
    long long ai = 0;
    double af = 0.0, ad = 0.0;  // large parts; small parts and whole terms
    float p1 = 0.f, p2 = 0.f, p3 = 0.f;
    const float unit = job.inst.junit;
    auto flush = [&]() {
        af += (double)p1;
        af += (double)p2;
        ad += (double)p3;
        p1 = p2 = p3 = 0.f;
    };
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
    const int per = L < 32 ? 32 / L : 1;            // rows per warp
    const int sub = L < 32 ? lane / L : 0, x0 = L < 32 ? lane - sub * L : lane;
    int held = 0;
    for (int row0 = warp * per; row0 < L * L; row0 += warps * per) {
        const int row = row0 + sub;
        if (sub >= per || row >= L * L) continue;
        const int z = row / L, y = row - z * L;
        const int base = row * L;
        const int up_y = (y + 1 == L ? row - (L - 1) : row + 1) * L, up_z = (z + 1 == L ? row - (L - 1) * L : row + L) * L;
        for (int x = x0; x < L; x += 32) {
            const int i = base + x;
            const int mi = mr[i];
            const int mn[3] = {mr[base + (x + 1 == L ? 0 : x + 1)], mr[up_y + x], mr[up_z + x]};
            if (JT == PB_J_PM1_I8) {
                const int8_t* J = static_cast<const int8_t*>(job.inst.J3);
                int t = 0;
#pragma unroll
                for (int d = 0; d < 3; ++d) t -= (int)J[(size_t)d * N + i] * mi * mn[d];
                if (job.inst.hraw) t -= static_cast<const int8_t*>(job.inst.hraw)[i] * mi;
                ai += t;
            } else {
                // the site's terms -v m, loaded together; one branch for those without a split
                const float* J = static_cast<const float*>(job.inst.J3);
                float x[4], q[4][3];
#pragma unroll
                for (int d = 0; d < 3; ++d) x[d] = __ldg(J + (size_t)d * N + i);
                x[3] = job.inst.hraw ? static_cast<const float*>(job.inst.hraw)[i] : 0.0f;
                uint32_t whole = 0;
#pragma unroll
                for (int d = 0; d < 4; ++d) {
                    if ((d < 3 ? mi * mn[d < 3 ? d : 0] : mi) > 0) x[d] = -x[d];
                    const bool split = split_exact(x[d], unit, q[d][0], q[d][1], q[d][2]);
                    whole |= split ? 0u : 1u << d;
                    p1 = __fadd_rn(p1, split ? q[d][0] : 0.0f);
                    p2 = __fadd_rn(p2, split ? q[d][1] : 0.0f);
                    p3 = __fadd_rn(p3, split ? q[d][2] : 0.0f);
                }
                if (whole) {
#pragma unroll
                    for (int d = 0; d < 4; ++d)
                        if (whole >> d & 1u) ad += (double)x[d];  // a field that is not finite is here too
                }
                if (++held == 16) {  // at most 64 terms per part
                    flush();
                    held = 0;
                }
            }
        }
    }
    if (JT == PB_J_F32) flush();
    for (int o = 16; o > 0; o >>= 1) {
        ai += __shfl_xor_sync(0xFFFFFFFFu, ai, o);
        af += __shfl_xor_sync(0xFFFFFFFFu, af, o);
        ad += __shfl_xor_sync(0xFFFFFFFFu, ad, o);
    }
    if (lane == 0) {
        red_i[warp] = ai;
        red_f[warp] = af;
        red_d[warp] = ad;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        long long si = 0;
        double sf = 0.0, sd = 0.0;
        for (int q = 0; q < warps; ++q) {
            si += red_i[q];
            sf += red_f[q];
            sd += red_d[q];
        }
        E[r] = (JT == PB_J_PM1_I8) ? (double)si : sf + sd;
    }
}

// Fields of given states with the anneal kernels' arithmetic.
__global__ void __launch_bounds__(256) ea_fields_kernel(EaDevice inst, const int8_t* __restrict__ m, int R,
                                                        float* __restrict__ out)
{
    const int L = inst.L, N = inst.N, half = inst.half;
    const long long j = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= (long long)R * N) return;
    const int r = (int)(j / N);
    const int i = (int)(j - (long long)r * N);
    const int x = i % L, y = (i / L) % L, z = i / (L * L);
    const int c = (x + y + z) & 1;
    const int k = i >> 1;
    const int8_t* mr = m + (size_t)r * N;
    const SiteGeom sg = site_of_rank(L, c, k);
    int kn[6];
    neighbour_ranks(L, sg, kn);
    // class rank -> site index of the other colour: i' = 2k' + parity
    uint32_t nb[6];
#pragma unroll
    for (int b = 0; b < 6; ++b) {
        const int kk = kn[b];
        const int row = kk / (L >> 1), qq = kk - row * (L >> 1);
        const int yy = row % L, zz = row / L;
        const int xx = 2 * qq + ((1 - c + yy + zz) & 1);
        const bool minus = mr[xx + L * (yy + L * zz)] < 0;
        nb[b] = (inst.jtype == PB_J_PM1_I8) ? (minus ? 1u : 0u) : (minus ? 0xBFu : 0x3Fu);
    }
    if (inst.jtype == PB_J_PM1_I8) {
        const uint32_t X = ea_pattern(nb[0], nb[1], nb[2], nb[3], nb[4], nb[5], inst.jbits[c * half + k]);
        const int h = inst.h8 ? inst.h8[c * half + k] : 0;
        out[j] = (float)(6 - 2 * __popc(X & 0xFCu) + h);
    } else {
        const size_t site = (size_t)c * half + k;
        const float4 ja = reinterpret_cast<const float4*>(inst.j6)[2 * site];
        const float4 jb = reinterpret_cast<const float4*>(inst.j6)[2 * site + 1];
        const float jv[6] = {ja.x, ja.y, ja.z, ja.w, jb.x, jb.y};
        out[j] = ea_field_f32(jv, inst.hf[site], nb, 0);
    }
}

}  // namespace

// ---------------------------------------------------------------------------
// Host launchers
// ---------------------------------------------------------------------------
int ea_resident_pick_wt(int L, int jtype, int has_h, int nF, int cap_words)
{
    const int h2 = L / 2;
    int best = 0;
    for (int wt = 1; wt <= kResidentMaxWT; wt *= 2) {
        if ((long long)h2 * L * wt > kResidentThreads / 2) break;
        if (ea_resident_smem(L, wt, jtype, has_h, nF) > kResidentSmemLimit) break;
        best = wt;
        if (wt >= cap_words) break;
    }
    return best;
}

// The limit is a property of the kernel, shared by every run of the process
// on a device: it only grows, so preparing a run never lowers the limit that
// another prepared run will launch with.
template <int K>
static cudaError_t ea_resident_attr(size_t smem)
{
    return cudaFuncSetAttribute(ea_resident_kernel<K>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
}

cudaError_t ea_resident_set_smem(int kernel, size_t smem)
{
    static std::mutex mu;
    static size_t current[kEaKernels][64] = {};
    if (kernel < 0 || kernel >= kEaKernels) return cudaErrorInvalidValue;
    int dev = 0;
    cudaGetDevice(&dev);
    std::lock_guard<std::mutex> lock(mu);
    size_t* cur = (dev >= 0 && dev < 64) ? &current[kernel][dev] : nullptr;
    if (cur && smem <= *cur) return cudaSuccess;
    const cudaError_t e = kernel == kEaKernelPm1        ? ea_resident_attr<kEaKernelPm1>(smem)
                          : kernel == kEaKernelPm1Split ? ea_resident_attr<kEaKernelPm1Split>(smem)
                          : kernel == kEaKernelF32      ? ea_resident_attr<kEaKernelF32>(smem)
                                                        : ea_resident_attr<kEaKernelF32L24>(smem);
    if (e == cudaSuccess && cur) *cur = smem;
    return e;
}

cudaError_t ea_launch_resident(int kernel, const EaJob* d_jobs, const EaWork* d_work, int n_work, int* d_counter,
                               size_t smem, int grid, int threads, bool after_previous, cudaStream_t st)
{
    if (kernel < 0 || kernel >= kEaKernels) return cudaErrorInvalidValue;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    if (after_previous) {
        attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[0].val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
    }
    if (kernel == kEaKernelPm1)
        return cudaLaunchKernelEx(&cfg, ea_resident_kernel<kEaKernelPm1>, d_jobs, d_work, n_work, d_counter);
    if (kernel == kEaKernelPm1Split)
        return cudaLaunchKernelEx(&cfg, ea_resident_kernel<kEaKernelPm1Split>, d_jobs, d_work, n_work, d_counter);
    if (kernel == kEaKernelF32)
        return cudaLaunchKernelEx(&cfg, ea_resident_kernel<kEaKernelF32>, d_jobs, d_work, n_work, d_counter);
    return cudaLaunchKernelEx(&cfg, ea_resident_kernel<kEaKernelF32L24>, d_jobs, d_work, n_work, d_counter);
}

cudaError_t ea_launch_philox_ceiling(uint64_t seed, int sweeps, int blocks, uint32_t* sink, cudaStream_t st)
{
    ea_philox_ceiling_kernel<<<blocks, kResidentThreads, 0, st>>>((uint32_t)seed, (uint32_t)(seed >> 32), sweeps, sink);
    return cudaGetLastError();
}

static unsigned blocks_for(long long n, int bs) { return (unsigned)((n + bs - 1) / bs); }

cudaError_t ea_launch_plain_init(const EaJob& job, cudaStream_t st)
{
    const long long n = 2LL * job.inst.half * job.WT;
    ea_plain_init_kernel<<<blocks_for(n, 256), 256, 0, st>>>(job);
    return cudaGetLastError();
}

cudaError_t ea_launch_plain_sweep(const EaJob& job, int s, cudaStream_t st)
{
    const long long n = (long long)job.inst.half * job.WT;
    const unsigned nb = blocks_for(n, 256);
    for (int c = 0; c < 2; ++c) {
        if (job.inst.jtype == PB_J_PM1_I8) {
            if (job.inst.has_h)
                ea_plain_half_kernel<PB_J_PM1_I8, true><<<nb, 256, 0, st>>>(job, c, s);
            else
                ea_plain_half_kernel<PB_J_PM1_I8, false><<<nb, 256, 0, st>>>(job, c, s);
        } else {
            ea_plain_half_kernel<PB_J_F32, false><<<nb, 256, 0, st>>>(job, c, s);
        }
    }
    return cudaGetLastError();
}

cudaError_t ea_launch_plain_energy(const EaJob& job, int s, bool init, cudaStream_t st)
{
    if (job.inst.jtype == PB_J_PM1_I8) {
        if (job.inst.has_h)
            ea_plain_energy_kernel<PB_J_PM1_I8, true><<<job.WT, 256, 0, st>>>(job, s, init ? 1 : 0);
        else
            ea_plain_energy_kernel<PB_J_PM1_I8, false><<<job.WT, 256, 0, st>>>(job, s, init ? 1 : 0);
    } else {
        ea_plain_energy_kernel<PB_J_F32, false><<<job.WT, 256, 0, st>>>(job, s, init ? 1 : 0);
    }
    return cudaGetLastError();
}

cudaError_t ea_launch_readout(const EaJob& job, const uint32_t* words, int8_t* out_pm, double* out_E, cudaStream_t st)
{
    const int h2 = job.inst.L / 2, V = ea_readout_sites(job.inst.L, reinterpret_cast<uintptr_t>(out_pm));
    const int bpr = (h2 / (V ? V : 1) * job.inst.L * job.inst.L + 255) / 256;
    const unsigned grid = (unsigned)bpr * (unsigned)job.R;
    if (V == 4)
        ea_readout_kernel<4><<<grid, 256, 0, st>>>(job, words, out_pm, bpr);
    else if (V == 2)
        ea_readout_kernel<2><<<grid, 256, 0, st>>>(job, words, out_pm, bpr);
    else if (V == 1)
        ea_readout_kernel<1><<<grid, 256, 0, st>>>(job, words, out_pm, bpr);
    else
        ea_readout_kernel<0><<<grid, 256, 0, st>>>(job, words, out_pm, bpr);
    if (job.groups) return cudaGetLastError();
    if (job.inst.jtype == PB_J_PM1_I8)
        ea_energy_kernel<PB_J_PM1_I8><<<job.R, 256, 0, st>>>(job, out_pm, out_E);
    else
        ea_energy_kernel<PB_J_F32><<<job.R, 256, 0, st>>>(job, out_pm, out_E);
    return cudaGetLastError();
}

cudaError_t ea_launch_fields(const EaDevice& inst, const int8_t* d_states, int R, float* d_out, cudaStream_t st)
{
    const long long n = (long long)R * inst.N;
    ea_fields_kernel<<<blocks_for(n, 256), 256, 0, st>>>(inst, d_states, R, d_out);
    return cudaGetLastError();
}

}  // namespace pb
