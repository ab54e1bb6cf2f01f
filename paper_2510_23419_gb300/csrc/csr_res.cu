// csr_res.cu -- resident form of the p-bit anneal on general sparse +-1 instances
// (arXiv 2510.23419: Eq. 1 on an arbitrary edge set, update groups of Sec.
// 1.2.2 from a proper colouring) without fields, degree <= 15 and at most
// kCsrResSpins spins: one CTA anneals one or two quads of 4 replicas from the
// initial state to the last sweep with every spin in shared memory, one bit per
// spin and replica, so a colour class costs a CTA barrier instead of a launch.
//
// A spin is a byte (bit 4 q + k: replica k of quad q, 1 <=> m = -1); a thread takes a
// word of 4 spins of one class (classes start on word boundaries).  Per neighbour
// slot it gathers 4 bytes, xors the coupling signs and adds the word into bit
// planes, so the count n of negative terms J m < 0 of 32 updates (F = deg - 2 n) is
// a few operations per slot; what is left per update is a Philox word, a
// threshold lookup and a compare.  The per-class launches that this replaces kept a
// byte per spin and replica in global memory and took 68 instructions per update
// and 5 launches per sweep on the L = 25 cube (4 colours): us per sweep, before -> after: 1024
// replicas 70.3 -> 28.4, 64 replicas 34.7 -> 19.7; L = 11, 256 replicas 28.9 -> 5.7.  What bounds it now: the
// part-filled rounds of a class (its words over 512 threads) and L2 latency of the rows; more
// threads did not help (768: 29.0, 1024: 29.4 us against 27.8 at 512 then).
//
// Energy: a row lists its neighbours in lower classes first.  When a spin is
// updated those hold their values of this sweep, so its unsatisfied bonds to them are
// final: their sum over all spins is U, and E = 2 U - (number of edges).
// They are counted in bit planes too and leave the registers once per sweep, or earlier where a thread's
// words of the next class could overflow the planes (kCsrResWords).
#include <algorithm>

#include "csr_launch.h"
#include "ea_kernels.cuh"
#include "ea_philox.cuh"

namespace pb {

namespace {

constexpr int kThreads = kCsrResThreads;
constexpr int kAcc = kCsrResPlanes;  // planes of a thread's energy count
static_assert((kCsrResSpins / 4 + kThreads - 1) / kThreads <= kCsrResWords, "energy planes hold a class");

// Add the bits of two words to the planes p (a bit-sliced counter of P bits).
template <int P>
__device__ __forceinline__ void add2(uint32_t (&p)[P], uint32_t a, uint32_t b)
{
    uint32_t c = (p[0] & a) | (b & (p[0] | a));
    p[0] ^= a ^ b;
#pragma unroll
    for (int k = 1; k < P; ++k) {
        const uint32_t t = p[k] & c;
        p[k] ^= c;
        c = t;
    }
}

// REGULAR: every spin has degree maxdeg.  P: planes of a neighbour count (3: degree <= 7, 4: <= 15).
template <int P, int Q, bool REGULAR>
__global__ void __launch_bounds__(kThreads, 1) csr_res_kernel(CsrJob job)
{
    extern __shared__ __align__(16) unsigned char sm[];
    const CsrResDevice& g = job.g.res;
    unsigned char* const spins = sm;  // byte Npad stays zero: the neighbour of unused slots
    uint32_t* const best = reinterpret_cast<uint32_t*>(sm + g.npad + 16);
    __shared__ uint32_t s_tab[2][32];  // threshold rows reversed (offset 4 (maxdeg - deg) + 8 n), by sweep parity
    __shared__ int32_t s_cls[256][4];  // class: as CsrResDevice::cls
    __shared__ int32_t s_U[2][4 * Q];
    __shared__ uint8_t s_imp[4 * Q];
    const int t = threadIdx.x, lane = t & 31;
    const int words = g.npad / 4, nc = job.g.n_colours, S = job.S, q0 = blockIdx.x * Q;
    const RoundKeys rk = round_keys(job.key0, job.key1);
    constexpr uint32_t kReps = Q == 2 ? 0xFFFFFFFFu : 0x0F0F0F0Fu;

    for (int i = t; i < 4 * nc; i += kThreads) s_cls[i >> 2][i & 3] = g.cls[i];
    for (int i = t; i < 2 * 4 * Q; i += kThreads) s_U[i / (4 * Q)][i % (4 * Q)] = 0;
    // the threshold row of a level: the window's entries, saturated outside it
    auto row_entry = [&](int lev, int e) {  // entry e of the reversed row
        const int f = job.nF - 1 - e;
        const int lo = job.win[3 * lev], w = job.win[3 * lev + 1], off = job.win[3 * lev + 2];
        return job.table[off + min(max(f - lo, 0), w - 1)];
    };
    __syncthreads();

    // initial state (tag 1)
    for (int c = 0; c < nc; ++c)
        for (int w = t; w < s_cls[c][1]; w += kThreads) {
            uint32_t v = 0;
            for (int j = 0; j < 4; ++j)
                for (int q = 0; q < Q; ++q) {
                    if (4 * w + j >= s_cls[c][2]) break;
                    const U4 r = philox10((uint32_t)(4 * w + j), 0u, (uint32_t)(q0 + q), (kTagInit << 24) | (uint32_t)c,
                                          job.key0, job.key1);
                    v |= ((r.x >> 31) | ((r.y >> 31) << 1) | ((r.z >> 31) << 2) | ((r.w >> 31) << 3)) << (8 * j + 4 * q);
                }
            reinterpret_cast<uint32_t*>(spins)[s_cls[c][0] + w] = v;
            best[s_cls[c][0] + w] = v;
        }
    if (t < 4) reinterpret_cast<uint32_t*>(spins + g.npad)[t] = 0;
    if (t < job.nF) s_tab[0][t] = row_entry(0, t);
    __syncthreads();

    uint32_t acc[kAcc];  // the sweep's unsatisfied bonds, per bit position (spin of the word, replica)
    // Word ww: planes n of its spins' negative terms over `all` slots, and low those over the first `lo`
    // (lower classes; both counts even).  The row entries of kAhead slots are loaded at once: they come
    // from L2, one dependent latency per word instead of one per two slots.
    constexpr int kAhead = 6;
    auto gather = [&](int ww, int lo, int all, uint32_t (&low)[P], uint32_t (&n)[P]) {
#pragma unroll
        for (int k = 0; k < P; ++k) low[k] = n[k] = 0;
        for (int u = 0; u < all; u += kAhead) {
            uint2 nb[kAhead];
            uint32_t sg[kAhead];
#pragma unroll
            for (int k = 0; k < kAhead; ++k)
                if (u + k < all) {
                    nb[k] = __ldg(g.nbr + (size_t)(u + k) * words + ww);
                    sg[k] = __ldg(g.sign + (size_t)(u + k) * words + ww);
                }
#pragma unroll
            for (int k = 0; k < kAhead; k += 2)
                if (u + k < all) {
                    uint32_t x[2];
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        const uint2 v = nb[k + e];
                        const uint32_t b0 = spins[v.x & 0xFFFFu], b1 = spins[v.x >> 16];
                        const uint32_t b2 = spins[v.y & 0xFFFFu], b3 = spins[v.y >> 16];
                        x[e] = __byte_perm(__byte_perm(b0, b1, 0x0040u), __byte_perm(b2, b3, 0x0040u), 0x5410u) ^
                               (sg[k + e] & kReps);
                    }
                    add2<P>(n, x[0], x[1]);
                    if (u + k + 2 == lo) {
#pragma unroll
                        for (int b = 0; b < P; ++b) low[b] = n[b];
                    }
                }
        }
    };
    // Unsatisfied bonds to the lower classes, given the count planes n of their negative terms: n for
    // m = +1, deg_low - n for m = -1 (mod 2^P: (n ^ m) + deg_low m + m), added to acc.
    auto count = [&](const uint32_t (&n)[P], uint32_t m, int ww) {
        const uint4 d4 = __ldg(g.lowdeg + ww);
        const uint32_t d[4] = {d4.x, d4.y, d4.z, d4.w};
        uint32_t u[P], c = m;
#pragma unroll
        for (int k = 0; k < P; ++k) {
            const uint32_t a = n[k] ^ m, b = d[k] & m;
            u[k] = a ^ b ^ c;
            c = (a & b) | (c & (a | b));
        }
        c = 0;
#pragma unroll
        for (int k = 0; k < kAcc; ++k) {
            if (k < P) {
                const uint32_t a = acc[k], b = u[k];
                acc[k] = a ^ b ^ c;
                c = (a & b) | (c & (a | b));
            } else {
                const uint32_t a = acc[k];
                acc[k] = a ^ c;
                c &= a;
            }
        }
    };
    auto clear = [&]() {
#pragma unroll
        for (int k = 0; k < kAcc; ++k) acc[k] = 0;
    };
    // The threads' counts per replica into s_U.
    auto flush = [&](int32_t* U) {
#pragma unroll
        for (int b = 0; b < 4 * Q; ++b) {
            int v = 0;
#pragma unroll
            for (int k = 0; k < kAcc; ++k) v += __popc(acc[k] & (0x01010101u << b)) << k;
            v = __reduce_add_sync(0xFFFFFFFFu, v);
            if (lane == 0 && v) atomicAdd(U + b, v);
        }
    };
    clear();
    for (int c = 0; c < nc; ++c) {
        const int slots = s_cls[c][3], lo = slots & 0xFF;
        for (int w = t; w < s_cls[c][1]; w += kThreads) {
            const int ww = s_cls[c][0] + w;
            uint32_t low[P], n[P];
            gather(ww, lo, lo, low, n);
            count(low, reinterpret_cast<uint32_t*>(spins)[ww], ww);
        }
        if (slots & kCsrResFlush) {
            flush(s_U[1]);
            clear();
        }
    }
    __syncthreads();

    // thread r < 4 Q keeps replica r's running best
    double Ebest = 0.0;
    int bsweep = -1, hit = -1;
    auto energy = [&](int par) {
        const double E = 2.0 * (double)s_U[par][t] - (double)g.edges;
        s_U[par][t] = 0;
        return E;
    };
    if (t < 4 * Q) Ebest = energy(1);
    auto finish = [&](int s) {
        if (t >= 4 * Q) return;
        const double E = energy(s & 1);
        const bool imp = E < Ebest;
        if (imp) {
            Ebest = E;
            bsweep = s;
        }
        if (job.has_target && hit < 0 && E <= job.target) hit = s;
        s_imp[t] = imp ? 1 : 0;
    };
    auto improved = [&]() {  // byte mask of the improved replicas, in every byte of a word
        uint32_t f = 0;
#pragma unroll
        for (int b = 0; b < 4 * Q; ++b) f |= (uint32_t)s_imp[b] << b;
        return f * 0x01010101u;
    };

    int lev = 0, in_lev = 0;
    uint32_t mask = 0;  // replicas whose energy improved in the previous sweep: their old spins go to the best state
    for (int s = 0; s < S; ++s) {
        // level of sweep s + 1, its row fetched beside the first class
        int nlev = lev, nin = in_lev + 1;
        if (nin == job.step) {
            nin = 0;
            ++nlev;
        }
        uint32_t next = 0;
        const bool fetch = t >= kThreads - 32 && kThreads - 1 - t < job.nF && s + 1 < S;
        if (fetch) next = row_entry(nlev, kThreads - 1 - t);
        if (s > 0) mask = improved();
        const unsigned char* row = reinterpret_cast<const unsigned char*>(s_tab[s & 1]);
        for (int c = 0; c < nc; ++c) {
            const int w0 = s_cls[c][0], nw = s_cls[c][1], nsp = s_cls[c][2], slots = s_cls[c][3];
            const int lo = slots & 0xFF, all = slots >> 16;
            PhiloxPre pre[Q];
#pragma unroll
            for (int q = 0; q < Q; ++q)
                pre[q] = philox_pre((uint32_t)s, (uint32_t)(q0 + q), (kTagDecision << 24) | (uint32_t)c, rk);
#pragma unroll 1
            for (int w = t; w < nw; w += kThreads) {
                const int ww = w0 + w;
                uint32_t p[P], n[P];
                gather(ww, lo, all, p, n);
                const uint32_t dg = REGULAR ? 0u : __ldg(g.degoff + ww);  // 4 (maxdeg - deg) of the word's spins
                // counts as nibbles: nibble 2 j + q of x[k] = n of (spin j, quad q, replica k)
                uint32_t x[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    x[k] = (n[0] >> k) & 0x11111111u;
#pragma unroll
                    for (int b = 1; b < P; ++b) x[k] |= (b >= k ? n[b] << (b - k) : n[b] >> (k - b)) & (0x11111111u << b);
                }
                uint32_t res = 0;
#pragma unroll
                for (int j = 0; j < 4; ++j)
#pragma unroll
                    for (int q = 0; q < Q; ++q) {
                        const U4 r = philox_c0((uint32_t)(4 * w + j), pre[q], rk);
                        const uint32_t ws[4] = {r.x, r.y, r.z, r.w};
                        const unsigned char* tb = row + (REGULAR ? 0u : (dg >> (8 * j)) & 0xFFu);
#pragma unroll
                        for (int k = 0; k < 4; ++k) {
                            constexpr uint32_t m = P == 3 ? 0x38u : 0x78u;
                            const int sh = 4 * (2 * j + q) - 3;
                            const uint32_t o = (sh < 0 ? x[k] << 3 : x[k] >> sh) & m;
                            const uint32_t T = *reinterpret_cast<const uint32_t*>(tb + o);
                            or_if_ge(ws[k], T, 1u << (8 * j + 4 * q + k), res);
                        }
                    }
                if (4 * w + 4 > nsp) res &= (1u << (8 * (nsp - 4 * w))) - 1u;  // the class's last word
                uint32_t* own = reinterpret_cast<uint32_t*>(spins) + ww;
                if (mask) {
                    const uint32_t old = *own;
                    best[ww] = (best[ww] & ~mask) | (old & mask);
                }
                *own = res;
                if (lo) count(p, res, ww);
            }
            if (c == 0 && fetch) s_tab[(s + 1) & 1][kThreads - 1 - t] = next;
            if (slots & kCsrResFlush) {
                flush(s_U[s & 1]);
                clear();
            }
            __syncthreads();
        }
        finish(s);
        __syncthreads();
        lev = nlev;
        in_lev = nin;
    }
    // the last sweep's improvements, then the states into the run's word layout (byte b: replica b of the quad)
    mask = S > 0 ? improved() : 0;
    for (int w = t; w < words; w += kThreads)
        best[w] = (best[w] & ~mask) | (reinterpret_cast<uint32_t*>(spins)[w] & mask);
    __syncthreads();
    for (int i = t; i < job.g.N; i += kThreads) {
        const int at = g.pos[i];
        const uint32_t f = spins[at], b = reinterpret_cast<unsigned char*>(best)[at];
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            if (q0 + q >= job.Rw) break;
            const uint32_t fq = (f >> (4 * q)) & 0xFu, bq = (b >> (4 * q)) & 0xFu;
            job.spins[(size_t)i * job.Rw + q0 + q] = (fq * 0x00204081u) & 0x01010101u;
            job.best[(size_t)i * job.Rw + q0 + q] = (bq * 0x00204081u) & 0x01010101u;
        }
    }
    if (t < 4 * Q && 4 * q0 + t < 4 * job.Rw) {
        const int r = 4 * q0 + t;
        job.E_best[r] = Ebest;
        job.best_sweep[r] = bsweep;
        job.hit_sweep[r] = hit;
    }
}

template <int P, int Q, bool REGULAR>
cudaError_t launch(const CsrJob& job, size_t smem, cudaStream_t st)
{
    cudaError_t e = cudaFuncSetAttribute(csr_res_kernel<P, Q, REGULAR>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)csr_res_smem(kCsrResSpins));
    if (e != cudaSuccess) return e;
    csr_res_kernel<P, Q, REGULAR><<<(unsigned)((job.Rw + Q - 1) / Q), kThreads, smem, st>>>(job);
    return cudaGetLastError();
}

}  // namespace

size_t csr_res_smem(int npad) { return (size_t)2 * npad + 16; }

cudaError_t csr_launch_res(const CsrJob& job, int sms, cudaStream_t st)
{
    const size_t smem = csr_res_smem(job.g.res.npad);
    // two quads share a word's gathers; one while its CTAs fit the SMs in one wave
    const bool two = csr_res_quads(job.Rw, sms) == 2, reg = job.g.res.regular != 0;
    if (job.g.maxdeg <= 7)
        return two ? (reg ? launch<3, 2, true>(job, smem, st) : launch<3, 2, false>(job, smem, st))
                   : (reg ? launch<3, 1, true>(job, smem, st) : launch<3, 1, false>(job, smem, st));
    return two ? (reg ? launch<4, 2, true>(job, smem, st) : launch<4, 2, false>(job, smem, st))
               : (reg ? launch<4, 1, true>(job, smem, st) : launch<4, 1, false>(job, smem, st));
}

}  // namespace pb
