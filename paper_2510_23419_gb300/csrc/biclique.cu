// biclique.cu -- CUDA-core kernels of the p-bit update on complete bipartite
// graphs K_{n,n} (arXiv 2510.23419, Sec. 3; update groups Sec. 1.2.2: the
// two sides are the two colour classes, every neighbour is shared by the
// whole class, so the field of a side is one dense product J M over replicas).
//
// The field F_A[r][i] = sum_j J[i][j] b[r][j] + h_i (Eq. 3) is an FP32 FMA
// tile product; the epilogue applies the p-bit decision (Eq. 2) with the
// Philox word of (i, s, r >> 2, side) and writes the new spins.  Fields of
// +-1 instances are exact integers in FP32 (|F| <= n + |h| < 2^24).
#include "biclique_launch.h"
#include "bit_count.cuh"
#include "ea_kernels.cuh"
#include "exact_split.cuh"

namespace pb {

namespace {

template <int SB>
struct SpinCode;
template <>
struct SpinCode<1> {
    using T = uint8_t;
    __device__ static float to_f(T v) { return __uint_as_float(0x3F800000u | ((uint32_t)(v & 0x80u) << 24)); }
    __device__ static T enc(bool minus) { return minus ? kE4m3Minus : kE4m3Plus; }
    __device__ static bool minus(T v) { return (v & 0x80u) != 0; }
};
template <>
struct SpinCode<2> {
    using T = uint16_t;
    __device__ static float to_f(T v) { return __uint_as_float((uint32_t)v << 16); }
    __device__ static T enc(bool minus) { return minus ? kBf16Minus : kBf16Plus; }
    __device__ static bool minus(T v) { return (v & 0x8000u) != 0; }
};


__global__ void __launch_bounds__(256) bq_init_kernel(BqJob job)
{
    const int n = job.inst.n;
    const long long tot = 2LL * job.Rpad * n;
    const long long j = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= tot) return;
    const int side = (int)(j / ((long long)job.Rpad * n));
    const long long rem = j - (long long)side * job.Rpad * n;
    const int r = (int)(rem / n);
    const int i = (int)(rem - (long long)r * n);
    const U4 w = philox10((uint32_t)i, 0u, (uint32_t)(r >> 2), (kTagInit << 24) | (uint32_t)side, job.key0, job.key1);
    const uint32_t ws[4] = {w.x, w.y, w.z, w.w};
    const bool minus = ws[r & 3] >= 0x80000000u;
    const size_t off = (size_t)r * job.ld + i;
    if (job.inst.jtype == PB_J_PM1_I8)
        static_cast<uint8_t*>(job.spins[side])[off] = minus ? kE4m3Minus : kE4m3Plus;
    else
        static_cast<uint16_t*>(job.spins[side])[off] = minus ? kBf16Minus : kBf16Plus;
}

// +-1 states (int8, [R][2n]) -> encoded spins of both sides.
__global__ void __launch_bounds__(256) bq_encode_kernel(BqJob job, const int8_t* __restrict__ m)
{
    const int n = job.inst.n;
    const long long j = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= (long long)job.R * 2 * n) return;
    const int r = (int)(j / (2 * n));
    const int c = (int)(j - (long long)r * 2 * n);
    const int side = c >= n ? 1 : 0;
    const int i = c - side * n;
    const bool minus = m[j] < 0;
    const size_t off = (size_t)r * job.ld + i;
    if (job.inst.jtype == PB_J_PM1_I8)
        static_cast<uint8_t*>(job.spins[side])[off] = minus ? kE4m3Minus : kE4m3Plus;
    else
        static_cast<uint16_t*>(job.spins[side])[off] = minus ? kBf16Minus : kBf16Plus;
}

constexpr int BM = kBqTileRows, BN = kBqTileReps, BK = 32;

template <int SB>
__global__ void __launch_bounds__(256) bq_cc_half_kernel(BqJob job, int side, int s_arg, const int32_t* sp, int decide,
                                                        float* fields_out)
{
    const int s = sp ? *sp : s_arg;
    if (decide && s >= job.S) return;
    using SC = SpinCode<SB>;
    using ST = typename SC::T;
    __shared__ __align__(16) float As[BK][BM + 4];
    __shared__ __align__(16) float Bs[BK][BN + 4];
    __shared__ float red[16][BN + 1];
    __shared__ float redh[16][BN + 1];

    const int n = job.inst.n;
    const float* __restrict__ Jm = side == 0 ? job.inst.Jf : job.inst.Jft;
    const ST* __restrict__ other = static_cast<const ST*>(job.spins[1 - side]);
    ST* __restrict__ own = static_cast<ST*>(job.spins[side]);
    const int i0 = blockIdx.x * BM;
    const int r0 = blockIdx.y * BN;
    const int t = threadIdx.x;
    const int ty = t >> 4, tx = t & 15;

    float acc[4][4];
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) acc[a][b] = 0.0f;

    const int lrow = t >> 2;          // 0..63
    const int lcol = (t & 3) * 8;     // 0, 8, 16, 24
    for (int j0 = 0; j0 < n; j0 += BK) {
        {
            const int i = i0 + lrow;
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const int j = j0 + lcol + q;
                As[lcol + q][lrow] = (i < n && j < n) ? __ldg(Jm + (size_t)i * n + j) : 0.0f;
            }
            const int r = r0 + lrow;
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const int j = j0 + lcol + q;
                Bs[lcol + q][lrow] = (j < n) ? SC::to_f(other[(size_t)r * job.ld + j]) : 0.0f;
            }
        }
        __syncthreads();
#pragma unroll 8
        for (int kk = 0; kk < BK; ++kk) {
            const float4 a = *reinterpret_cast<const float4*>(&As[kk][ty * 4]);
            const float4 b = *reinterpret_cast<const float4*>(&Bs[kk][tx * 4]);
            const float av[4] = {a.x, a.y, a.z, a.w};
            const float bv[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
            for (int x = 0; x < 4; ++x)
#pragma unroll
                for (int y = 0; y < 4; ++y) acc[x][y] = fmaf(av[x], bv[y], acc[x][y]);
        }
        __syncthreads();
    }

    // ---- epilogue: decisions (Eq. 2), energy partials ----
    const bool pm1 = job.inst.jtype == PB_J_PM1_I8;
    const uint32_t* trow = nullptr;
    float cexp = 0.0f;
    TabWindow win{0, 0, 1};
    if (pm1 && decide) {
        const int l = s / job.step;
        win = TabWindow{job.win[3 * l + 2], job.win[3 * l], job.win[3 * l + 1]};
    }
    if (pm1)
        trow = job.table + win.off;
    else
        cexp = f32_cexp(job.betaf[s / job.step]);
    float e_field[4] = {0.f, 0.f, 0.f, 0.f};  // -m F  (side B)
    float e_h[4] = {0.f, 0.f, 0.f, 0.f};      // -h m  (side A)
    const int rq = r0 + tx * 4;
#pragma unroll
    for (int x = 0; x < 4; ++x) {
        const int i = i0 + ty * 4 + x;
        if (i >= n) continue;
        const float hv = pm1 ? (job.inst.h8 ? (float)job.inst.h8[side * n + i] : 0.0f) : job.inst.hf[side * n + i];
        float F[4];
#pragma unroll
        for (int b = 0; b < 4; ++b) F[b] = acc[x][b] + hv;
        if (fields_out) {
#pragma unroll
            for (int b = 0; b < 4; ++b)
                if (rq + b < job.R) fields_out[(size_t)(rq + b) * 2 * n + side * n + i] = F[b];
            continue;
        }
        bool mn[4];
        if (decide) {
            const U4 w = philox10((uint32_t)i, (uint32_t)s, (uint32_t)(rq >> 2), (kTagDecision << 24) | (uint32_t)side,
                                  job.key0, job.key1);
            const uint32_t ws[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
            for (int b = 0; b < 4; ++b) {
                mn[b] = pm1 ? (ws[b] >= trow[min(max((int)F[b] - job.fmin, win.lo), win.lo + win.width - 1) - win.lo])
                            : (decide_f32(ws[b], F[b], cexp) != 0u);
                own[(size_t)(rq + b) * job.ld + i] = SC::enc(mn[b]);
            }
        } else {
#pragma unroll
            for (int b = 0; b < 4; ++b) mn[b] = SC::minus(own[(size_t)(rq + b) * job.ld + i]);
        }
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            if (side == 1) e_field[b] += mn[b] ? F[b] : -F[b];
            e_h[b] += mn[b] ? hv : -hv;
        }
    }
    if (fields_out) return;
#pragma unroll
    for (int b = 0; b < 4; ++b) {
        red[ty][tx * 4 + b] = e_field[b];
        redh[ty][tx * 4 + b] = e_h[b];
    }
    __syncthreads();
    if (t < BN) {
        float ef = 0.0f, eh = 0.0f;
        for (int q = 0; q < 16; ++q) {
            ef += red[q][t];
            eh += redh[q][t];
        }
        // side A: -h.a ; side B: -b.F_B (F_B includes h_B) -> partial rows [0] and [1]
        const size_t off = ((size_t)side * job.nblk + blockIdx.x) * job.Rpad + r0 + t;
        const float v = side == 0 ? eh : ef;
        if (pm1)
            static_cast<int32_t*>(job.part)[off] = (int32_t)v;
        else
            static_cast<float*>(job.part)[off] = v;
    }
}

// Energy of the state after the sweep (the row-tile partials of both sides,
// summed in a fixed order) and running best; 32 replicas per block, one thread
// per replica reads the partials (coalesced across replicas).  Best states are
// copied lazily: the live states alternate between two buffers per side by
// sweep parity, so the state of sweep s - 1 survives sweep s, and a replica's
// rows are copied only when an improving sweep is followed by one that does
// not improve (and once after the last sweep).
constexpr int kEndReps = 32;

// Copy the rows of the flagged replicas of a block (one warp per replica, eight
// independent 16-byte loads in flight per lane) from the live buffers of parity
// `par` into the best buffers.
__device__ __forceinline__ void bq_copy_flagged(const BqJob& job, int r0, const int* flag, int par)
{
    const int nvec = job.ld * (job.inst.jtype == PB_J_PM1_I8 ? 1 : 2) / 16;  // the row is a multiple of 16 bytes
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int q = warp; q < kEndReps; q += (int)(blockDim.x >> 5)) {
        if (!flag[q]) continue;
        const size_t row = (size_t)(r0 + q) * nvec;
        for (int side = 0; side < 2; ++side) {
            const uint4* __restrict__ src = static_cast<const uint4*>(job.buf[side][par]) + row;
            uint4* __restrict__ dst = static_cast<uint4*>(job.best[side]) + row;
            for (int k0 = lane; k0 < nvec; k0 += 32 * 8) {
                uint4 t[8];
#pragma unroll
                for (int u = 0; u < 8; ++u)
                    if (k0 + 32 * u < nvec) t[u] = src[k0 + 32 * u];
#pragma unroll
                for (int u = 0; u < 8; ++u)
                    if (k0 + 32 * u < nvec) dst[k0 + 32 * u] = t[u];
            }
        }
    }
}

__global__ void __launch_bounds__(256) bq_sweep_end_kernel(BqJob job, int s_arg, int init, const int32_t* sp_read,
                                                          int32_t* sp_write)
{
    // a programmatic dependent of the half-sweep before it in tensor-form runs that
    // set BqJob::pdl (otherwise both instructions do nothing)
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int s = sp_read ? *sp_read : s_arg;
    // read by the next sweep's launches; a max, because in stop mode the block that sees the
    // last replica reach the target raises it to S
    if (sp_write && blockIdx.x == 0 && threadIdx.x == 0) atomicMax(sp_write, s + 1);
    if (!init && s >= job.S) return;
    __shared__ int s_copy[kEndReps];
    constexpr int kSub = 8;  // partial-row subsets, one per warp
    __shared__ int32_t s_pi[kSub][kEndReps];
    __shared__ float s_pf[kSub][kEndReps];
    const int r0 = blockIdx.x * kEndReps;
    const bool pm1 = job.inst.jtype == PB_J_PM1_I8;
    {
        // warp k adds the partial rows b = k, k + 8, ... of both sides for the
        // block's 32 replicas (coalesced across replicas); the 8 subset sums are
        // then added in the fixed order k = 0..7
        const int k = threadIdx.x >> 5, r = r0 + (threadIdx.x & 31);
        const int rows = 2 * job.nblk;
        // side 0's rows hold -h.a and stay zero without a field: start at side 1's
        // rows then, when nblk is a multiple of kSub (always in the tensor form), so
        // that warp k adds the same side-1 rows in the same order, after the same
        // zeros: the same sums
        const int first = (job.inst.has_h || job.nblk % kSub) ? 0 : job.nblk;
        if (pm1) {
            const int32_t* p = static_cast<const int32_t*>(job.part);
            int32_t E = 0;
            for (int b = first + k; b < rows; b += kSub) E += p[(size_t)b * job.Rpad + r];
            s_pi[k][threadIdx.x & 31] = E;
        } else {
            const float* p = static_cast<const float*>(job.part);
            float E = 0.0f;
            for (int b = first + k; b < rows; b += kSub) E += p[(size_t)b * job.Rpad + r];
            s_pf[k][threadIdx.x & 31] = E;
        }
    }
    __syncthreads();
    if (threadIdx.x < kEndReps && r0 + (int)threadIdx.x >= job.R) {
        s_copy[threadIdx.x] = 0;  // padding replicas: nothing to record (the tensor form leaves them as they are)
    } else if (threadIdx.x < kEndReps) {
        const int r = r0 + threadIdx.x;
        bool imp, hit_now = false;
        const int prev = init ? -2 : job.best_sweep[r];
        const bool live = init || job.has_target != 2 || job.hit_sweep[r] < 0;  // stop mode: best frozen at the target
        if (pm1) {
            int32_t E = 0;
#pragma unroll
            for (int k = 0; k < kSub; ++k) E += s_pi[k][threadIdx.x];
            imp = init || (live && E < job.E_best_i[r]);
            if (imp) job.E_best_i[r] = E;
            hit_now = !init && job.has_target && job.hit_sweep[r] < 0 && E <= job.target_i;
        } else {
            float E = 0.0f;
#pragma unroll
            for (int k = 0; k < kSub; ++k) E += s_pf[k][threadIdx.x];
            imp = init || (live && E < job.E_best_f[r]);
            if (imp) job.E_best_f[r] = E;
            hit_now = !init && job.has_target && job.hit_sweep[r] < 0 && E <= job.target_f;
        }
        if (hit_now) {
            job.hit_sweep[r] = s;
            // stop mode: the last replica to reach the target ends the run after this sweep
            if (job.has_target == 2 && r < job.R && atomicAdd(job.stop, 1) + 1 == job.R) {
                job.stop[1] = s;
                if (sp_write) atomicMax(sp_write, job.S);
            }
        }
        if (init) job.hit_sweep[r] = -1;
        if (imp) job.best_sweep[r] = init ? -1 : s;
        // the best is state s - 1, and sweep s + 1 will overwrite its buffers: copy it now
        s_copy[threadIdx.x] = (!init && !imp && prev == s - 1) ? 1 : 0;
    }
    __syncthreads();
    if (!init) bq_copy_flagged(job, r0, s_copy, (s - 1) & 1);
}

// The sweep whose state the live buffers end with: S - 1, or the sweep after
// which a stop-mode run ended.
__device__ __forceinline__ int bq_last_sweep(const BqJob& job)
{
    return (job.has_target == 2 && job.stop[1] >= 0) ? job.stop[1] : job.S - 1;
}

__global__ void __launch_bounds__(256) bq_best_flush_kernel(BqJob job)
{
    __shared__ int s_copy[kEndReps];
    const int r0 = blockIdx.x * kEndReps;
    const int last = bq_last_sweep(job);
    if (threadIdx.x < kEndReps)
        s_copy[threadIdx.x] = (r0 + (int)threadIdx.x < job.R && job.best_sweep[r0 + threadIdx.x] == last) ? 1 : 0;
    __syncthreads();
    bq_copy_flagged(job, r0, s_copy, last & 1);
}

// Spin words of a state set: bit c of word [r][side][w] set <=> m of spin 32 w + c is -1.
__global__ void __launch_bounds__(256) bq_readout_kernel(BqJob job, int which, int8_t* __restrict__ out)
{
    // a thread reads 32 encoded spins and writes their 32 output bytes and, for +-1, their bit word
    const int n = job.inst.n, W = (n + 31) / 32;
    const long long j = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= 2LL * job.R * W) return;
    const int rs = (int)(j / W), w = (int)(j - (long long)rs * W);
    const int r = rs >> 1, side = rs & 1;
    const void* src_side;
    if (which)
        src_side = job.best[side];
    else if (job.has_target == 2 && job.stop && job.stop[1] >= 0)  // stopped early: the live buffers of that sweep
        src_side = job.buf[side][job.stop[1] & 1];
    else
        src_side = job.spins[side];
    const bool pm1 = job.inst.jtype == PB_J_PM1_I8;
    uint32_t bits = 0;
    // rows are multiples of 16 elements, so whole 16-byte loads stay inside the row
    if (pm1) {
        const uint4* src = reinterpret_cast<const uint4*>(static_cast<const uint8_t*>(src_side) + (size_t)r * job.ld) + 2 * w;
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            if (32 * w + 16 * q >= n) break;
            const uint4 v = src[q];
            const uint32_t x[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const uint32_t t = (x[u] >> 7) & 0x01010101u;  // the four sign bits to bits 0..3
                bits |= ((t | (t >> 7) | (t >> 14) | (t >> 21)) & 0xFu) << (16 * q + 4 * u);
            }
        }
    } else {
        const uint4* src = reinterpret_cast<const uint4*>(static_cast<const uint16_t*>(src_side) + (size_t)r * job.ld) + 4 * w;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            if (32 * w + 8 * q >= n) break;
            const uint4 v = src[q];
            const uint32_t x[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int u = 0; u < 4; ++u) bits |= (((x[u] >> 15) & 1u) | ((x[u] >> 30) & 2u)) << (8 * q + 2 * u);
        }
    }
    const int left = n - 32 * w;
    if (left < 32) bits &= (1u << left) - 1u;
    if (pm1) job.sbits[j] = bits;
    int8_t* dst = out + (size_t)r * 2 * n + (size_t)side * n + 32 * w;
    if (left >= 32 && (n & 3) == 0) {
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const uint32_t f = (bits >> (4 * u)) & 0xFu;
            const uint32_t t = (f & 1u) | ((f & 2u) << 7) | ((f & 4u) << 14) | ((f & 8u) << 21);
            reinterpret_cast<uint32_t*>(dst)[u] = 0x01010101u + t * 0xFEu;  // 0x01 = +1, 0xFF = -1
        }
    } else {
        for (int c = 0; c < min(left, 32); ++c) dst[c] = ((bits >> c) & 1u) ? (int8_t)-1 : (int8_t)1;
    }
}

// Sign words of +-1 couplings: bit c of word [i][w] set <=> J[i][32 w + c] = -1.
__global__ void __launch_bounds__(256) bq_sign_words_kernel(const int8_t* __restrict__ J, int n, uint32_t* __restrict__ out)
{
    const int W = (n + 31) / 32, lane = threadIdx.x & 31;
    const long long word = (long long)blockIdx.x * 8 + (threadIdx.x >> 5);  // a warp per word
    if (word >= (long long)n * W) return;
    const int i = (int)(word / W), j = (int)(word - (long long)i * W) * 32 + lane;
    const uint32_t m = __ballot_sync(0xFFFFFFFFu, j < n && J[(size_t)i * n + j] < 0);
    if (lane == 0) out[word] = m;
}

// Exact energy of returned states (Eq. 1 with the sign reading E = -sum J a b - sum h m).
// Tiled over 64 rows i x 64 replicas r, 4 x 4 per thread: U[i][r] = sum_j J[i][j] b[r][j], then
// the tile's part -sum_i a[r][i] U[i][r] goes to epart[row tile][r].
constexpr int kEt = 64;
constexpr int kEtLd = kEt + 4;  // row stride in shared memory: vector loads of 4 neighbours, no conflicts

// The tile's -sum_i a U per replica: the threads' rows, then the 16 row quads in order.
__device__ __forceinline__ void bq_energy_reduce(const BqJob& job, const double (&part)[4], int r0, double (&red)[16][kEt + 1])
{
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
#pragma unroll
    for (int b = 0; b < 4; ++b) red[ty][tx * 4 + b] = part[b];
    __syncthreads();
    if (threadIdx.x < kEt) {
        const int r = r0 + threadIdx.x;
        double t = 0.0;
        for (int q = 0; q < 16; ++q) t += red[q][threadIdx.x];
        if (r < job.R) job.epart[(size_t)blockIdx.x * job.R + r] = t;
    }
}

// +-1: U = n - 2 popc(J ^ b) on sign words, eight words at a time carry-save compressed to four
// population counts.  n = 4096, 4096 replicas: 0.64 ms per state set with its state copy (int8
// products with __dp4a and a byte per thread, which this replaces, 1.79 ms).
__global__ void __launch_bounds__(256) bq_energy_bits_kernel(BqJob job)
{
    const int n = job.inst.n, R = job.R, W = (n + 31) / 32;
    const int i0 = blockIdx.x * kEt, r0 = blockIdx.y * kEt;
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;  // replica quad, row quad
    constexpr int KW = 16;                                     // words per stage
    __shared__ __align__(16) uint32_t Js[KW][kEtLd];
    __shared__ __align__(16) uint32_t Bs[KW][kEtLd];
    __shared__ double red[16][kEt + 1];
    int pc[4][4];
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) pc[a][b] = 0;
    for (int w0 = 0; w0 < W; w0 += KW) {
        for (int e = threadIdx.x; e < kEt * KW; e += 256) {
            const int w = e % KW, q = e / KW;
            const bool in = w0 + w < W;
            Js[w][q] = in && i0 + q < n ? job.inst.Jbits[(size_t)(i0 + q) * W + w0 + w] : 0u;
            Bs[w][q] = in && r0 + q < R ? job.sbits[((size_t)(r0 + q) * 2 + 1) * W + w0 + w] : 0u;
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < KW; k += 8) {
            uint32_t jv[8][4], bv[8][4];
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const uint4 x = *reinterpret_cast<const uint4*>(&Js[k + u][ty * 4]);
                const uint4 y = *reinterpret_cast<const uint4*>(&Bs[k + u][tx * 4]);
                jv[u][0] = x.x, jv[u][1] = x.y, jv[u][2] = x.z, jv[u][3] = x.w;
                bv[u][0] = y.x, bv[u][1] = y.y, bv[u][2] = y.z, bv[u][3] = y.w;
            }
#pragma unroll
            for (int a = 0; a < 4; ++a)
#pragma unroll
                for (int b = 0; b < 4; ++b) {
                    uint32_t x[8];
#pragma unroll
                    for (int u = 0; u < 8; ++u) x[u] = jv[u][a] ^ bv[u][b];
                    pc[a][b] += popc_words<8>(x);
                }
        }
        __syncthreads();
    }
    double part[4];
#pragma unroll
    for (int b = 0; b < 4; ++b) {
        const int r = r0 + tx * 4 + b;
        int t = 0;  // |t| <= 4 n
#pragma unroll
        for (int a = 0; a < 4; ++a) {
            const int i = i0 + ty * 4 + a;
            if (i < n && r < R) {
                const int U = n - 2 * pc[a][b];
                t += (job.sbits[(size_t)r * 2 * W + (i >> 5)] >> (i & 31)) & 1u ? U : -U;
            }
        }
        part[b] = (double)t;
    }
    bq_energy_reduce(job, part, r0, red);
}

// Real couplings: split into two FP32 parts whose sums over 64 terms are exact (exact_split.cuh).  Every 64
// columns the two sums go into an unevaluated pair hi + lo by the error-free two-sum (Knuth), 1/32nd of
// the roundings of a two-sum per term: two fused multiply-adds per term instead of seven operations.  A coupling that
// has no such split goes into the pair by a two-sum of its own; the columns of a tile that hold one (for N(0,1)
// draws one in ten) are known to the whole CTA.  n = 2048, 1024 replicas: 0.75 ms per state set with
// its state copy (two-sum per term: 1.31 ms); shared-memory reads bound it.
__device__ __forceinline__ void two_sum_acc(float& hi, float& lo, float x)
{
    const float s = hi + x;
    const float bb = s - hi;
    const float err = (hi - (s - bb)) + (x - bb);
    hi = s;
    lo += err;
}

constexpr size_t kEnergyF32Smem = (size_t)4 * kEt * kEtLd * 4;

__global__ void __launch_bounds__(256) bq_energy_f32_kernel(BqJob job, const int8_t* __restrict__ m)
{
    extern __shared__ __align__(16) float sm[];
    const int n = job.inst.n, R = job.R;
    const int i0 = blockIdx.x * kEt, r0 = blockIdx.y * kEt;
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    float* const P[3] = {sm, sm + kEt * kEtLd, sm + 2 * kEt * kEtLd};  // parts of J, J not split: [column][row]
    float* const Bs = sm + 3 * kEt * kEtLd;                            // spins: [column][replica]
    __shared__ double red[16][kEt + 1];
    __shared__ __align__(8) uint8_t s_whole[8];  // bit per column: some row's J is not split
    const float unit = job.inst.junit;
    const float* J = static_cast<const float*>(job.inst.Jraw);
    float hi[4][4], lo[4][4];
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            hi[a][b] = 0.0f;
            lo[a][b] = 0.0f;
        }
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int j0 = 0; j0 < n; j0 += kEt) {
        bool whole = false;
        for (int e = threadIdx.x; e < kEt * kEt; e += 256) {
            // a warp takes 8 columns x 4 rows: whole sectors read, distinct banks written
            const int j = warp * 8 + (e & 7), q = (e >> 8) * 4 + ((e >> 3) & 3);
            const int i = i0 + q, r = r0 + q;
            const float x = (i < n && j0 + j < n) ? J[(size_t)i * n + j0 + j] : 0.0f;
            float q1, q2;
            const bool split = split_exact(x, unit, q1, q2);
            whole |= !split;
            P[0][j * kEtLd + q] = split ? q1 : 0.0f;
            P[1][j * kEtLd + q] = split ? q2 : 0.0f;
            P[2][j * kEtLd + q] = split ? 0.0f : x;
            Bs[j * kEtLd + q] = (r < R && j0 + j < n) ? (float)m[(size_t)r * 2 * n + n + j0 + j] : 1.0f;
        }
        uint32_t cols = __ballot_sync(0xFFFFFFFFu, whole);  // lanes 8 apart share a column
        cols |= cols >> 16;
        cols |= cols >> 8;
        if (lane == 0) s_whole[warp] = (uint8_t)cols;
        __syncthreads();
        float s[2][4][4];
#pragma unroll
        for (int d = 0; d < 2; ++d)
#pragma unroll
            for (int a = 0; a < 4; ++a)
#pragma unroll
                for (int b = 0; b < 4; ++b) s[d][a][b] = 0.0f;
#pragma unroll 2
        for (int j = 0; j < kEt; ++j) {
            const float4 bv = *reinterpret_cast<const float4*>(Bs + j * kEtLd + tx * 4);
            const float bb[4] = {bv.x, bv.y, bv.z, bv.w};
#pragma unroll
            for (int d = 0; d < 2; ++d) {
                const float4 jv = *reinterpret_cast<const float4*>(P[d] + j * kEtLd + ty * 4);
                const float ja[4] = {jv.x, jv.y, jv.z, jv.w};
#pragma unroll
                for (int a = 0; a < 4; ++a)
#pragma unroll
                    for (int b = 0; b < 4; ++b) s[d][a][b] = fmaf(ja[a], bb[b], s[d][a][b]);
            }
        }
#pragma unroll
        for (int d = 0; d < 2; ++d)
#pragma unroll
            for (int a = 0; a < 4; ++a)
#pragma unroll
                for (int b = 0; b < 4; ++b) two_sum_acc(hi[a][b], lo[a][b], s[d][a][b]);
        for (unsigned long long m = *reinterpret_cast<const unsigned long long*>(s_whole); m; m &= m - 1) {
            const int j = __ffsll((long long)m) - 1;
            const float4 bv = *reinterpret_cast<const float4*>(Bs + j * kEtLd + tx * 4);
            const float4 jv = *reinterpret_cast<const float4*>(P[2] + j * kEtLd + ty * 4);
            const float bb[4] = {bv.x, bv.y, bv.z, bv.w}, ja[4] = {jv.x, jv.y, jv.z, jv.w};
#pragma unroll
            for (int a = 0; a < 4; ++a)
#pragma unroll
                for (int b = 0; b < 4; ++b) two_sum_acc(hi[a][b], lo[a][b], ja[a] * bb[b]);
        }
        __syncthreads();
    }
    double part[4];
#pragma unroll
    for (int b = 0; b < 4; ++b) {
        const int r = r0 + tx * 4 + b;
        double t = 0.0;
#pragma unroll
        for (int a = 0; a < 4; ++a) {
            const int i = i0 + ty * 4 + a;
            if (i < n && r < R) t -= (double)m[(size_t)r * 2 * n + i] * ((double)hi[a][b] + (double)lo[a][b]);
        }
        part[b] = t;
    }
    bq_energy_reduce(job, part, r0, red);
}

// E[r] = sum over row tiles of epart (fixed order) - sum_c h_c m_c; one warp per replica.
template <int JT>
__global__ void __launch_bounds__(256) bq_energy_sum_kernel(BqJob job, const int8_t* __restrict__ m, double* __restrict__ E)
{
    const int n = job.inst.n, R = job.R;
    const int r = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (r >= R) return;
    const int nt = (n + kEt - 1) / kEt;
    double t = 0.0;
    for (int q = lane; q < nt; q += 32) t += job.epart[(size_t)q * R + r];
    if (job.inst.hraw) {
        for (int c = lane; c < 2 * n; c += 32) {
            const double hv = JT == PB_J_PM1_I8 ? (double)static_cast<const int8_t*>(job.inst.hraw)[c]
                                                : (double)static_cast<const float*>(job.inst.hraw)[c];
            t -= hv * (double)m[(size_t)r * 2 * n + c];
        }
    }
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xFFFFFFFFu, t, o);
    if (lane == 0) E[r] = t;
}

unsigned nblocks(long long n, int bs) { return (unsigned)((n + bs - 1) / bs); }

}  // namespace

cudaError_t bq_launch_init(const BqJob& job, cudaStream_t st)
{
    const long long tot = 2LL * job.Rpad * job.inst.n;
    bq_init_kernel<<<nblocks(tot, 256), 256, 0, st>>>(job);
    return cudaGetLastError();
}

cudaError_t bq_launch_encode(const BqJob& job, const int8_t* d_states, cudaStream_t st)
{
    bq_encode_kernel<<<nblocks((long long)job.R * 2 * job.inst.n, 256), 256, 0, st>>>(job, d_states);
    return cudaGetLastError();
}

cudaError_t bq_launch_cc_half(const BqJob& job, int side, int s, const int32_t* sp, int decide, float* fields_out,
                              cudaStream_t st)
{
    dim3 grid((unsigned)((job.inst.n + BM - 1) / BM), (unsigned)(job.Rpad / BN));
    if (job.inst.jtype == PB_J_PM1_I8)
        bq_cc_half_kernel<1><<<grid, 256, 0, st>>>(job, side, s, sp, decide, fields_out);
    else
        bq_cc_half_kernel<2><<<grid, 256, 0, st>>>(job, side, s, sp, decide, fields_out);
    return cudaGetLastError();
}

cudaError_t bq_launch_sweep_end(const BqJob& job, int s, int init, const int32_t* sp_read, int32_t* sp_write,
                                cudaStream_t st)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(job.Rpad / kEndReps));
    cfg.blockDim = dim3(256);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    if (job.pdl && sp_read) {  // inside a tensor-form sweep loop: a programmatic dependent of its half-sweep
        attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[0].val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
    }
    return cudaLaunchKernelEx(&cfg, bq_sweep_end_kernel, job, s, init, sp_read, sp_write);
}

cudaError_t bq_launch_best_flush(const BqJob& job, cudaStream_t st)
{
    bq_best_flush_kernel<<<job.Rpad / kEndReps, 256, 0, st>>>(job);
    return cudaGetLastError();
}

cudaError_t bq_launch_sign_words(const int8_t* J, int n, uint32_t* out, cudaStream_t st)
{
    bq_sign_words_kernel<<<nblocks((long long)n * ((n + 31) / 32), 8), 256, 0, st>>>(J, n, out);
    return cudaGetLastError();
}

cudaError_t bq_readout_set_smem()
{
    return cudaFuncSetAttribute(bq_energy_f32_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kEnergyF32Smem);
}

cudaError_t bq_launch_readout(const BqJob& job, int which, int8_t* out_pm, double* out_E, cudaStream_t st)
{
    const int W = (job.inst.n + 31) / 32;
    bq_readout_kernel<<<nblocks(2LL * job.R * W, 256), 256, 0, st>>>(job, which, out_pm);
    const dim3 grid((unsigned)((job.inst.n + kEt - 1) / kEt), (unsigned)((job.R + kEt - 1) / kEt));
    if (job.inst.jtype == PB_J_PM1_I8) {
        bq_energy_bits_kernel<<<grid, 256, 0, st>>>(job);
        bq_energy_sum_kernel<PB_J_PM1_I8><<<nblocks(job.R, 8), 256, 0, st>>>(job, out_pm, out_E);
    } else {
        bq_energy_f32_kernel<<<grid, 256, kEnergyF32Smem, st>>>(job, out_pm);
        bq_energy_sum_kernel<PB_J_F32><<<nblocks(job.R, 8), 256, 0, st>>>(job, out_pm, out_E);
    }
    return cudaGetLastError();
}

}  // namespace pb
