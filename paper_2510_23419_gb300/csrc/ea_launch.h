// ea_launch.h -- host/device interface of the EA (periodic L^3 cube) kernels.
#pragma once

#include "pb_common.h"

namespace pb {

// One anneal job as the kernels see it (plain form: one tile with WT = R/4
// rounded up; resident form: tiles of 4*WT replicas).  State buffers use the
// tile layout: word ((tile*2 + c)*half + k)*WT + w holds replicas
// tile*4*WT + 4w + (0..3) of the site of colour c and class rank k.
struct EaJob {
    EaDevice inst;
    uint32_t key0, key1;      // Philox key = seed
    int32_t S;                // sweeps
    int32_t step;             // sweeps per beta level (1 for explicit schedules)
    int32_t nF;               // PM1: threshold table width (F_max - F_min + 1)
    int32_t fmin;             // PM1: F_min
    const uint32_t* table;    // PM1: [levels][nF] thresholds
    const float* betaf;       // F32: [levels] beta as float
    int32_t R;                // replicas requested
    int32_t WT;               // words (4 replicas each) per site in one tile
    int32_t n_tiles;
    int32_t has_target;       // 0: none; 1: record the first sweep at the target; 2: also freeze the
                              // running best there and stop once every replica has reached it
    int32_t target_i;         // PM1 target energy (integer)
    float target_f;           // F32 target energy
    uint32_t* best_words;     // tile layout
    uint32_t* final_words;    // tile layout (plain form: the live state)
    int32_t* E_best_i;        // PM1 running-best energy  [n_tiles*4*WT]
    float* E_best_f;          // F32 running-best energy
    int32_t* best_sweep;      // [n_tiles*4*WT]
    int32_t* hit_sweep;       // [n_tiles*4*WT]
    int32_t* n_hit;           // plain form, has_target == 2: replicas that reached the target (device counter)
    int32_t s0;               // first sweep (resident form: > 0 only for a resumed run)
    int32_t resume;           // resident form: the initial state is final_words, the running best
                              // (best_words, E_best_*, best_sweep) is given
    int32_t groups;           // 0: state buffers in the byte layout above; else (resident +-1 runs) one bit
                              // per spin, `groups` sites per word: word ((tile*2 + c)*nw + wi)*WT + w,
                              // nw = half / groups, bit 8 b + g = replica b of the quad at class rank wi + g nw
    int32_t split;            // +-1: the job runs on the kernel of split words (EaKernel); FP32: threads per
                              // summation lane (ea_f32_split)
    int32_t threads;          // resident runs: threads of the CTA that take words or lanes
    double* E_out[2];         // resident +-1 runs: energies of the final and the best states [R], counted
                              // from the states by the tile itself
};

// Tile code of the resident kernels (chosen on the host, so the kernel
// branches on one word of the work item).  FP32 tiles:
enum EaTilePath : int32_t {
    kEaPathGeneric = 0,  // any even L <= 32
    kEaPathFast32 = 1,   // compile-time tile L = 32, WT = 1
    kEaPathFast16 = 2,   // L = 16, WT = 4
    kEaPathFast8 = 3,    // L = 8, WT = 16
    kEaPathFast24 = 7,   // compile-time tile L = 24, WT = 1 (576 of the CTA's threads hold sites)
};

// +-1 tiles (ea_bits.cuh): G sites per spin word, CPT Philox calls of a word per
// thread, the thread's words all in one (x, y) column or not, with fields or not.
__host__ __device__ constexpr int32_t ea_bits_path(int G, int CPT, bool column, bool has_h)
{
    return (1 << 16) | (G << 8) | (CPT << 4) | (column ? 2 : 0) | (has_h ? 1 : 0);
}
// Sites per spin word of a +-1 tile: gcd(L, 8) for an even L.
__host__ __device__ constexpr int ea_bits_groups(int L) { return L % 8 == 0 ? 8 : (L % 4 == 0 ? 4 : 2); }

struct EaWork {
    int32_t job;
    int32_t tile;
    int32_t path;  // EaTilePath, or ea_bits_path of a +-1 job
};

// Shared memory of one +-1 tile: byte offsets of its parts.  Spins: two buffers of
// class 0, one of class 1, then the best state; bond words and field bytes; two
// threshold rows (with fields); two sets of energy sums; improved flags.
struct EaBitsLayout {
    size_t best, bonds, h, tab, eacc, flags, total;
    int tab_bytes;  // of one row
};

__host__ __device__ inline EaBitsLayout ea_bits_layout(int L, int WT, int has_h, int nF)
{
    const size_t N = (size_t)L * L * L;
    const int G = ea_bits_groups(L);
    const size_t words = N / 2 / G * WT;  // of one class
    EaBitsLayout o{};
    size_t b = 3 * words * 4;
    o.best = b;
    b += 2 * words * 4;
    b = (b + 15) / 16 * 16;
    o.bonds = b;
    b += N / G * (G == 8 ? 8 : 4);
    o.h = b;
    if (has_h) b += N;
    b = (b + 15) / 16 * 16;
    o.tab = b;
    o.tab_bytes = has_h ? (nF + 3) / 4 * 16 : 0;
    b += 2 * (size_t)o.tab_bytes;
    o.eacc = b;
    b += 2 * (size_t)4 * WT * 4;
    o.flags = b;
    b += (size_t)4 * WT;
    o.total = (b + 127) / 128 * 128;
    return o;
}

// CTA of the +-1 kernel: 512 threads of 128 registers.  With 1024 threads of 64 the
// tiles ran 7% (L = 32) to 35% (L = 16, one quad) slower, with 256 threads 8% slower
// at L = 32 (too few warps).
constexpr int kBitsThreads = 512;

// Launch shape of a +-1 tile of the job.
struct EaBitsShape {
    int lanes;    // threads per spin word
    int threads;  // of the CTA that the tile keeps busy, whole warps
    bool column;  // a thread's words are in one (x, y) column
};
// One thread per word shares the word's neighbour loads and counts among all its G
// Philox calls.  Tiles of fewer than 256 words (8 warps) are bound by latency, not by
// the SM's pipes: with `split`, the calls of a word go to threads of their own, lanes of
// one word staying inside a warp (L = 6, 64 replicas: 0.9 against 1.2 us per sweep; at
// 256 words, L = 16, splitting lost 12%).
inline EaBitsShape ea_bits_shape(const EaJob& j, bool split)
{
    const int G = ea_bits_groups(j.inst.L);
    const int words = j.inst.N / 2 / G * j.WT;  // of one class
    EaBitsShape o{1, 0, false};
    while (split && 2 * o.lanes <= G && words * 2 * o.lanes <= kBitsThreads && words * o.lanes < 256 &&
           2 * o.lanes * j.WT <= 32)
        o.lanes *= 2;
    if (j.inst.has_h && o.lanes > 1)  // compiled with fields: one thread per word or one per call
        o.lanes = G * j.WT <= 32 && words * G <= kBitsThreads ? G : 1;
    // (Fewer threads with even shares of the words ran slower: L = 24 by 12%, as 14 warps load the four
    // schedulers of an SM unevenly.)
    const int need = words * o.lanes;
    o.threads = need >= kBitsThreads ? kBitsThreads : need < 128 ? 128 : (need + 31) / 32 * 32;
    const int columns = j.inst.L / 2 * j.inst.L * j.WT;
    o.column = need <= o.threads || (o.threads / o.lanes) % columns == 0;
    return o;
}

inline int32_t ea_tile_path_f32(int L, int WT)
{
    if (L == 32 && WT == 1) return kEaPathFast32;
    if (L == 16 && WT == 4) return kEaPathFast16;
    if (L == 8 && WT == 16) return kEaPathFast8;
    if (L == 24 && WT == 1) return kEaPathFast24;
    return kEaPathGeneric;
}

inline int32_t ea_tile_path(const EaJob& j)
{
    if (j.inst.jtype == PB_J_PM1_I8) {
        const EaBitsShape o = ea_bits_shape(j, j.split != 0);
        const int G = ea_bits_groups(j.inst.L), cpt = G / o.lanes;
        // compiled variants: one thread per word with fields has no column form, several have only that
        const bool column = cpt < G ? true : (j.inst.has_h ? false : o.column);
        return ea_bits_path(G, cpt, column, j.inst.has_h != 0);
    }
    return ea_tile_path_f32(j.inst.L, j.WT);
}

// FP32 tiles: `lanes` = L^2 WT summation lanes (at most 1024) on 512 threads, two per thread, or one
// per thread where they fit the kernel's CTA (`most`: ea_kernel_threads).  With 1024 threads of 64
// registers a thread had one site in flight; with 512 it has two.  608 replicas, N(0,1), us per sweep, 1024
// threads against this: L = 32 31.8 / 29.3, L = 16 6.9 / 5.7, L = 20 13.9 / 11.7, L = 24 15.7 / 14.1; 9728 of L = 8
// 8.5 / 7.6.
__host__ __device__ constexpr int ea_f32_threads(int lanes, int most) { return lanes <= most ? lanes : 512; }
// Threads that share a summation lane: the lanes of a lone small job leave most of the CTA idle.  The
// fewest that give the least sites per thread, within 512 threads (us per sweep at 64 replicas, one
// thread per lane against this: L = 6 2.50 / 1.44, L = 10 3.56 / 2.39; L = 16 6.77 / 5.57).
inline int ea_f32_split(const EaJob& j)
{
    if (ea_tile_path_f32(j.inst.L, j.WT) != kEaPathGeneric) return 1;
    const int lanes = j.inst.L * j.inst.L * j.WT, sites = j.inst.L / 2;
    int best = 1;
    for (int k = 2; k <= sites && k * lanes <= 512; ++k)
        if ((sites + k - 1) / k < (sites + best - 1) / best) best = k;
    return best;
}

// Threads of the CTA (of at most `most`) that a tile of the job keeps busy, whole warps.
inline int ea_tile_threads(const EaJob& j, int most)
{
    if (j.inst.jtype == PB_J_PM1_I8) return ea_bits_shape(j, j.split != 0).threads;
    const int lanes = j.inst.L * j.inst.L * j.WT;
    const int t = ((j.split > 1 ? j.split * lanes : ea_f32_threads(lanes, most)) + 31) / 32 * 32;
    return t < 128 ? 128 : t;
}

// Persistent resident kernels.  For +-1 couplings, one with a thread per spin word
// and one with several (a launch takes the second if all its +-1 tiles gain by it;
// with both forms in one kernel, their shared register allocation spilled 230 B a
// thread and L = 32 ran 6% slower).  Two for FP32, which
// differ in their compile-time tiles -- the L = 32 tile, or the L = 24 tile,
// beside L = 16, L = 8 and the runtime-shaped generic tile.  With both the
// L = 32 and the L = 24 tile in one kernel, the register allocation they share
// slowed the L = 32 tile by 8%.  A batch takes the L = 24 kernel when its FP32
// tiles include ones of 576 lanes (L = 24, or 16 replicas of L = 12) and no L = 32
// ones; otherwise L = 24 FP32 tiles run the generic tile of the first kernel.
enum EaKernel : int32_t {
    kEaKernelPm1 = 0,
    kEaKernelPm1Split = 1,
    kEaKernelF32 = 2,
    kEaKernelF32L24 = 3,
    kEaKernels = 4
};
// Most threads of a kernel's CTA.  576 threads leave 96 registers each (five warps on one scheduler), 512
// leave 128.
constexpr int ea_kernel_threads(int kernel) { return kernel == kEaKernelF32L24 ? 576 : 512; }
// The +-1 kernel of a launch: split words if every +-1 job of it has tiles that gain.
inline bool ea_bits_gains_by_split(const EaJob& j) { return ea_bits_shape(j, true).lanes > 1; }

// Shared memory of one resident tile, in bytes.
__host__ __device__ inline size_t ea_resident_smem(int L, int WT, int jtype, int has_h, int nF)
{
    if (jtype == PB_J_PM1_I8) return ea_bits_layout(L, WT, has_h, nF).total;
    const size_t N = (size_t)L * L * L;
    size_t b = N * (size_t)WT * 4;          // spins [2][half][WT]
    b += (size_t)(1024 / 32) * 4 * WT * 4;  // per-warp energy partials
    b += (size_t)(4 * WT + 15) / 16 * 16;   // improved flags
    // energy terms of shared summation lanes (generic tile, lanes <= 256): 16 bytes per lane and site of the
    // class (of both with fields)
    if ((size_t)L * L * WT <= 256) b += (size_t)(has_h ? 2 : 1) * (L / 2) * L * L * WT * 16;
    return (b + 127) / 128 * 128;
}

constexpr int kResidentThreads = 1024;
constexpr int kResidentMaxWT = 32;
constexpr size_t kResidentSmemLimit = 227 * 1024;

// Largest power-of-two WT <= min(32, cap) such that the column-words of a
// class give at most 1024 summation lanes (h2*L*WT <= kResidentThreads/2: two lanes,
// one per z parity, per column) and the tile fits shared memory; 0 if none.
int ea_resident_pick_wt(int L, int jtype, int has_h, int nF, int cap_words);

// Opt the persistent kernel `kernel` (EaKernel) into `smem` bytes of dynamic
// shared memory (outside any capture).
cudaError_t ea_resident_set_smem(int kernel, size_t smem);
// Persistent kernel `kernel` (EaKernel) over n_work items of its coupling
// type.  after_previous: programmatic dependent launch on the kernel launched
// just before it on `st` (its CTAs start as that kernel's CTAs leave; the
// caller orders any later consumer after both).
// threads: the largest ea_tile_threads of its jobs.
cudaError_t ea_launch_resident(int kernel, const EaJob* d_jobs, const EaWork* d_work, int n_work, int* d_counter,
                               size_t smem, int grid, int threads, bool after_previous, cudaStream_t st);
// Random-word ceiling: `blocks` CTAs of kResidentThreads threads, each thread drawing the
// decision words of 32 sites (one L = 32 column, both colours) per sweep; sink holds
// blocks * kResidentThreads words.  Updates counted: blocks * kResidentThreads * 32 * 4 per sweep.
cudaError_t ea_launch_philox_ceiling(uint64_t seed, int sweeps, int blocks, uint32_t* sink, cudaStream_t st);
cudaError_t ea_launch_plain_init(const EaJob& job, cudaStream_t st);
cudaError_t ea_launch_plain_sweep(const EaJob& job, int s, cudaStream_t st);
cudaError_t ea_launch_plain_energy(const EaJob& job, int s, bool init, cudaStream_t st);
// Words of each class that a thread of the readout takes: it stores twice as many bytes at once, at offsets that are
// multiples of that from the output's address, which a caller of pb_anneal_ea_noalloc is free to choose.  0: no
// alignment, single bytes.
inline int ea_readout_sites(int L, uintptr_t out)
{
    for (int v = 4; v; v /= 2)
        if (L / 2 % v == 0 && out % (2 * v) == 0) return v;
    return 0;
}
// State buffer -> [R][N] int8 +-1, and energies recomputed from those states
// (int64 for PM1, FP64 for F32; not where job.groups is set: the resident +-1
// tiles have written E_out themselves).
cudaError_t ea_launch_readout(const EaJob& job, const uint32_t* words, int8_t* out_pm, double* out_E,
                              cudaStream_t st);
cudaError_t ea_launch_fields(const EaDevice& inst, const int8_t* d_states, int R, float* d_out, cudaStream_t st);

}  // namespace pb
