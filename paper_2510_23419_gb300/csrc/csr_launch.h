// csr_launch.h -- host/device interface of the p-bit update on general sparse
// instances (arXiv 2510.23419: the general graph of Eq. 1, update groups of
// Sec. 1.2.2 from a proper colouring with k >= 2 colours).
#pragma once

#include "pb_common.h"

namespace pb {

// Rows of the resident form (csr_res.cu): +-1 instances without fields, degree <= 15,
// at most kCsrResSpins padded positions (else npad = 0).  Every class starts on a multiple of 4
// positions; a word is 4 consecutive positions, arrays over words hold one entry per
// position in its bytes or 16-bit halves.
struct CsrResDevice {
    int32_t npad;            // padded positions (a multiple of 4); byte npad of the state stays zero
    int32_t regular;         // every spin has the same degree
    int32_t edges;
    const uint2* nbr;        // [slots][npad / 4] neighbour positions (npad: unused slot), lower classes first
    const uint32_t* sign;    // [slots][npad / 4] bytes 0xFF <=> J = -1
    const uint4* lowdeg;     // [npad / 4] bit planes (bytes 0xFF / 0) of the degree into lower classes
    const uint32_t* degoff;  // [npad / 4] bytes 4 (maxdeg - degree)
    const int32_t* cls;      // [n_colours][4]: first word, words, spins, slots into lower classes | kCsrResFlush |
                             // all slots << 16
    const int32_t* pos;      // [N] position of label p
    int32_t rounds;          // of a sweep: sum over the classes of ceil(words / kCsrResThreads)
    int32_t slot_rounds;     // the same, weighted with the class's slots
    int32_t slot_words;      // sum over the classes of words x slots
};

// Device copy of a general instance.  Spins carry labels: the classes are
// listed one after the other, each in ascending original index, and a spin's
// label is its position in that list, so class c is the label range
// cls_off[c] .. cls_off[c+1]-1 and label - cls_off[c] is the class rank (the
// Philox counter word 0).  Each undirected edge (u, v, J) is stored from both
// ends in compressed rows over the labels (+-1 rows: the J = +1 half-edges
// first, each part in edge order); fields and colours are per label.  States
// cross the interface in the original order (orig / pos translate).
struct CsrDevice {
    int32_t N, jtype, n_colours, maxdeg, has_h, hmax;
    const int32_t* rowptr;   // [N + 1] rows by label
    const int32_t* rowneg;   // PM1: [N] first half-edge of row i with J = -1 (J = +1 ones come first)
    const int32_t* col;      // [2E] neighbour of each half-edge
    const int8_t* J8;        // [2E] +-1 couplings (PM1)
    const float* Jf;         // [2E] real couplings (F32)
    const int8_t* h8;        // [N] or null (PM1)
    const float* hf;         // [N] or null (F32)
    const int32_t* cls_off;  // [n_colours + 1] first label of each class
    const int32_t* orig;     // [N] original index of label p
    const int32_t* pos;      // [N] label of original vertex i
    const int32_t* colour;   // [N] colour of label p
    // +-1 instances of degree <= kCsrEllSlots (else null): row p as kCsrEllSlots
    // labels (the J = +1 neighbours first), unused slots naming label N, whose
    // spin words are kept zero; ell_nd[p] = (J = +1 count) | degree << 8
    const int4* ell;         // [N][kCsrEllSlots / 4]
    const uint16_t* ell_nd;  // [N]
    CsrResDevice res;        // resident form
};

// Spin words: 4 replicas per uint32, one byte each, byte = 0 <=> m = +1,
// 1 <=> m = -1; state [N][Rw], Rw = ceil(R / 4), replica r in byte r % 4 of word r / 4.
struct CsrJob {
    CsrDevice g;
    uint32_t key0, key1;
    int32_t S, step, nF, fmin;
    int32_t s0;              // first sweep (0, or the sweep a resumed run continues from)
    const uint32_t* table;   // PM1: threshold windows of all levels, concatenated
    const int32_t* win;      // PM1: [levels][3] (lo, width, off)
    const float* betaf;      // F32: [levels]
    int32_t R, Rw;
    uint32_t* spins;         // [N][Rw] (+ one zero row, label N, for the padded rows)
    uint32_t* best;          // [N][Rw]
    int32_t nchunk;          // vertex chunks of the energy partials
    double* part;            // [nchunk][4 Rw] energy partials (PM1: 2E as exact integers)
    int32_t ndchunk;         // class chunks of the sweep's energy changes, over all classes
    const int32_t* dchunk_off;  // [n_colours + 1] first class chunk of each class
    double* dpart;           // F32: [ndchunk][4 Rw] energy change of each class chunk in the last sweep
    unsigned long long* dacc;  // PM1: [4 Rw] energy change of the sweep so far (int64 two's complement)
    double* E_best;          // [4 Rw]
    int32_t* best_sweep;     // [4 Rw]
    int32_t* hit_sweep;      // [4 Rw]
    uint8_t* improved;       // [4 Rw] + 1 "any" flag at [4 Rw]
    int32_t has_target;        // 0 none, 1 record the target sweep, 2 also stop there (see pbit.h)
    int32_t* stop;             // has_target == 2: [0] replicas that reached the target, [1] the sweep after
                               // which all had (-1 while running); later launches return at once
    double target;
    double* E_cur;             // [4 Rw] energy after the last sweep
    // parallel tempering (null temp: annealing with the schedule)
    uint8_t* temp;             // [4 Rw] temperature index of every slot (= replica)
    int32_t* slot_of;          // [M][C] slot holding temperature t of chain r
    int32_t M, C;              // temperatures, chains; slot g = k C + r starts at temperature k
    const float* xdb;          // [M-1] (beta_{t+1} - beta_t) log2 e, rounded to FP32 (real couplings)
    const uint32_t* xtab;      // +-1: exchange thresholds floor(exp(dbeta_t * (-d)) 2^32), d = 1, 2, ...
    const int32_t* xwin;       // +-1: [M-1][2] (length, offset) of pair t's thresholds in xtab
    unsigned long long* n_accept;  // [M-1] accepted exchanges per pair
};

constexpr int kCsrResThreads = 512;
constexpr int kCsrResSpins = 65528;  // 16-bit positions; two bytes of shared memory each
constexpr int kCsrResDegree = 15;
// A thread counts its unsatisfied bonds in kCsrResPlanes bit planes: at most 15 per word, so kCsrResWords words
// before the count leaves the registers.  Every class deals its words to the threads anew, so thread 0 has a word of
// each of up to 255 classes: classes after which the count must leave carry kCsrResFlush (the last one always).
// (Decided in the kernel from the class table, this cost 0.3 of 4.6 us per sweep on the L = 5 cube.)
constexpr int kCsrResPlanes = 9;
constexpr int kCsrResWords = ((1 << kCsrResPlanes) - 1) / kCsrResDegree;
constexpr int kCsrResFlush = 1 << 8;
constexpr int kCsrChunk = 64;  // vertices per energy chunk
constexpr int kCsrLanesQ = 32;  // class kernel: replica words per block
constexpr int kCsrLanesV = 8;   // class kernel: vertex lanes per block
constexpr int kCsrEllSlots = 8;  // padded rows for +-1 instances of degree <= 8
constexpr int kCsrMaxVpt = 16;  // class kernel: most class spins one thread takes in a launch

// Which form a run takes.  A resident CTA sweeps all spins of one quad (two, once the quads outnumber the SMs) alone,
// whatever the replicas; a class launch spreads them over the chip.  So large graphs with few replicas are
// the launches' and the rest the resident form's.  us per sweep as fitted to both forms (within 25%), timed on cubes of
// side 5 to 39 and on random circulants of 4 000 to 60 000 spins and degree 2 to 14 with 1 to 1024 replicas; resident /
// launches, e.g.: side 25, 4 replicas 20 / 34; side 31, 64 replicas 33 / 40; side 37, 64 replicas 52 / 45, 256
// replicas 56 / 67; 60 000 spins of degree 8, 64 replicas 86 / 69, 512 replicas 91 / 132.  The choice it makes is
// the faster form at all but six of the 140 points (those by at most 10%).
inline int csr_res_quads(int Rw, int sms) { return Rw > sms ? 2 : 1; }
inline double csr_res_us(const CsrResDevice& g, int Rw, int sms)
{
    const int q = csr_res_quads(Rw, sms), waves = ((Rw + q - 1) / q + sms - 1) / sms;
    const double sw = g.slot_words / (double)kCsrResThreads;
    return waves * (q == 1 ? 0.97 * g.rounds + 0.047 * g.slot_rounds + 0.094 * sw - 0.7
                           : 1.8 * g.rounds + 0.027 * g.slot_rounds + 0.133 * sw - 1.3);
}
inline double csr_launches_us(int n_colours, int N, double degree, int Rw)
{
    const int more = Rw > 16 ? 4 * Rw - 64 : 0;  // replicas past the first 64, which cost no more than one quad
    return 6.4 * n_colours + N * (3.8e-4 + 4.6e-6 * degree + (Rw == 1 ? 1.4e-4 : 0.0) + more * (1.9e-6 + 1.3e-7 * degree));
}
// Seconds of an anneal of S sweeps in either form; compute: the part of it that needs the whole chip's SMs (a resident
// CTA holds one SM for the run's length, the launches' fixed cost holds none).
inline double csr_seconds(const CsrResDevice& g, int n_colours, int N, double degree, int Rw, int S, int sms, bool resident,
                          double* compute)
{
    const double us = resident ? csr_res_us(g, Rw, sms) : csr_launches_us(n_colours, N, degree, Rw);
    const int q = csr_res_quads(Rw, sms), ctas = (Rw + q - 1) / q;
    if (compute) *compute = 1e-6 * S * (resident ? us * (ctas < sms ? (double)ctas / sms : 1.0) : us - 6.4 * n_colours);
    return 1e-6 * S * us;
}
// Resident form: the whole anneal (states, bests, target sweeps) of a run whose instance has
// resident rows, in one launch.
size_t csr_res_smem(int npad);
cudaError_t csr_launch_res(const CsrJob& job, int sms, cudaStream_t st);
cudaError_t csr_launch_init(const CsrJob& job, cudaStream_t st);
// Blocks (class chunks) of one class launch for a class of ncls spins: whole
// waves of resident blocks (SMs x blocks per SM of the kernel variant), at most
// kCsrMaxVpt spins per thread; a function of the device and the shapes only, so
// a run's energy partials are summed in the same order whatever runs beside it.
// -1 on a CUDA error.
int csr_class_blocks(int jtype, bool temp, int Rw, int ncls, int maxdeg, int hmax);
// Update of colour class c in sweep s (Eq. 2, Eq. 3) and its energy changes
// (nchunks = csr_class_blocks(...) of the class).
cudaError_t csr_launch_class(const CsrJob& job, int c, int nchunks, int s, cudaStream_t st);
// Energy partials of the state `m` ([N][Rw] words); exact FP64 per term when exact != 0.
cudaError_t csr_launch_energy(const CsrJob& job, const uint32_t* m, int exact, cudaStream_t st);
// Parallel tempering: exchange of temperatures between adjacent pairs of every
// chain after sweep s (pairs t = s mod 2, t + 2, ...).
cudaError_t csr_launch_exchange(const CsrJob& job, int s, cudaStream_t st);
// Running best after sweep s (init 1: the initial state, whose energy comes from
// csr_launch_energy, becomes the best; init 2: a resumed run's state, whose
// energy is set and whose given best is kept; init 0: later sweeps add the class
// launches' energy changes to the previous energy) and the improved flags.  The
// next sweep's class launches copy the flagged replicas' state into the best
// state as they read it; csr_launch_snapshot does so after the last sweep.
cudaError_t csr_launch_sweep_end(const CsrJob& job, int s, int init, cudaStream_t st);
cudaError_t csr_launch_snapshot(const CsrJob& job, cudaStream_t st);
// States [R][N] int8 +-1 and energies (from the partials of the same state) of `m`.
cudaError_t csr_launch_readout(const CsrJob& job, const uint32_t* m, int8_t* out_pm, double* out_E, cudaStream_t st);
// Fields F[r][i] = sum_j J_ij m_j + h_i of given +-1 states [R][N] (written as [R][N] float).
cudaError_t csr_launch_fields(const CsrJob& job, const int8_t* states, float* out, cudaStream_t st);

}  // namespace pb
