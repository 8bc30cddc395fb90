// Diagonal-frame path of the on-chip instances (n <= 16): tables shared by the host planner
// (qng_frames_plan.cu), the host API and the kernels (qng_frames.cu).
//
// Every gate of this library is diagonal in some local Clifford frame: R_X is diagonal after a
// Hadamard on its qubit, R_Y after H S^dag, a (controlled) Pauli-string rotation after one such
// change per X or Y factor, CZ and Z as they stand. The planner therefore writes the circuit as
//     psi = tau_R D_R tau_{R-1} ... D_1 tau_0 |0...0>
// on a vector kept in a running local frame: a run D_r is a diagonal unitary (all of its rotations
// and sign gates at once), and a transition tau_r is Hadamards on some qubits and linear index
// permutations (CNOT networks). Pauli and phase gates, and the Hadamards of the circuit itself,
// only change the frame and cost nothing.
//
// What that gives the recurrence of Algorithm 1: all parameters of a run commute, so with Psi_r
// the vector after run r and b the column there, every inner product of the run is read off the one
// product p_m = conj(Psi_r[m]) b[m], <Psi|K_i|b> = sum_m k_i(m) p_m with k_i(m) in {0, +1, -1}, and
// one complex factor per amplitude takes b through all of the run's adjoint gates. A column costs two
// multiplications per amplitude and run; everything else is additions.
#pragma once

#include <cstdint>
#include <vector>

#include "qng_internal.h"

namespace qng {
namespace frames {

constexpr int kRegBitsMax = 4;  // a thread holds 2^kb amplitudes, kb index bits at a time (kb = 3 or 4)

// A transition of k Hadamards (unnormalised, sqrt 2 times an isometry each) and the run after it. Fixed point
// halves floor(k / 2) times inside the transition and leaves the odd sqrt 1/2 to the run's factor. float32 has the
// range to leave all of 2^(-k/2) to the factor, which costs nothing, but only to a bound: the table's products are
// multiples of 2^-61, so 2^-24 relative needs 2^(-k/2) well above 2^-37, and circuits of H and CNOT alone put any
// number of Hadamards into one transition. Longer transitions are halved inside as in fixed point.
constexpr int kTableHalf = 48;
inline int table_half(int k, bool fixed) { return fixed || k > kTableHalf ? (k & 1) : k; }

// A diagonal factor of a run. With par = parity(m & z) and on = ((m & ctrl) == cval):
//   kind 0 (rotation):  on ? cos(theta/2) - i lam sin(theta/2) : 1,  lam = sgn (-1)^par
//   kind 1 (sign gate): on ? lam : 1
//   kind 2 (S^dag):     par ? -i : 1
struct Member {
    int32_t kind;
    int32_t param;
    uint32_t z, ctrl, cval;
    int32_t sgn;
};

// A parameter of a run as the column kernel reads its inner product off the thread's 16 products:
// index bits split into the thread's own (zreg, sign16, incl16) and the others (z, ctrl, cval over
// the thread index).
struct Ip {
    uint16_t z, ctrl, cval;
    uint16_t zreg;     // parity mask over the thread's bits
    uint16_t incl16;   // the products that the controls include (all: no control)
    uint16_t sign16;   // the products whose sign flips
    int16_t sgn;
    uint16_t all16;    // every product of a thread
};

struct Run {
    int32_t mem_begin, mem_count;  // Member table
    int32_t ip_begin, ip_count;    // Ip table; parameters ip_first .. ip_first + ip_count - 1 in order
    int32_t ip_first;
    int32_t low;                   // lowest of the index bits a thread holds at this run
    int32_t khalf;                 // Hadamards since the run before (each is sqrt 2 times an isometry) that its
                                   // factor normalises; the others are halved away inside the transition
    int32_t simple;                // every parameter: no control, at most one of the thread's bits
};

// One step of the vector: exchange into arrangement `low` (through permutation perm >= 0), Hadamards
// on the thread's bits hm followed by `shift` halvings, then run `run` (>= 0).
struct UOp {
    int16_t low;    // -1: no exchange
    int16_t hm;
    int16_t shift;  // halvings after the Hadamards (float32: of long transitions only)
    int16_t rshift; // halvings right before the run (streaming, fixed point)
    int32_t perm;   // -1: none
    int32_t run;
};

struct Perm {
    uint32_t img[16];  // gather: new[m] = old[xor of img[b] over the bits b of m]
};

// Per-instance descriptor.
struct Inst {
    int32_t n, nE;            // qubits; index bits (at least kb)
    int32_t R, P;
    int32_t run_off;          // first Run
    int32_t fwd_off, fwd_cnt; // forward UOps
    int32_t bwd_off, bwd_cnt; // walk UOps (from the last run down to run 0)
    int32_t start0, end_low;  // arrangement before the first forward step / after the last
    int32_t cl;               // log2 CTAs per vector
    int32_t term_off, nterms; // Hamiltonian terms in the final frame
    int32_t eexp;             // <E> is summed in fixed point, units of 2^(eexp - 60)
    int32_t hchunks;          // CTAs of the H psi kernel for this instance
    int32_t ip_off;           // first Ip
    int32_t pad;
    int64_t a_off, d_off;     // checkpoints / factor tables, amplitude units (R << nE each)
    int64_t v_off;            // final vector and eta (1 << nE each)
    int64_t param_off, metric_off;
};

// A work item of the column kernel: ncol columns (cols[list..]) of run `run`, or the gradient column
// (ncol = 0).
struct Item {
    int32_t inst, run;
    int32_t list, ncol;
    int32_t entry;      // first step of the walk, index into the instance's walk UOps
    int32_t nip, nruns;  // parameters and runs the walk meets: the first ones, up to its own run
    int32_t pad;
};

struct TabItem {        // 512 entries of one run's factor table
    int32_t inst, run, first;
};

struct HItem {          // a CTA of the H psi kernel
    int32_t inst, chunk;
};

// One launch class: instances whose vectors use one CTA shape.
struct Class {
    int cl = 0;
    int kb = 4;                          // index bits per thread
    int threads = 0;                     // CTA size of the column kernel
    int fwd_threads = 0;                 // CTA size of the forward sweep
    int max_P = 0;
    bool general = false;                // some run is not simple
    int first_inst = 0, num_inst = 0;    // into order
    int first_item = 0, num_item = 0;    // metric and gradient columns, longest first
    int first_met = 0, num_met = 0;
    int first_grad = 0, num_grad = 0;
    int first_h = 0, num_h = 0;
    size_t smem_fwd = 0, smem_col = 0, smem_col_im = 0;
};

// Device pointers of the path (the workspace's tables and arrays).
struct FWork {
    bool chain = false;  // launches after the tables' follow on as a chain (launch_next)
    const Inst *inst;
    const Run *run;
    const Member *member;
    const Ip *ip;
    const UOp *uop;
    const Perm *perm;
    const DevTerm *term;
    const Item *item;
    const int32_t *cols;
    const int32_t *order;     // instances by class
    const TabItem *tab;
    const HItem *hitem;
    int32_t *bad_run;         // per run: an angle is not finite
    int32_t *bad;             // per instance
    unsigned long long *eacc; // per instance: <E> and |H psi|^2 in fixed point, the count of finished
    int32_t *etaexp;          //   CTAs; |H psi| <= 2^etaexp
    void *a, *d, *v, *eta;
    const double *theta;
    int32_t *status;
    double *pctrl, *sigma, *L, *Lim, *gradraw, *energy;
};

constexpr int kTabThreads = 128, kTabBits = 2, kTabAmps = 1 << kTabBits;
constexpr int kHThreads = 64, kHSplit = 4;  // H psi: threads per CTA, threads per amplitude

// The column kernel of that form takes runs that are not simple.
inline bool takes_general(int precision, int kb) { return precision != QNG_C128 || kb == 3; }
cudaError_t prepare(int precision, int kb, size_t smem_fwd, size_t smem_col, size_t smem_col_im);
cudaError_t launch_tables(const FWork &w, int ntab, int kb, int precision, cudaStream_t st);
cudaError_t launch_forward(const FWork &w, const Class &c, int precision, cudaStream_t st);
cudaError_t launch_hpsi(const FWork &w, int first, int num, int precision, cudaStream_t st);
cudaError_t launch_columns(const FWork &w, const Class &c, int precision, int first, int num, int metric_im,
                           cudaStream_t st);

struct Program {  // one instance, host side
    int n = 0, nE = 4, kb = 4;
    std::vector<Run> runs;
    std::vector<Member> members;
    std::vector<Ip> ips;
    std::vector<UOp> fwd, bwd;
    std::vector<int32_t> bwd_entry;  // index of run r's step in bwd
    std::vector<Perm> perms;
    std::vector<DevTerm> terms;
    int start0 = 0, end_low = 0;
};

// Build the program of one circuit on index bits [0, nE), kb of them per thread and the top cl
// distributed over CTAs; fixed: for fixed-point vectors, else for float32 ones.
// Indices in the program (members, perms) are relative to its own tables.
void build_program(const std::vector<qng_gate> &gates, const std::vector<uint64_t> &masks,
                   const std::vector<qng_pauli> &terms, int n, int kb, int cl, bool fixed, Program &out);

// ------------------------------------------------------------------------------------------
// Streaming: one instance whose vectors lie in global memory. A pass loads tiles of 2^tb amplitudes (the
// low bits and a window of tb - low consecutive others), runs its steps on each and stores them.
// A run's factor on amplitude m is lo[m mod 2^hl] hi[m >> hl] (-1)^parity(m & mask[m >> hl]).
struct SIp {
    uint32_t zall, z;  // the qubit's bit; the same unless a warp's own sums resolve it
    int16_t sgn;
    int16_t src;       // which warp sum of the products: 0 all, 1 + j signed by the thread's bit j,
                       // 8 + j signed by lane bit j
};

struct SPerm {         // gather within a tile: local source index
    uint32_t limg[16]; // image of each local bit
    uint32_t oimg[32]; // what a set bit outside the tile adds
};

struct SPass {
    int32_t s;         // first bit of the window
    int32_t load_low;  // arrangement the tile is loaded in
    int32_t op_begin, nops;
    int32_t run0;      // its first run, -1 without one
    int32_t shift;     // halvings of the fixed-point vector when it is stored
};

struct SEntry {        // where the walk's columns of a run start
    int32_t pass, op, low, pad;
};

struct SCol {          // a column: its parameter (P: the gradient column) and its run (R: the gradient's)
    int32_t col, run;
};

struct StreamProgram {
    int n = 0, kb = 4, tb = 12, low = 2, hl = 0;
    std::vector<Run> runs;
    std::vector<Member> members;
    std::vector<SIp> ips;
    std::vector<SPerm> perms;
    std::vector<UOp> ops;
    std::vector<SPass> fwd, bwd;
    std::vector<SEntry> entry;
    std::vector<DevTerm> terms;
};

// Tile bits for n qubits, and index bits per thread for that tile: 64 KiB for large vectors, smaller tiles where
// those would leave SMs idle (20 qubits complex64, energy and backward: 548 -> 470 us).
inline int stream_tile_bits(int precision, int n) {
    if (precision == QNG_C128) return n <= 19 ? 11 : 12;
    return n <= 19 ? 11 : (n == 20 ? 12 : 13);
}
inline int stream_reg_bits(int tb) { return tb == 13 ? 5 : 4; }
void build_stream(const std::vector<qng_gate> &gates, const std::vector<qng_pauli> &terms, int n, int kb, int tb, int low,
                  bool fixed, StreamProgram &out);

struct SWork {
    bool chain = false;  // as FWork's
    const Run *run;
    const Member *member;
    const SIp *ip;
    const SPerm *perm;
    const UOp *uop;
    const SEntry *entry;
    const SCol *col;
    const DevTerm *term;
    void *lo, *hi;            // factor tables, 2^hl and 2^(n-hl) entries per run
    uint32_t *mask;           // 2^(n-hl) per run
    void *a;                  // checkpoints, natural order, 2^n per run
    void *b;                  // column slots, 2^n each
    long long *acc;           // (P x P) sums of the metric, twice that with Im, in units of 2^-62
    long long *sacc, *gacc;   // <sigma_j>, units of 2^-62; the gradient, units of 2^(etaexp - 62)
    unsigned long long *eacc; // as in FWork
    int32_t *etaexp;
    const double *theta;
    int32_t *status, *bad;
    double *pctrl, *sigma, *L, *Lim, *gradraw, *energy;
    int32_t n, P, R, tb, low, hl, nterms, eexp, hblocks;
};

cudaError_t prepare_stream(int precision, int tb);
cudaError_t launch_stream_tables(const SWork &w, int precision, cudaStream_t st);
cudaError_t launch_stream_forward(const SWork &w, const SPass &p, int first, int slot, int precision, cudaStream_t st);
// Pass p of the walk over ncol columns col[col0 ..], column k in slot k.
cudaError_t launch_stream_walk(const SWork &w, const SPass &p, int pass, int col0, int ncol, int store, int precision,
                               int metric_im, cudaStream_t st);
// H psi: slot `in` -> slot `out`, and <E>.
cudaError_t launch_stream_hpsi(const SWork &w, int in, int out, int precision, cudaStream_t st);
// Sums to float64: what = 1 metric, 2 gradient (bits), 4 with Im.
cudaError_t launch_stream_finish(const SWork &w, int what, cudaStream_t st);

}  // namespace frames
}  // namespace qng
