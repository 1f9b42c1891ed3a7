// launch.h -- host-side launch wrappers of the library's kernels.
#pragma once

#include <cstdint>
#include <mutex>

#include <cuda_runtime.h>

#include "../../include/stab.h"
#include "stab_internal.h"

namespace stab {

constexpr int kMaxResidentQubits = 6;   // two buffers of 4^6 doubles = 64 KiB of shared memory
constexpr int kMaxResidentAdjoint = 6;  // four buffers of 4^6 doubles = 128 KiB
constexpr int kRotPerGradPass = 8;      // rotations per P_WIRE pass in gradient plans

// Whether a barrier's counter, which counts arrivals mod 2^32, has come to
// `want`: the two are never 2^31 apart (a CTA is at most one meeting ahead), so
// the sign of their difference tells, also where the count wraps (a chain of 600
// CTAs: after 7 million steps, 14 million gates).
__host__ __device__ inline bool arrivals_reached(uint32_t seen, uint32_t want) {
    return (int32_t)(seen - want) >= 0;
}

// A kernel's dynamic shared-memory limit belongs to the function, not to a
// launch: every thread and context of the process sees the same value.  It is
// only ever raised here, under a lock, so that one thread lowering it cannot
// fail another thread's larger launch.  One SmemLimit per kernel.
struct SmemLimit {
    std::mutex mu;
    size_t set[64] = {};   // per device: the limit so far (0: not asked yet)
};

template <typename K>
cudaError_t raise_smem_limit(K kernel, size_t smem, SmemLimit &lim) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    std::lock_guard<std::mutex> g(lim.mu);
    const bool tracked = dev >= 0 && dev < 64;
    if (!tracked || lim.set[dev] == 0) {
        // the default: what 48 KiB hold beside the kernel's static shared memory
        cudaFuncAttributes fa{};
        e = cudaFuncGetAttributes(&fa, kernel);
        if (e != cudaSuccess) return e;
        if (tracked) lim.set[dev] = (size_t)fa.maxDynamicSharedSizeBytes;
        if ((size_t)fa.maxDynamicSharedSizeBytes >= smem) return cudaSuccess;
    }
    if (tracked && lim.set[dev] >= smem) return cudaSuccess;
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e == cudaSuccess && tracked) lim.set[dev] = smem;
    return e;
}

struct StreamArgs {
    const Rec *stream;       // instruction stream (device), n_chunks x kChunkRecs records
    int32_t n_chunks;
    int32_t init;            // InitMode
    const DevTerm *terms;    // INIT_TERMS
    int32_t n_terms;
    int32_t n_vec;           // vectors (blocks); block b starts as Z_b for INIT_GENERATOR
    const double *in;        // INIT_LOAD: block b reads in + b * 4^n
    double *out;             // final vector of block b at out + b * 4^n (may be null)
    double *xfree_out;       // block b: sum of its x-free coefficients (may be null)
    int32_t *status;         // set to a nonzero code when a bounded wait gives up
};

// Split resident adjoint (two CTAs, two launches; see k_adjoint_split).
struct AdjointSplitArgs {
    const Rec *stream[2];    // phase 0: forward [0, cut), backward [cut, P); phase 1: backward
                             // [0, cut), forward [cut, P) -- all of the gradient plan
    int32_t n_chunks[2];
    int32_t phase;           // 0 or 1
    const DevTerm *terms;    // phase 0, CTA 1: O
    int32_t n_terms;
    double *rmid, *lmid;     // rho and lambda at the cut: phase 0 writes, phase 1 reads
    double *grad_rot;        // phase 1: one entry per rotation ordinal
    double *partials;        // phase 1, optional: per-thread dots [rotation ordinal][threads]
                             // (summed afterwards by k_reduce_partials); null: each pass
                             // reduces its rotations' dots over the CTA into grad_rot
    double *expect_out;      // phase 1: <O>
    int32_t *status;
};

struct AdjointStreamArgs {
    const Rec *fwd;          // forward stream of the gradient plan
    const Rec *bwd;          // backward stream of the gradient plan
    int32_t n_fwd_chunks;
    int32_t n_bwd_chunks;
    const DevTerm *terms;
    int32_t n_terms;
    double *grad_rot;        // one entry per rotation ordinal
    double *partials;        // optional, as in AdjointSplitArgs
    double *expect_out;      // <O>
    int32_t *status;
};
// Threads of the resident adjoint kernels' CTA at n qubits (the row length
// of their per-thread partials).
int resident_adjoint_threads(int n);
// Bytes of the resident adjoint's per-thread dot shares for n_rot rotations
// at n qubits, or 0 where the sweeps reduce each pass's dots themselves.
size_t resident_partial_bytes(int n, int64_t n_rot);

// One unit of the persistent batch kernel: one vector of one circuit.
struct BatchUnit {             // 64 bytes
    const Rec *stream;         // the circuit's forward (generators) or backward (<O>) stream
    int32_t n_chunks;
    int8_t n;                  // qubits (1 .. 8)
    int8_t init;               // INIT_GENERATOR or INIT_TERMS
    int16_t gen;               // generator index for INIT_GENERATOR
    const DevTerm *terms;      // INIT_TERMS
    int32_t n_terms;
    int32_t pad;
    double *out;               // final vector (may be null)
    double *xfree_out;         // <O> (may be null)
    int64_t cost;              // host-side ordering key
    int64_t reserved;
};
static_assert(sizeof(BatchUnit) == 64, "BatchUnit layout");

struct BatchArgs {
    const BatchUnit *units;
    int32_t n_units;
    int32_t *counter;          // next unit to take (zeroed before the launch)
    int32_t *status;
    double *slab;              // per-CTA global vectors for n > kMaxResidentQubits (may be null)
    size_t slab_doubles;       // doubles per CTA slab
    int32_t max_chunks;        // > 0: each unit runs only its first max_chunks chunks (timing
                               // samples; the outputs are then partial); 0: whole streams
    int32_t smem_n;            // units of n <= smem_n keep their vectors in shared memory, the
                               // others in the slab (0: kMaxResidentQubits)
};

// One slice of one unit of the serving iteration kernel (k_serve): a vector
// (or an adjoint pair) of one admitted request carried through a contiguous
// range of chunks of one of its instruction streams.  The request's state
// vectors live in its own device memory between launches; a slice starts
// from them (or from its initial value) and writes them back.
enum ServeKind : int8_t {
    SV_VEC = 0,        // one vector through a stream (forward or backward)
    SV_PAIR_BWD = 1,   // (lambda, rho) through a backward gradient stream, dots then ops
    SV_PAIR_FWD = 2,   // (lambda, rho) through a forward gradient stream, ops then dots
};

struct ServeUnit {             // 80 bytes
    const Rec *stream;         // first chunk of the slice
    int32_t n_chunks;          // chunks of the slice
    int8_t n;                  // qubits (1 .. kServeMaxQubits)
    int8_t kind;               // ServeKind
    int8_t init;               // INIT_RHO0 / INIT_TERMS (first slice of a vector), INIT_LOAD
    int8_t flags;              // SF_LAST | SF_ROWS
    const DevTerm *terms;      // INIT_TERMS
    int32_t n_terms;
    int32_t pad;
    const double *src;         // INIT_LOAD: the vector (SV_VEC) or lambda (pairs)
    const double *src2;        // INIT_LOAD, pairs: rho
    double *state;             // persistent state: SV_VEC [v | spare] (2 x 4^n doubles),
                               // pairs [lambda | rho | spare | spare] (4 x 4^n)
    double *grad_rot;          // pairs: the dots, by rotation ordinal
    double *xfree_out;         // SF_LAST: x-free sum of the vector (SV_VEC) or of lambda
    int64_t reserved;
};
static_assert(sizeof(ServeUnit) == 80, "ServeUnit layout");

constexpr int kServeMaxQubits = 8;
constexpr int SF_LAST = 1;     // the slice ends the unit's stream
constexpr int SF_ROWS = 2;     // SV_VEC at n <= 4: every wire pass one 3x3 map (lane quads)

struct ServeArgs {
    const ServeUnit *units;
    int32_t n_units;
    int32_t *counter;          // next unit to take (zeroed before the launch)
    int32_t *status;
    int32_t smem_buf;          // bytes of shared memory for state buffers: a unit whose
                               // buffers (2 or 4 x 4^n doubles) fit runs in shared memory
    int64_t *unit_cycles;      // per unit: SM clock cycles its slice took (may be null)
};

size_t serve_smem_bytes(int smem_buf);
cudaError_t serve_occupancy(size_t smem, int *ctas_per_sm);
cudaError_t launch_serve(const ServeArgs &a, int grid, size_t smem, cudaStream_t s);

size_t batch_smem_bytes(int max_n_in_smem);
int batch_threads();
cudaError_t batch_occupancy(size_t smem, int *ctas_per_sm);
cudaError_t launch_batch(const BatchArgs &a, int grid, size_t smem, cudaStream_t s);

}  // namespace stab

typedef struct stab_ctx stab_ctx;
struct stab_gate;

namespace stab {

// The context's main stream (work queued by the asynchronous entry points is
// complete once this stream is).
cudaStream_t ctx_stream(stab_ctx *ctx);

// Device memory the context's gradients may take for stored sweeps (0: none, the
// pair sweep's fixed number of vectors; else a failed allocation of them is
// STAB_E_NOMEM instead of the pair sweep), and a bound on what a circuit's take (0:
// more than any context takes, so the pair sweep runs).
void ctx_checkpoint_limit(stab_ctx *ctx, size_t bytes);
struct PlanCount;
size_t checkpoint_bound(int n, const PlanCount &k);
// Whether streamed sweeps may run as chains of tile steps, and a bound on the
// tables and steps that these take (<O>, or a gradient from stored sweeps).
void ctx_allow_chains(stab_ctx *ctx, bool on);
size_t chain_bound(int n, const PlanCount &k, bool grad);
// Bounds on what a streamed plan of the gates has: blocks of wire passes, Clifford
// passes, ranges that its wire passes are planned in.
struct PlanCount {
    size_t blocks = 0, cliffs = 0, ranges = 1;
    PlanCount(const struct ::stab_gate *gates, int64_t m);
};
// Hands back the memory of stored sweeps, then that of chains' tables, when the
// context holds more than `keep` of it (no call in flight); returns what it still
// holds.
size_t ctx_trim(stab_ctx *ctx, size_t keep);

// Density matrix from the forward-evolved coefficients of 2^n |0><0|:
// rho (device, 2 x 4^n doubles, interleaved complex, row-major).
cudaError_t launch_decode_rho(const double *r, int n, double *rho, cudaStream_t st);

// Kernel that waits on a barrier nothing completes (bounded), for the self-test.
cudaError_t launch_bounded_wait(int64_t polls, int32_t *status, cudaStream_t st);

// Records the CUDA error behind a STAB_E_CUDA status (stab_last_cuda_error).
void record_cuda_error(cudaError_t e);

// Whether runs of up to max_count gates are composed (or walked) by a warp each
// instead of a thread each: a thread takes about 2.3 us a gate (a sincos and a
// product, one after another), a warp about 6 us and, beyond the GPU's warps, 12
// ns a run (five shuffled products).
inline bool warp_per_run(int64_t n_runs, int max_count) {
    return max_count > 32 || (max_count > 4 && 2.3 * max_count > 6.0 + 0.012 * (double)n_runs);
}
// Composed 3x3 map of every run (maps[i].m), from the angle array on the
// device (max_count: the longest run).
cudaError_t launch_compose_maps(DevMap3 *maps, int n_maps, int max_count,
                                const int32_t *map_gate_idx, const RawGate *gates,
                                const double *thetas, cudaStream_t st);
int max_map_count(const DevMap3 *maps, size_t n_maps);   // host: the longest run

// Encode: the composed maps, then the lifting coefficients of every rotation op.
cudaError_t launch_encode(DevOp *ops, int n_ops, DevMap3 *maps, int n_maps, int max_count,
                          const int32_t *map_gate_idx, const RawGate *gates, const double *thetas,
                          cudaStream_t st);

// Stream encode: shear coefficients of the R_ROT records and the matrices of
// the R_MAP3 records listed in enc (indices into recs), copied from maps
// (composed before by launch_compose_maps).
cudaError_t launch_encode_stream(Rec *recs, const int32_t *enc, int n_enc, const DevMap3 *maps,
                                 const double *thetas, cudaStream_t st);

// Shared-memory-resident propagation, one CTA per vector (n <= kMaxResidentQubits).
cudaError_t launch_resident_stream(int n, const StreamArgs &a, cudaStream_t st);
int resident_lanes_per_group(int n);

// Streamed passes over n_vec vectors of 4^n doubles in global memory.
cudaError_t launch_fill(double *vec, int n, int n_vec, int init, const DevTerm *terms,
                        int n_terms, cudaStream_t st);
cudaError_t launch_stream_wire(double *vec, int n, int n_vec, const DevPass &p, const DevOp *ops,
                               const DevMap3 *maps, int inverse, cudaStream_t st);
cudaError_t launch_stream_cliff(const double *src, double *dst, int n, int n_vec,
                                const DevPass &p, const DevOp *ops, int inverse, cudaStream_t st);
cudaError_t launch_xfree_sum(const double *vec, int n, int n_vec, double *out, cudaStream_t st);
// *out = <a, b> over the 4^n entries, fixed order; partial: 256 doubles of scratch.
cudaError_t launch_dot(const double *a, const double *b, int n, double *partial, double *out,
                       cudaStream_t st);
// dst = a Clifford run as a signed gather (n <= 12).
cudaError_t launch_stream_pull(const double *src, double *dst, int n, int n_vec,
                               const DevPull *pull, cudaStream_t st);

// Several consecutive wire passes on at most kTileWires wires fused into one
// streamed launch: each CTA loads a tile (all 4^|Q| slots of the wires Q times
// some of the lowest other index bits) into shared memory, applies the passes
// in order and writes it back.
constexpr int kTileWires = 5;
constexpr int kTileMaxPasses = 8;
constexpr int kTileMaxBits = 10;        // 1024 doubles = 8 KiB of shared memory
constexpr int kTileThreads = (1 << kTileMaxBits) / 4;   // one group of four entries each

struct BitRuns {                        // deposit of a packed integer into index bits
    uint8_t n;
    uint8_t src[16], dst[16], len[16];
};

// Wires of a tile group: as few groups of about equal size as n wires need.
constexpr int tile_wires(int n) {
    const int groups = (n + kTileWires - 1) / kTileWires;
    return (n + groups - 1) / groups;
}

struct TileGroup {
    int32_t n_pass;
    int32_t tile_bits;                  // log2 entries per tile
    int32_t rest_bits;                  // 2n - tile_bits: log2 tiles per vector
    int32_t inverse;
    uint8_t lz[kTileMaxPasses], lx[kTileMaxPasses];   // tile-local bits of each pass's wire
    uint16_t n_ops[kTileMaxPasses];
    uint8_t n_rot[kTileMaxPasses];      // rotations of each pass (adjoint groups)
    uint32_t first[kTileMaxPasses];
    uint32_t map[kTileMaxPasses];       // each pass's composed map (k_stream_tile)
    BitRuns tile_runs;                  // local entry -> global index bits
    BitRuns rest_runs;                  // tile id -> global index bits
    // A Clifford gather folded into the tile loads (the Clifford pass that
    // precedes the group); null: plain loads.
    const DevPull *pull;
};

// src == dst, or (always with a folded Clifford gather) a different buffer.  ops
// null: the passes as composed maps (maps[tg.map[j]]); else as their ops (maps:
// the plan's long runs).
constexpr int kTileStagedOps = 96;      // ops of a group staged in shared memory (3 KiB)
cudaError_t launch_stream_tile(const double *src, double *dst, int n, int n_vec,
                               const TileGroup &tg, const DevMap3 *maps, const DevOp *ops,
                               cudaStream_t st);

// Whole sequences of tile steps in one cooperative launch: independent chains
// of steps, each a number of CTAs that meet at a barrier after every step.  A
// step gathers a tile, applies its passes and stores it.  Where each thread
// reads and writes is tabulated per shape (tile geometry, the wire whose groups
// the threads hold, the Clifford gather read through), so the chain only looks
// it up: entry k = 0 .. 3 (I, Z, X, Y) of thread t's group in tile m is at index
// tiles[4 m + k].x + threads[t].x, its source the xor of both tables' .y
// (pulled shapes; see DevPull for the sign).
struct ChainShape {
    BitRuns tile_runs, rest_runs;
    int32_t tile_bits, rest_bits;
    int32_t lz, lx, wire;               // the wire: tile-local bits, qubit
    int32_t pad;
    const DevPull *pull;                // null: entries are read in place
    uint2 *threads;                     // (offset, source | Q << 31) per thread
    uint4 *tiles;                       // (index, source | Q << 31, cross bits, 0) per entry
};
cudaError_t launch_chain_tables(const ChainShape *shapes, int n_shapes, int n, cudaStream_t st);

struct ChainStep {                      // 128 bytes
    const double *src;
    double *dst;
    const uint2 *in_threads, *out_threads;   // shapes of the first and the last pass's wire
    const uint4 *tiles;                 // of the first pass's shape
    const DevPull *pull;                // of that shape
    int32_t n_pass, inverse, rest_bits, pad;
    uint32_t out_k[4];                  // index bits of the last pass's wire for I, Z, X, Y
    uint8_t lz[kTileMaxPasses], lx[kTileMaxPasses];
    uint32_t map[kTileMaxPasses];
};
static_assert(sizeof(ChainStep) == 128, "ChainStep layout");
struct ChainDesc {                      // one chain, 64 bytes
    const ChainStep *steps;             // device
    const DevMap3 *maps;
    uint32_t *arrived;                  // its counter (128 bytes of its own), zero before the launch
    int32_t n_steps, n, n_vec;
    int32_t cta0, ctas;                 // its CTAs: [cta0, cta0 + ctas)
    int32_t pad[5];
};
static_assert(sizeof(ChainDesc) == 64, "ChainDesc layout");
struct ChainArgs {
    const ChainDesc *chains;            // device
    int32_t n_chains, grid, tile_bits;  // tiles of 2^tile_bits entries in every chain
    bool alone;                         // every chain one CTA, one vector, one tile
    int32_t *status;
};
constexpr int kChainMinN = 5;           // tiles of at least 2^9 entries
// CTAs of `threads` threads that fit on the device at once (0 on an error).
int chain_max_ctas(int threads);
cudaError_t launch_stream_chain(const ChainArgs &a, cudaStream_t st);

// The c of up to kTileWires wire runs of one block of wire passes, from rho and
// lambda at the block's end (lambda read through `pull` unless null).
struct DotJob {
    const double *rho, *lam;
    const DevPull *pull;
    int32_t n_wires;
    int32_t tile_bits, rest_bits;
    int32_t run[kTileWires];
    uint8_t lz[kTileWires], lx[kTileWires];   // tile-local bits of the wires
    BitRuns tile_runs, rest_runs;
};
// dots[(3 run + s) chunks + chunk], a CTA per job and chunk of its tiles.
cudaError_t launch_grad_dots(const DotJob *jobs, int n_jobs, int n, int chunks, double *dots,
                             cudaStream_t st);

// Adjoint gradient, shared-memory resident (n <= kMaxResidentAdjoint).
cudaError_t launch_adjoint_split(int n, const AdjointSplitArgs &a, cudaStream_t s);
cudaError_t launch_adjoint_stream(int n, const AdjointStreamArgs &a, cudaStream_t st);

// Streamed adjoint pieces.
int adjoint_stream_blocks(int n);
// One wire pass of the adjoint on (lambda, rho): backward (forward = 0: the
// dot at the post-gate pair, then the inverse gate) or forward (the gate, then
// the dot); partials[gate][block], adjoint_stream_blocks(n) blocks.
cudaError_t launch_adjoint_wire(double *lam, double *rho, int n, const DevPass &p,
                                const DevOp *ops, double *partials, int forward,
                                cudaStream_t st);
// Tile-fused reverse sweep on the contiguous pair (lambda, rho) for n <=
// kAdjTileMaxN: tiles of 2^kAdjTileBits entries, one per CTA and one group per
// thread, grid = adjoint_stream_blocks(n); partials[gate][block] as
// launch_adjoint_wire.
constexpr int kAdjTileMaxN = 8;
constexpr int kAdjTileBits = 9;
constexpr int kAdjTileWires = 4;
size_t adjoint_tile_smem(int tile_bits, int n_rot);   // n_rot: rotations of the group
cudaError_t launch_adjoint_tile(const double *src_pair, double *dst_pair, int n,
                                const TileGroup &tg, const DevOp *ops, double *partials,
                                cudaStream_t st);
cudaError_t launch_reduce_partials(const double *partials, int n_rot, int n_blocks,
                                   double *grad_rot, cudaStream_t st);
cudaError_t launch_gather_grads(const double *grad_rot, const int32_t *param_ptr,
                                const int32_t *param_rot, int n_params, double *grads,
                                cudaStream_t st);

// ---------------------------------------------------------------- segment unitaries (k_unitary.cu)

// 2 x 2 maps of the plan's wire runs from the angles (max_count: the longest run).
cudaError_t launch_uni_maps(const UniRun *runs, int n_runs, int max_count, const RawGate *gates,
                            const double *thetas, UniMap *maps, cudaStream_t st);

struct UniArgs {
    const UniOp *ops;
    const UniMap *maps;
    const UniSeg *segs;
    const UniPart *parts;
    int32_t n_segs;
    double2 *nodes;          // node matrices, 4^n complex entries each, column-major
    int32_t *node_parity;    // per node: U is kept times sqrt(2)^parity
    int32_t *node_count;     // per node: arrivals of its children (zero between launches)
};
// Every segment's unitary and the trees' inner nodes up to each part's root,
// one CTA per segment.
cudaError_t launch_uni_segments(int n, const UniArgs &a, cudaStream_t st);
// The parts' unitaries in plan order (at most kUniMaxParts).
constexpr int kUniMaxParts = 3;
struct UniRoots {
    const double2 *nodes;
    const int32_t *node_parity;
    int32_t n;
    int32_t root[kUniMaxParts];
};
// out[k] = the Pauli coefficients of U Z_k U^dagger, k < n, U the product of
// the roots, one CTA per generator.
cudaError_t launch_uni_images(int n, const UniRoots &r, double *out, cudaStream_t st);
// out = roots 1 times 0.
cudaError_t launch_uni_merge(int n, const UniRoots &r, double2 *out, int32_t *parity,
                             cudaStream_t st);
// psi = U |0>: *expect = <psi|O|psi> (may be null), r_out (may be null) = the
// coefficients of 2^n |psi><psi|; psi and phi (may be null): the states and
// the cotangents at the parts' boundaries, (r.n + 1) x 2^n entries each.
cudaError_t launch_uni_states(int n, const UniRoots &r, const DevTerm *terms, int n_terms,
                              double *expect, double2 *psi, double2 *phi, double *r_out,
                              cudaStream_t st);
// The three numbers c of every wire run at its end, as 2^n shares:
// dots[(3 run + s) 2^n + row] (see k_unitary.cu).
cudaError_t launch_uni_grad(int n, const UniArgs &a, const double2 *psi, const double2 *phi,
                            double *dots, cudaStream_t st);
// grad_gate[g] = d<O>/d(angle of gate g) for the rotations of the run-ordered
// gate array, from every run's c, given as `rows` shares each.
cudaError_t launch_run_grads(const UniRun *runs, int n_runs, int max_count, const RawGate *gates,
                             const double *thetas, const double *dots, int rows,
                             double *grad_gate, cudaStream_t st);

// ---------------------------------------------------------------- sparse term lists (k_sparse.cu)

// A key is z | x << n.
constexpr int kSpMaxBlocks = 608;        // partial sums of the x-free coefficients
constexpr int kSpSmallCap = 4096;        // list entries one CTA keeps in shared memory

// A rotation pulled back through the Clifford gates before it: about the Pauli
// string P instead of a wire's letter, so those gates need not touch the list.
struct SpRot {
    uint64_t P;                          // key of the string
    uint64_t anti;                       // parity(key & anti): the term anticommutes with P
    uint64_t letter;                     // parity(key & letter) == (flags & 1): it is the u term
    int32_t param;
    uint32_t flags;                      // bit 0 see above, bit 1: the string's sign is minus
};

struct SpTab {                           // tableau entry: image of X_q or Z_q, its sign
    uint64_t key;
    uint32_t neg;
    uint32_t pad;
};

// The tableau regrouped by chunks of 4 qubits (8 generators): per chunk the
// ordered products of all 256 subsets of its generator images.
constexpr int kSpChunkQubits = 4;
constexpr int kSpChunks = 8;             // 32 qubits
constexpr int kSpChunkEntries = kSpChunks * 256;
struct SpChunk {                         // x, z of the product string, phase exponent (mod 4)
    uint32_t x, z, e, pad;
};

enum { SP_RUNNING = 0, SP_OVERFLOW = 1, SP_THRESHOLD = 2 };

// Where a run stands: the list is the one before rotation `rot`, in buffer `buf`.
struct SpState {
    int64_t count;
    int32_t rot, buf;
    int32_t stop;                        // SP_OVERFLOW: rotation `rot` would not fit (not applied)
    int32_t err;                         // 1: a table probe ran out, 2: a wait (never expected)
    uint32_t arrived;                    // the grid barrier
    uint32_t blocks;                     // blocks of the x-free sum that are done
    double value;                        // the x-free sum
    int64_t pad[3];
};

struct SpRunArgs {
    SpState *st;
    int64_t *counts;                     // counts[r + 1] = order after rotation r
    const SpRot *rots;
    const double *cs;                    // cos, sin per slot
    int32_t n_rot, n, inverse;
    int32_t grid;                        // CTAs of the grid kernel, all resident
    int64_t cap, threshold;              // list capacity; stop above this order (0: never)
    const uint64_t *init;                // the initial list: keys, then coefficients
    uint64_t *keys[2];
    double *vals[2];
    uint64_t *table;                     // open-addressing table, all slots free between rotations
    int32_t *partner;                    // per term: position of its partner, -1 absent (and idle)
    uint64_t *tiles;                     // per tile: step tag and emitted terms
};

// cs[2 p] = cos(thetas[p]), cs[2 p + 1] = sin(thetas[p]) for every slot
cudaError_t launch_sp_cos_sin(const double *thetas, int64_t n_params, double *cs,
                              cudaStream_t st);
// chunks: kSpChunkEntries, from the tableau's 64 entries (2n used)
cudaError_t launch_sp_chunks(const SpTab *tab, int n, SpChunk *chunks, cudaStream_t st);
int sp_table_log(int64_t count);         // table slots (log2) for a list of `count` terms
int64_t sp_tiles(int64_t cap, int grid); // tile words for lists of up to `cap` terms
cudaError_t sp_run_grid(int device, int *grid);
// the rotations while the list fits one CTA's shared memory, from a.init
cudaError_t launch_sp_small(const SpRunArgs &a, cudaStream_t st);
// the rest, from the state, on the whole GPU (cooperative launch)
cudaError_t launch_sp_run(const SpRunArgs &a, cudaStream_t st);
// st->value: fixed-order sum of the coefficients whose images are x-free;
// parity(key & xcol[q]) is bit q of an image's x mask
cudaError_t launch_sp_xfree(const SpRunArgs &a, const uint64_t *xcol, const SpChunk *chunks,
                            double *partial, cudaStream_t st);
// the final list's images, in the order of the list: into `out` or `terms`
cudaError_t launch_sp_images(const uint64_t *keys, const double *vals, int64_t count, int n,
                             const SpChunk *chunks, DevTerm *out, stab_term *terms,
                             cudaStream_t st);

}  // namespace stab

struct stab_ctx;
namespace stab {
// <0^n| U^dagger O U |0^n> for the loaded circuit, O given as nt deduplicated
// device terms (stab_api.cpp); blocks until the value is on the host.
int expect_device_terms(stab_ctx *c, const DevTerm *terms, int64_t nt, double *out);
}  // namespace stab

namespace stab {
// Items of a batch whose vectors are too long for one CTA each: a context of
// the streamed kernels (loaded, observable set) gives its chains of tile steps,
// which the batch runs together with its other long items' in one launch.
// gens: the n generators, else <O>.  prepare: buffers, maps, steps; *chains
// (host, the context's) with cta0 and ctas for max_ctas CTAs alone.  Per run:
// fill, the chains, finish (out: 8 bytes, or n 4^n doubles).
int long_item_prepare(stab_ctx *c, bool gens, int max_ctas, const ChainDesc **chains,
                      int *n_chains);
int long_item_fill(stab_ctx *c, bool gens, cudaStream_t s);
int long_item_finish(stab_ctx *c, bool gens, double *out, cudaStream_t s);
}  // namespace stab
