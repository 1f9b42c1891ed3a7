// stab_api.cpp -- the C interface (include/stab.h): contexts, device buffers,
// circuit loading, and the launch sequences of every entry point.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <functional>
#include <map>
#include <new>
#include <string>
#include <thread>
#include <vector>

#include "../../include/stab.h"
#include "launch.h"
#include "host_pool.h"
#include "planner.h"
#include "tuner.h"

using namespace stab;

namespace {

thread_local int g_last_cuda = 0;

}  // namespace

void stab::record_cuda_error(cudaError_t e) { g_last_cuda = (int)e; }

namespace {

#define CK(expr)                                                    \
    do {                                                            \
        cudaError_t e_ = (expr);                                    \
        if (e_ != cudaSuccess) {                                    \
            g_last_cuda = (int)e_;                                  \
            return STAB_E_CUDA;                                     \
        }                                                           \
    } while (0)

#define RC(expr)                 \
    do {                         \
        int r_ = (expr);         \
        if (r_ != STAB_OK) return r_; \
    } while (0)

struct DevBuf {
    void *p = nullptr;
    size_t bytes = 0;
};

size_t align256(size_t b) { return (b + 255) & ~(size_t)255; }

// Resident plans with at least this many passes also get split streams.
constexpr int kSplitMinPasses = 64;
// n = 2, 3: the unitaries' tree is two levels of 3 us and the read-outs are one
// small launch, against a compose, two encodes and 0.1 us a pass and vector, so
// almost any plan is better off there (angles in, generators, <O>: n = 2, 20 gates 32
// -> 28 us, 100 gates 37 -> 31; n = 3 32 -> 30, 38 -> 33; gradients 60 -> 44 and 108
// -> 57).  At n = 4 the levels take 6 us and the read-out 256 rows: 34 -> 37, 40 ->
// 42 and even at 200 gates, about 64 passes; at n = 1 a plan is one run (37 -> 41).
constexpr int kUniMinPasses = 8;
// Resident adjoint: per-thread dot shares while the CTA has at most this many
// threads (n <= 5) and the shares take at most this many bytes.
constexpr int kPartialThreads = 256;
constexpr size_t kPartialBytes = (size_t)256 << 20;

}  // namespace

size_t stab::resident_partial_bytes(int n, int64_t n_rot) {
    const int t = resident_adjoint_threads(n);
    const size_t rows = (size_t)(n_rot > 0 ? n_rot : 0), cols = (size_t)(t > 0 ? t : 0);
    const size_t bytes = rows * cols * sizeof(double);
    return (t > 0 && t <= kPartialThreads && bytes <= kPartialBytes) ? bytes : 0;
}

namespace {

// Plans of at least this many passes build their instruction streams on
// several host threads.
constexpr int kThreadedStreamPasses = 2048;

// Device memory a context may take for the stored sweeps of a gradient; above
// it the pair sweep runs, which keeps a fixed number of vectors.
constexpr size_t kCheckpointBytes = (size_t)4 << 30;
// More than this goes back at a load whose circuit takes less than a quarter of it
// (a training loop's loads of like circuits keep theirs).
constexpr size_t kCheckpointRelease = (size_t)64 << 20;

// Instruction stream of a plan for the resident kernels, with the indices of
// the records the encode kernel fills (rotations and maps).
struct DevStreamBuf {
    std::vector<Rec> host;
    std::vector<int32_t> enc;
    // a long stream is built as two pieces at once: the second piece (its
    // encoded positions already offset) is uploaded right behind the first
    std::vector<Rec> tail;
    std::vector<int32_t> tail_enc;
    Rec *dev = nullptr;
    const int32_t *enc_dev = nullptr;
    int n_chunks = 0;
};

// A plan uploaded to the device: one buffer holding passes, ops, maps, map
// gate indices, raw gates, the slot CSR and (resident plans) the forward and
// backward instruction streams.
struct DevPlan {
    HostPlan host;
    int host_n = 0;                  // qubits of the plan
    bool streams = false;
    DevStreamBuf sf, sb;
    // split resident streams (see split_resident): forward passes [0, split)
    // and [split, P), backward passes [split, P) and (gradient plans) [0, split);
    // split < 0: none
    DevStreamBuf h1, h2, h2b, h1b;
    int split = -1;
    // n <= 4 (uni): K >= 2 parts, part k = passes [cuts[k],
    // cuts[k+1]), each cut into segments whose unitaries are composed at once
    // (see k_unitary.cu); no streams.
    bool uni = false;
    bool uni_identity = false;       // some wire run is the identity and holds no rotation, so
                                     // a gradient plan of its own would have other units
    std::vector<int> cuts;
    std::vector<UniOp> uops;
    std::vector<UniRun> uruns;
    std::vector<RawGate> ugates;
    std::vector<UniSeg> usegs;
    std::vector<UniPart> uparts;
    int uni_max_run = 0, uni_nodes = 0;
    UniArgs uargs{};
    const UniRun *uruns_dev = nullptr;
    const RawGate *ugates_dev = nullptr;
    std::vector<DevStreamBuf *> all_streams() { return {&sf, &sb, &h1, &h2, &h2b, &h1b}; }
    DevBuf buf;
    Program prog{};
    const int32_t *map_gate_idx = nullptr;
    std::vector<DevMap3> pass_maps;  // of prog.pass_maps, before composition
    int max_pass_gates = 0, wire_passes = 0;
    const int32_t *run_gates = nullptr;
    const RawGate *raw = nullptr;
    const int32_t *param_ptr = nullptr;
    const int32_t *param_rot = nullptr;
    bool built = false;
    bool encoded = false;
    bool ops_encoded = false, maps_encoded = false;   // streamed plans
};

// Pinned staging of uploads on the aux stream, so that the copies are queued and
// the caller does not wait for what is queued before them: a block that is filled
// from the front while copies are in flight and replaced when it is full (the old
// one goes when they are done).
struct Staging {
    size_t least = 0;      // bytes of a block
    char *p = nullptr;
    size_t bytes = 0, at = 0;
    std::vector<char *> full;
    cudaEvent_t copied = nullptr;   // behind the copies up to the last mark()
    bool unmarked = false;          // a copy was queued after it
    // idle: the caller knows that no copy is in flight.
    int take(size_t want, bool idle, char **out) {
        want = align256(want);
        if (!idle && !unmarked) {
            idle = !copied || cudaEventQuery(copied) == cudaSuccess;
            if (!idle) (void)cudaGetLastError();   // not ready
        }
        if (idle) {
            for (char *b : full) cudaFreeHost(b);
            full.clear();
            at = 0;
        }
        if (at + want > bytes) {
            const size_t last = at;
            if (p && at == 0) cudaFreeHost(p);
            else if (p) full.push_back(p);
            p = nullptr;
            bytes = at = 0;
            // room for what was in the old one and this, so that calls which take
            // turns settle in one block
            const size_t cap = std::max(least, last + want);
            CK(cudaMallocHost((void **)&p, cap));
            bytes = cap;
        }
        *out = p + at;
        at += want;
        unmarked = true;
        return STAB_OK;
    }
    int mark(cudaStream_t s) {
        if (!copied) CK(cudaEventCreateWithFlags(&copied, cudaEventDisableTiming));
        CK(cudaEventRecord(copied, s));
        unmarked = false;
        return STAB_OK;
    }
    void release() {
        full.push_back(p);
        for (char *b : full)
            if (b) cudaFreeHost(b);
        full.clear();
        p = nullptr;
        if (copied) cudaEventDestroy(copied);
        copied = nullptr;
    }
};

// Where chains' tables follow the terms (kChainMinN to kChainMaxN): what 10,000
// gates' gradient takes.  (A few bytes come out of pinned memory that the
// driver holds already, one of 512 KiB takes 0.1 ms: the first call at n = 2 takes
// 0.22 ms, 0.24 with 512 KiB.)
constexpr size_t kStagingTables = (size_t)512 << 10;

// A captured sequence of streamed launches, valid while its key is unchanged.
struct GraphCache {
    cudaGraphExec_t exec = nullptr;
    std::vector<const void *> key;
    std::vector<const void *> seen;  // key of the last run made without a graph
    int64_t launches = 0;            // kernels in the graph
    void *result = nullptr;          // buffer that ends up holding the result
    void reset() {
        if (exec) cudaGraphExecDestroy(exec);
        exec = nullptr;
        key.clear();
        seen.clear();
        launches = 0;
        result = nullptr;
    }
};

// Two chains of tile steps on the device (see k_stream_chain), valid while the
// key (plan, buffers) is unchanged.
struct ChainSet {
    std::vector<const void *> key;
    std::vector<ChainStep> host[2];
    std::vector<ChainShape> shapes;           // tables, one per distinct shape
    std::vector<int> in_shape[2], out_shape[2];   // per step
    std::map<std::string, int> known;         // shape -> its index
    void clear() {
        key.clear();
        shapes.clear();
        known.clear();
        for (int k = 0; k < 2; ++k) {
            host[k].clear();
            in_shape[k].clear();
            out_shape[k].clear();
        }
    }
    DevBuf dev, tables;
    ChainDesc desc[2];                        // of the chains with steps, in order
    int n_chains = 0, grid = 0;
    const ChainDesc *desc_dev = nullptr;
    uint32_t *arrived = nullptr;              // 32 words per chain
    bool alone = false;
    double *result[2] = {nullptr, nullptr};   // where each chain's vectors end up
};

}  // namespace

struct stab_ctx {
    int n = 0;
    int device = 0;
    int kernel = STAB_KERNEL_AUTO;
    int fuse = 1;
    stab_path_choice choice{};         // AUTO: the path tuner's choice for this n and GPU
    cudaStream_t st = nullptr;
    cudaStream_t aux = nullptr;
    cudaStream_t aux2 = nullptr;       // second branch of the split adjoint
    cudaEvent_t ev_fork = nullptr, ev_join = nullptr;
    bool own_st = false;
    cudaEvent_t ev_ready = nullptr;    // plan uploaded and encoded (on st); the aux work waits
                                       // on it (the observable's terms are uploaded on aux)
    cudaEvent_t ev_aux = nullptr;      // aux work done
    cudaEvent_t ev_gens = nullptr;     // readers of the generators queued so far (on st)
    cudaEvent_t ev_stage = nullptr;    // staging buffer free
    stab_alloc_fn alloc = nullptr;
    stab_free_fn free = nullptr;
    void *user = nullptr;

    bool loaded = false;
    bool gens_valid = false;
    std::vector<stab_gate> gates;
    int64_t n_params = 0;

    DevPlan fwd, grad;
    // gradients from stored sweeps (streamed; see ck_gradient): the fused plan
    // when fwd is not one, the runs and their gates; blocks of wire passes
    DevPlan ck;
    struct CkBlock {
        int p0, p1;                  // its wire passes
        std::vector<int> before;     // Clifford passes between the previous block and this one
    };
    std::vector<CkBlock> ck_blocks;
    std::vector<int> ck_after;       // Clifford passes after the last block
    std::vector<DotJob> ck_jobs;     // pointers filled in once the slots exist
    std::vector<int> ck_job_block;
    int ck_chunks = 1;
    bool ck_ready = false, ck_off = false;   // built for this plan; no room or not wanted
    size_t ck_bytes_max = kCheckpointBytes;
    bool ck_must = false;            // no room is an error (the caller tries again), not a reason
                                     // for the pair sweep
    DevBuf ckslots, ckjobs, ckdots;
    std::vector<const void *> key_ck;
    DevBuf thetas, gens, gens_tmp, lam, rho, tmp, tmp2, terms, scal, grad_rot, partials, grads;
    DevBuf gbuf;                     // gradients written inside captured graphs
    DevBuf lam2, tmp3;               // second-branch buffers of the split sweeps
    DevBuf dotbuf;                   // partial sums of the split expectation's inner product
    DevBuf gmid;                     // split resident adjoint: rho, then lambda, at the cut
    bool grad_uni = false;           // the gradient runs through the segments' unitaries
    bool grad_ran = false;           // a gradient was asked for since the circuit was loaded
    DevBuf ustates, udots;           // its states at the parts' boundaries, runs' dot shares
    // split sweeps of the small registers.  n <= 4: the wire runs' 2 x 2 maps,
    // the segments' and parts' unitaries.  n = 5, 6: the two halves of <O>:
    // meeting vectors, batch units, unit counter
    DevBuf umaps, unodes, rmid, lmid, units_e, cnt;
    std::vector<const void *> key_e;
    size_t split_smem = 0;
    int sms = 0;                     // SMs of the device
    int chain_ctas = 0;              // CTAs of a chain launch that fit on it at once
    bool chains_off = false;         // no room for the chains' tables: launches instead
    // the parts' unitaries were composed for these angles when tx_gen ==
    // param_gen; ev_tx marks their end on st
    int64_t param_gen = 0, tx_gen = -1;
    cudaEvent_t ev_tx = nullptr;
    DevBuf status;                   // int32 set by kernels whose bounded waits gave up
    GraphCache g_gens, g_expect, g_grad; // streamed launch sequences (n > resident sizes)
    ChainSet c_gens, c_expect, c_grad;   // the same as one launch, small vectors
    int64_t plan_gen = 0;            // bumped whenever a plan is rebuilt
    int32_t n_obs_terms = 0;
    bool obs_loaded = false;
    int64_t h2d_bytes = 0, d2h_bytes = 0;
    double *gens_cur = nullptr;      // buffer holding the evolved generators

    void *stage = nullptr;           // pinned host staging
    size_t stage_bytes = 0;
    Staging aux_stage;               // terms, chains' steps and shapes, gradients' jobs
    int64_t launches = 0;

    int dalloc(DevBuf &b, size_t bytes, cudaStream_t s) {
        if (b.bytes >= bytes && b.p) return STAB_OK;
        dfree(b, s);
        bytes = align256(bytes ? bytes : 256);
        void *p = nullptr;
        if (alloc) {
            p = alloc(bytes, (void *)s, user);
            if (!p) return STAB_E_NOMEM;
        } else {
            cudaError_t e = cudaMallocAsync(&p, bytes, s);
            if (e != cudaSuccess) {
                (void)cudaGetLastError();
                return e == cudaErrorMemoryAllocation ? STAB_E_NOMEM : (g_last_cuda = (int)e, STAB_E_CUDA);
            }
        }
        b.p = p;
        b.bytes = bytes;
        return STAB_OK;
    }
    void dfree(DevBuf &b, cudaStream_t s) {
        if (!b.p) return;
        // a buffer may be in use on either stream of the context
        if (st) cudaStreamSynchronize(st);
        if (aux) cudaStreamSynchronize(aux);
        if (aux2) cudaStreamSynchronize(aux2);
        if (free) free(b.p, b.bytes, (void *)s, user);
        else cudaFreeAsync(b.p, s);
        b.p = nullptr;
        b.bytes = 0;
    }
    int host_stage(void *&buf, size_t &cap, size_t bytes) {
        if (cap >= bytes && buf) return STAB_OK;
        if (buf) cudaFreeHost(buf);
        buf = nullptr;
        cap = 0;
        CK(cudaMallocHost(&buf, bytes));
        cap = bytes;
        return STAB_OK;
    }
    size_t vec_bytes() const { return (sizeof(double) << (2 * n)); }
    bool use_resident() const {
        const bool k = kernel == STAB_KERNEL_AUTO ? choice.resident != 0
                                                  : (kernel == STAB_KERNEL_RESIDENT ||
                                                     kernel == STAB_KERNEL_PLAIN);
        return k && n <= kMaxResidentQubits;
    }
    bool use_resident_adjoint() const {
        const bool k = kernel == STAB_KERNEL_AUTO ? choice.resident_adjoint != 0
                                                  : kernel == STAB_KERNEL_RESIDENT;
        return k && n <= kMaxResidentAdjoint;
    }
    PlanMode fwd_mode() const {
        const bool rows = use_resident() && resident_lanes_per_group(n) == 4;
        if (kernel == STAB_KERNEL_PLAIN || !fuse) return rows ? PLAN_PLAIN_ROWS : PLAN_PLAIN;
        return rows ? PLAN_ROWS : PLAN_FUSED;
    }
};

namespace {

// Uploads a host plan into its device buffer (one copy from pinned staging).
int upload_plan(stab_ctx *c, DevPlan &P) {
    HostPlan &H = P.host;
    // resident plans read only their streams (plus maps and raw gates for encoding)
    const size_t n_pass = P.streams ? 0 : H.passes.size();
    const size_t n_ops = P.streams ? 0 : H.ops.size();
    // streamed plans whose vectors are small enough for tile launches: every
    // wire pass's run as a composed map
    P.pass_maps.clear();
    P.max_pass_gates = P.wire_passes = 0;
    if (!P.streams && (uint64_t)c->vec_bytes() / sizeof(double) <= (uint64_t)c->choice.tile_limit &&
        H.run_first.size() == n_pass + 1) {
        P.pass_maps.resize(n_pass);
        for (size_t p = 0; p < n_pass; ++p) {
            DevMap3 &m = P.pass_maps[p];
            m.first = H.run_first[p];
            m.count = H.run_first[p + 1] - H.run_first[p];
            P.max_pass_gates = std::max(P.max_pass_gates, (int)m.count);
            P.wire_passes += H.passes[p].type == P_WIRE;
        }
    }
    const size_t n_pmaps = P.pass_maps.size(), n_rg = n_pmaps ? H.run_gates.size() : 0;
    // plans applied through segment unitaries read their own op list and runs
    const size_t n_maps = P.uni ? 0 : H.maps.size();
    const size_t n_midx = P.uni ? 0 : H.map_gate_idx.size();
    const size_t n_raw = P.uni ? 0 : H.raw.size();
    const size_t b_pass = align256(n_pass * sizeof(DevPass));
    const size_t b_ops = align256(n_ops * sizeof(DevOp));
    const size_t b_maps = align256(n_maps * sizeof(DevMap3));
    const size_t b_midx = align256(n_midx * sizeof(int32_t));
    const size_t b_raw = align256(n_raw * sizeof(RawGate));
    const size_t b_pptr = align256(H.param_ptr.size() * sizeof(int32_t));
    const size_t b_prot = align256(H.param_rot.size() * sizeof(int32_t));
    const size_t b_pulls = align256(H.pulls.size() * sizeof(DevPull));
    const std::vector<DevStreamBuf *> streams = P.all_streams();
    size_t b_streams = 0;
    for (const DevStreamBuf *S : streams)
        b_streams += align256((S->host.size() + S->tail.size()) * sizeof(Rec)) +
                     align256((S->enc.size() + S->tail_enc.size()) * 4);
    const size_t b_pmaps = align256(n_pmaps * sizeof(DevMap3)), b_rg = align256(n_rg * 4);
    const size_t b_uops = align256(P.uops.size() * sizeof(UniOp));
    const size_t b_uruns = align256(P.uruns.size() * sizeof(UniRun));
    const size_t b_ugates = align256(P.ugates.size() * sizeof(RawGate));
    const size_t b_usegs = align256(P.usegs.size() * sizeof(UniSeg));
    const size_t b_uparts = align256(P.uparts.size() * sizeof(UniPart));
    const size_t total = b_pass + b_ops + b_maps + b_midx + b_raw + b_pptr + b_prot + b_pulls +
                         b_streams + b_uops + b_uruns + b_ugates + b_usegs + b_uparts + b_pmaps + b_rg;
    RC(c->dalloc(P.buf, total, c->st));
    CK(cudaEventSynchronize(c->ev_stage));
    RC(c->host_stage(c->stage, c->stage_bytes, total));
    char *h = (char *)c->stage;
    char *d = (char *)P.buf.p;
    size_t off = 0;
    // large pieces are copied into the staging buffer by the host pool
    std::vector<std::function<void()>> copies;
    // [src, bytes) then [src2, bytes2) at the next `span` bytes of the buffer
    auto put = [&](const void *src, size_t bytes, size_t span, const void *src2 = nullptr,
                   size_t bytes2 = 0) {
        size_t o = off;
        for (int k = 0; k < 2; ++k) {
            const void *from = k ? src2 : src;
            const size_t b = k ? bytes2 : bytes;
            if (b >= ((size_t)1 << 18)) {
                char *dst = h + o;
                copies.push_back([dst, from, b] { std::memcpy(dst, from, b); });
            } else if (b) {
                std::memcpy(h + o, from, b);
            }
            o += b;
        }
        const size_t at = off;
        off += span;
        return d + at;
    };
    P.prog.passes = (const DevPass *)put(H.passes.data(), n_pass * sizeof(DevPass), b_pass);
    P.prog.ops = (const DevOp *)put(H.ops.data(), n_ops * sizeof(DevOp), b_ops);
    P.prog.maps = (const DevMap3 *)put(H.maps.data(), n_maps * sizeof(DevMap3), b_maps);
    P.map_gate_idx = (const int32_t *)put(H.map_gate_idx.data(), n_midx * 4, b_midx);
    P.raw = (const RawGate *)put(H.raw.data(), n_raw * sizeof(RawGate), b_raw);
    P.param_ptr = (const int32_t *)put(H.param_ptr.data(), H.param_ptr.size() * 4, b_pptr);
    P.param_rot = (const int32_t *)put(H.param_rot.data(), H.param_rot.size() * 4, b_prot);
    P.prog.pulls = (const DevPull *)put(H.pulls.data(), H.pulls.size() * sizeof(DevPull), b_pulls);
    for (DevStreamBuf *S : streams) {
        const size_t rb = S->host.size() * sizeof(Rec), tb = S->tail.size() * sizeof(Rec);
        S->dev = (Rec *)put(S->host.data(), rb, align256(rb + tb), S->tail.data(), tb);
        const size_t eb = S->enc.size() * 4, teb = S->tail_enc.size() * 4;
        S->enc_dev = (const int32_t *)put(S->enc.data(), eb, align256(eb + teb),
                                          S->tail_enc.data(), teb);
    }
    P.prog.pass_maps = nullptr;
    if (n_pmaps) {
        P.prog.pass_maps =
            (const DevMap3 *)put(P.pass_maps.data(), n_pmaps * sizeof(DevMap3), b_pmaps);
        P.run_gates = (const int32_t *)put(H.run_gates.data(), n_rg * 4, b_rg);
    }
    P.uargs = UniArgs{};
    P.uargs.ops = (const UniOp *)put(P.uops.data(), P.uops.size() * sizeof(UniOp), b_uops);
    P.uruns_dev = (const UniRun *)put(P.uruns.data(), P.uruns.size() * sizeof(UniRun), b_uruns);
    P.ugates_dev = (const RawGate *)put(P.ugates.data(), P.ugates.size() * sizeof(RawGate),
                                        b_ugates);
    P.uargs.segs = (const UniSeg *)put(P.usegs.data(), P.usegs.size() * sizeof(UniSeg), b_usegs);
    P.uargs.parts = (const UniPart *)put(P.uparts.data(), P.uparts.size() * sizeof(UniPart),
                                         b_uparts);
    P.uargs.n_segs = (int32_t)P.usegs.size();
    P.prog.n_passes = (int32_t)n_pass;
    P.prog.n_ops = (int32_t)n_ops;
    HostPool::run(copies);
    CK(cudaMemcpyAsync(P.buf.p, h, total, cudaMemcpyHostToDevice, c->st));
    CK(cudaEventRecord(c->ev_stage, c->st));
    c->h2d_bytes += (int64_t)total;
    P.built = true;
    P.encoded = false;
    return STAB_OK;
}

int encode_plan(stab_ctx *c, DevPlan &P) {
    const double *th = (const double *)c->thetas.p;
    if (P.uni) {
        CK(launch_uni_maps(P.uruns_dev, (int)P.uruns.size(), P.uni_max_run, P.ugates_dev, th,
                           (UniMap *)c->umaps.p, c->st));
        c->launches += !P.uruns.empty();
        P.encoded = true;
        return STAB_OK;
    }
    if (P.streams) {
        // resident plans: only the instruction streams are read by kernels;
        // each run's map is composed once and copied into every stream
        const int n_maps = (int)P.host.maps.size();
        if (n_maps > 0) {
            CK(launch_compose_maps(const_cast<DevMap3 *>(P.prog.maps), n_maps,
                                   max_map_count(P.host.maps.data(), P.host.maps.size()),
                                   P.map_gate_idx, P.raw, th, c->st));
            c->launches++;
        }
        for (DevStreamBuf *S : P.all_streams()) {
            const int n_enc = (int)(S->enc.size() + S->tail_enc.size());
            if (n_enc == 0) continue;
            CK(launch_encode_stream(S->dev, S->enc_dev, n_enc, P.prog.maps, th,
                                    c->st));
            c->launches++;
        }
        P.encoded = true;
        return STAB_OK;
    }
    // streamed plans: what the next call reads (stream_ops, stream_maps)
    P.ops_encoded = P.maps_encoded = false;
    P.encoded = true;
    return STAB_OK;
}

// The ops of a streamed plan for the current angles (a launch per pass reads
// them), or its composed pass maps (tile launches), on the context stream;
// ev_ready moves behind them.
int stream_ops(stab_ctx *c, DevPlan &P) {
    if (P.ops_encoded) return STAB_OK;
    const int n_ops = P.prog.n_ops, n_maps = (int)P.host.maps.size();
    if (n_ops > 0 || n_maps > 0)
        CK(launch_encode(const_cast<DevOp *>(P.prog.ops), n_ops,
                         const_cast<DevMap3 *>(P.prog.maps), n_maps,
                         max_map_count(P.host.maps.data(), P.host.maps.size()), P.map_gate_idx,
                         P.raw, (const double *)c->thetas.p, c->st));
    c->launches += (n_maps > 0) + (n_ops > 0);
    P.ops_encoded = true;
    CK(cudaEventRecord(c->ev_ready, c->st));
    return STAB_OK;
}

int stream_maps(stab_ctx *c, DevPlan &P) {
    if (P.maps_encoded) return STAB_OK;
    if (!P.pass_maps.empty()) {
        CK(launch_compose_maps(const_cast<DevMap3 *>(P.prog.pass_maps), (int)P.pass_maps.size(),
                               P.max_pass_gates, P.run_gates, P.raw,
                               (const double *)c->thetas.p, c->st));
        c->launches++;
    }
    P.maps_encoded = true;
    CK(cudaEventRecord(c->ev_ready, c->st));
    return STAB_OK;
}

// How wire passes on n_vec vectors run where the path choice allows tiles.
// Small vectors: as composed maps, nine FMAs a group, because launches and
// latency bound them.  From 2^18 entries on the FP64 pipe bounds a pass: maps
// only where the runs hold two rotations and more (three FMAs each as lifts), one
// vector's other plans as tiles of lifts, more vectors as a launch per pass.
// (n = 9, <O> of 1,000 gates: 2.7 rotations a run 0.44 ms in tiles of maps, 0.55 a
// launch per pass; 0.9 a run 0.90 in tiles of maps, 0.68 in tiles of lifts,
// 0.82 a launch per pass.  Nine generators, 300 gates: 1.79 ms in tiles of maps,
// 1.28 a launch per pass.)
enum TileForm { kNoTiles, kTileMaps, kTileOps };
TileForm tile_form(const stab_ctx *c, const DevPlan &P, int n_vec) {
    const uint64_t size = (uint64_t)n_vec << (2 * c->n);
    if (!P.prog.pass_maps || size > (uint64_t)c->choice.tile_limit) return kNoTiles;
    if (size < ((uint64_t)1 << 18) || P.host.n_rot >= 2 * P.wire_passes) return kTileMaps;
    return n_vec == 1 ? kTileOps : kNoTiles;
}

// What a sweep of n_vec vectors reads, for the current angles.
int stream_encode(stab_ctx *c, DevPlan &P, int n_vec) {
    return tile_form(c, P, n_vec) == kTileMaps ? stream_maps(c, P) : stream_ops(c, P);
}

// One instruction stream to build: passes [k0, k1) of the plan, forward or
// (backward) walked from k1 - 1 down to k0.
struct StreamSpec {
    DevStreamBuf *S;
    bool backward;
    int k0, k1;
};

// Streams of at least this many passes are built as two pieces at once.
constexpr int kStreamPiecePasses = 4096;

// Builds the streams, on the host pool when `threads` is set; there a long
// stream is built as two pieces at once, the first ending in R_NEXT on a
// chunk boundary (its pending pulls in an identity pass), the second in
// S.tail -- the same passes, pulls and ops as the one-piece stream.
void build_streams(const DevPlan &P, const std::vector<StreamSpec> &specs, bool threads) {
    std::vector<std::function<void()>> jobs;
    for (const StreamSpec &sp : specs) {
        DevStreamBuf *S = sp.S;
        S->tail.clear();
        S->tail_enc.clear();
        if (!threads || sp.k1 - sp.k0 < kStreamPiecePasses) {
            jobs.push_back([&P, sp] {
                build_stream(P.host, sp.backward, &sp.S->host, sp.k0, sp.k1, &sp.S->enc);
            });
            continue;
        }
        const int mid = sp.k0 + (sp.k1 - sp.k0) / 2;
        const int a0 = sp.backward ? mid : sp.k0, a1 = sp.backward ? sp.k1 : mid;
        const int b0 = sp.backward ? sp.k0 : mid, b1 = sp.backward ? mid : sp.k1;
        jobs.push_back([&P, sp, a0, a1] {
            build_stream(P.host, sp.backward, &sp.S->host, a0, a1, &sp.S->enc, false);
        });
        jobs.push_back([&P, sp, b0, b1] {
            build_stream(P.host, sp.backward, &sp.S->tail, b0, b1, &sp.S->tail_enc);
        });
    }
    if (threads) {
        HostPool::run(jobs);
    } else {
        for (auto &j : jobs) j();
    }
    for (const StreamSpec &sp : specs) {
        DevStreamBuf &S = *sp.S;
        for (int32_t &e : S.tail_enc) e += (int32_t)S.host.size();
        S.n_chunks = (int)((S.host.size() + S.tail.size()) / kChunkRecs);
    }
}

void clear_parts(DevPlan &P) {
    P.uni = P.uni_identity = false;
    P.cuts.clear();
    P.uops.clear();
    P.uruns.clear();
    P.ugates.clear();
    P.usegs.clear();
    P.uparts.clear();
}

// Forward and backward streams, built concurrently on host threads; with
// split_frac > 0 (and enough passes) also the split streams cut at that
// fraction of the passes.  A split gradient plan (grad) needs only the four
// half streams, not the whole-circuit ones.  Below kThreadedStreamPasses
// passes the streams are built on the calling thread: handing them to the
// pool would cost more than the work.
void make_streams(DevPlan &P, double split_frac = 0.0, bool grad = false) {
    P.streams = true;
    const int np = (int)P.host.passes.size();
    const bool threads = np >= kThreadedStreamPasses;
    clear_parts(P);
    P.split = (split_frac > 0.0 && np >= kSplitMinPasses) ? (int)(np * split_frac) : -1;
    // streams that are rebuilt keep their capacity; the others are released
    if (P.split < 0) P.h1 = P.h2 = P.h2b = DevStreamBuf();
    if (!(grad && P.split >= 0)) P.h1b = DevStreamBuf();
    if (grad && P.split >= 0) {
        P.sf = P.sb = DevStreamBuf();
        build_streams(P,
                      {{&P.h1b, true, 0, P.split},
                       {&P.h1, false, 0, P.split},
                       {&P.h2, false, P.split, np},
                       {&P.h2b, true, P.split, np}},
                      threads);
        return;
    }
    if (P.split < 0) {
        build_streams(P, {{&P.sf, false, 0, np}, {&P.sb, true, 0, np}}, threads);
        return;
    }
    // A split plan (n = 5, 6) reads the whole forward stream (generators,
    // density matrix) and the halves that <O> meets from, h1 and h2b; nothing
    // reads the whole backward stream.
    P.sb = P.h2 = DevStreamBuf();
    build_streams(P,
                  {{&P.h1, false, 0, P.split}, {&P.h2b, true, P.split, np}, {&P.sf, false, 0, np}},
                  threads);
}

void no_streams(DevPlan &P) {
    P.streams = false;
    P.sf = DevStreamBuf();
    P.sb = DevStreamBuf();
    P.h1 = P.h2 = P.h2b = P.h1b = DevStreamBuf();
    clear_parts(P);
    P.split = -1;
}

// Reads and clears the kernels' status word (synchronizes the context).
int check_status(stab_ctx *c) {
    if (!c->status.p) return STAB_OK;
    int32_t h = 0;
    CK(cudaStreamSynchronize(c->aux));
    CK(cudaMemcpyAsync(&h, c->status.p, sizeof(int32_t), cudaMemcpyDeviceToHost, c->st));
    CK(cudaStreamSynchronize(c->st));
    if (h != 0) {
        CK(cudaMemsetAsync(c->status.p, 0, sizeof(int32_t), c->st));
        CK(cudaStreamSynchronize(c->st));
        return STAB_E_TIMEOUT;
    }
    return STAB_OK;
}

int upload_thetas_host(stab_ctx *c, const double *thetas) {
    const size_t bytes = (size_t)(c->n_params > 0 ? c->n_params : 1) * sizeof(double);
    RC(c->dalloc(c->thetas, bytes, c->st));
    if (c->n_params == 0) return STAB_OK;
    CK(cudaEventSynchronize(c->ev_stage));
    RC(c->host_stage(c->stage, c->stage_bytes, bytes));
    std::memcpy(c->stage, thetas, (size_t)c->n_params * sizeof(double));
    CK(cudaMemcpyAsync(c->thetas.p, c->stage, (size_t)c->n_params * sizeof(double),
                       cudaMemcpyHostToDevice, c->st));
    CK(cudaEventRecord(c->ev_stage, c->st));
    c->h2d_bytes += c->n_params * (int64_t)sizeof(double);
    return STAB_OK;
}

// Uploads deduplicated observable terms on the main stream (pinned staging).
int upload_terms(stab_ctx *c, const stab_term *O, int64_t n_terms) {
    std::vector<DevTerm> t;
    RC(encode_terms(c->n, O, n_terms, &t));
    const size_t bytes = (t.size() ? t.size() : 1) * sizeof(DevTerm);
    // The terms are read on the aux stream (expectations, gradients), so they
    // are uploaded there, from the aux staging: the upload does not queue behind
    // generator work on the main stream.  The aux stream may still read the
    // previous terms.
    CK(cudaStreamSynchronize(c->aux));
    RC(c->dalloc(c->terms, bytes, c->aux));
    if (!t.empty()) {
        char *h = nullptr;
        RC(c->aux_stage.take(bytes, true, &h));
        std::memcpy(h, t.data(), t.size() * sizeof(DevTerm));
        CK(cudaMemcpyAsync(c->terms.p, h, t.size() * sizeof(DevTerm), cudaMemcpyHostToDevice,
                           c->aux));
        c->h2d_bytes += (int64_t)(t.size() * sizeof(DevTerm));
    }
    c->n_obs_terms = (int32_t)t.size();
    return STAB_OK;
}

// Tiles of a launch below which a tile takes no further bits: with 4 wires of
// n = 8 (2^8 entries) one more bit gives 128 tiles, one to an SM, whose four
// warps fill its sub-partitions and read two entries in a row.
constexpr int kMinTiles = 128;

void bit_runs(const std::vector<int> &bits, BitRuns *r) {
    // bit k of a packed integer goes to index bit bits[k] (bits ascending)
    std::memset(r, 0, sizeof(*r));
    for (size_t k = 0; k < bits.size();) {
        size_t j = k + 1;
        while (j < bits.size() && bits[j] == bits[j - 1] + 1) ++j;
        r->src[r->n] = (uint8_t)k;
        r->dst[r->n] = (uint8_t)bits[k];
        r->len[r->n] = (uint8_t)(j - k);
        r->n++;
        k = j;
    }
}

// Tile geometry for the wires: their x and z bits plus as many of the lowest
// other bits as keep at least min_tiles tiles (and 2^max_bits entries).  tile
// and rest receive the index bits of a tile's entries and of the tiles.
void tile_bits_of(int n, int n_vec, const std::vector<int> &wires, int min_tiles, int max_bits,
                  std::vector<int> *tile_out, std::vector<int> *rest_out) {
    std::vector<int> qbits;
    for (int q : wires) {
        qbits.push_back(q);
        qbits.push_back(n + q);
    }
    std::vector<int> others;
    for (int b = 0; b < 2 * n; ++b)
        if (std::find(qbits.begin(), qbits.end(), b) == qbits.end()) others.push_back(b);
    int c = 0;
    while (c < (int)others.size() && (int)qbits.size() + c + 1 <= max_bits &&
           ((int64_t)n_vec << (2 * n - ((int)qbits.size() + c + 1))) >= min_tiles)
        ++c;
    std::vector<int> &tile = *tile_out;
    tile = qbits;
    tile.insert(tile.end(), others.begin(), others.begin() + c);
    std::sort(tile.begin(), tile.end());
    rest_out->assign(others.begin() + c, others.end());
}

void make_tile_group(int n, int n_vec, const std::vector<DevPass> &passes,
                     const std::vector<const DevPass *> &group, int inverse, TileGroup *tg,
                     int min_tiles = kMinTiles, int max_bits = kTileMaxBits) {
    std::memset(tg, 0, sizeof(*tg));
    std::vector<int> wires, tile, rest;
    for (const DevPass *p : group)
        if (std::find(wires.begin(), wires.end(), (int)p->q) == wires.end()) wires.push_back(p->q);
    tile_bits_of(n, n_vec, wires, min_tiles, max_bits, &tile, &rest);
    tg->n_pass = (int32_t)group.size();
    tg->tile_bits = (int32_t)tile.size();
    tg->rest_bits = (int32_t)rest.size();
    tg->inverse = inverse;
    for (size_t j = 0; j < group.size(); ++j) {
        const int q = group[j]->q;
        tg->lz[j] = (uint8_t)(std::find(tile.begin(), tile.end(), q) - tile.begin());
        tg->lx[j] = (uint8_t)(std::find(tile.begin(), tile.end(), n + q) - tile.begin());
        tg->n_ops[j] = group[j]->n_ops;
        tg->first[j] = group[j]->first;
        tg->map[j] = (uint32_t)(group[j] - passes.data());
    }
    bit_runs(tile, &tg->tile_runs);
    bit_runs(rest, &tg->rest_runs);
}

// ---------------------------------------------------------------- split sweeps of small registers
//
// A resident vector walks the circuit's passes one after another on one SM.
// n <= 4 (from kUniMinPasses or kSplitMinPasses passes): the plan is cut into parts
// whose maps are carried by their unitaries, composed from segments that run
// at once (k_unitary.cu); the generators, rho and <O> are read off the parts'
// unitaries, the gradient off states carried through the segments.
// n = 5, 6: <O> = <lambda, r> with r = rho_0 through the first half and
// lambda = O backward through the second -- two vectors at once on two CTAs
// of the persistent batch kernel, then one inner product.

int later_parts(const stab_ctx *c) { return (int)c->fwd.uparts.size() - 1; }

// Parts of a long plan: two cut at gen_cut of the passes, or three -- at n = 4
// where the path choice says so (a first part of gen_cut, two equal ones), at
// n <= 3 from kPartMinPasses passes a part (equal ones).  Where the cuts lie
// costs nothing: every part's segments run at once.
constexpr int kPartMinPasses = 32;
std::vector<int> part_cuts(const stab_ctx *c) {
    const int np = (int)c->fwd.host.passes.size();
    if (c->n <= 3 && np >= 3 * kPartMinPasses)
        return {0, (int)((int64_t)np / 3), (int)((int64_t)np * 2 / 3), np};
    const int c1 = (int)(np * c->choice.gen_cut);
    if (c->n == 4 && c->choice.gen_parts == 3 && np >= 3 * kSplitMinPasses)
        return {0, c1, c1 + (np - c1) / 2, np};
    return {0, c1, np};
}

// Plans of one gate list in different modes hold the same sequence of units:
// a P_CLIFF pass, or a maximal stretch of consecutive P_WIRE passes on one
// wire (a gradient plan only cuts a wire's run into several passes).
bool unit_start(const HostPlan &P, size_t i) {
    if (i == 0) return true;
    const DevPass &p = P.passes[i], &q = P.passes[i - 1];
    return p.type != P_WIRE || q.type != P_WIRE || p.q != q.q;
}

// Segments of a plan with W wire passes.  A segment of W / K passes takes
// 0.6 us a pass at n = 4 (0.3 below) and a level of the tree over the K
// segments about 6 us (3), so the sum is least near ten passes a segment; it is
// flat there (n = 4, 500 passes: 72, 69, 70, 71, 81 us a step at 6, 10, 15, 30,
// 50; n = 2 and 3 alike).  At n = 4 a segment's eight warps fill an SM's FP64
// pipe, so more segments than SMs only add levels.
constexpr int kUniSegPasses = 10;
int uni_segments(int n, int W, int sms) {
    return std::max(1, std::min(n == 4 ? sms : 2 * sms, W / kUniSegPasses));
}

// The forward plan as parts [cuts[k], cuts[k + 1]) cut into segments at unit
// boundaries, each of about the same number of wire passes.
void make_uni(DevPlan &P, const std::vector<int> &cuts, int sms) {
    clear_parts(P);
    P.streams = P.uni = true;
    P.sf = P.sb = P.h1 = P.h2 = P.h2b = P.h1b = DevStreamBuf();
    P.cuts = cuts;
    P.split = (int)P.host.passes.size() >= kSplitMinPasses ? cuts[1] : -1;
    const HostPlan &H = P.host;
    const int np = (int)H.passes.size(), K = (int)cuts.size() - 1;
    std::vector<int> wires((size_t)np + 1, 0);   // wire passes before pass i
    for (int i = 0; i < np; ++i)
        wires[(size_t)i + 1] = wires[(size_t)i] + (H.passes[(size_t)i].type == P_WIRE);
    const int W = wires[(size_t)np], want = uni_segments(P.host_n, W, sms);
    P.uops.reserve((size_t)np + H.ops.size());
    P.uruns.reserve((size_t)W);
    P.ugates.reserve(H.map_gate_idx.size());
    P.uni_max_run = 0;
    int node = 0;
    for (int k = 0; k < K; ++k) {
        const int c0 = cuts[(size_t)k], c1 = cuts[(size_t)k + 1];
        const int w0 = wires[(size_t)c0], wp = wires[(size_t)c1] - w0;
        const int n_seg = std::max(1, (int)((int64_t)want * wp / std::max(1, W)));
        UniPart part{};
        part.seg_first = (int32_t)P.usegs.size();
        part.node = node;
        int at = c0;
        for (int j = 1; j <= n_seg && at < c1; ++j) {
            int end = c1;
            if (j < n_seg) {
                const int target = w0 + (int)((int64_t)wp * j / n_seg);
                end = at + 1;
                while (end < c1 && !(wires[(size_t)end] >= target && unit_start(H, (size_t)end)))
                    ++end;
            }
            UniSeg sg{};
            sg.op_first = (int32_t)P.uops.size();
            sg.map_first = (int32_t)P.uruns.size();
            sg.part = k;
            sg.index = (int32_t)P.usegs.size() - part.seg_first;
            int parity = 0;
            for (int i = at; i < end; ++i) {
                const DevPass &p = H.passes[(size_t)i];
                for (int o = 0; o < p.n_ops; ++o) {
                    const DevOp &op = H.ops[p.first + (uint32_t)o];
                    UniOp u{};
                    u.q0 = op.q;
                    if (p.type == P_CLIFF) {
                        u.kind = op.kind == K_CX ? UK_CX : UK_CZ;
                        u.q1 = op.q1;
                    } else {
                        u.kind = UK_WIRE;
                        const DevMap3 &mp = H.maps[(size_t)op.param];
                        UniRun r{(int32_t)P.ugates.size(), mp.count, parity};
                        uint32_t perm = kPermIdentity;
                        bool rotates = false;
                        for (int g = 0; g < mp.count; ++g) {
                            const RawGate rg =
                                H.raw[(size_t)H.map_gate_idx[(size_t)(mp.first + g)]];
                            parity ^= rg.op == STAB_H;
                            if (rg.op >= STAB_RX) rotates = true;
                            else if (!rotates) perm = perm_compose(perm, clifford_perm_code(rg.op));
                            P.ugates.push_back(rg);
                        }
                        r.parity |= parity << 1;
                        P.uruns.push_back(r);
                        if (!rotates && perm == kPermIdentity) P.uni_identity = true;
                        P.uni_max_run = std::max(P.uni_max_run, (int)mp.count);
                    }
                    P.uops.push_back(u);
                }
            }
            sg.n_ops = (int32_t)P.uops.size() - sg.op_first;
            sg.n_maps = (int32_t)P.uruns.size() - sg.map_first;
            sg.parity = parity;
            P.usegs.push_back(sg);
            at = end;
        }
        part.n_seg = (int32_t)P.usegs.size() - part.seg_first;
        int level = part.n_seg, root = node;
        while (level > 1) {
            root += level;
            level = (level + 1) / 2;
        }
        part.root = root;
        node = root + 1;
        P.uparts.push_back(part);
    }
    P.uni_nodes = node;
}

// Device buffers of the segments' maps and unitaries (the arrival counters
// zeroed; every launch leaves them so).  One node more than the trees hold:
// the first parts' product of a three-part plan.
int uni_buffers(stab_ctx *c) {
    DevPlan &P = c->fwd;
    const size_t E = (size_t)1 << (2 * c->n), nn = (size_t)P.uni_nodes + 1;
    RC(c->dalloc(c->umaps, std::max<size_t>(1, P.uruns.size()) * sizeof(UniMap), c->st));
    RC(c->dalloc(c->unodes, nn * (E * sizeof(double2) + 2 * sizeof(int32_t)), c->st));
    P.uargs.maps = (const UniMap *)c->umaps.p;
    P.uargs.nodes = (double2 *)c->unodes.p;
    P.uargs.node_parity = (int32_t *)(P.uargs.nodes + nn * E);
    P.uargs.node_count = P.uargs.node_parity + nn;
    CK(cudaMemsetAsync(P.uargs.node_count, 0, nn * sizeof(int32_t), c->st));
    return STAB_OK;
}

// The parts' unitaries on the context stream.
int uni_run(stab_ctx *c) {
    CK(launch_uni_segments(c->n, c->fwd.uargs, c->st));
    c->launches++;
    CK(cudaEventRecord(c->ev_tx, c->st));
    c->tx_gen = c->param_gen;
    return STAB_OK;
}

UniRoots uni_roots(const stab_ctx *c) {
    UniRoots r{};
    r.nodes = c->fwd.uargs.nodes;
    r.node_parity = c->fwd.uargs.node_parity;
    r.n = (int32_t)c->fwd.uparts.size();
    for (int k = 0; k < r.n; ++k) r.root[k] = c->fwd.uparts[(size_t)k].root;
    return r;
}

// Units of the expectation's split sweep on stream s (rebuilt when the plan
// or the observable's device terms change).
int split_units_e(stab_ctx *c, cudaStream_t s) {
    const size_t vb = c->vec_bytes();
    if (c->split_smem == 0) {
        c->split_smem = batch_smem_bytes(c->n);
        int occ = 0;
        CK(batch_occupancy(c->split_smem, &occ));
    }
    RC(c->dalloc(c->cnt, 256, s));
    RC(c->dalloc(c->rmid, vb, s));
    RC(c->dalloc(c->lmid, vb, s));
    RC(c->dalloc(c->dotbuf, 256 * sizeof(double), s));
    RC(c->dalloc(c->units_e, 2 * sizeof(BatchUnit), s));
    const int32_t nt = c->n_obs_terms;
    const std::vector<const void *> key = {(const void *)c->plan_gen, c->fwd.h1.dev,
                                           c->fwd.h2b.dev, c->terms.p, (const void *)(intptr_t)nt,
                                           c->rmid.p, c->lmid.p, c->units_e.p};
    if (key == c->key_e) return STAB_OK;
    BatchUnit U[2] = {};
    U[0].stream = c->fwd.h1.dev;
    U[0].n_chunks = c->fwd.h1.n_chunks;
    U[0].n = (int8_t)c->n;
    U[0].init = INIT_RHO0;
    U[0].out = (double *)c->rmid.p;
    U[1].stream = c->fwd.h2b.dev;
    U[1].n_chunks = c->fwd.h2b.n_chunks;
    U[1].n = (int8_t)c->n;
    U[1].init = INIT_TERMS;
    U[1].terms = (const DevTerm *)c->terms.p;
    U[1].n_terms = nt;
    U[1].out = (double *)c->lmid.p;
    CK(cudaMemcpyAsync(c->units_e.p, U, sizeof(U), cudaMemcpyHostToDevice, s));
    CK(cudaStreamSynchronize(s));
    c->key_e = key;
    return STAB_OK;
}

// A Clifford pass as one gather of its own.  One or two gates are walked per
// entry (their few index operations hide behind the loads: n = 10, random
// circuits of 107 gates 2.02 against 2.20 ms, n = 12 3.24 against 3.33), longer runs
// read through their linear map.
constexpr int kShortRun = 2;
cudaError_t launch_gather(const stab_ctx *c, const DevPlan &P, const DevPass &p, int inverse,
                          const double *src, double *dst, int n_vec, cudaStream_t s) {
    const size_t k = (size_t)(&p - P.host.passes.data());
    if (k >= P.host.pull_of.size() || (p.type == P_CLIFF && p.n_ops <= kShortRun))
        return launch_stream_cliff(src, dst, c->n, n_vec, p, P.prog.ops, inverse, s);
    return launch_stream_pull(src, dst, c->n, n_vec,
                              P.prog.pulls + 2 * P.host.pull_of[k] + (inverse ? 1 : 0), s);
}

// Streamed propagation of n_vec vectors through a plan; *cur / *alt are the
// ping-pong buffers (the result ends in *cur).  Consecutive wire passes on at
// most kTileWires wires run as one tile-fused launch (fused plans only; the
// gate-by-gate forms keep one launch per gate).
int run_streamed(stab_ctx *c, const DevPlan &P, double **cur, double **alt, int n_vec,
                 int inverse, cudaStream_t s, int k0 = 0, int k1 = -1) {
    const auto &passes = P.host.passes;
    if (k1 < 0) k1 = (int)passes.size();
    const int np = k1 - k0;   // passes [k0, k1), walked backward when inverse
    // tiles pay where a launch is small (launch-bound: few vectors, n <= 8); larger
    // launches are FP64-bound and run faster one wire per launch; the limit is
    // the path tuner's (measured per GPU model)
    const TileForm form = tile_form(c, P, n_vec);
    const bool fuse_tiles = form != kNoTiles;
    const size_t max_wires = (size_t)tile_wires(c->n);
    std::vector<const DevPass *> group;
    std::vector<int> wires;
    // with tiles, a Clifford gather is folded into the loads of the next group
    const DevPass *pending = nullptr;
    auto pull_of = [&](const DevPass *p) -> const DevPull * {
        const size_t k = (size_t)(p - passes.data());
        return k < P.host.pull_of.size() ? P.prog.pulls + 2 * P.host.pull_of[k] + (inverse ? 1 : 0)
                                         : nullptr;
    };
    auto gather_now = [&]() -> int {
        CK(launch_gather(c, P, *pending, inverse, *cur, *alt, n_vec, s));
        std::swap(*cur, *alt);
        c->launches++;
        pending = nullptr;
        return STAB_OK;
    };
    auto flush = [&]() -> int {
        if (group.empty()) return STAB_OK;
        if (!fuse_tiles) {
            CK(launch_stream_wire(*cur, c->n, n_vec, *group[0], P.prog.ops, P.prog.maps, inverse,
                                  s));
        } else {
            TileGroup tg;
            make_tile_group(c->n, n_vec, passes, group, inverse, &tg);
            double *dst = *cur;
            if (pending) {
                tg.pull = pull_of(pending);
                dst = *alt;
            }
            const bool maps = form == kTileMaps;
            CK(launch_stream_tile(*cur, dst, c->n, n_vec, tg,
                                  maps ? P.prog.pass_maps : P.prog.maps,
                                  maps ? nullptr : P.prog.ops, s));
            if (pending) {
                std::swap(*cur, *alt);
                pending = nullptr;
            }
        }
        c->launches++;
        group.clear();
        wires.clear();
        return STAB_OK;
    };
    for (int k = 0; k < np; ++k) {
        const DevPass &p = passes[inverse ? k1 - 1 - k : k0 + k];
        if (p.type == P_WIRE) {
            const bool known = std::find(wires.begin(), wires.end(), (int)p.q) != wires.end();
            if (!fuse_tiles || (int)group.size() == kTileMaxPasses ||
                (!known && wires.size() == max_wires)) {
                RC(flush());
            }
            group.push_back(&p);
            if (std::find(wires.begin(), wires.end(), (int)p.q) == wires.end())
                wires.push_back(p.q);
            continue;
        }
        RC(flush());
        if (pending) RC(gather_now());
        pending = &p;
        if (!fuse_tiles) RC(gather_now());
    }
    RC(flush());
    if (pending) RC(gather_now());
    return STAB_OK;
}

// ---------------------------------------------------------------- chains of tile steps
//
// Where a vector is small enough for tile launches (the path choice's
// tile_limit), the whole sequence of them runs as one cooperative launch.

int chain_tile_bits(int n) { return std::min(2 * n, std::max(9, 2 * tile_wires(n))); }

bool use_chain(const stab_ctx *c, const DevPlan &P, int n_vec) {
    return c->n >= kChainMinN && c->chain_ctas > 0 && !c->chains_off &&
           tile_form(c, P, n_vec) == kTileMaps;
}

// Whether generators and <O> take the chain: a cooperative launch and its
// tables cost about 7 us more than the first few launches of a graph (<O> of
// 100 gates: n = 6 67 against 59, n = 8 69 against 62; 300 gates: 100 / 100, 104 /
// 101; 1,000 gates: 210 / 244, 217 / 242), about the time of ten steps' gain;
// at n = 9 every SM has work either way and launches spread it better (300 /
// 1,000 / 3,000 gates: 178 / 465 / 1294 in a chain, 160 / 435 / 1204 launched).
// (A gradient's two chains take twice the steps and always gain.)
constexpr int kChainMinPasses = 40;
constexpr int kChainMaxN = 8;
bool use_chain_forward(const stab_ctx *c, const DevPlan &P, int n_vec) {
    return c->n <= kChainMaxN && (int)P.host.passes.size() >= kChainMinPasses &&
           use_chain(c, P, n_vec);
}

// One step of chain k: the wires' passes on src (through pull unless null) into
// dst; no passes: the gather alone.  Every step's tile has the same size.
void chain_step(const stab_ctx *c, const DevPlan &P, const std::vector<const DevPass *> &group,
                bool inverse, const DevPull *pull, const double *src, double *dst, ChainSet *C,
                int k) {
    const int n = c->n;
    std::vector<int> wires, tile, rest;
    for (const DevPass *p : group)
        if (std::find(wires.begin(), wires.end(), (int)p->q) == wires.end()) wires.push_back(p->q);
    // a gather alone: any wire's groups
    if (wires.empty()) wires.push_back(n - 1);
    tile_bits_of(n, 1, wires, 1, chain_tile_bits(n), &tile, &rest);
    auto local = [&](int bit) {
        return (int)(std::find(tile.begin(), tile.end(), bit) - tile.begin());
    };
    auto shape = [&](int wire, const DevPull *through) {
        ChainShape h{};
        bit_runs(tile, &h.tile_runs);
        bit_runs(rest, &h.rest_runs);
        h.tile_bits = (int32_t)tile.size();
        h.rest_bits = (int32_t)rest.size();
        h.wire = wire;
        h.lz = local(wire);
        h.lx = local(n + wire);
        h.pull = through;
        const std::string id((const char *)&h, sizeof(h));
        auto it = C->known.find(id);
        if (it != C->known.end()) return it->second;
        C->shapes.push_back(h);
        const int at = (int)C->shapes.size() - 1;
        C->known.emplace(id, at);
        return at;
    };
    ChainStep s{};
    s.src = src;
    s.dst = dst;
    s.pull = pull;
    s.n_pass = (int32_t)group.size();
    s.inverse = inverse;
    s.rest_bits = (int32_t)rest.size();
    for (size_t j = 0; j < group.size(); ++j) {
        s.lz[j] = (uint8_t)local(group[j]->q);
        s.lx[j] = (uint8_t)local(n + group[j]->q);
        s.map[j] = (uint32_t)(group[j] - P.host.passes.data());
    }
    const int in = group.empty() ? wires[0] : group.front()->q;
    const int out = group.empty() ? wires[0] : group.back()->q;
    for (uint32_t e = 0; e < 4; ++e) s.out_k[e] = (e & 1u) << out | (e >> 1) << (n + out);
    // the step's index comes from the unpulled wire bits of the first shape's
    // entry I, so the last wire's bits are clear in it as well
    C->host[k].push_back(s);
    C->in_shape[k].push_back(shape(in, pull));
    C->out_shape[k].push_back(shape(out, nullptr));
}

// Wire passes [p0, p1) of one block from src (through pull unless null) into dst.
void chain_block(const stab_ctx *c, const DevPlan &P, int p0, int p1, bool inverse,
                 const DevPull *pull, const double *src, double *dst, ChainSet *C, int ch) {
    const auto &passes = P.host.passes;
    std::vector<const DevPass *> group;
    std::vector<int> wires;
    for (int k = 0; k < p1 - p0; ++k) {
        const DevPass *p = &passes[(size_t)(inverse ? p1 - 1 - k : p0 + k)];
        const bool known = std::find(wires.begin(), wires.end(), (int)p->q) != wires.end();
        if ((int)group.size() == kTileMaxPasses ||
            (!known && (int)wires.size() == tile_wires(c->n))) {
            chain_step(c, P, group, inverse, pull, src, dst, C, ch);
            src = dst;
            pull = nullptr;
            group.clear();
            wires.clear();
            wires.push_back(p->q);
        } else if (!known) {
            wires.push_back(p->q);
        }
        group.push_back(p);
    }
    chain_step(c, P, group, inverse, pull, src, dst, C, ch);
}

// Passes [k0, k1) (walked backward when inverse) as steps between two buffers;
// returns the one that holds the result.
double *chain_passes(const stab_ctx *c, const DevPlan &P, double *cur, double *alt, bool inverse,
                     int k0, int k1, ChainSet *C, int ch) {
    const auto &passes = P.host.passes;
    auto pull_of = [&](int p) {
        return P.prog.pulls + 2 * P.host.pull_of[(size_t)p] + (inverse ? 1 : 0);
    };
    int pending = -1;
    auto gather = [&]() {
        chain_step(c, P, {}, inverse, pull_of(pending), cur, alt, C, ch);
        std::swap(cur, alt);
    };
    for (int k = 0; k < k1 - k0;) {
        const int p = inverse ? k1 - 1 - k : k0 + k;
        if (passes[(size_t)p].type != P_WIRE) {
            if (pending >= 0) gather();
            pending = p;
            ++k;
            continue;
        }
        int m = 0;   // the block's wire passes
        while (k + m < k1 - k0 && passes[(size_t)(inverse ? p - m : p + m)].type == P_WIRE) ++m;
        double *dst = pending >= 0 ? alt : cur;
        chain_block(c, P, inverse ? p - m + 1 : p, inverse ? p + 1 : p + m, inverse,
                    pending >= 0 ? pull_of(pending) : nullptr, cur, dst, C, ch);
        if (pending >= 0) std::swap(cur, alt);
        pending = -1;
        k += m;
    }
    if (pending >= 0) gather();
    return cur;
}

// Builds the shapes' tables, uploads both chains' steps (on s) and sizes their
// CTAs: one per tile, as far as max_ctas allows for all chains together.
int chain_upload(stab_ctx *c, ChainSet &C, const std::vector<const void *> &key,
                 const DevPlan &P, int n_vec, int max_ctas, cudaStream_t s) {
    const size_t n0 = C.host[0].size(), n1 = C.host[1].size(), ns = C.shapes.size();
    const size_t groups = (size_t)1 << (chain_tile_bits(c->n) - 2);
    const size_t tiles = (size_t)1 << (2 * c->n - chain_tile_bits(c->n));
    const size_t per = groups * sizeof(uint2) + 4 * tiles * sizeof(uint4);
    const size_t b_shapes = align256(ns * sizeof(ChainShape));
    const size_t b_steps = align256((n0 + n1) * sizeof(ChainStep));
    RC(c->dalloc(C.tables, b_shapes + ns * per, s));
    RC(c->dalloc(C.dev, b_steps + 256 + 2 * 128, s));
    char *base = (char *)C.tables.p + b_shapes;
    for (size_t k = 0; k < ns; ++k) {
        C.shapes[k].tiles = (uint4 *)(base + k * per);
        C.shapes[k].threads = (uint2 *)(base + k * per + 4 * tiles * sizeof(uint4));
    }
    ChainStep *d = (ChainStep *)C.dev.p;
    C.desc_dev = (const ChainDesc *)((char *)C.dev.p + b_steps);
    C.arrived = (uint32_t *)((char *)C.dev.p + b_steps + 256);
    C.n_chains = C.grid = 0;
    for (int k = 0; k < 2; ++k) {
        std::vector<ChainStep> &H = C.host[k];
        if (H.empty()) continue;
        for (size_t i = 0; i < H.size(); ++i) {
            const ChainShape &in = C.shapes[(size_t)C.in_shape[k][i]];
            H[i].in_threads = in.threads;
            H[i].tiles = in.tiles;
            H[i].out_threads = C.shapes[(size_t)C.out_shape[k][i]].threads;
        }
        ChainDesc e{};
        e.steps = d + (k ? n0 : 0);
        e.maps = P.prog.pass_maps;
        e.arrived = C.arrived + 32 * C.n_chains;
        e.n_steps = (int32_t)H.size();
        e.n = c->n;
        e.n_vec = n_vec;
        e.cta0 = C.grid;
        e.ctas = (int32_t)std::min<int64_t>((int64_t)n_vec * (int64_t)tiles,
                                            std::max(1, max_ctas / (n0 && n1 ? 2 : 1)));
        C.grid += e.ctas;
        C.desc[C.n_chains++] = e;
    }
    C.alone = n_vec == 1 && tiles == 1;
    // as on the device: steps, descriptors; then the shapes
    char *h = nullptr;
    RC(c->aux_stage.take(b_steps + 256 + b_shapes, false, &h));
    std::copy(C.host[0].begin(), C.host[0].end(), (ChainStep *)h);
    std::copy(C.host[1].begin(), C.host[1].end(), (ChainStep *)h + n0);
    std::memcpy(h + b_steps, C.desc, sizeof(C.desc));
    std::copy(C.shapes.begin(), C.shapes.end(), (ChainShape *)(h + b_steps + 256));
    CK(cudaMemcpyAsync(C.dev.p, h, b_steps + 256, cudaMemcpyHostToDevice, s));
    if (ns)
        CK(cudaMemcpyAsync(C.tables.p, h + b_steps + 256, ns * sizeof(ChainShape),
                           cudaMemcpyHostToDevice, s));
    RC(c->aux_stage.mark(s));
    CK(launch_chain_tables((const ChainShape *)C.tables.p, (int)ns, c->n, s));
    c->launches += ns > 0;
    C.key = key;
    return STAB_OK;
}

int chain_run(stab_ctx *c, const ChainSet &C, cudaStream_t s) {
    if (C.n_chains == 0) return STAB_OK;
    ChainArgs a{};
    a.chains = C.desc_dev;
    a.n_chains = C.n_chains;
    a.grid = C.grid;
    a.tile_bits = chain_tile_bits(c->n);
    a.alone = C.alone;
    a.status = (int32_t *)c->status.p;
    CK(cudaMemsetAsync(C.arrived, 0, 256, s));
    CK(launch_stream_chain(a, s));
    c->launches++;
    return STAB_OK;
}

// <O> as two chains that meet at half the passes: O backward (from lam), rho_0
// forward (from lam2).
int expect_chains(stab_ctx *c, const std::vector<const void *> &key, int max_ctas,
                  cudaStream_t s) {
    ChainSet &C = c->c_expect;
    const int np = (int)c->fwd.host.passes.size(), mid = np / 2;
    C.clear();
    C.result[0] = chain_passes(c, c->fwd, (double *)c->lam.p, (double *)c->tmp.p, true, mid, np,
                               &C, 0);
    C.result[1] = chain_passes(c, c->fwd, (double *)c->lam2.p, (double *)c->tmp3.p, false, 0, mid,
                               &C, 1);
    return chain_upload(c, C, key, c->fwd, 1, max_ctas, s);
}

int expect_fill(stab_ctx *c, cudaStream_t s) {
    const int32_t nt = c->n_obs_terms;
    CK(launch_fill((double *)c->lam.p, c->n, 1, INIT_TERMS, (const DevTerm *)c->terms.p, nt, s));
    CK(launch_fill((double *)c->lam2.p, c->n, 1, INIT_RHO0, nullptr, 0, s));
    c->launches += (nt ? 2 : 1) + 1;
    return STAB_OK;
}

// Replays the launch sequence `body` (queued on s) from a graph cached under
// `key`, capturing it first when the key changed.  s is the context's own
// non-blocking stream (the legacy default stream cannot be captured).  All
// buffers the body uses must be allocated before the call.
template <class F>
int run_graph(stab_ctx *c, GraphCache &g, const std::vector<const void *> &key, cudaStream_t s,
              F body) {
    if (!(g.exec && g.key == key) && g.seen != key) {
        // First run of this sequence: launched directly.  A sequence that is
        // run once (a served request, a one-off circuit) would only pay for
        // capturing and instantiating a graph; it is captured when it comes
        // again.
        if (g.exec) g.reset();
        const int rc = body(s, &g.result);
        if (rc != STAB_OK) return rc;
        g.seen = key;
        return STAB_OK;
    }
    if (!g.exec || g.key != key) {
        g.reset();
        cudaGraph_t graph = nullptr;
        const int64_t l0 = c->launches;
        CK(cudaStreamBeginCapture(s, cudaStreamCaptureModeThreadLocal));
        const int rc = body(s, &g.result);
        cudaError_t e = cudaStreamEndCapture(s, &graph);
        g.launches = c->launches - l0;
        c->launches = l0;
        if (rc != STAB_OK || e != cudaSuccess) {
            if (graph) cudaGraphDestroy(graph);
            g.reset();
            if (rc != STAB_OK) return rc;
            CK(e);
        }
        e = cudaGraphInstantiate(&g.exec, graph, 0);
        cudaGraphDestroy(graph);
        if (e != cudaSuccess) g.reset();
        CK(e);
        g.key = key;
    }
    CK(cudaGraphLaunch(g.exec, s));
    c->launches += g.launches;
    return STAB_OK;
}

void reset_graphs(stab_ctx *c) {
    c->g_gens.reset();
    c->g_expect.reset();
    c->g_grad.reset();
    c->plan_gen++;
}

// The pass of plan B that starts the unit starting at pass k of plan A, or -1
// when pass k starts no unit or the two plans' unit sequences differ (a run
// that is the identity and holds no rotation makes no pass in some modes).
// (stab_selftest_align; the gradient's uni_identity is the same condition.)
int aligned_pass(const HostPlan &A, int k, const HostPlan &B) {
    if (k <= 0 || k >= (int)A.passes.size() || !unit_start(A, (size_t)k)) return -1;
    // the units of both plans, as (type, wire), in order; the first pass of each in B
    std::vector<uint16_t> ua, ub;
    std::vector<int> start_b;
    int unit_k = -1;
    for (size_t i = 0; i < A.passes.size(); ++i)
        if (unit_start(A, i)) {
            if ((int)i == k) unit_k = (int)ua.size();
            ua.push_back((uint16_t)(A.passes[i].type << 8 | A.passes[i].q));
        }
    for (size_t i = 0; i < B.passes.size(); ++i)
        if (unit_start(B, i)) {
            ub.push_back((uint16_t)(B.passes[i].type << 8 | B.passes[i].q));
            start_b.push_back((int)i);
        }
    if (ua != ub || unit_k < 0) return -1;
    return start_b[(size_t)unit_k];
}

// The gradient of a plan with segment unitaries: only the slot -> rotations
// table (rotations by their place in the run-ordered gate array).
bool uni_grad_ok(const stab_ctx *c) {
    return c->use_resident() && c->use_resident_adjoint() && c->fwd.uni;
}

// Slot -> rotations, each by its place in the run-ordered gate array.
void slot_table(const std::vector<RawGate> &g, int64_t n_params, HostPlan *H) {
    H->param_ptr.assign((size_t)n_params + 1, 0);
    for (const RawGate &r : g)
        if (r.op >= STAB_RX) H->param_ptr[(size_t)r.param + 1]++;
    for (int64_t j = 0; j < n_params; ++j)
        H->param_ptr[(size_t)j + 1] += H->param_ptr[(size_t)j];
    H->param_rot.resize((size_t)H->param_ptr[(size_t)n_params]);
    std::vector<int32_t> at(H->param_ptr.begin(), H->param_ptr.end() - 1);
    for (size_t k = 0; k < g.size(); ++k)
        if (g[k].op >= STAB_RX) H->param_rot[(size_t)at[(size_t)g[k].param]++] = (int32_t)k;
}

int ensure_uni_grad(stab_ctx *c) {
    if (c->grad.built) return STAB_OK;
    c->grad.host = HostPlan();
    slot_table(c->fwd.ugates, c->n_params, &c->grad.host);
    no_streams(c->grad);
    RC(upload_plan(c, c->grad));
    c->grad.encoded = true;
    CK(cudaEventRecord(c->ev_ready, c->st));
    return STAB_OK;
}

// ---------------------------------------------------------------- gradients from stored sweeps
//
// Streamed gradients (n >= 5).  rho goes forward through the whole plan and
// lambda backward through it, each a chain of its own launches at once on two
// streams, and every block of wire passes leaves its result in a slot of its
// own; one launch then takes the three numbers c of every wire run from the
// two vectors at its block's end (k_grad_dots), one turns them into the
// rotations' derivatives.  Against carrying (lambda, rho) pairs from the
// middle to both ends with every rotation's dot on the way: two sweeps of a
// vector instead of three, six FMAs a group and run instead of three a
// rotation, off the sequential chain, and runs of any length composed.

const DevPlan &ck_plan(const stab_ctx *c) {
    return !c->use_resident() && c->fwd.host.mode == PLAN_FUSED ? c->fwd : c->ck;
}

// The blocks, runs and jobs of the plan (host side, once per circuit).
int ck_build(stab_ctx *c) {
    const int n = c->n;
    const bool own = &ck_plan(c) == &c->ck;
    no_streams(c->ck);
    if (own)
        build_plan(n, c->gates.data(), (int64_t)c->gates.size(), c->n_params, PLAN_FUSED,
                   &c->ck.host, true);
    else
        c->ck.host = HostPlan();
    const HostPlan &H = ck_plan(c).host;
    c->ck_blocks.clear();
    c->ck_after.clear();
    c->ck_jobs.clear();
    c->ck_job_block.clear();
    std::vector<RawGate> &gates = c->ck.ugates;
    std::vector<int> between;
    const int np = (int)H.passes.size();
    c->ck.uni_max_run = 0;
    for (int p = 0; p < np;) {
        if (H.passes[(size_t)p].type != P_WIRE) {
            between.push_back(p++);
            continue;
        }
        stab_ctx::CkBlock b;
        b.p0 = p;
        b.before.swap(between);
        std::vector<std::vector<int32_t>> wire((size_t)n);
        for (; p < np && H.passes[(size_t)p].type == P_WIRE; ++p) {
            std::vector<int32_t> &w = wire[H.passes[(size_t)p].q];
            w.insert(w.end(), H.run_gates.begin() + H.run_first[(size_t)p],
                     H.run_gates.begin() + H.run_first[(size_t)p + 1]);
        }
        b.p1 = p;
        // a run per wire that holds a rotation, a job per tile_wires of them
        std::vector<int> wires, runs;
        auto flush = [&]() {
            if (wires.empty()) return;
            DotJob J{};
            std::vector<int> tile, rest;
            tile_bits_of(n, 1, wires, 1, std::min(kTileMaxBits, 2 * n), &tile, &rest);
            J.n_wires = (int32_t)wires.size();
            J.tile_bits = (int32_t)tile.size();
            J.rest_bits = (int32_t)rest.size();
            for (size_t w = 0; w < wires.size(); ++w) {
                J.run[w] = runs[w];
                J.lz[w] = (uint8_t)(std::find(tile.begin(), tile.end(), wires[w]) - tile.begin());
                J.lx[w] =
                    (uint8_t)(std::find(tile.begin(), tile.end(), n + wires[w]) - tile.begin());
            }
            bit_runs(tile, &J.tile_runs);
            bit_runs(rest, &J.rest_runs);
            c->ck_jobs.push_back(J);
            c->ck_job_block.push_back((int)c->ck_blocks.size());
            wires.clear();
            runs.clear();
        };
        for (int q = 0; q < n; ++q) {
            bool rotates = false;
            for (int32_t g : wire[(size_t)q]) rotates |= c->gates[(size_t)g].op >= STAB_RX;
            if (!rotates) continue;
            UniRun r{(int32_t)gates.size(), (int32_t)wire[(size_t)q].size(), 0};
            for (int32_t g : wire[(size_t)q]) {
                const stab_gate &s = c->gates[(size_t)g];
                gates.push_back({s.op, s.q0, s.q1, s.flags, s.param});
            }
            c->ck.uni_max_run = std::max(c->ck.uni_max_run, (int)r.count);
            wires.push_back(q);
            runs.push_back((int)c->ck.uruns.size());
            c->ck.uruns.push_back(r);
            if ((int)wires.size() == tile_wires(n)) flush();
        }
        flush();
        c->ck_blocks.push_back(std::move(b));
    }
    c->ck_after = std::move(between);
    const int64_t tiles = (int64_t)1 << std::max(0, 2 * n - kTileMaxBits);
    const int64_t want = 16 * (int64_t)c->sms / std::max<int64_t>(1, (int64_t)c->ck_jobs.size()) + 1;
    c->ck_chunks = (int)std::min<int64_t>(std::min<int64_t>(64, tiles), want);
    HostPlan &K = c->ck.host;
    if (!own) K.mode = PLAN_FUSED;
    slot_table(gates, c->n_params, &K);
    RC(upload_plan(c, c->ck));
    c->ck.encoded = false;
    c->ck_ready = true;
    c->key_ck.clear();
    c->g_grad.reset();
    c->plan_gen++;
    return STAB_OK;
}

// Slots of 4^n doubles: [0, B) rho at the end of each block, [B, 2 B) lambda at
// its start, two spares of each chain, O, and one more wherever lambda passes
// several Clifford passes in a row (the dots read it between them).
constexpr size_t kCkSpares = 5;
size_t ck_slots(const stab_ctx *c) {
    size_t extra = kCkSpares;
    for (const auto &b : c->ck_blocks) extra += b.before.size() > 1 ? b.before.size() - 1 : 0;
    extra += c->ck_after.size() > 1 ? c->ck_after.size() - 1 : 0;
    return 2 * c->ck_blocks.size() + extra;
}

// Whether the streamed gradient runs from stored sweeps: a circuit with
// rotations whose slots fit (and could be allocated); else the pair sweep.
bool ck_usable(stab_ctx *c, int *rc) {
    *rc = STAB_OK;
    if (c->ck_off || c->ck_bytes_max == 0 || c->n_params == 0) return false;
    if (!c->ck_ready) *rc = ck_build(c);
    if (*rc != STAB_OK) return false;
    const size_t bytes = ck_slots(c) * c->vec_bytes();
    c->ck_off = c->ck_blocks.empty() || bytes > c->ck_bytes_max;
    if (c->ck_off) return false;
    const int room = c->dalloc(c->ckslots, bytes, c->aux);
    if (room == STAB_OK) return true;
    (void)cudaGetLastError();
    if (c->ck_must) *rc = room;
    else c->ck_off = true;
    return false;
}

// One block's wire passes from src (through Clifford pass `gather` unless
// negative) into dst, a launch each.
int ck_block(stab_ctx *c, const DevPlan &G, const stab_ctx::CkBlock &b, bool inverse,
             const double *src, int gather, double *dst, cudaStream_t s) {
    const int n = c->n, np = b.p1 - b.p0;
    if (gather >= 0) {
        CK(launch_gather(c, G, G.host.passes[(size_t)gather], inverse, src, dst, 1, s));
        c->launches++;
    } else if (src != dst) {
        CK(cudaMemcpyAsync(dst, src, c->vec_bytes(), cudaMemcpyDeviceToDevice, s));
    }
    for (int k = 0; k < np; ++k)
        CK(launch_stream_wire(dst, n, 1, G.host.passes[(size_t)(inverse ? b.p1 - 1 - k : b.p0 + k)],
                              G.prog.ops, G.prog.maps, inverse, s));
    c->launches += np;
    return STAB_OK;
}

// Clifford passes between block b and the next one (or the end).
const std::vector<int> &ck_between(const stab_ctx *c, int b) {
    return b + 1 < (int)c->ck_blocks.size() ? c->ck_blocks[(size_t)b + 1].before : c->ck_after;
}

// The jobs' pointers into the slots, uploaded on s: block b's dots read lambda
// through the first Clifford pass after the block.
int ck_upload_jobs(stab_ctx *c, cudaStream_t s) {
    const DevPlan &G = ck_plan(c);
    const int B = (int)c->ck_blocks.size();
    const double *slots = (const double *)c->ckslots.p;
    const size_t E = (size_t)1 << (2 * c->n);
    RC(c->dalloc(c->ckjobs, std::max<size_t>(1, c->ck_jobs.size()) * sizeof(DotJob), s));
    const std::vector<const void *> key = {(const void *)c->plan_gen, slots, G.prog.pulls,
                                           c->ckjobs.p};
    if (key == c->key_ck || c->ck_jobs.empty()) return STAB_OK;
    std::vector<size_t> src((size_t)B);
    size_t extra = 2 * (size_t)B + kCkSpares;
    for (int b = B - 1; b >= 0; --b) {
        const size_t m = ck_between(c, b).size();
        src[(size_t)b] = b == B - 1 ? 2 * (size_t)B + 4 : (size_t)(B + b + 1);
        if (m > 1) {
            extra += m - 1;
            src[(size_t)b] = extra - 1;
        }
    }
    for (size_t k = 0; k < c->ck_jobs.size(); ++k) {
        const int b = c->ck_job_block[k];
        const std::vector<int> &between = ck_between(c, b);
        DotJob &J = c->ck_jobs[k];
        J.rho = slots + (size_t)b * E;
        J.lam = slots + src[(size_t)b] * E;
        J.pull = between.empty() ? nullptr
                                 : G.prog.pulls + 2 * G.host.pull_of[(size_t)between[0]] + 1;
    }
    const size_t bytes = c->ck_jobs.size() * sizeof(DotJob);
    char *h = nullptr;
    RC(c->aux_stage.take(bytes, false, &h));
    std::memcpy(h, c->ck_jobs.data(), bytes);
    CK(cudaMemcpyAsync(c->ckjobs.p, h, bytes, cudaMemcpyHostToDevice, s));
    RC(c->aux_stage.mark(s));
    c->key_ck = key;
    return STAB_OK;
}

// The stored sweeps as two chains of steps: rho forward, lambda backward (the
// slots as in ck_gradient).
int ck_chains(stab_ctx *c, cudaStream_t s) {
    const DevPlan &G = ck_plan(c);
    const int B = (int)c->ck_blocks.size();
    const size_t E = (size_t)1 << (2 * c->n), at = 2 * (size_t)B;
    auto slot = [&](size_t k) { return (double *)c->ckslots.p + k * E; };
    auto pull = [&](int p, bool inverse) {
        return G.prog.pulls + 2 * G.host.pull_of[(size_t)p] + (inverse ? 1 : 0);
    };
    ChainSet &C = c->c_grad;
    const std::vector<const void *> key = {(const void *)c->plan_gen, c->ckslots.p, G.buf.p};
    if (C.key == key) return STAB_OK;
    C.clear();
    double *cur = c->ck_blocks[0].before.empty() ? slot(0) : slot(at);
    for (int b = 0; b < B; ++b) {
        const auto &blk = c->ck_blocks[(size_t)b];
        for (size_t k = 0; k + 1 < blk.before.size(); ++k) {
            double *to = cur == slot(at) ? slot(at + 1) : slot(at);
            chain_step(c, G, {}, false, pull(blk.before[k], false), cur, to, &C, 0);
            cur = to;
        }
        chain_block(c, G, blk.p0, blk.p1, false,
                    blk.before.empty() ? nullptr : pull(blk.before.back(), false), cur,
                    slot((size_t)b), &C, 0);
        cur = slot((size_t)b);
    }
    cur = slot(at + 4);
    size_t extra = at + kCkSpares;
    for (int b = B - 1; b >= 0; --b) {
        const auto &blk = c->ck_blocks[(size_t)b];
        const std::vector<int> &between = ck_between(c, b);
        for (size_t k = between.size(); k-- > 1;) {
            chain_step(c, G, {}, true, pull(between[k], true), cur, slot(extra), &C, 1);
            cur = slot(extra++);
        }
        chain_block(c, G, blk.p0, blk.p1, true, between.empty() ? nullptr : pull(between[0], true),
                    cur, slot((size_t)(B + b)), &C, 1);
        cur = slot((size_t)(B + b));
    }
    const std::vector<int> &lead = c->ck_blocks[0].before;
    for (size_t k = lead.size(); k-- > 0;) {
        double *to = cur == slot(at + 2) ? slot(at + 3) : slot(at + 2);
        chain_step(c, G, {}, true, pull(lead[k], true), cur, to, &C, 1);
        cur = to;
    }
    C.result[1] = cur;
    return chain_upload(c, C, key, G, 1, c->chain_ctas, s);
}

// The runs' numbers and the derivatives from the slots.
int ck_finish(stab_ctx *c, cudaStream_t gs) {
    CK(launch_grad_dots((const DotJob *)c->ckjobs.p, (int)c->ck_jobs.size(), c->n, c->ck_chunks,
                        (double *)c->ckdots.p, gs));
    CK(launch_run_grads(c->ck.uruns_dev, (int)c->ck.uruns.size(), c->ck.uni_max_run,
                        c->ck.ugates_dev, (const double *)c->thetas.p, (const double *)c->ckdots.p,
                        c->ck_chunks, (double *)c->grad_rot.p, gs));
    CK(launch_gather_grads((const double *)c->grad_rot.p, c->ck.param_ptr, c->ck.param_rot,
                           (int)c->n_params, (double *)c->gbuf.p, gs));
    c->launches += 2 + !c->ck_jobs.empty();
    return STAB_OK;
}

// The launches of a gradient from stored sweeps, queued on gs (and aux2).
int ck_gradient(stab_ctx *c, double *res, cudaStream_t gs) {
    const DevPlan &G = ck_plan(c);
    const int n = c->n, B = (int)c->ck_blocks.size();
    const size_t E = (size_t)1 << (2 * n), at = 2 * (size_t)B;
    auto slot = [&](size_t k) { return (double *)c->ckslots.p + k * E; };
    auto gather = [&](const double *from, double *to, int p, bool inverse,
                      cudaStream_t s) -> int {
        CK(launch_gather(c, G, G.host.passes[(size_t)p], inverse, from, to, 1, s));
        c->launches++;
        return STAB_OK;
    };
    auto block = [&](int b, bool inverse, const double *from, int p, double *to,
                     cudaStream_t s) -> int {
        return ck_block(c, G, c->ck_blocks[(size_t)b], inverse, from, p, to, s);
    };
    if (use_chain(c, G, 1)) {
        RC(ck_chains(c, gs));
        const double *lam0 = c->c_grad.result[1];
        CK(launch_fill(c->ck_blocks[0].before.empty() ? slot(0) : slot(at), n, 1, INIT_RHO0,
                       nullptr, 0, gs));
        CK(launch_fill(slot(at + 4), n, 1, INIT_TERMS, (const DevTerm *)c->terms.p,
                       c->n_obs_terms, gs));
        RC(chain_run(c, c->c_grad, gs));
        CK(launch_xfree_sum(lam0, n, 1, res, gs));
        c->launches += (c->n_obs_terms ? 3 : 2) + 1;
        return ck_finish(c, gs);
    }
    CK(cudaEventRecord(c->ev_fork, gs));
    CK(cudaStreamWaitEvent(c->aux2, c->ev_fork, 0));
    // rho forward
    double *cur = c->ck_blocks[0].before.empty() ? slot(0) : slot(at);
    CK(launch_fill(cur, n, 1, INIT_RHO0, nullptr, 0, gs));
    c->launches++;
    for (int b = 0; b < B; ++b) {
        const std::vector<int> &before = c->ck_blocks[(size_t)b].before;
        for (size_t k = 0; k + 1 < before.size(); ++k) {
            double *to = cur == slot(at) ? slot(at + 1) : slot(at);
            RC(gather(cur, to, before[k], false, gs));
            cur = to;
        }
        RC(block(b, false, cur, before.empty() ? -1 : before.back(), slot((size_t)b), gs));
        cur = slot((size_t)b);
    }
    // lambda backward
    cudaStream_t s2 = c->aux2;
    cur = slot(at + 4);
    CK(launch_fill(cur, n, 1, INIT_TERMS, (const DevTerm *)c->terms.p, c->n_obs_terms, s2));
    c->launches += c->n_obs_terms ? 2 : 1;
    size_t extra = at + kCkSpares;
    for (int b = B - 1; b >= 0; --b) {
        const std::vector<int> &between = ck_between(c, b);
        for (size_t k = between.size(); k-- > 1;) {
            RC(gather(cur, slot(extra), between[k], true, s2));
            cur = slot(extra++);
        }
        RC(block(b, true, cur, between.empty() ? -1 : between[0], slot((size_t)(B + b)), s2));
        cur = slot((size_t)(B + b));
    }
    // <O> = the x-free sum of lambda at the circuit's start
    const std::vector<int> &lead = c->ck_blocks[0].before;
    for (size_t k = lead.size(); k-- > 0;) {
        double *to = cur == slot(at + 2) ? slot(at + 3) : slot(at + 2);
        RC(gather(cur, to, lead[k], true, s2));
        cur = to;
    }
    CK(launch_xfree_sum(cur, n, 1, res, s2));
    c->launches++;
    CK(cudaEventRecord(c->ev_join, c->aux2));
    CK(cudaStreamWaitEvent(gs, c->ev_join, 0));
    return ck_finish(c, gs);
}

int ensure_grad_plan(stab_ctx *c) {
    if (!c->grad.built) {
        build_plan(c->n, c->gates.data(), (int64_t)c->gates.size(), c->n_params, PLAN_GRAD,
                   &c->grad.host, !c->use_resident_adjoint());
        // resident adjoint: split at half the passes (the AUTO kernel; the
        // RESIDENT choice keeps the single-CTA forward-then-reverse sweep)
        if (c->use_resident_adjoint()) {
            make_streams(c->grad, c->kernel == STAB_KERNEL_AUTO ? 0.5 : 0.0, true);
        } else {
            no_streams(c->grad);
        }
        c->g_grad.reset();
        c->plan_gen++;
        RC(upload_plan(c, c->grad));
    }
    if (!c->grad.encoded) RC(encode_plan(c, c->grad));
    if (!c->grad.streams) {
        // the pair sweep reads the ops, the first phase tiles where it may
        RC(stream_ops(c, c->grad));
        RC(stream_encode(c, c->grad, 1));
    }
    CK(cudaEventRecord(c->ev_ready, c->st));
    return STAB_OK;
}

}  // namespace

cudaStream_t stab::ctx_stream(stab_ctx *c) { return c ? c->st : nullptr; }
void stab::ctx_checkpoint_limit(stab_ctx *c, size_t bytes) {
    if (!c) return;
    c->ck_bytes_max = std::min(bytes, kCheckpointBytes);
    c->ck_must = bytes > 0;
}
void stab::ctx_allow_chains(stab_ctx *c, bool on) {
    if (c) c->chains_off = !on;
}
stab::PlanCount::PlanCount(const stab_gate *gates, int64_t m) {
    bool two = true, run_two = false;
    int64_t run = 0, pairs = 0;
    // a long run of single-qubit Clifford gates may become a gather inside its block
    auto end_run = [&]() {
        if (run >= 8) {
            ++ranges;
            blocks += !run_two;
            cliffs += !run_two;
        }
        run = 0;
        run_two = false;
    };
    for (int64_t i = 0; i < m; ++i) {
        const bool t = gates[i].op == STAB_CX || gates[i].op == STAB_CZ;
        if (t && (!two || i == 0)) ++cliffs;
        if (!t && two) ++blocks;
        two = t;
        pairs += t;
        if (gates[i].op >= STAB_RX) end_run();
        else ++run;
        run_two |= t;
    }
    end_run();
    cliffs += (size_t)(pairs / 65535);   // gates of a pass at most
    ranges += (size_t)(m / 16384);
}

size_t stab::checkpoint_bound(int n, const PlanCount &k) {
    // a slot more than ck_slots per Clifford pass at most
    const size_t bytes = (2 * k.blocks + k.cliffs + kCkSpares) * (sizeof(double) << (2 * n));
    return bytes <= kCheckpointBytes ? bytes : 0;
}
size_t stab::chain_bound(int n, const PlanCount &k, bool grad) {
    // the largest n whose vectors the path tuner gives to tiles; <O> see use_chain_forward
    if (n < kChainMinN || n > (grad ? 9 : kChainMaxN)) return 0;
    const size_t per_block = (size_t)((n + tile_wires(n) - 1) / tile_wires(n));
    const size_t dirs = grad ? 2 : 1;   // <O>: two chains of half the plan
    const size_t steps = dirs * ((k.blocks + k.ranges) * per_block + k.cliffs + 2);
    // shapes: one per wire set and first (or last) wire, and one per gather read through
    size_t sets = 0, choose = 1;
    for (int w = 1; w <= tile_wires(n); ++w) {
        choose = choose * (size_t)(n - w + 1) / (size_t)w;
        sets += choose * (size_t)w;
    }
    const size_t shapes = dirs * (k.blocks + k.cliffs + 2) + std::min(sets, 2 * steps);
    const size_t groups = (size_t)1 << (chain_tile_bits(n) - 2);
    const size_t tiles = (size_t)1 << (2 * n - chain_tile_bits(n));
    return steps * sizeof(ChainStep) +
           shapes * (sizeof(ChainShape) + groups * sizeof(uint2) + 4 * tiles * sizeof(uint4));
}
size_t stab::ctx_trim(stab_ctx *c, size_t keep) {
    if (!c) return 0;
    auto held = [&]() {
        size_t sum = c->ckslots.bytes;
        for (const ChainSet *C : {&c->c_gens, &c->c_expect, &c->c_grad})
            sum += C->tables.bytes + C->dev.bytes;
        return sum;
    };
    if (held() > keep) {
        c->dfree(c->ckslots, c->aux);
        c->key_ck.clear();
        c->c_grad.key.clear();
        c->g_grad.reset();
    }
    if (held() > keep)
        for (ChainSet *C : {&c->c_gens, &c->c_expect, &c->c_grad}) {
            c->dfree(C->tables, c->aux);
            c->dfree(C->dev, c->aux);
            C->clear();
        }
    return held();
}

extern "C" {

void stab_default_opts(stab_opts *o) {
    if (!o) return;
    std::memset(o, 0, sizeof(*o));
    o->device = -1;
    o->kernel = STAB_KERNEL_AUTO;
    o->fuse = 1;
}

int stab_version(void) { return STAB_VERSION; }

namespace {

// What a kernel applies from a stream, in order: every pull record (last
// listed first), then, for a pass with ops, its header (pull count cleared)
// and its op records.  False when the stream is malformed (a record that is
// not a header where one is due, a pass straddling a chunk, no R_END) or its
// encoded positions are not those of its R_ROT / R_MAP3 records.
bool stream_actions(const std::vector<Rec> &s, const std::vector<int32_t> &enc,
                    std::vector<Rec> *out) {
    std::vector<int32_t> pos;
    size_t r = 0;
    while (r < s.size()) {
        const Rec &h = s[r];
        if (h.kind == R_END) return pos == enc;
        if (h.kind == R_NEXT) {
            r = (r / kChunkRecs + 1) * kChunkRecs;
            continue;
        }
        const size_t len = 1 + (size_t)h.param + (size_t)h.gate;
        if (h.kind != R_PASS || h.param < 0 || h.gate < 0 ||
            r / kChunkRecs != (r + len - 1) / kChunkRecs || r + len > s.size())
            return false;
        for (int k = h.param; k > 0; --k) out->push_back(s[r + (size_t)k]);
        if (h.gate > 0) {
            Rec hh = h;
            hh.param = 0;
            hh.code = 0;   // the repeated-pull hint is not an action
            out->push_back(hh);
            for (int k = 0; k < h.gate; ++k) {
                const size_t i = r + 1 + (size_t)h.param + (size_t)k;
                if (s[i].kind == R_ROT || s[i].kind == R_MAP3) pos.push_back((int32_t)i);
                out->push_back(s[i]);
            }
        }
        r += len;
    }
    return false;
}

// Every pass header of a one-piece stream carries kPullRepeat exactly when
// its pull records equal those of the previous pull pass.
bool pull_repeat_flags_exact(const std::vector<Rec> &s) {
    std::vector<Rec> last;
    size_t r = 0;
    while (r < s.size()) {
        const Rec &h = s[r];
        if (h.kind == R_END) return true;
        if (h.kind == R_NEXT) {
            r = (r / kChunkRecs + 1) * kChunkRecs;
            continue;
        }
        if (h.kind != R_PASS || h.param < 0 || h.gate < 0) return false;
        if (h.param > 0) {
            bool same = (size_t)h.param == last.size();
            for (int k = 0; same && k < h.param; ++k) {
                const Rec &p = s[r + 1 + (size_t)k];
                same = p.kind == last[(size_t)k].kind && p.q == last[(size_t)k].q &&
                       p.q1 == last[(size_t)k].q1;
            }
            if (same != (h.code == kPullRepeat)) return false;
            last.assign(s.begin() + (long)r + 1, s.begin() + (long)r + 1 + h.param);
        } else if (h.code != 0) {
            return false;
        }
        r += 1 + (size_t)h.param + (size_t)h.gate;
    }
    return false;
}

}  // namespace

int stab_selftest_plan(int n, const stab_gate *gates, int64_t m, int64_t n_params, int mode) {
    if (n < 1 || n > STAB_MAX_QUBITS) return STAB_E_RANGE;
    if (mode < 0 || mode > 3) return STAB_E_RANGE;
    std::string msg;
    RC(validate_gates(n, gates, m, n_params, &msg));
    const PlanMode pm = mode == 0 ? PLAN_FUSED : mode == 1 ? PLAN_GRAD : mode == 2 ? PLAN_PLAIN
                                                                               : PLAN_ROWS;
    HostPlan a, b;
    build_plan(n, gates, m, n_params, pm, &a, false, true);
    build_plan(n, gates, m, n_params, pm, &b, false, false);
    auto same = [](const auto &x, const auto &y) {
        return x.size() == y.size() &&
               (x.empty() || std::memcmp(x.data(), y.data(), x.size() * sizeof(x[0])) == 0);
    };
    bool ok = same(a.passes, b.passes) && same(a.ops, b.ops) && same(a.maps, b.maps) &&
              same(a.map_gate_idx, b.map_gate_idx) && same(a.raw, b.raw) &&
              same(a.param_ptr, b.param_ptr) && same(a.param_rot, b.param_rot) &&
              a.n_rot == b.n_rot;
    for (bool backward : {false, true}) {
        std::vector<Rec> sa, sb;
        build_stream(a, backward, &sa);
        build_stream(b, backward, &sb);
        ok = ok && same(sa, sb) && pull_repeat_flags_exact(sa);
    }
    // one-piece against two-piece streams, compared as what a kernel applies:
    // pulls in application order, passes with ops (identity passes only pull)
    DevPlan P;
    P.host = std::move(b);
    const int np = (int)P.host.passes.size();
    for (bool backward : {false, true}) {
        DevStreamBuf one, two;
        build_streams(P, {{&one, backward, 0, np}}, false);
        build_streams(P, {{&two, backward, 0, np}}, true);
        std::vector<Rec> joined = two.host;
        joined.insert(joined.end(), two.tail.begin(), two.tail.end());
        std::vector<int32_t> enc = two.enc;
        enc.insert(enc.end(), two.tail_enc.begin(), two.tail_enc.end());
        std::vector<Rec> fa, fb;
        ok = ok && two.host.size() % kChunkRecs == 0 &&
             (size_t)two.n_chunks * kChunkRecs == joined.size() &&
             stream_actions(one.host, one.enc, &fa) && stream_actions(joined, enc, &fb) &&
             same(fa, fb);
    }
    return ok ? STAB_OK : STAB_E_STATE;
}

namespace {

// Rotation ordinals (sorted) and two-qubit gate count of passes [0, k) of a
// plan: maps list their gates, rotation ops carry their ordinals.
void prefix_content(const HostPlan &P, int k, std::vector<int32_t> *rots, int64_t *two_q) {
    rots->clear();
    *two_q = 0;
    for (int i = 0; i < k; ++i) {
        const DevPass &p = P.passes[(size_t)i];
        for (int j = 0; j < p.n_ops; ++j) {
            const DevOp &op = P.ops[p.first + (uint32_t)j];
            if (p.type == P_CLIFF) {
                ++*two_q;
            } else if (op.kind == K_ROT) {
                rots->push_back(op.gate);
            } else if (op.kind == K_MAP3) {
                const DevMap3 &mp = P.maps[(size_t)op.param];
                for (int g = 0; g < mp.count; ++g) {
                    const int32_t o = P.rot_ordinal[(size_t)P.map_gate_idx[(size_t)(mp.first + g)]];
                    if (o >= 0) rots->push_back(o);
                }
            }
        }
    }
    std::sort(rots->begin(), rots->end());
}

}  // namespace

int stab_selftest_align(int n, const stab_gate *gates, int64_t m, int64_t n_params,
                        int64_t *aligned) {
    if (n < 1 || n > STAB_MAX_QUBITS) return STAB_E_RANGE;
    std::string msg;
    RC(validate_gates(n, gates, m, n_params, &msg));
    HostPlan F, G;
    build_plan(n, gates, m, n_params, PLAN_ROWS, &F, false, true);
    build_plan(n, gates, m, n_params, PLAN_GRAD, &G, false, true);
    // rotation ordinals of the generator plan's maps need the gate -> ordinal table
    if (F.rot_ordinal.size() != (size_t)m) {
        F.rot_ordinal.assign((size_t)m, -1);
        int32_t nr = 0;
        for (int64_t i = 0; i < m; ++i)
            if (gates[i].op >= STAB_RX) F.rot_ordinal[(size_t)i] = nr++;
    }
    int64_t count = 0;
    bool refused = false;
    std::vector<int32_t> ra, rb;
    int64_t qa = 0, qb = 0;
    for (int k = 1; k < (int)F.passes.size(); ++k) {
        if (!unit_start(F, (size_t)k)) continue;
        const int g = aligned_pass(F, k, G);
        if (g < 0) {
            refused = true;
            break;
        }
        prefix_content(F, k, &ra, &qa);
        prefix_content(G, g, &rb, &qb);
        if (ra != rb || qa != qb) return STAB_E_STATE;
        ++count;
    }
    if (refused) {
        // the aligner refuses only where the plans' unit sequences differ
        std::vector<uint16_t> ua, ub;
        for (size_t i = 0; i < F.passes.size(); ++i)
            if (unit_start(F, i)) ua.push_back((uint16_t)(F.passes[i].type << 8 | F.passes[i].q));
        for (size_t i = 0; i < G.passes.size(); ++i)
            if (unit_start(G, i)) ub.push_back((uint16_t)(G.passes[i].type << 8 | G.passes[i].q));
        if (ua == ub) return STAB_E_STATE;
        count = 0;
    }
    if (aligned) *aligned = count;
    return STAB_OK;
}

int stab_selftest_pull(int n, const stab_gate *gates, int64_t m) {
    if (n < 1 || n > STAB_MAX_QUBITS) return STAB_E_RANGE;
    std::string msg;
    RC(validate_gates(n, gates, m, 0, &msg));   // no angle slots: Clifford gates only
    return check_pull(n, gates, m) ? STAB_OK : STAB_E_STATE;
}

int stab_selftest_barrier(int64_t ctas, int64_t step) {
    if (ctas < 1 || ctas > (1 << 20) || step < 0 || step > INT32_MAX) return STAB_E_RANGE;
    const int64_t want = ctas * (step + 1);   // as k_stream_chain counts: mod 2^32
    const uint32_t want32 = (uint32_t)ctas * (uint32_t)(step + 1);
    for (int64_t arrived = ctas * step; arrived <= want + ctas; ++arrived)
        if (arrivals_reached((uint32_t)arrived, want32) != (arrived >= want)) return STAB_E_STATE;
    return STAB_OK;
}

int stab_selftest_bounded_wait(int64_t polls) {
    if (polls < 0) return STAB_E_RANGE;
    cudaStream_t s = nullptr;
    CK(cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking));
    int32_t *d = nullptr;
    int32_t h = -1;
    cudaError_t e = cudaMallocAsync(&d, sizeof(int32_t), s);
    if (e == cudaSuccess) e = cudaMemsetAsync(d, 0, sizeof(int32_t), s);
    if (e == cudaSuccess) e = launch_bounded_wait(polls, d, s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(&h, d, sizeof(int32_t), cudaMemcpyDeviceToHost, s);
    if (d) cudaFreeAsync(d, s);
    cudaError_t e2 = cudaStreamSynchronize(s);
    cudaStreamDestroy(s);
    if (e == cudaSuccess) e = e2;
    CK(e);
    return h == 0 ? STAB_OK : STAB_E_TIMEOUT;
}

int stab_last_cuda_error(void) { return g_last_cuda; }

const char *stab_error_string(int s) {
    switch (s) {
    case STAB_OK: return "ok";
    case STAB_E_INVAL: return "invalid argument";
    case STAB_E_RANGE: return "value out of range";
    case STAB_E_NOMEM: return "out of device memory";
    case STAB_E_TIMEOUT: return "device wait timed out";
    case STAB_E_NONFINITE: return "non-finite angle or coefficient";
    case STAB_E_CUDA: return "CUDA runtime error";
    case STAB_E_STATE: return "call out of order";
    case STAB_E_BUSY: return "queue full";
    default: return "unknown status";
    }
}

namespace {

int create_ctx(int n, const stab_opts *opts, const stab_path_choice *forced, stab_ctx **out) {
    if (!out) return STAB_E_INVAL;
    *out = nullptr;
    if (n < 1 || n > STAB_MAX_QUBITS) return STAB_E_RANGE;
    stab_opts o;
    stab_default_opts(&o);
    if (opts) o = *opts;
    if (o.kernel < STAB_KERNEL_AUTO || o.kernel > STAB_KERNEL_PLAIN) return STAB_E_INVAL;
    if (o.kernel == STAB_KERNEL_RESIDENT && n > kMaxResidentQubits) return STAB_E_RANGE;
    if ((o.alloc == nullptr) != (o.free == nullptr)) return STAB_E_INVAL;
    int dev = o.device;
    cudaError_t e = cudaSuccess;
    if (dev < 0) e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaSetDevice(dev);
    if (e != cudaSuccess) {
        g_last_cuda = (int)e;
        return STAB_E_CUDA;
    }
    // the path the context runs: the tuner's choice for AUTO (measured on
    // first use of this n on this GPU model), the defaults otherwise
    stab_path_choice choice;
    stab_path_defaults(n, &choice);
    if (forced) choice = *forced;
    else if (o.kernel == STAB_KERNEL_AUTO && o.fuse) RC(resolve_path_choice(dev, n, &o, &choice));
    stab_ctx *c = new (std::nothrow) stab_ctx();
    if (!c) return STAB_E_NOMEM;
    c->n = n;
    c->fwd.host_n = c->grad.host_n = n;
    c->kernel = o.kernel;
    c->fuse = o.fuse;
    c->choice = choice;
    c->alloc = o.alloc;
    c->free = o.free;
    c->user = o.alloc_user;
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&c->sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess && n >= kChainMinN)
        c->chain_ctas = chain_max_ctas(1 << (chain_tile_bits(n) - 2));
    if (n >= kChainMinN && n <= kChainMaxN) c->aux_stage.least = kStagingTables;
    if (e == cudaSuccess) {
        c->device = dev;
        if (o.stream || o.stream_given) {
            c->st = (cudaStream_t)o.stream;
        } else {
            e = cudaStreamCreateWithFlags(&c->st, cudaStreamNonBlocking);
            c->own_st = (e == cudaSuccess);
        }
    }
    if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&c->aux, cudaStreamNonBlocking);
    if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&c->aux2, cudaStreamNonBlocking);
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&c->ev_fork, cudaEventDisableTiming);
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&c->ev_join, cudaEventDisableTiming);
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&c->ev_ready, cudaEventDisableTiming);
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&c->ev_tx, cudaEventDisableTiming);
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&c->ev_aux, cudaEventDisableTiming);
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&c->ev_gens, cudaEventDisableTiming);
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&c->ev_stage, cudaEventDisableTiming);
    if (e == cudaSuccess) e = cudaEventRecord(c->ev_stage, c->st);
    if (e == cudaSuccess) {
        const int r = c->dalloc(c->status, 256, c->st);
        if (r != STAB_OK) {
            stab_destroy(c);
            return r;
        }
        e = cudaMemsetAsync(c->status.p, 0, 256, c->st);
    }
    if (e != cudaSuccess) {
        g_last_cuda = (int)e;
        stab_destroy(c);
        return STAB_E_CUDA;
    }
    *out = c;
    return STAB_OK;
}

}  // namespace

}  // extern "C"

int stab::create_with_choice(int n, const stab_opts *opts, const stab_path_choice *choice,
                             stab_ctx **out) {
    if (!choice) return STAB_E_INVAL;
    return create_ctx(n, opts, choice, out);
}

extern "C" {

int stab_create(int n, const stab_opts *opts, stab_ctx **out) {
    return create_ctx(n, opts, nullptr, out);
}

int stab_path_current(stab_ctx *c, stab_path_choice *out) {
    if (!c || !out) return STAB_E_INVAL;
    *out = c->choice;
    return STAB_OK;
}

int stab_destroy(stab_ctx *c) {
    if (!c) return STAB_OK;
    cudaSetDevice(c->device);
    if (c->st) cudaStreamSynchronize(c->st);
    if (c->aux) cudaStreamSynchronize(c->aux);
    if (c->aux2) cudaStreamSynchronize(c->aux2);
    c->g_gens.reset();
    c->g_expect.reset();
    c->g_grad.reset();
    DevBuf *bufs[] = {&c->fwd.buf, &c->grad.buf, &c->thetas, &c->gens, &c->gens_tmp, &c->lam,
                      &c->rho, &c->tmp, &c->tmp2, &c->terms, &c->scal, &c->grad_rot,
                      &c->partials, &c->grads, &c->status, &c->gbuf, &c->lam2, &c->tmp3,
                      &c->dotbuf, &c->umaps, &c->unodes, &c->ustates, &c->udots, &c->rmid,
                      &c->lmid, &c->units_e, &c->cnt, &c->gmid, &c->ck.buf, &c->ckslots,
                      &c->ckjobs, &c->ckdots, &c->c_gens.dev, &c->c_expect.dev, &c->c_grad.dev,
                      &c->c_gens.tables, &c->c_expect.tables, &c->c_grad.tables};
    for (DevBuf *b : bufs) c->dfree(*b, c->st);
    if (c->st) cudaStreamSynchronize(c->st);
    c->aux_stage.release();
    if (c->stage) cudaFreeHost(c->stage);
    if (c->ev_ready) cudaEventDestroy(c->ev_ready);
    if (c->ev_tx) cudaEventDestroy(c->ev_tx);
    if (c->ev_aux) cudaEventDestroy(c->ev_aux);
    if (c->ev_gens) cudaEventDestroy(c->ev_gens);
    if (c->ev_stage) cudaEventDestroy(c->ev_stage);
    if (c->aux) cudaStreamDestroy(c->aux);
    if (c->aux2) cudaStreamDestroy(c->aux2);
    if (c->ev_fork) cudaEventDestroy(c->ev_fork);
    if (c->ev_join) cudaEventDestroy(c->ev_join);
    if (c->own_st && c->st) cudaStreamDestroy(c->st);
    delete c;
    return STAB_OK;
}

int stab_load_circuit(stab_ctx *c, const stab_gate *gates, int64_t m, const double *thetas,
                      int64_t n_params) {
    if (!c) return STAB_E_INVAL;
    std::string msg;
    RC(validate_gates(c->n, gates, m, n_params, &msg));
    RC(validate_thetas(thetas, n_params));
    CK(cudaSetDevice(c->device));
    // new state is built before the old one is dropped only where cheap; on an
    // error below the context reports STAB_E_STATE until a load succeeds
    c->loaded = false;
    c->gens_valid = false;
    c->gates.assign(gates, gates + m);
    c->n_params = n_params;
    c->grad.built = false;
    c->grad.encoded = false;
    c->grad_ran = c->ck_ready = c->ck_off = false;
    reset_graphs(c);
    if (c->ckslots.bytes > kCheckpointRelease &&
        checkpoint_bound(c->n, PlanCount(gates, m)) < c->ckslots.bytes / 4)
        ctx_trim(c, 0);
    build_plan(c->n, gates, m, n_params, c->fwd_mode(), &c->fwd.host, !c->use_resident());
    if (c->use_resident()) {
        // AUTO: at n <= 4 the parts' unitaries, at n = 5, 6 the two halves of <O>
        const bool split = c->kernel == STAB_KERNEL_AUTO && c->fuse;
        const int least = c->n == 2 || c->n == 3 ? kUniMinPasses : kSplitMinPasses;
        if (split && c->n <= kUniMaxQubits && (int)c->fwd.host.passes.size() >= least) {
            make_uni(c->fwd, part_cuts(c), c->sms);
        } else {
            make_streams(c->fwd, split ? c->choice.gen_cut : 0.0);
        }
    }
    else no_streams(c->fwd);
    RC(upload_thetas_host(c, thetas));
    RC(upload_plan(c, c->fwd));
    if (c->fwd.uni) RC(uni_buffers(c));
    RC(encode_plan(c, c->fwd));
    CK(cudaEventRecord(c->ev_ready, c->st));
    c->param_gen++;
    c->loaded = true;
    return STAB_OK;
}

int stab_set_params(stab_ctx *c, const double *thetas, int is_device) {
    if (!c) return STAB_E_INVAL;
    if (!c->loaded) return STAB_E_STATE;
    CK(cudaSetDevice(c->device));
    if (is_device) {
        if (c->n_params > 0) {
            if (!thetas) return STAB_E_INVAL;
            CK(cudaMemcpyAsync(c->thetas.p, thetas, (size_t)c->n_params * sizeof(double),
                               cudaMemcpyDeviceToDevice, c->st));
        }
    } else {
        RC(validate_thetas(thetas, c->n_params));
        RC(upload_thetas_host(c, thetas));
    }
    RC(encode_plan(c, c->fwd));
    c->grad.encoded = false;
    c->ck.encoded = false;
    c->gens_valid = false;
    c->param_gen++;
    CK(cudaEventRecord(c->ev_ready, c->st));
    return STAB_OK;
}

int stab_run_generators(stab_ctx *c) {
    if (!c) return STAB_E_INVAL;
    if (!c->loaded) return STAB_E_STATE;
    CK(cudaSetDevice(c->device));
    const int n = c->n;
    const size_t bytes = c->vec_bytes() * (size_t)n;
    RC(c->dalloc(c->gens, bytes, c->st));
    if (c->use_resident() && c->fwd.uni) {
        // the parts' unitaries for these angles may already be there (from
        // <O>, a gradient or the density matrix); then only the read-out is left
        if (c->tx_gen != c->param_gen) RC(uni_run(c));
        UniRoots r = uni_roots(c);
        if (n == 4 && r.n == 3) {
            // the read-out multiplies two unitaries; a third joins the first here
            const UniArgs &u = c->fwd.uargs;
            const int32_t spare = c->fwd.uni_nodes;
            CK(launch_uni_merge(n, r, u.nodes + (size_t)spare * ((size_t)1 << (2 * n)),
                                u.node_parity + spare, c->st));
            c->launches++;
            r.n = 2;
            r.root[0] = spare;
            r.root[1] = r.root[2];
        }
        CK(launch_uni_images(n, r, (double *)c->gens.p, c->st));
        c->launches++;
        c->gens_cur = (double *)c->gens.p;
    } else if (c->use_resident()) {
        StreamArgs a{};
        a.stream = c->fwd.sf.dev;
        a.n_chunks = c->fwd.sf.n_chunks;
        a.init = INIT_GENERATOR;
        a.n_vec = n;
        a.out = (double *)c->gens.p;
        a.status = (int32_t *)c->status.p;
        CK(launch_resident_stream(n, a, c->st));
        c->launches++;
        c->gens_cur = (double *)c->gens.p;
    } else {
        RC(c->dalloc(c->gens_tmp, bytes, c->st));
        RC(stream_encode(c, c->fwd, n));
        cudaStream_t s = c->aux;
        // behind all that is queued on st: the encoding, and copies of the last run's
        // generators that have not run yet
        CK(cudaEventRecord(c->ev_gens, c->st));
        CK(cudaStreamWaitEvent(s, c->ev_gens, 0));
        const std::vector<const void *> key = {(const void *)c->plan_gen, c->gens.p,
                                               c->gens_tmp.p};
        if (use_chain_forward(c, c->fwd, n)) {
            ChainSet &C = c->c_gens;
            if (C.key != key) {
                C.clear();
                C.result[0] = chain_passes(c, c->fwd, (double *)c->gens.p, (double *)c->gens_tmp.p,
                                           false, 0, (int)c->fwd.host.passes.size(), &C, 0);
                RC(chain_upload(c, C, key, c->fwd, n, c->chain_ctas, s));
            }
            CK(launch_fill((double *)c->gens.p, n, n, INIT_GENERATOR, nullptr, 0, s));
            c->launches++;
            RC(chain_run(c, C, s));
            c->g_gens.result = C.result[0];
        } else RC(run_graph(c, c->g_gens, key, s, [&](cudaStream_t gs, void **result) {
            double *cur = (double *)c->gens.p, *alt = (double *)c->gens_tmp.p;
            CK(launch_fill(cur, n, n, INIT_GENERATOR, nullptr, 0, gs));
            c->launches++;
            RC(run_streamed(c, c->fwd, &cur, &alt, n, 0, gs));
            *result = cur;
            return STAB_OK;
        }));
        c->gens_cur = (double *)c->g_gens.result;
        CK(cudaEventRecord(c->ev_aux, s));
        CK(cudaStreamWaitEvent(c->st, c->ev_aux, 0));
    }
    c->gens_valid = true;
    return STAB_OK;
}

int stab_apply_circuit(stab_ctx *c, const stab_gate *gates, int64_t m, const double *thetas,
                       int64_t n_params) {
    RC(stab_load_circuit(c, gates, m, thetas, n_params));
    return stab_run_generators(c);
}

int stab_get_generators(stab_ctx *c, double *out, int out_is_device) {
    if (!c || !out) return STAB_E_INVAL;
    if (!c->gens_valid) return STAB_E_STATE;
    CK(cudaSetDevice(c->device));
    const size_t bytes = c->vec_bytes() * (size_t)c->n;
    if (out_is_device) {
        CK(cudaMemcpyAsync(out, c->gens_cur, bytes, cudaMemcpyDeviceToDevice, c->st));
    } else {
        CK(cudaMemcpyAsync(out, c->gens_cur, bytes, cudaMemcpyDeviceToHost, c->st));
        CK(cudaStreamSynchronize(c->st));
        c->d2h_bytes += (int64_t)bytes;
        RC(check_status(c));
    }
    return STAB_OK;
}

const double *stab_generators_device(stab_ctx *c) {
    if (!c || !c->gens_valid) return nullptr;
    return c->gens_cur;
}

int stab_set_observable(stab_ctx *c, const stab_term *O, int64_t n_terms) {
    if (!c) return STAB_E_INVAL;
    CK(cudaSetDevice(c->device));
    c->obs_loaded = false;
    RC(upload_terms(c, O, n_terms));
    c->obs_loaded = true;
    return STAB_OK;
}

int stab_expect_async(stab_ctx *c, double *out_dev) {
    if (!c || !out_dev) return STAB_E_INVAL;
    if (!c->loaded || !c->obs_loaded) return STAB_E_STATE;
    CK(cudaSetDevice(c->device));
    cudaStream_t s = c->aux;
    if (!c->use_resident()) RC(stream_encode(c, c->fwd, 1));
    CK(cudaStreamWaitEvent(s, c->ev_ready, 0));
    const int32_t nt = c->n_obs_terms;
    if (c->use_resident() && c->fwd.uni) {
        // <O> = <psi|O|psi>, psi = U |0> through the parts' unitaries
        if (c->tx_gen != c->param_gen) RC(uni_run(c));
        CK(cudaStreamWaitEvent(s, c->ev_tx, 0));
        CK(launch_uni_states(c->n, uni_roots(c), (const DevTerm *)c->terms.p, nt, out_dev, nullptr,
                             nullptr, nullptr, s));
        c->launches++;
    } else if (c->use_resident() && c->fwd.split >= 0) {
        RC(split_units_e(c, s));
        BatchArgs a{};
        a.units = (const BatchUnit *)c->units_e.p;
        a.n_units = 2;
        a.counter = (int32_t *)c->cnt.p + 16;
        a.status = (int32_t *)c->status.p;
        CK(cudaMemsetAsync((int32_t *)c->cnt.p + 16, 0, 4, s));
        CK(launch_batch(a, 2, c->split_smem, s));
        CK(launch_dot((const double *)c->lmid.p, (const double *)c->rmid.p, c->n,
                      (double *)c->dotbuf.p, out_dev, s));
        c->launches += 3;
    } else if (c->use_resident()) {
        StreamArgs a{};
        a.stream = c->fwd.sb.dev;
        a.n_chunks = c->fwd.sb.n_chunks;
        a.init = INIT_TERMS;
        a.terms = (const DevTerm *)c->terms.p;
        a.n_terms = nt;
        a.n_vec = 1;
        a.xfree_out = out_dev;
        a.status = (int32_t *)c->status.p;
        CK(launch_resident_stream(c->n, a, s));
        c->launches++;
    } else {
        const size_t vb = c->vec_bytes();
        RC(c->dalloc(c->lam, vb, s));
        RC(c->dalloc(c->tmp, vb, s));
        RC(c->dalloc(c->scal, 64 * sizeof(double), s));
        // small vectors (the tile regime): O backward through the second half
        // of the circuit and rho_0 forward through the first half, at once on
        // two streams; <O> = <lambda_mid, r_mid> (orthogonal maps keep inner
        // products), half the sequential depth
        const bool split = c->fwd.host.mode != PLAN_PLAIN && c->fwd.host.mode != PLAN_PLAIN_ROWS &&
                           c->fwd.host.passes.size() >= 8;
        if (split) {
            RC(c->dalloc(c->lam2, vb, s));
            RC(c->dalloc(c->tmp3, vb, s));
            RC(c->dalloc(c->dotbuf, 256 * sizeof(double), s));
        }
        double *res = (double *)c->scal.p + 2;
        const std::vector<const void *> key = {(const void *)c->plan_gen, c->lam.p, c->tmp.p,
                                               c->lam2.p, c->tmp3.p, c->dotbuf.p,
                                               c->terms.p, (const void *)(intptr_t)nt, res,
                                               (const void *)(intptr_t)split};
        if (split && use_chain_forward(c, c->fwd, 1)) {
            ChainSet &C = c->c_expect;
            if (C.key != key) RC(expect_chains(c, key, c->chain_ctas, s));
            RC(expect_fill(c, s));
            RC(chain_run(c, C, s));
            CK(launch_dot(C.result[0], C.result[1], c->n, (double *)c->dotbuf.p, res, s));
            c->launches += 2;
        } else RC(run_graph(c, c->g_expect, key, s, [&](cudaStream_t gs, void **) {
            double *cur = (double *)c->lam.p, *alt = (double *)c->tmp.p;
            if (!split) {
                CK(launch_fill(cur, c->n, 1, INIT_TERMS, (const DevTerm *)c->terms.p, nt, gs));
                c->launches += nt ? 2 : 1;
                RC(run_streamed(c, c->fwd, &cur, &alt, 1, 1, gs));
                CK(launch_xfree_sum(cur, c->n, 1, res, gs));
                c->launches++;
                return STAB_OK;
            }
            const int np = (int)c->fwd.host.passes.size(), mid = np / 2;
            CK(cudaEventRecord(c->ev_fork, gs));
            CK(cudaStreamWaitEvent(c->aux2, c->ev_fork, 0));
            CK(launch_fill(cur, c->n, 1, INIT_TERMS, (const DevTerm *)c->terms.p, nt, gs));
            RC(run_streamed(c, c->fwd, &cur, &alt, 1, 1, gs, mid, np));
            double *rc = (double *)c->lam2.p, *ra = (double *)c->tmp3.p;
            CK(launch_fill(rc, c->n, 1, INIT_RHO0, nullptr, 0, c->aux2));
            RC(run_streamed(c, c->fwd, &rc, &ra, 1, 0, c->aux2, 0, mid));
            CK(cudaEventRecord(c->ev_join, c->aux2));
            CK(cudaStreamWaitEvent(gs, c->ev_join, 0));
            CK(launch_dot(cur, rc, c->n, (double *)c->dotbuf.p, res, gs));
            c->launches += (nt ? 2 : 1) + 1 + 2;
            return STAB_OK;
        }));
        CK(cudaMemcpyAsync(out_dev, res, sizeof(double), cudaMemcpyDeviceToDevice, s));
    }
    // join: later work on the main stream sees the result
    CK(cudaEventRecord(c->ev_aux, s));
    CK(cudaStreamWaitEvent(c->st, c->ev_aux, 0));
    return STAB_OK;
}

int stab_expect(stab_ctx *c, const stab_term *O, int64_t n_terms, double *out) {
    if (!c || !out) return STAB_E_INVAL;
    if (!c->loaded) return STAB_E_STATE;
    RC(stab_set_observable(c, O, n_terms));
    RC(c->dalloc(c->scal, 64 * sizeof(double), c->st));
    RC(stab_expect_async(c, (double *)c->scal.p));
    CK(cudaEventSynchronize(c->ev_stage));
    RC(c->host_stage(c->stage, c->stage_bytes, 64 * sizeof(double)));
    double *h = (double *)c->stage;
    CK(cudaMemcpyAsync(h, c->scal.p, sizeof(double), cudaMemcpyDeviceToHost, c->st));
    CK(cudaStreamSynchronize(c->st));
    c->d2h_bytes += (int64_t)sizeof(double);
    *out = *h;
    RC(check_status(c));
    return STAB_OK;
}

int stab_grad_async(stab_ctx *c, double *expect_dev, double *grads_dev) {
    if (!c) return STAB_E_INVAL;
    if (!c->loaded || !c->obs_loaded) return STAB_E_STATE;
    if (c->n_params > 0 && !grads_dev) return STAB_E_INVAL;
    CK(cudaSetDevice(c->device));
    c->grad_uni = uni_grad_ok(c);
    int rc = STAB_OK;
    const bool stored = !c->grad_uni && !c->use_resident_adjoint() && ck_usable(c, &rc);
    RC(rc);
    if (stored) {
        DevPlan &G = &ck_plan(c) == &c->ck ? c->ck : c->fwd;
        if (!G.encoded) RC(encode_plan(c, G));
        RC(use_chain(c, G, 1) ? stream_maps(c, G) : stream_ops(c, G));
        CK(cudaEventRecord(c->ev_ready, c->st));
    } else {
        RC(c->grad_uni ? ensure_uni_grad(c) : ensure_grad_plan(c));
    }
    c->grad_ran = true;
    cudaStream_t s = c->aux;
    CK(cudaStreamWaitEvent(s, c->ev_ready, 0));
    const int32_t nt = c->n_obs_terms;
    const int n = c->n;
    if (stored) {
        RC(c->dalloc(c->scal, 64 * sizeof(double), s));
        RC(c->dalloc(c->gbuf, (size_t)c->n_params * sizeof(double), s));
        RC(c->dalloc(c->grad_rot, std::max<size_t>(1, c->ck.ugates.size()) * sizeof(double), s));
        RC(c->dalloc(c->ckdots, std::max<size_t>(1, c->ck.uruns.size()) * 3 *
                                    (size_t)c->ck_chunks * sizeof(double), s));
        RC(ck_upload_jobs(c, s));
        double *res = (double *)c->scal.p + 3;
        const std::vector<const void *> key = {
            (const void *)c->plan_gen, c->ckslots.p, c->ckjobs.p, c->ckdots.p, c->grad_rot.p,
            c->gbuf.p, c->terms.p, (const void *)(intptr_t)nt, res, c->thetas.p, c->ck.buf.p};
        // the chain is one launch; long vectors' launches are replayed from a graph
        if (use_chain(c, ck_plan(c), 1)) RC(ck_gradient(c, res, s));
        else RC(run_graph(c, c->g_grad, key, s,
                          [&](cudaStream_t gs, void **) { return ck_gradient(c, res, gs); }));
        CK(cudaMemcpyAsync(expect_dev ? expect_dev : (double *)c->scal.p + 1, res, sizeof(double),
                           cudaMemcpyDeviceToDevice, s));
        CK(cudaMemcpyAsync(grads_dev, c->gbuf.p, (size_t)c->n_params * sizeof(double),
                           cudaMemcpyDeviceToDevice, s));
        CK(cudaEventRecord(c->ev_aux, s));
        CK(cudaStreamWaitEvent(c->st, c->ev_aux, 0));
        return STAB_OK;
    }
    if (c->grad_uni) {
        // the states at the parts' boundaries, then every segment at once
        const DevPlan &P = c->fwd;
        if (c->tx_gen != c->param_gen) RC(uni_run(c));
        CK(cudaStreamWaitEvent(s, c->ev_tx, 0));
        const size_t D = (size_t)1 << n, slots = P.uparts.size() + 1;
        const size_t n_runs = P.uruns.size(), n_gates = P.ugates.size();
        RC(c->dalloc(c->scal, 64 * sizeof(double), s));
        RC(c->dalloc(c->ustates, 2 * slots * D * sizeof(double2), s));
        RC(c->dalloc(c->udots, std::max<size_t>(1, n_runs) * 3 * D * sizeof(double), s));
        RC(c->dalloc(c->grad_rot, std::max<size_t>(1, n_gates) * sizeof(double), s));
        double2 *psi = (double2 *)c->ustates.p, *phi = psi + slots * D;
        CK(launch_uni_states(n, uni_roots(c), (const DevTerm *)c->terms.p, nt,
                             expect_dev ? expect_dev : (double *)c->scal.p + 1, psi, phi, nullptr,
                             s));
        c->launches++;
        if (c->n_params > 0) {
            CK(launch_uni_grad(n, P.uargs, psi, phi, (double *)c->udots.p, s));
            CK(launch_run_grads(P.uruns_dev, (int)n_runs, P.uni_max_run, P.ugates_dev,
                                (const double *)c->thetas.p, (const double *)c->udots.p, (int)D,
                                (double *)c->grad_rot.p, s));
            CK(launch_gather_grads((const double *)c->grad_rot.p, c->grad.param_ptr,
                                   c->grad.param_rot, (int)c->n_params, grads_dev, s));
            c->launches += 2 + (n_runs > 0);
        }
        CK(cudaEventRecord(c->ev_aux, s));
        CK(cudaStreamWaitEvent(c->st, c->ev_aux, 0));
        return STAB_OK;
    }
    const int n_rot = c->grad.host.n_rot;
    RC(c->dalloc(c->scal, 64 * sizeof(double), s));
    RC(c->dalloc(c->grad_rot, (size_t)(n_rot ? n_rot : 1) * sizeof(double), s));
    double *e_out = expect_dev ? expect_dev : (double *)c->scal.p + 1;
    // the resident sweeps store each thread's dot share per rotation (no
    // reduction on the sweep's critical path; one fixed-order sum after it)
    // while the CTA has at most kPartialThreads threads and the shares fit
    // kPartialBytes; otherwise each pass reduces its dots over the CTA
    double *partials = nullptr;
    const int part_threads = resident_adjoint_threads(n);
    if (c->use_resident_adjoint()) {
        const size_t bytes = resident_partial_bytes(n, n_rot);
        if (bytes > 0) {
            RC(c->dalloc(c->partials, bytes, s));
            partials = (double *)c->partials.p;
        }
    }
    if (c->use_resident_adjoint() && c->grad.split >= 0) {
        // meet in the middle: rho_0 forward through the first part and O
        // backward through the second, then the pair at the cut backward
        // through the first part and forward through the second
        const size_t E = (size_t)1 << (2 * n);
        RC(c->dalloc(c->gmid, 2 * E * sizeof(double), s));
        AdjointSplitArgs a{};
        a.stream[0] = c->grad.h1.dev;
        a.n_chunks[0] = c->grad.h1.n_chunks;
        a.stream[1] = c->grad.h2b.dev;
        a.n_chunks[1] = c->grad.h2b.n_chunks;
        a.phase = 0;
        a.terms = (const DevTerm *)c->terms.p;
        a.n_terms = nt;
        a.rmid = (double *)c->gmid.p;
        a.lmid = (double *)c->gmid.p + E;
        a.grad_rot = (double *)c->grad_rot.p;
        a.partials = partials;
        a.expect_out = e_out;
        a.status = (int32_t *)c->status.p;
        CK(launch_adjoint_split(n, a, s));
        a.stream[0] = c->grad.h1b.dev;
        a.n_chunks[0] = c->grad.h1b.n_chunks;
        a.stream[1] = c->grad.h2.dev;
        a.n_chunks[1] = c->grad.h2.n_chunks;
        a.phase = 1;
        CK(launch_adjoint_split(n, a, s));
        c->launches += 2;
        if (partials) {
            CK(launch_reduce_partials(partials, n_rot, part_threads, (double *)c->grad_rot.p, s));
            c->launches++;
        }
        if (c->n_params > 0) {
            CK(launch_gather_grads((const double *)c->grad_rot.p, c->grad.param_ptr,
                                   c->grad.param_rot, (int)c->n_params, grads_dev, s));
            c->launches++;
        }
    } else if (c->use_resident_adjoint()) {
        AdjointStreamArgs a{};
        a.fwd = c->grad.sf.dev;
        a.bwd = c->grad.sb.dev;
        a.n_fwd_chunks = c->grad.sf.n_chunks;
        a.n_bwd_chunks = c->grad.sb.n_chunks;
        a.terms = (const DevTerm *)c->terms.p;
        a.n_terms = nt;
        a.grad_rot = (double *)c->grad_rot.p;
        a.partials = partials;
        a.expect_out = e_out;
        a.status = (int32_t *)c->status.p;
        CK(launch_adjoint_stream(n, a, s));
        c->launches++;
        if (partials) {
            CK(launch_reduce_partials(partials, n_rot, part_threads, (double *)c->grad_rot.p, s));
            c->launches++;
        }
        if (c->n_params > 0) {
            CK(launch_gather_grads((const double *)c->grad_rot.p, c->grad.param_ptr,
                                   c->grad.param_rot, (int)c->n_params, grads_dev, s));
            c->launches++;
        }
    } else {
        // lambda and rho are one contiguous pair (lambda first), ping-ponged
        // with a second pair, so a Clifford gather moves both in one launch
        const size_t vb = c->vec_bytes();
        const uint64_t E = 1ull << (2 * n);
        RC(c->dalloc(c->lam, 2 * vb, s));
        RC(c->dalloc(c->tmp, 2 * vb, s));
        RC(c->dalloc(c->gbuf, (size_t)(c->n_params ? c->n_params : 1) * sizeof(double), s));
        const int nb = adjoint_stream_blocks(n);
        RC(c->dalloc(c->partials, (size_t)(n_rot ? n_rot : 1) * nb * sizeof(double), s));
        double *res = (double *)c->scal.p + 3;
        const bool tiles = n <= kAdjTileMaxN;
        RC(c->dalloc(c->lam2, 2 * vb, s));
        RC(c->dalloc(c->tmp3, 2 * vb, s));
        const std::vector<const void *> key = {
            (const void *)c->plan_gen, c->lam.p, c->tmp.p, c->lam2.p, c->tmp3.p, c->partials.p,
            c->grad_rot.p, c->gbuf.p, c->terms.p, (const void *)(intptr_t)nt, res};
        {
            // Pair sweep, for plans whose stored sweeps would not fit.  The
            // circuit's passes are cut in two halves at
            // `mid`.  Phase 1, two branches at once: r forward through the
            // first half, lambda backward through the second; both meet at
            // `mid`.  Phase 2, two branches at once: the pair (lambda, r)
            // backward through the first half and forward through the second
            // (every map is orthogonal, so lambda moves forward as r does),
            // each rotation's dot taken at its post-gate pair.  Half the
            // sequential depth of forward-then-reverse, and two chains of
            // launches share the GPU (measured faster at every n: 1.6x at
            // n = 8, 1.1-1.3x at n = 9..12).
            RC(run_graph(c, c->g_grad, key, s, [&](cudaStream_t gs, void **) {
                const auto &passes = c->grad.host.passes;
                const int np = (int)passes.size(), mid = np / 2;
                const DevOp *ops = c->grad.prog.ops;
                const auto &hops = c->grad.host.ops;
                double *A = (double *)c->lam.p, *B = (double *)c->tmp.p;
                double *Cb = (double *)c->lam2.p, *D = (double *)c->tmp3.p;
                auto fork = [&](cudaStream_t from, cudaStream_t to) -> int {
                    CK(cudaEventRecord(c->ev_fork, from));
                    CK(cudaStreamWaitEvent(to, c->ev_fork, 0));
                    return STAB_OK;
                };
                auto join = [&](cudaStream_t from, cudaStream_t to) -> int {
                    CK(cudaEventRecord(c->ev_join, from));
                    CK(cudaStreamWaitEvent(to, c->ev_join, 0));
                    return STAB_OK;
                };
                // the adjoint sweep of passes [k0, k1) on a pair, one way
                auto sweep = [&](double *&pr, double *&al, int k0, int k1, bool forward,
                                 cudaStream_t st) -> int {
                    std::vector<const DevPass *> group;
                    std::vector<int> wires;
                    const DevPass *pending = nullptr;
                    auto pull_of = [&](const DevPass *p) {
                        return c->grad.prog.pulls +
                               2 * c->grad.host.pull_of[(size_t)(p - passes.data())] +
                               (forward ? 0 : 1);
                    };
                    auto gather_now = [&]() -> int {
                        CK(launch_gather(c, c->grad, *pending, forward ? 0 : 1, pr, al, 2, st));
                        c->launches++;
                        std::swap(pr, al);
                        pending = nullptr;
                        return STAB_OK;
                    };
                    auto flush = [&]() -> int {
                        if (group.empty()) return STAB_OK;
                        if (!tiles) {
                            for (const DevPass *gp : group) {
                                CK(launch_adjoint_wire(pr, pr + E, n, *gp, ops,
                                                       (double *)c->partials.p, forward ? 1 : 0,
                                                       st));
                                c->launches++;
                            }
                            group.clear();
                            wires.clear();
                            return STAB_OK;
                        }
                        TileGroup tg;
                        make_tile_group(n, 1, passes, group, forward ? 0 : 1, &tg, nb,
                                        std::min(kAdjTileBits, 2 * n));
                        for (size_t j = 0; j < group.size(); ++j) {
                            int nr = 0;
                            for (int k = 0; k < group[j]->n_ops; ++k)
                                nr += hops[(size_t)group[j]->first + k].kind == K_ROT;
                            tg.n_rot[j] = (uint8_t)nr;
                        }
                        double *dst = pr;
                        if (pending) {
                            tg.pull = pull_of(pending);
                            dst = al;
                        }
                        CK(launch_adjoint_tile(pr, dst, n, tg, ops, (double *)c->partials.p, st));
                        c->launches++;
                        if (pending) {
                            std::swap(pr, al);
                            pending = nullptr;
                        }
                        group.clear();
                        wires.clear();
                        return STAB_OK;
                    };
                    for (int t = 0; t < k1 - k0; ++t) {
                        const DevPass &p = passes[forward ? k0 + t : k1 - 1 - t];
                        if (p.type == P_WIRE) {
                            const bool known =
                                std::find(wires.begin(), wires.end(), (int)p.q) != wires.end();
                            if ((int)group.size() == kTileMaxPasses ||
                                (!known && (int)wires.size() == kAdjTileWires))
                                RC(flush());
                            group.push_back(&p);
                            if (!known) wires.push_back(p.q);
                            continue;
                        }
                        RC(flush());
                        if (pending) RC(gather_now());
                        pending = &p;
                        if (!tiles) RC(gather_now());
                    }
                    RC(flush());
                    if (pending) RC(gather_now());
                    return STAB_OK;
                };
                // phase 1
                RC(fork(gs, c->aux2));
                double *rho = A + E, *rho_alt = B + E;
                CK(launch_fill(rho, n, 1, INIT_RHO0, nullptr, 0, gs));
                RC(run_streamed(c, c->grad, &rho, &rho_alt, 1, 0, gs, 0, mid));
                double *lam = Cb, *lam_alt = D;
                CK(launch_fill(lam, n, 1, INIT_TERMS, (const DevTerm *)c->terms.p, nt, c->aux2));
                RC(run_streamed(c, c->grad, &lam, &lam_alt, 1, 1, c->aux2, mid, np));
                c->launches += nt ? 3 : 2;
                RC(join(c->aux2, gs));
                // the meeting pair, once in each branch's buffers
                double *X = rho - E, *Xalt = X == A ? B : A;
                double *Y = lam, *Yalt = Y == Cb ? D : Cb;
                CK(cudaMemcpyAsync(X, lam, vb, cudaMemcpyDeviceToDevice, gs));
                CK(cudaMemcpyAsync(Y + E, rho, vb, cudaMemcpyDeviceToDevice, gs));
                // phase 2
                RC(fork(gs, c->aux2));
                RC(sweep(X, Xalt, 0, mid, false, gs));
                RC(sweep(Y, Yalt, mid, np, true, c->aux2));
                RC(join(c->aux2, gs));
                CK(launch_reduce_partials((const double *)c->partials.p, n_rot, nb,
                                          (double *)c->grad_rot.p, gs));
                CK(launch_xfree_sum(X, n, 1, res, gs));   // <O> = <lambda_0, rho_0>
                c->launches += 2;
                if (c->n_params > 0) {
                    CK(launch_gather_grads((const double *)c->grad_rot.p, c->grad.param_ptr,
                                           c->grad.param_rot, (int)c->n_params,
                                           (double *)c->gbuf.p, gs));
                    c->launches++;
                }
                return STAB_OK;
            }));
        }
        CK(cudaMemcpyAsync(e_out, res, sizeof(double), cudaMemcpyDeviceToDevice, s));
        if (c->n_params > 0)
            CK(cudaMemcpyAsync(grads_dev, c->gbuf.p, (size_t)c->n_params * sizeof(double),
                               cudaMemcpyDeviceToDevice, s));
    }
    CK(cudaEventRecord(c->ev_aux, s));
    CK(cudaStreamWaitEvent(c->st, c->ev_aux, 0));
    return STAB_OK;
}

int stab_set_grad_memory(stab_ctx *c, int64_t bytes) {
    if (!c) return STAB_E_INVAL;
    if (bytes < 0) return STAB_E_RANGE;
    CK(cudaSetDevice(c->device));
    c->ck_bytes_max = std::min((size_t)bytes, kCheckpointBytes);
    c->ck_off = false;   // decided anew by the next gradient
    if (c->ckslots.bytes > c->ck_bytes_max) ctx_trim(c, 0);
    return STAB_OK;
}

int stab_grad(stab_ctx *c, const stab_term *O, int64_t n_terms, double *expect_out,
              double *grads_out) {
    if (!c) return STAB_E_INVAL;
    if (!c->loaded) return STAB_E_STATE;
    if (c->n_params > 0 && !grads_out) return STAB_E_INVAL;
    RC(stab_set_observable(c, O, n_terms));
    RC(c->dalloc(c->grads, (size_t)(c->n_params ? c->n_params : 1) * sizeof(double), c->st));
    RC(c->dalloc(c->scal, 64 * sizeof(double), c->st));
    RC(stab_grad_async(c, (double *)c->scal.p, (double *)c->grads.p));
    const size_t gbytes = (size_t)c->n_params * sizeof(double);
    CK(cudaEventSynchronize(c->ev_stage));
    RC(c->host_stage(c->stage, c->stage_bytes, gbytes + 64 * sizeof(double)));
    double *h = (double *)c->stage;
    CK(cudaMemcpyAsync(h, c->scal.p, sizeof(double), cudaMemcpyDeviceToHost, c->st));
    if (gbytes) CK(cudaMemcpyAsync(h + 8, c->grads.p, gbytes, cudaMemcpyDeviceToHost, c->st));
    CK(cudaStreamSynchronize(c->st));
    c->d2h_bytes += (int64_t)(gbytes + sizeof(double));
    if (expect_out) *expect_out = h[0];
    if (gbytes) std::memcpy(grads_out, h + 8, gbytes);
    RC(check_status(c));
    return STAB_OK;
}

int stab_density_matrix(stab_ctx *c, double *out, int out_is_device) {
    if (!c || !out) return STAB_E_INVAL;
    if (!c->loaded) return STAB_E_STATE;
    CK(cudaSetDevice(c->device));
    const int n = c->n;
    const size_t vb = c->vec_bytes();
    RC(c->dalloc(c->rho, vb, c->st));
    double *r = (double *)c->rho.p;
    if (c->use_resident() && c->fwd.uni) {
        if (c->tx_gen != c->param_gen) RC(uni_run(c));
        CK(launch_uni_states(n, uni_roots(c), nullptr, 0, nullptr, nullptr, nullptr, r, c->st));
        c->launches++;
    } else if (c->use_resident()) {
        StreamArgs a{};
        a.stream = c->fwd.sf.dev;
        a.n_chunks = c->fwd.sf.n_chunks;
        a.init = INIT_RHO0;
        a.n_vec = 1;
        a.out = r;
        a.status = (int32_t *)c->status.p;
        CK(launch_resident_stream(n, a, c->st));
        c->launches++;
    } else {
        RC(c->dalloc(c->tmp2, vb, c->st));
        RC(stream_encode(c, c->fwd, 1));
        double *cur = r, *alt = (double *)c->tmp2.p;
        CK(launch_fill(cur, n, 1, INIT_RHO0, nullptr, 0, c->st));
        c->launches++;
        RC(run_streamed(c, c->fwd, &cur, &alt, 1, 0, c->st));
        r = cur;
    }
    const size_t rho_bytes = 2 * vb;
    if (out_is_device) {
        CK(launch_decode_rho(r, n, out, c->st));
        c->launches++;
        return STAB_OK;
    }
    RC(c->dalloc(c->tmp, rho_bytes, c->st));
    CK(launch_decode_rho(r, n, (double *)c->tmp.p, c->st));
    c->launches++;
    CK(cudaMemcpyAsync(out, c->tmp.p, rho_bytes, cudaMemcpyDeviceToHost, c->st));
    CK(cudaStreamSynchronize(c->st));
    c->d2h_bytes += (int64_t)rho_bytes;
    return check_status(c);
}

int stab_synchronize(stab_ctx *c) {
    if (!c) return STAB_E_INVAL;
    CK(cudaSetDevice(c->device));
    CK(cudaStreamSynchronize(c->st));
    CK(cudaStreamSynchronize(c->aux));
    return check_status(c);
}

int stab_plan_info(stab_ctx *c, int64_t *n_gates, int64_t *n_passes, int32_t *kernel) {
    if (!c) return STAB_E_INVAL;
    if (n_gates) *n_gates = (int64_t)c->gates.size();
    if (n_passes) *n_passes = (int64_t)c->fwd.host.passes.size();
    if (kernel) *kernel = c->use_resident() ? STAB_KERNEL_RESIDENT : STAB_KERNEL_STREAMED;
    return STAB_OK;
}

int stab_split_info(stab_ctx *c, int64_t *cut, int32_t *gen_units, int32_t *expect_units) {
    if (!c) return STAB_E_INVAL;
    const bool on = c->loaded && c->use_resident() && c->fwd.split >= 0;
    const int E = 1 << (2 * c->n);
    if (cut) *cut = on ? c->fwd.split : -1;
    if (gen_units) *gen_units = on && c->fwd.uni ? c->n + 1 + later_parts(c) * (E - 1) : 0;
    if (expect_units) *expect_units = on && !c->fwd.uni ? 2 : 0;
    return STAB_OK;
}

int64_t stab_launch_count(stab_ctx *c) { return c ? c->launches : 0; }

int stab_grad_parts(stab_ctx *c, int32_t *parts) {
    if (!c || !parts) return STAB_E_INVAL;
    *parts = !c->grad_ran                              ? 0
             : c->grad_uni && !c->fwd.uni_identity && c->fwd.split >= 0
                 ? (int32_t)c->fwd.uparts.size()
                 : 1;
    return STAB_OK;
}

int stab_transfer_bytes(stab_ctx *c, int64_t *h2d, int64_t *d2h) {
    if (!c) return STAB_E_INVAL;
    if (h2d) *h2d = c->h2d_bytes;
    if (d2h) *d2h = c->d2h_bytes;
    return STAB_OK;
}

}  // extern "C"

// ---------------------------------------------------------------- long items of a batch

int stab::long_item_prepare(stab_ctx *c, bool gens, int max_ctas, const ChainDesc **chains,
                            int *n_chains) {
    if (!c || !c->loaded || c->use_resident() || (!gens && !c->obs_loaded)) return STAB_E_STATE;
    const size_t vb = c->vec_bytes();
    const std::vector<const void *> key = {(const void *)c->plan_gen};
    ChainSet &C = gens ? c->c_gens : c->c_expect;
    RC(stream_maps(c, c->fwd));
    if (!c->fwd.prog.pass_maps && !c->fwd.host.passes.empty()) return STAB_E_STATE;
    if (gens) {
        const size_t bytes = vb * (size_t)c->n;
        RC(c->dalloc(c->gens, bytes, c->st));
        RC(c->dalloc(c->gens_tmp, bytes, c->st));
        C.clear();
        C.result[0] = chain_passes(c, c->fwd, (double *)c->gens.p, (double *)c->gens_tmp.p, false,
                                   0, (int)c->fwd.host.passes.size(), &C, 0);
        RC(chain_upload(c, C, key, c->fwd, c->n, max_ctas, c->st));
    } else {
        for (DevBuf *b : {&c->lam, &c->tmp, &c->lam2, &c->tmp3}) RC(c->dalloc(*b, vb, c->st));
        RC(c->dalloc(c->dotbuf, 256 * sizeof(double), c->st));
        RC(expect_chains(c, key, max_ctas, c->st));
        // the terms were allocated and copied on aux, and the batch reads them on
        // a stream of its own that waits for c->st alone
        CK(cudaStreamSynchronize(c->aux));
    }
    *chains = C.desc;
    *n_chains = C.n_chains;
    return STAB_OK;
}

int stab::long_item_fill(stab_ctx *c, bool gens, cudaStream_t s) {
    if (!gens) return expect_fill(c, s);
    CK(launch_fill((double *)c->gens.p, c->n, c->n, INIT_GENERATOR, nullptr, 0, s));
    return STAB_OK;
}

int stab::long_item_finish(stab_ctx *c, bool gens, double *out, cudaStream_t s) {
    if (gens) {
        CK(cudaMemcpyAsync(out, c->c_gens.result[0], c->vec_bytes() * (size_t)c->n,
                           cudaMemcpyDeviceToDevice, s));
        return STAB_OK;
    }
    CK(launch_dot(c->c_expect.result[0], c->c_expect.result[1], c->n, (double *)c->dotbuf.p, out,
                  s));
    return STAB_OK;
}

// Expectation of an observable already on the device as deduplicated terms
// (the sparse path's list when it switches to the dense vector).
int stab::expect_device_terms(stab_ctx *c, const DevTerm *terms, int64_t nt, double *out) {
    if (!c || !out || nt < 0 || nt > INT32_MAX || (nt > 0 && !terms)) return STAB_E_INVAL;
    if (!c->loaded) return STAB_E_STATE;
    CK(cudaSetDevice(c->device));
    c->obs_loaded = false;
    CK(cudaStreamSynchronize(c->aux));
    RC(c->dalloc(c->terms, (size_t)(nt ? nt : 1) * sizeof(DevTerm), c->st));
    if (nt)
        CK(cudaMemcpyAsync(c->terms.p, terms, (size_t)nt * sizeof(DevTerm),
                           cudaMemcpyDeviceToDevice, c->st));
    c->n_obs_terms = (int32_t)nt;
    CK(cudaEventRecord(c->ev_ready, c->st));
    c->obs_loaded = true;
    RC(c->dalloc(c->scal, 64 * sizeof(double), c->st));
    RC(stab_expect_async(c, (double *)c->scal.p));
    CK(cudaEventSynchronize(c->ev_stage));
    RC(c->host_stage(c->stage, c->stage_bytes, 64 * sizeof(double)));
    double *h = (double *)c->stage;
    CK(cudaMemcpyAsync(h, c->scal.p, sizeof(double), cudaMemcpyDeviceToHost, c->st));
    CK(cudaStreamSynchronize(c->st));
    c->d2h_bytes += (int64_t)sizeof(double);
    *out = *h;
    RC(check_status(c));
    return STAB_OK;
}

