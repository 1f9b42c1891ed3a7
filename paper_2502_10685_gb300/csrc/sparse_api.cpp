// sparse_api.cpp -- the sparse term-list entry points (include/stab.h): step
// plans, the run with capacity growth, and the switch to the dense path once
// the stabilizer order n' passes a threshold (Sec. II-B, Fig. 1).
//
// A plan is the gate list in application order (backward: reversed, inverse
// gates) cut into steps: maximal runs of Clifford gates and single rotations.
// On the device only rotations run, each about its string pulled back through
// the Clifford gates before it (k_sparse.cu); the images of the last list under
// all of those gates are the result.  A run is one launch while the list is
// short and one for the rest; its outcome and the orders are read once.  A
// rotation that would overflow is not applied; the buffers grow 8x (the list is
// copied over) and the run resumes at it.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <functional>
#include <map>
#include <new>
#include <string>
#include <vector>

#include "../../include/stab.h"
#include "host_pool.h"
#include "launch.h"
#include "planner.h"

using namespace stab;

namespace {

#define SCK(expr)                        \
    do {                                 \
        cudaError_t e_ = (expr);         \
        if (e_ != cudaSuccess) {         \
            record_cuda_error(e_);       \
            return STAB_E_CUDA;          \
        }                                \
    } while (0)

#define SRC(expr)                         \
    do {                                  \
        int r_ = (expr);                  \
        if (r_ != STAB_OK) return r_;     \
    } while (0)

constexpr int64_t kSpMinCap = 4096;
constexpr int64_t kSpMaxCap = 1ll << 30;

struct SpBuf {
    void *p = nullptr;
    size_t bytes = 0;
};

enum { SP_CLIFF = 0, SP_ROT = 1 };

struct SpGate {               // one Clifford gate, already inverted for
    uint8_t op, q0, q1, pad;  // backward plans (S <-> S^dagger)
};

struct SpStep {
    int kind;
    int first, count;         // Clifford run: gates [first, first + count)
    int64_t gate_lo, gate_hi; // circuit gates [gate_lo, gate_hi) the step covers
};

struct SpPlan {
    std::vector<SpStep> steps;
    std::vector<SpGate> gates;
    std::vector<SpRot> rots;
    std::vector<int64_t> rot_step;   // the rotations' steps
};

// The outcome of one propagation.
struct SpRun {
    int buf = 0;              // buffer holding the list
    int64_t step = 0;         // the list is the one before this step (== steps: all run)
    int64_t count = 0;
    bool stopped = false;     // threshold reached, or capacity exhausted
};

// The strings U^dagger X_q U and U^dagger Z_q U, kept while gates are appended
// to U: a gate g maps its wires' letters to products of at most two (g^dagger
// sigma g), so it rewrites at most two rows.  What U does to a string follows
// from the rows alone: bit x_q of the image of P is whether P anticommutes with
// U^dagger Z_q U, bit z_q whether it does with U^dagger X_q U.
struct SpPull {
    struct Row {
        uint64_t key;
        uint32_t e;           // i^e times the Hermitian string `key`
    };
    int n;
    uint64_t zm;
    Row x[32], z[32];

    explicit SpPull(int n_) : n(n_), zm((1ull << n_) - 1) {
        for (int q = 0; q < n; ++q) {
            x[q] = Row{1ull << (n + q), 0};
            z[q] = Row{1ull << q, 0};
        }
    }
    uint64_t flip(uint64_t k) const { return (k >> n) | ((k & zm) << n); }
    // see sp_mul_phase of k_sparse.cu
    Row mul(const Row &a, const Row &b) const {
        const uint32_t ax = (uint32_t)(a.key >> n), az = (uint32_t)(a.key & zm);
        const uint32_t bx = (uint32_t)(b.key >> n), bz = (uint32_t)(b.key & zm);
        const uint32_t A = ax & az, B = ax & ~az, C = ~ax & az;
        const uint32_t plus = (A & bz & ~bx) | (B & bz & bx) | (C & bx & ~bz);
        const uint32_t minus = (A & bx & ~bz) | (B & bz & ~bx) | (C & bx & bz);
        const uint32_t c = (uint32_t)__builtin_popcountll(((uint64_t)~minus << 32) | plus);
        return Row{a.key ^ b.key, (a.e + b.e + c) & 3u};
    }
    Row y(int q) const {      // Y = i X Z
        Row r = mul(x[q], z[q]);
        r.e = (r.e + 1u) & 3u;
        return r;
    }
    void apply(const SpGate &g) {
        const int a = g.q0, b = g.q1;
        switch (g.op) {
        case STAB_H: std::swap(x[a], z[a]); break;
        case STAB_S:          // S^dagger X S = -Y
            x[a] = y(a);
            x[a].e ^= 2u;
            break;
        case STAB_SDG: x[a] = y(a); break;
        case STAB_X: z[a].e ^= 2u; break;
        case STAB_Y:
            x[a].e ^= 2u;
            z[a].e ^= 2u;
            break;
        case STAB_Z: x[a].e ^= 2u; break;
        case STAB_CX:         // X_c -> X_c X_t, Z_t -> Z_c Z_t
            x[a] = mul(x[a], x[b]);
            z[b] = mul(z[a], z[b]);
            break;
        case STAB_CZ: {       // X_a -> X_a Z_b, X_b -> Z_a X_b
            x[a] = mul(x[a], z[b]);
            x[b] = mul(z[a], x[b]);
            break;
        }
        default: break;
        }
    }
    SpRot rotation(int q, int axis, int param) const {
        const Row P = axis == 0 ? x[q] : axis == 1 ? y(q) : z[q];
        // pairs (u, v): R_x: (Y, Z), R_y: (Z, X), R_z: (X, Y); u is the one with
        // x (Y of Y, Z), with z (Z of Z, X), without z (X of X, Y)
        SpRot r{};
        r.P = P.key;
        r.anti = flip(P.key);
        r.letter = flip(axis == 0 ? z[q].key : x[q].key);
        r.param = param;
        r.flags = (axis == 2 ? 0u : 1u) | P.e;
        return r;
    }
    uint64_t xcol(int q) const { return flip(z[q].key); }
    // U X_q U^dagger (entry q) and U Z_q U^dagger (entry n + q): the bits as
    // above; the sign is that of the rows' product over the bits, which gives
    // the generator back
    void tableau(SpTab *tab) const {
        for (int g = 0; g < 2 * n; ++g) {
            const uint64_t k = g < n ? 1ull << (n + g) : 1ull << (g - n);
            Row t{0, 0};
            uint64_t w = 0;
            for (int q = 0; q < n; ++q) {
                const bool wx = __builtin_parityll(k & flip(z[q].key));
                const bool wz = __builtin_parityll(k & flip(x[q].key));
                if (wx) t = mul(t, x[q]);
                if (wz) t = mul(t, z[q]);
                if (wx && wz) t.e = (t.e + 1u) & 3u;
                w |= ((uint64_t)wx << (n + q)) | ((uint64_t)wz << q);
            }
            tab[g] = SpTab{w, t.e >> 1, 0};
        }
    }
};

void build_sp_plan(const std::vector<stab_gate> &gates, bool backward, SpPlan *P, SpPull *U) {
    P->steps.clear();
    P->gates.clear();
    P->rots.clear();
    P->rot_step.clear();
    const int64_t m = (int64_t)gates.size();
    bool in_run = false;
    for (int64_t k = 0; k < m; ++k) {
        const int64_t i = backward ? m - 1 - k : k;
        const stab_gate &g = gates[i];
        if (g.op >= STAB_RX) {
            SpStep s{};
            s.kind = SP_ROT;
            s.gate_lo = i;
            s.gate_hi = i + 1;
            P->rots.push_back(U->rotation(g.q0, g.op - STAB_RX, g.param));
            P->rot_step.push_back((int64_t)P->steps.size());
            P->steps.push_back(s);
            in_run = false;
            continue;
        }
        uint8_t op = g.op;
        if (backward && op == STAB_S) op = STAB_SDG;
        else if (backward && op == STAB_SDG) op = STAB_S;
        if (!in_run) {
            SpStep s{};
            s.kind = SP_CLIFF;
            s.first = (int)P->gates.size();
            s.count = 0;
            s.gate_lo = i;
            s.gate_hi = i + 1;
            P->steps.push_back(s);
            in_run = true;
        }
        SpStep &s = P->steps.back();
        P->gates.push_back(SpGate{op, g.q0, g.q1, 0});
        U->apply(P->gates.back());
        s.count++;
        s.gate_lo = std::min(s.gate_lo, i);
        s.gate_hi = std::max(s.gate_hi, i + 1);
    }
}

// What the device needs of a plan's whole Clifford part: the tableau, then the
// masks of its x bits.
struct SpFinal {
    SpTab tab[64];
    uint64_t xcol[32];
};

void fill_final(const SpPull &U, SpFinal *f) {
    std::memset((void *)f, 0, sizeof *f);
    U.tableau(f->tab);
    for (int q = 0; q < U.n; ++q) f->xcol[q] = U.xcol(q);
}

// One direction of a loaded circuit.
struct SpDir {
    SpPlan plan;
    SpBuf rots, fin, chunks;
};

}  // namespace

struct stab_sparse {
    int n = 0;
    int device = 0;
    cudaStream_t st = nullptr;
    bool own_st = false;
    stab_opts opts{};
    int64_t max_terms = 0, cap = 0, threshold = 0;
    bool loaded = false;
    std::vector<stab_gate> gates;
    std::vector<double> thetas_h;
    int64_t n_params = 0;
    SpDir fwd, bwd;
    SpBuf thetas, cs, keys[2], vals[2], table, partner, tiles, init, run, partial, dterms, fin,
        chunks;
    int grid = 0;
    void *pinned = nullptr;
    size_t pinned_bytes = 0;
    std::vector<int64_t> history;
    stab_ctx *dense = nullptr;
    int32_t regrows = 0;
    bool table_dirty = false;   // a run that failed left slots claimed

    int dalloc(SpBuf &b, size_t bytes) {
        if (b.p && b.bytes >= bytes) return STAB_OK;
        dfree(b);
        bytes = (bytes + 255) & ~(size_t)255;
        if (bytes == 0) bytes = 256;
        void *p = nullptr;
        if (opts.alloc) {
            p = opts.alloc(bytes, (void *)st, opts.alloc_user);
            if (!p) return STAB_E_NOMEM;
        } else {
            cudaError_t e = cudaMallocAsync(&p, bytes, st);
            if (e != cudaSuccess) {
                (void)cudaGetLastError();
                if (e == cudaErrorMemoryAllocation) return STAB_E_NOMEM;
                record_cuda_error(e);
                return STAB_E_CUDA;
            }
        }
        b.p = p;
        b.bytes = bytes;
        return STAB_OK;
    }
    void dfree(SpBuf &b) {
        if (!b.p) return;
        cudaStreamSynchronize(st);
        if (opts.free) opts.free(b.p, b.bytes, (void *)st, opts.alloc_user);
        else cudaFreeAsync(b.p, st);
        b.p = nullptr;
        b.bytes = 0;
    }
    int stage(size_t bytes) {
        if (pinned && pinned_bytes >= bytes) return STAB_OK;
        if (pinned) cudaFreeHost(pinned);
        pinned = nullptr;
        pinned_bytes = 0;
        SCK(cudaMallocHost(&pinned, bytes));
        pinned_bytes = bytes;
        return STAB_OK;
    }

    int clear(int64_t c) {
        SCK(cudaMemsetAsync(table.p, 0xff, (size_t)8 << sp_table_log(c), st));
        SCK(cudaMemsetAsync(partner.p, 0xff, (size_t)c * 4, st));
        return STAB_OK;
    }

    // Capacity `c` for the list; the live list (count terms in buffer `from`)
    // moves to buffer 0.  The table's slots are all free, the partners all absent.
    int reserve(int64_t c, int from, int64_t count) {
        if (c <= cap && from == 0) return STAB_OK;
        c = std::max(c, cap);
        const bool grow = c > cap;
        cap = 0;   // until all buffers are there: after a failure the next run starts over
        SpBuf nk, nv;
        std::swap(nk, keys[0]);
        std::swap(nv, vals[0]);
        int r = dalloc(keys[0], (size_t)c * 8);
        if (r == STAB_OK) r = dalloc(vals[0], (size_t)c * 8);
        if (r == STAB_OK && count > 0) {
            const SpBuf &ok = from == 0 ? nk : keys[1], &ov = from == 0 ? nv : vals[1];
            cudaError_t e = cudaMemcpyAsync(keys[0].p, ok.p, (size_t)count * 8,
                                            cudaMemcpyDeviceToDevice, st);
            if (e == cudaSuccess)
                e = cudaMemcpyAsync(vals[0].p, ov.p, (size_t)count * 8, cudaMemcpyDeviceToDevice,
                                    st);
            if (e != cudaSuccess) {
                record_cuda_error(e);
                r = STAB_E_CUDA;
            }
        }
        dfree(nk);
        dfree(nv);
        SRC(r);
        if (grow) {
            SRC(dalloc(keys[1], (size_t)c * 8));
            SRC(dalloc(vals[1], (size_t)c * 8));
            SRC(dalloc(partner, (size_t)c * 4));
            SRC(dalloc(tiles, (size_t)sp_tiles(c, grid) * 8));
            SRC(dalloc(table, (size_t)8 << sp_table_log(c)));
            SRC(clear(c));
        }
        cap = c;
        return STAB_OK;
    }

    ~stab_sparse() {
        if (st) cudaStreamSynchronize(st);
        for (SpBuf *b : {&thetas, &cs, &keys[0], &keys[1], &vals[0], &vals[1], &table, &partner,
                         &tiles, &init, &run, &partial, &dterms, &fin, &chunks, &fwd.rots,
                         &fwd.fin, &fwd.chunks, &bwd.rots, &bwd.fin, &bwd.chunks})
            dfree(*b);
        if (pinned) cudaFreeHost(pinned);
        if (dense) stab_destroy(dense);
        if (own_st && st) cudaStreamDestroy(st);
    }
};

namespace {

// Runs the plan on a list.  With `sum`, the x-free sum of the last list's images
// is queued behind it and returned there (of no use when the run stopped).
int sp_run(stab_sparse *s, const SpDir &D, bool backward, const std::vector<uint64_t> &k0,
           const std::vector<double> &v0, SpRun *R, int64_t *order_max, double *sum) {
    const int64_t S = (int64_t)D.plan.steps.size(), rots = (int64_t)D.plan.rots.size();
    const int64_t n0 = (int64_t)k0.size();
    s->history.clear();
    s->regrows = 0;
    SRC(s->reserve(std::min(s->max_terms, std::max(kSpMinCap, 4 * n0)), 0, 0));
    if (n0 > s->cap) return STAB_E_RANGE;
    if (s->table_dirty) {
        SRC(s->clear(s->cap));
        s->table_dirty = false;
    }
    // state and orders come back in one copy; initial list and first order go in one
    const size_t back = sizeof(SpState) + (size_t)(rots + 1) * 8, there = (size_t)n0 * 16;
    const size_t back_pad = (back + 63) & ~(size_t)63;
    SRC(s->dalloc(s->run, back));
    SRC(s->dalloc(s->init, std::max<size_t>(there, 16)));
    SRC(s->stage(back_pad + there + sizeof(SpState) + 8));
    char *h = (char *)s->pinned;
    uint64_t *h_init = (uint64_t *)(h + back_pad);
    char *h_state = h + back_pad + there;
    std::copy(k0.begin(), k0.end(), h_init);
    std::memcpy(h_init + n0, v0.data(), (size_t)n0 * 8);
    SpState first{};
    first.count = n0;
    std::memcpy(h_state, &first, sizeof first);
    std::memcpy(h_state + sizeof first, &n0, 8);
    if (n0) SCK(cudaMemcpyAsync(s->init.p, h_init, there, cudaMemcpyHostToDevice, s->st));
    SCK(cudaMemcpyAsync(s->run.p, h_state, sizeof first + 8, cudaMemcpyHostToDevice, s->st));

    SpRunArgs a{};
    a.st = (SpState *)s->run.p;
    a.counts = (int64_t *)((char *)s->run.p + sizeof(SpState));
    a.rots = (const SpRot *)D.rots.p;
    a.cs = (const double *)s->cs.p;
    a.n_rot = (int32_t)rots;
    a.n = s->n;
    a.inverse = backward ? 1 : 0;
    a.grid = s->grid;
    a.threshold = s->threshold;
    a.init = (const uint64_t *)s->init.p;
    // a list that can outgrow one CTA's memory needs the grid behind it
    const int64_t small = std::min<int64_t>(s->cap, kSpSmallCap);
    bool grid = n0 > small;
    if (grid) {
        SCK(cudaMemcpyAsync(s->keys[0].p, s->init.p, (size_t)n0 * 8, cudaMemcpyDeviceToDevice,
                            s->st));
        SCK(cudaMemcpyAsync(s->vals[0].p, (char *)s->init.p + (size_t)n0 * 8, (size_t)n0 * 8,
                            cudaMemcpyDeviceToDevice, s->st));
    }
    int64_t bound = n0;
    for (int64_t r = 0; r < rots && bound <= small; ++r) bound *= 2;
    const bool one_cta = !grid;
    grid = rots > 0 && (grid || bound > small);
    SpState at{};
    for (bool again = false;; again = true) {
        a.cap = s->cap;
        for (int b = 0; b < 2; ++b) {
            a.keys[b] = (uint64_t *)s->keys[b].p;
            a.vals[b] = (double *)s->vals[b].p;
        }
        a.table = (uint64_t *)s->table.p;
        a.partner = (int32_t *)s->partner.p;
        a.tiles = (uint64_t *)s->tiles.p;
        if (one_cta && !again) SCK(launch_sp_small(a, s->st));
        if (grid) SCK(launch_sp_run(a, s->st));
        if (sum)
            SCK(launch_sp_xfree(a, ((const SpFinal *)D.fin.p)->xcol, (const SpChunk *)D.chunks.p,
                                (double *)s->partial.p, s->st));
        SCK(cudaMemcpyAsync(h, s->run.p, back, cudaMemcpyDeviceToHost, s->st));
        SCK(cudaStreamSynchronize(s->st));
        std::memcpy(&at, h, sizeof at);
        if (at.err != 0) {   // a table probe or a wait ran out (never expected)
            s->table_dirty = true;
            return at.err == 1 ? STAB_E_NOMEM : STAB_E_CUDA;
        }
        if (at.stop != SP_OVERFLOW || s->cap >= s->max_terms) break;
        SRC(s->reserve(std::min(s->max_terms, s->cap * 8), at.buf, at.count));
        s->regrows++;
        at.buf = 0;
        at.stop = SP_RUNNING;
        at.arrived = 0;
        std::memcpy(h_state, &at, sizeof at);
        SCK(cudaMemcpyAsync(s->run.p, h_state, sizeof at, cudaMemcpyHostToDevice, s->st));
    }
    R->buf = at.buf;
    R->count = at.count;
    // stopped behind rotation rot - 1 (threshold) or before rotation rot (no room)
    R->step = S;
    if (at.stop == SP_THRESHOLD) R->step = D.plan.rot_step[at.rot - 1] + 1;
    if (at.stop == SP_OVERFLOW) R->step = D.plan.rot_step[at.rot];
    R->stopped = at.stop == SP_OVERFLOW || R->step < S;
    const int64_t *counts = (const int64_t *)(h + sizeof(SpState));
    *order_max = n0;
    int64_t order = n0;
    for (int64_t j = 0, r = 0; j < R->step; ++j) {
        if (D.plan.steps[(size_t)j].kind == SP_ROT) order = counts[++r];
        s->history.push_back(order);
        *order_max = std::max(*order_max, order);
    }
    if (sum) *sum = at.value;
    return STAB_OK;
}

// The chunk table of the Clifford gates the list before step R.step has behind
// it: the loaded one, or one of the first steps alone.
int sp_chunks(stab_sparse *s, const SpDir &D, const SpRun &R, const SpChunk **out) {
    *out = (const SpChunk *)D.chunks.p;
    if (R.step == (int64_t)D.plan.steps.size()) return STAB_OK;
    SpPull U(s->n);
    for (int64_t j = 0; j < R.step; ++j) {
        const SpStep &st = D.plan.steps[(size_t)j];
        for (int g = 0; st.kind == SP_CLIFF && g < st.count; ++g)
            U.apply(D.plan.gates[(size_t)(st.first + g)]);
    }
    SRC(s->dalloc(s->fin, sizeof(SpFinal)));
    SRC(s->dalloc(s->chunks, kSpChunkEntries * sizeof(SpChunk)));
    SRC(s->stage(sizeof(SpFinal)));
    fill_final(U, (SpFinal *)s->pinned);
    SCK(cudaMemcpyAsync(s->fin.p, s->pinned, sizeof(SpFinal), cudaMemcpyHostToDevice, s->st));
    SCK(launch_sp_chunks(((const SpFinal *)s->fin.p)->tab, s->n, (SpChunk *)s->chunks.p, s->st));
    SCK(cudaStreamSynchronize(s->st));   // the staging buffer may be reused
    *out = (const SpChunk *)s->chunks.p;
    return STAB_OK;
}

int sp_encode_terms(int n, const stab_term *O, int64_t nt, std::vector<uint64_t> *k,
                    std::vector<double> *v) {
    k->clear();
    v->clear();
    if (nt < 0) return STAB_E_RANGE;
    if (nt > 0 && !O) return STAB_E_INVAL;
    const uint64_t lim = n >= 64 ? ~0ull : (1ull << n);
    std::map<uint64_t, double> acc;
    for (int64_t i = 0; i < nt; ++i) {
        if ((n < 64 && (O[i].x >= lim || O[i].z >= lim))) return STAB_E_INVAL;
        if (!std::isfinite(O[i].coeff)) return STAB_E_NONFINITE;
        acc[O[i].z | (O[i].x << n)] += O[i].coeff;
    }
    for (auto &kv : acc) {
        if (kv.second == 0.0) continue;
        k->push_back(kv.first);
        v->push_back(kv.second);
    }
    return STAB_OK;
}

void fill_info(stab_sparse *s, const SpRun &R, int64_t order_max, int64_t dense_gates,
               stab_sparse_info *info) {
    if (!info) return;
    info->order_final = R.count;
    info->order_max = order_max;
    info->steps = (int64_t)s->history.size();
    info->dense_gates = dense_gates;
    info->regrows = s->regrows;
    info->reserved = 0;
}

}  // namespace

extern "C" {

int stab_sparse_create(int n, int64_t max_terms, const stab_opts *opts, stab_sparse **out) {
    if (!out) return STAB_E_INVAL;
    *out = nullptr;
    if (n < 1 || n > STAB_SPARSE_MAX_QUBITS) return STAB_E_RANGE;
    if (max_terms < 1 || max_terms > kSpMaxCap) return STAB_E_RANGE;
    stab_opts o;
    stab_default_opts(&o);
    if (opts) o = *opts;
    if ((o.alloc == nullptr) != (o.free == nullptr)) return STAB_E_INVAL;
    stab_sparse *s = new (std::nothrow) stab_sparse();
    if (!s) return STAB_E_NOMEM;
    s->n = n;
    s->max_terms = max_terms;
    s->threshold = n <= STAB_MAX_QUBITS ? (int64_t)1 << (2 * n - 4 > 0 ? 2 * n - 4 : 0) : 0;
    if (s->threshold >= max_terms) s->threshold = max_terms / 2;
    int dev = o.device;
    cudaError_t e = cudaSuccess;
    if (dev < 0) e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaSetDevice(dev);
    if (e == cudaSuccess) {
        s->device = dev;
        if (o.stream || o.stream_given) {
            s->st = (cudaStream_t)o.stream;
        } else {
            e = cudaStreamCreateWithFlags(&s->st, cudaStreamNonBlocking);
            s->own_st = (e == cudaSuccess);
        }
    }
    if (e != cudaSuccess) {
        record_cuda_error(e);
        delete s;
        return STAB_E_CUDA;
    }
    // the dense context (created on demand) queues on the same stream
    o.device = dev;
    o.stream = (void *)s->st;
    o.stream_given = 1;
    s->opts = o;
    int r = s->dalloc(s->partial, (size_t)kSpMaxBlocks * 8);
    if (r == STAB_OK) {
        e = sp_run_grid(dev, &s->grid);
        if (e != cudaSuccess) {
            record_cuda_error(e);
            r = STAB_E_CUDA;
        }
    }
    if (r != STAB_OK) {
        delete s;
        return r;
    }
    *out = s;
    return STAB_OK;
}

int stab_sparse_destroy(stab_sparse *s) {
    if (!s) return STAB_OK;
    cudaSetDevice(s->device);
    delete s;
    return STAB_OK;
}

int stab_sparse_load_circuit(stab_sparse *s, const stab_gate *gates, int64_t m,
                             const double *thetas, int64_t n_params) {
    if (!s) return STAB_E_INVAL;
    SRC(validate_gates(s->n, gates, m, n_params, nullptr));
    SRC(validate_thetas(thetas, n_params));
    SCK(cudaSetDevice(s->device));
    s->loaded = false;
    s->gates.assign(gates, gates + m);
    s->thetas_h.assign(thetas, thetas + n_params);
    s->n_params = n_params;
    const size_t bt = (size_t)n_params * 8;
    SRC(s->dalloc(s->thetas, std::max<size_t>(bt, 8)));
    SRC(s->dalloc(s->cs, std::max<size_t>(2 * bt, 8)));
    SpDir *dirs[2] = {&s->fwd, &s->bwd};
    size_t need = bt;
    std::vector<SpFinal> fin(2);
    for (int k = 0; k < 2; ++k) {
        SpDir &D = *dirs[k];
        SpPull U(s->n);
        build_sp_plan(s->gates, k == 1, &D.plan, &U);
        fill_final(U, &fin[k]);
        const size_t br = D.plan.rots.size() * sizeof(SpRot);
        SRC(s->dalloc(D.rots, std::max<size_t>(br, 8)));
        SRC(s->dalloc(D.fin, sizeof(SpFinal)));
        SRC(s->dalloc(D.chunks, kSpChunkEntries * sizeof(SpChunk)));
        need += br + sizeof(SpFinal);
    }
    SRC(s->stage(need));
    char *h = (char *)s->pinned;
    auto put = [&](const SpBuf &d, const void *src, size_t bytes) {
        if (bytes == 0) return cudaSuccess;
        std::memcpy(h, src, bytes);
        const cudaError_t e = cudaMemcpyAsync(d.p, h, bytes, cudaMemcpyHostToDevice, s->st);
        h += bytes;
        return e;
    };
    SCK(put(s->thetas, s->thetas_h.data(), bt));
    SCK(launch_sp_cos_sin((const double *)s->thetas.p, n_params, (double *)s->cs.p, s->st));
    for (int k = 0; k < 2; ++k) {
        SpDir &D = *dirs[k];
        SCK(put(D.rots, D.plan.rots.data(), D.plan.rots.size() * sizeof(SpRot)));
        SCK(put(D.fin, &fin[k], sizeof(SpFinal)));
        SCK(launch_sp_chunks(((const SpFinal *)D.fin.p)->tab, s->n, (SpChunk *)D.chunks.p, s->st));
    }
    SCK(cudaStreamSynchronize(s->st));
    s->loaded = true;
    return STAB_OK;
}

int stab_sparse_set_dense_threshold(stab_sparse *s, int64_t order) {
    if (!s) return STAB_E_INVAL;
    if (order < 0 || (order > 0 && s->n > STAB_MAX_QUBITS)) return STAB_E_RANGE;
    s->threshold = order;
    return STAB_OK;
}

int stab_sparse_expect(stab_sparse *s, const stab_term *O, int64_t n_terms, double *out,
                       stab_sparse_info *info) {
    if (!s || !out) return STAB_E_INVAL;
    if (!s->loaded) return STAB_E_STATE;
    SCK(cudaSetDevice(s->device));
    std::vector<uint64_t> k0;
    std::vector<double> v0;
    SRC(sp_encode_terms(s->n, O, n_terms, &k0, &v0));
    SpRun R;
    int64_t order_max = 0;
    if (k0.empty()) {
        s->history.clear();
        *out = 0.0;
        fill_info(s, R, 0, -1, info);
        return STAB_OK;
    }
    double value = 0.0;
    SRC(sp_run(s, s->bwd, true, k0, v0, &R, &order_max, &value));
    int64_t dense_gates = -1;
    if (R.stopped) {
        // the rest of the circuit (backward: gates [0, g)) on the dense vector
        if (s->n > STAB_MAX_QUBITS) return STAB_E_RANGE;
        const int64_t g = s->bwd.plan.steps[R.step].gate_hi;
        if (!s->dense) SRC(stab_create(s->n, &s->opts, &s->dense));
        SRC(stab_load_circuit(s->dense, s->gates.data(), g, s->thetas_h.data(), s->n_params));
        SRC(s->dalloc(s->dterms, (size_t)std::max<int64_t>(R.count, 1) * sizeof(DevTerm)));
        const SpChunk *chunks;
        SRC(sp_chunks(s, s->bwd, R, &chunks));
        SCK(launch_sp_images((const uint64_t *)s->keys[R.buf].p, (const double *)s->vals[R.buf].p,
                             R.count, s->n, chunks, (DevTerm *)s->dterms.p, nullptr, s->st));
        SRC(expect_device_terms(s->dense, (const DevTerm *)s->dterms.p, R.count, out));
        dense_gates = g;
    } else {
        *out = value;
    }
    fill_info(s, R, order_max, dense_gates, info);
    return STAB_OK;
}

int stab_sparse_generator(stab_sparse *s, int k, int64_t max_out, stab_term *out,
                          int64_t *n_out, stab_sparse_info *info) {
    if (!s || !n_out || max_out < 0 || (max_out > 0 && !out)) return STAB_E_INVAL;
    if (!s->loaded) return STAB_E_STATE;
    if (k < 0 || k >= s->n) return STAB_E_RANGE;
    SCK(cudaSetDevice(s->device));
    const std::vector<uint64_t> k0 = {1ull << k};
    const std::vector<double> v0 = {1.0};
    const int64_t keep = s->threshold;
    s->threshold = 0;   // generators stay on the list
    SpRun R;
    int64_t order_max = 0;
    const int r = sp_run(s, s->fwd, false, k0, v0, &R, &order_max, nullptr);
    s->threshold = keep;
    SRC(r);
    if (R.stopped) return STAB_E_RANGE;
    *n_out = R.count;
    fill_info(s, R, order_max, -1, info);
    if (R.count > max_out) return STAB_E_RANGE;
    if (R.count == 0) return STAB_OK;
    const SpChunk *chunks;
    SRC(sp_chunks(s, s->fwd, R, &chunks));
    // the records are made there: 96,000 of them here took as long as the last rotations
    const size_t bytes = (size_t)R.count * sizeof(stab_term);
    SRC(s->dalloc(s->dterms, bytes));
    SRC(s->stage(bytes));
    SCK(launch_sp_images((const uint64_t *)s->keys[R.buf].p, (const double *)s->vals[R.buf].p,
                         R.count, s->n, chunks, nullptr, (stab_term *)s->dterms.p, s->st));
    SCK(cudaMemcpyAsync(s->pinned, s->dterms.p, bytes, cudaMemcpyDeviceToHost, s->st));
    SCK(cudaStreamSynchronize(s->st));
    // 2.3 MB (96,000 terms): 90 us on one core
    constexpr size_t kPart = 256 << 10;
    std::vector<std::function<void()>> jobs;
    for (size_t at = 0; at < bytes; at += kPart)
        jobs.push_back([=] {
            std::memcpy((char *)out + at, (const char *)s->pinned + at, std::min(kPart, bytes - at));
        });
    HostPool::run(jobs);
    return STAB_OK;
}

int stab_sparse_order_history(stab_sparse *s, int64_t *orders, int64_t max, int64_t *count) {
    if (!s || !count || max < 0 || (max > 0 && !orders)) return STAB_E_INVAL;
    const int64_t c = (int64_t)s->history.size();
    *count = c;
    for (int64_t i = 0; i < std::min(c, max); ++i) orders[i] = s->history[(size_t)i];
    return STAB_OK;
}

}  // extern "C"
