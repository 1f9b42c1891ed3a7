// k_unitary.cu -- plans at n <= 4 through the unitaries of their segments.
//
// Every map of the method is P -> U P U^dagger for a 2^n x 2^n unitary U, so a
// stretch of the plan is carried by that one matrix: the transfer matrix of
// the stretch (4^n x 4^n in the Pauli basis) has 4^n - 1 nontrivial columns,
// U has 4^n complex entries.  At n = 4 a wire pass costs 255 columns x 64
// groups x 9 FP64 instructions through the columns and 256 entries x 8
// through U, 1/70 of the work, and with that little work the plan can be cut
// into many segments that run at once and are multiplied in a tree.  The
// Pauli coefficients of the evolved generators, of rho and of <O> are read
// off at the end.  Measured on a GB300, new angles every call, against the
// columns of the later parts swept as vectors beside the first part (the
// gradient: pairs of vectors through the parts): generators and <O> at n = 4,
// 60,200 gates 2.50 -> 0.130 ms, 2,000 gates 149 -> 68 us, n = 3, 20,000 gates
// 700 -> 57 us; gradients at n = 4, 4,000 gates 909 -> 112 us, 60,200 gates
// 12.2 -> 0.237 ms, n = 3, 20,000 gates 3.19 -> 0.092 ms, n = 2, 4,000 gates 354 ->
// 74 us; short plans: n = 4, 260 gates 66 -> 50 us, n = 2, 100 gates 108 -> 57 us.
//
// Exactness on Clifford circuits: H is kept as [[1, 1], [1, -1]] and the
// factor sqrt(2) of an odd number of H gates as a parity beside the matrix
// (an even number is a power of two), so Clifford gates only move, negate, add
// and double entries and U P U^dagger comes out as an exact signed string.
// Global phases drop out of U P U^dagger and are not kept.
#include <cuda_runtime.h>

#include "device_ops.cuh"
#include "launch.h"

namespace stab {

namespace {

__device__ __forceinline__ double2 cmul(double2 a, double2 b) {
    return make_double2(fma(a.x, b.x, -a.y * b.y), fma(a.x, b.y, a.y * b.x));
}
// acc + a b
__device__ __forceinline__ double2 cfma(double2 a, double2 b, double2 acc) {
    return make_double2(fma(-a.y, b.y, fma(a.x, b.x, acc.x)),
                        fma(a.y, b.x, fma(a.x, b.y, acc.y)));
}
// acc + a conj(b)
__device__ __forceinline__ double2 cfma_conj(double2 a, double2 b, double2 acc) {
    return make_double2(fma(a.y, b.y, fma(a.x, b.x, acc.x)),
                        fma(a.y, b.x, fma(-a.x, b.y, acc.y)));
}

__device__ __forceinline__ double2 scaled(double2 a, double f) {
    return make_double2(f * a.x, f * a.y);
}
constexpr double kInvSqrt2 = 0.70710678118654752440;

// ---------------------------------------------------------------- wire maps

// M <- G M for one single-qubit gate, rows r0 = (m0, m1), r1 = (m2, m3);
// odd: H gates so far mod 2 (their factor sqrt(2) kept in M).
__device__ __forceinline__ void left_gate(double2 (&m)[4], const RawGate &g, const double *thetas,
                                          int &odd) {
    if (g.op >= 8) {
        double s, c;
        sincos(0.5 * thetas[g.param], &s, &c);
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const double2 a = m[k], b = m[2 + k];
            if (g.op == 8) {          // c a - i s b, c b - i s a
                m[k] = make_double2(fma(s, b.y, c * a.x), fma(-s, b.x, c * a.y));
                m[2 + k] = make_double2(fma(s, a.y, c * b.x), fma(-s, a.x, c * b.y));
            } else if (g.op == 9) {   // c a - s b, s a + c b
                m[k] = make_double2(fma(-s, b.x, c * a.x), fma(-s, b.y, c * a.y));
                m[2 + k] = make_double2(fma(s, a.x, c * b.x), fma(s, a.y, c * b.y));
            } else {                  // (c - i s) a, (c + i s) b
                m[k] = make_double2(fma(s, a.y, c * a.x), fma(-s, a.x, c * a.y));
                m[2 + k] = make_double2(fma(-s, b.y, c * b.x), fma(s, b.x, c * b.y));
            }
        }
        return;
    }
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const double2 a = m[k], b = m[2 + k];
        switch (g.op) {
        case 0: {   // H times sqrt(2); every second one takes the pair's factor 2 out
            const double w = odd ? 0.5 : 1.0;
            m[k] = make_double2(w * (a.x + b.x), w * (a.y + b.y));
            m[2 + k] = make_double2(w * (a.x - b.x), w * (a.y - b.y));
            break;
        }
        case 1: m[2 + k] = make_double2(-b.y, b.x); break;            // S
        case 2: m[2 + k] = make_double2(b.y, -b.x); break;            // S^dagger
        case 3: m[k] = b; m[2 + k] = a; break;                        // X
        case 4:                                                       // Y
            m[k] = make_double2(b.y, -b.x);
            m[2 + k] = make_double2(-a.y, a.x);
            break;
        case 5: m[2 + k] = make_double2(-b.x, -b.y); break;           // Z
        default: break;
        }
    }
    if (g.op == 0) odd ^= 1;
}

__device__ __forceinline__ void store_map(UniMap *out, const double2 (&m)[4]) {
    double2 *f = reinterpret_cast<double2 *>(out->f);
    f[0] = m[0];   // row bit 0: itself, its partner
    f[1] = m[1];
    f[2] = m[3];   // row bit 1
    f[3] = m[2];
}

// A thread per run, its gates in order.  Bound by the sincos of its gates.
__global__ void __launch_bounds__(64) k_uni_maps_seq(const UniRun *runs, int n_runs,
                                                     const RawGate *gates, const double *thetas,
                                                     UniMap *maps) {
    const int i = (int)(blockIdx.x * blockDim.x + threadIdx.x);
    if (i >= n_runs) return;
    const UniRun r = runs[i];
    int odd = r.parity & 1;
    double2 m[4] = {{1.0, 0.0}, {0.0, 0.0}, {0.0, 0.0}, {1.0, 0.0}};
    for (int k = 0; k < r.count; ++k) left_gate(m, gates[r.first + k], thetas, odd);
    store_map(maps + i, m);
}

// A warp per run: lane l composes a contiguous chunk of the run's gates, then
// an ordered shuffle tree multiplies the chunks (later times earlier).
__global__ void __launch_bounds__(128) k_uni_maps_warp(const UniRun *runs, int n_runs,
                                                       const RawGate *gates,
                                                       const double *thetas, UniMap *maps) {
    const int w = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5);
    const int lane = (int)(threadIdx.x & 31u);
    if (w >= n_runs) return;   // whole warps
    const UniRun r = runs[w];
    const int count = r.count;
    const int per = (count + 31) / 32;
    const int k0 = min(lane * per, count), k1 = min(k0 + per, count);
    // H gates before this lane's chunk, mod 2
    int h = 0;
    for (int k = k0; k < k1; ++k) h ^= gates[r.first + k].op == 0;
    const uint32_t hs = __ballot_sync(0xffffffffu, h);
    int odd = (r.parity ^ __popc(hs & ((1u << lane) - 1u))) & 1;
    double2 m[4] = {{1.0, 0.0}, {0.0, 0.0}, {0.0, 0.0}, {1.0, 0.0}};
    for (int k = k0; k < k1; ++k) left_gate(m, gates[r.first + k], thetas, odd);
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        double2 o[4], p[4];
#pragma unroll
        for (int j = 0; j < 4; ++j)
            o[j] = make_double2(__shfl_down_sync(0xffffffffu, m[j].x, d),
                                __shfl_down_sync(0xffffffffu, m[j].y, d));
        if ((lane & (2 * d - 1)) == 0) {
#pragma unroll
            for (int a = 0; a < 2; ++a)
#pragma unroll
                for (int b = 0; b < 2; ++b)
                    p[2 * a + b] = cfma(o[2 * a + 1], m[2 + b], cmul(o[2 * a], m[b]));
#pragma unroll
            for (int j = 0; j < 4; ++j) m[j] = p[j];
        }
    }
    if (lane == 0) store_map(maps + w, m);
}

// ---------------------------------------------------------------- segments

// One op on the entry (re, im) of row `row`, the rows of a column in
// consecutive lanes.
__device__ __forceinline__ void apply_wire(const double *map, int d, int row, double &re,
                                           double &im) {
    const double pr = __shfl_xor_sync(0xffffffffu, re, d);
    const double pi = __shfl_xor_sync(0xffffffffu, im, d);
    const double2 *f = reinterpret_cast<const double2 *>(map) + ((row & d) ? 2 : 0);
    const double2 m = f[0], q = f[1];
    const double nr = fma(-q.y, pi, fma(q.x, pr, fma(-m.y, im, m.x * re)));
    im = fma(q.y, pr, fma(q.x, pi, fma(m.y, re, m.x * im)));
    re = nr;
}

__device__ __forceinline__ void apply_two_qubit(const UniOp &op, int lane, int row, double &re,
                                                double &im) {
    if (op.kind == UK_CX) {
        const int from = lane ^ (((row >> op.q0) & 1) << op.q1);
        re = __shfl_sync(0xffffffffu, re, from);
        im = __shfl_sync(0xffffffffu, im, from);
    } else {
        const uint32_t neg = (uint32_t)((row >> op.q0) & (row >> op.q1) & 1);
        re = flip(re, neg);
        im = flip(im, neg);
    }
}

template <int N>
struct UCfg {
    static constexpr int D = 1 << N;
    static constexpr int E = D * D;
    static constexpr int T = E < 32 ? 32 : E;
};

constexpr int kUniStage = 256;   // ops staged at a time

// Matrices are stored by columns: entry (row, col) at col * D + row.

// out(row, col) = sum_k later(row, k) earlier(k, col), scaled, one entry per thread.
template <int N>
__device__ __forceinline__ double2 product_entry(const double2 *later, const double2 *earlier,
                                                 int row, int col, double scale) {
    constexpr int D = UCfg<N>::D;
    double2 acc = make_double2(0.0, 0.0);
#pragma unroll
    for (int k = 0; k < D; ++k) acc = cfma(later[k * D + row], earlier[col * D + k], acc);
    return make_double2(scale * acc.x, scale * acc.y);
}

// One CTA per segment.  A thread holds one entry of U; the 2^n rows of a
// column sit in one warp, so a wire pass gets its partner entry and a CNOT
// its source entry by shuffles, and the warps never wait for one another
// inside a stage.  Eight FP64 instructions per entry and wire pass: with
// eight warps on four sub-partitions (n = 4) the FP64 pipe is the bound.
// Then the tree: the second CTA to reach a node multiplies its two children
// and goes on upward, the first one leaves, so nothing waits.
template <int N>
__global__ void __launch_bounds__(UCfg<N>::T) k_uni_segments(UniArgs a) {
    constexpr int D = UCfg<N>::D, E = UCfg<N>::E, T = UCfg<N>::T;
    __shared__ UniOp sop[kUniStage];
    __shared__ __align__(16) double smap[kUniStage * 8];
    __shared__ double2 sa[E], sb[E];
    __shared__ int s_go;
    const UniSeg sg = a.segs[blockIdx.x];
    const int t = (int)threadIdx.x;
    const int row = t & (D - 1), col = t / D;
    const int lane = t & 31;
    double re = row == col ? 1.0 : 0.0, im = 0.0;
    int map_at = sg.map_first;
    for (int o0 = 0; o0 < sg.n_ops; o0 += kUniStage) {
        const int no = min(kUniStage, sg.n_ops - o0);
        int wires = 0;
        if (o0) __syncthreads();
        for (int k = t; k < no; k += T) sop[k] = a.ops[sg.op_first + o0 + k];
        // at most `no` maps belong to this stage; those that exist are copied
        const int nm = min(no, sg.map_first + sg.n_maps - map_at);
        const double2 *src = reinterpret_cast<const double2 *>(a.maps + map_at);
        for (int k = t; k < 4 * nm; k += T) reinterpret_cast<double2 *>(smap)[k] = src[k];
        __syncthreads();
        for (int k = 0; k < no; ++k) {
            const UniOp op = sop[k];
            if (op.kind == UK_WIRE) {
                apply_wire(smap + 8 * wires, 1 << op.q0, row, re, im);
                ++wires;
            } else {
                apply_two_qubit(op, lane, row, re, im);
            }
        }
        map_at += wires;
    }
    // up the part's tree
    const UniPart P = a.parts[sg.part];
    int node = P.node, level_n = P.n_seg, idx = sg.index, parity = sg.parity;
    double2 u = make_double2(re, im);
    const bool live = t < E;
    while (true) {
        const int at = node + idx;
        if (live) a.nodes[(size_t)at * E + t] = u;
        if (t == 0) a.node_parity[at] = parity;
        if (level_n == 1) return;   // the root
        const int up_n = (level_n + 1) / 2, up = node + level_n;
        if (idx == level_n - 1 && !(idx & 1)) {   // no sibling: the parent is this matrix
            node = up;
            level_n = up_n;
            idx >>= 1;
            continue;
        }
        __syncthreads();
        if (t == 0) {
            __threadfence();
            int32_t *cnt = a.node_count + up + (idx >> 1);
            const int before = atomicAdd(cnt, 1);
            if (before) *cnt = 0;   // both children are here: ready for the next launch
            __threadfence();
            s_go = before;
        }
        __syncthreads();
        if (!s_go) return;
        // the sibling: index idx ^ 1 of this level
        const int sib = node + (idx ^ 1);
        double2 *mine = (idx & 1) ? sa : sb, *other = (idx & 1) ? sb : sa;
        if (live) {
            mine[t] = u;
            const double2 *sp = a.nodes + (size_t)sib * E + t;
            other[t] = make_double2(__ldcg(&sp->x), __ldcg(&sp->y));
        }
        const int sib_parity = __ldcg(a.node_parity + sib);
        __syncthreads();
        // sa: the later child, sb: the earlier one
        const double scale = (parity & sib_parity) ? 0.5 : 1.0;
        if (live) u = product_entry<N>(sa, sb, row, col, scale);
        parity ^= sib_parity;
        node = up;
        level_n = up_n;
        idx >>= 1;
        __syncthreads();
    }
}

// ---------------------------------------------------------------- read-out

// Pauli coefficients of a Hermitian matrix B given by its entries
// h[x * D + b] = B(b, b ^ x): coefficient of P(x, z) = 2^-n Tr(P B) with
// P(x, z)|b> = i^|x & z| (-1)^{z.b} |b ^ x>, at index z | x << n.  The entries
// b and b ^ x are conjugates, so for x > 0 the sum runs over one b of each
// pair (x's highest bit clear) and keeps the part that does not cancel.
template <int N>
__device__ __forceinline__ double pauli_coefficient(const double2 *h, int x, int z) {
    constexpr int D = UCfg<N>::D;
    double sum = 0.0;
    if (x == 0) {
#pragma unroll
        for (int b = 0; b < D; ++b) sum += flip(h[b].x, (uint32_t)__popc(z & b) & 1u);
        return sum * (1.0 / D);
    }
    const int k = __popc(x & z) & 3;
    const int top = 31 - __clz(x);
    const double *v = reinterpret_cast<const double *>(h + x * D) + (k & 1);
#pragma unroll
    for (int j = 0; j < D / 2; ++j) {
        const int b = ((j >> top) << (top + 1)) | (j & ((1 << top) - 1));
        sum += flip(v[2 * b], (uint32_t)__popc(z & b) & 1u);
    }
    // i^k (sum + (-1)^k conj): 2 Re, -2 Im, -2 Re, 2 Im
    return (k == 1 || k == 2 ? -2.0 : 2.0) / D * sum;
}

template <int N>
__device__ __forceinline__ const double2 *root_matrix(const UniRoots &r, int p) {
    return r.nodes + (size_t)r.root[p] * UCfg<N>::E;
}
__device__ __forceinline__ int root_parity(const UniRoots &r, int p) {
    return r.node_parity[r.root[p]];
}

// One CTA per generator: W = the product of the parts' unitaries (later
// ones to the left), then the coefficients of
// W Z_k W^dagger.  FP64-bound: a product is 512 warp instructions on the SM's
// four sub-partitions at n = 4 (4.7 us).
template <int N>
__global__ void __launch_bounds__(UCfg<N>::T) k_uni_images(UniRoots roots, double *out) {
    constexpr int D = UCfg<N>::D, E = UCfg<N>::E;
    __shared__ double2 U[E], V[E];
    __shared__ double2 h[E];
    const int t = (int)threadIdx.x, k = (int)blockIdx.x;
    const int row = t & (D - 1), col = t / D;
    int parity = root_parity(roots, 0);
    if (t < E) U[t] = root_matrix<N>(roots, 0)[t];
    __syncthreads();
    for (int p = 1; p < roots.n; ++p) {
        if (t < E) V[t] = root_matrix<N>(roots, p)[t];
        __syncthreads();
        const int q = root_parity(roots, p);
        double2 u;
        if (t < E) u = product_entry<N>(V, U, row, col, (parity & q) ? 0.5 : 1.0);
        parity ^= q;
        __syncthreads();
        if (t < E) U[t] = u;
        __syncthreads();
    }
    const double scale = parity ? 0.5 : 1.0;   // both factors of U Z U^dagger
    // B(r, r ^ x) for one r of each conjugate pair, by packed threads
    constexpr int kPairs = (D - 1) * (D / 2);
    if (t < kPairs + D) {
        int x = 0, r = t - kPairs;
        if (t < kPairs) {
            x = 1 + t / (D / 2);
            const int top = 31 - __clz(x), j = t % (D / 2);
            r = ((j >> top) << (top + 1)) | (j & ((1 << top) - 1));
        }
        const int s = r ^ x;
        double2 acc = make_double2(0.0, 0.0);
#pragma unroll
        for (int c = 0; c < D; ++c) {
            const uint32_t neg = (uint32_t)(c >> k) & 1u;   // (Z_k)(c, c)
            double2 v = U[c * D + r];
            v.x = flip(v.x, neg);
            v.y = flip(v.y, neg);
            acc = cfma_conj(v, U[c * D + s], acc);
        }
        h[x * D + r] = make_double2(scale * acc.x, x ? scale * acc.y : 0.0);
    }
    __syncthreads();
    if (t < E) out[(size_t)k * E + t] = pauli_coefficient<N>(h, t >> N, t & (D - 1));
}

// One CTA: out = later times earlier (n = 4 plans of three parts).
template <int N>
__global__ void __launch_bounds__(UCfg<N>::T) k_uni_merge(UniRoots roots, double2 *out,
                                                          int32_t *out_parity) {
    constexpr int D = UCfg<N>::D, E = UCfg<N>::E;
    __shared__ double2 U[E], V[E];
    const int t = (int)threadIdx.x;
    if (t < E) {
        U[t] = root_matrix<N>(roots, 0)[t];
        V[t] = root_matrix<N>(roots, 1)[t];
    }
    __syncthreads();
    const int p = root_parity(roots, 0), q = root_parity(roots, 1);
    if (t < E) out[t] = product_entry<N>(V, U, t & (D - 1), t / D, (p & q) ? 0.5 : 1.0);
    if (t == 0) *out_parity = p ^ q;
}

// y = M v or (adjoint) M^dagger v, D entries, by one warp: lane = part * D +
// row for D <= 16 rows, each of the 32 / D parts summing D / (32 / D) terms,
// then a fixed shuffle tree over the parts.  v is read from lanes' registers
// through shared memory `s`; every lane returns row lane & (D - 1).
template <int N>
__device__ __forceinline__ double2 warp_matvec(const double2 *M, bool adjoint, double2 v,
                                               double2 *s) {
    constexpr int D = UCfg<N>::D;
    constexpr int P = 32 / D;              // lanes per row
    constexpr int per = D / P > 0 ? D / P : 1;
    const int lane = (int)(threadIdx.x & 31u), row = lane & (D - 1), part = lane / D;
    __syncwarp();
    if (lane < D) s[lane] = v;
    __syncwarp();
    double2 acc = make_double2(0.0, 0.0);
    double2 m[per];
#pragma unroll
    for (int j = 0; j < per; ++j) {
        const int k = part * per + j;
        if (k < D) {
            const double2 *e = adjoint ? M + row * D + k : M + k * D + row;
            m[j] = make_double2(__ldcg(&e->x), __ldcg(&e->y));
            if (adjoint) m[j].y = -m[j].y;
        }
    }
#pragma unroll
    for (int j = 0; j < per; ++j) {
        const int k = part * per + j;
        if (k < D) acc = cfma(m[j], s[k], acc);
    }
#pragma unroll
    for (int o = 16; o >= D; o >>= 1) {
        acc.x += __shfl_xor_sync(0xffffffffu, acc.x, o);
        acc.y += __shfl_xor_sync(0xffffffffu, acc.y, o);
    }
    return acc;
}

// One warp: psi = the circuit applied to |0>, <O> = <psi|O|psi> and (r_out) the
// Pauli coefficients of 2^n |psi><psi|.  For the gradient also psi at the start
// of every part (slots 0 .. n) and the cotangent phi_p = U_p^dagger ...
// U_{K-1}^dagger O psi at the same places, both normalised.
template <int N>
__global__ void __launch_bounds__(32) k_uni_states(UniRoots roots, const DevTerm *terms,
                                                   int n_terms, double *expect, double2 *psi,
                                                   double2 *phi, double *r_out) {
    constexpr int D = UCfg<N>::D, E = UCfg<N>::E;
    __shared__ double2 s[D], h[E];
    const int lane = (int)threadIdx.x, row = lane & (D - 1);
    double2 v = make_double2(row == 0 ? 1.0 : 0.0, 0.0);
    int parity = 0;
    for (int p = 0; p <= roots.n; ++p) {
        if (p) {
            v = warp_matvec<N>(root_matrix<N>(roots, p - 1), false, v, s);
            const int q = root_parity(roots, p - 1);
            if (parity & q) v = scaled(v, 0.5);   // two factors sqrt(2)
            parity ^= q;
        }
        if (psi && lane < D) psi[p * D + row] = parity ? scaled(v, kInvSqrt2) : v;
    }
    if (expect) {
        // w = O psi: lane (part, row) takes the terms part, part + 32 / D, ...
        double2 w = make_double2(0.0, 0.0);
        __syncwarp();
        if (lane < D) s[lane] = v;
        __syncwarp();
        for (int k = lane / D; k < n_terms; k += 32 / D) {
            const int x = (int)(terms[k].idx >> N), z = (int)(terms[k].idx & (D - 1));
            const int from = row ^ x, ph = (__popc(x & z) + 2 * __popc(z & from)) & 3;
            double2 u = s[from];   // times i^ph
            if (ph & 1) u = make_double2(-u.y, u.x);
            if (ph & 2) u = make_double2(-u.x, -u.y);
            w = make_double2(fma(terms[k].coeff, u.x, w.x), fma(terms[k].coeff, u.y, w.y));
        }
#pragma unroll
        for (int o = 16; o >= D; o >>= 1) {
            w.x += __shfl_xor_sync(0xffffffffu, w.x, o);
            w.y += __shfl_xor_sync(0xffffffffu, w.y, o);
        }
        double e = fma(v.x, w.x, v.y * w.y);
#pragma unroll
        for (int o = D / 2; o > 0; o >>= 1) e += __shfl_xor_sync(0xffffffffu, e, o);
        if (lane == 0) *expect = parity ? 0.5 * e : e;
        if (phi) {
            if (parity) w = scaled(w, kInvSqrt2);
            if (lane < D) phi[roots.n * D + row] = w;
            for (int p = roots.n - 1; p >= 0; --p) {
                w = warp_matvec<N>(root_matrix<N>(roots, p), true, w, s);
                if (root_parity(roots, p)) w = scaled(w, kInvSqrt2);
                if (lane < D) phi[p * D + row] = w;
            }
        }
    }
    if (r_out) {
        __syncwarp();
        if (lane < D) s[lane] = v;
        __syncwarp();
        const double f = parity ? 0.5 * D : (double)D;
        for (int t = lane; t < E; t += 32) {
            const int x = t / D, b = t & (D - 1);
            const double2 z = cfma_conj(s[b], s[b ^ x], make_double2(0.0, 0.0));
            h[t] = make_double2(f * z.x, x ? f * z.y : 0.0);
        }
        __syncwarp();
        for (int t = lane; t < E; t += 32)
            r_out[t] = pauli_coefficient<N>(h, t >> N, t & (D - 1));
    }
}

// ---------------------------------------------------------------- gradient
//
// d<O>/d theta_j = Im <phi_j| s |psi_j> after rotation j (s its Pauli axis on
// its wire): both states of <psi|O|psi> carried through the plan.  For one
// wire the three numbers c_s = Im <phi| s |psi>, s = X, Y, Z, turn with the
// wire's gates as a 3-vector (U^dagger s U is the turned axis) and do not
// change under gates on other wires, so the 3-vector at the end of a wire
// run gives every rotation of the run.

// psi through segments [0, index) of a part (fwd) or phi back through
// segments [index, n_seg), by one warp: a greedy cover of the range by tree
// nodes, at most two per level.
template <int N>
__device__ double2 walk_tree(const UniArgs &a, const UniPart &P, int index, bool fwd, double2 v,
                             double2 *s) {
    constexpr int E = UCfg<N>::E;
    int at = fwd ? 0 : P.n_seg;
    while (at != index) {
        // the largest node that starts (fwd) or ends at `at` inside the range
        int level = 0, first = P.node, count = P.n_seg, best = 0, to = at;
        while (true) {
            // node i of a level covers segments [i 2^level, (i + 1) 2^level), cut at n_seg
            const int i = (fwd ? at : at - 1) >> level;
            const int b = i << level, e = min((i + 1) << level, P.n_seg);
            if (fwd ? (b != at || e > index) : (e != at || b < index)) break;
            best = first + i;
            to = fwd ? e : b;
            if (count == 1) break;
            first += count;
            count = (count + 1) / 2;
            ++level;
        }
        v = warp_matvec<N>(a.nodes + (size_t)best * E, !fwd, v, s);
        if (a.node_parity[best]) v = scaled(v, kInvSqrt2);
        at = to;
    }
    return v;
}

// A CTA of two warps per segment: psi and phi at its start, one warp each;
// then warp 0 carries both through it (lanes 0 .. D - 1 psi, the next D phi)
// and after each wire run stores every row's share of c at dots[(3 run + s) D
// + row].  14 FP64 instructions a wire pass, the FP64 pipe of one
// sub-partition the bound.
template <int N>
__global__ void __launch_bounds__(64) k_uni_grad(UniArgs a, const double2 *psi,
                                                 const double2 *phi, double *dots) {
    constexpr int D = UCfg<N>::D;
    constexpr int kStage = kUniStage / 2;
    __shared__ UniOp sop[kStage];
    __shared__ __align__(16) double smap[kStage * 8];
    __shared__ double2 s[2][D];
    const UniSeg sg = a.segs[blockIdx.x];
    const int t = (int)threadIdx.x, w = t >> 5, lane = t & 31, row = lane & (D - 1);
    {
        const UniPart P = a.parts[sg.part];
        double2 v = w ? phi[(sg.part + 1) * D + row] : psi[sg.part * D + row];
        v = walk_tree<N>(a, P, sg.index, w == 0, v, s[w]);
        __syncwarp();
        if (lane < D) s[w][lane] = v;
    }
    __syncthreads();
    const bool cot = (lane / D) & 1;   // this lane holds an entry of phi
    double re = s[cot][row].x, im = s[cot][row].y;
    int map_at = sg.map_first;
    for (int o0 = 0; o0 < sg.n_ops; o0 += kStage) {
        const int no = min(kStage, sg.n_ops - o0);
        if (o0) __syncthreads();
        for (int k = t; k < no; k += 64) sop[k] = a.ops[sg.op_first + o0 + k];
        const int nm = min(no, sg.map_first + sg.n_maps - map_at);
        const double2 *src = reinterpret_cast<const double2 *>(a.maps + map_at);
        for (int k = t; k < 4 * nm; k += 64) reinterpret_cast<double2 *>(smap)[k] = src[k];
        __syncthreads();
        int wires = 0;
        for (int k = 0; k < no; ++k) {
            const UniOp op = sop[k];
            if (op.kind != UK_WIRE) {
                if (w == 0) apply_two_qubit(op, lane, row, re, im);
                continue;
            }
            if (w == 0) {
                const int d = 1 << op.q0;
                apply_wire(smap + 8 * wires, d, row, re, im);
                // on a psi lane: z = conj(phi_row) psi_row, y = conj(phi_row) psi_{row ^ d}
                const double fr = __shfl_xor_sync(0xffffffffu, re, D);
                const double fi = __shfl_xor_sync(0xffffffffu, im, D);
                const double pr = __shfl_xor_sync(0xffffffffu, re, d);
                const double pi = __shfl_xor_sync(0xffffffffu, im, d);
                const double cz = fma(fr, im, -fi * re), cx = fma(fr, pi, -fi * pr);
                const double cy = fma(fr, pr, fi * pi);
                const uint32_t one = (row & d) ? 1u : 0u;
                if (lane < D) {
                    double *out = dots + (size_t)(map_at + wires) * 3 * D + row;
                    out[0] = cx;
                    out[D] = flip(cy, one ^ 1u);   // Im(-i y) on bit 0, Im(i y) on bit 1
                    out[2 * D] = flip(cz, one);
                }
            }
            ++wires;
        }
        map_at += wires;
    }
}

// c before a gate from c after it.
__device__ __forceinline__ void turn_back(double (&c)[3], int op, double co, double si) {
    const double x = c[0], y = c[1], z = c[2];
    switch (op) {
    case 0: c[0] = z; c[1] = -y; c[2] = x; break;
    case 1: c[0] = y; c[1] = -x; break;
    case 2: c[0] = -y; c[1] = x; break;
    case 3: c[1] = -y; c[2] = -z; break;
    case 4: c[0] = -x; c[2] = -z; break;
    case 5: c[0] = -x; c[1] = -y; break;
    case 8: c[1] = fma(si, z, co * y); c[2] = fma(-si, y, co * z); break;
    case 9: c[2] = fma(si, x, co * z); c[0] = fma(-si, z, co * x); break;
    case 10: c[0] = fma(si, y, co * x); c[1] = fma(-si, x, co * y); break;
    default: break;
    }
}

// A run's gates [k0, k1), last first: each rotation's derivative is c's entry
// of its axis just after it.
__device__ __forceinline__ void walk_run(double (&c)[3], const RawGate *gates, int k0, int k1,
                                         const double *thetas, double *out) {
    for (int k = k1 - 1; k >= k0; --k) {
        const RawGate g = gates[k];
        double si = 0.0, co = 1.0;
        if (g.op >= 8) {
            if (out) out[k] = c[g.op - 8];
            sincos(thetas[g.param], &si, &co);
        }
        turn_back(c, g.op, co, si);
    }
}

// c of a run at its end: its `rows` shares in order, less the run's factor.
__device__ __forceinline__ void run_dots(const double *dots, int run, int rows, int parity,
                                         double (&c)[3]) {
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        const double *p = dots + ((size_t)run * 3 + j) * rows;
        double v = 0.0;
#pragma unroll 4
        for (int r = 0; r < rows; ++r) v += p[r];
        c[j] = parity ? 0.5 * v : v;
    }
}

// A thread per run.
__global__ void __launch_bounds__(64) k_walk_seq(const UniRun *runs, int n_runs,
                                                 const RawGate *gates, const double *thetas,
                                                 const double *dots, int rows,
                                                 double *grad_gate) {
    const int i = (int)(blockIdx.x * blockDim.x + threadIdx.x);
    if (i >= n_runs) return;
    const UniRun r = runs[i];
    double c[3];
    run_dots(dots, i, rows, r.parity >> 1, c);
    walk_run(c, gates, r.first, r.first + r.count, thetas, grad_gate);
}

// A warp per run: every lane turns the three unit vectors back through its
// chunk of the run, a suffix scan of these 3 x 3 maps gives c at the chunk's
// end, and the chunk is walked again.
__global__ void __launch_bounds__(128) k_walk_warp(const UniRun *runs, int n_runs,
                                                   const RawGate *gates, const double *thetas,
                                                   const double *dots, int rows,
                                                   double *grad_gate) {
    const int w = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5);
    const int lane = (int)(threadIdx.x & 31u);
    if (w >= n_runs) return;   // whole warps
    const UniRun r = runs[w];
    const int per = (r.count + 31) / 32;
    const int k0 = r.first + min(lane * per, r.count), k1 = r.first + min((lane + 1) * per, r.count);
    // m[j]: the unit vector j at the end of chunks lane .. lane + 2^s - 1, at their start
    double m[3][3] = {{1.0, 0.0, 0.0}, {0.0, 1.0, 0.0}, {0.0, 0.0, 1.0}};
    for (int k = k1 - 1; k >= k0; --k) {
        const RawGate g = gates[k];
        double si = 0.0, co = 1.0;
        if (g.op >= 8) sincos(thetas[g.param], &si, &co);
#pragma unroll
        for (int j = 0; j < 3; ++j) turn_back(m[j], g.op, co, si);
    }
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        double o[3][3], p[3][3];
#pragma unroll
        for (int j = 0; j < 3; ++j)
#pragma unroll
            for (int i = 0; i < 3; ++i) o[j][i] = __shfl_down_sync(0xffffffffu, m[j][i], d);
        if (lane + d < 32) {
            // the later chunks first: e_j -> o[j] -> sum_i o[j][i] m[i]
#pragma unroll
            for (int j = 0; j < 3; ++j)
#pragma unroll
                for (int i = 0; i < 3; ++i)
                    p[j][i] = fma(o[j][2], m[2][i], fma(o[j][1], m[1][i], o[j][0] * m[0][i]));
#pragma unroll
            for (int j = 0; j < 3; ++j)
#pragma unroll
                for (int i = 0; i < 3; ++i) m[j][i] = p[j][i];
        }
    }
    double e[3], c[3];
    run_dots(dots, w, rows, r.parity >> 1, e);
    // the chunks after this lane's
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        const double a0 = __shfl_down_sync(0xffffffffu, m[0][i], 1);
        const double a1 = __shfl_down_sync(0xffffffffu, m[1][i], 1);
        const double a2 = __shfl_down_sync(0xffffffffu, m[2][i], 1);
        c[i] = lane == 31 ? e[i] : fma(e[2], a2, fma(e[1], a1, e[0] * a0));
    }
    walk_run(c, gates, k0, k1, thetas, grad_gate);
}

template <int N>
cudaError_t segments_n(const UniArgs &a, cudaStream_t st) {
    k_uni_segments<N><<<a.n_segs, UCfg<N>::T, 0, st>>>(a);
    return cudaGetLastError();
}

template <int N>
cudaError_t images_n(const UniRoots &r, double *out, cudaStream_t st) {
    k_uni_images<N><<<N, UCfg<N>::T, 0, st>>>(r, out);
    return cudaGetLastError();
}

template <int N>
cudaError_t merge_n(const UniRoots &r, double2 *out, int32_t *parity, cudaStream_t st) {
    k_uni_merge<N><<<1, UCfg<N>::T, 0, st>>>(r, out, parity);
    return cudaGetLastError();
}

template <int N>
cudaError_t states_n(const UniRoots &r, const DevTerm *terms, int n_terms, double *expect,
                     double2 *psi, double2 *phi, double *r_out, cudaStream_t st) {
    k_uni_states<N><<<1, 32, 0, st>>>(r, terms, n_terms, expect, psi, phi, r_out);
    return cudaGetLastError();
}

template <int N>
cudaError_t grad_n(const UniArgs &a, const double2 *psi, const double2 *phi, double *dots,
                   cudaStream_t st) {
    k_uni_grad<N><<<a.n_segs, 64, 0, st>>>(a, psi, phi, dots);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_uni_maps(const UniRun *runs, int n_runs, int max_count, const RawGate *gates,
                            const double *thetas, UniMap *maps, cudaStream_t st) {
    if (n_runs == 0) return cudaSuccess;
    if (!warp_per_run(n_runs, max_count))
        k_uni_maps_seq<<<(n_runs + 63) / 64, 64, 0, st>>>(runs, n_runs, gates, thetas, maps);
    else
        k_uni_maps_warp<<<(n_runs + 3) / 4, 128, 0, st>>>(runs, n_runs, gates, thetas, maps);
    return cudaGetLastError();
}

cudaError_t launch_uni_segments(int n, const UniArgs &a, cudaStream_t st) {
    switch (n) {
    case 1: return segments_n<1>(a, st);
    case 2: return segments_n<2>(a, st);
    case 3: return segments_n<3>(a, st);
    case 4: return segments_n<4>(a, st);
    default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_uni_images(int n, const UniRoots &r, double *out, cudaStream_t st) {
    switch (n) {
    case 1: return images_n<1>(r, out, st);
    case 2: return images_n<2>(r, out, st);
    case 3: return images_n<3>(r, out, st);
    case 4: return images_n<4>(r, out, st);
    default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_uni_merge(int n, const UniRoots &r, double2 *out, int32_t *parity,
                             cudaStream_t st) {
    switch (n) {
    case 1: return merge_n<1>(r, out, parity, st);
    case 2: return merge_n<2>(r, out, parity, st);
    case 3: return merge_n<3>(r, out, parity, st);
    case 4: return merge_n<4>(r, out, parity, st);
    default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_uni_states(int n, const UniRoots &r, const DevTerm *terms, int n_terms,
                              double *expect, double2 *psi, double2 *phi, double *r_out,
                              cudaStream_t st) {
    switch (n) {
    case 1: return states_n<1>(r, terms, n_terms, expect, psi, phi, r_out, st);
    case 2: return states_n<2>(r, terms, n_terms, expect, psi, phi, r_out, st);
    case 3: return states_n<3>(r, terms, n_terms, expect, psi, phi, r_out, st);
    case 4: return states_n<4>(r, terms, n_terms, expect, psi, phi, r_out, st);
    default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_uni_grad(int n, const UniArgs &a, const double2 *psi, const double2 *phi,
                            double *dots, cudaStream_t st) {
    switch (n) {
    case 1: return grad_n<1>(a, psi, phi, dots, st);
    case 2: return grad_n<2>(a, psi, phi, dots, st);
    case 3: return grad_n<3>(a, psi, phi, dots, st);
    case 4: return grad_n<4>(a, psi, phi, dots, st);
    default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_run_grads(const UniRun *runs, int n_runs, int max_count, const RawGate *gates,
                             const double *thetas, const double *dots, int rows,
                             double *grad_gate, cudaStream_t st) {
    if (n_runs == 0) return cudaSuccess;
    if (!warp_per_run(n_runs, max_count))
        k_walk_seq<<<(n_runs + 63) / 64, 64, 0, st>>>(runs, n_runs, gates, thetas, dots, rows,
                                                      grad_gate);
    else
        k_walk_warp<<<(n_runs + 3) / 4, 128, 0, st>>>(runs, n_runs, gates, thetas, dots, rows,
                                                      grad_gate);
    return cudaGetLastError();
}

}  // namespace stab
