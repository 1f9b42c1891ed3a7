// k_stream.cu -- angle encoding and the streamed (HBM-resident) passes.
//
// Streamed passes keep the vectors in global memory and apply one fused pass
// per launch to every vector of the batch: a P_WIRE pass reads each group of
// the pass's wire once, runs all of the wire's ops on it in registers and
// writes it back in place; a P_CLIFF pass gathers every entry through the
// pass's signed permutation into a second buffer.
#include <cuda_runtime.h>

#include "device_ops.cuh"
#include "launch.h"
#include "pull.cuh"
#include "tma.cuh"

namespace stab {

namespace {

constexpr int kThreads = 256;

int grid_for(uint64_t work, int threads) {
    uint64_t b = (work + threads - 1) / threads;
    const uint64_t cap = 152ull * 16ull;  // grid-stride beyond 16 CTAs per SM
    if (b > cap) b = cap;
    if (b < 1) b = 1;
    return (int)b;
}

// 3x3 maps on the (X, Y, Z) coefficients of one wire (new = M old), Table I
// rows; Clifford gates as signed permutation matrices.
__device__ void gate_matrix3(const RawGate &g, const double *thetas, double M[9]) {
    for (int k = 0; k < 9; ++k) M[k] = 0.0;
    double c = 1.0, s = 0.0;
    if (g.op >= 8) sincos(thetas[g.param], &s, &c);
    switch (g.op) {
    case 0:  // H: X <- Z, Y <- -Y, Z <- X
        M[2] = 1.0; M[4] = -1.0; M[6] = 1.0; break;
    case 1:  // S: X <- -Y, Y <- X
        M[1] = -1.0; M[3] = 1.0; M[8] = 1.0; break;
    case 2:  // Sdg: X <- Y, Y <- -X
        M[1] = 1.0; M[3] = -1.0; M[8] = 1.0; break;
    case 3:  // X: Y, Z negated
        M[0] = 1.0; M[4] = -1.0; M[8] = -1.0; break;
    case 4:  // Y: X, Z negated
        M[0] = -1.0; M[4] = 1.0; M[8] = -1.0; break;
    case 5:  // Z: X, Y negated
        M[0] = -1.0; M[4] = -1.0; M[8] = 1.0; break;
    case 8:  // RX: Y' = cY - sZ, Z' = sY + cZ
        M[0] = 1.0; M[4] = c; M[5] = -s; M[7] = s; M[8] = c; break;
    case 9:  // RY: X' = cX + sZ, Z' = -sX + cZ
        M[0] = c; M[2] = s; M[4] = 1.0; M[6] = -s; M[8] = c; break;
    case 10: // RZ: X' = cX - sY, Y' = sX + cY
        M[0] = c; M[1] = -s; M[3] = s; M[4] = c; M[8] = 1.0; break;
    default:
        M[0] = M[4] = M[8] = 1.0; break;
    }
}

// Shear coefficients of an angle: theta is reduced to phi in [-pi/2, pi/2] up
// to a factor R(pi) = -1 on the pair (neg), so that t = -tan(phi/2) stays in
// [-1, 1].
__device__ void shear_coeffs(double theta, double &t, double &s, uint16_t &neg) {
    const double two_pi = 6.283185307179586476925286766559;
    const double pi = 3.1415926535897932384626433832795;
    double phi = remainder(theta, two_pi);
    neg = 0;
    if (phi > 0.5 * pi) { phi -= pi; neg = 1; }
    else if (phi < -0.5 * pi) { phi += pi; neg = 1; }
    t = -tan(0.5 * phi);
    s = sin(phi);
}

// 3x3 product C = A B (row-major).
__device__ __forceinline__ void mul3(const double A[9], const double B[9], double C[9]) {
#pragma unroll
    for (int r = 0; r < 3; ++r)
#pragma unroll
        for (int c = 0; c < 3; ++c)
            C[3 * r + c] = fma(A[3 * r + 2], B[6 + c], fma(A[3 * r + 1], B[3 + c], A[3 * r] * B[c]));
}

// Composed map of every run, one warp per map: lane l composes a contiguous
// chunk of the run's gates in order (the lanes evaluate their gates' sin/cos
// at once), then the 32 partial products are multiplied in order by a
// shuffle tree (later chunk times earlier chunk), log2(32) steps instead of a
// sequential walk over the whole run.
__global__ void k_compose_maps(DevMap3 *maps, int n_maps, const int32_t *map_gate_idx,
                               const RawGate *gates, const double *thetas) {
    const int w = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5);
    const int lane = (int)(threadIdx.x & 31u);
    if (w >= n_maps) return;   // whole warps
    const DevMap3 mp = maps[w];
    const int per = (mp.count + 31) / 32;
    const int k0 = min(lane * per, mp.count), k1 = min(k0 + per, mp.count);
    double M[9] = {1.0, 0.0, 0.0, 0.0, 1.0, 0.0, 0.0, 0.0, 1.0};
    for (int k = k0; k < k1; ++k) {
        double G[9], R[9];
        gate_matrix3(gates[map_gate_idx[mp.first + k]], thetas, G);
        mul3(G, M, R);
#pragma unroll
        for (int j = 0; j < 9; ++j) M[j] = R[j];
    }
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        double O[9], R[9];
#pragma unroll
        for (int j = 0; j < 9; ++j) O[j] = __shfl_down_sync(0xffffffffu, M[j], d);
        if ((lane & (2 * d - 1)) == 0) {
            mul3(O, M, R);
#pragma unroll
            for (int j = 0; j < 9; ++j) M[j] = R[j];
        }
    }
    if (lane == 0)
#pragma unroll
        for (int j = 0; j < 9; ++j) maps[w].m[j] = M[j];
}

// The same with a CTA of 1,024 threads per map, for runs of thousands of gates
// (n = 1, where a circuit is one run: 16,912 gates 1.24 ms with a warp, 0.31 so):
// warp w composes chunks 32 w .. 32 w + 31, the first warp the warps' products.
__global__ void __launch_bounds__(1024) k_compose_maps_cta(DevMap3 *maps,
                                                           const int32_t *map_gate_idx,
                                                           const RawGate *gates,
                                                           const double *thetas) {
    __shared__ double part[32][9];
    const int warp = (int)(threadIdx.x >> 5), lane = (int)(threadIdx.x & 31u);
    const DevMap3 &mp = maps[blockIdx.x];
    const int first = mp.first, count = mp.count, per = (count + 1023) / 1024;
    const int k0 = min((int)threadIdx.x * per, count), k1 = min(k0 + per, count);
    double M[9] = {1.0, 0.0, 0.0, 0.0, 1.0, 0.0, 0.0, 0.0, 1.0};
    for (int k = k0; k < k1; ++k) {
        double G[9], R[9];
        gate_matrix3(gates[map_gate_idx[first + k]], thetas, G);
        mul3(G, M, R);
#pragma unroll
        for (int j = 0; j < 9; ++j) M[j] = R[j];
    }
    for (int round = 0; round < 2; ++round) {
        if (round == 1) {
            __syncthreads();
            if (warp != 0) return;
#pragma unroll
            for (int j = 0; j < 9; ++j) M[j] = part[lane][j];
        }
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            double O[9], R[9];
#pragma unroll
            for (int j = 0; j < 9; ++j) O[j] = __shfl_down_sync(0xffffffffu, M[j], d);
            if ((lane & (2 * d - 1)) == 0) {
                mul3(O, M, R);
#pragma unroll
                for (int j = 0; j < 9; ++j) M[j] = R[j];
            }
        }
        if (lane == 0)
#pragma unroll
            for (int j = 0; j < 9; ++j) {
                if (round == 0) part[warp][j] = M[j];
                else maps[blockIdx.x].m[j] = M[j];
            }
    }
}

// Composed map of every run, one thread per map walking its gates in order:
// the form for plans of short runs (a warp per map would idle most lanes).
__global__ void k_compose_maps_seq(DevMap3 *maps, int n_maps, const int32_t *map_gate_idx,
                                   const RawGate *gates, const double *thetas) {
    const int i = (int)(blockIdx.x * blockDim.x + threadIdx.x);
    if (i >= n_maps) return;
    const DevMap3 mp = maps[i];
    double M[9] = {1.0, 0.0, 0.0, 0.0, 1.0, 0.0, 0.0, 0.0, 1.0};
    for (int k = 0; k < mp.count; ++k) {
        double G[9], R[9];
        gate_matrix3(gates[map_gate_idx[mp.first + k]], thetas, G);
        mul3(G, M, R);
#pragma unroll
        for (int j = 0; j < 9; ++j) M[j] = R[j];
    }
#pragma unroll
    for (int j = 0; j < 9; ++j) maps[i].m[j] = M[j];
}

// Angles -> stream records: shear coefficients of rotations, and the composed
// maps (from k_compose_maps) copied into the R_MAP3 data records, transposed
// (the inverse) in backward streams.
__global__ void k_encode_stream(Rec *recs, const int32_t *enc, int n_enc, const DevMap3 *maps,
                                const double *thetas) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n_enc) return;
    Rec &r = recs[enc[k]];
    if (r.kind == R_ROT) {
        double t, s;
        uint16_t neg;
        shear_coeffs(thetas[r.param], t, s, neg);
        r.t = r.inv ? -t : t;
        r.s = r.inv ? -s : s;
        r.code = neg;
    } else if (r.kind == R_MAP3) {
        const double *M = maps[r.param].m;
        double *dst = reinterpret_cast<double *>(&r + 1);
        for (int i = 0; i < 3; ++i)
            for (int j = 0; j < 3; ++j) dst[3 * i + j] = r.inv ? M[3 * j + i] : M[3 * i + j];
    }
}

__global__ void k_encode(DevOp *ops, int n_ops, const double *thetas) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n_ops && ops[i].kind == K_ROT) {
        double t, s;
        uint16_t neg;
        shear_coeffs(thetas[ops[i].param], t, s, neg);
        ops[i].t = t;
        ops[i].s = s;
        ops[i].perm = neg;
    }
}

__global__ void k_fill(double *vec, int n, int n_vec, int init) {
    const uint64_t E = 1ull << (2 * n);
    const uint64_t total = E * (uint64_t)n_vec;
    for (uint64_t t = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; t < total;
         t += (uint64_t)gridDim.x * blockDim.x) {
        const uint64_t v = t >> (2 * n), i = t & (E - 1);
        double val = 0.0;
        if (init == INIT_RHO0) val = i < (1ull << n) ? 1.0 : 0.0;
        else if (init == INIT_GENERATOR) val = (i == (1ull << v)) ? 1.0 : 0.0;
        vec[t] = val;
    }
}

__global__ void k_scatter_terms(double *vec, const DevTerm *terms, int n_terms) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k < n_terms) vec[terms[k].idx] = terms[k].coeff;
}

__global__ void __launch_bounds__(kThreads) k_stream_wire(double *vec, int n, int n_vec, DevPass p,
                                                          const DevOp *ops, const DevMap3 *maps,
                                                          int inverse) {
    const int q = p.q;
    const uint64_t E = 1ull << (2 * n);
    const uint64_t G = E >> 2;
    const uint64_t total = G * (uint64_t)n_vec;
    const uint64_t bx = 1ull << (n + q), bz = 1ull << q;
    const int n_ops = p.n_ops;
    for (uint64_t t = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; t < total;
         t += (uint64_t)gridDim.x * blockDim.x) {
        const uint64_t v = t >> (2 * n - 2), g = t & (G - 1);
        double *base = vec + v * E + group_base(g, n, q);
        double x = base[bx], y = base[bx | bz], z = base[bz];
        for (int j = 0; j < n_ops; ++j) {
            const DevOp op = ops[p.first + (inverse ? n_ops - 1 - j : j)];
            apply_op1(x, y, z, op, maps, inverse);
        }
        base[bx] = x;
        base[bx | bz] = y;
        base[bz] = z;
    }
}

__global__ void __launch_bounds__(kThreads) k_stream_cliff(const double *__restrict__ src,
                                                           double *__restrict__ dst, int n,
                                                           int n_vec, DevPass p, const DevOp *ops,
                                                           int inverse) {
    const uint64_t E = 1ull << (2 * n);
    const uint64_t total = E * (uint64_t)n_vec;
    for (uint64_t t = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; t < total;
         t += (uint64_t)gridDim.x * blockDim.x) {
        const uint64_t v = t >> (2 * n), i = t & (E - 1);
        uint32_t neg = 0;
        const uint64_t j = pull_pass(i, n, ops + p.first, p.n_ops, inverse, neg);
        dst[t] = flip(src[v * E + j], neg);
    }
}

// A Clifford run as one signed gather over whole vectors: a CTA takes 1,024
// consecutive entries, four per thread, so an entry costs a few popcounts
// beside its two memory accesses whatever the length of the run.  Bound by
// the scattered reads (n = 12, a ring of 12 CNOTs; <O> of 400 gates there
// 7.69 -> 6.42 ms against walking the ring's gates for every entry).
__global__ void __launch_bounds__(kThreads) k_stream_pull(const double *__restrict__ src,
                                                          double *__restrict__ dst, int n,
                                                          int n_vec, const DevPull *pull) {
    const LanePull L = load_pull(pull, n);
    const uint64_t E = 1ull << (2 * n);
    const uint32_t t = threadIdx.x;
    uint32_t oj[4] = {0, 0, 0, 0}, oq[4] = {0, 0, 0, 0};
    const int nb = 2 * n < 10 ? 2 * n : 10;
    for (int b = 0; b < nb; ++b)
#pragma unroll
        for (int k = 0; k < 4; ++k) off_bit(L, b, t | (uint32_t)k << 8, oj[k], oq[k]);
    const uint64_t per = (E + 1023) >> 10, chunks = per * (uint64_t)n_vec;
    for (uint64_t c = blockIdx.x; c < chunks; c += gridDim.x) {
        const uint64_t v = c / per, base = (c - v * per) << 10;
        const BasePull B = base_pull(L, (uint32_t)base);
        const double *S = src + v * E;
        double *D = dst + v * E;
        double val[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const uint32_t off = t | (uint32_t)k << 8;
            uint32_t neg;
            const uint32_t j = pull_entry(L, B, n, off, oj[k], oq[k], neg);
            if (base + off < E) val[k] = flip(S[j], neg);
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const uint32_t off = t | (uint32_t)k << 8;
            if (base + off < E) D[base + off] = val[k];
        }
    }
}

// Consecutive wire passes on at most kTileWires wires: a tile of up to 2^10
// entries (the wires' (z, x) bits and the lowest other bits) per CTA in shared
// memory, a group of four entries per thread and pass, the preceding Clifford
// run folded into the loads.  Small vectors are latency-bound here (n = 8: one
// warp per sub-partition and 36 FP64 instructions a launch), so a launch
// fetches everything it needs at once and a pass is the run's composed map:
// three independent rows of three FMAs and no op decoding, where lifts would
// be a chain of nine behind three decoded ops.  (n = 8, four wires with a
// folded CNOT ring, two sequences on the GPU: 11 us a launch with the ring's
// gates walked per entry, 7.3 with lifts, 6.9 so; k_stream_chain runs whole
// sequences, this kernel the steps of plans outside them.)  From n = 10 on a launch per wire pass is faster (600 gates: 661 against 794
// us): the FP64 pipe is full there and a tile's barriers only leave gaps.
// MAPS = false: the runs' ops instead (lifts, three FMAs a rotation), for
// vectors of 2^18 entries and more whose runs hold few rotations.
template <bool MAPS>
__global__ void __launch_bounds__(kTileThreads) k_stream_tile(const double *src, double *dst,
                                                              int n, int n_vec, TileGroup tg,
                                                              const DevMap3 *maps,
                                                              const DevOp *ops) {
    __shared__ double tile[1 << kTileMaxBits];
    __shared__ __align__(16) double smap[kTileMaxPasses][10];
    __shared__ __align__(16) DevOp sops[MAPS ? 1 : kTileStagedOps];
    const uint32_t T = 1u << tg.tile_bits;
    const uint32_t t = threadIdx.x, nt = blockDim.x;   // nt >= T / 4
    bool staged = false;
    if constexpr (MAPS) {
        // the maps, transposed (the inverse) for backward sweeps
        for (uint32_t k = t; k < (uint32_t)tg.n_pass * 9u; k += nt) {
            const uint32_t j = k / 9u, e = k - 9u * j;
            const uint32_t to = tg.inverse ? (e % 3u) * 3u + e / 3u : e;
            smap[j][to] = maps[tg.map[j]].m[e];
        }
    } else {
        int total = 0;
        for (int j = 0; j < tg.n_pass; ++j) total += tg.n_ops[j];
        staged = total <= kTileStagedOps;
        if (staged)
            for (int k = (int)t; k < total; k += (int)nt) {
                int j = 0, at = k;
                while (at >= (int)tg.n_ops[j]) at -= tg.n_ops[j++];
                sops[k] = ops[tg.first[j] + at];
            }
    }
    const bool pulled = tg.pull != nullptr;
    LanePull L{};
    if (pulled) L = load_pull(tg.pull, n);
    // entry t + k nt: this thread's offset, and one of the CTA for each k
    const uint32_t off = (uint32_t)deposit_runs(t, tg.tile_runs);
    uint32_t step[4], oj = 0, oq = 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) step[k] = (uint32_t)deposit_runs(k * nt, tg.tile_runs);
    if (pulled) {
        const int bits = 31 - __clz((int)nt);
        int at = 0;
        for (int r = 0; r < tg.tile_runs.n; ++r)
            for (int b = 0; b < tg.tile_runs.len[r] && at < bits; ++b, ++at)
                off_bit(L, tg.tile_runs.dst[r] + b, off, oj, oq);
    }
    const uint64_t E = 1ull << (2 * n);
    const uint64_t tiles = (uint64_t)n_vec << tg.rest_bits;
    for (uint64_t tb = blockIdx.x; tb < tiles; tb += gridDim.x) {
        const uint64_t v = tb >> tg.rest_bits;
        const uint32_t base =
            (uint32_t)deposit_runs(tb & ((1ull << tg.rest_bits) - 1ull), tg.rest_runs);
        const double *S = src + v * E;
        double *V = dst + v * E;
        double val[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const bool in = t + k * nt < T;
            uint32_t neg = 0, j = base + step[k] + off;
            if (pulled) {
                const BasePull B = base_pull(L, base + step[k]);
                j = pull_entry(L, B, n, off, oj, oq, neg);
            }
            if (in) val[k] = flip(S[j], neg);
        }
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (t + k * nt < T) tile[t + k * nt] = val[k];
        __syncthreads();
        int at = 0;
        for (int j = 0; j < tg.n_pass; ++j) {
            const int lz = tg.lz[j], lx = tg.lx[j];
            const int lo = lz < lx ? lz : lx, hi = lz < lx ? lx : lz;
            const uint32_t bz = 1u << lz, bx = 1u << lx;
            const int n_ops = tg.n_ops[j];
            const DevOp *pops = staged ? sops + at : ops + tg.first[j];
            at += n_ops;
            if (t < T / 4) {
                uint32_t b = ((t >> lo) << (lo + 1)) | (t & ((1u << lo) - 1u));
                b = ((b >> hi) << (hi + 1)) | (b & ((1u << hi) - 1u));
                double x = tile[b | bx], y = tile[b | bx | bz], z = tile[b | bz];
                if constexpr (MAPS) {
                    apply_map3(x, y, z, smap[j], false);
                } else {
                    DevOp next = pops[tg.inverse ? n_ops - 1 : 0];
                    for (int k = 0; k < n_ops; ++k) {
                        const DevOp op = next;
                        if (k + 1 < n_ops) next = pops[tg.inverse ? n_ops - 2 - k : k + 1];
                        apply_op1(x, y, z, op, maps, tg.inverse);
                    }
                }
                tile[b | bx] = x;
                tile[b | bx | bz] = y;
                tile[b | bz] = z;
            }
            __syncthreads();
        }
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (t + k * nt < T) V[base + step[k] + off] = tile[t + k * nt];
        __syncthreads();
    }
}

// Tables of one shape per CTA (see launch.h).
__global__ void __launch_bounds__(128) k_chain_tables(const ChainShape *shapes, int n) {
    __shared__ ChainShape S;
    __shared__ DevPull P;
    {
        const uint32_t *from = reinterpret_cast<const uint32_t *>(shapes + blockIdx.x);
        for (uint32_t k = threadIdx.x; k < sizeof(ChainShape) / 4; k += blockDim.x)
            reinterpret_cast<uint32_t *>(&S)[k] = from[k];
    }
    __syncthreads();
    if (S.pull) {
        const uint32_t *from = reinterpret_cast<const uint32_t *>(S.pull);
        for (uint32_t k = threadIdx.x; k < sizeof(DevPull) / 4; k += blockDim.x)
            reinterpret_cast<uint32_t *>(&P)[k] = from[k];
    }
    __syncthreads();
    const int lo = min(S.lz, S.lx), hi = max(S.lz, S.lx);
    const uint32_t groups = 1u << (S.tile_bits - 2);
    for (uint32_t t = threadIdx.x; t < groups; t += blockDim.x) {
        uint32_t b = ((t >> lo) << (lo + 1)) | (t & ((1u << lo) - 1u));
        b = ((b >> hi) << (hi + 1)) | (b & ((1u << hi) - 1u));
        const uint32_t off = (uint32_t)deposit_runs(b, S.tile_runs);
        uint32_t j = 0, q = 0;
        if (S.pull)
            for (int k = 0; k < 2 * n; ++k)
                if ((off >> k) & 1u) {
                    j ^= P.col[k];
                    q ^= (uint32_t)__popc(P.qrow[k] & off);
                }
        S.threads[t] = make_uint2(off, j | (q & 1u) << 31);
    }
    const uint64_t entries = 4ull << S.rest_bits;
    for (uint64_t m = threadIdx.x; m < entries; m += blockDim.x) {
        const uint32_t k = (uint32_t)m & 3u;
        const uint32_t i = (uint32_t)deposit_runs(m >> 2, S.rest_runs) |
                           ((k & 1u) << S.wire) | ((k >> 1) << (n + S.wire));
        uint32_t j = 0, q = 0, cross = 0;
        if (S.pull)
            for (int a = 0; a < 2 * n; ++a) {
                const uint32_t par = (uint32_t)__popc(P.qrow[a] & i) & 1u;
                cross ^= par << a;
                if ((i >> a) & 1u) {
                    j ^= P.col[a];
                    cross ^= P.qrow[a];
                    q ^= par;
                }
            }
        S.tiles[m] = make_uint4(i, j | q << 31, cross, 0u);
    }
}

// A chain of tile steps in one launch: the chain's CTAs stay and meet at a
// counter in global memory after every step.  Nothing a step needs besides
// its vector depends on the steps before it, so all of it (where the thread
// reads and writes, the maps) is loaded during the step before, and a step is
// its gather, its passes and the barrier's round trip.  The first pass's group
// is gathered straight into registers and the last pass's stored from them;
// shared memory carries the tile between passes.  The launch is cooperative
// (all CTAs resident) and every wait is bounded: a CTA that gives up sets the
// status word and leaves, and so do the others.
// Per step at n = 8, four wires, two chains on the GPU: 6.9 us as launches
// replayed from a graph, 6.3 in a chain that fetches after the barrier, 5.4
// so; of it 1.9 are FP64 (two CTAs share most SMs), 0.5 the barrier's wait.
// n = 7: 5.8 -> 4.2 us.
constexpr uint32_t kChainPolls = 1u << 22;   // a second or two

// ALONE: chains of one CTA each (n = 5) keep their vector in shared memory and
// meet nobody (3,000 gates: <O> 515 -> 406 us, gradient 1048 -> 788).  Four CTAs of 256
// threads fit an SM, so both chains of n = 9 (256 tiles each) have a CTA a tile.
template <bool ALONE>
__global__ void __launch_bounds__(kTileThreads, 4) k_stream_chain(ChainArgs a) {
    __shared__ double tile[1 << kTileMaxBits];
    __shared__ __align__(16) double smap[2][kTileMaxPasses * 9];
    __shared__ double solo[2][ALONE ? 1 << kTileMaxBits : 1];
    __shared__ ChainStep S[3];
    __shared__ ChainDesc C;
    __shared__ int s_ok;
    const uint32_t t = threadIdx.x;              // one group: blockDim.x = 2^tile_bits / 4
    for (int k = (int)t; k < a.n_chains; k += (int)blockDim.x) {
        const int c0 = a.chains[k].cta0;
        if ((int)blockIdx.x >= c0 && (int)blockIdx.x < c0 + a.chains[k].ctas) C = a.chains[k];
    }
    __syncthreads();
    const uint32_t rank = blockIdx.x - (uint32_t)C.cta0, ctas = (uint32_t)C.ctas;
    const int n_steps = C.n_steps, n_vec = C.n_vec, n = C.n;
    const ChainStep *steps = C.steps;
    const DevMap3 *all_maps = C.maps;
    uint32_t *arrived = C.arrived;
    const uint64_t E = 1ull << (2 * n);
    const uint32_t zmask = (1u << n) - 1u;
    constexpr uint32_t kWords = sizeof(ChainStep) / 4;   // <= blockDim.x
    // registers loaded one step ahead
    uint2 in_t{}, in_t1{};
    uint32_t out_off = 0, out_off1 = 0, r0 = 0, r1 = 0, r01 = 0, r11 = 0;
    uint4 tk[4], tk1[4];
    double mval = 0.0;
    uint32_t word = 0;
    const uint32_t mj = t / 9u, me = t - 9u * mj;
    // issues step s's loads (its description is in S[s % 3])
    auto fetch = [&](int s) {
        const ChainStep &d = S[s % 3];
        in_t1 = d.in_threads[t];
        out_off1 = d.out_threads[t].x;
        if (d.pull) {
            r01 = d.pull->r0;
            r11 = d.pull->r1;
        }
        if ((rank >> d.rest_bits) < (uint32_t)n_vec) {
            const uint4 *p = d.tiles + 4ull * (rank & ((1u << d.rest_bits) - 1u));
#pragma unroll
            for (int k = 0; k < 4; ++k) tk1[k] = p[k];
        }
        // thread (j, e) holds entry e of pass j's map, transposed (the inverse)
        // for backward sweeps
        if (mj < (uint32_t)d.n_pass)
            mval = all_maps[d.map[mj]].m[d.inverse ? (me % 3u) * 3u + me / 3u : me];
    };
    auto land = [&](int s) {   // fetched values of step s become current
        in_t = in_t1;
        out_off = out_off1;
        r0 = r01;
        r1 = r11;
#pragma unroll
        for (int k = 0; k < 4; ++k) tk[k] = tk1[k];
        if (mj < (uint32_t)S[s % 3].n_pass) smap[s & 1][t] = mval;
    };
    for (int s = 0; s < 2 && s < n_steps; ++s)
        if (t < kWords)
            reinterpret_cast<uint32_t *>(&S[s])[t] =
                reinterpret_cast<const uint32_t *>(steps + s)[t];
    __syncthreads();
    if (n_steps > 0) {
        fetch(0);
        land(0);
    }
    if (ALONE && n_steps > 0)
        for (uint32_t i = t; i < (uint32_t)E; i += blockDim.x) solo[0][i] = S[0].src[i];
    __syncthreads();
    for (int s = 0; s < n_steps; ++s) {
        const ChainStep &st = S[s % 3];
        const int n_pass = st.n_pass;
        const bool pulled = st.pull != nullptr;
        const double *maps = smap[s & 1];
        const uint64_t tiles = (uint64_t)n_vec << st.rest_bits;
        bool first = true;
        for (uint64_t tb = rank; tb < tiles; tb += ctas) {
            const uint64_t v = tb >> st.rest_bits;
            const double *src = st.src + v * E;
            double *dst = st.dst + v * E;
            if (!first) {
                const uint4 *p = st.tiles + 4ull * (tb & ((1ull << st.rest_bits) - 1ull));
#pragma unroll
                for (int k = 0; k < 4; ++k) tk[k] = p[k];
            }
            double val[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const uint32_t i = tk[k].x + in_t.x;
                uint32_t j = i, neg = 0;
                if (pulled) {
                    const uint32_t jq = tk[k].y ^ in_t.y;
                    j = jq & 0x7fffffffu;
                    const uint32_t q = (jq >> 31) ^ ((uint32_t)__popc(in_t.x & tk[k].z) & 1u);
                    neg = ((uint32_t)(__popc((i >> n) & i & zmask) + __popc(i & r0) +
                                      2 * __popc(i & r1) + 2 * (int)q -
                                      __popc((j >> n) & j & zmask)) >> 1) & 1u;
                }
                // written by other SMs in this launch: through L2
                val[k] = flip(ALONE ? solo[s & 1][j] : __ldcg(src + j), neg);
            }
            if (first) {
                // the next step's loads, in flight during this one
                if (s + 1 < n_steps) fetch(s + 1);
                if (s + 2 < n_steps && t < kWords)
                    word = reinterpret_cast<const uint32_t *>(steps + s + 2)[t];
                first = false;
            }
            if (n_pass > 0) apply_map3(val[2], val[3], val[1], maps, false);
            for (int j = 1; j < n_pass; ++j) {
                // through shared memory from pass j - 1's groups to pass j's
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int lz = st.lz[j - 1 + h], lx = st.lx[j - 1 + h];
                    const int lo = lz < lx ? lz : lx, hi = lz < lx ? lx : lz;
                    const uint32_t bz = 1u << lz, bx = 1u << lx;
                    uint32_t b = ((t >> lo) << (lo + 1)) | (t & ((1u << lo) - 1u));
                    b = ((b >> hi) << (hi + 1)) | (b & ((1u << hi) - 1u));
                    if (h == 0) {
                        // (the last pass's reads of this buffer are behind a barrier)
                        tile[b] = val[0];
                        tile[b | bz] = val[1];
                        tile[b | bx] = val[2];
                        tile[b | bx | bz] = val[3];
                        __syncthreads();
                    } else {
                        val[0] = tile[b];
                        val[1] = tile[b | bz];
                        val[2] = tile[b | bx];
                        val[3] = tile[b | bx | bz];
                        __syncthreads();
                    }
                }
                apply_map3(val[2], val[3], val[1], maps + 9 * j, false);
            }
            const uint32_t base = n_pass > 0 ? tk[0].x + out_off : 0u;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const uint32_t i = n_pass > 0 ? base + st.out_k[k] : tk[k].x + in_t.x;
                dst[i] = val[k];
                if (ALONE) solo[(s + 1) & 1][i] = val[k];
            }
        }
        if (s + 1 == n_steps) return;
        if (first) {   // a CTA without a tile in this step
            fetch(s + 1);
            if (s + 2 < n_steps && t < kWords)
                word = reinterpret_cast<const uint32_t *>(steps + s + 2)[t];
        }
        __syncthreads();
        if (t == 0 && !ALONE) {
            __threadfence();
            atomicAdd(arrived, 1u);
        }
        land(s + 1);
        if (s + 2 < n_steps && t < kWords)
            reinterpret_cast<uint32_t *>(&S[(s + 2) % 3])[t] = word;
        if (ALONE) {
            __syncthreads();
            continue;
        }
        if (t == 0) {
            const uint32_t want = ctas * (uint32_t)(s + 1);
            bool ok = false;
            for (uint32_t it = 0; it < kChainPolls && !ok; ++it) {
                uint32_t seen;
                asm volatile("ld.acquire.gpu.global.u32 %0, [%1];"
                             : "=r"(seen) : "l"(arrived) : "memory");
                ok = arrivals_reached(seen, want);
            }
            if (!ok && a.status) atomicExch(a.status, STAB_KSTATUS_TIMEOUT);
            s_ok = ok ? 1 : 0;
        }
        __syncthreads();
        if (!s_ok) return;
    }
}

// Deterministic sum of the 2^n x-free coefficients of each vector (one CTA
// per vector, fixed order).
__global__ void __launch_bounds__(kThreads) k_xfree_sum(const double *vec, int n, double *out) {
    __shared__ double red[kThreads / 32];
    const uint64_t E = 1ull << (2 * n);
    const double *v = vec + blockIdx.x * E;
    double acc = 0.0;
    for (int i = threadIdx.x; i < (1 << n); i += blockDim.x) acc += v[i];
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        double total = 0.0;
        for (int w = 0; w < kThreads / 32; ++w) total += red[w];
        out[blockIdx.x] = total;
    }
}

// Inner product <a, b> of two coefficient vectors in a fixed order: block b
// sums a contiguous slice (strided by the block's threads, then a shuffle
// tree), the last kernel the kDotBlocks partials in order.
constexpr int kDotBlocks = 256;

__global__ void __launch_bounds__(kThreads) k_dot_partial(const double *a, const double *b,
                                                          int n, double *partial) {
    __shared__ double red[kThreads / 32];
    const uint64_t E = 1ull << (2 * n);
    const uint64_t per = (E + gridDim.x - 1) / gridDim.x;
    const uint64_t lo = blockIdx.x * per, hi = lo + per < E ? lo + per : E;
    double acc = 0.0;
    for (uint64_t i = lo + threadIdx.x; i < hi; i += blockDim.x) acc = fma(a[i], b[i], acc);
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        double total = 0.0;
        for (int w = 0; w < kThreads / 32; ++w) total += red[w];
        partial[blockIdx.x] = total;
    }
}

__global__ void k_dot_final(const double *partial, int nblk, double *out) {
    const int lane = threadIdx.x;
    const int per = (nblk + 31) / 32;
    double t = 0.0;
    for (int k = lane * per; k < nblk && k < (lane + 1) * per; ++k) t += partial[k];
    for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
    if (lane == 0) *out = t;
}

// Waits on a barrier nothing completes, with a poll bound; records a timeout.
__global__ void k_bounded_wait(int64_t polls, int32_t *status) {
    __shared__ uint64_t bar;
    if (threadIdx.x == 0) {
        mbar_init(&bar, 1);
        mbar_fence_init();
        bool ok = polls == 0;
        for (int64_t i = 0; i < polls && !ok; ++i) ok = mbar_try_wait(&bar, 0);
        *status = ok ? 0 : STAB_KSTATUS_TIMEOUT;
    }
}

}  // namespace

cudaError_t launch_bounded_wait(int64_t polls, int32_t *status, cudaStream_t st) {
    k_bounded_wait<<<1, 32, 0, st>>>(polls, status);
    return cudaGetLastError();
}

int max_map_count(const DevMap3 *maps, size_t n_maps) {
    int m = 0;
    for (size_t i = 0; i < n_maps; ++i) m = maps[i].count > m ? maps[i].count : m;
    return m;
}

cudaError_t launch_compose_maps(DevMap3 *maps, int n_maps, int max_count,
                                const int32_t *map_gate_idx, const RawGate *gates,
                                const double *thetas, cudaStream_t st) {
    if (n_maps == 0) return cudaSuccess;
    // a CTA per map while the CTAs are few and a warp's lanes would walk 32 gates and more
    if (max_count >= 1024 && n_maps <= 1024)
        k_compose_maps_cta<<<n_maps, 1024, 0, st>>>(maps, map_gate_idx, gates, thetas);
    else if (!warp_per_run(n_maps, max_count))
        k_compose_maps_seq<<<(n_maps + 127) / 128, 128, 0, st>>>(maps, n_maps, map_gate_idx, gates,
                                                                 thetas);
    else
        k_compose_maps<<<(n_maps + 3) / 4, 128, 0, st>>>(maps, n_maps, map_gate_idx, gates,
                                                         thetas);
    return cudaGetLastError();
}

cudaError_t launch_encode(DevOp *ops, int n_ops, DevMap3 *maps, int n_maps, int max_count,
                          const int32_t *map_gate_idx, const RawGate *gates, const double *thetas,
                          cudaStream_t st) {
    cudaError_t e = launch_compose_maps(maps, n_maps, max_count, map_gate_idx, gates, thetas, st);
    if (e != cudaSuccess || n_ops == 0) return e;
    k_encode<<<(n_ops + 127) / 128, 128, 0, st>>>(ops, n_ops, thetas);
    return cudaGetLastError();
}

cudaError_t launch_encode_stream(Rec *recs, const int32_t *enc, int n_enc, const DevMap3 *maps,
                                 const double *thetas, cudaStream_t st) {
    if (n_enc == 0) return cudaSuccess;
    k_encode_stream<<<(n_enc + 127) / 128, 128, 0, st>>>(recs, enc, n_enc, maps, thetas);
    return cudaGetLastError();
}

cudaError_t launch_fill(double *vec, int n, int n_vec, int init, const DevTerm *terms,
                        int n_terms, cudaStream_t st) {
    const uint64_t total = (1ull << (2 * n)) * (uint64_t)n_vec;
    k_fill<<<grid_for(total, kThreads), kThreads, 0, st>>>(vec, n, n_vec, init);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess || init != INIT_TERMS || n_terms == 0) return e;
    k_scatter_terms<<<(n_terms + 127) / 128, 128, 0, st>>>(vec, terms, n_terms);
    return cudaGetLastError();
}

cudaError_t launch_stream_wire(double *vec, int n, int n_vec, const DevPass &p, const DevOp *ops,
                               const DevMap3 *maps, int inverse, cudaStream_t st) {
    const uint64_t total = (1ull << (2 * n - 2)) * (uint64_t)n_vec;
    k_stream_wire<<<grid_for(total, kThreads), kThreads, 0, st>>>(vec, n, n_vec, p, ops, maps,
                                                                   inverse);
    return cudaGetLastError();
}

cudaError_t launch_stream_pull(const double *src, double *dst, int n, int n_vec,
                               const DevPull *pull, cudaStream_t st) {
    const uint64_t per = ((1ull << (2 * n)) + 1023) >> 10;
    k_stream_pull<<<grid_for(per * (uint64_t)n_vec * kThreads, kThreads), kThreads, 0, st>>>(
        src, dst, n, n_vec, pull);
    return cudaGetLastError();
}

cudaError_t launch_stream_cliff(const double *src, double *dst, int n, int n_vec,
                                const DevPass &p, const DevOp *ops, int inverse, cudaStream_t st) {
    const uint64_t total = (1ull << (2 * n)) * (uint64_t)n_vec;
    k_stream_cliff<<<grid_for(total, kThreads), kThreads, 0, st>>>(src, dst, n, n_vec, p, ops,
                                                                    inverse);
    return cudaGetLastError();
}

cudaError_t launch_stream_tile(const double *src, double *dst, int n, int n_vec,
                               const TileGroup &tg, const DevMap3 *maps, const DevOp *ops,
                               cudaStream_t st) {
    const uint64_t tiles = (uint64_t)n_vec << tg.rest_bits;
    int threads = (1 << tg.tile_bits) / 4;
    if (threads < 32) threads = 32;
    uint64_t grid = tiles;
    if (grid > 152ull * 16ull) grid = 152ull * 16ull;
    if (ops)
        k_stream_tile<false><<<(int)grid, threads, 0, st>>>(src, dst, n, n_vec, tg, maps, ops);
    else
        k_stream_tile<true><<<(int)grid, threads, 0, st>>>(src, dst, n, n_vec, tg, maps, nullptr);
    return cudaGetLastError();
}

int chain_max_ctas(int threads) {
    int dev = 0, sms = 0, per = 0, coop = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_stream_chain<false>, threads, 0) !=
            cudaSuccess) {
        (void)cudaGetLastError();
        return 0;
    }
    return coop ? per * sms : 0;
}

cudaError_t launch_chain_tables(const ChainShape *shapes, int n_shapes, int n, cudaStream_t st) {
    if (n_shapes == 0) return cudaSuccess;
    k_chain_tables<<<n_shapes, 128, 0, st>>>(shapes, n);
    return cudaGetLastError();
}

cudaError_t launch_stream_chain(const ChainArgs &a, cudaStream_t st) {
    const int threads = 1 << (a.tile_bits - 2);
    if (a.n_chains < 1 || threads < (int)(sizeof(ChainStep) / 4) ||
        threads < 9 * kTileMaxPasses || threads > kTileThreads)
        return cudaErrorInvalidValue;
    ChainArgs args = a;
    void *params[] = {&args};
    return cudaLaunchCooperativeKernel(a.alone ? (const void *)k_stream_chain<true>
                                               : (const void *)k_stream_chain<false>,
                                       dim3((unsigned)a.grid), dim3((unsigned)threads), params, 0,
                                       st);
}

cudaError_t launch_dot(const double *a, const double *b, int n, double *partial, double *out,
                       cudaStream_t st) {
    k_dot_partial<<<kDotBlocks, kThreads, 0, st>>>(a, b, n, partial);
    k_dot_final<<<1, 32, 0, st>>>(partial, kDotBlocks, out);
    return cudaGetLastError();
}

cudaError_t launch_xfree_sum(const double *vec, int n, int n_vec, double *out, cudaStream_t st) {
    k_xfree_sum<<<n_vec, kThreads, 0, st>>>(vec, n, out);
    return cudaGetLastError();
}

}  // namespace stab
