// k_sparse.cu -- propagation of a Pauli-term list: the sparse (lambda, I)
// representation of a stabilizer (Sec. II-B), kept while its stabilizer
// order n' (the number of strings, Fig. 1) is small, so that n is limited by
// the list, not by a 4^n vector (keys z | x << n in 64 bits, n <= 32).
//
// Clifford gates do not touch the list.  A rotation behind a Clifford U acts on
// U's images as the rotation about the string U^dagger sigma U acts on the
// terms themselves, so every rotation is pulled back through the Clifford gates
// before it (SpRot, made once per circuit load) and the gates' tableau is
// applied to the last list alone.  (Mapping the whole list at each of 29
// Clifford runs took a quarter of a 32-qubit call of 28 rotations.)
//
// A rotation about P mixes the two strings of each anticommuting pair (u, v),
// v = u P up to a phase, as u' = c u - s v, v' = s u + c v (Table I); a term
// whose partner is absent spawns it.  The images stand where the u term stood
// (or the lone term), u first: the list order is the input order, independent
// of the grid.  Exact zeros are never stored.  Two phases:
//   pair  -- every anticommuting term puts its position at its pair's place in
//            an open-addressing table (both strings of a pair hash alike, so the
//            second one to come finds the first, and tells it);
//   write -- images, their positions by a scan, and the table is cleared.
// Short lists run in one CTA's shared memory, rotation after rotation
// (k_sp_small); from there on the whole GPU takes the rest in one cooperative
// launch (k_sp_run).  n = 32, 20,000 gates, 28 rotations, <O> up to 5.7 million
// terms: 2.10 -> 0.73 ms; one generator, 96,000 terms: 1.19 -> 0.37 ms; n = 13, 12
// rotations, 2,400 terms: 451 -> 90 us (before: five launches a rotation, the
// list mapped at every Clifford run).
#include <cuda_runtime.h>

#include "../../include/stab.h"
#include "launch.h"

namespace stab {

namespace {

constexpr int kSpThreads = 256;
constexpr uint64_t kSpFree = ~0ull;

// one population count for both halves: they run at an eighth of the integer rate
__device__ __forceinline__ uint32_t sp_parity(uint64_t x) {
    return (uint32_t)__popc((uint32_t)(x >> 32) ^ (uint32_t)x) & 1u;
}

__device__ __forceinline__ bool sp_nonzero(double x) {
    return (__double_as_longlong(x) << 1) != 0;   // off the FP64 pipe
}

__device__ __forceinline__ uint64_t sp_hash(uint64_t key) {
    return (key ^ (key >> 31)) * 0x9E3779B97F4A7C15ull;
}

// Exponent c (mod 4) of P(a) P(b) = i^c P(a xor b) for Hermitian Pauli strings
// given by x / z masks: per qubit, with a = Y: z_b - x_b; a = X: z_b (2 x_b - 1);
// a = Z: x_b (1 - 2 z_b) (the phase function of the stabilizer tableau
// algorithm of Aaronson and Gottesman), summed with one population count:
// the complement of `minus` counts 32 - |minus|.
__device__ __forceinline__ uint32_t sp_mul_phase(uint32_t ax, uint32_t az, uint32_t bx,
                                                 uint32_t bz) {
    const uint32_t A = ax & az, B = ax & ~az, C = ~ax & az;
    const uint32_t plus = (A & bz & ~bx) | (B & bz & bx) | (C & bx & ~bz);
    const uint32_t minus = (A & bx & ~bz) | (B & bz & ~bx) | (C & bx & bz);
    return (uint32_t)__popcll(((uint64_t)~minus << 32) | plus) & 3u;
}

__device__ __forceinline__ bool sp_anti(uint64_t key, const SpRot &d) {
    return sp_parity(key & d.anti) != 0;
}

__device__ __forceinline__ bool sp_is_u(uint64_t key, const SpRot &d) {
    return sp_parity(key & d.letter) == (d.flags & 1u);
}

__device__ __forceinline__ double sp_neg_if(double x, bool neg) {   // off the FP64 pipe, too
    return __longlong_as_double(__double_as_longlong(x) ^ ((long long)neg << 63));
}

// The images of a term under the rotation: up to two (key, value) pairs in the
// order u, v, their number returned.  i u P = +-v: with the minus, v enters and
// leaves negated.  The FP64 pipe takes an instruction of a warp every 76 clocks:
// a warp of lone terms issues the two products it needs, a warp with a pair
// (any_paired: in the whole warp) four more; tests for zero and signs are integer
// work (with them off the pipe and one population count a parity the n = 32 call
// went from 1.07 to 0.97 ms).  All lanes call this together.
__device__ __forceinline__ int sp_images(bool in, bool any_paired, uint64_t key, double val,
                                         bool paired, double pval, const SpRot &d, int n,
                                         double c, double s, uint64_t &k0, double &v0,
                                         uint64_t &k1, double &v1) {
    const bool is_u = sp_is_u(key, d);
    const uint64_t ku = is_u ? key : key ^ d.P;
    const uint32_t zm = (uint32_t)((1ull << n) - 1ull);
    const uint32_t e = 1u + (d.flags & 2u) +
                       sp_mul_phase((uint32_t)(ku >> n), (uint32_t)ku & zm, (uint32_t)(d.P >> n),
                                    (uint32_t)d.P & zm);
    const bool minus = (e & 2u) != 0;
    // u: (c u, +-s u); v = +-val: (-s v, c v), whose own sign comes back
    const double cx = c * val, sx = s * val;
    double ou = is_u ? cx : sp_neg_if(sx, !minus);
    double ov = is_u ? sp_neg_if(sx, minus) : cx;
    if (any_paired) {
        const double vv = sp_neg_if(pval, minus);
        const double pu = fma(c, val, -(s * vv));
        const double pv = sp_neg_if(fma(s, val, c * vv), minus);
        if (paired) {
            ou = pu;
            ov = pv;
        }
    }
    const bool anti = sp_anti(key, d);
    // a commuting term stays; of a pair, the u term writes both
    const bool mix = in && anti && (is_u || !paired);
    const bool u_on = mix && sp_nonzero(ou), v_on = mix && sp_nonzero(ov);
    k0 = mix ? (u_on ? ku : ku ^ d.P) : key;
    v0 = mix ? (u_on ? ou : ov) : val;
    k1 = ku ^ d.P;
    v1 = ov;
    return mix ? (u_on ? 1 : 0) + (v_on ? 1 : 0) : (in && !anti ? 1 : 0);
}

template <typename T>
__device__ T block_exclusive_scan(T x, T &total, T *sh) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    T incl = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const T y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
    }
    if (lane == 31) sh[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        T w = lane < (int)(blockDim.x >> 5) ? sh[lane] : (T)0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const T y = __shfl_up_sync(0xffffffffu, w, o);
            if (lane >= o) w += y;
        }
        sh[lane] = w;   // inclusive prefix over warps
    }
    __syncthreads();
    const T warp_before = warp > 0 ? sh[warp - 1] : (T)0;
    total = sh[(blockDim.x >> 5) - 1];
    return warp_before + incl - x;
}

// Every term needs its slot's cos and sin; evaluating sincos for each cost the
// FP64 pipe more than the rotation itself on short lists.
__global__ void k_sp_cos_sin(const double *thetas, int64_t n_params, double *cs) {
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p < n_params) sincos(thetas[p], &cs[2 * p + 1], &cs[2 * p]);
}

// Entry (chunk c, subset t) of a tableau's chunk table is the ordered product
// prod_{q in c} (U X_q U^dagger)^{x_q} (U Z_q U^dagger)^{z_q} of the generator
// images the subset selects (bit j of t: x of qubit 4c + j, bit 4 + j: its z),
// as a Hermitian string and a phase i^e.  One block per chunk, one thread per
// subset.
__global__ void k_sp_tab_chunks(const SpTab *tab, int n, SpChunk *chunks) {
    const int c = blockIdx.x, t = threadIdx.x;
    const uint64_t zmask = (1ull << n) - 1;
    uint32_t rx = 0, rz = 0, e = 0;
    for (int j = 0; j < kSpChunkQubits; ++j) {
        const int q = kSpChunkQubits * c + j;
        if (q >= n) break;
        for (int part = 0; part < 2; ++part) {   // X_q, then Z_q
            if (!((t >> (part * kSpChunkQubits + j)) & 1)) continue;
            const SpTab g = tab[part ? n + q : q];
            const uint32_t gx = (uint32_t)(g.key >> n), gz = (uint32_t)(g.key & zmask);
            e += sp_mul_phase(rx, rz, gx, gz) + (g.neg ? 2u : 0u);
            rx ^= gx;
            rz ^= gz;
        }
    }
    chunks[(size_t)blockIdx.x * 256 + t] = SpChunk{rx, rz, e & 3u, 0u};
}

// U P U^dagger from the tableau: P(x, z) = i^{|x & z|} prod_q X_q^{x_q} Z_q^{z_q}
// (Y = i X Z), so its image is i^{|x & z|} times the product of the generator
// images in that order, taken chunk by chunk: ceil(n / 4) lookups and string
// products.  A Hermitian image: e is 0 or 2 (mod 4).
__device__ __forceinline__ uint64_t sp_image(uint64_t k, int n, const SpChunk *chunks, bool &neg) {
    const uint32_t x = (uint32_t)(k >> n), z = (uint32_t)(k & ((1ull << n) - 1ull));
    uint32_t rx = 0, rz = 0, e = (uint32_t)__popc(x & z);
    for (int c = 0; c < (n + kSpChunkQubits - 1) / kSpChunkQubits; ++c) {
        const uint32_t sh = (uint32_t)(kSpChunkQubits * c);
        const SpChunk g = chunks[c * 256 + (((x >> sh) & 15u) | (((z >> sh) & 15u) << 4))];
        e += g.e + sp_mul_phase(rx, rz, g.x, g.z);
        rx ^= g.x;
        rz ^= g.z;
    }
    neg = (e & 2u) != 0;
    return ((uint64_t)rx << n) | rz;
}

__global__ void __launch_bounds__(kSpThreads) k_sp_images(const uint64_t *keys, const double *vals,
                                                           int64_t count, int n,
                                                           const SpChunk *chunks, DevTerm *out,
                                                           stab_term *terms) {
    __shared__ SpChunk sc[kSpChunks * 256];
    const int n_ch = (n + kSpChunkQubits - 1) / kSpChunkQubits;
    for (int k = threadIdx.x; k < n_ch * 256; k += blockDim.x) sc[k] = chunks[k];
    __syncthreads();
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < count;
         i += (int64_t)gridDim.x * blockDim.x) {
        bool neg;
        const uint64_t k = sp_image(keys[i], n, sc, neg);
        const double v = neg ? -vals[i] : vals[i];
        if (out) out[i] = DevTerm{v, k};
        if (terms) {
            terms[i].coeff = v;
            terms[i].x = k >> n;
            terms[i].z = k & ((1ull << n) - 1ull);
        }
    }
}

// ---------------------------------------------------------------- one CTA

// Lists of up to kSpSmallCap terms, in shared memory: two buffers of keys and
// coefficients, a table of positions of twice that (the key is looked up by the
// position), the partners.  A thread takes at most four neighbouring terms.  A
// rotation is the latency of its phases, 1.5 to 2 us up to 500 terms, then FP64:
// 6.5 at 2,500; as four launches it was about 16.  The rotation whose list would not
// fit is left to the grid kernel, which takes 10 us a rotation up to 150,000 terms.
constexpr int kSmallThreads = 1024, kSmallPer = kSpSmallCap / kSmallThreads;
constexpr int kSmallLog = 13, kSmallRots = 64;
struct SpSmall {
    uint64_t key[2][kSpSmallCap];
    double val[2][kSpSmallCap];
    int32_t table[1 << kSmallLog];
    int32_t partner[kSpSmallCap];
    SpRot rot[kSmallRots];
    double2 cs[kSmallRots];
    int32_t sh[32];
};
static_assert((1 << kSmallLog) >= 2 * kSpSmallCap, "a free slot is always near");

__global__ void __launch_bounds__(kSmallThreads, 1) k_sp_small(SpRunArgs a) {
    extern __shared__ __align__(16) unsigned char raw[];
    SpSmall &S = *reinterpret_cast<SpSmall *>(raw);
    const int t = threadIdx.x;
    int count = (int)a.st->count, cur = 0, r = 0, stop = SP_RUNNING;
    const int64_t lim = a.cap < kSpSmallCap ? a.cap : (int64_t)kSpSmallCap;
    for (int i = t; i < count; i += kSmallThreads) {
        S.key[0][i] = a.init[i];
        S.val[0][i] = __longlong_as_double((long long)a.init[count + i]);
    }
    for (int i = t; i < (1 << kSmallLog); i += kSmallThreads) S.table[i] = -1;
    for (int i = t; i < kSpSmallCap; i += kSmallThreads) S.partner[i] = -1;
    __syncthreads();
    for (; r < a.n_rot; ++r) {
        if (r % kSmallRots == 0) {
            if (t < kSmallRots && r + t < a.n_rot) {
                const SpRot d = a.rots[r + t];
                S.rot[t] = d;
                S.cs[t] = double2{a.cs[2 * d.param],
                                  a.inverse ? -a.cs[2 * d.param + 1] : a.cs[2 * d.param + 1]};
            }
            __syncthreads();
        }
        const SpRot d = S.rot[r % kSmallRots];
        const double2 cs = S.cs[r % kSmallRots];
        const int per = (count + kSmallThreads - 1) / kSmallThreads;
        const int i0 = t * per;
        int slot[kSmallPer];
#pragma unroll
        for (int j = 0; j < kSmallPer; ++j) {
            const int i = i0 + j;
            slot[j] = -1;
            if (j >= per || i >= count) continue;
            const uint64_t k = S.key[cur][i];
            if (!sp_anti(k, d)) continue;
            uint32_t s = (uint32_t)(sp_hash(sp_is_u(k, d) ? k : k ^ d.P) >> (64 - kSmallLog));
            for (int probe = 0; probe < (1 << kSmallLog); ++probe) {
                const int p = atomicCAS(&S.table[s], -1, i);
                if (p == -1) {
                    slot[j] = (int)s;
                    break;
                }
                if ((S.key[cur][p] ^ k) == d.P) {
                    S.partner[i] = p;
                    S.partner[p] = i;
                    break;
                }
                s = (s + 1u) & ((1u << kSmallLog) - 1u);
            }
        }
        __syncthreads();
        uint64_t k0[kSmallPer], k1[kSmallPer];
        double v0[kSmallPer], v1[kSmallPer];
        int e[kSmallPer], mine = 0;
#pragma unroll
        for (int j = 0; j < kSmallPer; ++j) {
            const int i = i0 + j;
            const bool in = j < per && i < count;
            e[j] = 0;
            if (!__any_sync(0xffffffffu, in)) continue;
            const int p = in ? S.partner[i] : -1;
            e[j] = sp_images(in, __any_sync(0xffffffffu, p >= 0), in ? S.key[cur][i] : 0ull,
                             in ? S.val[cur][i] : 0.0, p >= 0, p >= 0 ? S.val[cur][p] : 0.0, d,
                             a.n, cs.x, cs.y, k0[j], v0[j], k1[j], v1[j]);
            mine += e[j];
            if (p >= 0) S.partner[i] = -1;
            if (slot[j] >= 0) S.table[slot[j]] = -1;
        }
        int total;
        int at = block_exclusive_scan<int>(mine, total, S.sh);
        if (total > lim) break;
#pragma unroll
        for (int j = 0; j < kSmallPer; ++j) {
            if (e[j] > 0) {
                S.key[1 - cur][at] = k0[j];
                S.val[1 - cur][at] = v0[j];
                ++at;
            }
            if (e[j] > 1) {
                S.key[1 - cur][at] = k1[j];
                S.val[1 - cur][at] = v1[j];
                ++at;
            }
        }
        if (t == 0) a.counts[r + 1] = total;
        count = total;
        cur ^= 1;
        __syncthreads();
        if (a.threshold > 0 && total > a.threshold) {
            stop = SP_THRESHOLD;
            ++r;
            break;
        }
    }
    for (int i = t; i < count; i += kSmallThreads) {
        a.keys[0][i] = S.key[cur][i];
        a.vals[0][i] = S.val[cur][i];
    }
    if (t == 0) {
        a.st->count = count;
        a.st->rot = r;
        a.st->buf = 0;
        a.st->stop = stop;
    }
}

// ---------------------------------------------------------------- whole GPU

constexpr int kRunThreads = 512, kRunPer = 4;
constexpr int kRunWarps = kRunThreads / 32, kRunRots = 64;
constexpr uint32_t kRunPolls = 1u << 22;     // a second or two
constexpr int kTileBits = 32;                // a tile word: step tag, emitted terms

// Table slots (log2) for a list: four a term while that is no more than 8 MB
// (a claim that meets another costs a round trip to L2, and the slowest chain
// of a phase counts), one and a half beyond, where clearing counts.
__host__ __device__ __forceinline__ int sp_table_bits(int64_t count) {
    int l = 12;
    while (l < 20 && (1ll << l) < 4 * count) ++l;
    while ((1ll << l) < count + (count >> 1)) ++l;
    return l;
}

// Tiles of a list of up to `cap` terms: G a round, kRunPer * kRunThreads terms at most.
__host__ __device__ __forceinline__ int64_t sp_tile_words(int64_t cap, int64_t G) {
    return cap / (kRunPer * kRunThreads) + G;
}

// All CTAs of the cooperative launch meet; false once a wait gave up.
__device__ bool sp_grid_sync(SpState *st, uint32_t want, int *s_ok) {
    __syncthreads();
    if (threadIdx.x == 0) {
        asm volatile("red.release.gpu.global.add.u32 [%0], 1;" : : "l"(&st->arrived) : "memory");
        bool ok = false;
        for (uint32_t it = 0; it < kRunPolls && !ok; ++it) {
            uint32_t seen;
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];"
                         : "=r"(seen) : "l"(&st->arrived) : "memory");
            ok = arrivals_reached(seen, want);
        }
        if (!ok) atomicExch(&st->err, 2);
        *s_ok = ok ? 1 : 0;
    }
    __syncthreads();
    return *s_ok != 0;
}

// Rotations from the state's on, two grid barriers each.  Up to 200,000 terms the
// barriers' 2 to 3 us and the phases' own round trips are the time; of 3.8 million
// (0.15 ms) the pair phase is 48 us of table atomics, the write phase 71 us of FP64
// and issue (its lists take 25 us of HBM).  The table takes the list's size (1.5
// slots a term at least, 8 bytes each: 64 MB there, where one of the capacity's size
// and 16 bytes was 512 MB, out of L2).  Positions: a tile of the write phase needs the emitted terms before it.  CTA b holds tiles b,
// b + G, ...: between two of its tiles lie exactly G - 1 others, whose totals
// it reads at once (a thread each, tagged with the step, so no clearing); the
// tiles are all in flight on resident CTAs, which publish before they wait.
// What other CTAs wrote is read past L1.
struct SpTile {
    uint64_t key[2 * kRunPer * kRunThreads];
    double val[2 * kRunPer * kRunThreads];
    SpRot rot[kRunRots];
    double2 cs[kRunRots];
    int64_t red[kRunWarps];
    int32_t wt[kRunPer * kRunWarps];
    int32_t own, ok;
};

__global__ void __launch_bounds__(kRunThreads, 2) k_sp_run(SpRunArgs a) {
    extern __shared__ __align__(16) unsigned char raw[];
    SpTile &S = *reinterpret_cast<SpTile *>(raw);
    SpState *st = a.st;
    int64_t count = st->count;
    int r = st->rot, cur = st->buf, stop = st->stop;
    if (stop != SP_RUNNING || r >= a.n_rot) return;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int64_t G = gridDim.x, b = blockIdx.x;
    uint32_t meets = 0;
    // tags of an earlier launch could match this one's
    {
        const int64_t words = sp_tile_words(a.cap, G);
        for (int64_t i = b * kRunThreads + t; i < words; i += G * kRunThreads) a.tiles[i] = 0;
    }
    const int r0 = r;
    for (; r < a.n_rot; ++r) {
        if ((r - r0) % kRunRots == 0) {
            if (t < kRunRots && r + t < a.n_rot) {
                const SpRot f = a.rots[r + t];
                S.rot[t] = f;
                S.cs[t] = double2{a.cs[2 * f.param],
                                  a.inverse ? -a.cs[2 * f.param + 1] : a.cs[2 * f.param + 1]};
            }
            __syncthreads();
        }
        const SpRot d = S.rot[(r - r0) % kRunRots];
        const double c = S.cs[(r - r0) % kRunRots].x, s = S.cs[(r - r0) % kRunRots].y;
        const uint64_t *keys = cur ? a.keys[1] : a.keys[0];
        const double *vals = cur ? a.vals[1] : a.vals[0];
        const int log_h = sp_table_bits(count);
        const uint32_t mask = (1u << log_h) - 1u;
        // as many rounds as full tiles would take, of equal tiles (whole warps: a
        // full tile in a last round that few CTAs have took as long as one that
        // all have, and so did a short list in few full tiles)
        const int64_t full = G * kRunPer * kRunThreads, rounds = count > full ? (count + full - 1) / full : 1;
        const int64_t even = (count + G * rounds - 1) / (G * rounds);
        const int tile_terms = count > 0 ? (int)((even + 31) / 32 * 32) : 32;
        // pair
        uint64_t next[kRunPer];
        auto look = [&](int64_t base) {
#pragma unroll
            for (int j = 0; j < kRunPer; ++j) {
                const int64_t i = base + j * kRunThreads + t;
                next[j] = j * kRunThreads + t < tile_terms && i < count ? __ldcg((const unsigned long long *)keys + i) : 0ull;
            }
        };
        look(b * tile_terms);
        for (int64_t base = b * tile_terms; base < count; base += G * tile_terms) {
            uint64_t k[kRunPer], old[kRunPer], mine[kRunPer];
            uint32_t slot[kRunPer];
            bool anti[kRunPer];
#pragma unroll
            for (int j = 0; j < kRunPer; ++j) k[j] = next[j];
            look(base + G * tile_terms);
#pragma unroll
            for (int j = 0; j < kRunPer; ++j) {
                // no key (zero, or past the end) is one that commutes with all
                anti[j] = sp_anti(k[j], d);
                const uint64_t h = sp_hash(sp_is_u(k[j], d) ? k[j] : k[j] ^ d.P);
                slot[j] = (uint32_t)(h >> (64 - log_h));
                mine[j] = ((uint64_t)(uint32_t)(h >> (32 - log_h)) << 32) |
                          (uint32_t)(base + j * kRunThreads + t);
                old[j] = kSpFree;
                if (anti[j])
                    old[j] = atomicCAS((unsigned long long *)a.table + slot[j], kSpFree, mine[j]);
            }
            // the terms that met an occupied slot look on together (one after the
            // other: 83 -> 48 us of this phase at 3.8 million terms), each at its own
            // odd step: neighbouring slots grow long chains of round trips, and the
            // whole GPU waits for the longest (500,000 terms, this phase and its
            // barrier: 14.8 -> 8.3 us)
            for (uint32_t probe = 0;; ++probe) {
                bool more = false;
#pragma unroll
                for (int j = 0; j < kRunPer; ++j) {
                    if (old[j] == kSpFree) continue;
                    if ((uint32_t)(old[j] >> 32) == (uint32_t)(mine[j] >> 32)) {
                        const uint32_t p = (uint32_t)old[j];
                        if ((__ldcg((const unsigned long long *)keys + p) ^ k[j]) == d.P) {
                            const uint32_t i = (uint32_t)mine[j];
                            a.partner[i] = (int32_t)p;
                            a.partner[p] = (int32_t)i;
                            old[j] = kSpFree;
                            continue;
                        }
                    }
                    slot[j] = (slot[j] + ((uint32_t)(mine[j] >> 32) | 1u)) & mask;
                    more = true;
                }
                if (!more) break;
                if (probe > mask) {          // only guards against a corrupted table
                    atomicExch(&st->err, 1);
                    break;
                }
#pragma unroll
                for (int j = 0; j < kRunPer; ++j)
                    if (old[j] != kSpFree)
                        old[j] = atomicCAS((unsigned long long *)a.table + slot[j], kSpFree,
                                           mine[j]);
            }
        }
        if (!sp_grid_sync(st, (uint32_t)G * ++meets, &S.ok)) return;
        // write
        const int64_t n_tiles = count > 0 ? (count + tile_terms - 1) / tile_terms : 1;
        uint64_t *keys_out = cur ? a.keys[0] : a.keys[1];
        double *vals_out = cur ? a.vals[0] : a.vals[1];
        const uint64_t tag = (uint64_t)(uint32_t)(r + 1) << kTileBits;
        {
            const uint4 free4{~0u, ~0u, ~0u, ~0u};
            const int64_t quads = (int64_t)1 << (log_h - 1);
            for (int64_t i = b * kRunThreads + t; i < quads; i += G * kRunThreads)
                reinterpret_cast<uint4 *>(a.table)[i] = free4;
        }
        int64_t before = 0;                  // emitted by this CTA's last tile and all before it
        uint64_t k[kRunPer];
        double v[kRunPer];
        int32_t p[kRunPer];
        auto fetch = [&](int64_t tile) {
#pragma unroll
            for (int j = 0; j < kRunPer; ++j) {
                const int64_t i = tile * tile_terms + j * kRunThreads + t;
                const bool in = j * kRunThreads + t < tile_terms && i < count;
                k[j] = in ? __ldcg((const unsigned long long *)keys + i) : 0ull;
                v[j] = in ? __ldcg(vals + i) : 0.0;
                p[j] = in ? __ldcg(a.partner + i) : -1;
            }
        };
        fetch(b);
        for (int64_t tile = b; tile < n_tiles; tile += G) {
            uint64_t k1[kRunPer];
            double v1[kRunPer], pv[kRunPer];
            int32_t at[kRunPer];
            int e[kRunPer];
#pragma unroll
            for (int j = 0; j < kRunPer; ++j) {
                const int64_t i = tile * tile_terms + j * kRunThreads + t;
                pv[j] = 0.0;
                if (p[j] >= 0) {
                    pv[j] = __ldcg(vals + p[j]);
                    a.partner[i] = -1;
                }
            }
#pragma unroll
            for (int j = 0; j < kRunPer; ++j) {
                const bool in = j * kRunThreads + t < tile_terms &&
                                tile * tile_terms + j * kRunThreads + t < count;
                e[j] = 0;
                if (__any_sync(0xffffffffu, in)) {
                    const uint64_t key = k[j];
                    const double val = v[j];
                    e[j] = sp_images(in, __any_sync(0xffffffffu, p[j] >= 0), key, val, p[j] >= 0,
                                     pv[j], d, a.n, c, s, k[j], v[j], k1[j], v1[j]);
                }
                const uint32_t one = __ballot_sync(0xffffffffu, e[j] > 0);
                const uint32_t two = __ballot_sync(0xffffffffu, e[j] > 1);
                const uint32_t lt = (1u << lane) - 1u;
                at[j] = __popc(one & lt) + __popc(two & lt);
                if (lane == 0) S.wt[j * kRunWarps + warp] = __popc(one) + __popc(two);
            }
            __syncthreads();
            if (warp == 0) {                 // exclusive scan of the warp totals
                constexpr int kTot = kRunPer * kRunWarps / 32;
                int x[kTot], incl = 0;
#pragma unroll
                for (int k2 = 0; k2 < kTot; ++k2) {
                    x[k2] = incl;
                    incl += S.wt[kTot * lane + k2];
                }
                const int mine = incl;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int y = __shfl_up_sync(0xffffffffu, incl, o);
                    if (lane >= o) incl += y;
                }
#pragma unroll
                for (int k2 = 0; k2 < kTot; ++k2) S.wt[kTot * lane + k2] = incl - mine + x[k2];
                if (lane == 31) {
                    *(volatile unsigned long long *)(a.tiles + tile) = tag | (uint32_t)incl;
                    S.own = incl;
                }
            }
            __syncthreads();
            const int own = S.own;
#pragma unroll
            for (int j = 0; j < kRunPer; ++j) {
                const int o = S.wt[j * kRunWarps + warp] + at[j];
                if (e[j] > 0) {
                    S.key[o] = k[j];
                    S.val[o] = v[j];
                }
                if (e[j] > 1) {
                    S.key[o + 1] = k1[j];
                    S.val[o + 1] = v1[j];
                }
            }
            if (tile + G < n_tiles) fetch(tile + G);
            // the tiles between this CTA's last one and this one
            int64_t sum = 0;
            bool ok = true;
            for (int64_t u = tile - G + 1 + t; u < tile; u += kRunThreads) {
                if (u < 0) continue;
                uint64_t w = 0;
                uint32_t it = 0;
                do {
                    w = *(volatile unsigned long long *)(a.tiles + u);
                } while ((w >> kTileBits) != (tag >> kTileBits) && ++it < kRunPolls);
                if ((w >> kTileBits) != (tag >> kTileBits)) ok = false;
                sum += (int64_t)(uint32_t)w;
            }
            for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
            if (lane == 0) S.red[warp] = sum;
            if (!__syncthreads_and(ok)) {
                if (t == 0) atomicExch(&st->err, 2);
                return;
            }
            for (int w = 0; w < kRunWarps; ++w) before += S.red[w];
            for (int i = t; i < own; i += kRunThreads) {
                if (before + i < a.cap) {
                    keys_out[before + i] = S.key[i];
                    vals_out[before + i] = S.val[i];
                }
            }
            before += own;
            if (tile == n_tiles - 1 && t == 0) a.counts[r + 1] = before;
            __syncthreads();                 // the tile's arrays are used again
        }
        if (!sp_grid_sync(st, (uint32_t)G * ++meets, &S.ok)) return;
        const int64_t total = __ldcg((const long long *)a.counts + r + 1);
        if (total > a.cap) {
            stop = SP_OVERFLOW;
            break;
        }
        count = total;
        cur ^= 1;
        if (a.threshold > 0 && total > a.threshold) {
            stop = SP_THRESHOLD;
            ++r;
            break;
        }
    }
    if (b == 0 && t == 0) {
        st->count = count;
        st->rot = r;
        st->buf = cur;
        st->stop = stop;
    }
}

// Fixed-order sum of the coefficients whose images are x-free, in one launch:
// block sums over contiguous ranges, then one warp of the last block to finish
// (lane l a contiguous slice of the partials, then a shuffle tree).  The bits
// of an image's x mask are tried one by one: of lists that are all but random,
// a term takes two.
__global__ void __launch_bounds__(kSpThreads) k_sp_xfree(SpRunArgs a, const uint64_t *xcol,
                                                          const SpChunk *chunks,
                                                          double *partial) {
    __shared__ double red[kSpThreads / 32];
    __shared__ uint64_t col[32];
    __shared__ int last;
    const int n = a.n;
    if ((int)threadIdx.x < n) col[threadIdx.x] = xcol[threadIdx.x];
    __syncthreads();
    const int64_t count = a.st->count;
    const uint64_t *keys = a.keys[a.st->buf];
    const double *vals = a.vals[a.st->buf];
    const int64_t per = (count + gridDim.x - 1) / gridDim.x;
    const int64_t lo = min((int64_t)blockIdx.x * per, count), hi = min(lo + per, count);
    double acc = 0.0;
    constexpr int kAhead = 8;
    for (int64_t i0 = lo + threadIdx.x; i0 < hi; i0 += kAhead * kSpThreads) {
        uint64_t k[kAhead];
#pragma unroll
        for (int j = 0; j < kAhead; ++j)
            k[j] = i0 + j * kSpThreads < hi ? keys[i0 + j * kSpThreads] : 0ull;
#pragma unroll
        for (int j = 0; j < kAhead; ++j) {
            const int64_t i = i0 + j * kSpThreads;
            int q = i < hi ? 0 : -1;
            while (q >= 0 && q < n && !sp_parity(k[j] & col[q])) ++q;
            if (q == n) {
                bool neg;
                (void)sp_image(k[j], n, chunks, neg);
                acc += neg ? -vals[i] : vals[i];
            }
        }
    }
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < kSpThreads / 32; ++w) t += red[w];
        partial[blockIdx.x] = t;
        __threadfence();
        last = atomicAdd(&a.st->blocks, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!last || threadIdx.x >= 32) return;
    __threadfence();
    constexpr int kPer = kSpMaxBlocks / 32;
    static_assert(kPer * 32 == kSpMaxBlocks, "whole slices");
    double p[kPer], t = 0.0;
#pragma unroll
    for (int j = 0; j < kPer; ++j) p[j] = __ldcg(partial + threadIdx.x * kPer + j);
#pragma unroll
    for (int j = 0; j < kPer; ++j) t += p[j];
    for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
    if (threadIdx.x == 0) {
        a.st->value = t;
        a.st->blocks = 0;
    }
}

}  // namespace

cudaError_t launch_sp_cos_sin(const double *thetas, int64_t n_params, double *cs,
                              cudaStream_t st) {
    if (n_params <= 0) return cudaSuccess;
    k_sp_cos_sin<<<(unsigned)((n_params + 255) / 256), 256, 0, st>>>(thetas, n_params, cs);
    return cudaGetLastError();
}

cudaError_t launch_sp_chunks(const SpTab *tab, int n, SpChunk *chunks, cudaStream_t st) {
    k_sp_tab_chunks<<<kSpChunks, 256, 0, st>>>(tab, n, chunks);
    return cudaGetLastError();
}

int sp_table_log(int64_t count) { return sp_table_bits(count); }

int64_t sp_tiles(int64_t cap, int grid) { return sp_tile_words(cap, grid); }

cudaError_t sp_run_grid(int device, int *grid) {
    int sms = 0, per = 0;
    cudaError_t e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_sp_run, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)sizeof(SpTile));
    if (e == cudaSuccess)
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_sp_run, kRunThreads,
                                                          sizeof(SpTile));
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_sp_small, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)sizeof(SpSmall));
    if (e != cudaSuccess) return e;
    *grid = sms * (per < 2 ? per : 2);
    return *grid > 0 ? cudaSuccess : cudaErrorInvalidConfiguration;
}

cudaError_t launch_sp_small(const SpRunArgs &a, cudaStream_t st) {
    k_sp_small<<<1, kSmallThreads, sizeof(SpSmall), st>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_sp_run(const SpRunArgs &a, cudaStream_t st) {
    SpRunArgs args = a;
    void *params[] = {&args};
    return cudaLaunchCooperativeKernel((const void *)k_sp_run, dim3((unsigned)a.grid),
                                       dim3(kRunThreads), params, sizeof(SpTile), st);
}

cudaError_t launch_sp_xfree(const SpRunArgs &a, const uint64_t *xcol, const SpChunk *chunks,
                            double *partial, cudaStream_t st) {
    k_sp_xfree<<<kSpMaxBlocks, kSpThreads, 0, st>>>(a, xcol, chunks, partial);
    return cudaGetLastError();
}

cudaError_t launch_sp_images(const uint64_t *keys, const double *vals, int64_t count, int n,
                             const SpChunk *chunks, DevTerm *out, stab_term *terms,
                             cudaStream_t st) {
    if (count <= 0) return cudaSuccess;
    int64_t blocks = (count + 511) / 512;
    if (blocks > kSpMaxBlocks) blocks = kSpMaxBlocks;
    k_sp_images<<<(unsigned)blocks, kSpThreads, 0, st>>>(keys, vals, count, n, chunks, out,
                                                         terms);
    return cudaGetLastError();
}

}  // namespace stab
