// k_resident.cu -- propagation with the whole 4^n coefficient vector resident
// in shared memory, one CTA per vector (n <= 6), reading an instruction stream
// staged chunk by chunk with bulk copies (see tma.cuh).
//
// The CTA walks the passes of the loaded circuit (the sequential Map stage of
// Sec. IV-B).  Each pass reads its wire's groups from one shared buffer --
// pulling every entry through the preceding run of two-qubit Clifford gates
// (map_CX of Sec. III-C, and CZ) -- applies the wire's ops and writes the
// other buffer; the buffers then swap.  Two thread mappings:
//   LPG = 4 (n <= 4): the wire run is one composed 3x3 map and a quad of
//     lanes holds a group (slots I, X, Y, Z); each lane pulls its own entry,
//     gets the other two through warp shuffles and computes its output row:
//     three dependent FP64 instructions per pass.  An FP64 instruction costs
//     ~68 cycles per warp on this GPU whatever the active-lane mask, so this is
//     the shortest pass; the next pass's source index is computed while the
//     current pass's FP64 chain is in flight.
//   LPG = 1 (n = 5, 6): one lane per group running the ops in registers
//     (lifting rotations, 3 FMAs per rotation): the fewest FP64 instructions.
// The adjoint kernel carries the cotangent and the forward vector backward
// together and reduces each rotation's gradient dot at the end of its pass.
#include <cuda_runtime.h>

#include "resident.cuh"

namespace stab {

namespace {

using namespace resident;

template <int N, int LPG>
__global__ void __launch_bounds__(SCfg<N, LPG>::T) k_resident_stream(StreamArgs a) {
    using C = SCfg<N, LPG>;
    extern __shared__ __align__(128) unsigned char smem[];
    Stager st;
    st.s0 = a.stream;
    st.s1 = nullptr;
    st.n0 = a.n_chunks;
    st.n_total = a.n_chunks;
    stager_setup(st, smem);
    double *red = reinterpret_cast<double *>(smem + kOffRed);
    double *bufA = reinterpret_cast<double *>(smem + kSmemHeader);
    double *bufB = bufA + C::E;
    st.start();

    const int b = blockIdx.x;
    for (int i = threadIdx.x; i < C::E; i += C::T) {
        double v = 0.0;
        if (a.init == INIT_RHO0) v = (i < (1 << N)) ? 1.0 : 0.0;
        else if (a.init == INIT_LOAD) v = a.in[(size_t)b * C::E + i];
        bufA[i] = v;
    }
    __syncthreads();
    if (a.init == INIT_GENERATOR) {
        if (threadIdx.x == 0) bufA[1u << b] = 1.0;   // Z_b: z bit b set
    } else if (a.init == INIT_TERMS) {
        for (int k = threadIdx.x; k < a.n_terms; k += C::T) bufA[a.terms[k].idx] = a.terms[k].coeff;
    }
    __syncthreads();

    double *res = run_stream<N, LPG>(st, 0, a.n_chunks, bufA, bufB, a.status);
    if (res == nullptr) return;
    if (a.out) {
        double *o = a.out + (size_t)b * C::E;
        for (int i = threadIdx.x; i < C::E; i += C::T) o[i] = res[i];
    }
    if (a.xfree_out) {
        double acc = 0.0;
        for (int i = threadIdx.x; i < (1 << N); i += C::T) acc += res[i];
        const double total = block_sum<C::T>(acc, red);
        if (threadIdx.x == 0) a.xfree_out[b] = total;
    }
}

// ---------------------------------------------------------------- adjoint

template <int N>
__global__ void __launch_bounds__(SCfg<N, 1>::T) k_adjoint_stream(AdjointStreamArgs a) {
    using C = SCfg<N, 1>;
    extern __shared__ __align__(128) unsigned char smem[];
    Stager st;
    st.s0 = a.fwd;
    st.s1 = a.bwd;
    st.n0 = a.n_fwd_chunks;
    st.n_total = a.n_fwd_chunks + a.n_bwd_chunks;
    stager_setup(st, smem);
    double *red = reinterpret_cast<double *>(smem + kOffRed);
    double *rA = reinterpret_cast<double *>(smem + kSmemHeader);
    double *rB = rA + C::E, *lA = rB + C::E, *lB = lA + C::E;
    st.start();
    for (int i = threadIdx.x; i < C::E; i += C::T) {
        rA[i] = i < (1 << N) ? 1.0 : 0.0;
        lA[i] = 0.0;
    }
    __syncthreads();
    for (int k = threadIdx.x; k < a.n_terms; k += C::T) lA[a.terms[k].idx] = a.terms[k].coeff;
    __syncthreads();

    // forward: r_m = M_m ... M_1 rho_0
    double *rho = run_stream<N, 1>(st, 0, a.n_fwd_chunks, rA, rB, a.status);
    if (rho == nullptr) return;
    double *rho_n = rho == rA ? rB : rA;
    double *lam = lA, *lam_n = lB;
    // no pull reuse at n = 5 here: with the forward sweep in the same kernel
    // the eight cached registers spill
    if (!adjoint_sweep<N, C::T, (N <= 4)>(st, a.n_fwd_chunks, st.n_total, lam, lam_n, rho,
                                          rho_n, a.grad_rot, a.status, smem, false, a.partials))
        return;
    double acc = 0.0;
    for (int i = threadIdx.x; i < (1 << N); i += C::T) acc += lam[i];
    const double total = block_sum<C::T>(acc, red);
    if (threadIdx.x == 0 && a.expect_out) *a.expect_out = total;
}

// Split adjoint, two CTAs, two launches (phase 0, then phase 1):
//   phase 0: CTA 0 carries rho_0 forward through the first part (stream 0)
//     into rmid, CTA 1 carries O backward through the second part (stream 1)
//     into lmid;
//   phase 1: both CTAs start from the pair (lmid, rmid) at the cut: CTA 0
//     sweeps it backward through the first part (stream 0) and also writes
//     <O> (x-free sum of lambda_0), CTA 1 forward through the second part
//     (stream 1); each rotation's dot lands in the part that holds it.
template <int N>
__global__ void __launch_bounds__(SCfg<N, 1>::T) k_adjoint_split(AdjointSplitArgs a) {
    using C = SCfg<N, 1>;
    extern __shared__ __align__(128) unsigned char smem[];
    const int b = blockIdx.x;
    Stager st;
    const bool fwd = b == 1;
    st.s0 = b == 0 ? a.stream[0] : a.stream[1];
    st.n0 = b == 0 ? a.n_chunks[0] : a.n_chunks[1];
    st.s1 = nullptr;
    st.n_total = st.n0;
    stager_setup(st, smem);
    double *red = reinterpret_cast<double *>(smem + kOffRed);
    double *rA = reinterpret_cast<double *>(smem + kSmemHeader);
    double *rB = rA + C::E, *lA = rB + C::E, *lB = lA + C::E;
    st.start();
    if (a.phase == 0) {
        for (int i = threadIdx.x; i < C::E; i += C::T)
            rA[i] = (b == 0 && i < (1 << N)) ? 1.0 : 0.0;
        __syncthreads();
        if (b == 1)
            for (int k = threadIdx.x; k < a.n_terms; k += C::T) rA[a.terms[k].idx] = a.terms[k].coeff;
        __syncthreads();
        const double *v = run_stream<N, 1>(st, 0, st.n_total, rA, rB, a.status);
        if (v == nullptr) return;
        double *out = b == 0 ? a.rmid : a.lmid;
        for (int i = threadIdx.x; i < C::E; i += C::T) out[i] = v[i];
        return;
    }
    for (int i = threadIdx.x; i < C::E; i += C::T) {
        rA[i] = a.rmid[i];
        lA[i] = a.lmid[i];
    }
    __syncthreads();
    double *rho = rA, *rho_n = rB, *lam = lA, *lam_n = lB;
    const bool ok = adjoint_sweep<N>(st, 0, st.n_total, lam, lam_n, rho, rho_n, a.grad_rot,
                                     a.status, smem, fwd, a.partials);
    if (!ok || b != 0) return;
    double acc = 0.0;
    for (int i = threadIdx.x; i < (1 << N); i += C::T) acc += lam[i];
    const double total = block_sum<C::T>(acc, red);
    if (threadIdx.x == 0 && a.expect_out) *a.expect_out = total;
}

template <int N, int LPG>
cudaError_t launch_stream_n(const StreamArgs &a, cudaStream_t s) {
    using C = SCfg<N, LPG>;
    const size_t smem = kSmemHeader + 2 * (size_t)C::E * sizeof(double);
    static SmemLimit lim;
    cudaError_t e = raise_smem_limit(k_resident_stream<N, LPG>, smem, lim);
    if (e != cudaSuccess) return e;
    k_resident_stream<N, LPG><<<a.n_vec, C::T, smem, s>>>(a);
    return cudaGetLastError();
}

template <int N>
cudaError_t launch_adjoint_split_n(const AdjointSplitArgs &a, cudaStream_t s) {
    using C = SCfg<N, 1>;
    const size_t smem = kSmemHeader + 4 * (size_t)C::E * sizeof(double);
    static SmemLimit lim;
    cudaError_t e = raise_smem_limit(k_adjoint_split<N>, smem, lim);
    if (e != cudaSuccess) return e;
    k_adjoint_split<N><<<2, C::T, smem, s>>>(a);
    return cudaGetLastError();
}

template <int N>
cudaError_t launch_adjoint_stream_n(const AdjointStreamArgs &a, cudaStream_t s) {
    using C = SCfg<N, 1>;
    const size_t smem = kSmemHeader + 4 * (size_t)C::E * sizeof(double);
    static SmemLimit lim;
    cudaError_t e = raise_smem_limit(k_adjoint_stream<N>, smem, lim);
    if (e != cudaSuccess) return e;
    k_adjoint_stream<N><<<1, C::T, smem, s>>>(a);
    return cudaGetLastError();
}

}  // namespace

int resident_lanes_per_group(int n) { return n <= 4 ? 4 : 1; }

cudaError_t launch_resident_stream(int n, const StreamArgs &a, cudaStream_t s) {
    switch (n) {
    case 1: return launch_stream_n<1, 4>(a, s);
    case 2: return launch_stream_n<2, 4>(a, s);
    case 3: return launch_stream_n<3, 4>(a, s);
    case 4: return launch_stream_n<4, 4>(a, s);
    case 5: return launch_stream_n<5, 1>(a, s);
    case 6: return launch_stream_n<6, 1>(a, s);
    default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_adjoint_stream(int n, const AdjointStreamArgs &a, cudaStream_t s) {
    switch (n) {
    case 1: return launch_adjoint_stream_n<1>(a, s);
    case 2: return launch_adjoint_stream_n<2>(a, s);
    case 3: return launch_adjoint_stream_n<3>(a, s);
    case 4: return launch_adjoint_stream_n<4>(a, s);
    case 5: return launch_adjoint_stream_n<5>(a, s);
    case 6: return launch_adjoint_stream_n<6>(a, s);
    default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_adjoint_split(int n, const AdjointSplitArgs &a, cudaStream_t s) {
    switch (n) {
    case 1: return launch_adjoint_split_n<1>(a, s);
    case 2: return launch_adjoint_split_n<2>(a, s);
    case 3: return launch_adjoint_split_n<3>(a, s);
    case 4: return launch_adjoint_split_n<4>(a, s);
    case 5: return launch_adjoint_split_n<5>(a, s);
    case 6: return launch_adjoint_split_n<6>(a, s);
    default: return cudaErrorInvalidValue;
    }
}

int resident_adjoint_threads(int n) {
    switch (n) {
    case 1: return SCfg<1, 1>::T;
    case 2: return SCfg<2, 1>::T;
    case 3: return SCfg<3, 1>::T;
    case 4: return SCfg<4, 1>::T;
    case 5: return SCfg<5, 1>::T;
    case 6: return SCfg<6, 1>::T;
    default: return 0;
    }
}

}  // namespace stab
