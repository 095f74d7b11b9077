// k_gates.cu -- H, S, S^dag, T, T^dag, CNOT and general two-qubit gates
// (4x4 complex matrices) on a complex64 state vector (the Clifford
// preconditioning circuits, T doping and brick-wall circuits of the paper), applied
// in fused blocks: a run of consecutive gates acting inside a set of at most
// GATE_BLOCK_Q qubits (always containing qubits 0..4, so every tile is made of
// 256-byte contiguous runs) is applied to each 2^Q-amplitude tile with one
// global read and one global write of psi per block.
//
// Inside a block the tile passes through the registers in rounds. In a round
// every thread holds the 32 amplitudes of five local qubits (the round's slots;
// the others select the thread), and a gate is arithmetic in registers when
// its qubits are slots; a phase gate runs on any qubit and a CNOT needs only its
// target among the slots. Between rounds the tile is redistributed through
// shared memory with one barrier. The host orders a block's gates into rounds
// (sre_api.cu, run_gate_list). One barrier and one trip through shared memory
// per gate, as an in-place update of the shared tile takes, bound the kernel
// before: 1000 random Clifford + T gates at N = 26 took 31 ms in 32 blocks, now
// 17 ms (2.3 rounds a block; instruction issue bounds it, DRAM would take 5 ms);
// 552 two-qubit gates at N = 24 10.9 ms in 29 blocks, now 8.2 ms (4.3 rounds a
// block; 4.0 ms at the full FP32 rate).
#include "k_misc.cuh"

namespace sre {

struct GateBlockParams {
    int Q;                       // qubits in the block (GATE_BLOCK_Q in the rounds kernel)
    int n_other;                 // qubits outside the block
    unsigned char local[GATE_BLOCK_Q];   // global qubit of local bit i (ascending)
    unsigned char other[32];             // global qubit of tile bit i (ascending)
    int r0, nr;                  // rounds [r0, r0 + nr)
    int g0, ng;                  // gate rows of the block
};

namespace {

constexpr int GT = 256;                     // threads
constexpr int GE = 1 << GATE_ROUND_SLOTS;   // amplitudes per thread

// Shared-memory position of local index e: the nibbles above the lowest one
// are folded into it, so that lanes whose bits fall in different residues
// mod 4 (the host picks them so) hit different banks. Linear over GF(2).
__device__ __forceinline__ uint32_t gphys(uint32_t e) { return e ^ ((e >> 4) & 15u) ^ ((e >> 8) & 15u) ^ ((e >> 12) & 15u); }

template <int S>
__device__ __forceinline__ void gate_h(float2 (&v)[GE]) {
    const float2 r2 = make_float2(0.70710678118654752440f, 0.70710678118654752440f);
#pragma unroll
    for (int k = 0; k < GE; ++k)
        if (!(k & (1 << S))) {
            const float2 u = v[k], w = v[k | (1 << S)];
            v[k] = mul2(r2, add2(u, w));
            v[k | (1 << S)] = mul2(r2, sub2(u, w));
        }
}

// phase on the amplitudes whose index has all bits of MASK
template <int MASK>
__device__ __forceinline__ void gate_phase(float2 (&v)[GE], float cr, float ci) {
#pragma unroll
    for (int k = 0; k < GE; ++k)
        if ((k & MASK) == MASK) {
            const float2 u = v[k];
            v[k] = make_float2(cr * u.x - ci * u.y, cr * u.y + ci * u.x);
        }
}

// e^{i pi ph / 4}
__device__ __forceinline__ void phase_of(int ph, float &cr, float &ci) {
    const float r2 = 0.70710678118654752440f;
    const float a = (ph & 1) ? r2 : (ph & 2) ? 0.f : 1.f;     // |cos|
    const float b = (ph & 1) ? r2 : (ph & 2) ? 1.f : 0.f;     // |sin|
    cr = ((ph + 2) & 4) ? -a : a;
    ci = (ph & 4) ? -b : b;
}

// exchange of target pairs among the amplitudes whose index has all bits of CM,
// where the bits of m are set (m is all ones or zero). By exclusive or: as a
// plain exchange the compiler permutes registers, and where the gates' branches
// meet it then copies all 64 of them, three times the work of the gate itself.
template <int CM, int T>
__device__ __forceinline__ void gate_cx(float2 (&v)[GE], uint32_t m) {
#pragma unroll
    for (int k = 0; k < GE; ++k)
        if ((k & CM) == CM && !(k & (1 << T))) {
            float2 &a = v[k], &b = v[k | (1 << T)];
            const uint32_t tx = (__float_as_uint(a.x) ^ __float_as_uint(b.x)) & m;
            const uint32_t ty = (__float_as_uint(a.y) ^ __float_as_uint(b.y)) & m;
            a = make_float2(__uint_as_float(__float_as_uint(a.x) ^ tx), __uint_as_float(__float_as_uint(a.y) ^ ty));
            b = make_float2(__uint_as_float(__float_as_uint(b.x) ^ tx), __uint_as_float(__float_as_uint(b.y) ^ ty));
        }
}

// 4x4 matrix (16 entries, row-major) on slots A < B, local index bit(A) + 2 bit(B)
template <int A, int B>
__device__ __forceinline__ void gate_u2(float2 (&v)[GE], const float2 *u) {
    float2 m[16];
    const float4 *u4 = reinterpret_cast<const float4 *>(u);
#pragma unroll
    for (int e = 0; e < 8; ++e) {
        const float4 q = u4[e];
        m[2 * e] = make_float2(q.x, q.y);
        m[2 * e + 1] = make_float2(q.z, q.w);
    }
#pragma unroll
    for (int k = 0; k < GE; ++k)
        if (!(k & (1 << A)) && !(k & (1 << B))) {
            const int idx[4] = {k, k | (1 << A), k | (1 << B), k | (1 << A) | (1 << B)};
            float2 w[4];
#pragma unroll
            for (int l = 0; l < 4; ++l) w[l] = v[idx[l]];
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                float re = 0.f, im = 0.f;
#pragma unroll
                for (int l = 0; l < 4; ++l) {
                    re = fmaf(m[4 * r + l].x, w[l].x, fmaf(-m[4 * r + l].y, w[l].y, re));
                    im = fmaf(m[4 * r + l].x, w[l].y, fmaf(m[4 * r + l].y, w[l].x, im));
                }
                v[idx[r]] = make_float2(re, im);
            }
        }
}

} // namespace

// U2: the list holds two-qubit matrices only; otherwise none.
template <bool U2>
__global__ void __launch_bounds__(GT, 2) gate_block_kernel(float2 *psi, const GateRow *gates, const GateRound *rounds,
                                                           const float2 *mats, const GateBlockParams p) {
    extern __shared__ __align__(16) float2 amp[];
    __shared__ unsigned long long hioff[1 << (GATE_BLOCK_Q - GATE_BLOCK_LOW)];
    const unsigned long long tile = blockIdx.x + ((unsigned long long)blockIdx.y << 15);
    if (tile >= (1ULL << p.n_other)) return;   // uniform over the CTA
    unsigned long long base = 0;
    for (int i = 0; i < p.n_other; ++i) base |= ((tile >> i) & 1ULL) << p.other[i];
    // local bits 0..LOW-1 are global bits 0..LOW-1 (contiguous runs); the
    // global offset of the remaining local bits h = l >> LOW, one table entry
    // per value of h
    static_assert(GT == 1 << (GATE_BLOCK_Q - GATE_BLOCK_LOW), "one entry per thread");
    {
        unsigned long long o = base;
#pragma unroll
        for (int i = GATE_BLOCK_LOW; i < GATE_BLOCK_Q; ++i)
            o |= (unsigned long long)((threadIdx.x >> (i - GATE_BLOCK_LOW)) & 1) << p.local[i];
        hioff[threadIdx.x] = o;
    }
    // the block's two-qubit matrices, once per CTA (read back as broadcasts)
    float2 *msm = amp + (1 << GATE_BLOCK_Q);
    if constexpr (U2)
        for (int e = threadIdx.x; e < 16 * p.ng; e += GT) msm[e] = __ldg(mats + 16 * (size_t)p.g0 + e);
    __syncthreads();
    constexpr int LOWM = (1 << GATE_BLOCK_LOW) - 1;
    {
        // all loads of a thread in flight; thread t takes the indices t + 256 i
        float2 q[GE];
        const float2 *src = psi + (threadIdx.x & LOWM);
#pragma unroll
        for (int i = 0; i < GE; ++i) q[i] = src[hioff[(threadIdx.x >> GATE_BLOCK_LOW) + (GT >> GATE_BLOCK_LOW) * i]];
        const uint32_t at = gphys(threadIdx.x);
#pragma unroll
        for (int i = 0; i < GE; ++i) amp[at ^ gphys(GT * i)] = q[i];
    }
    const uint32_t t = threadIdx.x;
    static_assert(GT == 1 << (GATE_BLOCK_Q - GATE_ROUND_SLOTS), "a thread per coset of the slots");
    float2 v[GE];
    for (int ri = 0; ri < p.nr; ++ri) {
        const GateRound R = rounds[p.r0 + ri];
        __syncthreads();
        // amplitude k of thread t: byte address at ^ ok (positions are linear over GF(2))
        uint32_t at = 0, so[GATE_ROUND_SLOTS];
#pragma unroll
        for (int i = 0; i < GATE_BLOCK_Q - GATE_ROUND_SLOTS; ++i) at |= ((t >> i) & 1u) << R.thr[i];
        at = gphys(at) * (uint32_t)sizeof(float2);
#pragma unroll
        for (int i = 0; i < GATE_ROUND_SLOTS; ++i) so[i] = gphys(1u << R.slot[i]) * (uint32_t)sizeof(float2);
        char *sm = reinterpret_cast<char *>(amp);
        {
            // the 32 positions in Gray-code order, one exclusive or each
#pragma unroll
            for (int i = 0; i < GE; ++i) {
                if (i) at ^= so[__ffs(i) - 1];
                v[i ^ (i >> 1)] = *reinterpret_cast<const float2 *>(sm + at);
            }
            // phase gates on thread bits multiply all of a thread's amplitudes,
            // which commutes with the gates on its slots: they add up in ph (units
            // of pi / 4) and are applied once
            int ph = 0;
            uint32_t all;
            asm volatile("mov.u32 %0, -1;" : "=r"(all));
            GateRow next = gates[R.g0];
            for (int gi = R.g0; gi < R.g0 + R.ng; ++gi) {
                const GateRow G = next;
                if (gi + 1 < R.g0 + R.ng) next = gates[gi + 1];
                if constexpr (U2) {
                    const float2 *u = msm + 16 * (gi - p.g0);
                    switch (G.op) {
#define U(c, a, b) case c: gate_u2<a, b>(v, u); break;
                    U(0, 0, 1) U(1, 0, 2) U(2, 1, 2) U(3, 0, 3) U(4, 1, 3) U(5, 2, 3)
                    U(6, 0, 4) U(7, 1, 4) U(8, 2, 4) U(9, 3, 4)
#undef U
                    default: break;
                    }
                } else {
                    const uint32_t on = ((t >> G.q1) & 1u) ? ~0u : 0u;     // a thread bit controls the gate
                    switch (G.op) {
#define H(s) case GC_H + s: gate_h<s>(v); break;
                    H(0) H(1) H(2) H(3) H(4)
#undef H
#define P(s) case GC_PHASE + s: { float cr, ci; phase_of(G.q0, cr, ci); gate_phase<1 << s>(v, cr, ci); } break;
                    P(0) P(1) P(2) P(3) P(4)
#undef P
                    case GC_PHASE_THREAD: ph += G.q0 & on; break;
#define X(c, s) case GC_CX + 5 * c + s: gate_cx<1 << c, s>(v, all); break;
                    X(0, 1) X(0, 2) X(0, 3) X(0, 4) X(1, 0) X(1, 2) X(1, 3) X(1, 4) X(2, 0) X(2, 1) X(2, 3) X(2, 4)
                    X(3, 0) X(3, 1) X(3, 2) X(3, 4) X(4, 0) X(4, 1) X(4, 2) X(4, 3)
#undef X
#define Y(s) case GC_CX_THREAD + s: gate_cx<0, s>(v, on); break;
                    Y(0) Y(1) Y(2) Y(3) Y(4)
#undef Y
                    default: break;
                    }
                }
            }
            if constexpr (!U2) {
                if (ph & 7) {
                    float cr, ci;
                    phase_of(ph & 7, cr, ci);
                    gate_phase<0>(v, cr, ci);
                }
            }
            // back to the places this thread read, in reverse: no other thread
            // touches them in this round
#pragma unroll
            for (int i = GE - 1; i >= 0; --i) {
                *reinterpret_cast<float2 *>(sm + at) = v[i ^ (i >> 1)];
                if (i) at ^= so[__ffs(i) - 1];
            }
        }
    }
    __syncthreads();
    float2 *dst = psi + (threadIdx.x & LOWM);
    const uint32_t at = gphys(threadIdx.x);
#pragma unroll
    for (int i = 0; i < GE; ++i)
        dst[hioff[(threadIdx.x >> GATE_BLOCK_LOW) + (GT >> GATE_BLOCK_LOW) * i]] = amp[at ^ gphys(GT * i)];
}

// One barrier per gate, every thread on the pairs of each gate in the shared
// tile (gates_in_place says for which lists). Rows: opcodes and local qubits.
__global__ void __launch_bounds__(GT) gate_inplace_kernel(float2 *psi, const GateRow *gates, const float2 *mats,
                                                          const GateBlockParams p) {
    extern __shared__ __align__(16) float2 amp[];
    __shared__ unsigned long long hioff[1 << (GATE_BLOCK_Q - GATE_BLOCK_LOW)];
    // rows and matrices come through shared memory, GS gates at a time
    constexpr int GS = 64;
    __shared__ GateRow srow[GS];
    __shared__ __align__(16) float2 smat[16 * GS];
    const unsigned long long tile = blockIdx.x + ((unsigned long long)blockIdx.y << 15);
    if (tile >= (1ULL << p.n_other)) return;   // uniform over the CTA
    unsigned long long base = 0;
    for (int i = 0; i < p.n_other; ++i) base |= ((tile >> i) & 1ULL) << p.other[i];
    const int L = 1 << p.Q;
    const int low = p.Q < GATE_BLOCK_LOW ? p.Q : GATE_BLOCK_LOW, lm = (1 << low) - 1;
    for (int h = threadIdx.x; h < 1 << (p.Q - low); h += GT) {
        unsigned long long o = base;
        for (int i = low; i < p.Q; ++i) o |= (unsigned long long)((h >> (i - low)) & 1) << p.local[i];
        hioff[h] = o;
    }
    __syncthreads();
    for (int l = threadIdx.x; l < L; l += GT) amp[l] = psi[hioff[l >> low] | (unsigned long long)(l & lm)];
    const float r2 = 0.70710678118654752440f;
    for (int gi = 0; gi < p.ng; ++gi) {
        const int ci = gi & (GS - 1);
        if (ci == 0) {
            const int nc = p.ng - gi < GS ? p.ng - gi : GS;
            __syncthreads();
            for (int e = threadIdx.x; e < nc; e += GT) srow[e] = gates[p.g0 + gi + e];
            if (mats)
                for (int e = threadIdx.x; e < 16 * nc; e += GT) smat[e] = __ldg(mats + 16 * (size_t)(p.g0 + gi) + e);
        }
        __syncthreads();
        const GateRow G = srow[ci];
        const int b0 = 1 << G.q0;
        if (G.op == GATE_OP_U2) {   // 4x4 matrix, local index bit(q0) + 2 bit(q1)
            float2 m[16];
#pragma unroll
            for (int e = 0; e < 16; ++e) m[e] = smat[16 * ci + e];
            const int b1 = 1 << G.q1;
            const int lo = G.q0 < G.q1 ? G.q0 : G.q1, hi = G.q0 < G.q1 ? G.q1 : G.q0;
            for (int pi = threadIdx.x; pi < L / 4; pi += GT) {
                int i = ((pi >> lo) << (lo + 1)) | (pi & ((1 << lo) - 1));
                i = ((i >> hi) << (hi + 1)) | (i & ((1 << hi) - 1));
                const int idx[4] = {i, i | b0, i | b1, i | b0 | b1};
                float2 v[4];
#pragma unroll
                for (int l = 0; l < 4; ++l) v[l] = amp[idx[l]];
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    float re = 0.f, im = 0.f;
#pragma unroll
                    for (int l = 0; l < 4; ++l) {
                        re = fmaf(m[4 * r + l].x, v[l].x, fmaf(-m[4 * r + l].y, v[l].y, re));
                        im = fmaf(m[4 * r + l].x, v[l].y, fmaf(m[4 * r + l].y, v[l].x, im));
                    }
                    amp[idx[r]] = make_float2(re, im);
                }
            }
        } else if (G.op == 0) {   // H
            for (int pi = threadIdx.x; pi < L / 2; pi += GT) {
                const int i = ((pi >> G.q0) << (G.q0 + 1)) | (pi & (b0 - 1));
                const float2 u = amp[i], w = amp[i | b0];
                amp[i] = make_float2(r2 * (u.x + w.x), r2 * (u.y + w.y));
                amp[i | b0] = make_float2(r2 * (u.x - w.x), r2 * (u.y - w.y));
            }
        } else if (G.op == 3) {   // CNOT q0 -> q1
            const int b1 = 1 << G.q1;
            const int lo = G.q0 < G.q1 ? G.q0 : G.q1, hi = G.q0 < G.q1 ? G.q1 : G.q0;
            for (int pi = threadIdx.x; pi < L / 4; pi += GT) {
                int i = ((pi >> lo) << (lo + 1)) | (pi & ((1 << lo) - 1));
                i = ((i >> hi) << (hi + 1)) | (i & ((1 << hi) - 1));
                i |= b0;
                const float2 u = amp[i];
                amp[i] = amp[i | b1];
                amp[i | b1] = u;
            }
        } else {   // diagonal phase on |1> of q0
            float cr, ci;
            phase_of(G.op == 1 ? 2 : G.op == 2 ? 6 : G.op == 4 ? 1 : 7, cr, ci);
            for (int pi = threadIdx.x; pi < L / 2; pi += GT) {
                const int i = ((pi >> G.q0) << (G.q0 + 1)) | (pi & (b0 - 1)) | b0;
                const float2 u = amp[i];
                amp[i] = make_float2(cr * u.x - ci * u.y, cr * u.y + ci * u.x);
            }
        }
    }
    __syncthreads();
    for (int l = threadIdx.x; l < L; l += GT) psi[hioff[l >> low] | (unsigned long long)(l & lm)] = amp[l];
}

cudaError_t launch_gate_blocks(float2 *psi, int N, const GateRow *gates_dev, const GateRound *rounds_dev,
                               const float2 *mats_dev, const GateBlock *blocks, int n_blocks, cudaStream_t st) {
    int max_ng = 0;
    for (int b = 0; b < n_blocks; ++b) max_ng = blocks[b].ng > max_ng ? blocks[b].ng : max_ng;
    const size_t tile_max = sizeof(float2) << (N < GATE_BLOCK_Q ? N : GATE_BLOCK_Q);
    const size_t smem_max = rounds_dev && mats_dev ? tile_max + sizeof(float2) * 16 * (size_t)max_ng : tile_max;
    if (smem_max > 200 * 1024) return cudaErrorInvalidValue;
    static SmemOptIn optin[3];
    const int which = !rounds_dev ? 0 : mats_dev ? 1 : 2;
    const cudaError_t ea = optin[which].allow(which == 0 ? (const void *)gate_inplace_kernel
                                              : which == 1 ? (const void *)gate_block_kernel<true>
                                                           : (const void *)gate_block_kernel<false>, smem_max);
    if (ea != cudaSuccess) return ea;
    for (int b = 0; b < n_blocks; ++b) {
        GateBlockParams p;
        p.r0 = blocks[b].r0;
        p.nr = blocks[b].nr;
        p.g0 = blocks[b].g0;
        p.ng = blocks[b].ng;
        p.Q = 0;
        bool in[64] = {false};
        for (int i = 0; i < GATE_BLOCK_Q; ++i) {
            const unsigned char q = blocks[b].qubit[i];
            if (q == 255) break;
            p.local[p.Q++] = q;
            in[q] = true;
        }
        p.n_other = 0;
        for (int q = 0; q < N; ++q)
            if (!in[q]) p.other[p.n_other++] = (unsigned char)q;
        const unsigned long long tiles = 1ULL << p.n_other;
        const dim3 grid((unsigned)(tiles < 32768 ? tiles : 32768), (unsigned)(tiles < 32768 ? 1 : tiles >> 15));
        const size_t tile_bytes = sizeof(float2) << p.Q, mat_bytes = sizeof(float2) * 16 * (size_t)p.ng;
        if (!rounds_dev) gate_inplace_kernel<<<grid, GT, tile_bytes, st>>>(psi, gates_dev, mats_dev, p);
        else if (mats_dev) gate_block_kernel<true><<<grid, GT, tile_bytes + mat_bytes, st>>>(psi, gates_dev, rounds_dev, mats_dev, p);
        else gate_block_kernel<false><<<grid, GT, tile_bytes, st>>>(psi, gates_dev, rounds_dev, nullptr, p);
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

} // namespace sre
