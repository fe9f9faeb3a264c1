// Flooding-schedule decoding of small batches: one CTA per shot, several
// lanes per node.
//
// A batch that leaves SMs idle is bound by the latency of its slowest shot's
// iterations, i.e. by the instructions a warp issues one after the other
// between two barriers.  decode_kernel gives each thread one or two nodes with
// all their edges, about 270 instructions per node and iteration.  Here L lanes
// share a node (L = 4: one edge each; L = 2: two edges; L = 1: all four), so
// that a lane's chain holds the work of 4 / L edges: the check rule's partial
// products and the posterior's sums cross the lanes by shuffles, and the
// per-qubit values (posterior, decision, the four exponentials) are computed by
// every lane of the node.  Adjacency, prior and variant state stay in registers;
// shared memory holds the edge messages only.  Tables are read with plain loads
// and the shots are assigned to the CTAs statically, so a call is one launch:
// no queue to reset before it.  The host picks L (launch_small in decode.cu,
// with the measurements).  Calls back to back: one toric d = 15 EWAInit shot 13.1 us
// against 18.1 in the queue kernel, 152 planar d = 9 Momentum shots at p = 0.05 52
// against 64 there with one node per thread and 94 with two.
//
// Arithmetic and results are decode_shot's bit for bit (decode_kernel.cuh):
// every step is the same operation on the same operands, up to the order of the
// two operands of an addition.
#pragma once

#include <cuda_runtime.h>

#include "decode_kernel.cuh"

namespace bpq {
namespace dk {

// The value of the lane that holds the other pair of positions (0, 1 or 2, 3).
template <int L>
__device__ __forceinline__ float other_pair(float v) {
    return L == 1 ? v : __shfl_xor_sync(0xffffffffu, v, L / 2);
}

template <int VARIANT, int L>
__global__ void __launch_bounds__(1024, 1) decode_small_kernel(const DecodeArgs a, int runs, float clip) {
    constexpr bool PHI = PhiForm<VARIANT>::value;
    constexpr int E = 4 / L;  // edges per lane: positions E h .. E h + E - 1
    extern __shared__ __align__(16) uint8_t smem[];
    float *slots = reinterpret_cast<float *>(smem);  // slot p * n_pad + j: qubit j's p-th edge
    const int tid = threadIdx.x, x = tid / L, h = tid % L;
    const bool has_check = x < a.M, has_qubit = x < a.N;
    const int Np = a.n_pad, max_iter = a.max_iter;
    const float vclip = PHI ? a.phi_clip : a.delta_clip;
#ifdef BPQ_DEBUG
    // a lane for every node, slots for every qubit (the same for the whole CTA;
    // an early return happens before any barrier)
    if (16u * (uint32_t)Np > dynamic_smem_bytes() || Np < a.N || (a.M > a.N ? a.M : a.N) * L > (int)blockDim.x ||
        8u * (uint32_t)a.M > a.table_bytes || a.off_var_pauli + (uint32_t)a.N > a.table_bytes) {
        if (tid == 0) atomicExch(a.work + 1, kBoundsError);
        return;
    }
#endif

    // ---- the lane's edges of check x and positions of qubit x ----
    uint32_t slot[E];
    uint32_t used = 0;  // bit e: the lane's position e of the qubit holds an edge
    float Pi[3] = {0.f, 0.f, 0.f};
#pragma unroll
    for (int e = 0; e < E; ++e) slot[e] = kNoSlot;
    if (has_check) {
        const uint16_t *cs = reinterpret_cast<const uint16_t *>(a.table) + 4 * x + E * h;
#pragma unroll
        for (int e = 0; e < E; ++e) {
            slot[e] = __ldg(cs + e);
            // a slot index is an edge slot (< 4 n_pad) or no slot
            if (slot[e] != kNoSlot && !BPQ_IN_BOUNDS(slot[e], 4 * Np, a.work + 1)) slot[e] = kNoSlot;
        }
    }
    if (has_qubit) {
        const uint32_t vp = (uint32_t)__ldg(a.table + a.off_var_pauli + x) >> (2 * E * h);
#pragma unroll
        for (int e = 0; e < E; ++e) used |= ((vp >> (2 * e)) & 3u ? 1u : 0u) << e;
        prior_llr(a, x, Pi);
    }
    float *own = slots + (size_t)E * h * Np + x;
    // lanes 0 .. L/2 - 1 hold the X positions (0, 1), the others the Z
    // positions (2, 3); with L = 1 a lane holds both
    const bool zlane = L > 1 && h >= L / 2;
#ifndef BPQ_DEBUG
    if (blockIdx.x == 0 && tid < 2) a.work[tid] = 0u;  // no queue, no device-side error
#endif  // (reset by the host before a checked launch, whose CTAs may set it)

    // once: the grid is B.  (Without the loop statement the compiler's code is slower:
    // toric d = 3 AEWA, 4800 shots, 118 against 136 us; planar d = 4 Momentum,
    // 8000 shots, 90 against 105.)
    for (int shot = blockIdx.x; shot < a.B; shot += gridDim.x) {
        uint32_t sb = 0;  // the check's syndrome bit
        if (has_check) sb = (__ldg(a.syn + (size_t)shot * a.W + (x >> 5)) >> (x & 31)) & 1u;
        uint32_t d = 0;
        int conv = 0, iters = 0;
        for (int run = 0; run < runs && !conv; ++run) {
            // AEWA-BP (runs = 11): alpha = 1.0, 0.9, ..., 0.0, as decode_kernel
            const float alpha = runs > 1 ? (float)(10 - run) / 10.0f : a.alpha;
            const ShotParams sp = shot_params<PHI>(a, alpha);
            // s1: Q^(t-1), or EWAInit's next prior; s2: g, G, or EWAInit's alpha Pi^(0)
            float s1[3], s2[3];
#pragma unroll
            for (int w = 0; w < 3; ++w) {
                s1[w] = Pi[w];
                s2[w] = VARIANT == BPQ_EWAINIT ? alpha * Pi[w] : 0.f;
            }
            // v->c messages of the lane's positions from Q and the incoming
            // messages win; ab: whether the decision anticommutes with the X
            // (bit 0) and the Z positions (bit 1)
            auto emit = [&](const float (&Q)[3], const float (&win)[E], uint32_t ab) {
                const float c0 = fminf(0.f, fminf(Q[0], fminf(Q[1], Q[2])));
                const float e0 = ex2(c0);
                const float eX = ex2(__fsub_rn(c0, Q[0])), eY = ex2(__fsub_rn(c0, Q[1])), eZ = ex2(__fsub_rn(c0, Q[2]));
#pragma unroll
                for (int e = 0; e < E; ++e) {
                    const bool z = L == 1 ? e >= 2 : zlane;
                    const float C = __fadd_rn(e0, z ? eZ : eX), Ab = __fadd_rn(eY, z ? eX : eZ);
                    const float A = __fmul_rn(Ab, ex2(win[e]));
                    const uint32_t neg = __float_as_uint(__fsub_rn(C, A)) & 0x80000000u;
                    const float mn = fminf(C, A);
                    float dl;
                    if (PHI)
                        dl = log1p_rel(__fmul_rn(__fmul_rn(2.0f, mn), rcp(__fsub_rn(fmaxf(C, A), mn))));
                    else
                        dl = __fmul_rn(__fadd_rn(mn, mn), rcp(__fadd_rn(C, A)));
                    const uint32_t bits = (__float_as_uint(fmaxf(dl, vclip)) & ~1u) | (z ? ab >> 1 : ab & 1u) | neg;
                    // unused positions hold 0
                    if (has_qubit) own[e * Np] = (used >> e) & 1u ? __uint_as_float(bits) : 0.f;
                }
            };
            const float none[E] = {};
            emit(Pi, none, 0u);  // eq. (init)
            __syncthreads();
            conv = 0;
            for (int t = 1;; ++t) {
                // ---- check pass: syndrome test of the previous decision, then eq. (h_update) ----
                uint32_t u[E], ux = 0;
                float mag[E];
#pragma unroll
                for (int e = 0; e < E; ++e) {
                    u[e] = slot[e] != kNoSlot ? __float_as_uint(slots[slot[e]]) : 0u;
                    mag[e] = __uint_as_float(u[e] & 0x7FFFFFFEu);
                    ux ^= u[e];
                }
                if (L == 4) ux ^= __shfl_xor_sync(0xffffffffu, ux, 1);
                if (L >= 2) ux ^= __shfl_xor_sync(0xffffffffu, ux, L / 2);
                ux ^= sb | (sb << 31);
                // partner: the magnitude of the other edge of the same pair;
                // opp: the pair product (sum) of the other pair
                const float mate = L == 4 ? __shfl_xor_sync(0xffffffffu, mag[0], 1) : 0.f;
                float ext[E];
                if (L == 1) {
                    const float d01 = PHI ? __fadd_rn(mag[0], mag[1 % E]) : oplus(mag[0], mag[1 % E]);
                    const float d23 = PHI ? __fadd_rn(mag[2 % E], mag[3 % E]) : oplus(mag[2 % E], mag[3 % E]);
#pragma unroll
                    for (int e = 0; e < E; ++e)
                        ext[e] = PHI ? __fadd_rn(mag[(e ^ 1) % E], e < 2 ? d23 : d01)
                                     : oplus(mag[(e ^ 1) % E], e < 2 ? d23 : d01);
                } else {
                    const float m1 = L == 4 ? mate : mag[1 % E];
                    const float opp = other_pair<L>(PHI ? __fadd_rn(mag[0], m1) : oplus(mag[0], m1));
#pragma unroll
                    for (int e = 0; e < E; ++e) {
                        const float m = L == 4 ? mate : mag[(e ^ 1) % E];
                        ext[e] = PHI ? __fadd_rn(m, opp) : oplus(m, opp);
                    }
                }
                // (a slot is read and written by the same lane)
#pragma unroll
                for (int e = 0; e < E; ++e) {
                    const float w = fminf(PHI ? phi_check(ext[e]) : c2v_magnitude(ext[e]), clip);
                    if (slot[e] != kNoSlot)
                        slots[slot[e]] = __uint_as_float(__float_as_uint(w) ^ ((ux ^ u[e]) & 0x80000000u));
                }
                const int any = __syncthreads_or((int)(ux & 1u) & (int)(has_check && t > 1));
                if (t > 1 && !any) {
                    conv = 1;
                    iters = t - 1;
                    break;
                }
                if (t > max_iter) {
                    iters = max_iter;
                    break;
                }
                // ---- variable pass: posterior of the variant, decision, eq. (v_update)/(mombp5) ----
                float win[E];
#pragma unroll
                for (int e = 0; e < E; ++e) win[e] = has_qubit ? own[e * Np] : 0.f;
                float S[3];
                if (L == 1) {
                    S[2] = __fadd_rn(win[0], win[1 % E]);
                    S[0] = __fadd_rn(win[2 % E], win[3 % E]);
                } else {
                    const float s = __fadd_rn(win[0], L == 4 ? __shfl_xor_sync(0xffffffffu, win[0], 1) : win[1 % E]);
                    const float o = other_pair<L>(s);
                    S[2] = zlane ? o : s;
                    S[0] = zlane ? s : o;
                }
                S[1] = __fadd_rn(S[0], S[2]);
                float Q[3];
#pragma unroll
                for (int w = 0; w < 3; ++w) {
                    if (VARIANT == BPQ_PLAIN) {
                        Q[w] = __fadd_rn(Pi[w], S[w]);
                    } else if (VARIANT == BPQ_EWAINIT) {
                        Q[w] = __fadd_rn(s1[w], S[w]);
                        s1[w] = __fmaf_rn(1.f - alpha, Q[w], s2[w]);
                    } else if (VARIANT == BPQ_MOMENTUM) {
                        s2[w] = momentum_g(sp, s1[w], Pi[w], S[w], s2[w]);
                        Q[w] = s1[w] = momentum_q(sp, s1[w], s2[w]);
                    } else {
                        const float gp = adagrad_gp(s1[w], Pi[w], S[w]);
                        s2[w] = adagrad_G(s2[w], gp, t >= 2 || sp.ada_from1);
                        Q[w] = s1[w] = t == 1 ? __fadd_rn(Pi[w], S[w]) : adagrad_q(sp, s1[w], gp, s2[w]);
                    }
                }
                const float mq = fminf(Q[0], fminf(Q[1], Q[2]));
                d = mq > 0.f ? 0u : Q[0] == mq ? 1u : Q[1] == mq ? 2u : 3u;
                emit(Q, win, anti_bits_split(d));
                __syncthreads();
            }
        }
        if (has_qubit && h == 0 && BPQ_IN_BOUNDS((size_t)shot * a.N + x, (size_t)a.B * a.N, a.work + 1))
            a.est[(size_t)shot * a.N + x] = (uint8_t)d;
        if (tid == 0 && BPQ_IN_BOUNDS(shot, a.B, a.work + 1)) {
            a.conv[shot] = (uint8_t)conv;
            a.iters[shot] = (uint8_t)iters;
        }
    }
}

}  // namespace dk

}  // namespace bpq
