// Differentiable unrolled decoders (bpq_train_*): a fixed number T of
// flooding iterations without the stopping rule, with per-iteration
// trainable parameters, in two models:
//
//   EWAInit (Sec. III-B, Algorithm 2), EWA weight alpha_t:
//     Pi^(t)     = alpha_t Pi^(0) + (1 - alpha_t) Q^(t-1)              (t > 1)
//     Q^(t)      = Pi^(t) + S^(t)
//   Momentum (Sec. III-A1, eqs. (mombp1)-(mombp3)), step alpha_t, rate gamma_t:
//     g^(t)      = gamma_t g^(t-1) + (1 - gamma_t) (Q^(t-1) - Pi^(0) - S^(t))
//     Q^(t)      = Q^(t-1) - alpha_t g^(t),          Q^(0) = Pi^(0), g^(0) = 0
//
// and, in both, per-iteration damping beta_t of the variable-to-check
// messages and a weight w_e on every check-to-variable message (neural-BP
// style; the paper's conclusion names neural BP as a direction):
//
//   m_c->v^(t)  = clip(w_e (-1)^{s_i} r_e),  r_e = 2 atanh prod_{f != e} tanh(m_v->c^(t-1)_f / 2)
//   S^(t)       = sum of anticommuting m_c->v^(t)
//   m_v->c^(t)  = (1 - beta_t) clip(lambda_H(Q^(t) - own message)) + beta_t m_v->c^(t-1)
//
// Two losses:
//   posterior:  mean over shots and qubits of -log softmax(0, -Q_X, -Q_Y, -Q_Z)[true Pauli]
//               of the final posterior Q^(T);
//   coset:      mean over shots and iterations t = 1..T of
//                 mean over checks i of -log P_t(<E^, H_i> = s_i)
//               + mean over logical operators L of -log P_t(<E^, L> = <E, L>),
//               where E^ is drawn from the product of the posterior marginals
//               of iteration t (pi_W proportional to e^{-Q_W}, Q_I = 0) and E is
//               the true error: the probability that the soft decision of every
//               iteration satisfies the syndrome and lies in the true error's
//               coset (neural-BP decoders for quantum codes train on this kind
//               of loss).  The parity distribution of a check or logical is the
//               (P(even), P(odd)) convolution over its qubits of each qubit's
//               (commute, anticommute) probabilities, sums of positive terms, so
//               small probabilities keep their relative accuracy.
//
// At constant alpha (and gamma), beta_t = 0, w_e = 1 the forward pass is
// EWAInit-BP (Momentum-BP).  One CTA decodes one shot (thread x owns check
// x and qubit x).  The forward kernel stores a checkpoint (m_v->c, Q, and g
// for Momentum) every K iterations; the backward kernel recomputes each
// K-iteration segment from its checkpoint into shared memory and runs the
// adjoint through it in reverse.  Both run the same step functions, so the
// recomputation reproduces the forward pass exactly.  Per-shot gradient rows
// are reduced over shots by a separate kernel, so results are deterministic.
// Arithmetic is fp32 with accurate library functions; divisions are approximate
// (2 ulp, see hfun).
//
// The kernels are bound by instructions (the library functions' sequences), so
// the formulas are arranged to call them as rarely as the mathematics allows,
// without losing relative accuracy at either end of the messages' range:
//  * check node: with q_f = 2 / expm1(|m_f|), e^phi(|m_f|) = 1 + q_f, so the
//    sum of phi's over the other edges is ln(1 + E_n), E_n the q_f combined by
//    a [+] b = a + b + ab (positive terms only), and |r_n| = phi of that sum =
//    log1p(2 / E_n): one expm1 and one log1p per edge.
//  * its derivative: d r_n / d m_f = sinh(r_n) / sinh(m_f) (from 1 - tanh^2 =
//    1 / cosh^2; it avoids the 1 / (1 - P^2) of the product form), which with
//    sinh(ln(1 + y)) = y (y + 2) / (2 (y + 1)) and sinh(x) sinh(phi(x)) = 1 is
//    h(q_f) / h(E_n), h(y) = y (y + 2) / (y + 1): no hyperbolic function.
//  * variable node: the own message cancels out of every ratio but one,
//    lambda_H(Q - own) = Lambda_H - m_own, Lambda_H = ln(1 + e^{-Q_H}) -
//    ln(e^{-Q_a} + e^{-Q_b}), which the edges of one Pauli type share, and the
//    derivatives with respect to Q are those of Lambda_H, with respect to the
//    own message -1.
//  * coset loss: a qubit's (commute, anticommute) probabilities depend on the
//    Pauli only, and their derivatives are products of probabilities (no
//    difference of a probability and 1).
// Training step (Momentum, coset loss, planar d = 9, T = 25, 4096 shots), with
// phi, its inverse, lambda and their derivatives evaluated per edge: 932 us
// forward, 3590 us backward, gradients 1.4e-6 off float64; so arranged: 652 us,
// 2018 us, 1.8e-7; with adjacency in registers and approximate divisions 635 us,
// 1604 us, 2.9e-7.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>

#include "bpq_internal.h"
#include "decode_launch.h"

using bpq::fail;

namespace bpq {
namespace tr {

constexpr int kEWAInit = BPQ_TRAIN_EWAINIT, kMomentum = BPQ_TRAIN_MOMENTUM;
constexpr int kCoset = BPQ_TRAIN_LOSS_COSET;
constexpr int kMaxLogicals = 4;
constexpr float kMinProb = 1e-30f;  // -log P is taken of max(P, kMinProb); no gradient below

struct TrainArgs {
    const uint8_t *table;
    uint32_t off_var_pauli;
    const int32_t *chk_ptr;
    const uint32_t *syn;
    const uint8_t *err;
    const float *prior, *alpha, *beta, *w, *gamma;
    int N, M, E, W, B, T, K, nck, n_pad;
    int ck_floats;     // floats per checkpoint: 7 n_pad (EWAInit) or 10 n_pad (Momentum)
    int width;         // floats per gradient row: 2T + E (+ T for Momentum)
    float clip;
    int loss_kind;     // BPQ_TRAIN_LOSS_POSTERIOR or BPQ_TRAIN_LOSS_COSET
    const uint8_t *logicals;  // coset loss: [n_log][N] Pauli codes
    int n_log;
    float *ckpt;       // [B][nck][ck_floats]: m_v->c (4 n_pad slots), Q (3 n_pad), g (3 n_pad)
    float *loss_shot;  // [B] sum over qubits of the cross-entropy
    float *Q_out;      // optional [B][N][3]
    float *rows;       // [B][width] per-shot gradients: alpha | beta | w | gamma
};

__device__ __forceinline__ uint32_t anti(uint32_t a, uint32_t b) { return (a != 0u) & (b != 0u) & (a != b); }

// ---------------------------------------------------------------- steps shared by both kernels

// The thread's check and qubit.
struct Adj {
    uint32_t sl[4];   // message slots of the owned check's edges (kNoSlot: none)
    uint32_t vp;      // qubit Paulis, 2 bits per slot 4 x + k (0: unused)
    int ce;           // canonical index of the check's first edge
    float sigma;      // (-1)^{s_i}
    float ws[4];      // w_e (-1)^{s_i} of the owned check's edges
    uint32_t logp;    // Pauli of logical operator l on the qubit in bits 2l, 2l + 1 (coset loss)
};

__device__ __forceinline__ Adj load_adj(const TrainArgs &a, int x, int shot) {
    Adj d;
    d.vp = d.logp = 0;
    d.ce = 0;
    d.sigma = 1.f;
#pragma unroll
    for (int n = 0; n < 4; ++n) {
        d.sl[n] = kNoSlot;
        d.ws[n] = 0.f;
    }
    if (x < a.M) {
        const uint2 s = reinterpret_cast<const uint2 *>(a.table)[x];
        d.sl[0] = s.x & 0xFFFFu;
        d.sl[1] = s.x >> 16;
        d.sl[2] = s.y & 0xFFFFu;
        d.sl[3] = s.y >> 16;
        d.ce = a.chk_ptr[x];
        if ((a.syn[(size_t)shot * a.W + (x >> 5)] >> (x & 31)) & 1u) d.sigma = -1.f;
#pragma unroll
        for (int n = 0; n < 4; ++n)
            if (d.sl[n] != kNoSlot) d.ws[n] = a.w[d.ce + n] * d.sigma;
    }
    if (x < a.N) {
        d.vp = a.table[a.off_var_pauli + x];
        for (int l = 0; l < a.n_log; ++l) d.logp |= (a.logicals[(size_t)l * a.N + x] & 3u) << (2 * l);
    }
    return d;
}

__device__ __forceinline__ uint32_t slot_pauli(uint32_t vp, int k) { return (vp >> (2 * k)) & 3u; }

// Prior LLRs Pi^(0) of qubit x.
__device__ __forceinline__ void prior_llr(const TrainArgs &a, int x, float (&P)[3]) {
    const float px = a.prior[3 * x], py = a.prior[3 * x + 1], pz = a.prior[3 * x + 2];
    const float pI = 1.f - px - py - pz;
    P[0] = logf(pI / px);
    P[1] = logf(pI / py);
    P[2] = logf(pI / pz);
}

// a [+] b = (1 + a)(1 + b) - 1.
__device__ __forceinline__ float boxsum(float a, float b) { return __fmaf_rn(a, b, __fadd_rn(a, b)); }
// Divisions: __fdividef is within 2 ulp and a fifth of the instructions of the
// rounded one, for denominators of at most 2^126 (above, it gives 0).  expm1 of a
// message is the one denominator that can be larger (messages above 87.3, with a
// msg_clip that allows them); it goes in as its quarter.
// h(y) = y (y + 2) / (y + 1).
__device__ __forceinline__ float hfun(float y) { return __fmul_rn(y, __fadd_rn(1.f, __fdividef(1.f, __fadd_rn(y, 1.f)))); }

// Check node of the owned check from m_v->c in v: q_f of each edge, E_n, the
// signs (bit n: m_n < 0), r_n = 2 atanh prod_{f != n} tanh(m_f / 2), and the
// messages m_c->v = clip(w_e (-1)^{s_i} r_n).  q is at most 1e12 (messages
// below 2e-12), so that no product overflows.
struct CheckNode {
    float q[4], E[4], r[4], out[4];
    uint32_t neg;
};

__device__ __forceinline__ void check_node(const TrainArgs &a, const Adj &d, const float *v, CheckNode &c) {
    c.neg = 0;
#pragma unroll
    for (int n = 0; n < 4; ++n) {
        c.q[n] = 0.f;
        if (d.sl[n] != kNoSlot) {
            const float m = v[d.sl[n]];
            c.q[n] = fminf(__fdividef(0.5f, 0.25f * expm1f(fabsf(m))), 1e12f);
            c.neg |= (m < 0.f ? 1u : 0u) << n;
        }
    }
    const float d01 = boxsum(c.q[0], c.q[1]), d23 = boxsum(c.q[2], c.q[3]);
    c.E[0] = boxsum(c.q[1], d23);
    c.E[1] = boxsum(c.q[0], d23);
    c.E[2] = boxsum(c.q[3], d01);
    c.E[3] = boxsum(c.q[2], d01);
    const uint32_t odd = __popc(c.neg) & 1u;
#pragma unroll
    for (int n = 0; n < 4; ++n) {
        const float mag = log1pf(__fdividef(2.0f, c.E[n]));
        c.r[n] = ((c.neg >> n) & 1u) != odd ? -mag : mag;
        c.out[n] = 0.f;
        if (d.sl[n] != kNoSlot)
            c.out[n] = fminf(fmaxf(__fmul_rn(d.ws[n], c.r[n]), -a.clip), a.clip);
    }
}

// Lambda_H of one Pauli type H with the other two a, b.  Prior probabilities of
// 0 make Q infinite: with Qa = Qb = inf (noise of one Pauli only) the ratio has no
// denominator and Lambda_H is inf; the minimum turns the NaN of inf - inf into 0.
__device__ __forceinline__ float lambda_type(float QH, float Qa, float Qb) {
    const float lc = __fadd_rn(fmaxf(0.f, -QH), log1pf(expf(-fabsf(QH))));
    const float la = __fadd_rn(fmaxf(-Qa, -Qb), log1pf(expf(fminf(-fabsf(__fsub_rn(Qa, Qb)), 0.f))));
    return __fsub_rn(lc, la);
}

// Lambda of the types X, Y, Z that the qubit's edges have.
__device__ __forceinline__ void lambda_types(uint32_t vp, const float (&Q)[3], float (&L)[3]) {
    const uint32_t lo = vp & 0x55u, hi = (vp >> 1) & 0x55u;
    L[0] = (lo & ~hi) ? lambda_type(Q[0], Q[1], Q[2]) : 0.f;
    L[1] = (hi & ~lo) ? lambda_type(Q[1], Q[0], Q[2]) : 0.f;
    L[2] = (lo & hi) ? lambda_type(Q[2], Q[0], Q[1]) : 0.f;
}
__device__ __forceinline__ float pick3(const float (&v)[3], uint32_t p) { return p == 1u ? v[0] : p == 2u ? v[1] : v[2]; }

__device__ __forceinline__ float clipped(const TrainArgs &a, float x) { return fminf(fmaxf(x, -a.clip), a.clip); }

// S_W: the sum of the qubit's incoming messages that anticommute with W.
__device__ __forceinline__ void incoming_sums(uint32_t vp, const float (&cin)[4], float (&S)[3]) {
    S[0] = S[1] = S[2] = 0.f;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const uint32_t p = slot_pauli(vp, k);
#pragma unroll
        for (int w = 0; w < 3; ++w) S[w] = __fadd_rn(S[w], anti(w + 1, p) ? cin[k] : 0.f);
    }
}

// Variable node of iteration t: the posterior Q (from Q^(t-1); g for
// Momentum) and the outgoing messages v (from m_v->c^(t-1)), both updated in
// place, from the incoming messages cin (0 where unused).
template <int MODEL>
__device__ __forceinline__ void variable_node(const TrainArgs &a, uint32_t vp, const float (&Pi0)[3],
                                              const float (&cin)[4], int t, float (&Q)[3], float (&g)[3], float (&v)[4]) {
    const float al = a.alpha[t - 1], be = a.beta[t - 1];
    float S[3], L[3];
    incoming_sums(vp, cin, S);
#pragma unroll
    for (int w = 0; w < 3; ++w) {
        if (MODEL == kMomentum) {
            const float gm = a.gamma[t - 1], D = __fsub_rn(__fsub_rn(Q[w], Pi0[w]), S[w]);
            g[w] = __fmaf_rn(gm, g[w], __fmul_rn(__fsub_rn(1.f, gm), D));
            Q[w] = __fmaf_rn(-al, g[w], Q[w]);
        } else {
            const float pit = t > 1 ? __fmaf_rn(al, Pi0[w], __fmul_rn(__fsub_rn(1.f, al), Q[w])) : Pi0[w];
            Q[w] = __fadd_rn(pit, S[w]);
        }
    }
    lambda_types(vp, Q, L);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const uint32_t p = slot_pauli(vp, k);
        const float m = clipped(a, __fsub_rn(pick3(L, p), cin[k]));
        v[k] = p ? __fmaf_rn(be, v[k], __fmul_rn(__fsub_rn(1.f, be), m)) : 0.f;
    }
}

// Eq. (init): lambda(Pi^(0)) on the qubit's edges.
__device__ __forceinline__ void initial_messages(const TrainArgs &a, uint32_t vp, const float (&Pi0)[3], float (&v)[4]) {
    float L[3];
    lambda_types(vp, Pi0, L);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const uint32_t p = slot_pauli(vp, k);
        v[k] = p ? clipped(a, pick3(L, p)) : 0.f;
    }
}

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

__device__ __forceinline__ float4 load4(const float *p) { return *reinterpret_cast<const float4 *>(p); }
__device__ __forceinline__ void get4(const float *p, float (&v)[4]) {
    const float4 q = load4(p);
    v[0] = q.x, v[1] = q.y, v[2] = q.z, v[3] = q.w;
}
__device__ __forceinline__ void put4(float *p, const float (&v)[4]) {
    *reinterpret_cast<float4 *>(p) = make_float4(v[0], v[1], v[2], v[3]);
}

// ---------------------------------------------------------------- coset loss

// Parity distribution (P(even), P(odd)) of the sum of two independent bits
// with distributions x and y.
__device__ __forceinline__ float2 parity_combine(float2 x, float2 y) {
    return make_float2(x.x * y.x + x.y * y.y, x.x * y.y + x.y * y.x);
}

// Posterior marginals (pi_I, pi_X, pi_Y, pi_Z) of a qubit: pi_W proportional
// to e^{-Q_W}, Q_I = 0.
__device__ __forceinline__ void marginals(const float (&Q)[3], float (&pi)[4]) {
    const float c0 = fminf(0.f, fminf(Q[0], fminf(Q[1], Q[2])));
    const float e[4] = {expf(c0), expf(c0 - Q[0]), expf(c0 - Q[1]), expf(c0 - Q[2])};
    const float z = __fdividef(1.f, e[0] + e[1] + e[2] + e[3]);
#pragma unroll
    for (int k = 0; k < 4; ++k) pi[k] = e[k] * z;
}

// (P(the qubit's error commutes with P), P(it anticommutes)); (1, 0) for P = I.
__device__ __forceinline__ float2 comm_anti(const float (&pi)[4], uint32_t P) {
    const float pX = pi[1], pY = pi[2], pZ = pi[3];
    return P == 0u   ? make_float2(1.f, 0.f)
           : P == 1u ? make_float2(pi[0] + pX, pY + pZ)
           : P == 2u ? make_float2(pi[0] + pY, pX + pZ)
                     : make_float2(pi[0] + pZ, pX + pY);
}

// What the logical operators need from one warp: the parity distribution over
// its qubits and, for the gradient, sum ln |c - a| and the number of negative
// c - a.  A chunk of operators is gathered per barrier: as many as 32 float4 hold
// for the CTA's warps.
__host__ __device__ inline int logical_chunk(int n_log, int warps) { return n_log * warps <= 32 ? n_log : 32 / warps; }

template <bool GRAD>
__device__ __forceinline__ float4 logical_partial(float2 ca, bool has) {
    float4 r = make_float4(1.f, 0.f, 0.f, 0.f);
    if (!__any_sync(0xffffffffu, has)) return r;
    float2 eo = has ? ca : make_float2(1.f, 0.f);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
        eo = parity_combine(eo, make_float2(__shfl_xor_sync(0xffffffffu, eo.x, o), __shfl_xor_sync(0xffffffffu, eo.y, o)));
    r.x = eo.x;
    r.y = eo.y;
    if (GRAD) {
        const float u = ca.x - ca.y;
        r.z = warp_sum(has ? logf(fmaxf(fabsf(u), 1e-30f)) : 0.f);
        r.w = (float)__popc(__ballot_sync(0xffffffffu, has && u < 0.f));
    }
    return r;
}

// The CTA's total for operator i of a chunk of n (after a barrier).
template <bool GRAD>
__device__ __forceinline__ float4 logical_total(const float4 *part, int i, int n, int warps) {
    float4 t = make_float4(1.f, 0.f, 0.f, 0.f);
    for (int k = 0; k < warps; ++k) {
        const float4 p = part[k * n + i];
        const float2 eo = parity_combine(make_float2(t.x, t.y), make_float2(p.x, p.y));
        t.x = eo.x;
        t.y = eo.y;
        if (GRAD) {
            t.z += p.z;
            t.w += p.w;
        }
    }
    return t;
}

// Pauli of logical operator l on the thread's qubit.
__device__ __forceinline__ uint32_t logical_pauli(const Adj &d, int l) { return (d.logp >> (2 * l)) & 3u; }

// Parities <E, L> of the true error with the logical operators (bit l), the
// same on every thread.
__device__ __forceinline__ uint32_t true_logical_parities(const TrainArgs &a, const Adj &d, int x, int shot) {
    uint32_t tau = 0;
    const uint32_t e = x < a.N ? a.err[(size_t)shot * a.N + x] : 0u;
    for (int l = 0; l < a.n_log; ++l)
        tau |= (uint32_t)(__syncthreads_count((int)anti(e, logical_pauli(d, l))) & 1) << l;
    return tau;
}

// -log P of one side of a parity distribution; the likely side's from the other,
// so that a small loss keeps its relative accuracy.
__device__ __forceinline__ float neg_log(float P, float other) {
    return P > other ? -log1pf(-other) : -logf(fmaxf(P, kMinProb));
}

// Forward: one CTA per shot.  Per iteration two barriers: the check threads
// (which also take the coset loss's check terms of the previous iteration), the
// qubit threads.  The messages of an edge share a slot (m_v->c is replaced by
// m_c->v and back); the qubit's own copies, Q and g stay in registers.
template <int MODEL, bool COSET>
__global__ void __launch_bounds__(1024, 1) train_forward_kernel(const TrainArgs a) {
    extern __shared__ __align__(16) float sm[];
    const int Np = a.n_pad;
    float *msg = sm;                                                   // [4 Np]
    float2 *ub = reinterpret_cast<float2 *>(sm + 4 * Np);              // [4 Np] edge parity distributions (coset)
    float4 *part = reinterpret_cast<float4 *>(sm + 12 * Np);           // [chunk][warps] (coset)
    __shared__ float red[32];
    const int x = threadIdx.x, shot = blockIdx.x, warp = x >> 5, warps = blockDim.x >> 5;
    const Adj d = load_adj(a, x, shot);
    const uint32_t tau = COSET ? true_logical_parities(a, d, x, shot) : 0u;
    const bool qubit = x < a.N, check = x < a.M;
    float Pi0[3] = {0.f, 0.f, 0.f}, Q[3] = {0.f, 0.f, 0.f}, g[3] = {0.f, 0.f, 0.f}, v[4] = {0.f, 0.f, 0.f, 0.f};
    if (qubit) {
        prior_llr(a, x, Pi0);
#pragma unroll
        for (int w = 0; w < 3; ++w) Q[w] = Pi0[w];
        initial_messages(a, d.vp, Pi0, v);
        put4(msg + 4 * x, v);
    }
    const int chunk = logical_chunk(a.n_log, warps);
    float loss = 0.f, loss_log = 0.f;
    // the coset loss's check terms of the iteration whose ub is complete
    auto check_terms = [&]() {
        if (!check) return;
        float2 eo = make_float2(1.f, 0.f);
#pragma unroll
        for (int n = 0; n < 4; ++n)
            if (d.sl[n] != kNoSlot) eo = parity_combine(eo, ub[d.sl[n]]);
        loss += d.sigma < 0.f ? neg_log(eo.y, eo.x) : neg_log(eo.x, eo.y);
    };
    auto logical_terms = [&](int l0, int n) {
        if (x < n) {
            const float4 t = logical_total<false>(part, x, n, warps);
            loss_log += ((tau >> (l0 + x)) & 1u) ? neg_log(t.y, t.x) : neg_log(t.x, t.y);
        }
    };
    __syncthreads();
    float *ck = a.ckpt + (size_t)shot * a.nck * a.ck_floats;
    for (int t = 1; t <= a.T; ++t) {
        if ((t - 1) % a.K == 0 && qubit) {  // checkpoint (m_v->c^(t-1), Q^(t-1), g^(t-1))
            float *c = ck + (size_t)((t - 1) / a.K) * a.ck_floats;
            put4(c + 4 * x, v);
#pragma unroll
            for (int w = 0; w < 3; ++w) {
                c[(4 + w) * Np + x] = Q[w];
                if (MODEL == kMomentum) c[(7 + w) * Np + x] = g[w];
            }
        }
        if (check) {
            CheckNode c;
            check_node(a, d, msg, c);
#pragma unroll
            for (int n = 0; n < 4; ++n)
                if (d.sl[n] != kNoSlot) msg[d.sl[n]] = c.out[n];
        }
        if (COSET && t > 1) {
            check_terms();
            logical_terms(a.n_log - ((a.n_log - 1) % chunk + 1), (a.n_log - 1) % chunk + 1);
        }
        __syncthreads();
        float pi[4] = {1.f, 0.f, 0.f, 0.f};
        if (qubit) {
            float cin[4];
            get4(msg + 4 * x, cin);
#pragma unroll
            for (int k = 0; k < 4; ++k)
                if (!slot_pauli(d.vp, k)) cin[k] = 0.f;
            variable_node<MODEL>(a, d.vp, Pi0, cin, t, Q, g, v);
            put4(msg + 4 * x, v);
            if (COSET) {
                marginals(Q, pi);
#pragma unroll
                for (int k = 0; k < 4; ++k) ub[4 * x + k] = comm_anti(pi, slot_pauli(d.vp, k));
            }
        }
        if (COSET) {
            // the last chunk of operators waits for the barrier below, earlier
            // ones (many warps) have barriers of their own
            for (int l0 = 0; l0 < a.n_log; l0 += chunk) {
                const int n = min(chunk, a.n_log - l0);
                for (int i = 0; i < n; ++i) {
                    const uint32_t P = logical_pauli(d, l0 + i);
                    const float4 r = logical_partial<false>(comm_anti(pi, P), P != 0u);
                    if ((x & 31) == 0) part[warp * n + i] = r;
                }
                if (l0 + chunk < a.n_log) {
                    __syncthreads();
                    logical_terms(l0, n);
                    __syncthreads();
                }
            }
        }
        __syncthreads();
    }
    if (COSET) {
        check_terms();
        logical_terms(a.n_log - ((a.n_log - 1) % chunk + 1), (a.n_log - 1) % chunk + 1);
        // (a code without checks has no check terms)
        loss = ((a.M ? loss / (float)a.M : 0.f) + loss_log / (float)a.n_log) / (float)a.T;
    } else if (qubit) {
        // cross-entropy of the final posterior against the true error; the
        // largest term enters through log1p, so that a small loss keeps its
        // relative accuracy
        const float z[4] = {0.f, -Q[0], -Q[1], -Q[2]};
        int top = 0;
        float zm = z[0];
#pragma unroll
        for (int k = 1; k < 4; ++k)
            if (z[k] > zm) {
                zm = z[k];
                top = k;
            }
        float rest = 0.f;
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (k != top) rest += expf(z[k] - zm);
        const int e = a.err[(size_t)shot * a.N + x];
        loss = (e == 0 ? zm : zm + Q[e == 1 ? 0 : e == 2 ? 1 : 2]) + log1pf(rest);
    }
    if (qubit && a.Q_out)
        for (int w = 0; w < 3; ++w) a.Q_out[((size_t)shot * a.N + x) * 3 + w] = Q[w];
    loss = warp_sum(loss);
    if ((x & 31) == 0) red[warp] = loss;
    __syncthreads();
    if (warp == 0) {
        const float tot = warp_sum(x < warps ? red[x] : 0.f);
        if (x == 0) a.loss_shot[shot] = tot;
    }
}

// Shared memory of the backward kernel, in floats.
inline size_t backward_floats(int Np, int K, bool momentum, int n_log, int warps) {
    // m_v->c history | m_c->v | its adjoint | adjoint of m_v->c | edge
    // parities' second half | Q (and g) history | logical partials | warp sums
    return (size_t)4 * Np * (K + 1 + 4) + (size_t)3 * Np * (K + 1) * (momentum ? 2 : 1) +
           (size_t)(4 * logical_chunk(n_log, warps) + 3) * warps;
}

// Backward: one CTA per shot; segments of K iterations recomputed from the
// checkpoints into shared memory, adjoint in reverse.  An adjoint iteration t
// has three steps, a barrier after each:
//   1. check threads: the check-node derivative of iteration t + 1 (step B) and
//      the check node of iteration t (its m_c->v, and q, E, r kept in registers
//      for step B); qubit threads: iteration t's edge parities (coset);
//   2. check threads: the coset loss's gradient with respect to the edge
//      parities (coset only);
//   3. qubit threads: the coset gradient with respect to Q^(t), then damping,
//      lambda, posterior and prior (step A).
// With P_match = (1 + sigma prod_j u_j) / 2 (u_j = c_j - a_j, sigma = +-1 the
// target parity), d (-log P_match) / d u_j = -sigma U'_j / (2 P_match), U'_j
// the product over the other qubits, and d u_j / d Q_W = 2 pi_W (c_j -
// [W commutes with the operator's Pauli on j]), i.e. 2 pi_W c_j where W
// anticommutes and -2 pi_W a_j where it commutes.
// SMALL: CTAs of at most 320 threads take up to 96 registers a thread (20 warps
// per SM): planar d = 9, whose shared memory holds five CTAs of five warps, runs
// 1731 us with five and 72 registers, 1639 us with four and 80.
template <int MODEL, bool COSET, bool SMALL>
__global__ void __launch_bounds__(SMALL ? 320 : 1024, SMALL ? 2 : 1) train_backward_kernel(const TrainArgs a) {
    extern __shared__ __align__(16) float sm[];
    const int Np = a.n_pad, K = a.K, S4 = 4 * Np;
    float *vh = sm;                               // [K+1][S4]  m_v->c^(t0 .. t0+K)
    // edge parities, [S4] float2: over m_v->c^(t0+K), which the adjoint never
    // reads, and the S4 floats after it
    float2 *ub = reinterpret_cast<float2 *>(vh + (size_t)K * S4);
    float *cm = vh + (size_t)(K + 2) * S4;        // [S4] m_c->v^(t)
    float *cbar = cm + S4;                        // [S4] adjoint of m_c->v^(t)
    float *vbar = cbar + S4;                      // [S4] adjoint of m_v->c^(t)
    float *Qh = vbar + S4;                        // [K+1][3Np]  Q^(t0 .. t0+K)
    float *gh = Qh + (size_t)(K + 1) * 3 * Np;    // [K+1][3Np]  g^(t0 .. t0+K) (Momentum only)
    float4 *part = reinterpret_cast<float4 *>(gh + (MODEL == kMomentum ? (size_t)(K + 1) * 3 * Np : 0));
    float *red = reinterpret_cast<float *>(part + logical_chunk(a.n_log, blockDim.x >> 5) * (blockDim.x >> 5));  // [3 warps]
    const int x = threadIdx.x, shot = blockIdx.x, warp = x >> 5, warps = blockDim.x >> 5;
    const Adj d = load_adj(a, x, shot);
    const uint32_t tau = COSET ? true_logical_parities(a, d, x, shot) : 0u;
    const bool qubit = x < a.N, check = x < a.M;
    float Pi0[3] = {0.f, 0.f, 0.f};
    if (qubit) prior_llr(a, x, Pi0);
    const float zero4[4] = {0.f, 0.f, 0.f, 0.f};
    if (qubit) put4(vbar + 4 * x, zero4);
    float Qbar[3] = {0.f, 0.f, 0.f};  // adjoint of Q^(t) of the owned qubit
    float gbar[3] = {0.f, 0.f, 0.f};  // adjoint of g^(t) (Momentum)
    float wbar[4] = {0.f, 0.f, 0.f, 0.f};
    float *row = a.rows + (size_t)shot * a.width;
    const int chunk = logical_chunk(a.n_log, warps);
    const float scale_c = 1.f / ((float)a.B * (float)a.T * (float)a.M);
    const float scale_l = 1.f / ((float)a.B * (float)a.T * (float)a.n_log);
    CheckNode c;
    // step B of the iteration whose check node is in c and whose m_v->c^(t-1)
    // is v: message weights and the check-node derivative; also the sums over
    // the qubits of that iteration's parameter gradients
    auto step_b = [&](int t) {
        if (check) {
            float G[4];
#pragma unroll
            for (int n = 0; n < 4; ++n) {
                G[n] = 0.f;
                if (d.sl[n] == kNoSlot) continue;
                const float cb = cbar[d.sl[n]];
                if (fabsf(d.ws[n] * c.r[n]) <= a.clip) {
                    wbar[n] += cb * d.sigma * c.r[n];
                    const float h = __fdividef(cb * d.ws[n], hfun(c.E[n]));
                    G[n] = c.r[n] < 0.f ? -h : h;
                }
            }
            const float G01 = G[0] + G[1], G23 = G[2] + G[3];
            const float acc[4] = {G[1] + G23, G[0] + G23, G01 + G[3], G01 + G[2]};
#pragma unroll
            for (int f = 0; f < 4; ++f)
                if (d.sl[f] != kNoSlot) {
                    const float h = hfun(c.q[f]) * acc[f];  // d r_n / d m_f
                    vbar[d.sl[f]] += ((c.neg >> f) & 1u) ? -h : h;
                }
        }
        if (x < 3) {
            float s = 0.f;
            for (int k = 0; k < warps; ++k) s += red[3 * k + x];
            if (x == 0) row[t - 1] = (MODEL == kMomentum || t > 1) ? s : 0.f;
            if (x == 1) row[a.T + t - 1] = s;
            if (x == 2 && MODEL == kMomentum) row[2 * a.T + a.E + t - 1] = s;
        }
    };
    __syncthreads();

    for (int seg = a.nck - 1; seg >= 0; --seg) {
        const int t0 = seg * K, t1 = min(a.T, t0 + K);
        // ---- recompute iterations t0+1 .. t1 from the segment's checkpoint ----
        {
            const float *ck = a.ckpt + ((size_t)shot * a.nck + seg) * a.ck_floats;
            float Q[3] = {0.f, 0.f, 0.f}, g[3] = {0.f, 0.f, 0.f}, v[4] = {0.f, 0.f, 0.f, 0.f};
            if (qubit) {
                get4(ck + 4 * x, v);
                put4(vh + 4 * x, v);
#pragma unroll
                for (int w = 0; w < 3; ++w) {
                    Qh[w * Np + x] = Q[w] = ck[(4 + w) * Np + x];
                    if (MODEL == kMomentum) gh[w * Np + x] = g[w] = ck[(7 + w) * Np + x];
                }
            }
            __syncthreads();
            for (int t = t0 + 1; t <= t1; ++t) {
                const int s = t - t0;
                if (check) {
                    check_node(a, d, vh + (size_t)(s - 1) * S4, c);
#pragma unroll
                    for (int n = 0; n < 4; ++n)
                        if (d.sl[n] != kNoSlot) cm[d.sl[n]] = c.out[n];
                }
                __syncthreads();
                if (qubit) {
                    float cin[4];
                    get4(cm + 4 * x, cin);
#pragma unroll
                    for (int k = 0; k < 4; ++k)
                        if (!slot_pauli(d.vp, k)) cin[k] = 0.f;
                    variable_node<MODEL>(a, d.vp, Pi0, cin, t, Q, g, v);
                    put4(vh + (size_t)s * S4 + 4 * x, v);
#pragma unroll
                    for (int w = 0; w < 3; ++w) {
                        Qh[(3 * s + w) * Np + x] = Q[w];
                        if (MODEL == kMomentum) gh[(3 * s + w) * Np + x] = g[w];
                    }
                }
                __syncthreads();
            }
            // ---- posterior loss: gradient at the last iteration ----
            if (!COSET && t1 == a.T && qubit) {
                const float z[4] = {0.f, -Q[0], -Q[1], -Q[2]};
                const float zm = fmaxf(fmaxf(z[0], z[1]), fmaxf(z[2], z[3]));
                float se = 0.f;
                for (int k = 0; k < 4; ++k) se += expf(z[k] - zm);
                const int e = a.err[(size_t)shot * a.N + x];
                const float scale = 1.f / ((float)a.B * (float)a.N);
                for (int w = 0; w < 3; ++w) {
                    const float pw = expf(z[w + 1] - zm) / se;
                    Qbar[w] = -(pw - (e == w + 1 ? 1.f : 0.f)) * scale;  // d CE / d Q_W = -(p_W - [W = true])
                }
            }
        }
        // ---- adjoint through iterations t1 .. t0+1 ----
        for (int t = t1; t > t0; --t) {
            const int s = t - t0;
            const float *v_prev = vh + (size_t)(s - 1) * S4;  // m_v->c^(t-1)
            // step 1
            if (t < t1) step_b(t + 1);
            if (check) {
                if (t < t1) {  // (at t1 the recomputation has just left c and cm)
                    check_node(a, d, v_prev, c);
#pragma unroll
                    for (int n = 0; n < 4; ++n)
                        if (d.sl[n] != kNoSlot) cm[d.sl[n]] = c.out[n];
                }
            }
            float Q[3] = {0.f, 0.f, 0.f}, pi[4] = {1.f, 0.f, 0.f, 0.f};
            if (qubit) {
#pragma unroll
                for (int w = 0; w < 3; ++w) Q[w] = Qh[(3 * s + w) * Np + x];
                if (COSET) {
                    marginals(Q, pi);
#pragma unroll
                    for (int k = 0; k < 4; ++k) ub[4 * x + k] = comm_anti(pi, slot_pauli(d.vp, k));
                }
            }
            if (COSET) {
                for (int l0 = 0; l0 < a.n_log; l0 += chunk) {
                    const int n = min(chunk, a.n_log - l0);
                    for (int i = 0; i < n; ++i) {
                        const uint32_t P = logical_pauli(d, l0 + i);
                        const float4 r = logical_partial<true>(comm_anti(pi, P), P != 0u);
                        if ((x & 31) == 0) part[warp * n + i] = r;
                    }
                    __syncthreads();
                    if (l0 == 0 && check) {
                        // step 2: the gradient with respect to each edge's u, over its parity
                        float2 in[4], eo = make_float2(1.f, 0.f);
#pragma unroll
                        for (int m = 0; m < 4; ++m) {
                            in[m] = d.sl[m] != kNoSlot ? ub[d.sl[m]] : make_float2(1.f, 0.f);
                            eo = parity_combine(eo, in[m]);
                        }
                        const float P = d.sigma < 0.f ? eo.y : eo.x;
                        const float g0 = P > kMinProb ? -d.sigma * __fdividef(scale_c, P) : 0.f;
                        float u[4];
#pragma unroll
                        for (int m = 0; m < 4; ++m) u[m] = in[m].x - in[m].y;
                        const float u01 = u[0] * u[1], u23 = u[2] * u[3];
                        const float U[4] = {u[1] * u23, u[0] * u23, u01 * u[3], u01 * u[2]};
#pragma unroll
                        for (int m = 0; m < 4; ++m)
                            if (d.sl[m] != kNoSlot) ub[d.sl[m]].x = g0 * U[m];
                    }
                    // the operators' gradient (the CTA's totals of this chunk)
                    for (int i = 0; i < n; ++i) {
                        const uint32_t P = logical_pauli(d, l0 + i);
                        if (!P) continue;
                        const float4 tot = logical_total<true>(part, i, n, warps);
                        const bool odd = (tau >> (l0 + i)) & 1u;
                        const float Pm = odd ? tot.y : tot.x;
                        if (!(Pm > kMinProb)) continue;
                        const float2 ca = comm_anti(pi, P);
                        const float u = ca.x - ca.y, lg = logf(fmaxf(fabsf(u), 1e-30f));
                        const int others = (int)tot.w - (u < 0.f ? 1 : 0);
                        const float U = expf(tot.z - lg);  // product over the others
                        const float gl = (((others & 1) != 0) == odd ? -U : U) * __fdividef(scale_l, Pm);
#pragma unroll
                        for (int w = 0; w < 3; ++w) Qbar[w] += gl * pi[w + 1] * (anti(w + 1, P) ? ca.x : -ca.y);
                    }
                    __syncthreads();
                }
                // step 3: the check terms' gradient with respect to Q^(t)
                if (qubit) {
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const uint32_t p = slot_pauli(d.vp, k);
                        if (!p) continue;
                        const float ge = ub[4 * x + k].x;
                        const float2 ca = comm_anti(pi, p);
#pragma unroll
                        for (int w = 0; w < 3; ++w) Qbar[w] += ge * pi[w + 1] * (anti(w + 1, p) ? ca.x : -ca.y);
                    }
                }
            } else {
                __syncthreads();
            }
            // step A (qubit threads): damping, lambda, posterior, prior
            const float al = a.alpha[t - 1], be = a.beta[t - 1];
            float bb = 0.f, ab = 0.f, gb = 0.f;
            if (qubit) {
                float cin[4], vb[4], vp4[4], cb[4], Lam[3], Lsum[3] = {0.f, 0.f, 0.f};
                get4(cm + 4 * x, cin);
                get4(vbar + 4 * x, vb);
                get4(v_prev + 4 * x, vp4);
                lambda_types(d.vp, Q, Lam);
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const uint32_t p = slot_pauli(d.vp, k);
                    cb[k] = 0.f;
                    if (!p) {
                        cin[k] = vb[k] = 0.f;
                        continue;
                    }
                    const float lam = __fsub_rn(pick3(Lam, p), cin[k]);
                    bb += vb[k] * (vp4[k] - clipped(a, lam));
                    // a clipped lambda passes no gradient
                    const float Lb = fabsf(lam) <= a.clip ? (1.f - be) * vb[k] : 0.f;
                    cb[k] = -Lb;
#pragma unroll
                    for (int h = 0; h < 3; ++h) Lsum[h] += p == (uint32_t)h + 1u ? Lb : 0.f;
                }
                // d Lambda_H / d Q: -sigmoid(-Q_H) for H, the softmax of (-Q_a, -Q_b) for the others
                float Qtot[3];
#pragma unroll
                for (int w = 0; w < 3; ++w) Qtot[w] = Qbar[w];
#pragma unroll
                for (int h = 0; h < 3; ++h) {
                    if (Lsum[h] == 0.f) continue;
                    const int i = h == 0 ? 1 : 0, j = h == 2 ? 1 : 2;
                    const float uh = expf(-fabsf(Q[h])), ud = expf(-fabsf(Q[i] - Q[j]));
                    const float sh = __fdividef(Q[h] < 0.f ? 1.f : uh, 1.f + uh), sd = __fdividef(1.f, 1.f + ud);
                    Qtot[h] -= Lsum[h] * sh;
                    const bool first = Q[i] < Q[j];  // the larger share: of the smaller Q
                    Qtot[i] += Lsum[h] * (first ? sd : ud * sd);
                    Qtot[j] += Lsum[h] * (first ? ud * sd : sd);
                }
                float Sbar[3], Qp[3];
#pragma unroll
                for (int w = 0; w < 3; ++w) Qp[w] = Qh[(3 * (s - 1) + w) * Np + x];
                if (MODEL == kMomentum) {
                    // Q^(t) = Q^(t-1) - alpha g^(t);  g^(t) = gamma g^(t-1) + (1 - gamma) D,
                    // D = Q^(t-1) - Pi^(0) - S^(t)
                    const float gm = a.gamma[t - 1];
                    float S[3];
                    incoming_sums(d.vp, cin, S);
#pragma unroll
                    for (int w = 0; w < 3; ++w) {
                        const float gtot = gbar[w] - al * Qtot[w];  // adjoint of g^(t)
                        const float D = Qp[w] - Pi0[w] - S[w];
                        ab -= Qtot[w] * gh[(3 * s + w) * Np + x];
                        gb += gtot * (gh[(3 * (s - 1) + w) * Np + x] - D);
                        Sbar[w] = -(1.f - gm) * gtot;
                        Qbar[w] = Qtot[w] + (1.f - gm) * gtot;  // adjoint of Q^(t-1)
                        gbar[w] = gm * gtot;                    // adjoint of g^(t-1)
                    }
                } else {
#pragma unroll
                    for (int w = 0; w < 3; ++w) {
                        Sbar[w] = Qtot[w];
                        ab += Qtot[w] * (Pi0[w] - Qp[w]);
                        Qbar[w] = t > 1 ? (1.f - al) * Qtot[w] : 0.f;
                    }
                }
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const uint32_t p = slot_pauli(d.vp, k);
#pragma unroll
                    for (int w = 0; w < 3; ++w) cb[k] += anti(w + 1, p) ? Sbar[w] : 0.f;
                    vb[k] *= be;  // damping path to m_v->c^(t-1)
                }
                put4(cbar + 4 * x, cb);
                put4(vbar + 4 * x, vb);
            }
            ab = warp_sum(ab);
            bb = warp_sum(bb);
            if (MODEL == kMomentum) gb = warp_sum(gb);
            if ((x & 31) == 0) {
                red[3 * warp] = ab;
                red[3 * warp + 1] = bb;
                red[3 * warp + 2] = gb;
            }
            __syncthreads();
        }
        step_b(t0 + 1);
        __syncthreads();
    }
    if (check)
        for (int n = 0; n < 4; ++n)
            if (d.sl[n] != kNoSlot) row[2 * a.T + d.ce + n] = wbar[n];
}

template <int MODEL, bool COSET>
void (*pick_size(int threads))(const TrainArgs) {
    return threads <= 320 ? train_backward_kernel<MODEL, COSET, true> : train_backward_kernel<MODEL, COSET, false>;
}
void (*pick_backward(bool momentum, bool coset, int threads))(const TrainArgs) {
    if (momentum) return coset ? pick_size<kMomentum, true>(threads) : pick_size<kMomentum, false>(threads);
    return coset ? pick_size<kEWAInit, true>(threads) : pick_size<kEWAInit, false>(threads);
}

// Sums over the shots: out_k = scale * sum_b rows[b][k], the columns k of the
// rows divided into up to four consecutive ranges, each with its own output.
// A CTA takes kReduceCols columns (one 32-byte sector of a row) with
// kReduceLanes row lanes: lane r sums rows r, r + kReduceLanes, ... and the
// lanes' sums are combined in a fixed tree, so results are deterministic.
// The kernel is bound by the latency of its loads; many lanes per column keep
// enough of them in flight.  One thread per column walking all rows took
// 280 us per gradient (4096 rows of 603 floats, four launches) and 85 us for
// the loss; this takes 8 us for all gradients and 3 us for the loss.
constexpr int kReduceCols = 8, kReduceLanes = 64;
struct ReduceOut {
    float *out[4];
    int end[4];  // first column after the range
};
__global__ void __launch_bounds__(kReduceCols *kReduceLanes) reduce_rows_kernel(const float *rows, int B, int width,
                                                                               ReduceOut o, float scale) {
    __shared__ float part[kReduceLanes][kReduceCols];
    const int c = threadIdx.x % kReduceCols, r = threadIdx.x / kReduceCols;
    const int k = blockIdx.x * kReduceCols + c;
    float s = 0.f;
    if (k < width) {
        const float *p = rows + k;
#pragma unroll 8
        for (int b = r; b < B; b += kReduceLanes) s += __ldg(p + (size_t)b * width);
    }
    part[r][c] = s;
    for (int h = kReduceLanes / 2; h > 0; h >>= 1) {
        __syncthreads();
        if (r < h) part[r][c] += part[r + h][c];
    }
    if (r == 0 && k < width) {
        int g = 0, begin = 0;
        while (k >= o.end[g]) begin = o.end[g++];
        o.out[g][k - begin] = part[0][c] * scale;
    }
}

void launch_reduce(const float *rows, int B, int width, const ReduceOut &o, float scale, cudaStream_t st) {
    reduce_rows_kernel<<<(width + kReduceCols - 1) / kReduceCols, kReduceCols * kReduceLanes, 0, st>>>(rows, B, width,
                                                                                                      o, scale);
}

size_t a256(size_t x) { return (x + 255) & ~size_t(255); }

int fill(const bpq_tanner *t, int model, const uint32_t *syn, const uint8_t *err, const float *prior, int B, int T,
         int K, const float *alpha, const float *beta, const float *gamma, const float *w, float clip,
         const bpq_train_loss *loss, void *work, size_t work_bytes, TrainArgs &a) {
    int rc = need_uploaded(t);
    if (rc) return rc;
    if (model != kEWAInit && model != kMomentum) return fail(BPQ_EINVAL, "unknown training model");
    if (B < 1 || T < 1 || T > 255 || K < 1) return fail(BPQ_EINVAL, "bad B, T or checkpoint interval");
    if (!syn || !err || !prior || !alpha || !beta || !w || !work) return fail(BPQ_EINVAL, "NULL argument");
    if (misaligned(work, kBufferAlign)) return fail(BPQ_EINVAL, "workspace not 16-byte aligned");
    if (misaligned(syn, kWordAlign) || misaligned(prior, kWordAlign) || misaligned(alpha, kWordAlign) ||
        misaligned(beta, kWordAlign) || misaligned(w, kWordAlign) || (gamma && misaligned(gamma, kWordAlign)))
        return fail(BPQ_EINVAL, "an input array not 4-byte aligned");
    if (model == kMomentum && !gamma) return fail(BPQ_EINVAL, "the Momentum model needs gamma");
    if (!(clip > 0.f)) return fail(BPQ_EINVAL, "msg_clip must be positive");
    const int kind = loss ? loss->kind : BPQ_TRAIN_LOSS_POSTERIOR;
    if (kind != BPQ_TRAIN_LOSS_POSTERIOR && kind != BPQ_TRAIN_LOSS_COSET) return fail(BPQ_EINVAL, "unknown loss");
    if (kind == BPQ_TRAIN_LOSS_COSET && (!loss->logicals_dev || loss->n_logicals < 1 ||
                                         loss->n_logicals > kMaxLogicals))
        return fail(BPQ_EINVAL, "the coset loss needs 1 to 4 logical operators");
    if (std::max(t->N, t->M) > 1024) return fail(BPQ_EINVAL, "training kernels take codes of up to 1024 nodes");
    if (work_bytes < bpq_train_workspace_bytes(t, model, B, T, K))
        return fail(BPQ_EINVAL, "training workspace too small");
    a = TrainArgs{};
    a.table = t->d_table;
    a.off_var_pauli = t->off_var_pauli;
    a.chk_ptr = t->d_chk_ptr;
    a.syn = syn;
    a.err = err;
    a.prior = prior;
    a.alpha = alpha;
    a.beta = beta;
    a.w = w;
    a.gamma = gamma;
    a.N = t->N;
    a.M = t->M;
    a.E = t->E;
    a.W = (t->M + 31) / 32;
    a.B = B;
    a.T = T;
    a.K = K;
    a.nck = (T + K - 1) / K;
    a.n_pad = (t->N + 3) & ~3;
    a.ck_floats = (model == kMomentum ? 10 : 7) * a.n_pad;
    a.width = (model == kMomentum ? 3 : 2) * T + t->E;
    a.clip = clip;
    a.loss_kind = kind;
    a.logicals = kind == BPQ_TRAIN_LOSS_COSET ? loss->logicals_dev : nullptr;
    a.n_log = kind == BPQ_TRAIN_LOSS_COSET ? loss->n_logicals : 0;
    uint8_t *p = static_cast<uint8_t *>(work);
    a.ckpt = reinterpret_cast<float *>(p);
    p += a256(sizeof(float) * (size_t)B * a.nck * a.ck_floats);
    a.loss_shot = reinterpret_cast<float *>(p);
    p += a256(sizeof(float) * B);
    a.rows = reinterpret_cast<float *>(p);
    return BPQ_OK;
}

int threads_for(const bpq_tanner *t) { return ((std::max(t->N, t->M) + 31) / 32) * 32; }

}  // namespace tr
}  // namespace bpq

extern "C" {

size_t bpq_train_workspace_bytes(const bpq_tanner *t, int model, int B, int T, int ckpt_every) {
    if (!t || B < 1 || T < 1 || ckpt_every < 1) return 0;
    if (model != BPQ_TRAIN_EWAINIT && model != BPQ_TRAIN_MOMENTUM) return 0;
    const size_t np = (size_t)((t->N + 3) & ~3);
    const size_t nck = (size_t)((T + ckpt_every - 1) / ckpt_every);
    const size_t per_ck = (model == BPQ_TRAIN_MOMENTUM ? 10 : 7) * np;
    const size_t width = (size_t)(model == BPQ_TRAIN_MOMENTUM ? 3 : 2) * T + t->E;
    return bpq::tr::a256(sizeof(float) * (size_t)B * nck * per_ck) + bpq::tr::a256(sizeof(float) * B) +
           bpq::tr::a256(sizeof(float) * (size_t)B * width);
}

int bpq_train_forward(const bpq_tanner *t, int model, const uint32_t *syn_dev, const uint8_t *err_dev,
                      const float *prior_dev, int B, int T, int ckpt_every, const float *alpha_dev,
                      const float *beta_dev, const float *gamma_dev, const float *w_dev, float msg_clip,
                      const bpq_train_loss *loss, float *loss_dev, float *Q_dev, void *work_dev, size_t work_bytes,
                      void *stream) {
    bpq::tr::TrainArgs a;
    int rc = bpq::tr::fill(t, model, syn_dev, err_dev, prior_dev, B, T, ckpt_every, alpha_dev, beta_dev, gamma_dev,
                           w_dev, msg_clip, loss, work_dev, work_bytes, a);
    if (rc) return rc;
    if (!loss_dev) return fail(BPQ_EINVAL, "NULL loss output");
    a.Q_out = Q_dev;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const bool mom = model == BPQ_TRAIN_MOMENTUM;
    const bool coset = a.loss_kind == BPQ_TRAIN_LOSS_COSET;
    const int threads = bpq::tr::threads_for(t), warps = threads / 32;
    const size_t smem = sizeof(float) * ((coset ? 12 : 4) * (size_t)a.n_pad +
                                         4 * (size_t)bpq::tr::logical_chunk(a.n_log, warps) * warps);
    if (smem > 227 * 1024) return fail(BPQ_EINVAL, "code too large for the training kernels' shared memory");
    using namespace bpq::tr;
    void (*fn)(const TrainArgs) = mom ? (coset ? train_forward_kernel<kMomentum, true> : train_forward_kernel<kMomentum, false>)
                                      : (coset ? train_forward_kernel<kEWAInit, true> : train_forward_kernel<kEWAInit, false>);
    // what a code of 1024 nodes takes with the coset loss
    rc = bpq::allow_smem(fn, sizeof(float) * (12 * 1024 + 4 * 32), "train forward attribute");
    if (rc) return rc;
    fn<<<B, threads, smem, st>>>(a);
    // per-shot sums: over qubits (posterior loss) or already normalised (coset loss)
    bpq::tr::launch_reduce(a.loss_shot, B, 1, {{loss_dev}, {1}},
                           coset ? 1.f / (float)B : 1.f / ((float)B * (float)t->N), st);
    return bpq::cuda_check(cudaGetLastError(), "train forward launch");
}

int bpq_train_backward(const bpq_tanner *t, int model, const uint32_t *syn_dev, const uint8_t *err_dev,
                       const float *prior_dev, int B, int T, int ckpt_every, const float *alpha_dev,
                       const float *beta_dev, const float *gamma_dev, const float *w_dev, float msg_clip,
                       const bpq_train_loss *loss, float *grad_alpha_dev, float *grad_beta_dev,
                       float *grad_gamma_dev, float *grad_w_dev, void *work_dev, size_t work_bytes, void *stream) {
    bpq::tr::TrainArgs a;
    int rc = bpq::tr::fill(t, model, syn_dev, err_dev, prior_dev, B, T, ckpt_every, alpha_dev, beta_dev, gamma_dev,
                           w_dev, msg_clip, loss, work_dev, work_bytes, a);
    if (rc) return rc;
    const bool mom = model == BPQ_TRAIN_MOMENTUM;
    if (!grad_alpha_dev || !grad_beta_dev || !grad_w_dev || (mom && !grad_gamma_dev))
        return fail(BPQ_EINVAL, "NULL gradient output");
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const int threads = bpq::tr::threads_for(t);
    const size_t smem = sizeof(float) * bpq::tr::backward_floats(a.n_pad, a.K, mom, a.n_log, threads / 32);
    if (smem > 227 * 1024) return fail(BPQ_EINVAL, "checkpoint interval too long for shared memory");
    void (*fn)(const bpq::tr::TrainArgs) = bpq::tr::pick_backward(mom, a.loss_kind == BPQ_TRAIN_LOSS_COSET, threads);
    rc = bpq::allow_smem(fn, bpq::kMaxDynamicSmem, "train backward attribute");
    if (rc) return rc;
    fn<<<B, threads, smem, st>>>(a);
    // per-shot rows hold [alpha | beta | w | gamma]
    bpq::tr::launch_reduce(a.rows, B, a.width,
                           {{grad_alpha_dev, grad_beta_dev, grad_w_dev, mom ? grad_gamma_dev : nullptr},
                            {T, 2 * T, 2 * T + t->E, a.width}}, 1.f, st);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return fail(BPQ_ECUDA, std::string("train backward launch: ") + cudaGetErrorString(e));
    return BPQ_OK;
}

}  // extern "C"
