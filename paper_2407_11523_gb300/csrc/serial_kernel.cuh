// Serial-schedule decoding kernels (bpq_decode_serial, bpq_decode_serial_trace):
// Algorithm 1's serial update, where the qubits are visited in index order
// and qubit j, at its turn, takes the c->v messages of its checks from the
// v->c messages as they stand (this sweep's for the qubits before j, the
// previous sweep's for those after it), updates its posterior and sends its
// new v->c messages.
//
// GB300 mapping.  Qubit j depends, within a sweep, only on the earlier
// qubits that share a check with it, and the later ones depend on j; any order
// of the qubits that keeps this relation gives exactly the serial order's
// result.  The host arranges the sweep in steps of at most 16 (or 8) mutually
// independent qubits, each after all the earlier qubits that share a check with
// it (list scheduling, longest remaining chain first, build_serial_table); a
// __syncwarp separates the steps.  LANES lanes decode one shot, so a warp decodes
// 32 / LANES shots in lockstep over the steps, and Q lanes share a qubit:
//   LANES = 32, Q = 2: steps of 16, each lane two of a qubit's four edges;
//   LANES = 16, Q = 1: steps of 16, two shots per warp;
//   LANES = 8,  Q = 1: steps of 8, four shots per warp.
// A surface code's dependency chain is about 2L steps long and L qubits wide: on
// its levels a lane per qubit and a warp per shot keep under half the lanes
// busy (toric d = 15: 32 levels for 450 qubits, 44 %; planar d = 7: 14 for 85,
// 19 %).  Steps of 16 are 38 and 14, steps of 8 are 62 and 16.  What bounds it: a
// step is one chain of dependent operations, issued at about one instruction in
// two cycles by a warp, so the time is set by the instructions a lane executes
// per step and by how many warps share a scheduler, which shared memory limits
// (toric d = 15: 15 shots per SM).  Two lanes per qubit shorten the chain (480
// against 660 cycles per step); narrow groups issue fewer instructions per shot
// where shots are small (serial_mode in serial.cu has the rule and figures).
//
// The shot's edge messages, its variant state and one byte per qubit (the
// syndrome bits of its checks) sit in shared memory; the
// per-qubit tables are staged once per CTA by a bulk TMA copy.  Persistent
// CTAs; groups take shots from an atomic queue, each at the end of the sweep in
// which its shot stops.
//
// Layout.  Per-qubit arrays (prior, state, the qubit byte) are indexed by
// the qubit's position v in the sweep's step order, so the lanes of a step
// touch consecutive words; message slots are assigned by the host so that
// the lanes of one access fall in distinct banks where possible (modulo LANES
// with several shots per warp, which lie a multiple of 32 words plus LANES
// apart, so that their accesses to the same slot fall in different banks).  The
// tables serve all shots of the warp with one read, and the next step's entries
// are read before the current step's work.  Every qubit runs four edges: padding
// edges write the trash slot and read a slot that holds a message of no
// information (delta 1, phi infinite), whose c->v message is 0; the missing
// edges of a check read the zero slot (delta 0, the identity of the check rule).
// So the per-edge work is straight code with no branch or select on the degree.  SPLIT (split-layout codes,
// bpq_tanner::split): edges 0, 1 of a qubit have Pauli X and edges 2, 3 Pauli Z
// (or are padding), so the sums and the per-edge Pauli choices are fixed by the
// position.
//
// Stopping rule.  The syndrome test of a check needs the decisions of all
// its qubits in this sweep; the last of them in the sweep order sees the
// others' new messages (their least significant bits carry the
// anticommutation of each decision with the edge's Pauli) when it updates,
// so it tests the check at its turn and the group ORs the mismatches at the
// end of the sweep: the same test as a separate pass over the checks after
// the sweep.
//
// Arithmetic is that of the parallel kernel (decode_kernel.cuh): v->c
// messages stored as sign * delta (AdaGrad-BP: sign * phi) with the
// decision's anticommutation bit in the least significant bit, and
// log-likelihoods in bits; every step is an explicit intrinsic, so no
// contraction choice of the compiler can make two widths differ.
#pragma once

#include <cuda_runtime.h>

#include "bpq_internal.h"
#include "decode_kernel.cuh"
#include "decode_launch.h"

namespace bpq {

struct SerialArgs {
    const uint8_t *table;  // bpq_tanner::SerialTable of the width (see build_serial_table)
    uint32_t table_bytes;  // bytes staged in shared memory
    uint32_t off_meta, off_steps;               // inside the staged part
    uint32_t off_qubit, off_chk, off_canon;     // in global memory only
    int nsteps;
    const uint32_t *syn;   // [B][W]
    const float *prior;    // [N][3]
    uint8_t *est, *conv, *iters;
    uint32_t *work;        // [0] next shot, [1] device error word
    float *tr_v2c, *tr_c2v, *tr_Q;
    uint8_t *tr_dec;
    int N, M, E, W, B, max_iter;
    int n_pad;             // N rounded up to 4 (per-qubit array stride)
    uint32_t zero_slot;    // message slots: [0, zero_slot) edges, then zero, no information, trash
    uint32_t shot_words;   // shared memory of one shot: messages | state | syndrome | qubit bytes
    uint32_t off_state, off_syn, off_qb, off_dec;  // word offsets inside it
    float alpha, gamma, eps, clip, clip2, delta_clip, phi_clip;
    int ada_from1;
    int warps;             // warps that decode (SerialHelpers)
};

namespace sk {

using namespace dk;

__device__ __forceinline__ float2 f2(float x) { return make_float2(x, x); }

// Per-qubit state arrays (each n_pad floats) of the serial kernels: EWAInit
// Q^(t-1); Momentum Q^(t-1), g; AdaGrad Q^(t-1), G.  The kernels and serial_launch's sizing both read this.
__host__ __device__ constexpr int serial_state_arrays(int variant) {
    return variant == BPQ_PLAIN ? 0 : variant == BPQ_EWAINIT ? 3 : 6;
}

// Whether a launch of few shots has further warps, which share the staging of the
// prior and the initial messages (three logarithms and the message rule per
// qubit: one warp takes a qubit per lane at a time) and get no shot.  One shot,
// EWAInit, us, without / with: toric d = 27 128 / 103, d = 20 77 / 63, planar d = 25
// 130 / 110, d = 11 19.6 / 16.4; staging on the sweep's own arrays before (one warp,
// no initial messages) 105, 67, 113, 18.2.  Not for AdaGrad, whose sweeps the
// compiler's code for it slows (toric d = 15, 30000 shots, 5.95 ms against 5.52).
template <int VARIANT>
struct SerialHelpers {
    static constexpr bool value = VARIANT != BPQ_ADAGRAD;
};

// The four edge Paulis of a qubit one per byte (anti_bytes' format).
__device__ __forceinline__ uint32_t pauli_bytes(uint32_t pauli) {
    return (pauli & 3u) | (((pauli >> 2) & 3u) << 8) | (((pauli >> 4) & 3u) << 16) | (((pauli >> 6) & 3u) << 24);
}

// |m_{c->v}| in bits of two edges from the magnitudes of each one's check's
// other three v->c messages (eq. (h_update)), clipped.
template <bool PHI>
__device__ __forceinline__ float2 c2v_mag2(const SerialArgs &a, float2 m0, float2 m1, float2 m2) {
    if (PHI) {
        const float2 s = __fadd2_rn(__fadd2_rn(m0, m1), m2);
        return make_float2(fminf(phi_check(s.x), a.clip2), fminf(phi_check(s.y), a.clip2));
    }
    const float2 D = oplus2(oplus2(m0, m1), m2);
    const float2 r = __ffma2_rn(make_float2(2.0f, 2.0f), make_float2(rcp(D.x), rcp(D.y)), make_float2(-1.0f, -1.0f));
    return make_float2(fminf(lg2(r.x), a.clip2), fminf(lg2(r.y), a.clip2));
}

// Q_W of the variant for one qubit of one shot at sweep t from Pi_W, S_W and
// the state (qp = Q^(t-1), s2 = g or G); updates the state.
template <int VARIANT>
__device__ __forceinline__ float posterior(const SerialArgs &a, float Pi, float S, float &qp, float &s2, int t,
                                           float alpha) {
    if (VARIANT == BPQ_PLAIN) return __fadd_rn(Pi, S);  // eq. (p_update)
    if (VARIANT == BPQ_EWAINIT) {
        // eq. (EWAInit) for the qubit at its turn
        const float base = t > 1 ? __fmaf_rn(alpha, Pi, __fmul_rn(1.f - alpha, qp)) : Pi;
        qp = __fadd_rn(base, S);
        return qp;
    }
    if (VARIANT == BPQ_MOMENTUM) {
        // eqs. (mombp1), (mombp2)
        s2 = __fmaf_rn(a.gamma, s2, __fmul_rn(1.f - a.gamma, __fsub_rn(__fsub_rn(qp, Pi), S)));
        qp = __fmaf_rn(-a.alpha, s2, qp);
        return qp;
    }
    // eq. (boost) from t = 2; G accumulates g'^2
    const float gp = __fsub_rn(__fsub_rn(qp, Pi), S);
    if (t >= 2 || a.ada_from1) s2 = __fmaf_rn(gp, gp, s2);
    qp = t == 1 ? __fadd_rn(Pi, S) : __fmaf_rn(-__fmul_rn(a.alpha, gp), rcp(__fadd_rn(sqrt_approx(s2), a.eps)), qp);
    return qp;
}

// Hard decision: I if all Q_W > 0, else the first minimum of X, Y, Z.
__device__ __forceinline__ uint32_t decide(float QX, float QY, float QZ) {
    const bool y = QY < QX;
    const float m = y ? QY : QX;
    const uint32_t d = QZ < m ? 3u : y ? 2u : 1u;
    return QX > 0.f && QY > 0.f && QZ > 0.f ? 0u : d;
}

// Message bits of two edges: sign * delta (sign * phi with PHI) from each
// one's C and A (eq. (v_update) as C / A ratios), least significant bit = ab.
template <bool PHI>
__device__ __forceinline__ uint2 v2c_bits2(const SerialArgs &a, float2 C, float2 A, uint2 ab) {
    const float2 cma = __fadd2_rn(C, make_float2(-A.x, -A.y));  // sign bit: A > C
    float2 dl;
    if (PHI) {
        const float mx0 = fmaxf(C.x, A.x), mn0 = fminf(C.x, A.x), mx1 = fmaxf(C.y, A.y), mn1 = fminf(C.y, A.y);
        dl.x = fmaxf(log1p_rel(__fmul_rn(__fmul_rn(2.0f, mn0), rcp(__fsub_rn(mx0, mn0)))), a.phi_clip);
        dl.y = fmaxf(log1p_rel(__fmul_rn(__fmul_rn(2.0f, mn1), rcp(__fsub_rn(mx1, mn1)))), a.phi_clip);
    } else {
        const float2 m = make_float2(fminf(C.x, A.x), fminf(C.y, A.y)), sum = __fadd2_rn(C, A);
        const float2 r = __fmul2_rn(__fadd2_rn(m, m), make_float2(rcp(sum.x), rcp(sum.y)));
        dl = make_float2(fmaxf(r.x, a.delta_clip), fmaxf(r.y, a.delta_clip));
    }
    const uint32_t b0 = (__float_as_uint(dl.x) & ~1u) | ab.x, b1 = (__float_as_uint(dl.y) & ~1u) | ab.y;
    return make_uint2(b0 | (__float_as_uint(cma.x) & 0x80000000u), b1 | (__float_as_uint(cma.y) & 0x80000000u));
}

// One qubit's entry of the step table, a 16-byte half for each pair of edges
// (0, 1 and 2, 3): the byte offsets of the message slots of the two own edges
// (own) and of the three other edges of each one's check (oth); and a word with
// H_ij of edge k in bits 2k, 2k+1, "last" in bits 8-11 (the qubit is the last of
// edge k's check in the sweep) and "real" in bits 12-15 (edge k exists).
struct SerialHalf {
    uint4 w;
    __device__ __forceinline__ uint32_t half(int n) const {
        const uint32_t x = n < 2 ? w.x : n < 4 ? w.y : n < 6 ? w.z : w.w;
        return (n & 1) ? x >> 16 : x & 0xFFFFu;
    }
    __device__ __forceinline__ uint32_t own(int e) const { return half(e); }
    __device__ __forceinline__ uint32_t oth(int e, int f) const { return half(2 + 3 * e + f); }
};

// The CTA's tables in shared memory.
struct SerialTab {
    const uint4 *half;      // [2][N]
    const uint32_t *meta;
    const uint16_t *steps;  // first position of each step
    const float *Pi;        // [3][n_pad] prior, in step order
    const float *init;      // initial messages: [2][n_pad] for X and Z edges (SPLIT), [3][n_pad] for X, Y, Z
};

// What a lane reads of qubit v: both halves (Q = 1), or half h (Q = 2).
template <int Q>
struct SerialRec {
    SerialHalf pair[2 / Q];
    uint32_t meta;
    __device__ __forceinline__ SerialRec(const SerialArgs &a, const SerialTab &t, int v, int h) {
#pragma unroll
        for (int i = 0; i < 2 / Q; ++i) pair[i].w = t.half[(Q == 1 ? i : h) * a.N + v];
        meta = t.meta[v];
    }
};

// Shared memory of one shot: messages | state | syndrome words | one byte per
// qubit with the syndrome bits of its edges' checks (edge k's in bits 2k and
// 2k + 1) | plain BP, which keeps no posterior: one byte per qubit with its
// decision.
struct ShotMem {
    uint8_t *msg;
    float *state;
    uint32_t *syn;
    uint8_t *qb, *dec;
};

__device__ __forceinline__ float &slot_at(uint8_t *msg, uint32_t off) { return *reinterpret_cast<float *>(msg + off); }

// C = 1 + e^{-Q_H} and A's factor of eq. (v_update) for H = X, Y, Z, with the
// common shift c0 (see decode_kernel.cuh).
struct Lambda {
    float CX, CY, CZ, AX, AY, AZ;
    __device__ __forceinline__ Lambda(float QX, float QY, float QZ) {
        const float c0 = fminf(0.f, fminf(QX, fminf(QY, QZ)));
        const float e0 = ex2(c0);
        const float eX = ex2(__fsub_rn(c0, QX)), eY = ex2(__fsub_rn(c0, QY)), eZ = ex2(__fsub_rn(c0, QZ));
        CX = __fadd_rn(e0, eX), CY = __fadd_rn(e0, eY), CZ = __fadd_rn(e0, eZ);
        AX = __fadd_rn(eY, eZ), AY = __fadd_rn(eX, eZ), AZ = __fadd_rn(eX, eY);
    }
    __device__ __forceinline__ float C(uint32_t p) const { return p == 1u ? CX : p == 2u ? CY : CZ; }
    __device__ __forceinline__ float A(uint32_t p) const { return p == 1u ? AX : p == 2u ? AY : AZ; }
};

template <bool SPLIT>
__device__ __forceinline__ uint32_t edge_pauli(uint32_t pauli, int k) {
    return SPLIT ? (k < 2 ? 1u : 3u) : (pauli >> (2 * k)) & 3u;
}

// The update of the qubit at sweep position v in sweep t (t >= 1): c->v
// messages of its checks (eq. (h_update), from the messages as they stand),
// posterior of the variant, decision, new v->c messages.  Q = 1: one lane does
// all of it; Q = 2: two adjacent lanes, h = 0 edges 0 and 1, h = 1 edges 2 and 3,
// both the posterior (act: whether the lanes have a qubit; all lanes of the warp
// call, those without one read entries of qubit 0 and drop what they compute).  Returns the syndrome mismatch of the lane's checks that this qubit is
// the last of (bit 0).
template <int VARIANT, bool TRACE, bool SPLIT, int Q>
__device__ __forceinline__ uint32_t update_qubit(const SerialArgs &a, const ShotMem &m, const SerialTab &tab,
                                                 const SerialRec<Q> &r, int v, int h, int t, int shot, bool act) {
    constexpr bool PHI = PhiForm<VARIANT>::value;
    constexpr int NS = serial_state_arrays(VARIANT);
    constexpr int P = 2 / Q;  // pairs of edges of the lane
    const int Np = a.n_pad;
    const uint32_t qb = m.qb[v], pauli = r.meta & 0xFFu;
    float Pi[3], qp[3], s2[3];
#pragma unroll
    for (int w = 0; w < 3; ++w) {
        Pi[w] = tab.Pi[w * Np + v];
        qp[w] = NS >= 3 ? m.state[w * Np + v] : 0.f;
        s2[w] = NS == 6 ? m.state[(3 + w) * Np + v] : 0.f;
    }
    if (Q == 2 && NS >= 3) __syncwarp();  // both lanes have read the state that both will write (the same values)
    const uint16_t *ce = reinterpret_cast<const uint16_t *>(a.table + a.off_canon) + 4 * v;  // traces only
    float win[2 * P];
    uint32_t x[2 * P];  // bit 31: the sign of the edge's c->v message; bit 0: its check's parity without this edge
#pragma unroll
    for (int i = 0; i < P; ++i) {
        float mag[2][3];
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            uint32_t u[3];
#pragma unroll
            for (int f = 0; f < 3; ++f) {
                u[f] = __float_as_uint(slot_at(m.msg, r.pair[i].oth(e, f)));
                mag[e][f] = __uint_as_float(u[f] & 0x7FFFFFFEu);
            }
            // the syndrome bit at bits 31 and 0
            x[2 * i + e] = u[0] ^ u[1] ^ u[2] ^ __funnelshift_r(qb, qb, 4 * (Q == 1 ? i : h) + 2 * e + 1);
        }
        const float2 w = c2v_mag2<PHI>(a, make_float2(mag[0][0], mag[1][0]), make_float2(mag[0][1], mag[1][1]),
                                       make_float2(mag[0][2], mag[1][2]));
        win[2 * i] = __uint_as_float(__float_as_uint(w.x) ^ (x[2 * i] & 0x80000000u));
        win[2 * i + 1] = __uint_as_float(__float_as_uint(w.y) ^ (x[2 * i + 1] & 0x80000000u));
    }
    float S[3];
    if (SPLIT) {
        // edges 0, 1 anticommute with Z and Y, edges 2, 3 with X and Y
        const float s0 = __fadd_rn(win[0], win[1]);
        const float s1 = Q == 1 ? __fadd_rn(win[2 * P - 2], win[2 * P - 1]) : __shfl_xor_sync(0xffffffffu, s0, 1);
        S[2] = Q == 1 || h == 0 ? s0 : s1;
        S[0] = Q == 1 || h == 0 ? s1 : s0;
        S[1] = __fadd_rn(S[0], S[2]);
    } else if (Q == 1) {
        const float w4[4] = {win[0], win[1], win[2 * P - 2], win[2 * P - 1]};
        anticommuting_sums(pauli, w4, S[0], S[1], S[2]);
    } else {
        const float o0 = __shfl_xor_sync(0xffffffffu, win[0], 1), o1 = __shfl_xor_sync(0xffffffffu, win[1], 1);
        const float w4[4] = {h ? o0 : win[0], h ? o1 : win[1], h ? win[0] : o0, h ? win[1] : o1};
        anticommuting_sums(pauli, w4, S[0], S[1], S[2]);
    }
    float Qv[3];
#pragma unroll
    for (int w = 0; w < 3; ++w) {
        Qv[w] = posterior<VARIANT>(a, Pi[w], S[w], qp[w], s2[w], t, a.alpha);
        if (act && NS >= 3) m.state[w * Np + v] = qp[w];
        if (act && NS == 6) m.state[(3 + w) * Np + v] = s2[w];
    }
    const uint32_t d = decide(Qv[0], Qv[1], Qv[2]);
    if (act && NS == 0) m.dec[v] = (uint8_t)d;
    // whether the decision anticommutes with each edge
    uint32_t ab[2 * P];
    if (SPLIT) {
        const uint32_t b = anti_bits_split(d);
#pragma unroll
        for (int i = 0; i < P; ++i) ab[2 * i] = ab[2 * i + 1] = (Q == 1 ? i : h) ? b >> 1 : b & 1u;
    } else {
        const uint32_t b = anti_bytes(d, pauli_bytes(pauli)) >> (Q == 1 ? 0 : 16 * h);
#pragma unroll
        for (int k = 0; k < 2 * P; ++k) ab[k] = (b >> (8 * k)) & 1u;
    }
    const uint32_t last = r.meta >> (8 + (Q == 1 ? 0 : 2 * h));
    uint32_t mismatch = 0;
#pragma unroll
    for (int k = 0; k < 2 * P; ++k) mismatch |= (x[k] ^ ab[k]) & (last >> k);
    // eq. (v_update)/(mombp5)
    const Lambda lam(Qv[0], Qv[1], Qv[2]);
#pragma unroll
    for (int i = 0; i < P; ++i) {
        const int pr = Q == 1 ? i : h;  // edges 2 pr, 2 pr + 1
        float2 C, F;
        if (SPLIT) {
            C = f2(pr ? lam.CZ : lam.CX);
            F = f2(pr ? lam.AZ : lam.AX);
        } else {
            const uint32_t p0 = (pauli >> (4 * pr)) & 3u, p1 = (pauli >> (4 * pr + 2)) & 3u;
            C = make_float2(lam.C(p0), lam.C(p1));
            F = make_float2(lam.A(p0), lam.A(p1));
        }
        const float2 A = __fmul2_rn(F, make_float2(ex2(win[2 * i]), ex2(win[2 * i + 1])));
        const uint2 out = v2c_bits2<PHI>(a, C, A, make_uint2(ab[2 * i], ab[2 * i + 1]));
        if (act) {
            slot_at(m.msg, r.pair[i].own(0)) = __uint_as_float(out.x);
            slot_at(m.msg, r.pair[i].own(1)) = __uint_as_float(out.y);
        }
        if (TRACE && act)
            for (int e = 0; e < 2; ++e) {
                const int k = 2 * pr + e;
                if (!((r.meta >> (12 + k)) & 1u)) continue;
                if (a.tr_c2v)
                    a.tr_c2v[((size_t)shot * a.max_iter + (t - 1)) * a.E + ce[k]] = kLn2 * win[2 * i + e];
                if (a.tr_v2c)
                    a.tr_v2c[((size_t)shot * (a.max_iter + 1) + t) * a.E + ce[k]] =
                        fminf(fmaxf(kLn2 * (lg2(e ? C.y : C.x) - lg2(e ? A.y : A.x)), -a.clip), a.clip);
            }
    }
    if (TRACE && act && h == 0) {
        const size_t o = (size_t)shot * a.max_iter + (t - 1);
        const int j = reinterpret_cast<const uint16_t *>(a.table + a.off_qubit)[v];
        if (a.tr_Q) {
            a.tr_Q[(o * a.N + j) * 3 + 0] = kLn2 * Qv[0];
            a.tr_Q[(o * a.N + j) * 3 + 1] = kLn2 * Qv[1];
            a.tr_Q[(o * a.N + j) * 3 + 2] = kLn2 * Qv[2];
        }
        if (a.tr_dec) a.tr_dec[o * a.N + j] = (uint8_t)d;
    }
    return act ? mismatch & 1u : 0u;
}

// Eq. (init) for one shot (lane ln of LANES): the qubit bytes take the
// syndrome bits of each qubit's checks; Q^(0) = Pi^(0), g^(0) = G^(0) = 0;
// lambda(Pi^(0)) on every edge.
template <int VARIANT, bool TRACE, bool SPLIT, int LANES>
__device__ __forceinline__ void init_shot(const SerialArgs &a, const ShotMem &m, const SerialTab &tab, int ln, int shot) {
    constexpr int NS = serial_state_arrays(VARIANT);
    const int Np = a.n_pad;
    const uint2 *chk = reinterpret_cast<const uint2 *>(a.table + a.off_chk);
    for (int v = ln; v < a.N; v += LANES) {
        const SerialHalf h0{tab.half[v]}, h1{tab.half[a.N + v]};
        const uint32_t meta = tab.meta[v], real = (meta >> 12) & 15u;
        const uint2 c2 = __ldg(chk + v);
        const uint32_t chks[4] = {c2.x & 0xFFFFu, c2.x >> 16, c2.y & 0xFFFFu, c2.y >> 16};
        const uint32_t own[4] = {h0.own(0), h0.own(1), h1.own(0), h1.own(1)};
        uint32_t q = 0;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            q |= (((real >> k) & 1u) ? (m.syn[chks[k] >> 5] >> (chks[k] & 31)) & 1u : 0u) * (3u << (2 * k));
            const uint32_t p = edge_pauli<SPLIT>(meta, k);
            slot_at(m.msg, own[k]) = tab.init[(SPLIT ? (k < 2 ? 0 : 1) : p ? (int)p - 1 : 0) * Np + v];
        }
        m.qb[v] = (uint8_t)q;
#pragma unroll
        for (int w = 0; w < 3; ++w) {
            if (NS >= 3) m.state[w * Np + v] = tab.Pi[w * Np + v];
            if (NS == 6) m.state[(3 + w) * Np + v] = 0.f;
        }
        if (TRACE && a.tr_v2c) {
            const uint16_t *ce = reinterpret_cast<const uint16_t *>(a.table + a.off_canon) + 4 * v;
            const Lambda lam(tab.Pi[v], tab.Pi[Np + v], tab.Pi[2 * Np + v]);
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const uint32_t p = edge_pauli<SPLIT>(meta, k);
                const float l = fminf(fmaxf(kLn2 * (lg2(lam.C(p)) - lg2(__fmul_rn(lam.A(p), ex2(0.f)))), -a.clip), a.clip);
                if ((real >> k) & 1u) a.tr_v2c[(size_t)shot * (a.max_iter + 1) * a.E + ce[k]] = l;
            }
        }
    }
}

// Stage the step table (bulk TMA), the prior LLRs Pi_{v,W} = log2(p^I / p^W)
// and the initial messages in step order, and the constant slots of every shot.
// Returns false (after setting the error word) if the copy did not complete.
template <int VARIANT, bool SPLIT>
__device__ __forceinline__ bool stage_serial(const SerialArgs &a, uint8_t *smem, int shots, SerialTab &tab,
                                             uint32_t **shots_out) {
    constexpr bool PHI = PhiForm<VARIANT>::value;
    uint64_t *mbar = reinterpret_cast<uint64_t *>(smem);
    uint8_t *base = smem + 128;
    const int Np = a.n_pad;
    float *Pi = reinterpret_cast<float *>(base + a.table_bytes);
    float *init = Pi + 3 * Np;
    uint32_t *mem = reinterpret_cast<uint32_t *>(init + (SPLIT ? 2 : 3) * Np);
    const int tid = threadIdx.x;
    if (tid == 0) {
        mbar_init(mbar, 1);
        fence_mbar_init();
    }
    __syncthreads();
    if (tid == 0) {
        mbar_expect_tx(mbar, a.table_bytes);
        bulk_g2s(base, a.table, a.table_bytes, mbar);
    }
    for (int s = tid; s < shots; s += blockDim.x) {
        uint32_t *special = mem + (size_t)s * a.shot_words + a.zero_slot;
        special[0] = 0u;
        special[1] = __float_as_uint(PHI ? INFINITY : 1.0f);
    }
    const uint16_t *qubit = reinterpret_cast<const uint16_t *>(a.table + a.off_qubit);
    for (int v = tid; v < a.N; v += blockDim.x) {
        const int j = __ldg(qubit + v);
        const float px = a.prior[3 * j], py = a.prior[3 * j + 1], pz = a.prior[3 * j + 2];
        const float pI = 1.0f - px - py - pz;
        const float P[3] = {log2f(pI / px), log2f(pI / py), log2f(pI / pz)};
        const Lambda lam(P[0], P[1], P[2]);
#pragma unroll
        for (int w = 0; w < 3; ++w) {
            Pi[w * Np + v] = P[w];
            // decision bit 0, no incoming message
            if (!SPLIT || w != 1) {
                const float C = lam.C(w + 1), A = __fmul_rn(lam.A(w + 1), ex2(0.f));
                init[(SPLIT ? w / 2 : w) * Np + v] =
                    __uint_as_float(v2c_bits2<PHI>(a, make_float2(C, C), make_float2(A, A), make_uint2(0u, 0u)).x);
            }
        }
    }
    const bool staged = mbar_wait_bounded(mbar, 0, 1u << 22);
    if (__syncthreads_or(!staged)) {
        if (tid == 0) atomicExch(a.work + 1, 1u);
        mbar_wait_bounded(mbar, 0, 1u << 22);
        return false;
    }
    tab.half = reinterpret_cast<const uint4 *>(base);
    tab.meta = reinterpret_cast<const uint32_t *>(base + a.off_meta);
    tab.steps = reinterpret_cast<const uint16_t *>(base + a.off_steps);
    tab.Pi = Pi;
    tab.init = init;
    *shots_out = mem;
    return true;
}

// Most warps of a CTA: a whole warp per shot takes 64 registers a thread,
// narrower groups 128 (shared memory holds fewer of their warps).
__host__ __device__ constexpr int serial_max_warps(int lanes) { return lanes == 32 ? 32 : 16; }

// Persistent kernel: LANES lanes decode a shot, Q lanes a qubit, so a step
// holds LANES / Q qubits (TRACE: exactly max_iter sweeps).
template <int VARIANT, bool TRACE, bool SPLIT, int LANES, int Q>
__global__ void __launch_bounds__(32 * serial_max_warps(LANES), 1) serial_kernel(const SerialArgs a) {
    extern __shared__ __align__(16) uint8_t smem[];
    constexpr int K = 32 / LANES;  // shots per warp
    SerialTab tab;
    uint32_t *mem;
    constexpr bool HELPERS = SerialHelpers<VARIANT>::value;
    if (!stage_serial<VARIANT, SPLIT>(a, smem, K * (HELPERS ? a.warps : (int)(blockDim.x >> 5)), tab, &mem)) return;
    const int lane = threadIdx.x & 31, g = lane / LANES, ln = lane % LANES;
    const int h = ln % Q, pos = ln / Q;
    ShotMem m;
    {
        uint32_t *p = mem + (size_t)(K * (threadIdx.x >> 5) + g) * a.shot_words;
        m.msg = reinterpret_cast<uint8_t *>(p);
        m.state = reinterpret_cast<float *>(p + a.off_state);
        m.syn = p + a.off_syn;
        m.qb = reinterpret_cast<uint8_t *>(p + a.off_qb);
        m.dec = reinterpret_cast<uint8_t *>(p + a.off_dec);
    }
    const uint32_t group_mask = LANES == 32 ? 0xffffffffu : ((1u << (LANES % 32)) - 1u) << (g * LANES);
    int shot = 0, t = 0;
    bool live = true, start = true;
    for (;;) {
        // groups whose shot has stopped take the next one
        if (__any_sync(0xffffffffu, start)) {
            // a warp that only staged the tables: no shot, and it ends here.  (A return
            // above the loop costs every warp of it: toric d = 15, 10^5 shots, EWAInit
            // 3.26 ms against 3.16.)
            int s = HELPERS ? a.B : 0;
            if (start && ln == 0 && (!HELPERS || (int)(threadIdx.x >> 5) < a.warps)) s = (int)atomicAdd(a.work, 1u);
            s = __shfl_sync(0xffffffffu, s, g * LANES);
            if (start) {
                shot = s;
                live = shot < a.B;
                t = 0;
                if (live)
                    for (int w = ln; w < a.W; w += LANES) m.syn[w] = __ldg(a.syn + (size_t)shot * a.W + w);
            }
            __syncwarp();
            if (start && live) init_shot<VARIANT, TRACE, SPLIT, LANES>(a, m, tab, ln, shot);
            __syncwarp();
            if (!__any_sync(0xffffffffu, live)) break;
        }
        // one sweep
        ++t;
        uint32_t mismatch = 0;
        int v = pos, end = tab.steps[1];
        bool act = live && v < end;
        if (v >= end) v = 0;
        SerialRec<Q> r(a, tab, v, h);
        for (int s = 1; s <= a.nsteps; ++s) {
            // the next step's entry, while this one's messages are on their way
            int v2 = end + pos;
            end = s < a.nsteps ? tab.steps[s + 1] : 0;
            const bool act2 = live && v2 < end;
            if (v2 >= end) v2 = 0;
            const SerialRec<Q> r2(a, tab, v2, h);
            if (Q == 2)
                mismatch |= update_qubit<VARIANT, TRACE, SPLIT, Q>(a, m, tab, r, v, h, t, shot, act);
            else if (act)
                mismatch |= update_qubit<VARIANT, TRACE, SPLIT, Q>(a, m, tab, r, v, h, t, shot, true);
            __syncwarp();
            r = r2;
            v = v2;
            act = act2;
        }
        const bool bad = (__ballot_sync(0xffffffffu, mismatch) & group_mask) != 0;
        start = live && (TRACE ? t == a.max_iter : (!bad || t == a.max_iter));
        if (start) {
            if (!TRACE || a.est) {
                const uint16_t *qubit = reinterpret_cast<const uint16_t *>(a.table + a.off_qubit);
                for (int u = ln; u < a.N; u += LANES)
                    a.est[(size_t)shot * a.N + __ldg(qubit + u)] =
                        (uint8_t)(serial_state_arrays(VARIANT) == 0
                                      ? m.dec[u]
                                      : decide(m.state[u], m.state[a.n_pad + u], m.state[2 * a.n_pad + u]));
            }
            if (ln == 0 && (!TRACE || a.conv)) {
                a.conv[shot] = (uint8_t)(bad ? 0 : 1);
                a.iters[shot] = (uint8_t)t;
            }
        }
        __syncwarp();
    }
}

using SerialKernelFn = void (*)(const SerialArgs);
// The kernels of a variant, one translation unit per group width; split: the
// code has the split layout.  32 lanes per shot, two per qubit (serial.cu); 16
// and 8 lanes, one per qubit.
SerialKernelFn pick_serial32(int variant, bool trace, bool split);
SerialKernelFn pick_serial16(int variant, bool split);  // serial16.cu
SerialKernelFn pick_serial8(int variant, bool split);   // serial8.cu

#define BPQ_SERIAL_CASE(V, TRACE, LANES, Q) \
    case V: return split ? serial_kernel<V, TRACE, true, LANES, Q> : serial_kernel<V, TRACE, false, LANES, Q>;
#define BPQ_SERIAL_SWITCH(TRACE, LANES, Q)              \
    switch (variant) {                                  \
        BPQ_SERIAL_CASE(BPQ_PLAIN, TRACE, LANES, Q)     \
        BPQ_SERIAL_CASE(BPQ_MOMENTUM, TRACE, LANES, Q)  \
        BPQ_SERIAL_CASE(BPQ_ADAGRAD, TRACE, LANES, Q)   \
        BPQ_SERIAL_CASE(BPQ_EWAINIT, TRACE, LANES, Q)   \
    }                                                   \
    return nullptr;

}  // namespace sk

}  // namespace bpq
