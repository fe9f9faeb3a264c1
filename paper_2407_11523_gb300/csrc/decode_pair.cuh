// Two shots per thread: the flooding-schedule decoder of decode_kernel.cuh
// for codes in the split table layout, with every thread working on the
// same nodes of two shots at once ("lanes" 0 and 1).  Each message slot is a
// float2 holding the edge's message in both shots, so one 64-bit shared-
// memory access and one address serve two shots, and every floating-point
// step of the update rules runs as one packed f32x2 instruction over the two
// lanes.  Each lane rounds exactly as the one-shot kernel's scalar operation,
// so per-shot results are bit-identical to decode_kernel's.
//
// The lanes are independent shots with their own iteration counts: when a
// lane's decision satisfies its syndrome (or it reaches max_iter) the group
// writes that shot's outputs and the lane takes the next shot from the work
// queue at once, restarting from the initial messages of eq. (init) (which
// do not depend on the shot, since the prior is shared) while the other lane
// carries on.  The group synchronises on its barrier twice per iteration:
// after the check pass, which also publishes the lanes' syndrome-test votes
// (warp votes gathered in a shared flag word), and after the variable pass.
//
// What bounds it: per check and qubit of a warp (two shots), toric d = 15,
// about 300 issue slots, of which 117 go to the half-rate ALU pipe (minima,
// masks, sign and parity bits), and 40 special-function operations, which
// occupy their unit for 265 cycles (ex2 4 cycles a warp instruction, rcp and lg2
// 8, measured) of the 405 that pass; HBM traffic is negligible.  So the kernel
// spends shared memory to save instructions and registers:
//  * the slot addresses of a check are read from a per-CTA table of byte
//    offsets (one 128-bit load, no unpacking; one shot group per CTA, or
//    one-warp groups) in
//    place of packed indices in registers.  That also frees the registers that
//    tied a thread to two nodes: a thread loops over any number of nodes, so
//    large codes can take small groups, more of which fit an SM.
//    kPairGroups (several larger groups per CTA, or one where the smaller table
//    brings a third more CTAs onto an SM): 16-bit slot indices, half the size.
//  * a syndrome bit enters as one word whose bits 31 (sign) and 0 (parity)
//    are both the bit; a register per lane is rotated from check to check.
//  * the decision is kept as its two anticommutation bits, which the messages
//    need, and turned into a Pauli code only when the shot stops.
// EWAInit-BP, 10^5 toric d = 15 shots at p = 0.08 (256 threads): 5.73 ms with
// adjacency in registers, 5.50 ms so.
#pragma once

#include "decode_kernel.cuh"

namespace bpq {
namespace dk {

__device__ __forceinline__ float2 f2(float x) { return make_float2(x, x); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 neg2(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __fadd2_rn(a, neg2(b)); }
__device__ __forceinline__ float2 min2(float2 a, float2 b) { return make_float2(fminf(a.x, b.x), fminf(a.y, b.y)); }
__device__ __forceinline__ float2 max2(float2 a, float2 b) { return make_float2(fmaxf(a.x, b.x), fmaxf(a.y, b.y)); }
__device__ __forceinline__ float2 rcp2(float2 a) { return make_float2(rcp(a.x), rcp(a.y)); }
__device__ __forceinline__ float2 ex22(float2 a) { return make_float2(ex2(a.x), ex2(a.y)); }
__device__ __forceinline__ uint2 bits2(float2 a) { return make_uint2(__float_as_uint(a.x), __float_as_uint(a.y)); }

// phi_check and log1p_rel on both lanes (the same steps, packed).
__device__ __forceinline__ float2 phi_check2(float2 S) {
    float2 q = fma2(S, f2(1.0f / 720.0f), f2(1.0f / 120.0f));
    q = fma2(S, q, f2(1.0f / 24.0f));
    q = fma2(S, q, f2(1.0f / 6.0f));
    q = fma2(S, q, f2(0.5f));
    q = fma2(S, q, f2(1.0f));
    const float2 poly = mul2(S, q);
    const float2 arg = mul2(S, f2(kLog2e));
    const float2 big = add2(make_float2(ex2_always(arg.x), ex2_always(arg.y)), f2(-1.0f));
    const float2 em1 = make_float2(S.x < 0.25f ? poly.x : big.x, S.y < 0.25f ? poly.y : big.y);
    const float2 r = fma2(f2(2.0f), rcp2(em1), f2(1.0f));
    return make_float2(lg2(r.x), lg2(r.y));
}
__device__ __forceinline__ float2 log1p_rel2(float2 r) {
    float2 q = fma2(r, f2(0.2f), f2(-0.25f));
    q = fma2(r, q, f2(1.0f / 3.0f));
    q = fma2(r, q, f2(-0.5f));
    q = fma2(r, q, f2(1.0f));
    const float2 poly = mul2(r, q);
    const float2 r1 = add2(f2(1.0f), r);
    const float2 big = mul2(f2(kLn2), make_float2(lg2_always(r1.x), lg2_always(r1.y)));
    return make_float2(r.x < 0.0625f ? poly.x : big.x, r.y < 0.0625f ? poly.y : big.y);
}

// Plain BP adds the prior to every posterior, so its table holds each value
// twice (a packed operand); the others keep one copy.
template <int VARIANT>
struct PairPrior {
    static constexpr int copies = pair_prior_copies(VARIANT);
};

// Shared memory of the CTA: header | idx (int4 or ushort4 per check) | used
// positions of each qubit (bytes) | Pi [3][n_pad] | initial messages
// [4 n_pad] | groups.  A group: two vote words (16 bytes), the float2 message
// slots (4 n_pad + the zero slot, padded to 4 n_pad + 4) and
// the variant state (float2 [arrays][n_pad]).
struct PairMem {
    const uint8_t *idx, *used;
    const float *PiS, *init;
    uint32_t *votes;
    uint8_t *slots;  // byte-addressed float2 slots
    float2 *state;
};

template <int VARIANT, int MODE>
__device__ __forceinline__ PairMem pair_mem(const DecodeArgs &a, uint8_t *smem, int group) {
    PairMem m;
    const PairOffsets o = pair_offsets(VARIANT, MODE != kPairGroups, a.M, a.n_pad);
    m.idx = smem + o.idx;
    m.used = smem + o.used;
    m.PiS = reinterpret_cast<const float *>(smem + o.prior);
    m.init = reinterpret_cast<const float *>(smem + o.init);
    uint8_t *g = smem + o.groups + (MODE == kPairOne ? 0u : (uint32_t)group * a.group_bytes);
    m.votes = reinterpret_cast<uint32_t *>(g);
    m.slots = g + kPairVoteBytes;
    m.state = reinterpret_cast<float2 *>(m.slots) + a.slots_floats;
    return m;
}

// Byte offsets (from the group's slots) of the four message slots of check i.
template <int MODE>
__device__ __forceinline__ uint4 pair_slots(const uint8_t *idx, int i) {
    if (MODE != kPairGroups) return reinterpret_cast<const uint4 *>(idx)[i];
    const uint2 s = reinterpret_cast<const uint2 *>(idx)[i];
    return make_uint4((s.x & 0xFFFFu) * 8u, (s.x >> 16) * 8u, (s.y & 0xFFFFu) * 8u, (s.y >> 16) * 8u);
}

// Barrier of the group: of the CTA when it holds one group, of the warp.
template <int MODE>
__device__ __forceinline__ void pair_sync(int G, int bar_id) {
    if (MODE == kPairOne)
        __syncthreads();
    else if (MODE == kPairWarps)
        __syncwarp();
    else
        group_sync(G, bar_id);
}

// Barrier over the group that returns, per lane, whether any thread's vote
// is set: bit k of the result for bit k of `votes`.  Each warp ORs its two
// warp-wide votes into the shared word votes_smem[parity] before the
// barrier; the word of the other parity, read in the previous iteration, is
// cleared before the next barrier so that the next iteration finds it zero.
template <int MODE>
__device__ __forceinline__ uint32_t group_any2(int G, int bar_id, uint32_t votes, uint32_t *votes_smem, int tg,
                                               uint32_t parity) {
    const uint32_t w = __reduce_or_sync(0xffffffffu, votes);
    if (MODE == kPairWarps || (MODE == kPairGroups && G == 1)) {
        __syncwarp();
        return w;
    }
    if ((tg & 31) == 0 && w) atomicOr(votes_smem + parity, w);
    pair_sync<MODE>(G, bar_id);
    const uint32_t any = *reinterpret_cast<volatile uint32_t *>(votes_smem + parity);
    if (tg == 0) votes_smem[parity ^ 1u] = 0u;
    return any;
}

// Variable-to-check messages of one qubit for both lanes (split layout):
// emit_v2c's arithmetic, each step one f32x2 instruction over the lanes.  mq:
// min(Q_X, Q_Y, Q_Z) of each lane; ax, az: whether each lane's decision
// anticommutes with the X positions (0, 1) and the Z positions (2, 3).
template <bool PHI, bool FULL>
__device__ __forceinline__ void emit_v2c_pair(float vclip, float2 *slots, int Np, uint32_t used, float2 QX, float2 QY,
                                              float2 QZ, float2 mq, const float2 (&win)[4], uint2 ax, uint2 az) {
    const float2 c0 = min2(f2(0.f), mq);
    const float2 e0 = ex22(c0);
    const float2 eX = ex22(sub2(c0, QX)), eY = ex22(sub2(c0, QY)), eZ = ex22(sub2(c0, QZ));
    // C = 1 + e^{-Q_H} and the two anticommuting terms for H = X (positions
    // 0, 1) and H = Z (positions 2, 3)
    const float2 CX = add2(e0, eX), AX = add2(eY, eZ), CZ = add2(e0, eZ), AZ = add2(eX, eY);
#pragma unroll
    for (int n = 0; n < 4; ++n) {
        const float2 C = n < 2 ? CX : CZ;
        const float2 A = mul2(n < 2 ? AX : AZ, ex22(win[n]));
        const uint2 neg = bits2(sub2(C, A));  // sign bit: A > C, i.e. lambda < 0
        float2 dl;
        if (PHI) {
            const float2 mx = max2(C, A), mn = min2(C, A);
            dl = max2(log1p_rel2(mul2(mul2(f2(2.0f), mn), rcp2(sub2(mx, mn)))), f2(vclip));
        } else {
            const float2 m = min2(C, A);
            dl = max2(mul2(add2(m, m), rcp2(add2(C, A))), f2(vclip));
        }
        const uint2 d = bits2(dl), ab = n < 2 ? ax : az;
        const uint32_t b0 = (d.x & ~1u) | ab.x, b1 = (d.y & ~1u) | ab.y;
        if (FULL || ((used >> n) & 1u))
            slots[n * Np] = make_float2(__uint_as_float(b0 | (neg.x & 0x80000000u)),
                                        __uint_as_float(b1 | (neg.y & 0x80000000u)));
    }
}

// Decode shots two at a time with a group of G warps (thread tg of 32G)
// until the queue is empty.  Each thread owns the nodes tg, tg + T, ... (at
// most kPairMaxNodes).
template <int VARIANT, bool FULL, int MODE>
__device__ __forceinline__ void decode_pairs(const DecodeArgs &a, const PairMem &m, int T, int tg, int G, int bar_id,
                                             int *grp_shot) {
    constexpr bool PHI = PhiForm<VARIANT>::value;
    constexpr int NS = StateArrays<VARIANT>::n;
    const ShotParams sp = shot_params<PHI>(a, a.alpha);
    const int N = sp.N, M = sp.M, Np = sp.Np;
    const uint32_t zero = 8u * (4u * (uint32_t)Np);  // byte offset of the zero slot
    uint8_t *slots = m.slots;
    float2 *state = m.state;
    const float *PiS = m.PiS, *init = m.init;
    uint32_t parity = 0;

    // start both lanes
    if (tg == 0) {
        grp_shot[0] = (int)atomicAdd(a.work, 1u);
        grp_shot[1] = (int)atomicAdd(a.work, 1u);
        m.votes[0] = m.votes[1] = 0u;
    }
    pair_sync<MODE>(G, bar_id);
    int shot[2] = {grp_shot[0], grp_shot[1]};
    int t[2] = {1, 1};
    // syndrome bits of the owned checks: that of the k-th is at bits 31 and 0
    // of the lane's word rotated left by 2k
    uint32_t syn[2];
    // decisions of the owned qubits, two bits each (anticommutes with X, with
    // Z), the last owned qubit lowest
    uint32_t dec[2] = {0u, 0u};
    auto load_syndrome = [&](int lane) {
        uint32_t w = 0;
        if (shot[lane] < a.B) {
            const uint32_t *src = a.syn + (size_t)shot[lane] * a.W;
            for (int i = tg, k = 0; i < M; i += T, k += 2)
                if ((__ldg(src + (i >> 5)) >> (i & 31)) & 1u) w |= __funnelshift_r(0x80000001u, 0x80000001u, k);
        }
        syn[lane] = w;
    };
    // eq. (init) for `lanes` (bit k = lane k): the shot-independent initial
    // messages, Q^(0) = Pi^(0), g^(0) = G^(0) = 0, EWAInit's Pi^(1) = Pi^(0)
    auto restart = [&](uint32_t lanes) {
        for (int j = tg; j < N; j += T) {
#pragma unroll
            for (int n = 0; n < 4; ++n) {
                float *s = reinterpret_cast<float *>(slots) + 2 * (n * Np + j);
                const float v = init[n * Np + j];
                if (lanes & 1u) s[0] = v;
                if (lanes & 2u) s[1] = v;
            }
            if (NS >= 3) {
#pragma unroll
                for (int w = 0; w < 3; ++w) {
                    const float pw = PiS[w * Np + j];
                    float *s = reinterpret_cast<float *>(state + w * Np + j);
                    float *s3 = reinterpret_cast<float *>(state + (3 + w) * Np + j);
                    const float v3 = VARIANT == BPQ_EWAINIT ? a.alpha * pw : 0.f;
                    if (lanes & 1u) { s[0] = pw; s3[0] = v3; }
                    if (lanes & 2u) { s[1] = pw; s3[1] = v3; }
                }
            }
        }
    };
    if (shot[0] >= a.B && shot[1] >= a.B) return;
    load_syndrome(0);
    load_syndrome(1);
    restart(3u);
    pair_sync<MODE>(G, bar_id);

    for (;;) {
        uint32_t mis0 = 0, mis1 = 0;  // bit 0: a check of the lane fails the syndrome test
        uint32_t w0 = syn[0], w1 = syn[1];
        // ---- check pass: syndrome tests of the lanes' previous decisions, then eq. (h_update) ----
#pragma unroll 1
        for (int i = tg; i < M; i += T) {
            const uint4 o4 = pair_slots<MODE>(m.idx, i);
            const uint32_t off[4] = {o4.x, o4.y, o4.z, o4.w};
            uint2 u[4];
#pragma unroll
            for (int n = 0; n < 4; ++n) u[n] = *reinterpret_cast<const uint2 *>(slots + off[n]);
            // bit 31: (-1)^{s_i} times the product of the incoming signs; bit 0:
            // the parity of the previous decision on this check's edges plus s_i
            const uint32_t x0 = u[0].x ^ u[1].x ^ u[2].x ^ u[3].x ^ w0, x1 = u[0].y ^ u[1].y ^ u[2].y ^ u[3].y ^ w1;
            w0 = __funnelshift_l(w0, w0, 2);
            w1 = __funnelshift_l(w1, w1, 2);
            mis0 |= x0;
            mis1 |= x1;
            float2 ext[4];
            float2 mag[4];
#pragma unroll
            for (int n = 0; n < 4; ++n)
                mag[n] = make_float2(__uint_as_float(u[n].x & 0x7FFFFFFEu), __uint_as_float(u[n].y & 0x7FFFFFFEu));
            if (PHI) {
                const float2 e01 = add2(mag[0], mag[1]), e23 = add2(mag[2], mag[3]);
                ext[0] = add2(mag[1], e23);
                ext[1] = add2(mag[0], e23);
                ext[2] = add2(e01, mag[3]);
                ext[3] = add2(e01, mag[2]);
            } else {
                // a (+) b = a + b - ab, as oplus
                const float2 d01 = fma2(neg2(mag[0]), mag[1], add2(mag[0], mag[1]));
                const float2 d23 = fma2(neg2(mag[2]), mag[3], add2(mag[2], mag[3]));
                ext[0] = fma2(neg2(mag[1]), d23, add2(mag[1], d23));
                ext[1] = fma2(neg2(mag[0]), d23, add2(mag[0], d23));
                ext[2] = fma2(neg2(mag[3]), d01, add2(mag[3], d01));
                ext[3] = fma2(neg2(mag[2]), d01, add2(mag[2], d01));
            }
#pragma unroll
            for (int n = 0; n < 4; ++n) {
                float2 w;
                if (PHI) {
                    w = phi_check2(ext[n]);
                } else {
                    // c2v_magnitude on both lanes
                    const float2 q = fma2(f2(2.0f), rcp2(ext[n]), f2(-1.0f));
                    w = make_float2(lg2(q.x), lg2(q.y));
                }
                if (!(FULL && !PHI)) w = min2(w, f2(sp.clip2));
                const uint2 wb = bits2(w);
                const uint2 out = make_uint2(wb.x ^ ((x0 ^ u[n].x) & 0x80000000u), wb.y ^ ((x1 ^ u[n].y) & 0x80000000u));
                if (FULL || off[n] != zero) *reinterpret_cast<uint2 *>(slots + off[n]) = out;
            }
        }
        // a lane's first check pass has no previous decision to test
        const uint32_t mismatch = (t[0] > 1 ? mis0 & 1u : 0u) | (t[1] > 1 ? (mis1 & 1u) << 1 : 0u);
        const uint32_t any = group_any2<MODE>(G, bar_id, mismatch, m.votes, tg, parity);
        parity ^= 1u;
        uint32_t fin = 0;
#pragma unroll
        for (int l = 0; l < 2; ++l) {
            if (shot[l] >= a.B) continue;
            const bool conv = t[l] > 1 && !((any >> l) & 1u);
            if (conv || t[l] > sp.max_iter) {
                fin |= 1u << l;
                // outputs: the decision of the lane's last iteration
                uint8_t *est = a.est + (size_t)shot[l] * N;
                int sh = 2 * ((N - tg + T - 1) / T);
                for (int j = tg; j < N; j += T) {
                    sh -= 2;
                    const uint32_t d = dec[l] >> sh, dx = d & 1u, dz = (d >> 1) & 1u;
                    if (BPQ_IN_BOUNDS((size_t)shot[l] * N + j, (size_t)a.B * N, a.work + 1))
                        est[j] = (uint8_t)((dx << 1) | (dx ^ dz));
                }
                if (tg == 0 && BPQ_IN_BOUNDS(shot[l], a.B, a.work + 1)) {
                    a.conv[shot[l]] = conv ? 1 : 0;
                    a.iters[shot[l]] = (uint8_t)(conv ? t[l] - 1 : sp.max_iter);
                    grp_shot[l] = (int)atomicAdd(a.work, 1u);
                }
            }
        }

        // ---- variable pass: posterior of the variant, decision, eq. (v_update)/(mombp5) ----
        dec[0] = dec[1] = 0u;
#pragma unroll 1
        for (int j = tg; j < N; j += T) {
            float2 *sj = reinterpret_cast<float2 *>(slots) + j;
            float2 *st = state + j;
            const uint32_t used = FULL ? 15u : m.used[j];
            float2 win[4];
#pragma unroll
            for (int n = 0; n < 4; ++n) win[n] = sj[n * Np];
            // positions 0, 1: X-type edges (anticommute with Z and Y); 2, 3:
            // Z-type edges (with X and Y); unused slots hold 0
            const float2 SZ = add2(win[0], win[1]), SX = add2(win[2], win[3]);
            const float2 SY = add2(SX, SZ);
            float2 Q[3];
            if (VARIANT == BPQ_EWAINIT) {
                // eq. (EWAInit): Q^(t) = Pi^(t) + S, Pi^(t+1) = alpha Pi^(0) + (1-alpha) Q^(t)
                const float2 oma = f2(1.f - sp.alpha);
                Q[0] = add2(st[0], SX);
                Q[1] = add2(st[Np], SY);
                Q[2] = add2(st[2 * Np], SZ);
                st[0] = fma2(oma, Q[0], st[3 * Np]);
                st[Np] = fma2(oma, Q[1], st[4 * Np]);
                st[2 * Np] = fma2(oma, Q[2], st[5 * Np]);
            } else {
                const float2 S[3] = {SX, SY, SZ};
#pragma unroll
                for (int w = 0; w < 3; ++w) {
                    const float2 Pi = PairPrior<VARIANT>::copies == 2
                                          ? reinterpret_cast<const float2 *>(PiS)[w * Np + j]
                                          : f2(PiS[w * Np + j]);
                    if (VARIANT == BPQ_PLAIN) {
                        Q[w] = add2(Pi, S[w]);  // eq. (p_update)
                    } else if (VARIANT == BPQ_MOMENTUM) {
                        // momentum_g and momentum_q on both lanes
                        const float2 qp = st[w * Np], grad = sub2(sub2(qp, Pi), S[w]);
                        const float2 g = fma2(f2(sp.gamma), st[(3 + w) * Np], mul2(f2(1.f - sp.gamma), grad));
                        Q[w] = fma2(f2(-sp.alpha), g, qp);
                        st[w * Np] = Q[w];
                        st[(3 + w) * Np] = g;
                    } else {
                        // adagrad_gp, adagrad_G and adagrad_q on both lanes
                        const float2 qp = st[w * Np], G2 = st[(3 + w) * Np], gp = sub2(sub2(qp, Pi), S[w]);
                        const float2 acc = fma2(gp, gp, G2);
                        const float2 Gs = make_float2(t[0] >= 2 || sp.ada_from1 ? acc.x : G2.x,
                                                      t[1] >= 2 || sp.ada_from1 ? acc.y : G2.y);
                        const float2 den = add2(make_float2(sqrt_approx(Gs.x), sqrt_approx(Gs.y)), f2(sp.eps));
                        const float2 step = fma2(mul2(f2(-sp.alpha), gp), rcp2(den), qp), first = add2(Pi, S[w]);
                        Q[w] = make_float2(t[0] == 1 ? first.x : step.x, t[1] == 1 ? first.y : step.y);
                        st[w * Np] = Q[w];
                        st[(3 + w) * Np] = Gs;
                    }
                }
            }
            // hard decision per lane: I if all Q_W > 0, else the first minimum of
            // X, Y, Z; kept as whether it anticommutes with X (it is Y or Z) and
            // with Z (it is X or Y)
            const float2 mq = min2(Q[0], min2(Q[1], Q[2]));
            const bool some0 = !(mq.x > 0.f), some1 = !(mq.y > 0.f);
            const uint2 ax = make_uint2(some0 && Q[0].x != mq.x, some1 && Q[0].y != mq.y);
            const uint2 az = make_uint2(some0 && (Q[0].x == mq.x || Q[1].x == mq.x),
                                        some1 && (Q[0].y == mq.y || Q[1].y == mq.y));
            dec[0] = 4u * dec[0] + (ax.x + 2u * az.x);
            dec[1] = 4u * dec[1] + (ax.y + 2u * az.y);
            emit_v2c_pair<PHI, FULL>(sp.vclip, sj, Np, used, Q[0], Q[1], Q[2], mq, win, ax, az);
        }
        if (fin) restart(fin);  // finished lanes start their next shot from eq. (init)
        pair_sync<MODE>(G, bar_id);
        if (fin) {
#pragma unroll
            for (int l = 0; l < 2; ++l)
                if ((fin >> l) & 1u) {
                    shot[l] = grp_shot[l];
                    t[l] = 0;
                    load_syndrome(l);
                }
            if (shot[0] >= a.B && shot[1] >= a.B) break;
        }
        ++t[0];
        ++t[1];
    }
}

// One code per launch, two shots per thread: a persistent grid whose shot
// groups take shots from the global queue until the batch is exhausted.
template <int VARIANT, bool FULL, int MODE>
__global__ void __launch_bounds__(1024, 1) decode_pair_kernel(const DecodeArgs a) {
    extern __shared__ __align__(16) uint8_t smem[];
    int *grp_shot = reinterpret_cast<int *>(smem + 16);

    const int tid = threadIdx.x;
    const int T = MODE == kPairOne ? (int)blockDim.x : MODE == kPairWarps ? 32 : a.G * 32;
    const int G = MODE == kPairGroups ? a.G : T / 32;
    const int group = MODE == kPairOne ? 0 : tid / T;
    const int tg = MODE == kPairOne ? tid : tid - group * T;
    const int bar_id = 1 + group;
    const PairMem m = pair_mem<VARIANT, MODE>(a, smem, group);
    const PairOffsets o = pair_offsets(VARIANT, MODE != kPairGroups, a.M, a.n_pad);
    const uint32_t kZero = 4u * (uint32_t)a.n_pad;
#ifdef BPQ_DEBUG
    {
        const size_t need = (size_t)o.groups + (size_t)(blockDim.x / T) * a.group_bytes;
        const bool ok = need <= dynamic_smem_bytes() && a.n_pad >= a.N && a.slots_floats >= 4u * a.n_pad + 2u &&
                        a.group_bytes >= kPairVoteBytes + 8u * (a.slots_floats +
                                                               (uint32_t)StateArrays<VARIANT>::n * a.n_pad) &&
                        (a.off_var_pauli + (uint32_t)a.N <= a.table_bytes) && blockDim.x / T <= kMaxPairGroupsPerCta &&
                        (a.M > a.N ? a.M : a.N) <= kPairMaxNodes * T;
        if (!ok) {
            if (tid == 0) atomicExch(a.work + 1, kBoundsError);
            return;
        }
    }
#endif

    // ---- the CTA's tables, from the code's table in global memory ----
    float *PiS = reinterpret_cast<float *>(smem + o.prior);
    for (int i = tid; i < a.M; i += blockDim.x) {
        const uint2 s = __ldg(reinterpret_cast<const uint2 *>(a.table) + i);
        uint32_t sl[4] = {s.x & 0xFFFFu, s.x >> 16, s.y & 0xFFFFu, s.y >> 16};
        for (int n = 0; n < 4; ++n) {
            if (sl[n] == kNoSlot || !BPQ_IN_BOUNDS(sl[n], kZero, a.work + 1)) sl[n] = kZero;
        }
        if (MODE != kPairGroups)
            reinterpret_cast<uint4 *>(smem + o.idx)[i] = make_uint4(8u * sl[0], 8u * sl[1], 8u * sl[2], 8u * sl[3]);
        else
            reinterpret_cast<uint2 *>(smem + o.idx)[i] = make_uint2(sl[0] | (sl[1] << 16), sl[2] | (sl[3] << 16));
    }
    // the prior, and the initial messages of eq. (init), lambda(Pi^(0)) on
    // every edge: the one-shot kernel's variable pass with no incoming
    // messages (unused positions of padded qubits hold 0)
    {
        const ShotParams sp = shot_params<PhiForm<VARIANT>::value>(a, a.alpha);
        float *init = reinterpret_cast<float *>(smem + o.init);
        const float z4[4] = {0.f, 0.f, 0.f, 0.f};
        constexpr int PC = PairPrior<VARIANT>::copies;
        for (int j = tid; j < a.N; j += blockDim.x) {
            const uint32_t vp = __ldg(a.table + a.off_var_pauli + j);
            float P[3];
            prior_llr(a, j, P);
            for (int w = 0; w < 3; ++w)
                for (int c = 0; c < PC; ++c) PiS[PC * (w * a.n_pad + j) + c] = P[w];
            smem[o.used + j] = (uint8_t)(((vp & 3u) ? 1u : 0u) | ((vp & 12u) ? 2u : 0u) | ((vp & 48u) ? 4u : 0u) |
                                         ((vp & 192u) ? 8u : 0u));
            emit_v2c<false, true, PhiForm<VARIANT>::value, true, FULL>(a, sp, init, j, 0, 0, vp, P[0], P[1], P[2], z4,
                                                                      0u);
        }
        // the zero slot, and the unused positions (padded qubits), read 0 in both lanes
        float2 *slots = reinterpret_cast<float2 *>(m.slots);
        for (uint32_t s = (FULL ? kZero : 0u) + tg; s <= kZero; s += T) slots[s] = make_float2(0.f, 0.f);
    }
    __syncthreads();
    decode_pairs<VARIANT, FULL, MODE>(a, m, T, tg, G, bar_id, grp_shot + 2 * group);
}

}  // namespace dk

// The two-shots-per-thread kernels of one variant (split tables; FULL for
// tables without padding), by PairMode.
#define BPQ_DEFINE_PICK_PAIR(NAME, V, FULLV)                                             \
    DecodeKernelFn NAME(int mode) {                                                      \
        return mode == kPairOne     ? dk::decode_pair_kernel<V, FULLV, kPairOne>         \
               : mode == kPairWarps ? dk::decode_pair_kernel<V, FULLV, kPairWarps>       \
                                    : dk::decode_pair_kernel<V, FULLV, kPairGroups>;     \
    }

}  // namespace bpq
