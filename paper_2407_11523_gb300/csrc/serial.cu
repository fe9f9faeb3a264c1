// Host side of the serial-schedule decoders (serial_kernel.cuh) and the
// kernels with a whole warp per shot; narrower groups are instantiated in
// serial16.cu and serial8.cu.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>

#include "serial_kernel.cuh"

namespace bpq {
namespace sk {

namespace {
SerialKernelFn pick_trace(int variant, bool split) { BPQ_SERIAL_SWITCH(true, 32, 2) }
SerialKernelFn pick_decode(int variant, bool split) { BPQ_SERIAL_SWITCH(false, 32, 2) }
}  // namespace

SerialKernelFn pick_serial32(int variant, bool trace, bool split) {
    return trace ? pick_trace(variant, split) : pick_decode(variant, split);
}

}  // namespace sk

namespace {

// The ways to decode: lanes per shot, and the step table they use (32 lanes
// take two per qubit, hence the 16-qubit steps).
enum SerialMode { kSerial32 = 0, kSerial16 = 1, kSerial8 = 2 };
constexpr int kModeLanes[3] = {32, 16, 8}, kModeTable[3] = {0, 0, 1};

constexpr int kSerialStageWarps = 16;  // within every kernel's serial_max_warps

// Shared memory of a launch.
struct SerialShape {
    int lanes, warps;        // warps: that fit (0: not even one)
    size_t fixed, shot_bytes;
    uint32_t off_state, off_syn, off_qb, off_dec, shot_words;
    size_t smem(int n) const { return fixed + (size_t)n * (32 / lanes) * shot_bytes; }
};

SerialShape serial_shape(const bpq_tanner *t, int variant, int mode) {
    const SerialTable &s = t->serial[kModeTable[mode]];
    const uint32_t n_pad = (uint32_t)((t->N + 3) & ~3);
    SerialShape r;
    r.lanes = kModeLanes[mode];
    r.fixed = 128 + s.off_qubit + (size_t)(12 + (t->split ? 8 : 12)) * n_pad;
    // messages (and three constant slots) | state | syndrome words | qubit bytes
    r.off_state = ((uint32_t)s.slots + 3u + 3u) & ~3u;
    r.off_syn = r.off_state + (uint32_t)sk::serial_state_arrays(variant) * n_pad;
    r.off_qb = r.off_syn + (uint32_t)(((t->M + 31) / 32 + 3) & ~3);
    r.off_dec = r.off_qb + n_pad / 4;
    r.shot_words = r.off_dec + (sk::serial_state_arrays(variant) ? 0u : n_pad / 4);
    const size_t limit = 227 * 1024;
    auto warp_bytes = [&](uint32_t words) { return (32 / r.lanes) * 4 * (size_t)words; };
    if (r.lanes < 32) {
        // the shots of a warp `lanes` banks apart, unless that keeps the only warp out
        const uint32_t spread = r.shot_words + (uint32_t)(r.lanes - (int)(r.shot_words % 32) + 32) % 32;
        if (r.fixed + warp_bytes(spread) <= limit) r.shot_words = spread;
    }
    r.shot_bytes = 4 * (size_t)r.shot_words;
    r.warps = r.fixed + warp_bytes(r.shot_words) > limit
                  ? 0
                  : (int)std::min<size_t>(sk::serial_max_warps(r.lanes), (limit - r.fixed) / warp_bytes(r.shot_words));
    return r;
}

// The mode of a batch: the least of an estimate of its time, for ten sweeps a
// shot and a slowest shot that runs max_iter, from figures measured on GB300: a
// step costs a warp about 190 issue slots with two lanes per qubit and 290
// with one (shared by the warp's shots), and 480 or 660 cycles when the warp has
// its scheduler to itself; a scheduler issues 0.28 slots a cycle per resident
// warp, 0.85 at most.  So narrow groups are for small codes, whose shots fit
// shared memory many times, in large batches.  Measured, 32 / 16 / 8 lanes per
// shot (ms, EWAInit): planar d = 7, 10^6 shots 7.30 / 6.02 / 4.33, 10^5 1.11 /
// 1.10 / 1.04, 20000 0.51 / 0.58 / 0.65; planar d = 11, 10^5 3.19 / 2.86 / 2.89;
// toric d = 10, 10^5 1.78 / 1.75 / 1.96; toric d = 15, 10^6 24.0 / 25.1 / 45.5;
// planar d = 25, 20000 5.8 / 7.1 / 14.5.  (A warp per shot on the dependency
// levels, one lane per qubit, took 10.2, 1.68, 0.76, 4.77, 2.64, 30.1, 6.57.)
int serial_mode(const bpq_tanner *t, int variant, int max_iter, int B) {
    if (t->serial_shots_per_warp) return t->serial_shots_per_warp == 1 ? kSerial32 : kSerial16;
    int best = kSerial32;
    double least = 0;
    for (int mode = kSerial32; mode <= kSerial8; ++mode) {
        const SerialShape s = serial_shape(t, variant, mode);
        if (s.warps < 1) continue;
        const double steps = t->serial[kModeTable[mode]].steps, per_warp = 32 / s.lanes;
        const double busy = std::min<double>(s.warps, std::ceil(B / (per_warp * t->num_sms)));
        const double slots = steps * (mode == kSerial32 ? 190 : 290 / per_warp);
        const double cycles = 10.0 * B * slots / (std::min(0.85, 0.07 * busy) * 4 * t->num_sms) +
                              max_iter * steps * (mode == kSerial32 ? 480 : 660);
        if (mode == kSerial32 || cycles < least) {
            best = mode;
            least = cycles;
        }
    }
    return best;
}

// Validate, fill the arguments from the parallel decoder's (parameters in
// the kernel's units) and launch.
int serial_launch(const bpq_tanner *t, const uint32_t *syn, const float *prior, int variant, const bpq_params *params,
                  int max_iter, int B, void *work, bool trace, uint8_t *est, uint8_t *conv, uint8_t *iters,
                  float *tr_v2c, float *tr_c2v, float *tr_Q, uint8_t *tr_dec, cudaStream_t st) {
    int rc = need_uploaded(t);
    if (rc) return rc;
    if (variant < BPQ_PLAIN || variant > BPQ_EWAINIT)
        return fail(BPQ_EINVAL, "the serial schedule takes plain, Momentum, AdaGrad or EWAInit BP");
    DecodeArgs d;
    rc = fill_decode_args(t, syn, prior, variant, params, max_iter, B, work, d);
    if (rc) return rc;
    if (B == 0) return BPQ_OK;
    if (!trace && (!est || !conv || !iters)) return fail(BPQ_EINVAL, "NULL output");
    const int mode = trace ? kSerial32 : serial_mode(t, variant, max_iter, B);
    const SerialTable &s = t->serial[kModeTable[mode]];
    const SerialShape shape = serial_shape(t, variant, mode);
    if (shape.warps < 1)
        return fail(BPQ_EINVAL, mode == kSerial32 ? "code too large for the serial kernel's shared memory"
                                           : "two shots per warp do not fit in shared memory for this code");
    SerialArgs a;
    std::memset(&a, 0, sizeof a);
    a.table = t->d_serial[kModeTable[mode]];
    a.table_bytes = s.off_qubit;
    a.off_meta = s.off_meta;
    a.off_steps = s.off_steps;
    a.off_qubit = s.off_qubit;
    a.off_chk = s.off_chk;
    a.off_canon = s.off_canon;
    a.nsteps = s.steps;
    a.syn = syn;
    a.prior = prior;
    a.est = est;
    a.conv = conv;
    a.iters = iters;
    a.work = static_cast<uint32_t *>(work);
    a.tr_v2c = tr_v2c;
    a.tr_c2v = tr_c2v;
    a.tr_Q = tr_Q;
    a.tr_dec = tr_dec;
    a.N = t->N;
    a.M = t->M;
    a.E = t->E;
    a.W = (t->M + 31) / 32;
    a.B = B;
    a.max_iter = max_iter;
    a.n_pad = (t->N + 3) & ~3;
    a.zero_slot = (uint32_t)s.slots;
    a.shot_words = shape.shot_words;
    a.off_state = shape.off_state;
    a.off_syn = shape.off_syn;
    a.off_qb = shape.off_qb;
    a.off_dec = shape.off_dec;
    a.alpha = d.alpha;
    a.gamma = d.gamma;
    a.eps = d.eps;
    a.clip = d.clip;
    a.clip2 = d.clip2;
    a.delta_clip = d.delta_clip;
    a.phi_clip = d.phi_clip;
    a.ada_from1 = d.ada_from1;

    // small batches: spread over the SMs instead of filling the first ones
    const long per_warp = 32 / shape.lanes, wave = per_warp * t->num_sms;
    const int warps = (int)std::min<long>(shape.warps, (B + wave - 1) / wave);
    const size_t smem = shape.smem(warps);
    // the further warps of SerialHelpers
    a.warps = warps;
    const int threads =
        32 * (variant == BPQ_ADAGRAD ? warps : std::max(warps, std::min(kSerialStageWarps, (t->N + 31) / 32)));
    sk::SerialKernelFn fn = mode == kSerial32   ? sk::pick_serial32(variant, trace, t->split)
                            : mode == kSerial16 ? sk::pick_serial16(variant, t->split)
                                                : sk::pick_serial8(variant, t->split);
    if (!fn) return fail(BPQ_EINVAL, "no serial kernel for this variant");
    rc = allow_smem(fn, kMaxDynamicSmem, "cudaFuncSetAttribute");
    if (rc) return rc;
    int per_sm = 0;
    cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, threads, smem);
    if (e != cudaSuccess || per_sm < 1) return fail(BPQ_ECUDA, "serial kernel does not fit on an SM");
    long ctas = (long)per_sm * t->num_sms;
    const long per_cta = warps * per_warp;
    const long need = (B + per_cta - 1) / per_cta;
    if (ctas > need) ctas = need;
    rc = cuda_check(cudaMemsetAsync(work, 0, 8, st), "workspace reset");
    if (rc) return rc;
    fn<<<(unsigned)std::max(1L, ctas), threads, smem, st>>>(a);
    return cuda_check(cudaGetLastError(), "serial decode launch");
}

}  // namespace
}  // namespace bpq

using bpq::fail;

extern "C" {

int bpq_decode_serial(const bpq_tanner *t, const uint32_t *syn_dev, const float *prior_dev, int variant,
                      const bpq_params *params, int max_iter, int B, uint8_t *est_dev, uint8_t *conv_dev,
                      uint8_t *iters_dev, void *work_dev, void *stream) {
    return bpq::serial_launch(t, syn_dev, prior_dev, variant, params, max_iter, B, work_dev, false, est_dev, conv_dev,
                              iters_dev, nullptr, nullptr, nullptr, nullptr, static_cast<cudaStream_t>(stream));
}

int bpq_set_serial_shots_per_warp(bpq_tanner *t, int shots_per_warp) {
    if (!t) return fail(BPQ_EINVAL, "tanner is NULL");
    if (shots_per_warp < 0 || shots_per_warp > 2) return fail(BPQ_EINVAL, "shots per warp must be 0, 1 or 2");
    t->serial_shots_per_warp = shots_per_warp;
    return BPQ_OK;
}

int bpq_decode_serial_trace(const bpq_tanner *t, const uint32_t *syn_dev, const float *prior_dev, int variant,
                            const bpq_params *params, int T, int B, float *m_v2c_dev, float *m_c2v_dev, float *Q_dev,
                            uint8_t *dec_dev, void *work_dev, void *stream) {
    return bpq::serial_launch(t, syn_dev, prior_dev, variant, params, T, B, work_dev, true, nullptr, nullptr, nullptr,
                              m_v2c_dev, m_c2v_dev, Q_dev, dec_dev, static_cast<cudaStream_t>(stream));
}

}  // extern "C"
