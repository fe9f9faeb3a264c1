// C-ABI entry points of libbpq (declared in include/bpq.h): device upload of
// the Tanner graph, the Philox Pauli-channel sampler, argument checking and
// launch of the decoder, the logical-failure classifier.
#include <cuda_runtime.h>

#include <cmath>
#include <cstring>
#include <mutex>
#include <new>

#include "bpq_internal.h"
#include "decode_launch.h"

using bpq::fail;

namespace bpq {
namespace {

// ---------------------------------------------------------------- Philox4x64-10
// Salmon, Moraes, Dror, Shaw, "Parallel random numbers: as easy as 1, 2, 3"
// (SC 2011): 10 rounds of two 64x64->128 multiplications, Weyl key schedule.
// One round maps (x0, x1, x2, x3) to (hi(M1 x2) ^ x1 ^ k0, lo(M1 x2),
// hi(M0 x0) ^ x3 ^ k1, lo(M0 x0)).  The counter is (shot, block, 0, 0), so
// with one shot per lane the products of the first three rounds that do not
// see the block (round 0: M0 shot; round 1: M1 x2; round 2: M0 x0) are the
// same for all blocks of the shot and are computed once (PhiloxShot).
constexpr uint64_t kPhiloxM0 = 0xD2E7470EE14C6C93ULL, kPhiloxM1 = 0xCA5A826395121157ULL;
constexpr uint64_t kPhiloxW0 = 0x9E3779B97F4A7C15ULL, kPhiloxW1 = 0xBB67AE8584CAA73BULL;

// 64 x 64 -> 128 bit product (both halves from one expression: the compiler
// shares the partial products; a chain of 32 x 32 -> 64 multiply-adds written
// out was a third slower).
__device__ __forceinline__ void mul_wide64(uint64_t a, uint64_t m, uint64_t &hi, uint64_t &lo) {
    hi = __umul64hi(a, m);
    lo = a * m;
}

struct PhiloxShot {
    uint64_t lo_shot;          // lo(M0 shot): x3 after round 0
    uint64_t x1_r1;            // x1 after round 1
    uint64_t hi0_r2, lo0_r2;   // M0 x0 of round 2
};

__device__ __forceinline__ PhiloxShot philox_shot(uint64_t shot, uint64_t seed) {
    PhiloxShot s;
    uint64_t hi;
    mul_wide64(shot, kPhiloxM0, hi, s.lo_shot);          // round 0 (keys seed, 0): x2 = hi
    uint64_t hi1;
    mul_wide64(hi, kPhiloxM1, hi1, s.x1_r1);             // round 1: x0 = hi1 ^ 0 ^ (seed + W0)
    mul_wide64(hi1 ^ (seed + kPhiloxW0), kPhiloxM0, s.hi0_r2, s.lo0_r2);
    return s;
}

// The four words of `block` of the shot.
__device__ __forceinline__ void philox_block(const PhiloxShot &s, uint64_t block, uint64_t seed, uint64_t (&u)[4]) {
    uint64_t hi, lo;
    // round 0: x0 = block ^ seed; round 1: x2 = hi(M0 x0) ^ lo_shot ^ W1, x3 = lo(M0 x0)
    mul_wide64(block ^ seed, kPhiloxM0, hi, lo);
    const uint64_t x2r1 = hi ^ s.lo_shot ^ kPhiloxW1, x3r1 = lo;
    // round 2
    mul_wide64(x2r1, kPhiloxM1, hi, lo);
    uint64_t x0 = hi ^ s.x1_r1 ^ (seed + 2 * kPhiloxW0), x1 = lo;
    uint64_t x2 = s.hi0_r2 ^ x3r1 ^ (2 * kPhiloxW1), x3 = s.lo0_r2;
#pragma unroll
    for (int r = 3; r < 10; ++r) {
        uint64_t h0, l0, h1, l1;
        mul_wide64(x0, kPhiloxM0, h0, l0);
        mul_wide64(x2, kPhiloxM1, h1, l1);
        x0 = h1 ^ x1 ^ (seed + (uint64_t)r * kPhiloxW0);
        x1 = l1;
        x2 = h0 ^ x3 ^ ((uint64_t)r * kPhiloxW1);
        x3 = l0;
    }
    u[0] = x0;
    u[1] = x1;
    u[2] = x2;
    u[3] = x3;
}

// Transpose of a 32 x 32 bit matrix held one row per lane: bit c of lane r
// becomes bit r of lane c.
__device__ __forceinline__ uint32_t warp_transpose32(uint32_t x, int lane) {
    constexpr uint32_t mask[5] = {0x0000FFFFu, 0x00FF00FFu, 0x0F0F0F0Fu, 0x33333333u, 0x55555555u};
#pragma unroll
    for (int s = 0; s < 5; ++s) {
        const int k = 16 >> s;
        const uint32_t y = __shfl_xor_sync(0xffffffffu, x, k);
        x = (lane & k) ? (x & ~mask[s]) | ((y & ~mask[s]) >> k) : (x & mask[s]) | ((y & mask[s]) << k);
    }
    return x;
}

// Which planes of a qubit's two-bit code enter <., p>: the code's parity
// with mask m(p), m(X) = 2, m(Y) = 1, m(Z) = 3 (codes 0 I, 1 X, 2 Y, 3 Z: bit
// 1 is the Z part, bit 0 ^ bit 1 the X part), on words of 32 shots.
__device__ __forceinline__ uint32_t anti_word(uint2 c, uint32_t p) {
    return (p == 2u || p == 3u ? c.x : 0u) ^ (p == 1u || p == 3u ? c.y : 0u);
}

// XOR over a check's qubits of anti_word (planes: one uint2 per qubit).
__device__ __forceinline__ uint32_t check_word(const uint16_t *chk_slot, const uint8_t *chk_pauli, int i,
                                               const uint2 *planes) {
    const uint32_t cp = chk_pauli[i];
    const uint2 s = *reinterpret_cast<const uint2 *>(chk_slot + 4 * i);
    const uint32_t sl[4] = {s.x & 0xFFFFu, s.x >> 16, s.y & 0xFFFFu, s.y >> 16};
    uint32_t w = 0;
#pragma unroll
    for (int n = 0; n < 4; ++n)
        if (sl[n] != kNoSlot) {
            const uint32_t p = (cp >> (2 * n)) & 3u;
            const uint2 c = planes[sl[n] >> 2];
            w ^= p == 2u ? c.x : p == 1u ? c.y : c.x ^ c.y;
        }
    return w;
}

// Errors and syndromes of 32 consecutive shots per CTA.  Lane s of every warp
// is shot s; the warps share the shot's blocks of four qubits.  A block's codes go to
// shared memory one word per (shot, block), and warp votes turn them into bit
// planes (one word per qubit and code bit, bit s = shot s), from which a
// thread forms one check's syndrome for all 32 shots with four loads; 32 x 32
// bit transposes give the packed words.  Errors and syndromes of the tile are
// contiguous in memory and leave in 32-bit stores.
// Bound: the Philox multiplications (15 of the 20 per block are left per
// shot).  The two kernels this replaces (errors, then syndromes from the errors
// in memory, a byte load per edge) took 305 + 431 us for 10^6 planar d = 7 shots.
// Shared memory: codes [32][cw] | planes uint2[N] | syn [32][W].
__global__ void sample_kernel(const uint16_t *chk_slot, const uint8_t *chk_pauli, int N, int M, int W, int B,
                              uint64_t seed, uint64_t shot0, uint64_t tx, uint64_t ty, uint64_t tz, uint8_t *err,
                              uint32_t *syn) {
    extern __shared__ __align__(16) uint8_t smem[];
    const int nblk = (N + 3) / 4, cw = nblk | 1;  // odd row stride: lanes (shots) hit distinct banks
    uint32_t *codes = reinterpret_cast<uint32_t *>(smem);
    uint2 *planes = reinterpret_cast<uint2 *>(codes + 32 * cw);
    uint32_t *words = reinterpret_cast<uint32_t *>(planes + N);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    const long b0 = 32L * blockIdx.x;
    const int cnt = B - b0 < 32 ? (int)(B - b0) : 32;

    const PhiloxShot ps = philox_shot(shot0 + (uint64_t)(b0 + lane), seed);
    for (int blk = warp; blk < nblk; blk += nwarps) {
        uint64_t u[4];
        philox_block(ps, (uint64_t)blk, seed, u);
        uint32_t word = 0;
        uint2 mine = make_uint2(0u, 0u);
#pragma unroll
        for (int l = 0; l < 4; ++l) {
            // thresholds tx <= ty <= tz: X below tx, Y below ty, Z below tz
            const bool bx = u[l] < tx, by = u[l] < ty, bz = u[l] < tz;
            const uint32_t code = bx ? 1u : by ? 2u : bz ? 3u : 0u;
            word |= code << (8 * l);
            // bit 0 of the code: X or Z; bit 1: Y or Z
            const uint32_t vx = __ballot_sync(0xffffffffu, bx), vy = __ballot_sync(0xffffffffu, by),
                           vz = __ballot_sync(0xffffffffu, bz);
            if (lane == l) mine = make_uint2(vx | (vz & ~vy), vz & ~vx);
        }
        codes[lane * cw + blk] = word;
        if (lane < 4 && 4 * blk + lane < N) planes[4 * blk + lane] = mine;
    }
    __syncthreads();

    for (int i0 = 32 * warp; i0 < M; i0 += 32 * nwarps) {
        const int i = i0 + lane;
        const uint32_t w = warp_transpose32(i < M ? check_word(chk_slot, chk_pauli, i, planes) : 0u, lane);
        words[lane * W + (i0 >> 5)] = w;
    }
    // the tile's errors: byte o is qubit o % N of shot o / N (o < 2^16 and
    // N <= 2^11, so the product with ceil(2^32 / N) gives o / N exactly)
    uint8_t *e = err + b0 * N;
    const uint8_t *cb = reinterpret_cast<const uint8_t *>(codes);
    const uint32_t inv = 0xFFFFFFFFu / (uint32_t)N + 1u;
    const int bytes = cnt * N;
    int done = 0;
    if ((reinterpret_cast<uintptr_t>(e) & 3u) == 0 && N >= 4) {
        done = bytes & ~3;
        for (int o = 4 * threadIdx.x; o < done; o += 4 * blockDim.x) {
            const int s = (int)__umulhi((uint32_t)o, inv), j = o - s * N;
            const uint32_t *row = codes + s * cw + (j >> 2);
            uint32_t v = __funnelshift_r(row[0], row[1], 8 * (j & 3));
            const int left = N - j;  // codes of this shot from j on
            if (left < 4) v = (v & ((1u << (8 * left)) - 1u)) | (codes[(s + 1) * cw] << (8 * left));
            *reinterpret_cast<uint32_t *>(e + o) = v;
        }
    }
    for (int o = done + threadIdx.x; o < bytes; o += blockDim.x) {
        const int s = o / N;
        e[o] = cb[4 * s * cw + (o - s * N)];
    }
    __syncthreads();
    for (int k = threadIdx.x; k < cnt * W; k += blockDim.x) syn[b0 * W + k] = words[k];
}

// The same for few shots: one CTA per shot, whose threads draw blocks of four
// qubits and then test a check each.  sample_kernel gives a shot one lane, so few
// shots leave most of the chip idle and a large code's blocks follow one another
// (planar d = 31, 1 to 2000 shots: 36 us whatever the number).  Bound: the launch,
// then the Philox chain.  Errors and syndromes, us a call, tile kernel / this:
// planar d = 31, 40 shots 36 / 9.3, 1500 37 / 25.6, 2000 37 / 34, 3000 37 / 47;
// planar d = 18, 300 15 / 8.7, 1500 15.4 / 12.8, 2000 15.4 / 15.3, 3000 15.4 /
// 21; codes of up to 200 qubits the same up to 3000 shots (8.5).
__global__ void sample_shot_kernel(const uint16_t *chk_slot, const uint8_t *chk_pauli, int N, int M, int W,
                                   uint64_t seed, uint64_t shot0, uint64_t tx, uint64_t ty, uint64_t tz, uint8_t *err,
                                   uint32_t *syn) {
    __shared__ uint32_t codes[kMaxNodes / 4];  // one code per byte
    const int nblk = (N + 3) / 4;
    const PhiloxShot ps = philox_shot(shot0 + blockIdx.x, seed);
    for (int blk = threadIdx.x; blk < nblk; blk += blockDim.x) {
        uint64_t u[4];
        philox_block(ps, (uint64_t)blk, seed, u);
        uint32_t word = 0;
#pragma unroll
        for (int l = 0; l < 4; ++l) word |= (u[l] < tx ? 1u : u[l] < ty ? 2u : u[l] < tz ? 3u : 0u) << (8 * l);
        codes[blk] = word;
    }
    __syncthreads();
    const uint8_t *code = reinterpret_cast<const uint8_t *>(codes);
    uint8_t *e = err + (size_t)blockIdx.x * N;
    for (int j = threadIdx.x; j < N; j += blockDim.x) e[j] = code[j];
    for (int i0 = threadIdx.x & ~31; i0 < M; i0 += blockDim.x) {
        const int i = i0 + (threadIdx.x & 31);
        uint32_t odd = 0;
        if (i < M) {
            const uint32_t cp = chk_pauli[i];
            const uint2 s = *reinterpret_cast<const uint2 *>(chk_slot + 4 * i);
            const uint32_t sl[4] = {s.x & 0xFFFFu, s.x >> 16, s.y & 0xFFFFu, s.y >> 16};
#pragma unroll
            for (int n = 0; n < 4; ++n) {
                const uint32_t p = (cp >> (2 * n)) & 3u;  // the mask of anti_word: 2, 1, 3 for X, Y, Z
                if (sl[n] != kNoSlot) odd ^= __popc(code[sl[n] >> 2] & (p == 3u ? 3u : 3u - p));
            }
        }
        const uint32_t word = __ballot_sync(0xffffffffu, odd & 1u);
        if ((threadIdx.x & 31) == 0) syn[(size_t)blockIdx.x * W + (i0 >> 5)] = word;
    }
}
// Batches of at most this many shots per SM (1824 on a GB300) take it.
constexpr long kSampleShotsPerSm = 12;

// Bytes of shared memory of sample_kernel (W words of 32 checks): grows with N and W.
constexpr size_t sample_smem(int N, int W) {
    return 4 * (size_t)32 * (((N + 3) / 4) | 1) + 8 * (size_t)N + 4 * (size_t)32 * W;
}

// Four codes, one per byte; values above 3 (no Pauli code) count as I.
__device__ __forceinline__ uint32_t valid_codes(uint32_t v) {
    const uint32_t bad = v & 0xFCFCFCFCu;
    if (bad == 0) return v;
    uint32_t r = 0;
    for (int l = 0; l < 4; ++l)
        if (!((bad >> (8 * l)) & 0xFFu)) r |= v & (0xFFu << (8 * l));
    return r;
}

constexpr int check_logical_stride(int N) { return N % 4 ? N : 4 * ((N / 4) | 1); }
// (no N below kMaxNodes = 2048 takes more than 2048 does)
constexpr size_t check_logical_smem(int N) {
    return (((size_t)32 * check_logical_stride(N) + 7) & ~size_t(7)) + 8 * (size_t)N + 8;
}

// Classification of 32 consecutive shots per CTA: residual R = E^ E; 1 if R
// anticommutes with a check, 2 if it commutes with all checks but not with all
// logical operators.  The codes of a product are the XOR of the codes, so the
// tile's residuals are the XOR of the two arrays, read once in 32-bit words;
// warp votes turn them into bit planes (bit s of a qubit's word = shot s), and
// a thread then tests one check for all 32 shots with four loads.
// Bound: the tile's passes through shared memory; one warp per shot with
// byte loads per edge took 775 us for 10^6 planar d = 7 shots; this takes
// 104 us (174 MB of memory traffic).
// Shared memory: residuals, 32 rows of `stride` bytes | planes uint2[N] | two
// words.  Rows are contiguous as in memory when N is no multiple of 4, else
// padded to an odd number of words (lanes read the same qubit of 32 rows).
__global__ void check_logical_kernel(const uint16_t *chk_slot, const uint8_t *chk_pauli, const uint8_t *logicals,
                                     int nlog, int N, int M, int B, int stride, const uint8_t *err,
                                     const uint8_t *est, uint8_t *fail_out) {
    extern __shared__ __align__(16) uint8_t smem[];
    uint2 *planes = reinterpret_cast<uint2 *>(smem + ((32 * stride + 7) & ~7));
    uint32_t *verdict = reinterpret_cast<uint32_t *>(planes + N);  // [0] detected, [1] logical (bit = shot)
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    const long b0 = 32L * blockIdx.x;
    const int cnt = B - b0 < 32 ? (int)(B - b0) : 32;
    const uint8_t *e = err + b0 * N, *h = est + b0 * N;
    if (threadIdx.x < 2) verdict[threadIdx.x] = 0u;
    const int bytes = cnt * N;
    const bool words = ((reinterpret_cast<uintptr_t>(e) | reinterpret_cast<uintptr_t>(h)) & 3u) == 0;
    const int done = words ? bytes & ~3 : 0;
    for (int o = 4 * threadIdx.x; o < done; o += 4 * blockDim.x) {
        const uint32_t r = valid_codes(__ldg(reinterpret_cast<const uint32_t *>(e + o))) ^
                           valid_codes(__ldg(reinterpret_cast<const uint32_t *>(h + o)));
        const int at = stride == N ? o : (o / N) * stride + o % N;  // padded rows: N and stride multiples of 4
        *reinterpret_cast<uint32_t *>(smem + at) = r;
    }
    for (int o = done + threadIdx.x; o < bytes; o += blockDim.x) {
        const int s = o / N;
        smem[s * stride + (o - s * N)] = (uint8_t)(valid_codes(e[o]) ^ valid_codes(h[o]));
    }
    __syncthreads();
    const uint8_t *row = smem + (lane < cnt ? lane : 0) * stride;
    for (int j0 = 32 * warp; j0 < N; j0 += 32 * nwarps) {
        uint2 mine = make_uint2(0u, 0u);
        const int n = N - j0 < 32 ? N - j0 : 32;
        for (int l = 0; l < n; ++l) {
            const uint32_t c = row[j0 + l];
            const uint32_t p0 = __ballot_sync(0xffffffffu, c & 1u), p1 = __ballot_sync(0xffffffffu, c & 2u);
            if (lane == l) mine = make_uint2(p0, p1);
        }
        if (lane < n) planes[j0 + lane] = mine;
    }
    __syncthreads();
    uint32_t det = 0;
    for (int i = threadIdx.x; i < M; i += blockDim.x) det |= check_word(chk_slot, chk_pauli, i, planes);
    det = __reduce_or_sync(0xffffffffu, det);
    if (lane == 0 && det) atomicOr(verdict, det);
    for (int l = warp; l < nlog; l += nwarps) {
        uint32_t par = 0;
        for (int j = lane; j < N; j += 32) par ^= anti_word(planes[j], logicals[(size_t)l * N + j]);
        par = __reduce_xor_sync(0xffffffffu, par);
        if (lane == 0 && par) atomicOr(verdict + 1, par);
    }
    __syncthreads();
    if (warp == 0 && lane < cnt)
        fail_out[b0 + lane] = ((verdict[0] >> lane) & 1u) ? 1 : ((verdict[1] >> lane) & 1u) ? 2 : 0;
}


// Peak probes: `iters` rounds of 8 independent dependency chains per thread of
// either MUFU.EX2 (x <- 2^-x, stays in [0.5, 1)) or FFMA.
__global__ void probe_kernel(int which, int iters, float *sink) {
    float x[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) x[k] = 0.25f + 0.01f * k + 1e-6f * threadIdx.x;
    if (which == 0) {
        for (int it = 0; it < iters; ++it) {
#pragma unroll
            for (int k = 0; k < 8; ++k) asm volatile("ex2.approx.ftz.f32 %0, %1;" : "=f"(x[k]) : "f"(-x[k]));
        }
    } else {
        const float a = 0.999f, b = 0.001f;
        for (int it = 0; it < iters; ++it) {
#pragma unroll
            for (int k = 0; k < 8; ++k) x[k] = fmaf(x[k], a, b);
        }
    }
    float s = 0.f;
#pragma unroll
    for (int k = 0; k < 8; ++k) s += x[k];
    if (s == 12345.678f) sink[0] = s;  // keeps the chains live
}

uint64_t threshold(double c) {
    if (c <= 0.0) return 0;
    return (uint64_t)std::ldexp(c, 64);
}

int launch_grid(long items, int per_block) {
    const long g = (items + per_block - 1) / per_block;
    return (int)(g < 1 ? 1 : g);
}

// Warps of a CTA that works on a tile of 32 shots in `units` equal steps (32
// threads each): about six steps a warp where there are tiles for every SM
// (the tile's barriers and per-warp set-up cost less then), one step a warp
// while the tiles leave SMs idle.
int tile_warps(const bpq_tanner *t, int B, int units) {
    const long tiles = (B + 31L) / 32;
    const int most = units < 1 ? 1 : units > 16 ? 16 : units;
    if (tiles < 4L * t->num_sms) return most;
    const int w = (units + 5) / 6;
    return w < 4 ? (most < 4 ? most : 4) : w > 16 ? 16 : w;
}

// ---------------------------------------------------------------- no-allocation staging
// Device memory for bpq_decode_host_noalloc: a fixed array in the library's
// own image, so that callers that cannot allocate device memory can still
// decode.  It is created when the library is loaded on a device and held
// until the process exits.
constexpr size_t kNoAllocBytes = size_t(8) << 20;
static __device__ __align__(256) uint8_t g_noalloc_scratch[kNoAllocBytes];

constexpr int kMaxDevices = 64;
std::mutex g_noalloc_mu;
void *g_noalloc_ptr[kMaxDevices] = {};

// Device address of g_noalloc_scratch on `device` (which must be current).
// In host code the symbol's name is only a host-side stand-in, so its device
// address is looked up once per device and cached.
int noalloc_scratch(int device, void **out) {
    if (device < 0 || device >= kMaxDevices) return fail(BPQ_EINVAL, "device index out of range");
    std::lock_guard<std::mutex> lock(g_noalloc_mu);
    if (!g_noalloc_ptr[device]) {
        void *p = nullptr;
        cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
        if (e != cudaSuccess || !p)
            return fail(BPQ_ECUDA, std::string("cudaGetSymbolAddress: ") + cudaGetErrorString(e));
        g_noalloc_ptr[device] = p;
    }
    *out = g_noalloc_ptr[device];
    return BPQ_OK;
}

}  // namespace

int need_uploaded(const bpq_tanner *t) {
    if (!t) return fail(BPQ_EINVAL, "tanner is NULL");
    if (!t->dev_blob) return fail(BPQ_ESTATE, "tanner not uploaded to a device");
    cudaError_t e = cudaSetDevice(t->device);
    if (e != cudaSuccess) return fail(BPQ_ECUDA, std::string("cudaSetDevice: ") + cudaGetErrorString(e));
    return BPQ_OK;
}

int cuda_check(cudaError_t e, const char *what) {
    if (e == cudaSuccess) return BPQ_OK;
    return fail(BPQ_ECUDA, std::string(what) + ": " + cudaGetErrorString(e));
}

// 1 - tanh(c/2) = 2 / (e^c + 1): the smallest delta of a message clipped to |m| <= c
float delta_of_clip(float c) { return (float)(2.0 / (std::exp((double)c) + 1.0)); }
// phi(c) = log1p(2 / expm1(c)) = -ln tanh(c/2): the smallest phi of a clipped message
float phi_of_clip(float c) { return (float)std::log1p(2.0 / std::expm1((double)c)); }

int check_params(int variant, const bpq_params *params, bpq_params *out) {
    if (variant < BPQ_PLAIN || variant > BPQ_AEWA) return fail(BPQ_EINVAL, "unknown variant");
    if (params) *out = *params;
    else bpq_default_params(variant, out);
    if (!(out->msg_clip > 0.0f && out->msg_clip <= 80.0f)) return fail(BPQ_EINVAL, "msg_clip must be in (0, 80]");
    if (!std::isfinite(out->alpha) || !std::isfinite(out->gamma) || !std::isfinite(out->eps) || out->eps < 0.0f)
        return fail(BPQ_EINVAL, "non-finite parameter");
    return BPQ_OK;
}

int fill_decode_args(const bpq_tanner *t, const uint32_t *syn, const float *prior, int variant,
                     const bpq_params *params, int max_iter, int B, void *work, DecodeArgs &a) {
    bpq_params p;
    int rc = check_params(variant, params, &p);
    if (rc) return rc;
    if (B < 0) return fail(BPQ_EINVAL, "B < 0");
    if (max_iter < 1 || max_iter > 255) return fail(BPQ_EINVAL, "max_iter must be in [1, 255]");
    if (B > 0 && (!syn || !prior || !work)) return fail(BPQ_EINVAL, "NULL input or workspace");
    if (misaligned(work, kBufferAlign)) return fail(BPQ_EINVAL, "workspace not 16-byte aligned");
    if (misaligned(syn, kWordAlign) || misaligned(prior, kWordAlign))
        return fail(BPQ_EINVAL, "syndromes or priors not 4-byte aligned");
    std::memset(&a, 0, sizeof a);
    a.split = t->full ? 2 : t->split ? 1 : 0;
    a.table = t->split ? t->d_table_split : t->d_table;
    a.table_bytes = (uint32_t)t->table.size();
    a.off_chk_pauli = t->off_chk_pauli;
    a.off_var_pauli = t->off_var_pauli;
    a.syn = syn;
    a.prior = prior;
    a.work = static_cast<uint32_t *>(work);
    a.var_canon = t->split ? t->d_var_canon_split : t->d_var_canon;
    a.chk_ptr = t->d_chk_ptr;
    a.N = t->N;
    a.M = t->M;
    a.E = t->E;
    a.W = (t->M + 31) / 32;
    a.B = B;
    a.max_iter = max_iter;
    // the kernel keeps log-likelihoods in bits: AdaGrad's step alpha and eps
    // are log-likelihoods too, the EWA and momentum weights are pure numbers
    const float log2e = 1.4426950408889634f;
    a.alpha = variant == BPQ_ADAGRAD ? p.alpha * log2e : p.alpha;
    a.gamma = p.gamma;
    a.eps = p.eps * log2e;
    a.clip = p.msg_clip;
    a.clip2 = p.msg_clip * log2e;
    a.delta_clip = delta_of_clip(p.msg_clip);
    a.phi_clip = phi_of_clip(p.msg_clip);
    a.ada_from1 = p.adagrad_g_from_iter1 ? 1 : 0;
    return BPQ_OK;
}

int cuda_set_device(int device) {
    cudaError_t e = cudaSetDevice(device);
    if (e != cudaSuccess) return fail(BPQ_ECUDA, std::string("cudaSetDevice: ") + cudaGetErrorString(e));
    return BPQ_OK;
}

// Copy streams of one device for the pipelined host path (created on first
// use, kept for the life of the process).
struct HostPipe {
    cudaStream_t h2d = nullptr, d2h = nullptr, comp = nullptr;
};
std::mutex g_pipe_mu;
HostPipe g_pipe[64];

int host_pipe(int device, HostPipe **out) {
    if (device < 0 || device >= 64) return fail(BPQ_EINVAL, "device index out of range");
    std::lock_guard<std::mutex> lock(g_pipe_mu);
    HostPipe &hp = g_pipe[device];
    if (!hp.h2d) {
        int rc = cuda_check(cudaStreamCreateWithFlags(&hp.h2d, cudaStreamNonBlocking), "copy stream");
        if (rc) return rc;
        rc = cuda_check(cudaStreamCreateWithFlags(&hp.d2h, cudaStreamNonBlocking), "copy stream");
        if (rc) return rc;
        rc = cuda_check(cudaStreamCreateWithFlags(&hp.comp, cudaStreamNonBlocking), "decode stream");
        if (rc) return rc;
    }
    *out = &hp;
    return BPQ_OK;
}

// bpq_decode_host.  With `pipelined`, batches of at least 2 x kChunkShots
// shots are cut into up to kMaxChunks chunks whose host-to-device copies
// (one copy stream), decodes and device-to-host copies (a second copy
// stream) overlap, ordered by events.  Consecutive chunks decode on two
// streams (the caller's and a library stream, each with its own workspace),
// so that a chunk's CTAs take the SMs that the previous chunk's last, slowest
// shots leave free.  Without `pipelined` (the no-allocation path) everything
// runs on the caller's stream in order.
int decode_host_impl(const bpq_tanner *t, const uint32_t *syn_host, const float *prior_host, int variant,
                     const bpq_params *params, int max_iter, int B, uint8_t *est_host, uint8_t *conv_host,
                     uint8_t *iters_host, void *dev_buf, size_t dev_buf_bytes, void *stream, bool pipelined) {
    constexpr int kChunkShots = 1 << 16, kMaxChunks = 8;
    int rc = need_uploaded(t);
    if (rc) return rc;
    if (B < 0) return fail(BPQ_EINVAL, "B < 0");
    if (B == 0) return BPQ_OK;
    if (!syn_host || !prior_host || !est_host || !conv_host || !iters_host || !dev_buf)
        return fail(BPQ_EINVAL, "NULL argument");
    if (bpq::misaligned(dev_buf, bpq::kBufferAlign)) return fail(BPQ_EINVAL, "device buffer not 16-byte aligned");
    if (dev_buf_bytes < bpq_decode_host_bytes(t, B)) return fail(BPQ_EINVAL, "device buffer too small");
    auto al = [](size_t x) { return (x + 255) & ~size_t(255); };
    const size_t W = (t->M + 31) / 32, N = (size_t)t->N;
    uint8_t *p = static_cast<uint8_t *>(dev_buf);
    void *work = p;
    p += al(kWorkspaceBytes);
    void *work2 = p;  // the second decode stream's workspace
    p += al(kWorkspaceBytes);
    uint32_t *syn = reinterpret_cast<uint32_t *>(p);
    p += al(sizeof(uint32_t) * W * B);
    float *prior = reinterpret_cast<float *>(p);
    p += al(sizeof(float) * 3 * t->N);
    uint8_t *est = p;
    p += al((size_t)B * N);
    uint8_t *conv = p;
    p += al(B);
    uint8_t *iters = p;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const int chunks = pipelined ? std::min(kMaxChunks, B / kChunkShots) : 1;
    if (chunks < 2) {
        rc = cuda_check(cudaMemcpyAsync(syn, syn_host, sizeof(uint32_t) * W * B, cudaMemcpyHostToDevice, st), "H2D");
        if (!rc)
            rc = cuda_check(cudaMemcpyAsync(prior, prior_host, sizeof(float) * 3 * t->N, cudaMemcpyHostToDevice, st),
                            "H2D");
        if (!rc) rc = bpq_decode(t, syn, prior, variant, params, max_iter, B, est, conv, iters, work, stream);
        if (!rc) rc = cuda_check(cudaMemcpyAsync(est_host, est, (size_t)B * N, cudaMemcpyDeviceToHost, st), "D2H");
        if (!rc) rc = cuda_check(cudaMemcpyAsync(conv_host, conv, B, cudaMemcpyDeviceToHost, st), "D2H");
        if (!rc) rc = cuda_check(cudaMemcpyAsync(iters_host, iters, B, cudaMemcpyDeviceToHost, st), "D2H");
        if (rc) return rc;
        return cuda_check(cudaStreamSynchronize(st), "stream sync");
    }
    HostPipe *hp = nullptr;
    rc = host_pipe(t->device, &hp);
    if (rc) return rc;
    cudaEvent_t ev[2 * kMaxChunks + 1];
    int made = 0;
    for (; made < 2 * chunks + 1 && !rc; ++made)
        rc = cuda_check(cudaEventCreateWithFlags(&ev[made], cudaEventDisableTiming), "event");
    if (!rc) {
        // the copies start after whatever the caller queued on its stream
        rc = cuda_check(cudaEventRecord(ev[2 * chunks], st), "event");
        if (!rc) rc = cuda_check(cudaStreamWaitEvent(hp->h2d, ev[2 * chunks], 0), "wait");
        if (!rc)
            rc = cuda_check(cudaMemcpyAsync(prior, prior_host, sizeof(float) * 3 * t->N, cudaMemcpyHostToDevice,
                                            hp->h2d), "H2D");
    }
    for (int c = 0; c < chunks && !rc; ++c) {
        const int b0 = (int)((long)B * c / chunks), nb = (int)((long)B * (c + 1) / chunks) - b0;
        cudaStream_t cs = (c & 1) ? hp->comp : st;
        rc = cuda_check(cudaMemcpyAsync(syn + W * b0, syn_host + W * b0, sizeof(uint32_t) * W * nb,
                                        cudaMemcpyHostToDevice, hp->h2d), "H2D");
        if (!rc) rc = cuda_check(cudaEventRecord(ev[2 * c], hp->h2d), "event");
        if (!rc) rc = cuda_check(cudaStreamWaitEvent(cs, ev[2 * c], 0), "wait");
        if (!rc)
            rc = bpq_decode(t, syn + W * b0, prior, variant, params, max_iter, nb, est + N * b0, conv + b0,
                            iters + b0, (c & 1) ? work2 : work, cs);
        if (!rc) rc = cuda_check(cudaEventRecord(ev[2 * c + 1], cs), "event");
        if (!rc) rc = cuda_check(cudaStreamWaitEvent(hp->d2h, ev[2 * c + 1], 0), "wait");
        if (!rc)
            rc = cuda_check(cudaMemcpyAsync(est_host + N * b0, est + N * b0, N * nb, cudaMemcpyDeviceToHost, hp->d2h),
                            "D2H");
        if (!rc) rc = cuda_check(cudaMemcpyAsync(conv_host + b0, conv + b0, nb, cudaMemcpyDeviceToHost, hp->d2h), "D2H");
        if (!rc)
            rc = cuda_check(cudaMemcpyAsync(iters_host + b0, iters + b0, nb, cudaMemcpyDeviceToHost, hp->d2h), "D2H");
    }
    // drain everything that was queued, also after an error
    const int rc_d2h = cuda_check(cudaStreamSynchronize(hp->d2h), "stream sync");
    const int rc_h2d = cuda_check(cudaStreamSynchronize(hp->h2d), "stream sync");
    const int rc_cp = cuda_check(cudaStreamSynchronize(hp->comp), "stream sync");
    const int rc_st = cuda_check(cudaStreamSynchronize(st), "stream sync");
    for (int k = 0; k < made; ++k) cudaEventDestroy(ev[k]);
    return rc ? rc : rc_d2h ? rc_d2h : rc_h2d ? rc_h2d : rc_cp ? rc_cp : rc_st;
}

}  // namespace bpq

extern "C" {

int bpq_tanner_upload(bpq_tanner *t, int device) {
    if (!t) return fail(BPQ_EINVAL, "tanner is NULL");
    if (t->dev_blob) return fail(BPQ_ESTATE, "tanner already uploaded");
    int rc = bpq::cuda_check(cudaSetDevice(device), "cudaSetDevice");
    if (rc) return rc;
    int sms = 0;
    rc = bpq::cuda_check(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device), "SM count");
    if (rc) return rc;
    auto al = [](size_t x) { return (x + 255) & ~size_t(255); };
    const size_t o_tab = 0;
    const size_t o_canon = al(t->table.size());
    const size_t o_ptr = o_canon + al(sizeof(int32_t) * t->var_canon.size());
    const size_t o_log = o_ptr + al(sizeof(int32_t) * t->chk_ptr.size());
    const size_t o_tab2 = o_log + al(t->logicals.size() + 1);
    const size_t o_canon2 = o_tab2 + al(t->table_split.size());
    size_t o_serial[bpq::kSerialTables];
    size_t total = o_canon2 + al(sizeof(int32_t) * t->var_canon_split.size());
    for (int k = 0; k < bpq::kSerialTables; ++k) {
        o_serial[k] = total;
        total += al(t->serial[k].data.size());
    }
    void *blob = nullptr;
    rc = bpq::cuda_check(cudaMalloc(&blob, total), "cudaMalloc");
    if (rc) return rc;
    uint8_t *b = static_cast<uint8_t *>(blob);
    cudaError_t e = cudaMemcpy(b + o_tab, t->table.data(), t->table.size(), cudaMemcpyHostToDevice);
    if (e == cudaSuccess)
        e = cudaMemcpy(b + o_canon, t->var_canon.data(), sizeof(int32_t) * t->var_canon.size(), cudaMemcpyHostToDevice);
    if (e == cudaSuccess)
        e = cudaMemcpy(b + o_ptr, t->chk_ptr.data(), sizeof(int32_t) * t->chk_ptr.size(), cudaMemcpyHostToDevice);
    if (e == cudaSuccess && !t->logicals.empty())
        e = cudaMemcpy(b + o_log, t->logicals.data(), t->logicals.size(), cudaMemcpyHostToDevice);
    if (e == cudaSuccess && t->split)
        e = cudaMemcpy(b + o_tab2, t->table_split.data(), t->table_split.size(), cudaMemcpyHostToDevice);
    if (e == cudaSuccess && t->split)
        e = cudaMemcpy(b + o_canon2, t->var_canon_split.data(), sizeof(int32_t) * t->var_canon_split.size(),
                       cudaMemcpyHostToDevice);
    for (int k = 0; k < bpq::kSerialTables && e == cudaSuccess; ++k)
        e = cudaMemcpy(b + o_serial[k], t->serial[k].data.data(), t->serial[k].data.size(), cudaMemcpyHostToDevice);
    if (e != cudaSuccess) {
        cudaFree(blob);
        return bpq::cuda_check(e, "cudaMemcpy");
    }
    t->dev_blob = blob;
    t->device = device;
    t->num_sms = sms;
    t->d_table = b + o_tab;
    t->d_var_canon = reinterpret_cast<const int32_t *>(b + o_canon);
    t->d_chk_ptr = reinterpret_cast<const int32_t *>(b + o_ptr);
    t->d_logicals = t->logicals.empty() ? nullptr : b + o_log;
    t->d_table_split = t->split ? b + o_tab2 : nullptr;
    t->d_var_canon_split = t->split ? reinterpret_cast<const int32_t *>(b + o_canon2) : nullptr;
    for (int k = 0; k < bpq::kSerialTables; ++k) t->d_serial[k] = b + o_serial[k];
    return BPQ_OK;
}

void bpq_free_tanner(bpq_tanner *t) {
    if (!t) return;
    if (t->dev_blob) {
        cudaSetDevice(t->device);
        cudaFree(t->dev_blob);
    }
    delete t;
}

int bpq_sample(const bpq_tanner *t, double px, double py, double pz, uint64_t seed, uint64_t shot0, int B,
               uint8_t *err_dev, uint32_t *syn_dev, void *stream) {
    int rc = bpq::need_uploaded(t);
    if (rc) return rc;
    if (B < 0) return fail(BPQ_EINVAL, "B < 0");
    if (!(px >= 0 && py >= 0 && pz >= 0)) return fail(BPQ_EINVAL, "negative probability");
    const double cx = px, cy = cx + py, cz = cy + pz;
    if (!(cz < 1.0)) return fail(BPQ_EINVAL, "px + py + pz must be < 1");
    if (B == 0) return BPQ_OK;
    if (!err_dev || !syn_dev) return fail(BPQ_EINVAL, "NULL output");
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const int nblk = (t->N + 3) / 4, W = (t->M + 31) / 32;
    const uint16_t *chk_slot = reinterpret_cast<const uint16_t *>(t->d_table);
    const uint8_t *chk_pauli = t->d_table + t->off_chk_pauli;
    const uint64_t tx = bpq::threshold(cx), ty = bpq::threshold(cy), tz = bpq::threshold(cz);
    if (B <= bpq::kSampleShotsPerSm * t->num_sms) {
        // a block a thread and two checks a thread, where 512 threads reach that
        const int threads = std::min(512, (std::max(nblk, t->M / 2) / 32 + 1) * 32);
        bpq::sample_shot_kernel<<<(unsigned)B, threads, 0, st>>>(chk_slot, chk_pauli, t->N, t->M, W, seed, shot0, tx,
                                                                 ty, tz, err_dev, syn_dev);
        return bpq::cuda_check(cudaGetLastError(), "sample launch");
    }
    const size_t smem = bpq::sample_smem(t->N, W);
    if (smem > 48 * 1024) {
        rc = bpq::allow_smem(bpq::sample_kernel, bpq::sample_smem(bpq::kMaxNodes, bpq::kMaxNodes / 32),
                             "sample attribute");
        if (rc) return rc;
    }
    bpq::sample_kernel<<<bpq::launch_grid(B, 32), 32 * bpq::tile_warps(t, B, nblk), smem, st>>>(
        chk_slot, chk_pauli, t->N, t->M, W, B, seed, shot0, tx, ty, tz, err_dev, syn_dev);
    return bpq::cuda_check(cudaGetLastError(), "sample launch");
}

size_t bpq_decode_workspace_bytes(void) { return bpq::kWorkspaceBytes; }

int bpq_decode(const bpq_tanner *t, const uint32_t *syn_dev, const float *prior_dev, int variant,
               const bpq_params *params, int max_iter, int B, uint8_t *est_dev, uint8_t *conv_dev,
               uint8_t *iters_dev, void *work_dev, void *stream) {
    int rc = bpq::need_uploaded(t);
    if (rc) return rc;
    bpq::DecodeArgs a;
    rc = bpq::fill_decode_args(t, syn_dev, prior_dev, variant, params, max_iter, B, work_dev, a);
    if (rc) return rc;
    if (B == 0) return BPQ_OK;
    if (!est_dev || !conv_dev || !iters_dev) return fail(BPQ_EINVAL, "NULL output");
    a.est = est_dev;
    a.conv = conv_dev;
    a.iters = iters_dev;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    return bpq::decode_launch(t, a, variant, false, st);
}

int bpq_decode_status(const void *work_dev, void *stream, int *device_error) {
    if (!work_dev || !device_error) return fail(BPQ_EINVAL, "NULL argument");
    uint32_t w[2] = {0, 0};
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    int rc = bpq::cuda_check(cudaMemcpyAsync(w, work_dev, sizeof w, cudaMemcpyDeviceToHost, st), "status copy");
    if (rc) return rc;
    rc = bpq::cuda_check(cudaStreamSynchronize(st), "status sync");
    if (rc) return rc;
    *device_error = (int)w[1];
    return BPQ_OK;
}

size_t bpq_decode_host_bytes(const bpq_tanner *t, int B) {
    if (!t || B < 0) return 0;
    auto al = [](size_t x) { return (x + 255) & ~size_t(255); };
    const size_t W = (t->M + 31) / 32;
    return 2 * al(bpq::kWorkspaceBytes) + al(sizeof(uint32_t) * W * B) + al(sizeof(float) * 3 * t->N) +
           al((size_t)B * t->N) + al(B) + al(B);
}

int bpq_decode_host(const bpq_tanner *t, const uint32_t *syn_host, const float *prior_host, int variant,
                    const bpq_params *params, int max_iter, int B, uint8_t *est_host, uint8_t *conv_host,
                    uint8_t *iters_host, void *dev_buf, size_t dev_buf_bytes, void *stream) {
    return bpq::decode_host_impl(t, syn_host, prior_host, variant, params, max_iter, B, est_host, conv_host,
                                 iters_host, dev_buf, dev_buf_bytes, stream, true);
}

int bpq_decode_host_noalloc(const bpq_tanner *t, const uint32_t *syn_host, const float *prior_host, int variant,
                            const bpq_params *params, int max_iter, int B, uint8_t *est_host, uint8_t *conv_host,
                            uint8_t *iters_host, void *stream) {
    int rc = bpq::need_uploaded(t);
    if (rc) return rc;
    if (B < 0) return fail(BPQ_EINVAL, "B < 0");
    const size_t need = bpq_decode_host_bytes(t, B);
    if (need > bpq::kNoAllocBytes)
        return fail(BPQ_EINVAL, "batch too large for the fixed 8 MiB device staging area: at most " +
                                    std::to_string(bpq_decode_host_noalloc_max_shots(t)) + " shots of this code");
    void *scratch = nullptr;
    rc = bpq::noalloc_scratch(t->device, &scratch);
    if (rc) return rc;
    // so that the first call of a variant and layout covers every batch size
    rc = bpq::decode_preload(t, variant);
    if (rc) return rc;
    return bpq::decode_host_impl(t, syn_host, prior_host, variant, params, max_iter, B, est_host, conv_host,
                                 iters_host, scratch, bpq::kNoAllocBytes, stream, false);
}

int bpq_decode_host_noalloc_max_shots(const bpq_tanner *t) {
    if (!t) return fail(BPQ_EINVAL, "tanner is NULL");
    int lo = 0, hi = 1 << 24;
    while (lo < hi) {  // largest B whose staging fits
        const int mid = lo + (hi - lo + 1) / 2;
        if (bpq_decode_host_bytes(t, mid) <= bpq::kNoAllocBytes) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

int bpq_decode_trace(const bpq_tanner *t, const uint32_t *syn_dev, const float *prior_dev, int variant,
                     const bpq_params *params, int T, int B, float *m_v2c_dev, float *m_c2v_dev, float *Q_dev,
                     uint8_t *dec_dev, void *work_dev, void *stream) {
    int rc = bpq::need_uploaded(t);
    if (rc) return rc;
    bpq::DecodeArgs a;
    rc = bpq::fill_decode_args(t, syn_dev, prior_dev, variant, params, T, B, work_dev, a);
    if (rc) return rc;
    if (B == 0) return BPQ_OK;
    a.tr_v2c = m_v2c_dev;
    a.tr_c2v = m_c2v_dev;
    a.tr_Q = Q_dev;
    a.tr_dec = dec_dev;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    return bpq::decode_launch(t, a, variant, true, st);
}

int bpq_set_launch(bpq_tanner *t, int threads_per_shot, int shots_per_cta) {
    if (!t) return fail(BPQ_EINVAL, "tanner is NULL");
    if (threads_per_shot < 0 || shots_per_cta < 0 || shots_per_cta > 32) return fail(BPQ_EINVAL, "bad launch shape");
    const int old_t = t->threads_per_shot, old_s = t->shots_per_cta;
    t->threads_per_shot = threads_per_shot;
    t->shots_per_cta = shots_per_cta;
    bpq::LaunchShape s;
    int rc = bpq::decode_uses_pairs(t, BPQ_MOMENTUM, false) ? bpq::decode_pair_shape(t, BPQ_MOMENTUM, &s)
                                                            : bpq::decode_launch_shape(t, -1, &s);
    if (rc) {
        t->threads_per_shot = old_t;
        t->shots_per_cta = old_s;
    }
    return rc;
}

int bpq_set_shots_per_thread(bpq_tanner *t, int shots_per_thread) {
    if (!t) return fail(BPQ_EINVAL, "tanner is NULL");
    if (shots_per_thread < 0 || shots_per_thread > 2) return fail(BPQ_EINVAL, "shots per thread must be 0, 1 or 2");
    if (shots_per_thread == 2 && !t->split)
        return fail(BPQ_EINVAL, "two shots per thread need the split table layout (see bpq_tanner_layout)");
    const int old = t->shots_per_thread;
    t->shots_per_thread = shots_per_thread;
    bpq::LaunchShape s;
    int rc = bpq::decode_uses_pairs(t, BPQ_MOMENTUM, false) ? bpq::decode_pair_shape(t, BPQ_MOMENTUM, &s)
                                                            : bpq::decode_launch_shape(t, -1, &s);
    if (rc) t->shots_per_thread = old;
    return rc;
}

int bpq_set_debug_checks(bpq_tanner *t, int on) {
    if (!t) return fail(BPQ_EINVAL, "tanner is NULL");
    t->debug_checks = on != 0;
    return BPQ_OK;
}

int bpq_get_shots_per_thread(const bpq_tanner *t, int variant, int *shots_per_thread) {
    if (!t || !shots_per_thread) return fail(BPQ_EINVAL, "NULL argument");
    *shots_per_thread = bpq::decode_uses_pairs(t, variant, false) ? 2 : 1;
    return BPQ_OK;
}

int bpq_autotune(bpq_tanner *t, const uint32_t *syn_dev, const float *prior_dev, int variant,
                 const bpq_params *params, int max_iter, int B, uint8_t *est_dev, uint8_t *conv_dev,
                 uint8_t *iters_dev, void *work_dev, void *stream, int *threads_per_shot, int *shots_per_cta,
                 float *best_ms) {
    int rc = bpq::need_uploaded(t);
    if (rc) return rc;
    if (B < 1) return fail(BPQ_EINVAL, "autotune needs a non-empty sample");
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const int nodes = t->N > t->M ? t->N : t->M;
    const int old_t = t->threads_per_shot, old_s = t->shots_per_cta, old_k = t->shots_per_thread;
    int best_T = 0, best_S = 0, best_K = 0;
    bool found = false;
    float best = 1e30f;
    cudaEvent_t e0, e1;
    rc = bpq::cuda_check(cudaEventCreate(&e0), "cudaEventCreate");
    if (rc) return rc;
    rc = bpq::cuda_check(cudaEventCreate(&e1), "cudaEventCreate");
    if (rc) { cudaEventDestroy(e0); return rc; }
    auto time_shape = [&](int T, int S, int K) {
        t->threads_per_shot = T;
        t->shots_per_cta = S;
        t->shots_per_thread = K;
        float ms = 0.f;
        for (int rep = 0; rep < 3 && !rc; ++rep) {  // one warm-up, two timed
            if (rep == 1) rc = bpq::cuda_check(cudaEventRecord(e0, st), "cudaEventRecord");
            if (!rc)
                rc = bpq_decode(t, syn_dev, prior_dev, variant, params, max_iter, B, est_dev, conv_dev, iters_dev,
                                work_dev, stream);
        }
        if (!rc) rc = bpq::cuda_check(cudaEventRecord(e1, st), "cudaEventRecord");
        if (!rc) rc = bpq::cuda_check(cudaEventSynchronize(e1), "cudaEventSynchronize");
        if (!rc) rc = bpq::cuda_check(cudaEventElapsedTime(&ms, e0, e1), "cudaEventElapsedTime");
        if (!rc && ms / 2 < best) {
            best = ms / 2;
            best_T = T;
            best_S = S;
            best_K = K;
            found = true;
        }
    };
    // candidate shapes: the automatic choice, which small batches need (a stored
    // shape keeps to the queue kernels: 150 planar d = 9 Momentum shots at p =
    // 0.06 27 us automatic, 34 with the best stored shape); one or (split tables,
    // not AEWA-BP) two shots per thread; 1..4 nodes per thread (1..2 with two
    // shots per thread); 1..32 shot groups per CTA
    time_shape(0, 0, 0);
    const bool can_pair = t->split && variant >= BPQ_PLAIN && variant <= BPQ_EWAINIT;
    for (int K = 1; K <= (can_pair ? 2 : 1) && !rc; ++K)
    for (int npt = 1; npt <= (K == 2 ? 2 : bpq::kMaxNodesPerThread) && !rc; ++npt) {
        const int T = (((nodes + npt - 1) / npt + 31) / 32) * 32;
        if (T > bpq::kMaxThreadsPerShot) continue;
        if (npt > 1 && (((nodes + npt - 2) / (npt - 1) + 31) / 32) * 32 == T) continue;  // same T as npt-1
        for (int S : {1, 2, 4, 8, 15, 28, 32}) {
            if (S * T > (npt <= 2 ? 1024 : 512) || (S > 15 && T > 32) || (S > 1 && S * T < 64)) continue;
            if ((K == 2 && S > bpq::kMaxPairGroupsPerCta) || (K == 1 && S == 28)) continue;
            t->threads_per_shot = T;
            t->shots_per_cta = S;
            t->shots_per_thread = K;
            bpq::LaunchShape shape;
            if (K == 2 ? bpq::decode_pair_shape(t, variant, &shape) : bpq::decode_launch_shape(t, variant, &shape))
                continue;
            if (!rc) time_shape(T, S, K);
        }
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    if (rc || !found) {
        t->threads_per_shot = old_t;
        t->shots_per_cta = old_s;
        t->shots_per_thread = old_k;
        return rc ? rc : fail(BPQ_EINVAL, "no launch shape fits this code");
    }
    t->threads_per_shot = best_T;
    t->shots_per_cta = best_S;
    t->shots_per_thread = best_K;
    if (threads_per_shot) *threads_per_shot = best_T;
    if (shots_per_cta) *shots_per_cta = best_S;
    if (best_ms) *best_ms = best;
    return BPQ_OK;
}

int bpq_get_launch(const bpq_tanner *t, int *threads_per_shot, int *shots_per_cta, int *ctas) {
    if (!t) return fail(BPQ_EINVAL, "tanner is NULL");
    bpq::LaunchShape s;
    int rc = bpq::decode_uses_pairs(t, BPQ_MOMENTUM, false) ? bpq::decode_pair_shape(t, BPQ_MOMENTUM, &s)
                                                            : bpq::decode_launch_shape(t, -1, &s);
    if (rc) return rc;
    if (threads_per_shot) *threads_per_shot = s.T;
    if (shots_per_cta) *shots_per_cta = s.groups_per_cta;
    if (ctas) *ctas = 0;
    return BPQ_OK;
}

int bpq_probe_peak(int which, int blocks, int threads, int iters, float *sink_dev, void *stream) {
    if (which < 0 || which > 1 || blocks < 1 || threads < 32 || threads > 1024 || iters < 1 || !sink_dev)
        return fail(BPQ_EINVAL, "bad probe arguments");
    bpq::probe_kernel<<<blocks, threads, 0, static_cast<cudaStream_t>(stream)>>>(which, iters, sink_dev);
    return bpq::cuda_check(cudaGetLastError(), "probe launch");
}

int bpq_check_logical(const bpq_tanner *t, const uint8_t *err_dev, const uint8_t *est_dev, int B, uint8_t *fail_dev,
                      void *stream) {
    int rc = bpq::need_uploaded(t);
    if (rc) return rc;
    if (B < 0) return fail(BPQ_EINVAL, "B < 0");
    if (t->logicals.empty()) return fail(BPQ_ESTATE, "no logical operators known");
    if (B == 0) return BPQ_OK;
    if (!err_dev || !est_dev || !fail_dev) return fail(BPQ_EINVAL, "NULL argument");
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const int stride = bpq::check_logical_stride(t->N);
    const size_t smem = bpq::check_logical_smem(t->N);
    if (smem > 48 * 1024) {
        rc = bpq::allow_smem(bpq::check_logical_kernel, bpq::check_logical_smem(bpq::kMaxNodes),
                             "check_logical attribute");
        if (rc) return rc;
    }
    bpq::check_logical_kernel<<<bpq::launch_grid(B, 32), 32 * bpq::tile_warps(t, B, (t->N + 31) / 32), smem, st>>>(
        reinterpret_cast<const uint16_t *>(t->d_table), t->d_table + t->off_chk_pauli, t->d_logicals,
        (int)(t->logicals.size() / t->N), t->N, t->M, B, stride, err_dev, est_dev, fail_dev);
    return bpq::cuda_check(cudaGetLastError(), "check_logical launch");
}

}  // extern "C"
