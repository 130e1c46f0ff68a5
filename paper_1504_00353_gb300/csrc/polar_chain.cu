// Communication chain on the GPU around the decoder, for frame- and bit-error
// rates (the simulations behind the paper's error-rate figures, Sec. III):
// random information bits, the systematic encoder, BPSK over AWGN with
// float32 or int8 channel LLRs, and error counting.
//
// Random numbers come from Philox-4x32-10 (Salmon, Moraes, Dror, Shaw,
// "Parallel random numbers: as easy as 1, 2, 3", SC 2011), a counter-based
// generator: every output is a pure function of (key, counter), so any frame
// of any batch can be regenerated. Normals are Box-Muller pairs of its words.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <mutex>
#include <random>
#include <vector>

#include "polar_gb300.h"
#include "polar_internal.h"

using namespace polar;

namespace {

// ---------------------------------------------------------------- Philox-4x32-10

struct U4 {
    uint32_t x, y, z, w;
};

// One round: two 32x32 -> 64-bit products, their halves mixed with the key.
__host__ __device__ inline void philox_round(U4 &c, uint32_t k0, uint32_t k1) {
    const uint64_t p0 = uint64_t(0xD2511F53u) * c.x;
    const uint64_t p1 = uint64_t(0xCD9E8D57u) * c.z;
    const uint32_t hi0 = uint32_t(p0 >> 32), lo0 = uint32_t(p0);
    const uint32_t hi1 = uint32_t(p1 >> 32), lo1 = uint32_t(p1);
    c = U4{hi1 ^ c.y ^ k0, lo1, hi0 ^ c.w ^ k1, lo0};
}

// Ten rounds, the key bumped by the Weyl constants between rounds.
__host__ __device__ inline U4 philox4x32_10(U4 c, uint32_t k0, uint32_t k1) {
    for (int r = 0; r < 10; ++r) {
        if (r) {
            k0 += 0x9E3779B9u;
            k1 += 0xBB67AE85u;
        }
        philox_round(c, k0, k1);
    }
    return c;
}

// Counter layout: (word index, frame low, frame high, stream).
constexpr uint32_t kStreamInfo = 1u, kStreamNoise = 2u;

__device__ inline U4 draw(uint64_t seed, uint32_t stream, uint64_t frame, uint32_t j) {
    return philox4x32_10(U4{j, uint32_t(frame), uint32_t(frame >> 32), stream}, uint32_t(seed),
                         uint32_t(seed >> 32));
}

// ---------------------------------------------------------------- kernels

// Information bits: row f of `info` (ceil(K/8) bytes) from Philox words; bits
// at and beyond K are zero. `lanes` (a power of two) lanes make consecutive
// draws of 16 bytes of one row and store aligned 32-bit words at any row
// alignment, the bytes shifted through the neighbouring lane's draw; only a
// row's ends are stored as bytes. (Storing the 16 bytes of a draw one by one:
// 19 us for 1,024 rows of 3,687 bytes, now 9, most of it the launch.)
__global__ void random_info_kernel(uint8_t *info, uint32_t K, uint32_t lanes, size_t n_frames,
                                   uint64_t seed, uint64_t frame0) {
    const uint32_t row = (K + 7) / 8, draws = (row + 15) / 16, chunks = (draws + lanes - 1) / lanes;
    const uint32_t lane = threadIdx.x & (lanes - 1u);
    const size_t groups = size_t(gridDim.x) * blockDim.x / lanes;
    const size_t total = n_frames * chunks, turns = (total + groups - 1) / groups;
    size_t t = (blockIdx.x * size_t(blockDim.x) + threadIdx.x) / lanes;
    for (size_t k = 0; k < turns; ++k, t += groups) {  // every lane of a warp makes every turn
        const size_t f = t / chunks;
        const uint32_t j = static_cast<uint32_t>(t % chunks) * lanes + lane;
        const U4 r = draw(seed, kStreamInfo, frame0 + f, j);
        uint32_t v[5] = {0u, r.x, r.y, r.z, r.w};
#pragma unroll
        for (uint32_t k = 0; k < 4; ++k) {  // clear what lies beyond K
            const uint32_t bit0 = 128u * j + 32u * k;
            if (bit0 + 32 > K) v[k + 1] &= bit0 < K ? (1u << (K - bit0)) - 1u : 0u;
        }
        const uint32_t prev = __shfl_up_sync(0xffffffffu, v[4], 1, lanes);
        if (t >= total) continue;
        v[0] = lane ? prev : 0u;
        uint8_t *dst = info + f * row;
        const uint32_t sh = static_cast<uint32_t>(reinterpret_cast<uintptr_t>(dst)) & 3u;
        const int64_t left = row, base = int64_t(16) * (j - lane);  // first byte of the lanes' chunk
#pragma unroll
        for (uint32_t k = 0; k < 4; ++k) {
            const uint32_t word = __funnelshift_l(v[k], v[k + 1], 8u * sh);
            const int64_t at = int64_t(16) * j + 4 * k - sh;  // first byte of this aligned word
            if (at >= base && at + 4 <= left) {
                *reinterpret_cast<uint32_t *>(dst + at) = word;
            } else {
                for (int b = 0; b < 4; ++b)
                    if (at + b >= base && at + b < left) dst[at + b] = static_cast<uint8_t>(word >> (8 * b));
            }
        }
        if (sh && lane == lanes - 1u)  // the chunk's last sh bytes
            for (uint32_t b = 4u - sh; b < 4u; ++b)
                if (int64_t(16) * j + 12 + b < left)
                    dst[int64_t(16) * j + 12 + b] = static_cast<uint8_t>(v[4] >> (8 * b));
    }
}

// 32 bits from bit k of a packed LSB-first byte row (zeros beyond the row): two
// aligned words where both lie inside the row, else its bytes.
__device__ inline uint32_t bits32(const uint8_t *row, uint32_t row_bytes, uint32_t k) {
    const uint8_t *p = row + (k >> 3);
    const uint32_t sh = static_cast<uint32_t>(reinterpret_cast<uintptr_t>(p)) & 3u;
    if (p - sh >= row && p - sh + 8 <= row + row_bytes) {
        const uint32_t *w = reinterpret_cast<const uint32_t *>(p - sh);
        const uint32_t bit = 8u * sh + (k & 7u);
        const uint32_t lo = __ldg(w), hi = __ldg(w + 1);
        return bit ? __funnelshift_r(lo, hi, bit) : lo;
    }
    uint64_t v = 0;
    const uint32_t b0 = k >> 3;
    for (uint32_t b = 0; b < 5; ++b)
        if (b0 + b < row_bytes) v |= uint64_t(row[b0 + b]) << (8 * b);
    return static_cast<uint32_t>(v >> (k & 7));
}

// x <- x F^{(x)n} (x[i] ^= x[i + h] where bit h of i is clear, for every h < N;
// the stages commute) over the part of the index inside one warp: the bits of a
// word, the P words a lane holds (word lane P + r in x[r]) and the lanes.
template <uint32_t P>
__device__ inline void transform_warp(uint32_t (&x)[P], uint32_t N, uint32_t lane) {
    constexpr uint32_t M[5] = {0x55555555u, 0x33333333u, 0x0F0F0F0Fu, 0x00FF00FFu, 0x0000FFFFu};
#pragma unroll
    for (uint32_t l = 0; l < 5; ++l)
        if ((1u << l) < N) {
#pragma unroll
            for (uint32_t r = 0; r < P; ++r) x[r] ^= (x[r] >> (1u << l)) & M[l];
        }
#pragma unroll
    for (uint32_t h = 1; h < P; h *= 2)
#pragma unroll
        for (uint32_t r = 0; r < P; ++r)
            if (!(r & h)) x[r] ^= x[r + h];
    for (uint32_t h = 1; h < 32 && 32u * P * h < N; h *= 2) {
        const uint32_t keep = lane & h ? 0u : 0xffffffffu;
#pragma unroll
        for (uint32_t r = 0; r < P; ++r) x[r] ^= __shfl_xor_sync(0xffffffffu, x[r], h) & keep;
    }
}

// The stages across the `warps` (<= P) parts of a frame, each 32 P words long:
// thread t takes word positions t, t + T, ... of all parts.
template <uint32_t P, class Sink>
__device__ inline void transform_parts(const uint32_t *xs, uint32_t warps, uint32_t nw, uint32_t t,
                                       const Sink &sink) {
    for (uint32_t p = t; p < 32u * P && p < nw; p += 32u * warps) {
        uint32_t y[P];
#pragma unroll
        for (uint32_t i = 0; i < P; ++i) y[i] = i < warps ? xs[p + 32u * P * i] : 0u;
#pragma unroll
        for (uint32_t h = 1; h < P; h *= 2)
            if (h < warps) {
#pragma unroll
                for (uint32_t i = 0; i < P; ++i)
                    if (!(i & h)) y[i] ^= y[i + h];
            }
#pragma unroll
        for (uint32_t i = 0; i < P; ++i)
            if (i < warps) sink(p + 32u * P * i, y[i]);
    }
}

// Systematic encoding (two transforms with the frozen positions cleared in
// between): info bits to the information set, transform, clear the frozen set,
// transform. `warps` warps hold a frame's words in registers, P per lane; only
// the gather of the information bits, the stages across warps and the output
// order go through shared memory. Words that mix frozen and information bits
// (records `part`, see KernelArgs::ext_part) are spread by the expand of
// "Hacker's Delight" (7-5), the packing steps undone in reverse. Bound by its
// instructions and, for short codes, by launch width: one warp per frame up to
// N = 4096, so a block of 128 threads encodes four (a block per frame with every
// stage in shared memory: 74 us for 16,384 frames of N = 1024, 35 us for 1,024
// of N = 32768; now 13 and 17).
template <uint32_t P>
__global__ void __launch_bounds__(P < 8 ? 128 : 32 * P)
    encode_kernel(const uint8_t *info, uint8_t *cw, const uint32_t *ext_mask,
                  const uint32_t *ext_pre, const uint32_t *part, uint32_t n_part, uint32_t N,
                  uint32_t K, uint32_t warps, size_t n_frames) {
    extern __shared__ uint32_t xs_all[];
    const uint32_t nw = N >= 32 ? N / 32 : 1, in_row = (K + 7) / 8, out_row = (N + 7) / 8;
    const uint32_t T = 32u * warps, per_block = blockDim.x / T;
    const uint32_t slot = threadIdx.x / T, t = threadIdx.x % T, lane = threadIdx.x & 31u;
    uint32_t *xs = xs_all + slot * nw;
    auto sync = [&] {
        if (warps == 1) __syncwarp();
        else __syncthreads();  // then one frame per block: every thread is here
    };
    for (size_t f = blockIdx.x * size_t(per_block) + slot; f < n_frames;
         f += size_t(gridDim.x) * per_block) {
        const uint8_t *d = info + f * in_row;
        for (uint32_t w = t; w < nw; w += T) {
            const uint32_t m = __ldg(ext_mask + w);
            xs[w] = m ? bits32(d, in_row, __ldg(ext_pre + w)) : 0u;
        }
        sync();
        for (uint32_t i = t; i < n_part; i += T) {
            const uint4 *rec = reinterpret_cast<const uint4 *>(part) + 2 * i;
            const uint4 p = __ldg(rec), q = __ldg(rec + 1);
            const uint32_t v[5] = {p.z, p.w, q.x, q.y, q.z};
            uint32_t x = xs[p.x];
#pragma unroll
            for (int k = 4; k >= 0; --k) x = (x & ~v[k]) | ((x << (1 << k)) & v[k]);
            xs[p.x] = x & p.y;
        }
        sync();
        if (warps > 1) {
            transform_parts<P>(xs, warps, nw, t, [&](uint32_t w, uint32_t y) { xs[w] = y; });
            sync();
        }
        uint32_t x[P];
        const uint32_t w0 = t * P;
#pragma unroll
        for (uint32_t r = 0; r < P; ++r) x[r] = w0 + r < nw ? xs[w0 + r] : 0u;
        transform_warp<P>(x, N, lane);
#pragma unroll
        for (uint32_t r = 0; r < P; ++r) x[r] &= w0 + r < nw ? __ldg(ext_mask + w0 + r) : 0u;
        transform_warp<P>(x, N, lane);
#pragma unroll
        for (uint32_t r = 0; r < P; ++r)
            if (w0 + r < nw) xs[w0 + r] = x[r];
        sync();
        uint8_t *o = cw + f * size_t(out_row);
        if (N >= 32 && reinterpret_cast<uintptr_t>(cw) % 4 == 0) {
            uint32_t *ow = reinterpret_cast<uint32_t *>(o);
            transform_parts<P>(xs, warps, nw, t, [&](uint32_t w, uint32_t y) { ow[w] = y; });
        } else {
            transform_parts<P>(xs, warps, nw, t, [&](uint32_t w, uint32_t y) {
                if (N < 8) y &= (1u << N) - 1u;
                for (uint32_t b = 0; b < 4 && 4 * w + b < out_row; ++b)
                    o[4 * w + b] = static_cast<uint8_t>(y >> (8 * b));
            });
        }
        sync();
    }
}

// BPSK (bit 0 -> +1) over AWGN: y = s + sigma n, LLR = 2 y / sigma^2 in
// float32, or q = clamp(rint(8 LLR), -127, 127) for int8. Four elements per
// Philox draw (two Box-Muller pairs). Bound by its arithmetic (Philox, two
// logarithms, square roots and sine-cosine pairs per four values); N is a power
// of two, so the frame and element come from a shift, and the four values leave
// in one store where VEC says the row allows it (64-bit divisions and scalar
// stores before: 101 us for 1,024 int8 frames of N = 32768, now 81).
template <typename T, bool VEC>
__global__ void awgn_kernel(const uint8_t *cw, T *llr, uint32_t N, uint32_t log2quads,
                            size_t n_frames, float sigma, float scale, uint64_t seed,
                            uint64_t frame0) {
    const uint32_t row = (N + 7) / 8;
    const size_t total = n_frames << log2quads;
    for (size_t t = blockIdx.x * size_t(blockDim.x) + threadIdx.x; t < total;
         t += size_t(gridDim.x) * blockDim.x) {
        const size_t f = t >> log2quads;
        const uint32_t j = static_cast<uint32_t>(t) & ((1u << log2quads) - 1u);
        const U4 r = draw(seed, kStreamNoise, frame0 + f, j);
        const float u1a = (float(r.x) + 1.0f) * 2.3283064365386963e-10f;  // (0, 1]
        const float u1b = (float(r.z) + 1.0f) * 2.3283064365386963e-10f;
        const float ra = sqrtf(-2.0f * logf(u1a)), rb = sqrtf(-2.0f * logf(u1b));
        float sa, ca, sb, cb;
        sincospif(2.0f * (float(r.y) * 2.3283064365386963e-10f), &sa, &ca);
        sincospif(2.0f * (float(r.w) * 2.3283064365386963e-10f), &sb, &cb);
        const float nz[4] = {ra * ca, ra * sa, rb * cb, rb * sb};
        const uint32_t x = cw[f * row + (j >> 1)] >> (4u * (j & 1u));  // the four codeword bits
        T q[4];
#pragma unroll
        for (uint32_t e = 0; e < 4; ++e) {
            const float s = (x >> e) & 1u ? -1.0f : 1.0f;
            const float l = scale * (s + sigma * nz[e]);
            if constexpr (sizeof(T) == 1) {
                q[e] = static_cast<T>(fminf(fmaxf(rintf(8.0f * l), -127.0f), 127.0f));
            } else {
                q[e] = l;
            }
        }
        T *out = llr + f * size_t(N) + 4 * size_t(j);
        if constexpr (VEC) {
            if constexpr (sizeof(T) == 1) *reinterpret_cast<char4 *>(out) = make_char4(q[0], q[1], q[2], q[3]);
            else *reinterpret_cast<float4 *>(out) = make_float4(q[0], q[1], q[2], q[3]);
        } else {
            for (uint32_t e = 0; e < 4 && 4 * j + e < N; ++e) out[e] = q[e];
        }
    }
}

// Frame and bit errors between two packed rows per frame: counters[0] +=
// frames that differ, counters[1] += differing bits. `lanes` (a power of two)
// lanes share a frame and read 16-byte vectors where both rows have the same
// alignment, bytes elsewhere; a warp joins its sums before a block adds them once.
// Reads every byte once: bound by memory and launch. (One thread per frame reading
// bytes: 307 us for 1,024 rows of 3,687 bytes, now 9. An atomic per lane on the
// block's sums: 20.8 us for 5,000 rows of 6 bytes that all differ, now 4.)
__global__ void __launch_bounds__(256)
    count_errors_kernel(const uint8_t *a, const uint8_t *b, uint32_t row, uint32_t lanes,
                        size_t n_frames, unsigned long long *counters) {
    __shared__ unsigned long long sums[2];
    if (threadIdx.x < 2) sums[threadIdx.x] = 0;
    __syncthreads();
    unsigned long long fe = 0, be = 0;
    const uint32_t l = threadIdx.x & (lanes - 1u);
    const size_t groups = size_t(gridDim.x) * blockDim.x / lanes;
    const size_t g0 = (blockIdx.x * size_t(blockDim.x) + threadIdx.x) / lanes;
    // every lane of a warp makes the same number of turns, so the sums can use full-warp shuffles
    const size_t turns = (n_frames + groups - 1) / groups;
    for (size_t k = 0; k < turns; ++k) {
        const size_t f = g0 + k * groups;
        uint32_t bits = 0;
        if (f < n_frames) {
            const uint8_t *p = a + f * row, *q = b + f * row;
            uint32_t head = row, nv = 0;
            if (((reinterpret_cast<uintptr_t>(p) ^ reinterpret_cast<uintptr_t>(q)) & 15u) == 0) {
                head = min(row, static_cast<uint32_t>(-reinterpret_cast<uintptr_t>(p)) & 15u);
                nv = (row - head) / 16;
            }
            const uint4 *pv = reinterpret_cast<const uint4 *>(p + head);
            const uint4 *qv = reinterpret_cast<const uint4 *>(q + head);
            for (uint32_t i = l; i < nv; i += lanes) {
                const uint4 x = pv[i], y = qv[i];
                bits += __popc(x.x ^ y.x) + __popc(x.y ^ y.y) + __popc(x.z ^ y.z) + __popc(x.w ^ y.w);
            }
            for (uint32_t i = l; i < head; i += lanes) bits += __popc(uint32_t(p[i] ^ q[i]));
            for (uint32_t i = head + 16 * nv + l; i < row; i += lanes) bits += __popc(uint32_t(p[i] ^ q[i]));
        }
        for (uint32_t m = lanes / 2; m >= 1; m /= 2) bits += __shfl_xor_sync(0xffffffffu, bits, m);
        if (l == 0) {
            fe += bits ? 1u : 0u;
            be += bits;
        }
    }
    for (uint32_t m = 16; m >= 1; m /= 2) {  // only the lanes with l = 0 hold counts
        fe += __shfl_xor_sync(0xffffffffu, fe, m);
        be += __shfl_xor_sync(0xffffffffu, be, m);
    }
    if ((threadIdx.x & 31u) == 0 && fe) {
        atomicAdd(&sums[0], fe);
        atomicAdd(&sums[1], be);
    }
    __syncthreads();
    if (threadIdx.x < 2 && sums[threadIdx.x]) atomicAdd(&counters[threadIdx.x], sums[threadIdx.x]);
}

// ---------------------------------------------------------------- host helpers

polar_status status_of(cudaError_t e) {
    if (e == cudaSuccess) return POLAR_OK;
    cudaGetLastError();
    return e == cudaErrorMemoryAllocation ? POLAR_ENOMEM : POLAR_ECUDA;
}

int grid_for(size_t work, uint32_t threads) {
    int sms = 0, dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const size_t g = (work + threads - 1) / threads;
    return static_cast<int>(std::max<size_t>(1, std::min<size_t>(g, size_t(std::max(sms, 1)) * 16)));
}

// Whether the two-step encoder reproduces the information bits for this frozen
// set (checked once per handle on random words, on the host): true for the
// domination-contiguous sets polar constructions give.
bool systematic_ok(polar_code *c) {
    std::lock_guard<std::mutex> g(c->mu);
    if (c->systematic_checked) return c->systematic_valid;
    const uint32_t K = c->K;
    const size_t row = (K + 7) / 8;
    std::mt19937_64 rng(0x5eedu);
    bool ok = true;
    std::vector<uint8_t> d(row), x((c->N + 7) / 8);
    for (int t = 0; t < 16 && ok && K; ++t) {
        for (auto &b : d) b = static_cast<uint8_t>(rng());
        if (K % 8) d[row - 1] &= static_cast<uint8_t>((1u << (K % 8)) - 1u);
        ok = polar_encode_systematic(c, d.data(), x.data(), 1) == POLAR_OK;
    }
    c->systematic_checked = true;
    c->systematic_valid = ok;
    return ok;
}

}  // namespace

extern "C" {

polar_status polar_random_info(const polar_code_t *code, uint8_t *info_packed, size_t n_frames,
                               uint64_t seed, uint64_t frame0, polar_stream_t stream) {
    if (!code) return POLAR_EINVAL;
    if (n_frames == 0 || code->K == 0) return POLAR_OK;
    if (!info_packed) return POLAR_EINVAL;
    const uint32_t draws = ((code->K + 7) / 8 + 15) / 16;
    uint32_t lanes = 1;
    while (lanes < 32 && lanes < draws) lanes *= 2;
    random_info_kernel<<<grid_for(n_frames * ((draws + lanes - 1) / lanes) * lanes, 256), 256, 0,
                         reinterpret_cast<cudaStream_t>(stream)>>>(info_packed, code->K, lanes,
                                                                   n_frames, seed, frame0);
    return status_of(cudaGetLastError());
}

polar_status polar_encode_systematic_device(const polar_code_t *code, const uint8_t *info_packed,
                                            uint8_t *codeword_packed, size_t n_frames,
                                            polar_stream_t stream) {
    if (!code) return POLAR_EINVAL;
    if (n_frames == 0) return POLAR_OK;
    if ((!info_packed && code->K) || !codeword_packed) return POLAR_EINVAL;
    polar_code *c = const_cast<polar_code *>(code);
    if (!systematic_ok(c)) return POLAR_EINVAL;
    int device = -1;
    if (cudaGetDevice(&device) != cudaSuccess) return status_of(cudaErrorNoDevice);
    DeviceState *ds = nullptr;
    const polar_status st = code_device_state(c, device, &ds);
    if (st != POLAR_OK) return st;
    // words per lane and warps per frame: one warp of up to four words up to
    // N = 4096, then up to four warps, then both (the stages across warps need
    // warps <= words). More words on fewer warps only lengthen a frame's chain:
    // with eight words before a second warp 100 frames of N = 8192 and 16384 took
    // 10.3 us instead of 6.2, 5,000 took 16.4 and 26.6 instead of 14.3 and 20.5;
    // with two words N = 8192 and more are the same, 20,000 frames of N = 4096
    // 26.7 instead of 22.5.
    const uint32_t nw = c->N >= 32 ? c->N / 32 : 1;
    uint32_t P = 1, warps = 1;
    while (32 * P < nw && P < 4) P *= 2;
    while (32 * P * warps < nw) {
        if (warps < P) warps *= 2;
        else P *= 2;
    }
    const uint32_t per_block = warps == 1 ? 4 : 1;
    const size_t smem = size_t(per_block) * nw * sizeof(uint32_t);  // 128 KB at N = 2^20
    auto kernel = P == 1    ? encode_kernel<1>
                  : P == 2  ? encode_kernel<2>
                  : P == 4  ? encode_kernel<4>
                  : P == 8  ? encode_kernel<8>
                  : P == 16 ? encode_kernel<16>
                            : encode_kernel<32>;
    if (smem > 48 * 1024) {  // N >= 2^19, P = 32
        static std::mutex mu;
        static size_t raised[64] = {};
        std::lock_guard<std::mutex> g(mu);
        if (device < 64 && raised[device] < smem) {
            const cudaError_t e = cudaFuncSetAttribute(
                kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
            if (e != cudaSuccess) return status_of(e);
            raised[device] = smem;
        }
    }
    const uint32_t threads = 32 * warps * per_block;
    kernel<<<grid_for(((n_frames + per_block - 1) / per_block) * threads, threads), threads, smem,
             reinterpret_cast<cudaStream_t>(stream)>>>(
        info_packed, codeword_packed, ds->tables + c->at_mask(), ds->tables + c->at_pre(),
        ds->tables, static_cast<uint32_t>(c->ext_part.size() / 8), c->N, c->K, warps, n_frames);
    return status_of(cudaGetLastError());
}

polar_status polar_channel_awgn(const polar_code_t *code, const uint8_t *codeword_packed,
                                void *llr, int is_i8, size_t n_frames, float ebn0_db,
                                uint64_t seed, uint64_t frame0, polar_stream_t stream) {
    if (!code) return POLAR_EINVAL;
    if (n_frames == 0) return POLAR_OK;
    if (!codeword_packed || !llr || code->K == 0) return POLAR_EINVAL;
    const double rate = double(code->K) / code->N;
    const double s2 = 1.0 / (2.0 * rate * std::pow(10.0, ebn0_db / 10.0));
    const float sigma = static_cast<float>(std::sqrt(s2)), scale = static_cast<float>(2.0 / s2);
    const uint32_t quads = (code->N + 3) / 4;
    const uint32_t lq = static_cast<uint32_t>(log2u(quads));
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    const int grid = grid_for(n_frames * quads, 256);
    auto run = [&](auto kernel, auto *out) {
        kernel<<<grid, 256, 0, s>>>(codeword_packed, out, code->N, lq, n_frames, sigma, scale, seed, frame0);
    };
    const bool vec = code->N >= 4 && reinterpret_cast<uintptr_t>(llr) % (is_i8 ? 4 : 16) == 0;
    if (is_i8)
        run(vec ? awgn_kernel<int8_t, true> : awgn_kernel<int8_t, false>, static_cast<int8_t *>(llr));
    else
        run(vec ? awgn_kernel<float, true> : awgn_kernel<float, false>, static_cast<float *>(llr));
    return status_of(cudaGetLastError());
}

polar_status polar_count_errors(const polar_code_t *code, const uint8_t *decoded,
                                const uint8_t *sent, size_t n_frames,
                                unsigned long long *counters, polar_stream_t stream) {
    if (!code || !counters) return POLAR_EINVAL;
    if (n_frames == 0 || code->K == 0) return POLAR_OK;
    if (!decoded || !sent) return POLAR_EINVAL;
    const uint32_t row = (code->K + 7) / 8;
    uint32_t lanes = 1;
    while (lanes < 32 && 16 * lanes < row) lanes *= 2;
    count_errors_kernel<<<grid_for(n_frames * lanes, 256), 256, 0,
                          reinterpret_cast<cudaStream_t>(stream)>>>(decoded, sent, row, lanes,
                                                                    n_frames, counters);
    return status_of(cudaGetLastError());
}

polar_status polar_fer_run(const polar_code_t *code, int is_i8, float ebn0_db, uint64_t seed,
                           size_t n_frames, size_t batch, uint64_t *frame_errors,
                           uint64_t *bit_errors) {
    if (!code || !frame_errors || !bit_errors || code->K == 0) return POLAR_EINVAL;
    *frame_errors = *bit_errors = 0;
    if (n_frames == 0) return POLAR_OK;
    if (batch == 0) batch = 16384;
    batch = std::min(batch, n_frames);
    const size_t in_row = (code->K + 7) / 8, cw_row = (code->N + 7) / 8;
    const size_t es = is_i8 ? 1 : 4;
    uint8_t *d = nullptr, *x = nullptr, *out = nullptr;
    void *llr = nullptr;
    unsigned long long *cnt = nullptr;
    cudaStream_t s = nullptr;
    cudaError_t e = cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking);
    if (e == cudaSuccess) e = cudaMalloc(&d, batch * in_row);
    if (e == cudaSuccess) e = cudaMalloc(&x, batch * cw_row);
    if (e == cudaSuccess) e = cudaMalloc(&out, batch * in_row);
    if (e == cudaSuccess) e = cudaMalloc(&llr, batch * code->N * es);
    if (e == cudaSuccess) e = cudaMalloc(&cnt, 2 * sizeof(unsigned long long));
    if (e == cudaSuccess) e = cudaMemsetAsync(cnt, 0, 2 * sizeof(unsigned long long), s);
    polar_status st = status_of(e);
    const polar_stream_t ps = reinterpret_cast<polar_stream_t>(s);
    for (size_t f0 = 0; f0 < n_frames && st == POLAR_OK; f0 += batch) {
        const size_t n = std::min(batch, n_frames - f0);
        st = polar_random_info(code, d, n, seed, f0, ps);
        if (st == POLAR_OK) st = polar_encode_systematic_device(code, d, x, n, ps);
        if (st == POLAR_OK) st = polar_channel_awgn(code, x, llr, is_i8, n, ebn0_db, seed, f0, ps);
        if (st == POLAR_OK)
            st = is_i8 ? polar_decode_i8(code, static_cast<const int8_t *>(llr), out, n, ps)
                       : polar_decode(code, static_cast<const float *>(llr), out, n, ps);
        if (st == POLAR_OK) st = polar_count_errors(code, out, d, n, cnt, ps);
    }
    unsigned long long h[2] = {0, 0};
    if (st == POLAR_OK) st = status_of(cudaMemcpyAsync(h, cnt, sizeof h, cudaMemcpyDeviceToHost, s));
    if (s) {
        const cudaError_t e2 = cudaStreamSynchronize(s);
        if (st == POLAR_OK) st = status_of(e2);
    }
    if (st == POLAR_OK) st = polar_code_check(const_cast<polar_code_t *>(code), ps);
    *frame_errors = h[0];
    *bit_errors = h[1];
    cudaFree(d);
    cudaFree(x);
    cudaFree(out);
    cudaFree(llr);
    cudaFree(cnt);
    if (s) cudaStreamDestroy(s);
    return st;
}

}  // extern "C"
