// Device building blocks of the Fast-SSC decoder (sm_103a), shared by the
// operation-list interpreter (polar_kernels.cu, compiled by nvcc) and by the
// per-code specialised decoders that polar_codegen.cpp emits and compiles at
// run time with NVRTC. The file therefore includes no host header when
// __CUDACC_RTC__ is defined.
//
// Method: Giard et al., "Low-Latency Software Polar Decoders" (arXiv 1504.00353),
// Sec. II-C/II-D: min-sum F (Eq. 1), G (Eq. 2) and G_0R, Combine (Eq. 3) and
// Combine_0R, Rate-0, Rate-1 (Eq. 4), Repetition and SPC nodes.
//
// Memory layout (Sec. III-B): the alpha stage of node size n occupies elements
// [n, 2n) of a per-CTA array, in shared memory for n <= S and in per-CTA
// device scratch above that; beta is one N-bit array (node (off, n) owns bits
// [off, off+n), Combine rewrites only the left half), bit-packed in shared
// memory. float32: F is an exact min with the XOR of the sign bits (beta in
// {+0,-0}), G adds alpha_v[i] with its sign flipped by beta_l (Listing 3): one
// IEEE add. int8: G is a saturating add followed by max(-127) (Listing 4);
// in memory-level operations the int8 values are computed as f16 pairs, which
// is exact for them (see op_i8x4). Every operation agrees bit for bit with a
// scalar evaluation in the same order.
#pragma once

#ifdef __CUDACC_RTC__
typedef unsigned int uint32_t;
typedef int int32_t;
typedef unsigned long long uint64_t;
typedef signed char int8_t;
typedef unsigned char uint8_t;
typedef unsigned long size_t;
typedef unsigned long uintptr_t;
#else
#include <cstddef>
#include <cstdint>
#endif

namespace polar {

// Operation kinds of the depth-first Fast-SSC list (Sec. II-D, Listing 1).
enum OpKind : uint32_t {
    OP_F = 0,     // alpha_l = f(alpha_v[i], alpha_v[i + N_v/2])          (Eq. 1)
    OP_G = 1,     // alpha_r = g(alpha_v[i], alpha_v[i + N_v/2], beta_l)  (Eq. 2)
    OP_G0R = 2,   // G with an all-zero beta_l (left child Rate-0)
    OP_C = 3,     // beta_v[i] ^= beta_v[i + N_v/2], i < N_v/2            (Eq. 3)
    OP_C0R = 4,   // beta_v[i] = beta_v[i + N_v/2] (left child Rate-0)
    OP_R0 = 5,    // beta_v = 0 (Rate-0 right child, or a Rate-0 root)
    OP_R1 = 6,    // beta_v[i] = alpha_v[i] < 0                           (Eq. 4)
    OP_REP = 7,   // Repetition: threshold of the folded sum, replicated
    OP_SPC = 8,   // SPC: hard decisions, flip least-|alpha| bit on odd parity
};

// How an operation reads its input stage: RD_NORMAL; RD_STREAM, an L2
// evict-first policy (the channel LLRs, read far apart in time); RD_LAST, the
// last read of a scratch stage before it is rewritten: evict-first, and the
// generated code then discards the lines (discard_l2) so that the dead data is
// never written back to DRAM. Hints only: the values read are the same.
enum : uint32_t { RD_NORMAL = 0, RD_STREAM = 1, RD_LAST = 2 };

// How an operation stores a scratch stage (two bits per output stage): ST_FAR, an
// L2 evict-first policy, for the widest stage (N/2), which is read again only after
// a whole half of the tree; ST_NEAR, evict-last, for the narrower ones, which are
// read soon and discarded after their last read. The frames in flight hold more
// scratch than L2, beside the streaming channel. (4,096 frames of (32768, 29492):
// ST_FAR int8 248 -> 238 us, float32 806 -> 786; ST_NEAR int8 213 -> 206, float32
// 712 -> 705.)
enum : uint32_t { ST_NORMAL = 0, ST_FAR = 1, ST_NEAR = 2 };

// One operation as the interpreter reads it: a 32-bit word
//   bits 0-3   kind (OpKind)
//   bits 4-8   log2(N_v)
//   bit  9     inside a register-resident subtree (N_v <= kRegSubtree)
//   bit  10    first op of such a subtree: (N_v, off) is the subtree root
//   bit  11    last op of such a subtree: store its bits to beta
//   bits 12-31 off >> log2(N_v), off = index of the node's first leaf
enum : uint32_t {
    OPW_REG = 1u << 9,
    OPW_REG_ENTER = 1u << 10,
    OPW_REG_EXIT = 1u << 11,
};

__host__ __device__ inline uint32_t op_kind(uint32_t w) { return w & 0xFu; }
__host__ __device__ inline uint32_t op_log2n(uint32_t w) { return (w >> 4) & 0x1Fu; }
__host__ __device__ inline uint32_t op_off(uint32_t w) { return (w >> 12) << op_log2n(w); }

// Largest subtree the interpreter decodes in the registers of one warp: the largest
// for which a node's side tells where its bits go (two rows of 32 float32 bits).
constexpr uint32_t kRegSubtree = 64;

// Kernel parameters (identical layout for the interpreter and the generated
// decoders).
struct KernelArgs {
    const uint32_t *ops;           // n_ops packed operation words
    const uint32_t *trace_offs;    // per op: offset of its F/G/G_0R outputs in a trace row
    const uint32_t *ext_mask;      // info mask of each beta word (NW words)
    const uint32_t *ext_part;      // words mixing frozen and info bits: n_part records of 8 words
                                   // (word, mask, five compress masks, 0), 16-byte aligned
    const uint32_t *ext_start;     // per output word: first beta word << 5 | its info bits to skip
    int *status;                   // error flags (bit 0: a bounded wait expired)
    const void *llr;
    uint8_t *out;
    float *trace;
    void *gscratch;
    size_t n_frames;
    size_t trace_stride;           // floats per frame
    size_t gstride;                // scratch elements per CTA
    uint32_t n_ops;
    uint32_t N, log2N, K;
    uint32_t S;                    // smem_stage_max (already clipped to N/2)
    uint32_t log2W;                // ops with log2(N_v) <= log2W run on warp 0 alone
    uint32_t NW;                   // beta words (max(1, N/32))
    uint32_t KW;                   // output 32-bit words (ceil(K/32))
    uint32_t n_part;               // records of ext_part
    uint32_t out_row;              // bytes per output row (ceil(K/8))
};

__host__ __device__ constexpr size_t align_up(size_t v, size_t a) { return (v + a - 1) / a * a; }

// One code of a mixed batch, as the batch kernel sees it.
struct CodeDesc {
    const uint32_t *ext_mask;      // as in KernelArgs
    const uint32_t *ext_part;
    const uint32_t *ext_start;
    uint32_t N, K, NW, KW, out_row, n_part;
    uint32_t S;                    // smem_stage_max of this code (clipped to N/2)
};

// Parameters of the mixed-batch kernel: frame i belongs to code code_id[i],
// its LLRs start at element llr_off[i] of llr, its packed bits at byte
// out_off[i] of out. CTAs claim frames with an atomic counter.
struct BatchArgs {
    const CodeDesc *codes;
    const uint32_t *code_id;
    const unsigned long long *llr_off;
    const unsigned long long *out_off;
    const void *llr;
    uint8_t *out;
    unsigned int *counter;         // next unclaimed frame; zero before the launch
    void *gscratch;
    size_t gstride;                // scratch elements per frame slot (max over codes)
    size_t n_frames;
    uint32_t smem_alpha_elems;     // alpha region: max over codes of 2 * S
    uint32_t smem_beta_words;      // beta region: max over codes of NW
};

// Shared-memory bytes of one frame slot of the batch kernel (alpha, beta,
// reduction slots), computed identically on host and device.
__host__ __device__ inline size_t batch_slot_bytes(uint32_t alpha_elems, uint32_t beta_words,
                                                   uint32_t es) {
    return align_up(align_up(size_t(alpha_elems) * es, 128) + align_up(size_t(beta_words) * 4, 16) +
                        32 * 8 + 32 * 4,
                    128);
}


// Shared-memory carve-up, computed identically on host and device.
struct SmemLayout {
    size_t alpha, beta, rkey, rpar, chan0, chan1, mbar, total;
    __host__ __device__ SmemLayout(uint32_t N, uint32_t S, uint32_t es, bool stage) {
        const uint32_t Se = S < N / 2 ? S : N / 2;
        const uint32_t NW = N >= 32 ? N / 32 : 1;
        size_t o = 0;
        alpha = o;
        o = align_up(o + size_t(2) * Se * es, 128);
        beta = o;
        o = align_up(o + size_t(NW) * 4, 16);
        rkey = o;
        o += 32 * 8;
        rpar = o;
        o = align_up(o + 32 * 4, 128);
        chan0 = chan1 = o;
        if (stage) {
            chan0 = o;
            o = align_up(o + size_t(N) * es, 128);
            chan1 = o;
            o = align_up(o + size_t(N) * es, 128);
        }
        mbar = o;
        o += 16;
        total = align_up(o, 16);
    }
};

#if defined(__CUDACC__)

constexpr unsigned long long kWaitNs = 2000000000ull;  // bounded mbarrier wait: 2 s
constexpr uint32_t kWaitPolls = 1u << 28;              // and at most this many polls
constexpr uint32_t kFull = 0xffffffffu;

// ---------------------------------------------------------------- element ops

// Eq. 1: min(|a|, |b|) carrying the XOR of the two signs, one instruction.
__device__ __forceinline__ float f_f32(float a, float b) {
    float r;
    asm("min.xorsign.abs.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
    return r;
}
// Eq. 2 with beta_l as the sign bit of alpha_v[i] (Listing 3): one IEEE add.
__device__ __forceinline__ float g_f32(float a, float b, uint32_t bit) {
    return b + __uint_as_float(__float_as_uint(a) ^ (bit << 31));
}
__device__ __forceinline__ int sat127(int v) { return max(-127, min(127, v)); }
// Eq. 1 on integers: max(min(a, b), -max(a, b)) equals sgn(a) sgn(b) min(|a|, |b|)
// (both positive: min(a, b); both negative: -max(a, b) = min(|a|, |b|); mixed
// signs: the negative one of min(a, b) and -max(a, b) with the smaller magnitude).
__device__ __forceinline__ int f_i8s(int a, int b) { return max(min(a, b), -max(a, b)); }
__device__ __forceinline__ int g_i8s(int a, int b, uint32_t bit) {
    return sat127(bit ? b - a : b + a);
}

// Element op on the accumulator type (float, or int holding an int8 value).
__device__ __forceinline__ float op_f(float a, float b) { return f_f32(a, b); }
__device__ __forceinline__ int op_f(int a, int b) { return f_i8s(a, b); }
__device__ __forceinline__ float op_g(float a, float b, uint32_t bit) { return g_f32(a, b, bit); }
__device__ __forceinline__ int op_g(int a, int b, uint32_t bit) { return g_i8s(a, b, bit); }
__device__ __forceinline__ float op_add(float a, float b) { return a + b; }
__device__ __forceinline__ int op_add(int a, int b) { return sat127(a + b); }

// Four int8 lanes per 32-bit word, computed as two f16x2 pairs. Every int8
// value and every sum of two of them is an integer of magnitude <= 254, exact
// in f16, so F (one min.xorsign.abs, Eq. 1), G and G_0R (one IEEE add, Eq. 2,
// then the clamp to [-127, 127] that the saturating byte add followed by
// max(-127) gives) are exact: the results are the byte results bit for bit.
// The arithmetic runs on the FP16 units instead of byte-wise integer sequences.
__device__ __forceinline__ uint32_t prmt(uint32_t a, uint32_t b, uint32_t sel) {
    uint32_t r;
    asm("prmt.b32 %0, %1, %2, %3;" : "=r"(r) : "r"(a), "r"(b), "r"(sel));
    return r;
}
__device__ __forceinline__ uint32_t hadd2(uint32_t a, uint32_t b) {
    uint32_t r;
    asm("add.rn.f16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
    return r;
}
// Eq. 1 on two f16 lanes: min(|a|, |b|) carrying the XOR of the signs.
__device__ __forceinline__ uint32_t hf2(uint32_t a, uint32_t b) {
    uint32_t r;
    asm("min.xorsign.abs.f16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
    return r;
}
// Clamp both f16 lanes to [-127, 127] in one instruction: Eq. 1 with the constant
// 127 (0x57F0) is min(|v|, 127) with the sign of v.
__device__ __forceinline__ uint32_t hsat2(uint32_t v) { return hf2(v, 0x57F057F0u); }

// Four int8 LLRs as two f16x2 words: bytes 0, 1 in lo, bytes 2, 3 in hi.
struct H4 {
    uint32_t lo, hi;
};
// Byte x (in [-127, 127]) flipped to x + 128 = x ^ 0x80 under the exponent
// byte 0x64 is the f16 1024 + x + 128 (f16 steps by 1 in [1024, 2048)); adding
// -1152 (0xE480) leaves x exactly.
__device__ __forceinline__ H4 h4_unpack(uint32_t w) {
    const uint32_t u = w ^ 0x80808080u;
    return {hadd2(prmt(u, 0x64646464u, 0x4140u), 0xE480E480u),
            hadd2(prmt(u, 0x64646464u, 0x4342u), 0xE480E480u)};
}
// Back to bytes: for an integer x in [-254, 254], 1280 + x (0x6500 = 1280) lies
// in [1024, 2048), so its mantissa is 256 + x, whose low byte is x mod 256: the
// two's-complement byte. (-0 maps to 0.)
__device__ __forceinline__ uint32_t h4_pack(H4 v) {
    return prmt(hadd2(v.lo, 0x65006500u), hadd2(v.hi, 0x65006500u), 0x6420u);
}
// beta_l of 16 consecutive values (bit k for value k) as a word from which the sign
// bits of values 2i and 2i + 1, bits 15 and 31 of an f16 pair, are one shift left by
// 15 - 2i (a multiply per pair before: 4,096 int8 frames of (32768, 29492) 223 -> 216
// us, 16,384 mixed frames 312 -> 302 us).
__device__ __forceinline__ uint32_t spread16(uint32_t bits) { return bits | (bits << 15); }
// F / G / G_0R on four LLRs, values 4j..4j + 3 of the sixteen of `spread`. G flips
// the sign of alpha_v[i] where beta_l is 1 (Listing 3's sign XOR).
__device__ __forceinline__ H4 h4_flip(H4 a, uint32_t spread, uint32_t j) {
    return {a.lo ^ ((spread << (15u - 4u * j)) & 0x80008000u),
            a.hi ^ ((spread << (13u - 4u * j)) & 0x80008000u)};
}
template <uint32_t KIND>
__device__ __forceinline__ H4 h4_op(H4 a, H4 b, uint32_t spread, uint32_t j) {
    if constexpr (KIND == OP_F) {
        return {hf2(a.lo, b.lo), hf2(a.hi, b.hi)};
    } else if constexpr (KIND == OP_G) {
        a = h4_flip(a, spread, j);
        return {hsat2(hadd2(b.lo, a.lo)), hsat2(hadd2(b.hi, a.hi))};
    } else {
        return {hsat2(hadd2(b.lo, a.lo)), hsat2(hadd2(b.hi, a.hi))};
    }
}
template <uint32_t KIND>
__device__ __forceinline__ uint32_t op_i8x4(uint32_t a, uint32_t b, uint32_t spread, uint32_t j) {
    return h4_pack(h4_op<KIND>(h4_unpack(a), h4_unpack(b), spread, j));
}

// 32-bit word j of a 16-byte vector (j a constant after unrolling).
__device__ __forceinline__ uint32_t vword(const uint4 &v, uint32_t j) {
    return j == 0 ? v.x : (j == 1 ? v.y : (j == 2 ? v.z : v.w));
}
__device__ __forceinline__ void set_vword(uint4 &v, uint32_t j, uint32_t w) {
    if (j == 0) v.x = w;
    else if (j == 1) v.y = w;
    else if (j == 2) v.z = w;
    else v.w = w;
}

__device__ __forceinline__ bool is_neg(float a) { return a < 0.0f; }
__device__ __forceinline__ bool is_neg(int8_t a) { return a < 0; }

__device__ __forceinline__ unsigned long long spc_key(float a, uint32_t idx) {
    return (static_cast<unsigned long long>(__float_as_uint(fabsf(a))) << 32) | idx;
}
__device__ __forceinline__ unsigned long long spc_key(int8_t a, uint32_t idx) {
    return (static_cast<unsigned long long>(abs(static_cast<int>(a))) << 32) | idx;
}

template <typename T> struct Llr;
template <> struct Llr<float> {
    static constexpr uint32_t V = 4;  // elements per 16-byte vector
    using Acc = float;
    using Vec = float4;
};
template <> struct Llr<int8_t> {
    static constexpr uint32_t V = 16;
    using Acc = int;
    using Vec = uint4;
};

// ---------------------------------------------------------------- hinted device-memory reads

__device__ __forceinline__ unsigned long long evict_first_policy() {
    unsigned long long p;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
    return p;
}
template <uint32_t RD>
__device__ __forceinline__ uint4 ldv(const uint4 *p, unsigned long long pol) {
    if constexpr (RD == RD_NORMAL) {
        return *p;
    } else {
        uint4 r;
        asm volatile("ld.global.L2::cache_hint.v4.u32 {%0, %1, %2, %3}, [%4], %5;"
                     : "=r"(r.x), "=r"(r.y), "=r"(r.z), "=r"(r.w) : "l"(p), "l"(pol) : "memory");
        return r;
    }
}
template <uint32_t RD>
__device__ __forceinline__ float4 ldv(const float4 *p, unsigned long long pol) {
    if constexpr (RD == RD_NORMAL) {
        return *p;
    } else {
        float4 r;
        asm volatile("ld.global.L2::cache_hint.v4.f32 {%0, %1, %2, %3}, [%4], %5;"
                     : "=f"(r.x), "=f"(r.y), "=f"(r.z), "=f"(r.w) : "l"(p), "l"(pol) : "memory");
        return r;
    }
}
__device__ __forceinline__ unsigned long long evict_last_policy() {
    unsigned long long p;
    asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(p));
    return p;
}
struct Policies {  // the policies an operation needs, made once
    unsigned long long first, last;
    template <uint32_t RD, uint32_t WR>
    __device__ __forceinline__ static Policies of() {
        constexpr bool far = ((WR | (WR >> 2) | (WR >> 4)) & 1u) != 0u;
        constexpr bool near = ((WR | (WR >> 2) | (WR >> 4)) & 2u) != 0u;
        return {RD != RD_NORMAL || far ? evict_first_policy() : 0ull, near ? evict_last_policy() : 0ull};
    }
};
template <uint32_t ST, class Vec>
__device__ __forceinline__ void stv(Vec *p, const Vec &v, const Policies &pol) {
    if constexpr (ST == ST_NORMAL) {
        *p = v;
    } else {
        const uint4 x = *reinterpret_cast<const uint4 *>(&v);
        asm volatile("st.global.L2::cache_hint.v4.u32 [%0], {%1, %2, %3, %4}, %5;"
                     ::"l"(p), "r"(x.x), "r"(x.y), "r"(x.z), "r"(x.w),
                     "l"(ST == ST_FAR ? pol.first : pol.last) : "memory");
    }
}
__device__ __forceinline__ unsigned long long policy_for(uint32_t rd) {
    return rd == RD_NORMAL ? 0ull : evict_first_policy();
}

// ---------------------------------------------------------------- groups

struct WarpGrp {
    static constexpr bool kCta = false;
    __device__ static uint32_t rank() { return threadIdx.x & 31u; }
    __device__ static uint32_t size() { return 32u; }
    __device__ static void sync() { __syncwarp(); }
};
struct CtaGrp {
    static constexpr bool kCta = true;
    __device__ static uint32_t rank() { return threadIdx.x; }
    __device__ static uint32_t size() { return blockDim.x; }
    __device__ static void sync() { __syncthreads(); }
};

// Drop [p, p + bytes) of a scratch stage from L2 without writing it back
// (discard.global.L2: afterwards the bytes are undefined until written again).
// Call after a group barrier that follows the stage's last read; p 128-byte
// aligned, bytes a multiple of 128.
template <class Grp>
__device__ __forceinline__ void discard_l2(const void *p, uint32_t bytes) {
    for (uint32_t off = Grp::rank() * 128u; off < bytes; off += Grp::size() * 128u)
        asm volatile("discard.global.L2 [%0], 128;" ::"l"(static_cast<const char *>(p) + off)
                     : "memory");
}

// ---------------------------------------------------------------- beta helpers

// Replace bits [off, off+n) (n <= 32, inside one word) with the low n bits of v.
__device__ __forceinline__ void write_field(uint32_t *beta, uint32_t off, uint32_t n, uint32_t v) {
    if (n >= 32) {
        beta[off >> 5] = v;
        return;
    }
    const uint32_t p = off & 31u;
    const uint32_t fm = ((1u << n) - 1u) << p;
    uint32_t w = beta[off >> 5];
    w = (w & ~fm) | ((v << p) & fm);
    beta[off >> 5] = w;
}

__device__ __forceinline__ uint32_t bits_at(const uint32_t *beta, uint32_t pos, uint32_t nbits) {
    const uint32_t w = beta[pos >> 5] >> (pos & 31u);
    return nbits >= 32 ? w : (w & ((1u << nbits) - 1u));
}

// ---------------------------------------------------------------- F / G / G_0R in memory

template <uint32_t KIND>
__device__ __forceinline__ float4 fg4(float4 a, float4 b, uint32_t bits) {
    float4 r;
    if (KIND == OP_F) {
        r.x = f_f32(a.x, b.x); r.y = f_f32(a.y, b.y); r.z = f_f32(a.z, b.z); r.w = f_f32(a.w, b.w);
    } else if (KIND == OP_G) {
        r.x = g_f32(a.x, b.x, bits & 1u);
        r.y = g_f32(a.y, b.y, (bits >> 1) & 1u);
        r.z = g_f32(a.z, b.z, (bits >> 2) & 1u);
        r.w = g_f32(a.w, b.w, (bits >> 3) & 1u);
    } else {
        r.x = b.x + a.x; r.y = b.y + a.y; r.z = b.z + a.z; r.w = b.w + a.w;
    }
    return r;
}
template <uint32_t KIND>
__device__ __forceinline__ uint4 fg4(uint4 a, uint4 b, uint32_t bits) {
    uint4 r;
    const uint32_t s = spread16(bits);
    r.x = op_i8x4<KIND>(a.x, b.x, s, 0);
    r.y = op_i8x4<KIND>(a.y, b.y, s, 1);
    r.z = op_i8x4<KIND>(a.z, b.z, s, 2);
    r.w = op_i8x4<KIND>(a.w, b.w, s, 3);
    return r;
}

template <uint32_t KIND, typename T>
__device__ __forceinline__ T fg_scalar(T a, T b, uint32_t bit) {
    using Acc = typename Llr<T>::Acc;
    const Acc x = a, y = b;
    return static_cast<T>(KIND == OP_F ? op_f(x, y) : (KIND == OP_G ? op_g(x, y, bit) : op_add(x, y)));
}

// out[i] = op(in[i], in[i + h]) for i < h; in and out never overlap. Four vectors
// per thread are loaded before any is used, so device-memory operands (the
// channel at the root, scratch stages) overlap their latency.
template <typename T, class Grp, uint32_t KIND, uint32_t RD = RD_NORMAL, uint32_t WR = 0u>
__device__ __forceinline__ void op_fg(const T *__restrict__ in, T *__restrict__ out, uint32_t h,
                                      const uint32_t *beta, uint32_t o) {
    using Vec = typename Llr<T>::Vec;
    constexpr uint32_t V = Llr<T>::V;
    if (h >= V) {
        const uint32_t nv = h / V, G = Grp::size();
        const Vec *va = reinterpret_cast<const Vec *>(in);
        const Vec *vb = reinterpret_cast<const Vec *>(in + h);
        Vec *vo = reinterpret_cast<Vec *>(out);
        const Policies pol = Policies::of<RD, WR>();
        uint32_t v = Grp::rank();
        for (; v + 3 * G < nv; v += 4 * G) {
            Vec a[4], b[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                a[k] = ldv<RD>(va + v + k * G, pol.first);
                b[k] = ldv<RD>(vb + v + k * G, pol.first);
            }
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const uint32_t bits = KIND == OP_G ? bits_at(beta, o + (v + k * G) * V, V) : 0u;
                stv<WR & 3u>(vo + v + k * G, fg4<KIND>(a[k], b[k], bits), pol);
            }
        }
        for (; v < nv; v += G) {
            const uint32_t bits = KIND == OP_G ? bits_at(beta, o + v * V, V) : 0u;
            stv<WR & 3u>(vo + v, fg4<KIND>(ldv<RD>(va + v, pol.first), ldv<RD>(vb + v, pol.first), bits), pol);
        }
    } else {
        for (uint32_t i = Grp::rank(); i < h; i += Grp::size()) {
            const uint32_t bit = KIND == OP_G ? bits_at(beta, o + i, 1) : 0u;
            out[i] = fg_scalar<KIND, T>(in[i], in[i + h], bit);
        }
    }
}

// A chain of L = 2 or 3 operations down the tree, fused: K0 on node (o, n)
// (F, G or G_0R), then K1 and K2 (F or G_0R) on the node of the next stage
// that the previous operation produced the LLRs of. In list order these are
// consecutive operations, each reading the stage the one before it just
// wrote. Here every thread loads the 2^L inputs of one column of outputs
// (elements j + m n / 2^L of stage n) once, keeps the intermediate values in
// registers and stores each intermediate stage as well (a later operation
// reads it again) and the last one. Element by element this is the same
// arithmetic as the L operations one after another. stage1/2/3 = stages n/2,
// n/4, n/8; (n >> L) must be a multiple of the vector width.
// STORE: bit 0 stores stage n/2, bit 1 stage n/4 (for L = 3; the last stage
// is always stored): an intermediate stage that no later operation reads is
// not written at all. RD: how the input stage is read (see RD_LAST).
template <typename T, class Grp, uint32_t L, uint32_t K0, uint32_t K1, uint32_t K2,
          uint32_t STORE = 3u, uint32_t RD = RD_NORMAL, uint32_t WR = 0u>
__device__ __forceinline__ void op_chain(const T *__restrict__ in, T *__restrict__ stage1,
                                         T *__restrict__ stage2, T *__restrict__ stage3,
                                         uint32_t n, const uint32_t *beta, uint32_t o) {
    using Vec = typename Llr<T>::Vec;
    constexpr uint32_t V = Llr<T>::V, M = 1u << L;
    const uint32_t nvc = (n >> L) / V;  // vector columns of the last stage
    const Vec *vi = reinterpret_cast<const Vec *>(in);
    Vec *v1 = reinterpret_cast<Vec *>(stage1);
    Vec *v2 = reinterpret_cast<Vec *>(stage2);
    Vec *v3 = reinterpret_cast<Vec *>(stage3);
    const Policies pol = Policies::of<RD, WR>();
    for (uint32_t c = Grp::rank(); c < nvc; c += Grp::size()) {
        Vec x[M];
#pragma unroll
        for (uint32_t m = 0; m < M; ++m) x[m] = ldv<RD>(vi + c + m * nvc, pol.first);
        if constexpr (sizeof(T) == 1) {
            // int8: word by word in f16 pairs; intermediate stages are packed
            // back to bytes only where they are stored
            uint32_t gb[M / 2];
#pragma unroll
            for (uint32_t m = 0; m < M / 2; ++m)
                gb[m] = K0 == OP_G ? spread16(bits_at(beta, o + (c + m * nvc) * V, V)) : 0u;
            Vec y[M / 2], z[M / 4], w;
#pragma unroll
            for (uint32_t j = 0; j < 4; ++j) {
                H4 xh[M], yh[M / 2], zh[M / 4];
#pragma unroll
                for (uint32_t m = 0; m < M; ++m) xh[m] = h4_unpack(vword(x[m], j));
#pragma unroll
                for (uint32_t m = 0; m < M / 2; ++m) {
                    yh[m] = h4_op<K0>(xh[m], xh[m + M / 2], gb[m], j);
                    if (STORE & 1u) set_vword(y[m], j, h4_pack(yh[m]));
                }
#pragma unroll
                for (uint32_t m = 0; m < M / 4; ++m) {
                    zh[m] = h4_op<K1>(yh[m], yh[m + M / 4], 0u, j);
                    if (L == 2 || (STORE & 2u)) set_vword(z[m], j, h4_pack(zh[m]));
                }
                if constexpr (L == 3) set_vword(w, j, h4_pack(h4_op<K2>(zh[0], zh[1], 0u, j)));
            }
#pragma unroll
            for (uint32_t m = 0; m < M / 2; ++m)
                if (STORE & 1u) stv<WR & 3u>(v1 + c + m * nvc, y[m], pol);
#pragma unroll
            for (uint32_t m = 0; m < M / 4; ++m)
                if (L == 2 || (STORE & 2u)) stv<(WR >> 2) & 3u>(v2 + c + m * nvc, z[m], pol);
            if constexpr (L == 3) stv<(WR >> 4) & 3u>(v3 + c, w, pol);
        } else {
            Vec y[M / 2];
#pragma unroll
            for (uint32_t m = 0; m < M / 2; ++m) {
                const uint32_t bits = K0 == OP_G ? bits_at(beta, o + (c + m * nvc) * V, V) : 0u;
                y[m] = fg4<K0>(x[m], x[m + M / 2], bits);
                if (STORE & 1u) stv<WR & 3u>(v1 + c + m * nvc, y[m], pol);
            }
            Vec z[M / 4];
#pragma unroll
            for (uint32_t m = 0; m < M / 4; ++m) {
                z[m] = fg4<K1>(y[m], y[m + M / 4], 0u);
                if (L == 2 || (STORE & 2u)) stv<(WR >> 2) & 3u>(v2 + c + m * nvc, z[m], pol);
            }
            if constexpr (L == 3) stv<(WR >> 4) & 3u>(v3 + c, fg4<K2>(z[0], z[1], 0u), pol);
        }
    }
}

// ---------------------------------------------------------------- Combine / Rate-0 in memory

template <class Grp>
__device__ __forceinline__ void op_combine(uint32_t *beta, uint32_t n, uint32_t o, bool copy) {
    const uint32_t h = n >> 1;
    if (h >= 32) {
        const uint32_t wl = o >> 5, wr = (o + h) >> 5, nw = h >> 5;
        for (uint32_t j = Grp::rank(); j < nw; j += Grp::size()) {
            const uint32_t r = beta[wr + j];
            beta[wl + j] = copy ? r : (beta[wl + j] ^ r);
        }
    } else if (Grp::rank() == 0) {
        const uint32_t p = o & 31u, fm = (1u << h) - 1u;
        uint32_t w = beta[o >> 5];
        const uint32_t r = (w >> (p + h)) & fm;
        const uint32_t l = copy ? r : (((w >> p) & fm) ^ r);
        beta[o >> 5] = (w & ~(fm << p)) | (l << p);
    }
}

template <class Grp>
__device__ __forceinline__ void op_r0(uint32_t *beta, uint32_t n, uint32_t o) {
    if (n >= 32) {
        for (uint32_t j = Grp::rank(); j < (n >> 5); j += Grp::size()) beta[(o >> 5) + j] = 0u;
    } else if (Grp::rank() == 0) {
        write_field(beta, o, n, 0u);
    }
}

// ---------------------------------------------------------------- node decoders in memory

// Sign bits of the 16 int8 values of v, value k at bit k. Per word the sign
// bits 7, 15, 23, 31 are moved to bits 28..31 by one multiply (the partial
// products of 0x00204081 land on distinct bits, so nothing carries).
__device__ __forceinline__ uint32_t sign_bits16(uint4 v) {
    const uint32_t m0 = ((v.x & 0x80808080u) * 0x00204081u) >> 28;
    const uint32_t m1 = ((v.y & 0x80808080u) * 0x00204081u) >> 28;
    const uint32_t m2 = ((v.z & 0x80808080u) * 0x00204081u) >> 28;
    const uint32_t m3 = ((v.w & 0x80808080u) * 0x00204081u) >> 28;
    return m0 | (m1 << 4) | (m2 << 8) | (m3 << 12);
}

// Rate-1 (Eq. 4) on int8 LLRs, n >= 32: 16 values per lane per 16-byte load;
// lanes 2j and 2j + 1 of a warp hold the two halves of one beta word. Four
// loads per lane are in flight before the first is used.
template <class Grp>
__device__ __forceinline__ void op_r1_i8v(const int8_t *__restrict__ in, uint32_t *beta,
                                          uint32_t n, uint32_t o) {
    const uint4 *v = reinterpret_cast<const uint4 *>(in);
    const uint32_t nv = n >> 4, lane = threadIdx.x & 31u;
    const uint32_t w0 = Grp::kCta ? (threadIdx.x & ~31u) : 0u;
    const uint32_t step = Grp::kCta ? blockDim.x : 32u;
    for (uint32_t base = w0; base < nv; base += 4 * step) {
        uint32_t m[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const uint32_t i = base + k * step + lane;
            m[k] = i < nv ? sign_bits16(v[i]) : 0u;
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const uint32_t i = base + k * step + lane;
            const uint32_t hi = __shfl_down_sync(kFull, m[k], 1);
            if (i < nv && !(lane & 1u)) beta[(o >> 5) + (i >> 1)] = m[k] | (hi << 16);
        }
    }
}

// Rate-1 (Eq. 4) on float32 LLRs, n >= 128: four values per lane per 16-byte
// load; the eight lanes 8w..8w+7 of a warp hold the 32 values of one beta word
// and OR their 4-bit pieces together with three shuffles. Four loads per lane
// are in flight before the first is used.
template <class Grp>
__device__ __forceinline__ void op_r1_f32v(const float *__restrict__ in, uint32_t *beta,
                                           uint32_t n, uint32_t o) {
    const float4 *v = reinterpret_cast<const float4 *>(in);
    const uint32_t nv = n >> 2, lane = threadIdx.x & 31u;
    const uint32_t w0 = Grp::kCta ? (threadIdx.x & ~31u) : 0u;
    const uint32_t step = Grp::kCta ? blockDim.x : 32u;
    for (uint32_t base = w0; base < nv; base += 4 * step) {
        uint32_t m[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const uint32_t i = base + k * step + lane;
            uint32_t b = 0;
            if (i < nv) {
                const float4 x = v[i];  // x + 0 has its sign set exactly when x < 0 (-0 decides 0)
                b = (__float_as_uint(x.x + 0.0f) >> 31) | ((__float_as_uint(x.y + 0.0f) >> 30) & 2u) |
                    ((__float_as_uint(x.z + 0.0f) >> 29) & 4u) | ((__float_as_uint(x.w + 0.0f) >> 28) & 8u);
            }
            m[k] = b << (4u * (lane & 7u));
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const uint32_t i = base + k * step + lane;
            uint32_t w = m[k];
            w |= __shfl_xor_sync(kFull, w, 1);
            w |= __shfl_xor_sync(kFull, w, 2);
            w |= __shfl_xor_sync(kFull, w, 4);
            if (i < nv && !(lane & 7u)) beta[(o >> 5) + (i >> 3)] = w;
        }
    }
}

// Rate-1 (Eq. 4): one ballot per 32 consecutive elements; four chunks loaded ahead.
template <typename T, class Grp>
__device__ __forceinline__ void op_r1(const T *__restrict__ in, uint32_t *beta, uint32_t n,
                                      uint32_t o) {
    if constexpr (sizeof(T) == 1) {
        if (n >= 32) {
            op_r1_i8v<Grp>(reinterpret_cast<const int8_t *>(in), beta, n, o);
            return;
        }
    } else {
        if (n >= 128) {
            op_r1_f32v<Grp>(reinterpret_cast<const float *>(in), beta, n, o);
            return;
        }
    }
    const uint32_t lane = threadIdx.x & 31u;
    const uint32_t w0 = Grp::kCta ? (threadIdx.x >> 5) : 0u;
    const uint32_t ws = Grp::kCta ? (blockDim.x >> 5) : 1u;
    const uint32_t nch = (n + 31u) >> 5;
    uint32_t c = w0;
    for (; c + 3 * ws < nch; c += 4 * ws) {
        T a[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) a[k] = in[((c + k * ws) << 5) + lane];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const uint32_t bal = __ballot_sync(kFull, is_neg(a[k]));
            if (lane == 0) beta[(o >> 5) + c + k * ws] = bal;
        }
    }
    for (; c < nch; c += ws) {
        const uint32_t idx = (c << 5) + lane;
        const bool neg = idx < n && is_neg(in[idx]);
        const uint32_t bal = __ballot_sync(kFull, neg);
        if (lane == 0) write_field(beta, o + (c << 5), n < 32 ? n : 32, bal);
    }
}

// Signs of G on the 16 int8 values of one vector pair, value k at bit k (bits = beta_l).
// The clamp of the int8 sum keeps its sign, and the sums are never -0 (a byte 0
// enters as +0).
__device__ __forceinline__ uint32_t g_signs(uint4 a, uint4 b, uint32_t bits) {
    uint32_t t = 0;
    const uint32_t s = spread16(bits);
#pragma unroll
    for (uint32_t j = 0; j < 4; ++j) {
        const H4 x = h4_flip(h4_unpack(vword(a, j)), s, j);
        const H4 y = h4_unpack(vword(b, j));
        const uint32_t lo = hadd2(y.lo, x.lo), hi = hadd2(y.hi, x.hi);
        t |= (((lo >> 15) & 0x00010001u) | ((hi >> 13) & 0x00040004u)) << (4 * j);
    }
    return (t | (t >> 15)) & 0xFFFFu;
}
// int8 G of node (o, 2h) and the Rate-1 decision of its right child (o + h, h) in one
// pass of a warp, h >= 32: the child's LLRs are only looked at for their signs, so
// they are neither stored nor read back. In a high-rate code the wide right children
// are Rate-1 nodes. Loads four vector pairs ahead; two lanes join their bits into a
// word. For several frames per CTA (the generator says why): two operations instead,
// 206 us, now 202 for 4,096 frames of (32768, 29492), 16,384 mixed frames 283, now 275.
template <uint32_t RD = RD_NORMAL>
__device__ __forceinline__ void op_g_r1(const int8_t *__restrict__ in, uint32_t h, uint32_t *beta,
                                        uint32_t o) {
    using Vec = uint4;
    constexpr uint32_t V = 16, L = 2;
    const Vec *va = reinterpret_cast<const Vec *>(in);
    const Vec *vb = reinterpret_cast<const Vec *>(in + h);
    const uint32_t nv = h / V, lane = threadIdx.x & 31u;
    const unsigned long long pol = policy_for(RD);
    for (uint32_t base = 0; base < nv; base += 4 * 32u) {
        Vec a[4], b[4];
#pragma unroll
        for (uint32_t k = 0; k < 4; ++k) {
            const uint32_t i = base + 32u * k + lane;
            if (i < nv) {
                a[k] = ldv<RD>(va + i, pol);
                b[k] = ldv<RD>(vb + i, pol);
            }
        }
#pragma unroll
        for (uint32_t k = 0; k < 4; ++k) {
            const uint32_t i = base + 32u * k + lane;
            uint32_t m = i < nv ? g_signs(a[k], b[k], bits_at(beta, o + i * V, V)) : 0u;
            m <<= V * (lane & (L - 1u));
#pragma unroll
            for (uint32_t x = 1; x < L; x *= 2) m |= __shfl_xor_sync(kFull, m, x);
            if (i < nv && !(lane & (L - 1u))) beta[((o + h) >> 5) + i / L] = m;
        }
    }
}

// SPC on int8 LLRs, n >= 512 (see op_spc): 16 values per lane per 16-byte load, four
// loads ahead. A vector's least magnitude is a chain of Eq. 1 over its f16 pairs
// (signs ignored), and its f16 bits above the vector's index make one key, whose
// minimum over the group names the first vector that holds the node's least
// magnitude; the value is looked up there at the end. (One value per lane per load
// before, four loads ahead: a 4,096-value node of a throughput frame waited 32 times
// for memory: 216 -> 206 us for 4,096 frames of (32768, 29492).)
template <class Grp>
__device__ __forceinline__ void op_spc_i8v(const int8_t *__restrict__ in, uint32_t *beta, uint32_t n,
                                           uint32_t o, unsigned long long *rkey, uint32_t *rpar) {
    const uint4 *v = reinterpret_cast<const uint4 *>(in);
    const uint32_t nv = n >> 4, lane = threadIdx.x & 31u;
    const uint32_t w0 = Grp::kCta ? (threadIdx.x & ~31u) : 0u, step = Grp::size();
    uint32_t key = kFull, par = 0;
    for (uint32_t base = w0; base < nv; base += 4 * step) {
        uint4 x[4];
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (base + k * step + lane < nv) x[k] = v[base + k * step + lane];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const uint32_t i = base + k * step + lane;
            uint32_t m = 0;
            if (i < nv) {
                m = sign_bits16(x[k]);
                par ^= m;
                const H4 p = h4_unpack(x[k].x), q = h4_unpack(x[k].y), r = h4_unpack(x[k].z),
                         s = h4_unpack(x[k].w);
                const uint32_t least = hf2(hf2(hf2(p.lo, p.hi), hf2(q.lo, q.hi)),
                                           hf2(hf2(r.lo, r.hi), hf2(s.lo, s.hi))) & 0x7fff7fffu;
                key = min(key, (min(least & 0xffffu, least >> 16) << 16) | i);
            }
            const uint32_t hi = __shfl_down_sync(kFull, m, 1);
            if (i < nv && !(lane & 1u)) beta[(o >> 5) + (i >> 1)] = m | (hi << 16);
        }
    }
    key = __reduce_min_sync(kFull, key);
    par = __reduce_xor_sync(kFull, par);
    if (Grp::kCta) {
        const uint32_t w = threadIdx.x >> 5;
        if (lane == 0) {
            rkey[w] = key;
            rpar[w] = par;
        }
        Grp::sync();
        if (w != 0) return;
        const bool has = lane < (Grp::size() >> 5);
        key = __reduce_min_sync(kFull, has ? static_cast<uint32_t>(rkey[lane]) : kFull);
        par = __reduce_xor_sync(kFull, has ? rpar[lane] : 0u);
    } else {
        Grp::sync();  // the words written above, before one of them is changed
    }
    const uint32_t first = (key & 0xffffu) << 4;
    const float a = fabsf(static_cast<float>(in[first + (lane & 15u)]));
    float mag;
    asm("{\n .reg .b16 h, g;\n mov.b32 {g, h}, %1;\n cvt.f32.f16 %0, h;\n}\n" : "=f"(mag) : "r"(key));
    const uint32_t at = __ballot_sync(kFull, a == mag);
    if (lane == 0 && (__popc(par) & 1u)) {
        const uint32_t pos = o + first + static_cast<uint32_t>(__ffs(static_cast<int>(at))) - 1u;
        beta[pos >> 5] ^= 1u << (pos & 31u);
    }
}

// SPC: hard decisions, their parity, flip the least-|alpha| (lowest index)
// decision when the parity is odd (Listing 2 returns the first lane equal to
// the minimum).
// VEC = false keeps the one-value form for int8 too: in the out-of-line copies, where the
// vector form multiplies the compile time of a list of thousands of calls, and in the
// interpreter, whose 64 registers its four vectors overrun (208 bytes of spills; one int8
// frame of (32768, 29491): 539 us, 599 with it).
template <typename T, class Grp, bool VEC = true>
__device__ __forceinline__ void op_spc(const T *__restrict__ in, uint32_t *beta, uint32_t n,
                                       uint32_t o, unsigned long long *rkey, uint32_t *rpar) {
    if constexpr (VEC && sizeof(T) == 1) {
        if (n >= 512) {
            op_spc_i8v<Grp>(reinterpret_cast<const int8_t *>(in), beta, n, o, rkey, rpar);
            return;
        }
    }
    const uint32_t lane = threadIdx.x & 31u;
    const uint32_t w0 = Grp::kCta ? (threadIdx.x >> 5) : 0u;
    const uint32_t ws = Grp::kCta ? (blockDim.x >> 5) : 1u;
    const uint32_t nch = (n + 31u) >> 5;
    unsigned long long kmin = ~0ull;
    uint32_t par = 0;
    uint32_t c = w0;
    for (; c + 3 * ws < nch; c += 4 * ws) {
        T a[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) a[k] = in[((c + k * ws) << 5) + lane];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const uint32_t bal = __ballot_sync(kFull, is_neg(a[k]));
            par ^= __popc(bal) & 1u;
            if (lane == 0) beta[(o >> 5) + c + k * ws] = bal;
            const unsigned long long key = spc_key(a[k], ((c + k * ws) << 5) + lane);
            kmin = key < kmin ? key : kmin;
        }
    }
    for (; c < nch; c += ws) {
        const uint32_t idx = (c << 5) + lane;
        const bool valid = idx < n;
        const T a = valid ? in[idx] : T(0);
        const uint32_t bal = __ballot_sync(kFull, valid && is_neg(a));
        par ^= __popc(bal) & 1u;
        if (lane == 0) write_field(beta, o + (c << 5), n < 32 ? n : 32, bal);
        if (valid) {
            const unsigned long long key = spc_key(a, idx);
            kmin = key < kmin ? key : kmin;
        }
    }
#pragma unroll
    for (uint32_t s = 16; s > 0; s >>= 1) {
        const unsigned long long t = __shfl_xor_sync(kFull, kmin, s);
        kmin = t < kmin ? t : kmin;
    }
    if (Grp::kCta) {
        const uint32_t w = threadIdx.x >> 5;
        if (lane == 0) {
            rkey[w] = kmin;
            rpar[w] = par;
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            uint32_t p = 0;
            for (uint32_t i = 0; i < ws; ++i) {
                kmin = rkey[i] < kmin ? rkey[i] : kmin;
                p ^= rpar[i];
            }
            if (p) {
                const uint32_t pos = o + static_cast<uint32_t>(kmin & 0xffffffffull);
                beta[pos >> 5] ^= 1u << (pos & 31u);
            }
        }
    } else if (lane == 0 && par) {
        const uint32_t pos = o + static_cast<uint32_t>(kmin & 0xffffffffull);
        beta[pos >> 5] ^= 1u << (pos & 31u);
    }
}

// Repetition: the sum of alpha_v folded as t[i] <- t[i] + t[i + m],
// m = n/2, n/4, ..., 1 (the G_0R chain SC computes on this node); the bit is
// (sum < 0), replicated. Folds above 64 values run in memory (tmp = the free
// stage n/2), the last ones as warp shuffles with the same pairing.
template <typename T, class Grp>
__device__ __forceinline__ void op_rep(const T *in, T *tmp, uint32_t *beta, uint32_t n,
                                       uint32_t o) {
    using Acc = typename Llr<T>::Acc;
    uint32_t len = n;
    const T *src = in;
    while (len > 64) {
        const uint32_t m = len >> 1;
        if (src == tmp) {
            for (uint32_t i = Grp::rank(); i < m; i += Grp::size())
                tmp[i] = fg_scalar<OP_G0R, T>(tmp[i], tmp[i + m], 0u);
        } else {
            op_fg<T, Grp, OP_G0R>(src, tmp, m, nullptr, 0);
        }
        Grp::sync();
        src = tmp;
        len = m;
    }
    // the last folds: warp 0 of the CTA (CTA group), or the calling warp
    if (!Grp::kCta || threadIdx.x < 32) {
        const uint32_t lane = threadIdx.x & 31u;
        Acc x;
        uint32_t cur;
        if (len == 64) {
            x = op_add(static_cast<Acc>(src[lane]), static_cast<Acc>(src[lane + 32]));
            cur = 32;
        } else {
            x = lane < len ? static_cast<Acc>(src[lane]) : Acc(0);
            cur = len;
        }
        while (cur > 1) {
            cur >>= 1;
            const Acc y = __shfl_down_sync(kFull, x, cur);
            if (lane < cur) x = op_add(x, y);
        }
        const Acc s = __shfl_sync(kFull, x, 0);
        const uint32_t word = s < Acc(0) ? kFull : 0u;
        if (n >= 32) {
            for (uint32_t j = lane; j < (n >> 5); j += 32) beta[(o >> 5) + j] = word;
        } else if (lane == 0) {
            write_field(beta, o, n, word);
        }
    }
}

// ---------------------------------------------------------------- frame state

template <typename T>
struct Frame {
    const T *chan;     // channel LLRs of the frame (shared or device memory)
    T *s_alpha;        // shared alpha array (stage n at [n, 2n), n <= S)
    T *g_alpha;        // device scratch (stage n at [n - 2S, 2n - 2S), n > S)
    uint32_t *beta;    // shared beta bits
    unsigned long long *rkey;
    uint32_t *rpar;
    uint32_t N, S;
    __device__ __forceinline__ const T *stage_in(uint32_t n) const {
        return n == N ? chan : (n <= S ? s_alpha + n : g_alpha + (n - 2 * S));
    }
    __device__ __forceinline__ T *stage(uint32_t n) const {
        return n <= S ? s_alpha + n : g_alpha + (n - 2 * S);
    }
};

template <typename T, class Grp>
__device__ __forceinline__ void exec_op(uint32_t kind, uint32_t n, uint32_t o, const Frame<T> &fr) {
    switch (kind) {
    case OP_F: op_fg<T, Grp, OP_F>(fr.stage_in(n), fr.stage(n >> 1), n >> 1, fr.beta, o); break;
    case OP_G: op_fg<T, Grp, OP_G>(fr.stage_in(n), fr.stage(n >> 1), n >> 1, fr.beta, o); break;
    case OP_G0R: op_fg<T, Grp, OP_G0R>(fr.stage_in(n), fr.stage(n >> 1), n >> 1, fr.beta, o); break;
    case OP_C: op_combine<Grp>(fr.beta, n, o, false); break;
    case OP_C0R: op_combine<Grp>(fr.beta, n, o, true); break;
    case OP_R0: op_r0<Grp>(fr.beta, n, o); break;
    case OP_R1: op_r1<T, Grp>(fr.stage_in(n), fr.beta, n, o); break;
    case OP_REP: op_rep<T, Grp>(fr.stage_in(n), fr.stage(n >> 1), fr.beta, n, o); break;
    default: op_spc<T, Grp, false>(fr.stage_in(n), fr.beta, n, o, fr.rkey, fr.rpar); break;
    }
}

// ---------------------------------------------------------------- packed output

// Write a frame's information bits: the estimate x_hat (beta) restricted to the
// information set, packed LSB first into out_row bytes; beta is used up.
// First the few words that mix frozen and information bits are packed to their
// bottoms in place: the compress of H. S. Warren, "Hacker's Delight" (7-4), five
// moves right by 1, 2, 4, 8, 16 with masks the host made once. Then one lane
// forms one 32-bit output word from the beta words it draws on (two for a dense
// set), and a warp stores 32 of them as aligned words whatever the row's
// alignment, the bytes shifted through the neighbouring lane's word.
// Packing is instruction-bound. A bit-by-bit loop was a fifth of a throughput
// frame's instructions; with the compress done per output word and lane, where
// one mixed word made its whole warp wait, it was an eighth. (1024, 512), 10,000
// float32 frames: 45.1, 32.9, 31.0 us; (32768, 29492), 4,096 int8 frames: 327,
// 275, 260 us for the three forms.
template <class Grp, class Tables>
__device__ __forceinline__ void pack_bits(uint32_t *beta, const Tables &a, uint8_t *out) {
    const uint32_t lane = threadIdx.x & 31u;
    const uint32_t first = Grp::kCta ? (threadIdx.x & ~31u) : 0u;
    const uint32_t step = Grp::kCta ? blockDim.x : 32u;
    const uint32_t sh = static_cast<uint32_t>(reinterpret_cast<uintptr_t>(out)) & 3u;
    for (uint32_t i = Grp::rank(); i < a.n_part; i += Grp::size()) {
        const uint4 *rec = reinterpret_cast<const uint4 *>(a.ext_part) + 2 * i;
        const uint4 p = __ldg(rec), q = __ldg(rec + 1);
        const uint32_t v[5] = {p.z, p.w, q.x, q.y, q.z};
        uint32_t x = beta[p.x] & p.y;
#pragma unroll
        for (int k = 0; k < 5; ++k) x = (x & ~v[k]) | ((x & v[k]) >> (1 << k));
        beta[p.x] = x;
    }
    Grp::sync();
    for (uint32_t u0 = first; u0 < a.KW; u0 += step) {
        uint32_t acc = 0;
        if (u0 + lane < a.KW) {
            const uint32_t st = __ldg(a.ext_start + u0 + lane);
            uint32_t w = st >> 5;
            // the word the output word starts in, without the bits before it
            uint32_t pos = __popc(__ldg(a.ext_mask + w)) - (st & 31u);
            acc = beta[w] >> (st & 31u);
            while (pos < 32 && ++w < a.NW) {
                const uint32_t c = __popc(__ldg(a.ext_mask + w));
                if (c) acc |= beta[w] << pos;
                pos += c;
            }
        }
        // this lane's aligned word: bytes [4 lane - sh, 4 lane - sh + 4) of the
        // warp's `left` bytes
        const uint32_t prev = __shfl_up_sync(kFull, acc, 1);
        const uint32_t word = __funnelshift_l(lane ? prev : 0u, acc, 8u * sh);
        const int lo = static_cast<int>(4u * lane) - static_cast<int>(sh);
        const int left = static_cast<int>(min(128u, a.out_row - 4u * u0));
        uint8_t *dst = out + 4u * size_t(u0) + lo;
        if (lo >= 0 && lo + 4 <= left) {
            *reinterpret_cast<uint32_t *>(dst) = word;
        } else {
#pragma unroll
            for (int b = 0; b < 4; ++b)
                if (lo + b >= 0 && lo + b < left) dst[b] = static_cast<uint8_t>(word >> (8 * b));
        }
        if (sh && lane == 31u) {  // the last sh bytes of the last lane's word
            for (uint32_t b = 4u - sh; b < 4u; ++b)
                if (static_cast<int>(124u + b) < left)
                    out[4u * size_t(u0) + 124u + b] = static_cast<uint8_t>(acc >> (8 * b));
        }
    }
}

// ---------------------------------------------------------------- bulk copy

__device__ __forceinline__ uint32_t smem_u32(const void *p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ unsigned long long globaltimer() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}
__device__ __forceinline__ void mbar_init(uint64_t *bar) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void bulk_load(void *dst, const void *src, uint32_t bytes, uint64_t *bar) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;"
                 ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
        ::"r"(smem_u32(dst)), "l"(src), "r"(bytes), "r"(smem_u32(bar)) : "memory");
}
// Bounded wait for the phase with the given parity; false after limit_ns (or
// kWaitPolls polls).
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, uint32_t parity,
                                          unsigned long long limit_ns = kWaitNs) {
    const unsigned long long t0 = globaltimer();
    for (uint32_t i = 0; i < kWaitPolls; ++i) {
        uint32_t ok;
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
            " selp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(ok) : "r"(smem_u32(bar)), "r"(parity) : "memory");
        if (ok) return true;
        if ((i & 63u) == 63u && globaltimer() - t0 > limit_ns) return false;
    }
    return false;
}

// ---------------------------------------------------------------- frame loop

// Persistent loop over the frames of a launch: frame f goes to CTA f % grid.
// For each frame `body(fr, trace_row)` runs the operation list; afterwards the
// estimate x_hat restricted to A is packed LSB first (output word u = info bits
// [32u, 32u+32)). With STAGE the frame's LLRs are brought into shared memory
// by cp.async.bulk, two frames ahead of use.
template <typename T, bool TRACE, bool STAGE, class Body>
__device__ __forceinline__ void run_frames(const KernelArgs &a, const Body &body) {
    extern __shared__ __align__(128) unsigned char smem[];
    const SmemLayout L(a.N, a.S, sizeof(T), STAGE);
    const uint32_t tid = threadIdx.x;

    Frame<T> fr;
    fr.s_alpha = reinterpret_cast<T *>(smem + L.alpha);
    fr.g_alpha = a.gscratch ? static_cast<T *>(a.gscratch) + size_t(blockIdx.x) * a.gstride
                            : nullptr;
    fr.beta = reinterpret_cast<uint32_t *>(smem + L.beta);
    fr.rkey = reinterpret_cast<unsigned long long *>(smem + L.rkey);
    fr.rpar = reinterpret_cast<uint32_t *>(smem + L.rpar);
    fr.N = a.N;
    fr.S = a.S;

    T *const chan0 = reinterpret_cast<T *>(smem + L.chan0);
    T *const chan1 = reinterpret_cast<T *>(smem + L.chan1);
    uint64_t *mbar = reinterpret_cast<uint64_t *>(smem + L.mbar);
    const uint32_t chan_bytes = a.N * static_cast<uint32_t>(sizeof(T));
    const T *llr = static_cast<const T *>(a.llr);
    const size_t G = gridDim.x;

    if (STAGE) {
        if (tid == 0) {
            mbar_init(&mbar[0]);
            mbar_init(&mbar[1]);
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
            if (blockIdx.x < a.n_frames)
                bulk_load(chan0, llr + size_t(blockIdx.x) * a.N, chan_bytes, &mbar[0]);
            if (blockIdx.x + G < a.n_frames)
                bulk_load(chan1, llr + (blockIdx.x + G) * a.N, chan_bytes, &mbar[1]);
        }
        __syncthreads();
    }

    uint32_t it = 0;
    for (size_t f = blockIdx.x; f < a.n_frames; f += G, ++it) {
        if (STAGE) {
            const uint32_t b = it & 1u;
            const bool bad = !mbar_wait(&mbar[b], (it >> 1) & 1u);
            if (__syncthreads_or(bad)) {
                if (tid == 0) atomicOr(a.status, 1);
                // let any copy still in flight land before the CTA's shared memory is released
                mbar_wait(&mbar[b], (it >> 1) & 1u);
                if (f + G < a.n_frames) mbar_wait(&mbar[b ^ 1u], ((it + 1) >> 1) & 1u);
                return;
            }
            fr.chan = b ? chan1 : chan0;
        } else {
            fr.chan = llr + f * a.N;
        }
        float *trace_row = TRACE ? a.trace + f * a.trace_stride : nullptr;

        body(fr, trace_row);

        pack_bits<CtaGrp>(fr.beta, a, a.out + f * a.out_row);
        __syncthreads();

        if (STAGE && tid == 0 && f + 2 * G < a.n_frames) {
            // every thread is done reading this buffer (barrier above); order those
            // generic-proxy reads before the async-proxy write of the next frame
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            bulk_load((it & 1u) ? chan1 : chan0, llr + (f + 2 * G) * a.N, chan_bytes,
                      &mbar[it & 1u]);
        }
    }
}

// Persistent loop with several frames per CTA, one per warp: the CTA's
// F = blockDim.x / 32 warps decode F frames side by side, each with its own
// shared-memory region and scratch, running the same straight-line decoder
// (every group operation of the body is warp-level). Barriers in the body keep
// the warps in step, so that they share the instructions they fetch. In the
// last group, warps without a frame decode frame 0 again and store nothing, so
// that every warp passes the same barriers.
template <typename T, class Body>
__device__ __forceinline__ void run_warp_frames(const KernelArgs &a, const Body &body) {
    extern __shared__ __align__(128) unsigned char smem[];
    const SmemLayout L(a.N, a.S, sizeof(T), false);
    const size_t per_frame = align_up(L.total, 128);
    const uint32_t lane = threadIdx.x & 31u, w = threadIdx.x >> 5, F = blockDim.x >> 5;
    unsigned char *base = smem + size_t(w) * per_frame;
    Frame<T> fr;
    fr.s_alpha = reinterpret_cast<T *>(base + L.alpha);
    fr.beta = reinterpret_cast<uint32_t *>(base + L.beta);
    fr.rkey = reinterpret_cast<unsigned long long *>(base + L.rkey);
    fr.rpar = reinterpret_cast<uint32_t *>(base + L.rpar);
    fr.g_alpha = a.gscratch
                     ? static_cast<T *>(a.gscratch) + (size_t(blockIdx.x) * F + w) * a.gstride
                     : nullptr;
    fr.N = a.N;
    fr.S = a.S;
    const T *llr = static_cast<const T *>(a.llr);
    const size_t groups = (a.n_frames + F - 1) / F;
    for (size_t g = blockIdx.x; g < groups; g += gridDim.x) {
        const size_t f = g * F + w;
        const bool valid = f < a.n_frames;
        fr.chan = llr + (valid ? f : 0) * a.N;
        body(fr, nullptr);
        if (valid) pack_bits<WarpGrp>(fr.beta, a, a.out + f * a.out_row);
        __syncthreads();
    }
}

// ---------------------------------------------------------------- out-of-line forms

// The memory-resident operations as real calls with run-time sizes: the compact
// form of a generated decoder uses them so that code size grows with the number
// of distinct subtrees, not with the length of the operation list.
template <typename T, class Grp, uint32_t KIND, uint32_t RD = RD_NORMAL, uint32_t WR = 0u>
__device__ __noinline__ void mem_fg(const T *in, T *out, uint32_t h, const uint32_t *beta,
                                    uint32_t o) {
    op_fg<T, Grp, KIND, RD, WR>(in, out, h, beta, o);
}
template <typename T, class Grp, uint32_t L, uint32_t K0, uint32_t K1, uint32_t K2,
          uint32_t STORE = 3u, uint32_t RD = RD_NORMAL, uint32_t WR = 0u>
__device__ __noinline__ void mem_chain(const T *in, T *stage1, T *stage2, T *stage3, uint32_t n,
                                       const uint32_t *beta, uint32_t o) {
    op_chain<T, Grp, L, K0, K1, K2, STORE, RD, WR>(in, stage1, stage2, stage3, n, beta, o);
}
template <class Grp>
__device__ __noinline__ void mem_combine(uint32_t *beta, uint32_t n, uint32_t o, bool copy) {
    op_combine<Grp>(beta, n, o, copy);
}
template <class Grp>
__device__ __noinline__ void mem_r0(uint32_t *beta, uint32_t n, uint32_t o) {
    op_r0<Grp>(beta, n, o);
}
template <typename T, class Grp>
__device__ __noinline__ void mem_r1(const T *in, uint32_t *beta, uint32_t n, uint32_t o) {
    op_r1<T, Grp>(in, beta, n, o);
}
template <typename T, class Grp>
__device__ __noinline__ void mem_rep(const T *in, T *tmp, uint32_t *beta, uint32_t n, uint32_t o) {
    op_rep<T, Grp>(in, tmp, beta, n, o);
}
template <typename T, class Grp>
__device__ __noinline__ void mem_spc(const T *in, uint32_t *beta, uint32_t n, uint32_t o,
                                     unsigned long long *rkey, uint32_t *rpar) {
    op_spc<T, Grp, false>(in, beta, n, o, rkey, rpar);
}

// ---------------------------------------------------------------- mixed batches

// Persistent loop of the mixed-batch kernel: each CTA claims the next frame,
// points its Frame at the frame's code (shared base pointers, per-code N and
// S), runs `body(code_id, fr)` and packs the frame's information bits.
template <typename T, class Body>
__device__ __forceinline__ void run_batch(const BatchArgs &a, const Body &body) {
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ unsigned int s_item;
    const uint32_t tid = threadIdx.x;
    const size_t alpha_bytes = align_up(size_t(a.smem_alpha_elems) * sizeof(T), 128);
    const size_t beta_bytes = align_up(size_t(a.smem_beta_words) * 4, 16);
    Frame<T> fr;
    fr.s_alpha = reinterpret_cast<T *>(smem);
    fr.beta = reinterpret_cast<uint32_t *>(smem + alpha_bytes);
    fr.rkey = reinterpret_cast<unsigned long long *>(smem + alpha_bytes + beta_bytes);
    fr.rpar = reinterpret_cast<uint32_t *>(smem + alpha_bytes + beta_bytes + 32 * 8);
    fr.g_alpha = a.gscratch ? static_cast<T *>(a.gscratch) + size_t(blockIdx.x) * a.gstride : nullptr;
    const T *llr = static_cast<const T *>(a.llr);
    for (;;) {
        if (tid == 0) s_item = atomicAdd(a.counter, 1u);
        __syncthreads();
        const size_t item = s_item;
        __syncthreads();  // every thread has read s_item before it is overwritten
        if (item >= a.n_frames) break;
        const uint32_t cid = __ldg(a.code_id + item);
        const CodeDesc d = a.codes[cid];
        fr.N = d.N;
        fr.S = d.S;
        fr.chan = llr + __ldg(a.llr_off + item);
        body(cid, fr);
        pack_bits<CtaGrp>(fr.beta, d, a.out + __ldg(a.out_off + item));
        __syncthreads();
    }
}

// Persistent loop of the mixed-batch kernel with several frames per CTA, one
// per warp: the CTA claims F = blockDim.x / 32 consecutive frames of the list
// (listed longest code first, so they are almost always frames of one code)
// and its warps run that code's body side by side, each on its own frame,
// shared-memory slot and scratch slot, meeting at the CTA barriers the
// warp-level bodies place after each register subtree. When the F frames
// belong to several codes, the CTA runs the body of each of those codes in
// turn; in a turn, a warp whose frame is of another code decodes a copy of the
// turn's first frame of that code and stores nothing, so that every warp passes
// the same barriers. The same holds for the warps past the end of the list.
template <typename T, class Body>
__device__ __forceinline__ void run_batch_warps(const BatchArgs &a, const Body &body) {
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ unsigned int s_base;
    __shared__ uint32_t s_cid[32];
    const uint32_t lane = threadIdx.x & 31u, w = threadIdx.x >> 5, F = blockDim.x >> 5;
    const size_t slot = batch_slot_bytes(a.smem_alpha_elems, a.smem_beta_words, sizeof(T));
    unsigned char *base = smem + size_t(w) * slot;
    const size_t alpha_bytes = align_up(size_t(a.smem_alpha_elems) * sizeof(T), 128);
    const size_t beta_bytes = align_up(size_t(a.smem_beta_words) * 4, 16);
    Frame<T> fr;
    fr.s_alpha = reinterpret_cast<T *>(base);
    fr.beta = reinterpret_cast<uint32_t *>(base + alpha_bytes);
    fr.rkey = reinterpret_cast<unsigned long long *>(base + alpha_bytes + beta_bytes);
    fr.rpar = reinterpret_cast<uint32_t *>(base + alpha_bytes + beta_bytes + 32 * 8);
    fr.g_alpha = a.gscratch ? static_cast<T *>(a.gscratch) + (size_t(blockIdx.x) * F + w) * a.gstride
                            : nullptr;
    const T *llr = static_cast<const T *>(a.llr);
    for (;;) {
        if (threadIdx.x == 0) s_base = atomicAdd(a.counter, F);
        __syncthreads();
        const size_t first = s_base;
        if (first >= a.n_frames) break;
        const size_t item = first + w;
        if (lane == 0) s_cid[w] = __ldg(a.code_id + (item < a.n_frames ? item : first));
        __syncthreads();
        const uint32_t mine = s_cid[w];
        for (uint32_t k = 0; k < F; ++k) {
            const uint32_t cid = s_cid[k];
            bool seen = false;
            for (uint32_t j = 0; j < k; ++j) seen |= s_cid[j] == cid;
            if (seen) continue;  // this code's turn has been run
            const bool own = mine == cid && item < a.n_frames;
            const size_t src = own ? item : first + k;
            const CodeDesc d = a.codes[cid];
            fr.N = d.N;
            fr.S = d.S;
            fr.chan = llr + __ldg(a.llr_off + src);
            body(cid, fr);
            if (own) pack_bits<WarpGrp>(fr.beta, d, a.out + __ldg(a.out_off + item));
            __syncthreads();
        }
    }
}

// ---------------------------------------------------------------- specialised subtrees

// Compile-time loop: f(UC<I>{}) for I in [B, E). Indices reach the body as
// template constants, so arrays indexed by them stay in registers.
template <uint32_t V> struct UC {
    static constexpr uint32_t value = V;
};
template <uint32_t B, uint32_t E, class F>
__device__ __forceinline__ void static_for(F &&f) {
    if constexpr (B < E) {
        f(UC<B>{});
        static_for<B + 1, E>(f);
    }
}

// Register-subtree values. A 32-bit register holds W values of one lane: one
// float (W = 1), or for int8 LLRs two f16 (W = 2; integers of magnitude <= 254
// are exact in f16, see op_i8x4). int8 keeps its saturation: every sum is
// clamped to [-127, 127], which is what the saturating byte add followed by
// max(-127) gives. Bits are sign bits (SGN): beta = 1 is a set sign, so G flips
// signs with one XOR and a hard decision is the sign of x + 0, which is set
// exactly when x < 0 (-0 + 0 = +0, and a NaN sum is the positive NaN).
template <typename T> struct SubVal;
template <> struct SubVal<float> {
    static constexpr uint32_t W = 1, SGN = 0x80000000u;
    __device__ static __forceinline__ uint32_t f(uint32_t a, uint32_t b) {
        return __float_as_uint(f_f32(__uint_as_float(a), __uint_as_float(b)));
    }
    __device__ static __forceinline__ uint32_t add(uint32_t a, uint32_t b) {
        return __float_as_uint(__uint_as_float(a) + __uint_as_float(b));
    }
    __device__ static __forceinline__ uint32_t add_sign(uint32_t a, uint32_t b) { return hard(add(a, b)); }
    __device__ static __forceinline__ uint32_t hard(uint32_t a) {
        return __float_as_uint(__uint_as_float(a) + 0.0f);
    }
};
template <> struct SubVal<int8_t> {
    static constexpr uint32_t W = 2, SGN = 0x80008000u;
    __device__ static __forceinline__ uint32_t f(uint32_t a, uint32_t b) { return hf2(a, b); }
    __device__ static __forceinline__ uint32_t add(uint32_t a, uint32_t b) { return hsat2(hadd2(a, b)); }
    // a sum of which only the hard decision is used: the clamp keeps the sign
    __device__ static __forceinline__ uint32_t add_sign(uint32_t a, uint32_t b) { return hard(hadd2(a, b)); }
    __device__ static __forceinline__ uint32_t hard(uint32_t a) { return hadd2(a, 0u); }
};

__host__ __device__ constexpr uint32_t clog2(uint32_t v) { return v <= 1 ? 0u : 1u + clog2(v / 2); }

// Subtree of at most R leaves decoded by one warp in registers with compile-time
// node sizes and offsets (the generated decoders).
//
// Layout. A row is one register per lane: E = 32 W values of a node. Value e of
// a stage of n >= E values sits in row e / E, half (e / 32) % W, lane e % 32, so F
// and G of nodes of 2E and more values are lane-local. At n = E with W = 2 the
// two operands are the halves of one register. A stage of n <= 32 values is
// kept replicated: every lane li (and both halves) holds value li % n. Then the
// partner operand of F and G is one shuffle away (lane li ^ n/2), is kept from F
// for the G of the same node, no lane idles and none needs a predicate, every
// lane ends a Repetition fold with the sum, Combine is one logic instruction
// and a Rate-1 node one addition. (Before: stage n on lanes n..2n-1 and bits in
// a word common to the warp, with two shuffles and a select for F and for G, and
// a ballot and a bit-field insert for every node.) The narrow nodes (n <= 32)
// are nine tenths of a frame's operations and set both the length of a frame's
// serial chain and, through their instructions, the rate of a full GPU.
// Measured before and after this layout (int8 unless named): one frame of
// (32768, 29492) 77.9 -> 67.8 us, 4096 of them 352 -> 327 us (float32 883 -> 829),
// 2,001 frames of (2048, 1707) 24.6 -> 20.5 us.
// LEAN (the interpreter): the masks of operand b are formed when used, five
// registers fewer for one more logic instruction in a narrow G.
template <typename T, uint32_t R, bool LEAN = false>
struct RegSub {
    using V = SubVal<T>;
    static constexpr uint32_t G = 32, W = V::W, SGN = V::SGN, E = G * W;
    static constexpr uint32_t NR = R >= E ? R / E : 1;
    uint32_t v32[32], v16[16], v8[8], v4[4], v2[2], v1;  // stages of n >= E values: n / E rows
    uint32_t t[7], y[7];       // stage 2^k < E (replicated); partner operand of node 2^k <= E
    uint32_t B[NR];            // bits of nodes of n >= E values, by row
    uint32_t bl[7], br[7];     // bits of left / right nodes of 2^k < E values (replicated)
    uint32_t ca[5], cb[5];     // sign mask on lanes with bit k of the lane index clear / set
    uint32_t li;               // lane

    __device__ __forceinline__ void init() {
        li = threadIdx.x & 31u;
        static_for<0, 5>([&](auto kc) {
            constexpr uint32_t k = decltype(kc)::value;
            ca[k] = (li >> k) & 1u ? 0u : SGN;
            cb[k] = SGN ^ ca[k];
        });
    }

    template <uint32_t n, uint32_t k>
    __device__ __forceinline__ uint32_t &row() {
        if constexpr (n < E) return t[clog2(n)];
        else if constexpr (n / E == 32) return v32[k];
        else if constexpr (n / E == 16) return v16[k];
        else if constexpr (n / E == 8) return v8[k];
        else if constexpr (n / E == 4) return v4[k];
        else if constexpr (n / E == 2) return v2[k];
        else return v1;
    }
    // Bits of node (n, p), n < E (or its row when n = E).
    template <uint32_t n, uint32_t p>
    __device__ __forceinline__ uint32_t &bits() {
        if constexpr (n >= E) return B[p / E];
        else if constexpr ((p & n) != 0) return br[clog2(n)];
        else return bl[clog2(n)];
    }
    // The other operand's lanes for a node of n <= E values.
    template <uint32_t n>
    __device__ __forceinline__ uint32_t partner(uint32_t x) {
        if constexpr (W == 2 && n == E) return prmt(x, x, 0x1032u);
        else return __shfl_xor_sync(kFull, x, n / 2);
    }
    // Sign mask of the values that are operand a (index < n/2) / b of a node of n <= E.
    template <uint32_t n>
    __device__ __forceinline__ uint32_t mask_a() {
        if constexpr (W == 2 && n == E) return 0x00008000u;
        else return ca[clog2(n) - 1];
    }
    template <uint32_t n>
    __device__ __forceinline__ uint32_t mask_b() {
        if constexpr (W == 2 && n == E) return 0x80000000u;
        else if constexpr (LEAN) return SGN ^ ca[clog2(n) - 1];
        else return cb[clog2(n) - 1];
    }
    // Whether the signs of the n <= 32 values x (replicated) have odd parity, as
    // sign masks (SGN or 0 in every lane): one copy of the values is XORed over the
    // warp. (A ballot and a population count before: 20 cycles more in the chain.)
    template <uint32_t n>
    __device__ __forceinline__ uint32_t odd_signs(uint32_t x) {
        uint32_t keep = SGN;
        static_for<clog2(n), 5>([&](auto kc) { keep &= ca[decltype(kc)::value]; });
        return __reduce_xor_sync(kFull, x & keep);
    }

    // Load the subtree root's LLRs (stage n0).
    template <uint32_t n0>
    __device__ __forceinline__ void enter(const T *src) {
        init();
        if constexpr (n0 >= E) {
            static_for<0, n0 / E>([&](auto kc) {
                constexpr uint32_t k = decltype(kc)::value;
                if constexpr (W == 1) row<n0, k>() = __float_as_uint(src[E * k + li]);
                else row<n0, k>() = pair(src[E * k + li], src[E * k + G + li]);
            });
        } else {
            const T x = src[li & (n0 - 1u)];
            if constexpr (W == 1) t[clog2(n0)] = __float_as_uint(x);
            else t[clog2(n0)] = pair(x, x);
        }
    }
    // Two int8 values as f16x2: 0x6480 + x is the f16 1152 + x (x in [-127, 127]
    // keeps the exponent), and the sum of the two halves never carries.
    __device__ static __forceinline__ uint32_t pair(int32_t lo, int32_t hi) {
        return hadd2(0x64806480u + static_cast<uint32_t>(lo) + (static_cast<uint32_t>(hi) << 16),
                     0xE480E480u);
    }

    // Store the subtree's n0 bits at leaf offset o0 of beta. The words are the same
    // on every lane, so lane 0 stores them, 16 bytes at a time (o0 is a multiple of
    // n0, so the words are 16-byte aligned from 128 leaves up).
    template <uint32_t n0>
    __device__ __forceinline__ void exit(uint32_t *beta, uint32_t o0) {
        if constexpr (n0 < E) {
            const uint32_t m = __ballot_sync(kFull, static_cast<int32_t>(bl[clog2(n0)]) < 0);
            if (li == 0) write_field(beta, o0, n0, m);
        } else {
            uint32_t w[n0 / 32];
            static_for<0, n0 / 32>([&](auto kc) {
                constexpr uint32_t k = decltype(kc)::value;
                constexpr uint32_t m = (W == 2 && k % 2 == 0) ? 0x8000u : 0x80000000u;
                w[k] = __ballot_sync(kFull, (B[k / W] & m) != 0u);
            });
            if (li == 0) {
                static_for<0, n0 / 32>([&](auto kc) {
                    constexpr uint32_t k = decltype(kc)::value;
                    if constexpr (n0 >= 128) {
                        if constexpr (k % 4 == 0)
                            *reinterpret_cast<uint4 *>(beta + (o0 >> 5) + k) =
                                make_uint4(w[k], w[k + 1], w[k + 2], w[k + 3]);
                    } else {
                        beta[(o0 >> 5) + k] = w[k];
                    }
                });
            }
        }
    }

    // F / G / G_0R of a node of n leaves at subtree offset p.
    template <uint32_t KIND, uint32_t n, uint32_t p>
    __device__ __forceinline__ void fg() {
        if constexpr (n >= 2 * E) {
            constexpr uint32_t K = n / (2 * E);
            static_for<0, K>([&](auto kc) {
                constexpr uint32_t k = decltype(kc)::value;
                const uint32_t a = row<n, k>(), b = row<n, k + K>();
                uint32_t r;
                if constexpr (KIND == OP_F) r = V::f(a, b);
                else if constexpr (KIND == OP_G) r = V::add(b, a ^ (B[p / E + k] & SGN));
                else r = V::add(b, a);
                row<n / 2, k>() = r;
            });
        } else {
            const uint32_t x = row<n, 0>();
            if constexpr (KIND == OP_G) {
                const uint32_t w = bits<n / 2, p>(), z = y[clog2(n)];
                row<n / 2, 0>() = V::add(x ^ (w & mask_a<n>()), z ^ (w & mask_b<n>()));
            } else {
                const uint32_t z = partner<n>(x);
                y[clog2(n)] = z;
                row<n / 2, 0>() = KIND == OP_F ? V::f(x, z) : V::add(x, z);
            }
        }
    }

    // G of a node of n leaves at p and the Rate-1 decision of its right child in one.
    template <uint32_t n, uint32_t p>
    __device__ __forceinline__ void g_r1() {
        constexpr uint32_t h = n / 2;
        if constexpr (n >= 2 * E) {
            constexpr uint32_t K = n / (2 * E);
            static_for<0, K>([&](auto kc) {
                constexpr uint32_t k = decltype(kc)::value;
                B[(p + h) / E + k] = V::add_sign(row<n, k + K>(), row<n, k>() ^ (B[p / E + k] & SGN));
            });
        } else {
            const uint32_t w = bits<h, p>();
            bits<h, p + h>() = V::add_sign(row<n, 0>() ^ (w & mask_a<n>()),
                                           y[clog2(n)] ^ (w & mask_b<n>()));
        }
    }

    // Combine (copy = false) / Combine_0R (copy = true) of a node of n leaves at p.
    template <uint32_t n, uint32_t p, bool copy>
    __device__ __forceinline__ void combine() {
        constexpr uint32_t h = n / 2;
        if constexpr (n >= 2 * E) {
            static_for<0, h / E>([&](auto kc) {
                constexpr uint32_t k = decltype(kc)::value;
                const uint32_t r = B[(p + h) / E + k];
                B[p / E + k] = copy ? r : (B[p / E + k] ^ r);
            });
        } else {
            const uint32_t r = bits<h, p + h>();
            bits<n, p>() = copy ? r : (r ^ (bits<h, p>() & mask_a<n>()));
        }
    }

    // Rate-0 subtree root of n leaves.
    template <uint32_t n, uint32_t p>
    __device__ __forceinline__ void r0() {
        if constexpr (n >= E) {
            static_for<0, n / E>([&](auto kc) { B[p / E + decltype(kc)::value] = 0u; });
        } else {
            bits<n, p>() = 0u;
        }
    }
    // Rate-0 right child (n leaves at p) of a split node, which has no Combine:
    // the parent's left bits stay, its right bits are zero.
    template <uint32_t n, uint32_t p>
    __device__ __forceinline__ void r0_right() {
        if constexpr (n >= E) r0<n, p>();
        else bits<2 * n, p - n>() = bits<n, p - n>() & mask_a<2 * n>();
    }

    template <uint32_t n, uint32_t p>
    __device__ __forceinline__ void r1() {
        if constexpr (n >= E) {
            static_for<0, n / E>([&](auto kc) {
                constexpr uint32_t k = decltype(kc)::value;
                B[p / E + k] = V::hard(row<n, k>());
            });
        } else {
            bits<n, p>() = V::hard(t[clog2(n)]);
        }
    }

    // Folds a[k] <- a[k] + a[k + m] for m = K/2, ..., 1 over K rows.
    template <uint32_t K>
    __device__ __forceinline__ void fold_rows(uint32_t (&a)[K]) {
        if constexpr (K > 1) {
            static_for<0, K / 2>([&](auto kc) {
                constexpr uint32_t k = decltype(kc)::value;
                a[k] = V::add(a[k], a[k + K / 2]);
            });
            fold_rows<K / 2>(reinterpret_cast<uint32_t(&)[K / 2]>(a));
        }
    }
    // Repetition sum of a node of n <= E values x: t[i] + t[i + m] for m = n/2 .. 1,
    // on every lane (a + b = b + a, so partners agree); the sign of its sum + 0.
    template <uint32_t n>
    __device__ __forceinline__ uint32_t rep_small(uint32_t x) {
        static_for<0, clog2(n)>([&](auto kc) {
            constexpr uint32_t m = n >> decltype(kc)::value;
            x = V::add(x, partner<m>(x));
        });
        return V::hard(x);
    }
    template <uint32_t n, uint32_t p>
    __device__ __forceinline__ void rep() {
        if constexpr (n >= E) {
            constexpr uint32_t K = n / E;
            uint32_t a[K];
            static_for<0, K>([&](auto kc) {
                constexpr uint32_t k = decltype(kc)::value;
                a[k] = row<n, k>();
            });
            fold_rows<K>(a);
            const uint32_t w = rep_small<E>(a[0]);
            static_for<0, K>([&](auto kc) { B[p / E + decltype(kc)::value] = w; });
        } else {
            bits<n, p>() = rep_small<n>(t[clog2(n)]);
        }
    }

    // SPC bits of a replicated node of n <= 32 values x: the sign of the value of
    // least magnitude, the lowest index of equals (Listing 2), flips on odd parity.
    // float32: the least magnitude over the warp, then its lowest lane; the shift
    // brings that lane's ballot bit to its sign. int8: magnitude and index fit one key.
    template <uint32_t n>
    __device__ __forceinline__ uint32_t spc_small(uint32_t x) {
        const uint32_t d = V::hard(x), e = li & (n - 1u), odd = odd_signs<n>(d);
        if constexpr (W == 1) {
            const uint32_t mag = x & 0x7fffffffu, mn = __reduce_min_sync(kFull, mag);
            const uint32_t at = __ballot_sync(kFull, mag == mn);
            return d ^ (((at & (0u - at)) << (31u - e)) & odd);
        } else {
            const uint32_t key = (x & 0x7fff0000u) | e;
            return d ^ (key == __reduce_min_sync(kFull, key) ? odd : 0u);
        }
    }
    template <uint32_t n, uint32_t p>
    __device__ __forceinline__ void spc() {
        if constexpr (n <= 32) {
            bits<n, p>() = spc_small<n>(row<n, 0>());
        } else {
            constexpr uint32_t K = n / E;
            uint32_t par = 0;
            static_for<0, K>([&](auto kc) {
                constexpr uint32_t k = decltype(kc)::value;
                const uint32_t d = V::hard(row<n, k>());
                B[p / E + k] = d;
                par ^= d;
            });
            if constexpr (W == 2) par ^= par << 16;
            const bool odd = static_cast<int32_t>(__reduce_xor_sync(kFull, par)) < 0;
            if constexpr (W == 1) {
                uint32_t mk = kFull;
                static_for<0, K>([&](auto kc) {
                    mk = min(mk, row<n, decltype(kc)::value>() & 0x7fffffffu);
                });
                const uint32_t mn = __reduce_min_sync(kFull, mk);
                uint32_t e = kFull;  // lowest index of this lane with that magnitude
                static_for<0, K>([&](auto kc) {
                    constexpr uint32_t k = K - 1 - decltype(kc)::value;
                    if ((row<n, k>() & 0x7fffffffu) == mn) e = E * k + li;
                });
                e = __reduce_min_sync(kFull, e);
                const uint32_t at = odd ? e - li : kFull;  // E k on the lane that flips row k
                static_for<0, K>([&](auto kc) {
                    constexpr uint32_t k = decltype(kc)::value;
                    if (at == E * k) B[p / E + k] ^= SGN;
                });
            } else {
                uint32_t key = kFull;  // f16 magnitude, then 32-value chunk, then lane
                static_for<0, K>([&](auto kc) {
                    constexpr uint32_t k = decltype(kc)::value;
                    const uint32_t x = row<n, k>();
                    key = min(key, ((x << 16) & 0x7fff0000u) | (64u * k));
                    key = min(key, (x & 0x7fff0000u) | (64u * k + 32u));
                });
                key |= li;
                const uint32_t mn = __reduce_min_sync(kFull, key);
                const uint32_t c = (key == mn && odd) ? (mn & 0xffffu) >> 5 : kFull;  // chunk to flip
                static_for<0, K>([&](auto kc) {
                    constexpr uint32_t k = decltype(kc)::value;
                    if (c == 2 * k) B[p / E + k] ^= 0x00008000u;
                    if (c == 2 * k + 1) B[p / E + k] ^= 0x80000000u;
                });
            }
        }
    }
};

// Pointer to stage n of a generated decoder with compile-time N and S.
template <typename T, uint32_t N, uint32_t S, uint32_t n>
__device__ __forceinline__ const T *gen_in(const Frame<T> &fr) {
    if constexpr (n == N) return fr.chan;
    else if constexpr (n <= S) return fr.s_alpha + n;
    else return fr.g_alpha + (n - 2 * S);
}
template <typename T, uint32_t S, uint32_t n>
__device__ __forceinline__ T *gen_out(const Frame<T> &fr) {
    if constexpr (n <= S) return fr.s_alpha + n;
    else return fr.g_alpha + (n - 2 * S);
}

#endif  // __CUDACC__

}  // namespace polar
