// Fast-SSC decoding kernels for sm_103a (GB300).
//
// Method: Giard et al., "Low-Latency Software Polar Decoders" (arXiv 1504.00353),
// Sec. II-C/II-D. One CTA decodes one frame at a time and loops over frames
// (persistent grid sized to the resident-CTA count). The frame's operation list
// (the depth-first Fast-SSC call list of Listing 1, built on the host) is
// interpreted in order, at three granularities:
//   - wide operations (node size N_v > warp_stage_max) use every thread of the
//     CTA, loads issued ahead of use, one __syncthreads after each;
//   - narrower operations run on warp 0 alone with __syncwarp between them while
//     the other warps jump past the run (the host stores the run's end);
//   - subtrees of at most 64 leaves run entirely in registers of warp 0, in the
//     layout of the specialised decoders (RegSub in polar_ops.cuh), each
//     operation reached by one jump on its kind, size and side.
// Memory layout (Sec. III-B): the alpha stage for node size n occupies elements
// [n, 2n) of a per-CTA array, in shared memory for n <= smem_stage_max and in
// per-CTA device scratch above that; beta is one N-bit array in shared memory
// (node (off, n) owns bits [off, off+n), Combine rewrites only the left half).
// The channel LLRs are read in place from device memory with 16-byte vector
// loads, or (stage_channel) copied to shared memory with cp.async.bulk under an
// mbarrier, double buffered so the next frame's copy overlaps this frame.
// float32: F is an exact min with the XOR of the sign bits (beta in {+0,-0},
// Sec. III-B), G adds alpha_v[i] with its sign flipped by beta_l (Listing 3),
// one IEEE add. int8: G is a saturating add then max(-127) (Listing 4).
// Both agree bit for bit with a scalar evaluation in the same order.
#include <cuda_runtime.h>

#include <cstdint>
#include <mutex>
#include <set>
#include <utility>

#include "polar_internal.h"

namespace polar {
namespace {

template <typename T, class Grp>
__device__ __forceinline__ void trace_store(uint32_t kind, uint32_t n, uint32_t trace_off,
                                            const Frame<T> &fr, float *trace_row) {
    if (kind > OP_G0R) return;
    const uint32_t h = n >> 1;
    const T *src = fr.stage(h);
    for (uint32_t i = Grp::rank(); i < h; i += Grp::size())
        trace_row[trace_off + i] = static_cast<float>(src[i]);
}

// ---------------------------------------------------------------- register subtrees

// A subtree of at most kRegSubtree leaves decoded by warp 0 in registers: the
// layout and the operations of the specialised decoders (RegSub), reached from
// the list through one jump on an operation's kind, size and side (whether its
// node is the right child of its parent), so that an operation is its handful of
// instructions behind the jump. (Before: shuffles, selects and bit fields with
// run-time sizes, some 120 instructions for each operation of the list, waiting on
// one another.) The kernel has 64 registers, so that a CTA of 1024 threads fits, and
// the registers of a subtree nearly fill them: enter clears every one, which ends
// their lives between subtrees. Left as they were, they stayed allocated across the
// memory-level operations and those spilled: 408 (float32) and 660 (int8) bytes, now
// none. 1,000 frames of (1024, 512), float32 92 us before this layout, 82 with the
// spills, 72 now; int8 96, 82, 70; 4,000 of (32768, 29491) int8 2,935, 2,997, 2,574.
template <typename T, bool TRACE>
struct RegTree {
    using Sub = RegSub<T, kRegSubtree, true>;
    Sub r;
    uint32_t log2n0, o0;

    // f(UC<log2 n>{}) for the run-time log2 n <= log2 kRegSubtree.
    template <uint32_t L = 0, class F>
    __device__ __forceinline__ static void with_size(uint32_t l, F &&f) {
        if constexpr ((1u << L) <= kRegSubtree) {
            if (l == L) f(UC<L>{});
            else with_size<L + 1>(l, f);
        }
    }
    __device__ __forceinline__ void enter(const T *src, uint32_t l, uint32_t o) {
        log2n0 = l;
        o0 = o;
        r = Sub();
        with_size(l, [&](auto lc) { r.template enter<(1u << decltype(lc)::value)>(src); });
    }
    __device__ __forceinline__ void exit(uint32_t *beta) {
        with_size(log2n0, [&](auto lc) { r.template exit<(1u << decltype(lc)::value)>(beta, o0); });
    }

    template <uint32_t KIND, uint32_t n>
    __device__ __forceinline__ void fg(float *row) {
        r.template fg<KIND, n, 0>();
        if constexpr (TRACE) {  // the n/2 outputs: value i on lane i
            const uint32_t lane = threadIdx.x & 31u, v = r.template row<n / 2, 0>();
            if (lane < n / 2) {
                if constexpr (sizeof(T) == 1) {
                    float x;
                    asm("{\n .reg .b16 l, h;\n mov.b32 {l, h}, %1;\n cvt.f32.f16 %0, l;\n}\n" : "=f"(x) : "r"(v));
                    row[lane] = x;
                } else {
                    row[lane] = __uint_as_float(v);
                }
            }
        }
    }

    // Execute the operation of word w; row: where its F/G/G_0R outputs are traced.
    __device__ __forceinline__ void exec(uint32_t w, float *row) {
        // a node's bits go to its parent's left or right side; the subtree's root
        // counts as a left child, and the last operation completes the root
        const bool inner = !(w & OPW_REG_EXIT);
        const uint32_t side = inner ? (w >> 12) & 1u : 0u, up = inner ? (w >> 13) & 1u : 0u;
        // dense keys, so that the switch is a jump table
        const uint32_t key = (op_log2n(w) * 9u + op_kind(w)) * 2u + (op_kind(w) == OP_R0 ? up : side);
#define POLAR_KEY(kind, l, s) (((l) * 9u + (kind)) * 2u + (s))
#define POLAR_FG(l)                                                            \
    case POLAR_KEY(OP_F, l, 0): case POLAR_KEY(OP_F, l, 1): fg<OP_F, (1u << l)>(row); break;       \
    case POLAR_KEY(OP_G, l, 0): case POLAR_KEY(OP_G, l, 1): fg<OP_G, (1u << l)>(row); break;       \
    case POLAR_KEY(OP_G0R, l, 0): case POLAR_KEY(OP_G0R, l, 1): fg<OP_G0R, (1u << l)>(row); break;
#define POLAR_NODE(l, s)                                                       \
    case POLAR_KEY(OP_R1, l, s): r.template r1<(1u << l), (s << l)>(); break;      \
    case POLAR_KEY(OP_REP, l, s): r.template rep<(1u << l), (s << l)>(); break;    \
    case POLAR_KEY(OP_SPC, l, s): r.template spc<(1u << l), (s << l)>(); break;
#define POLAR_COMBINE(l, s)                                                    \
    case POLAR_KEY(OP_C, l, s): r.template combine<(1u << l), (s << l), false>(); break;           \
    case POLAR_KEY(OP_C0R, l, s): r.template combine<(1u << l), (s << l), true>(); break;
// a Rate-0 right child of n = 2^l leaves whose parent is on side s
#define POLAR_R0(l, s) \
    case POLAR_KEY(OP_R0, l, s): r.template r0_right<(1u << l), ((s << (l + 1)) + (1u << l))>(); break;
        switch (key) {
            POLAR_FG(1) POLAR_FG(2) POLAR_FG(3) POLAR_FG(4) POLAR_FG(5) POLAR_FG(6)
            POLAR_NODE(0, 0) POLAR_NODE(1, 0) POLAR_NODE(2, 0) POLAR_NODE(3, 0) POLAR_NODE(4, 0)
            POLAR_NODE(5, 0) POLAR_NODE(6, 0) POLAR_NODE(0, 1) POLAR_NODE(1, 1) POLAR_NODE(2, 1)
            POLAR_NODE(3, 1) POLAR_NODE(4, 1) POLAR_NODE(5, 1)
            POLAR_COMBINE(1, 0) POLAR_COMBINE(2, 0) POLAR_COMBINE(3, 0) POLAR_COMBINE(4, 0)
            POLAR_COMBINE(5, 0) POLAR_COMBINE(6, 0) POLAR_COMBINE(1, 1) POLAR_COMBINE(2, 1)
            POLAR_COMBINE(3, 1) POLAR_COMBINE(4, 1) POLAR_COMBINE(5, 1)
            POLAR_R0(0, 0) POLAR_R0(1, 0) POLAR_R0(2, 0) POLAR_R0(3, 0) POLAR_R0(4, 0) POLAR_R0(5, 0)
            POLAR_R0(0, 1) POLAR_R0(1, 1) POLAR_R0(2, 1) POLAR_R0(3, 1) POLAR_R0(4, 1)
        default: break;
        }
#undef POLAR_KEY
#undef POLAR_FG
#undef POLAR_NODE
#undef POLAR_COMBINE
#undef POLAR_R0
    }

    // A subtree that is one Rate-0 node.
    __device__ __forceinline__ void r0_root() {
        with_size(log2n0, [&](auto lc) { r.template r0<(1u << decltype(lc)::value), 0>(); });
    }
};

// The operation list as one warp sees it: a 32-op window in registers (op
// base + l on lane l) and the following window already requested, so an op is
// one shuffle away and device-memory latency is hidden 32 ops ahead. Indices
// passed to get() never decrease.
struct OpWindow {
    const uint32_t *ops;
    uint32_t n, base, cur, nxt, lane;

    __device__ __forceinline__ uint32_t fetch(uint32_t i) const {
        return i < n ? __ldg(ops + i) : 0u;
    }
    __device__ __forceinline__ void start(const uint32_t *p, uint32_t count, uint32_t l) {
        ops = p;
        n = count;
        lane = l;
        base = 0;
        cur = fetch(l);
        nxt = fetch(32 + l);
    }
    __device__ __forceinline__ void advance() {
        base += 32;
        cur = nxt;
        nxt = fetch(base + 32 + lane);
    }
    __device__ __forceinline__ uint32_t get(uint32_t j) {
        while (j - base >= 32) advance();
        return __shfl_sync(kFull, cur, j - base);
    }
    // First index >= i whose node is wider than 2^log2W (n if none).
    __device__ __forceinline__ uint32_t skip_narrow(uint32_t i, uint32_t log2W) {
        for (;;) {
            while (i - base >= 32) advance();
            const bool stop = lane >= i - base && base + lane < n && op_log2n(cur) > log2W;
            const uint32_t b = __ballot_sync(kFull, stop);
            if (b) return base + __ffs(b) - 1;
            if (base + 32 >= n) return n;
            i = base + 32;
        }
    }
};

// ---------------------------------------------------------------- interpreter body

// Runs the operation list of one frame: narrow runs on warp 0 (register
// subtrees or memory ops), wide ops on the whole CTA.
template <typename T, bool TRACE>
struct InterpBody {
    const KernelArgs &a;
    __device__ __forceinline__ void operator()(const Frame<T> &fr, float *trace_row) const {
        const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
        OpWindow win;
        win.start(a.ops, a.n_ops, lane);
        uint32_t i = 0;
        while (i < a.n_ops) {
            uint32_t w = win.get(i);
            if (op_log2n(w) <= a.log2W) {
                // a run of narrow ops: warp 0 executes it, the other warps skip it
                if (warp == 0) {
                    uint32_t j = i;
                    for (;;) {
                        const uint32_t kind = op_kind(w), n = 1u << op_log2n(w), o = op_off(w);
                        if (w & OPW_REG_ENTER) {  // a register subtree, to its last operation
                            RegTree<T, TRACE> rt;
                            rt.enter(fr.stage_in(n), op_log2n(w), o);
                            if (kind == OP_R0) rt.r0_root();
                            else
                                for (;;) {
                                    const uint32_t x = w & OPW_REG_EXIT ? 0u : win.get(j + 1);
                                    rt.exec(w, TRACE ? trace_row + __ldg(a.trace_offs + j) : nullptr);
                                    if (w & OPW_REG_EXIT) break;
                                    w = x;
                                    ++j;
                                }
                            rt.exit(fr.beta);
                            __syncwarp();
                        } else {
                            exec_op<T, WarpGrp>(kind, n, o, fr);
                            __syncwarp();
                            if (TRACE) {
                                trace_store<T, WarpGrp>(kind, n, __ldg(a.trace_offs + j), fr, trace_row);
                                __syncwarp();
                            }
                        }
                        if (++j >= a.n_ops) break;
                        w = win.get(j);
                        if (op_log2n(w) > a.log2W) break;
                    }
                    i = j;
                } else {
                    i = win.skip_narrow(i, a.log2W);
                }
                __syncthreads();
            } else {
                const uint32_t kind = op_kind(w), n = 1u << op_log2n(w);
                exec_op<T, CtaGrp>(kind, n, op_off(w), fr);
                __syncthreads();
                if (TRACE) trace_store<T, CtaGrp>(kind, n, __ldg(a.trace_offs + i), fr, trace_row);
                ++i;
            }
        }
    }
};

template <typename T, bool TRACE, bool STAGE>
__global__ void __launch_bounds__(1024) fastssc_decode_kernel(const KernelArgs a) {
    run_frames<T, TRACE, STAGE>(a, InterpBody<T, TRACE>{a});
}

template <typename T, bool TRACE, bool STAGE>
const void *kernel_ptr() {
    return reinterpret_cast<const void *>(&fastssc_decode_kernel<T, TRACE, STAGE>);
}

const void *select_kernel(bool is_i8, bool trace, bool stage) {
    if (is_i8) {
        if (trace) return stage ? kernel_ptr<int8_t, true, true>() : kernel_ptr<int8_t, true, false>();
        return stage ? kernel_ptr<int8_t, false, true>() : kernel_ptr<int8_t, false, false>();
    }
    if (trace) return stage ? kernel_ptr<float, true, true>() : kernel_ptr<float, true, false>();
    return stage ? kernel_ptr<float, false, true>() : kernel_ptr<float, false, false>();
}


}  // namespace

// Raise a kernel variant's dynamic shared-memory limit to the device's opt-in
// maximum, once per (variant, device). It is never lowered afterwards, so any
// shape the host selects can launch.
cudaError_t ensure_smem_limit(const void *k) {
    static std::mutex mu;
    static std::set<std::pair<const void *, int>> done;
    int device = 0;
    cudaError_t e = cudaGetDevice(&device);
    if (e != cudaSuccess) return e;
    std::lock_guard<std::mutex> g(mu);
    if (done.count({k, device})) return cudaSuccess;
    int optin = 0;
    e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, device);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, optin);
    if (e == cudaSuccess) done.insert({k, device});
    return e;
}


// Fixed device scratch for polar_decode_noalloc: the alpha stages above the
// shared-memory cap of every resident CTA live here instead of in memory taken
// with cudaMallocAsync. Every GPU that loads this library holds the array until
// the process exits; all calls on a device share it.
static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoAllocScratchBytes];

cudaError_t noalloc_scratch(void **ptr) {
    static std::mutex mu;
    static void *addr[kMaxDevices] = {};
    int device = 0;
    cudaError_t e = cudaGetDevice(&device);
    if (e != cudaSuccess) return e;
    if (device < 0 || static_cast<size_t>(device) >= kMaxDevices) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> g(mu);
    if (!addr[device]) {
        // Host code only knows a stand-in for the array; its device address is
        // looked up once per device, with that device current.
        void *p = nullptr;
        e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
        if (e != cudaSuccess) return e;
        addr[device] = p;
    }
    *ptr = addr[device];
    return cudaSuccess;
}

size_t kernel_smem_bytes(uint32_t N, uint32_t S, uint32_t threads, bool is_i8, bool stage) {
    (void)threads;
    return SmemLayout(N, S, is_i8 ? 1u : 4u, stage).total;
}

int kernel_max_ctas_per_sm(bool is_i8, bool stage, uint32_t threads, size_t smem_bytes) {
    const void *k = select_kernel(is_i8, false, stage);
    if (ensure_smem_limit(k) != cudaSuccess) return 0;
    int n = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k, static_cast<int>(threads),
                                                      smem_bytes) != cudaSuccess)
        return 0;
    return n;
}

// Self-test of the bounded wait: an mbarrier that expects one arrival which
// never comes; the wait gives up after limit_ns, exactly as the channel-staging
// wait does, and reports through the status word. No copy is in flight, so the
// CTA can leave at once.
__global__ void bounded_wait_selftest_kernel(int *status, unsigned long long limit_ns) {
    __shared__ uint64_t bar;
    if (threadIdx.x == 0) {
        mbar_init(&bar);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        if (!mbar_wait(&bar, 0u, limit_ns)) atomicOr(status, 1);
    }
}

cudaError_t launch_bounded_wait_selftest(int *status, unsigned long long limit_ns,
                                         cudaStream_t stream) {
    bounded_wait_selftest_kernel<<<1, 32, 0, stream>>>(status, limit_ns);
    return cudaGetLastError();
}

cudaError_t launch_decode(bool is_i8, bool trace, bool stage, const LaunchShape &shape,
                          const KernelArgs &args, cudaStream_t stream) {
    const void *k = select_kernel(is_i8, trace, stage);
    cudaError_t e = ensure_smem_limit(k);
    if (e != cudaSuccess) return e;
    void *params[] = {const_cast<KernelArgs *>(&args)};
    return cudaLaunchKernel(k, dim3(shape.grid), dim3(shape.threads), params, shape.smem_bytes,
                            stream);
}

}  // namespace polar
