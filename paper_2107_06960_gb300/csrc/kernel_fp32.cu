// fp32 kernel: fused-tile execution (MAFAT, Sec. 4) on CUDA cores.
//
// Runs the same task list and persistent scheduler as the tensor-core kernel, with fp32
// activations, weights and accumulation: an implicit GEMM on the FFMA pipe, which bounds
// it (152 SMs x 128 lanes).  Tensor cores would need the fp32 operands split in several
// 16-bit parts, and their accumulation is less exact than a chain of fmaf.
//
// One CTA of 128 threads computes one item: up to f32_groups groups of 8 neighbouring
// pixels of a row of the task's conv region x f32_nb output channels.  Groups of 8 pixels,
// not 16 x 8 blocks, are what a region is cut into, so that the 19- or 5-pixel regions of
// the later layers waste little.  A thread owns one group x CT channels (8 CT accumulators):
//   acc[o][x] = sum over input channel chunks, ky, kx, channels of w * in
// in that order whatever the item's shape, so every tiling of a plan and every CT give the
// same bits.  Per channel quad and kernel row it loads 10 pixels x 4 channels once from shared
// memory (16 bytes each) and uses them for three taps x CT channels.  Operands come by
// cp.async through a ring of chunks (one quad of a 3x3, four of a 1x1; the zero padding is
// cp.async's zero fill), weights packed on the host in the order the loop reads them.  Then
//   z = scale[o] * acc + bias[o];  out = z > 0 ? z : 0.1 z
// and, for a fused max-pool, the 2x2 maximum: rows 2r and 2r + 1 of a group column are
// neighbouring groups of one warp (one exchange), neighbouring pixels are in one thread.
//
// Which CT (8, 4, 2, or 1 with half the groups) a stage runs is the planner's choice
// (f32_shape): large stages take CT = 8, which is nearest the FFMA rate; stages with fewer
// than about three such items per SM take narrower ones, which spread over more warps.
//
// Measured on GB300: a 3x3 128 -> 256 convolution of 152x152 at 50 TFLOP/s (0.27 ms; a thread
// per pixel reading both operands from L1 took ~30 times as long), 1x1 256 -> 128 at 25; the
// 16-layer network at 416x416 29.06 -> 0.83 ms, two 96x96 frames 53.9 -> 0.30 ms (the shapes'
// choice and, for the two frames, the hand-out order included).  Those small frames are bound by
// their chain of 12 dependent layers (10-45 us each: a 64-chunk item of CT = 1, alone on its SM,
// takes ~0.7 us a chunk; F32Cost in planner.h has the times of the other shapes).  Measured and not kept: the halo held twice in shared
// memory so that pair instructions need no moves (42 instead of 50 TFLOP/s: 30 % more loads);
// a chunk's rows unrolled (a lone warp's instruction fetches); 128 registers and 4 CTAs per SM.
#include "sched.cuh"

namespace {

constexpr int kThreads = 128;
constexpr int kSmemFloats = 17 * 1024;  // ring of chunks: 4 of the largest item shape, up to 8 of the others
constexpr int kSmemBytes = kSmemFloats * 4;
constexpr int kCtasPerSm = 3;           // 168 registers a thread, 68 KB of shared memory

__device__ __forceinline__ const float* buf_ptr(const MafatKParams& p, int kind) {
    switch (kind) {
        case MAFAT_BUF_USER_IN: return (const float*)p.user_in;
        case MAFAT_BUF_CUT: return (const float*)p.cut;
        case MAFAT_BUF_SCRATCH:
        case MAFAT_BUF_MAP: return (const float*)p.scratch;
        default: return (const float*)p.user_out;
    }
}

// 16 or 4 bytes of global memory into shared memory; bytes = 0 writes zeros, on = false nothing.
// No branch: a chunk's copies are a straight run (a branch per copy restarts the instruction
// fetch of a scheduler that has one warp to issue from).
__device__ __forceinline__ void cp16(uint32_t dst, const float* src, int bytes, bool on = true) {
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %3, 0;\n\t"
                 "@p cp.async.cg.shared.global [%0], [%1], 16, %2;\n\t}" ::"r"(dst), "l"(src), "r"(bytes), "r"((int)on)
                 : "memory");
}
__device__ __forceinline__ void cp4(uint32_t dst, const float* src, int bytes) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// Weights of one (tap, channel) row for a thread's CT channels, as packed pairs of channels
// (CT = 1: one float).  Channel lane l owns channels 4l .. 4l + 3 and 32 + 4l .. for CT = 8,
// else CT l .. CT l + CT - 1.
template <int CT>
struct Wt {
    unsigned long long v[CT / 2];
    __device__ __forceinline__ void load(const float* row, int l) {
        if constexpr (CT == 8) {
            const ulonglong2 a = reinterpret_cast<const ulonglong2*>(row)[l], b = reinterpret_cast<const ulonglong2*>(row)[8 + l];
            v[0] = a.x, v[1] = a.y, v[2] = b.x, v[3] = b.y;
        } else if constexpr (CT == 4) {
            const ulonglong2 a = reinterpret_cast<const ulonglong2*>(row)[l];
            v[0] = a.x, v[1] = a.y;
        } else {
            v[0] = reinterpret_cast<const unsigned long long*>(row)[l];
        }
    }
};
template <>
struct Wt<1> {
    float v[1];
    __device__ __forceinline__ void load(const float* row, int l) { v[0] = row[l]; }
};

// Accumulators of one pixel: CT channels, in pairs.  fma.rn.f32x2 rounds each half as fmaf does;
// it takes half the operand reads of two FFMA, which the register file holds to ~50 of 80
// TFLOP/s in an 8 x 8 outer product (measured: 62 TFLOP/s with pairs).
template <int CT>
struct Acc {
    unsigned long long v[CT / 2];
    __device__ __forceinline__ void zero() {
#pragma unroll
        for (int o = 0; o < CT / 2; ++o) v[o] = 0ull;
    }
    __device__ __forceinline__ void fma(const Wt<CT>& w, float a) {
        unsigned long long aa;
        asm("mov.b64 %0, {%1, %1};" : "=l"(aa) : "f"(a));
#pragma unroll
        for (int o = 0; o < CT / 2; ++o) asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(v[o]) : "l"(w.v[o]), "l"(aa));
    }
    __device__ __forceinline__ float get(int o) const {
        float lo, hi;
        asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v[o >> 1]));
        return o & 1 ? hi : lo;
    }
};
template <>
struct Acc<1> {
    float v[1];
    __device__ __forceinline__ void zero() { v[0] = 0.f; }
    __device__ __forceinline__ void fma(const Wt<1>& w, float a) { v[0] = fmaf(w.v[0], a, v[0]); }
    __device__ __forceinline__ float get(int) const { return v[0]; }
};

__device__ __forceinline__ float pick(const float4& v, int c) { return c == 0 ? v.x : c == 1 ? v.y : c == 2 ? v.z : v.w; }

// One item.  L channel lanes x G groups = 128 threads; NB = L CT output channels.
template <int K, int L, int CT>
__device__ __forceinline__ void run_item(const MafatKParams& p, const MafatItemDev& it, const MafatTaskDev& tk,
                                         const MafatStageDev& st, float* smem, int ticket) {
    constexpr int G = kThreads / L, NB = L * CT;
    constexpr int kPx = K == 3 ? 30 : 8;                 // pixels copied per group and quad
    constexpr int kGroupPx = K == 3 ? 30 : 9;            // their slots in shared memory (a pad against bank conflicts)
    constexpr int kQuads = K == 3 ? 1 : 4;               // channel quads per chunk
    constexpr int kSlots = G * kPx * (K == 3 ? 1 : 4);   // 16-byte copies of a chunk
    constexpr int kPer = (kSlots + kThreads - 1) / kThreads;
    constexpr int kW16 = K * K * 4 * kQuads * NB / 4;    // 16-byte pieces of a chunk's weights
    constexpr int kAFloats = G * kGroupPx * 4 * kQuads, kStageFloats = kAFloats + kW16 * 4;
    // chunks in flight hide the L2 latency (~1 us under load) of narrow items, whose chunks take ~0.25 us
    constexpr int kStages = kSmemFloats / kStageFloats < 8 ? kSmemFloats / kStageFloats : 8;
    static_assert(kStages >= 3, "chunk ring");
    const int tid = threadIdx.x;
    const int gi = tid / L, l = tid % L;
    const int lin0 = (it.bx * 32768 + it.by) * G;        // first group of the item
    const int gx = tk.nbx;                               // groups per row
    const int n_chunks = st.f32_chunks;
    const uint32_t sbase = (uint32_t)__cvta_generic_to_shared(smem);
    // group g of the task -> conv position; groups past the region's end get a row past it
    auto locate = [&](int g, int& Y, int& X) {
        int y, x;
        if (st.f32_rect) {  // 16 rows x 1 group column blocks, stacked along rows
            const int nby = (tk.ch + G - 1) / G;
            const int blk = g / G;
            x = blk / nby;
            y = (blk - x * nby) * G + g % G;
        } else if (st.pool) {
            const int pr = (g >> 1) / gx;
            y = 2 * pr + (g & 1);
            x = (g >> 1) - pr * gx;
        } else {
            y = g / gx;
            x = g - y * gx;
        }
        Y = tk.cy0 + y;
        X = tk.cx0 + 8 * x;
    };
    int Yg, Xg;
    locate(lin0 + gi, Yg, Xg);
    const int y_end = tk.cy0 + tk.ch, x_end = tk.cx0 + tk.cw;
    const bool live = Yg < y_end && Xg < x_end;
    const bool warp_live = __any_sync(0xffffffffu, live);

    const bool nhwc = tk.in_kind == MAFAT_BUF_USER_IN;  // the caller's image; all else is octet-planar
    const float* const in = buf_ptr(p, tk.in_kind) + tk.in_off;
    const int64_t plane = nhwc ? 8 : (int64_t)tk.in_h * tk.in_w * 8;  // elements from an octet to the next
    const int cin = st.cin, pix_stride = nhwc ? cin : 8;
    const bool wide = !nhwc || (cin & 3) == 0;          // a quad of channels is one aligned 16-byte read
    // this thread's copies of a chunk, s = tid + 128 i: quad of the chunk and place in the chunk's
    // slot (both fold to constants and a term of tid), and the pixel in the input buffer (-1: zero
    // padding)
    auto slot_q = [&](int i) { return K == 3 ? 0 : i * (kThreads / (G * kPx)) + tid / (G * kPx); };
    const uint32_t dst0 = K == 3 ? tid * 16u
                                 : (uint32_t)((tid / (G * kPx) * G * kGroupPx + tid % (G * kPx) / 8 * kGroupPx + tid % 8) * 16);
    constexpr uint32_t kDstStep = K == 3 ? kThreads * 16u : (uint32_t)(kThreads / (G * kPx) * G * kGroupPx * 16);
    int off[kPer];
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
        const int s = tid + i * kThreads;
        const int r = s % (G * kPx), g = r / kPx, e = r - g * kPx;
        off[i] = -1;
        if (s < kSlots) {
            int Y, X;
            locate(lin0 + g, Y, X);
            const int x_in = X + (K == 3 ? e % 10 - 1 : e);
            const int ly = Y + (K == 3 ? e / 10 - 1 : 0) - tk.in_y0, lx = x_in - tk.in_x0;
            const bool needed = Y < y_end && X < x_end && x_in < x_end + (K == 3 ? 1 : 0);
            if (needed && ly >= 0 && ly < tk.in_h && lx >= 0 && lx < tk.in_w) off[i] = ly * tk.in_w + lx;
        }
    }
    const float* wsrc = p.w_f32 + st.f32_w_off + ((size_t)it.nb * n_chunks) * (kW16 * 4);
    auto issue_w = [&](int c, int stage) {
        const uint32_t dst = sbase + (uint32_t)(stage * kStageFloats + kAFloats) * 4u + tid * 16;
        const float* s = wsrc + (size_t)c * (kW16 * 4) + tid * 4;
#pragma unroll
        for (int i = 0; i < (kW16 + kThreads - 1) / kThreads; ++i)
            cp16(dst + i * kThreads * 16, s + i * kThreads * 4, 16, (i + 1) * kThreads <= kW16 || tid + i * kThreads < kW16);
    };
    auto issue_a = [&](int c, int stage) {
        const uint32_t dst = sbase + (uint32_t)(stage * kStageFloats) * 4u;
        if (wide) {
#pragma unroll
            for (int i = 0; i < kPer; ++i) {
                const int q = c * kQuads + slot_q(i);
                const float* src = in + ((int64_t)(q >> 1) * plane + 4 * (q & 1)) + (int64_t)off[i] * pix_stride;
                const bool ok = off[i] >= 0 && 4 * q < cin;
                cp16(dst + dst0 + i * kDstStep, ok ? src : in, ok ? 16 : 0, (i + 1) * kThreads <= kSlots || tid + i * kThreads < kSlots);
            }
        } else {  // an image whose pixels are no multiple of 16 bytes: channel by channel
#pragma unroll 1
            for (int i = 0; i < kPer; ++i) {
                if (tid + i * kThreads >= kSlots) break;
                int o = -1;
#pragma unroll
                for (int k = 0; k < kPer; ++k)
                    if (k == i) o = off[k];
                const int q = c * kQuads + slot_q(i);
                const float* src = in + (int64_t)(o < 0 ? 0 : o) * cin + 4 * q;
                for (int ch = 0; ch < 4; ++ch) {
                    const bool ok = o >= 0 && 4 * q + ch < cin;
                    cp4(dst + dst0 + i * kDstStep + 4 * ch, ok ? src + ch : in, ok ? 4 : 0);
                }
            }
        }
    };

    // weights do not depend on other tiles: the first chunks' go out before the waits
#pragma unroll
    for (int c = 0; c < kStages - 1; ++c)
        if (c < n_chunks) issue_w(c, c);
    if (tid == 0) {
        mafat_dev::wait_item_deps(p.ctr, it, p.timeout_ns);
        if (tk.dep_count > 0) mafat_dev::wait_dep_list(p.ctr, p.deps, tk.dep_first, tk.dep_count, p.timeout_ns);
        if (p.trace) mafat_dev::trace_put(p.trace, ticket, 1, mafat_dev::globaltimer_ns());
    }
    __syncthreads();
#pragma unroll
    for (int c = 0; c < kStages - 1; ++c) {
        if (c < n_chunks) issue_a(c, c);
        cp_commit();
    }

    Acc<CT> sum[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) sum[j].zero();
    int stage = 0, fill = kStages - 1;  // ring slots of chunk c and of chunk c + kStages - 1
    for (int c = 0; c < n_chunks; ++c) {
        cp_wait<kStages - 2>();
        __syncthreads();  // chunk c has landed for every thread, and chunk c - 1's slot is free
        if (c + kStages - 1 < n_chunks) {
            issue_w(c + kStages - 1, fill);
            issue_a(c + kStages - 1, fill);
        }
        cp_commit();
        const float* as = smem + stage * kStageFloats;
        stage = stage + 1 == kStages ? 0 : stage + 1;
        fill = fill + 1 == kStages ? 0 : fill + 1;
        if (!warp_live) continue;
        // rows of the chunk: kernel rows of a 3x3, channel quads of a 1x1; a row has kSteps
        // (tap, channel) steps of 8 CT multiply-adds.  Rolled: a chunk in one straight run does not
        // fit the instruction cache of a scheduler that has one or two warps (measured: 40 % of
        // the stalls of a narrow item were instruction fetches).
        constexpr int kRows = K == 3 ? 3 : kQuads, kSteps = 4 * K, kCols = K == 3 ? 10 : 8;
        const float4* ap = reinterpret_cast<const float4*>(as) + gi * kGroupPx;
        const float* wr = as + kAFloats;
#pragma unroll 1
        for (int r = 0; r < kRows; ++r, ap += K == 3 ? 10 : G * kGroupPx, wr += kSteps * NB) {
            float4 a[kCols];
#pragma unroll
            for (int j = 0; j < kCols; ++j) a[j] = ap[j];
            constexpr int kAhead = CT <= 2 ? kSteps : 2;  // weight rows read ahead
            Wt<CT> w[kAhead];
#pragma unroll
            for (int i = 0; i < kAhead; ++i) w[i].load(wr + i * NB, l);
#pragma unroll
            for (int i = 0; i < kSteps; ++i) {
#pragma unroll
                for (int j = 0; j < 8; ++j) sum[j].fma(w[i % kAhead], pick(a[j + (i >> 2)], i & 3));
                if (i + kAhead < kSteps) w[i % kAhead].load(wr + (i + kAhead) * NB, l);
            }
        }
    }

    // folded batch-norm, leaky ReLU, pool, stores
    if (warp_live) {
        auto chan = [&](int o) {  // channel within the item of this thread's o-th
            if constexpr (CT == 8)
                return (o & 4) * 8 + 4 * l + (o & 3);
            else
                return CT * l + o;
        };
        const int ch0 = it.nb * NB;
        float acc[CT][8];
#pragma unroll
        for (int o = 0; o < CT; ++o) {
            const int ch = ch0 + chan(o);
            const float sc = ch < st.cout ? __ldg(p.scale + st.sb_off + ch) : 0.f;
            const float bi = ch < st.cout ? __ldg(p.bias + st.sb_off + ch) : 0.f;
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const float z = sc * sum[j].get(o) + bi;
                acc[o][j] = z > 0.f ? z : 0.1f * z;
            }
        }
        float* out = (float*)(tk.out_kind == MAFAT_BUF_USER_OUT ? p.user_out
                              : tk.out_kind == MAFAT_BUF_CUT    ? p.cut
                                                                : p.scratch) + tk.out_off;
        constexpr int V = CT >= 4 ? 4 : CT;  // channels of one store
        int oy = Yg, ox = Xg, n = min(8, x_end - Xg);
        bool store = live;
        if (st.pool) {
#pragma unroll
            for (int o = 0; o < CT; ++o)
#pragma unroll
                for (int j = 0; j < 8; ++j) acc[o][j] = fmaxf(acc[o][j], __shfl_xor_sync(0xffffffffu, acc[o][j], L));
#pragma unroll
            for (int o = 0; o < CT; ++o)
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[o][j] = fmaxf(acc[o][2 * j], acc[o][2 * j + 1]);
            store = live && (Yg & 1) == 0;
            oy >>= 1;
            ox >>= 1;
            n >>= 1;  // a pooled region has even extents
        }
        if (store) {
            const size_t pix0 = (size_t)(oy - tk.out_y0) * tk.out_w + (ox - tk.out_x0);
            const size_t plane = (size_t)tk.out_h * tk.out_w * 8;
#pragma unroll
            for (int o = 0; o < CT; o += V) {
                const int ch = ch0 + chan(o);
                if (ch >= st.cout) continue;
                float* dst = tk.out_nhwc ? out + pix0 * st.cout + ch
                                         : out + (size_t)(ch >> 3) * plane + pix0 * 8 + (ch & 7);
                const int step = tk.out_nhwc ? st.cout : 8;
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    if (j >= n) break;
                    if constexpr (V == 4)
                        *reinterpret_cast<float4*>(dst) = make_float4(acc[o][j], acc[o + 1][j], acc[o + 2][j], acc[o + 3][j]);
                    else if constexpr (V == 2)
                        *reinterpret_cast<float2*>(dst) = make_float2(acc[o][j], acc[o + 1][j]);
                    else
                        *dst = acc[o][j];
                    dst += step;
                }
            }
        }
    }
}

__global__ void __launch_bounds__(kThreads, kCtasPerSm) mafat_fp32_kernel(const __grid_constant__ MafatKParams p) {
    extern __shared__ __align__(16) float smem[];
    __shared__ int s_ticket;
    const int tid = threadIdx.x;
    while (true) {
        if (tid == 0) s_ticket = (int)atomicAdd(&p.ctr[MAFAT_CTR_TICKET], 1u);
        __syncthreads();
        const int ticket = s_ticket;
        if (ticket >= p.n_items) break;
        const MafatItemDev it = p.items[ticket];
        const MafatTaskDev& tk = p.tasks[it.task];
        const MafatStageDev& st = p.stages[it.stage];
        if (p.trace && tid == 0) {
            mafat_dev::trace_put(p.trace, ticket, 0, mafat_dev::globaltimer_ns());
            mafat_dev::trace_put(p.trace, ticket, 4, mafat_dev::smid());
        }
        const int ct = st.f32_ct;
        if (st.k == 3) {
            if (ct == 8) run_item<3, 8, 8>(p, it, tk, st, smem, ticket);
            else if (ct == 4) run_item<3, 8, 4>(p, it, tk, st, smem, ticket);
            else if (ct == 2) run_item<3, 8, 2>(p, it, tk, st, smem, ticket);
            else run_item<3, 16, 1>(p, it, tk, st, smem, ticket);
        } else {
            if (ct == 8) run_item<1, 8, 8>(p, it, tk, st, smem, ticket);
            else if (ct == 4) run_item<1, 8, 4>(p, it, tk, st, smem, ticket);
            else if (ct == 2) run_item<1, 8, 2>(p, it, tk, st, smem, ticket);
            else run_item<1, 16, 1>(p, it, tk, st, smem, ticket);
        }
        __syncthreads();
        // the barrier orders every thread's stores before this thread's release
        if (tid == 0) {
            mafat_dev::publish_item(p.ctr, it, tk.done_ctr);
            if (p.trace) {
                const uint64_t t = mafat_dev::globaltimer_ns();
                mafat_dev::trace_put(p.trace, ticket, 2, t);
                mafat_dev::trace_put(p.trace, ticket, 3, t);
            }
        }
    }
    mafat_dev::finish_cta(p.ctr, p.n_ctr);
}

}  // namespace

namespace {
// One thread per (frame, octet, y, x), x fastest, so that the 8-element writes of a
// warp are contiguous; channels at or above c are written as zero.
template <typename T>
__global__ void __launch_bounds__(256) to_planar_kernel(const T* __restrict__ in, T* __restrict__ out, int frames,
                                                        int h, int w, int c, int c8) {
    const int64_t total = (int64_t)frames * c8 * h * w;
    const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= total) return;
    const int x = (int)(idx % w);
    int64_t r = idx / w;
    const int y = (int)(r % h);
    r /= h;
    const int o = (int)(r % c8);
    const int f = (int)(r / c8);
    const T* src = in + (((int64_t)f * h + y) * w + x) * c;
    T v[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        const int ch = o * 8 + k;
        v[k] = ch < c ? src[ch] : T(0);
    }
    T* dst = out + idx * 8;  // [f][o][y][x][8] in idx order, 16-byte aligned
    if constexpr (sizeof(T) == 2) {
        uint4 q;
        q.x = (uint32_t)v[0] | ((uint32_t)v[1] << 16);
        q.y = (uint32_t)v[2] | ((uint32_t)v[3] << 16);
        q.z = (uint32_t)v[4] | ((uint32_t)v[5] << 16);
        q.w = (uint32_t)v[6] | ((uint32_t)v[7] << 16);
        *reinterpret_cast<uint4*>(dst) = q;
    } else {
        reinterpret_cast<float4*>(dst)[0] = make_float4(v[0], v[1], v[2], v[3]);
        reinterpret_cast<float4*>(dst)[1] = make_float4(v[4], v[5], v[6], v[7]);
    }
}
}  // namespace

cudaError_t mafat_launch_to_planar(const void* nhwc, void* planar, int frames, int h, int w, int c, int c8,
                                   int elem_bytes, cudaStream_t s) {
    const int64_t total = (int64_t)frames * c8 * h * w;
    if (total <= 0) return cudaSuccess;
    const unsigned grid = (unsigned)((total + 255) / 256);
    if (elem_bytes == 2)
        to_planar_kernel<uint16_t><<<grid, 256, 0, s>>>((const uint16_t*)nhwc, (uint16_t*)planar, frames, h, w, c, c8);
    else
        to_planar_kernel<float><<<grid, 256, 0, s>>>((const float*)nhwc, (float*)planar, frames, h, w, c, c8);
    return cudaGetLastError();
}

int mafat_fp32_ctas_per_sm() { return kCtasPerSm; }
size_t mafat_fp32_smem_bytes() { return (size_t)kSmemBytes; }

cudaError_t mafat_prepare_fp32() {
    return cudaFuncSetAttribute(mafat_fp32_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes);
}

cudaError_t mafat_launch_fp32(const MafatKParams& p, int grid, cudaStream_t s) {
    mafat_fp32_kernel<<<grid, kThreads, kSmemBytes, s>>>(p);
    return cudaGetLastError();
}
