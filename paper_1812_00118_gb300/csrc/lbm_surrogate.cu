// Kernels of the learned warm-start surrogate (include/lbm_surrogate.h):
// periodic 3x3 convolutions on BF16 tensor cores with FP32 accumulation, and
// the elementwise, pooling, loss and optimiser kernels around them.
//
// Tensors are channels-last: pixel p = (n H + y) W + x, element (p, c) at
// p * stride + c (a channel stride larger than the channel count lets a
// layer read or write a slice of a wider tensor, which is how the skip
// concatenation is laid out).  Conv weights are [Co][9][Ci] (tap = 3 dy + dx,
// input channels fastest).  Channel counts of convolutions are multiples of
// 16 (zero-padded by the caller), pixel counts multiples of 16.
//
// The forward (and input-gradient) convolution runs on the tcgen05 tensor
// cores with the accumulator in tensor memory: conv_row_kernel for images
// whose width is a multiple of 128 and whose ring of rows and weights fit
// shared memory, else conv_flat_kernel where its cells and two taps' weights
// fit and the image is not too wide, else conv_tc_kernel (conv3x3 below has the
// rule).  So does the weight gradient, a GEMM over pixels, for widths that are
// multiples of 32 (conv_wgrad_row_kernel), with the warp-level mma.sync
// m16n8k16 BF16 kernel (fragments gathered straight from the channels-last
// tensors) for the rest.  All are implicit GEMMs without an im2col buffer.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <stdint.h>

#include "lbm.h"
#include "lbm_surrogate.h"

namespace {

using bf16 = __nv_bfloat16;

int check(cudaError_t e) { return e == cudaSuccess ? LBM_OK : LBM_ECUDA; }

__device__ __forceinline__ void mma_bf16(float (&d)[4], const uint32_t (&a)[4], const uint32_t (&b)[2]) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

__device__ __forceinline__ uint32_t pack_pair(const bf16* lo, const bf16* hi) {
    const uint32_t a = *reinterpret_cast<const unsigned short*>(lo);
    const uint32_t b = *reinterpret_cast<const unsigned short*>(hi);
    return a | (b << 16);
}

// pixel p shifted by (dy, dx) with periodic wrap inside its image
__device__ __forceinline__ long long shift_pixel(long long p, int H, int W, int dy, int dx) {
    const long long hw = (long long)H * W;
    const long long n = p / hw;
    const int r = (int)(p - n * hw);
    int y = r / W + dy, x = r % W + dx;
    y = y < 0 ? y + H : (y >= H ? y - H : y);
    x = x < 0 ? x + W : (x >= W ? x - W : x);
    return n * hw + (long long)y * W + x;
}

// ---------------------------------------------------------------- tcgen05 convolution
// The forward convolution (and the input-gradient convolution, the same
// operation on flipped weights) as an implicit GEMM on the fifth-generation
// tensor cores: D[pixel, co] = sum over (tap, ci) of A[pixel, (tap, ci)]
// B[(tap, ci), co], with A the shifted activations and B the weights, both
// bf16 and K-major (channels contiguous), D in FP32 in tensor memory.
//
// A CTA of 128 threads owns 128 consecutive pixels and every output channel
// (MMA shape M = 128, N = Co, K = 16).  The K loop runs over stages (tap,
// block of up to 64 input channels).  Per stage every thread copies its
// pixel's shifted channel row (16-byte cp.async; rows past the last pixel
// are zero-filled) and a share of the tap's weight rows into one of four
// shared-memory buffers, in the no-swizzle canonical layout of the tensor
// core: 8 x 16-byte core matrices, rows 16 bytes apart, 8-row groups 128
// bytes apart (stride byte offset), the 8-channel chunks one after another
// (leading byte offset = rows x 16 bytes).  The copies run two stages ahead
// of the MMAs: once a stage's copies have landed, warp 0 issues its MMAs
// and commits them to the buffer's mbarrier, and a buffer is refilled only
// after its mbarrier shows the MMAs that read it done.  The epilogue reads
// the accumulator back with tcgen05.ld (warp w reads lanes 32w..32w+31, one
// pixel per thread), adds the bias and stores FP32.
//
// Every wait is bounded: a wait that gives up sets *err (read by
// lbm_sg_status) and the CTA skips its epilogue, frees its tensor memory and
// returns.
constexpr int kTcM = 128;        // pixels per CTA (MMA M)
constexpr int kTcK = 64;         // input channels per stage
constexpr int kTcBuf = 4;        // stage buffers in shared memory
constexpr int kTcAhead = 2;      // stages whose copies are in flight ahead of the MMAs
constexpr long kTcPolls = 1L << 24;

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, uint32_t src_bytes) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(src_bytes) : "memory");
}

__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}

// true once the phase of the given parity has completed; false after `polls` tries
__device__ __forceinline__ bool mbar_wait_bounded(uint32_t bar, uint32_t parity, long polls) {
    for (long i = 0; i < polls; ++i)
        if (mbar_try(bar, parity)) return true;
    return false;
}

// shared-memory matrix descriptor, no swizzle: start address, leading and
// stride byte offsets (all in 16-byte units), descriptor version 1
__device__ __forceinline__ uint64_t tc_smem_desc(uint32_t addr, uint32_t lbo, uint32_t sbo) {
    return (uint64_t)((addr >> 4) & 0x3FFFu) | ((uint64_t)((lbo >> 4) & 0x3FFFu) << 16) |
           ((uint64_t)((sbo >> 4) & 0x3FFFu) << 32) | ((uint64_t)1 << 46);
}

// instruction descriptor of kind::f16: FP32 accumulator, bf16 A and B, both
// K-major, N / 8 and M / 16
__host__ __device__ constexpr uint32_t tc_idesc_bf16(int M, int N) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

// The issuing thread of a warp: 1 in one lane (the same at every call), 0 in
// the others.
__device__ __forceinline__ uint32_t tc_elect() {
    uint32_t e;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(e));
    return e;
}

// One MMA, issued by the lane with el != 0; every lane of the warp calls it.
__device__ __forceinline__ void tc_mma(uint32_t el, uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t idesc,
                                       uint32_t acc) {
    asm volatile(
        "{\n\t.reg .pred p, q;\n\tsetp.ne.b32 p, %4, 0;\n\tsetp.ne.b32 q, %5, 0;\n\t"
        "@q tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
        "l"(a), "l"(b), "r"(idesc), "r"(acc), "r"(el)
        : "memory");
}

// mbarrier arrival once every MMA the lane with el != 0 has issued is done
__device__ __forceinline__ void tc_commit(uint32_t el, uint32_t bar) {
    if (el)
        asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar)
                     : "memory");
}

// n MMAs of K = 16 into one accumulator, operand descriptors a step apart (the
// address field counts 16-byte units and never carries out of its 14 bits); the
// first one starts the sum unless `acc`.  Called by a whole warp with uniform
// arguments, and straight-line for the counts that occur (powers of two): the
// descriptors then stay in uniform registers and the issue keeps up with the
// tensor core.  (clk per MMA of M = 128, K = 16, N = 32 / 128, one CTA: 40 / 64;
// in a loop of one MMA per pass 120; from a branch of one thread that steps the
// descriptors 155; the core itself needs 64 at N = 128, and 32 to read A.)
template <int N>
__device__ __forceinline__ void tc_mma_fixed(uint32_t el, uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t a_step,
                                             uint32_t b_step, uint32_t idesc, bool acc) {
#pragma unroll
    for (int k = 0; k < N; ++k)
        tc_mma(el, d_tmem, a + (uint64_t)k * a_step, b + (uint64_t)k * b_step, idesc, (k > 0 || acc) ? 1u : 0u);
}
__device__ __forceinline__ void tc_mma_run(uint32_t el, uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t a_step,
                                           uint32_t b_step, uint32_t idesc, int n, bool acc) {
    for (int k = 0; k < n;) {
        const uint64_t ak = a + (uint64_t)((uint32_t)k * a_step), bk = b + (uint64_t)((uint32_t)k * b_step);
        const bool on = acc || k > 0;
        if (n - k >= 8) { tc_mma_fixed<8>(el, d_tmem, ak, bk, a_step, b_step, idesc, on); k += 8; }
        else if (n - k >= 4) { tc_mma_fixed<4>(el, d_tmem, ak, bk, a_step, b_step, idesc, on); k += 4; }
        else if (n - k >= 2) { tc_mma_fixed<2>(el, d_tmem, ak, bk, a_step, b_step, idesc, on); k += 2; }
        else { tc_mma_fixed<1>(el, d_tmem, ak, bk, a_step, b_step, idesc, on); k += 1; }
    }
}

// 16 consecutive FP32 columns of the thread's lane
__device__ __forceinline__ void tc_ld16(uint32_t taddr, float (&v)[16]) {
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

// ---- roles of the march kernels: eight worker warps copy operands in and write
// results out, one more warp issues the MMAs; mbarriers are all that ties them.
// The issuing warp has no copies of its own in flight, so its proxy fence (the
// copies land through the generic proxy, the MMAs read through the async one)
// waits for nothing; executed by threads with cp.async outstanding, the fence
// waits for all of them and no copy runs ahead of the MMAs.
constexpr int kWorkers = 256;
constexpr int kRoleThreads = kWorkers + 32;

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("{\n\t.reg .b64 t;\n\tmbarrier.arrive.shared::cta.b64 t, [%0];\n\t}" ::"r"(bar) : "memory");
}
// arrival of this thread once all its cp.async so far have landed
__device__ __forceinline__ void mbar_arrive_copies(uint32_t bar) {
    asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(bar) : "memory");
}
// Wait for the phase of parity k & 1 of a barrier (its k-th, from 0); false once
// it, or another wait of the CTA, has given up (*failed).
__device__ __forceinline__ bool mbar_wait_phase(uint32_t bar, int k, volatile int* failed) {
    const uint32_t parity = (uint32_t)k & 1u;
    if (mbar_try(bar, parity)) return true;
    for (long i = 0; i < kTcPolls; ++i) {
        if (mbar_try(bar, parity)) return true;
        if ((i & 255) == 255 && *failed) return false;
    }
    *failed = 1;
    return false;
}

// The (row, 16-byte group) pairs of an operand a worker copies: `groups` per row,
// neighbouring workers on neighbouring groups.  Where the groups divide the
// workers (channel counts that are powers of two up to 2048) a worker keeps its
// group and steps through the rows without a division.
template <typename F>
__device__ __forceinline__ void for_groups(int tid, int rows, int groups, F&& f) {
    if ((groups & (groups - 1)) == 0 && groups <= kWorkers) {
        const int sh = 31 - __clz(groups), c = tid & (groups - 1), step = kWorkers >> sh;
        for (int q = tid >> sh; q < rows; q += step) f(q, c);
    } else {
        for (int e = tid; e < rows * groups; e += kWorkers) {
            const int q = e / groups;
            f(q, e - q * groups);
        }
    }
}

// A whole 32-byte sector per lane: lanes write pixels a row stride apart, and
// two 16-byte stores per sector cost L2 two partial writes (16 -> 32 channels at
// 8 x 256^2: 32 us, 27 with this).
__device__ __forceinline__ void st_global_32(void* p, const uint32_t (&v)[8]) {
    asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "r"(v[0]), "r"(v[1]), "r"(v[2]),
                 "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7])
                 : "memory");
}

// 16 channels of one pixel of a convolution's output, as FP32 or (ACT) as the
// bf16 values after the ReLU, which is all the next layer and the backward
// pass read of them; `vec`: every pixel's channels start on a 32-byte boundary.
// bias: 16 floats, 16-byte aligned (zeros where there is none).
template <bool ACT>
__device__ __forceinline__ void conv_store16(void* y, long long at, float (&v)[16], const float* bias, bool vec) {
#pragma unroll
    for (int i = 0; i < 16; i += 4) {
        const float4 b = *reinterpret_cast<const float4*>(bias + i);
        v[i] += b.x; v[i + 1] += b.y; v[i + 2] += b.z; v[i + 3] += b.w;
    }
    if constexpr (ACT) {
        bf16* out = (bf16*)y + at;
        __nv_bfloat162 h[8];
#pragma unroll
        for (int i = 0; i < 8; ++i)
            h[i] = __floats2bfloat162_rn(fmaxf(v[2 * i], 0.0f), fmaxf(v[2 * i + 1], 0.0f));
        if (vec) {
            uint32_t q[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) q[i] = *reinterpret_cast<const uint32_t*>(&h[i]);
            st_global_32(out, q);
        } else {
#pragma unroll
            for (int i = 0; i < 8; ++i) { out[2 * i] = h[i].x; out[2 * i + 1] = h[i].y; }
        }
    } else {
        float* out = (float*)y + at;
        if (vec) {
#pragma unroll
            for (int i = 0; i < 16; i += 8) {
                uint32_t q[8];
#pragma unroll
                for (int k = 0; k < 8; ++k) q[k] = __float_as_uint(v[i + k]);
                st_global_32(out + i, q);
            }
        } else {
#pragma unroll
            for (int i = 0; i < 16; ++i) out[i] = v[i];
        }
    }
}
template <bool ACT>
__device__ __forceinline__ bool conv_vec(const void* y, int csy) {
    return (csy & (ACT ? 15 : 7)) == 0 && ((uintptr_t)y & 31) == 0;
}

template <bool ACT>
__global__ void __launch_bounds__(128, 1)
conv_tc_kernel(const bf16* __restrict__ x, int csx, const bf16* __restrict__ w, const float* __restrict__ bias,
               void* __restrict__ y, int csy, long long M, int H, int W, int Ci, int Co, int* err) {
    extern __shared__ __align__(1024) unsigned char smem[];
    __shared__ __align__(8) uint64_t bars[kTcBuf];
    __shared__ __align__(16) float bias_s[128];
    __shared__ uint32_t tmem_slot;
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;   // warp: uniform
    const long long p0 = (long long)blockIdx.x * kTcM;
    const int kcap = Ci < kTcK ? Ci : kTcK;   // channels per stage buffer
    const uint32_t a_bytes = kTcM * kcap * 2, stage_bytes = a_bytes + (uint32_t)Co * kcap * 2;
    const uint32_t sb = smem_u32(smem);
    // buffer b: A at sb + b stage_bytes, B a_bytes after it; its barrier at bar0 + 8 b
    const uint32_t bar0 = smem_u32(&bars[0]);
    const uint32_t ncols = Co <= 32 ? 32u : (Co <= 64 ? 64u : 128u);
    if (tid < Co) bias_s[tid] = bias ? bias[tid] : 0.0f;
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)),
                     "r"(ncols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid == 0) {
        for (int b = 0; b < kTcBuf; ++b)
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar0 + 8 * b) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = tmem_slot;
    const uint32_t idesc = tc_idesc_bf16(kTcM, Co);
    const int nkb = (Ci + kTcK - 1) / kTcK;
    const int nst = 9 * nkb;
    const long long p = p0 + tid;
    const bool in = p < M;
    // the copies of stage st into buffer st % kTcBuf, as one commit group
    auto issue = [&](int st) {
        const uint32_t a_s = sb + (st % kTcBuf) * stage_bytes, b_s = a_s + a_bytes;
        const int tap = st / nkb, kc0 = (st % nkb) * kTcK;
        const int kw = Ci - kc0 < kTcK ? Ci - kc0 : kTcK;
        const bf16* src = x + (in ? shift_pixel(p, H, W, tap / 3 - 1, tap % 3 - 1) : 0) * csx + kc0;
        for (int c = 0; c < kw / 8; ++c) cp_async16(a_s + c * (kTcM * 16) + tid * 16, src + c * 8, in ? 16u : 0u);
        for (int k = tid; k < Co * (kw / 8); k += kTcM) {
            const int co = k % Co, c = k / Co;
            cp_async16(b_s + c * (Co * 16) + co * 16, w + ((long long)co * 9 + tap) * Ci + kc0 + c * 8, 16u);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    // stage s commits to barrier s % kTcBuf: its (s / kTcBuf)-th phase
    auto wait_stage = [&](int st) {
        return mbar_wait_bounded(bar0 + 8 * (st % kTcBuf), (uint32_t)(st / kTcBuf) & 1u, kTcPolls);
    };
    bool ok = true;
    int issued = 0;   // stages whose MMAs were issued and committed
    for (int st = 0; st < kTcAhead && st < nst; ++st) issue(st);
    for (int st = 0; st < nst; ++st) {
        // copies run kTcAhead stages ahead; buffer (st + kTcAhead) % kTcBuf was
        // last read by the MMAs of stage st + kTcAhead - kTcBuf
        const int nxt = st + kTcAhead;
        if (nxt < nst) {
            if (nxt >= kTcBuf && !__syncthreads_and(wait_stage(nxt - kTcBuf))) {
                ok = false;
                break;
            }
            issue(nxt);
        }
        // stage st's group is complete once at most the newer ones are pending
        const int newer = (nst - 1 < st + kTcAhead ? nst - 1 : st + kTcAhead) - st;
        if (newer >= 2) asm volatile("cp.async.wait_group 2;" ::: "memory");
        else if (newer == 1) asm volatile("cp.async.wait_group 1;" ::: "memory");
        else asm volatile("cp.async.wait_group 0;" ::: "memory");
        // the copies were written through the generic proxy; the MMAs read through the async proxy
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncthreads();
        if (warp == 0) {
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint32_t el = tc_elect();
            const uint32_t a_s = sb + (st % kTcBuf) * stage_bytes, b_s = a_s + a_bytes;
            const int kc0 = (st % nkb) * kTcK;
            const int kw = Ci - kc0 < kTcK ? Ci - kc0 : kTcK;
            tc_mma_run(el, tmem, tc_smem_desc(a_s, kTcM * 16, 128), tc_smem_desc(b_s, Co * 16, 128), 2 * kTcM, 2 * Co,
                       idesc, kw / 16, st > 0);
            tc_commit(el, bar0 + 8 * (st % kTcBuf));
        }
        issued = st + 1;
    }
    // copies still in flight on the failure path land before the CTA leaves
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    // the last committed stage completes after every earlier MMA of the CTA
    // (waited for on the failure path too, before the tensor memory is freed)
    if (issued > 0) {
        const bool done = wait_stage(issued - 1);
        ok = __syncthreads_and(ok && done) != 0;
    }
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (ok) {
        const long long pr = p0 + 32 * warp + lane;
        const uint32_t trow = tmem + ((uint32_t)(32 * warp) << 16);
        const bool vec = conv_vec<ACT>(y, csy);
        for (int c0 = 0; c0 < Co; c0 += 16) {
            float v[16];
            tc_ld16(trow + (uint32_t)c0, v);
            if (pr < M) conv_store16<ACT>(y, pr * csy + c0, v, bias_s + c0, vec);
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(ncols) : "memory");
    if (!ok && tid == 0) atomicExch(err, 1);
}

// kTcBuf stage buffers of A (128 pixels) and B (Co weight rows), min(Ci, kTcK) channels each
size_t conv_tc_smem_bytes(int Ci, int Co) {
    const size_t k = Ci < kTcK ? (size_t)Ci : (size_t)kTcK;
    return (size_t)kTcBuf * (kTcM + (size_t)Co) * k * 2;
}

__device__ int g_sg_err;   // a bounded wait of a surrogate kernel gave up

// ---------------------------------------------------------------- tcgen05 convolution, row march
// The same convolution for images whose width is a multiple of 128: a CTA
// owns a 128-pixel segment of one image row and marches down a chunk of
// rows.  The shifted activations of a 3x3 tap are then rows of a halo
// strip: for row r the taps read input rows r - 1, r, r + 1 at pixel
// offsets -1, 0, +1 around the segment.  The strip is a ring of input rows
// (130 pixels each, the periodic neighbours included) in the tensor core's
// no-swizzle K-major layout, one 16-byte row per (pixel, 8 channels): a tap's
// A operand is the strip row of its dy started (1 + dx) pixels in, 128 rows
// of 16 bytes, 8-row core matrices 128 bytes apart, 8-channel planes an odd
// multiple of 16 bytes apart (the 8 groups of a pixel, copied by neighbouring
// threads, fall into different banks).  Every input row is copied into shared
// memory once (the tap kernel above copies it nine times) and the weights of
// all nine taps stay resident for the whole march.
//
// Worker warps copy the ring's rows ahead of the MMAs (a row's slot is refilled
// as soon as the last row that reads it is done) and write out one of two
// tensor-memory accumulators while the other is summed; a warp of its own
// issues the MMAs.  (On 128 threads that wrote out row j - 1 and copied row
// j + 1 before issuing row j the 64 -> 32 layer at 8 x 256^2 took 126 us with its
// FP32 output; this takes 52 to 54, and 43 with the ReLU in the epilogue and bf16
// out.)  Every wait is bounded, as in the tap kernel.
constexpr int kRowM = 128;          // pixels of a row segment (MMA M)
constexpr int kRowHalo = kRowM + 2;
constexpr int kRowSlots = 6;        // ring rows at most (at least 4)
constexpr size_t kRowSmemMax = 220 * 1024;

__host__ __device__ constexpr uint32_t row_plane_bytes() { return (kRowHalo | 1) * 16; }
__host__ __device__ inline uint32_t row_slot_bytes(int Ci) { return (uint32_t)(Ci / 8) * row_plane_bytes(); }
// weights: [tap][ci chunk][co], chunks an odd multiple of 16 bytes apart
__host__ __device__ inline uint32_t row_w_chunk(int Co) { return (uint32_t)(Co + 1) * 16; }
__host__ __device__ inline uint32_t row_w_bytes(int Ci, int Co) { return 9u * (uint32_t)(Ci / 8) * row_w_chunk(Co); }
// ring rows that fit beside the weights with `per_sm` CTAs on an SM (below 4:
// they do not fit)
inline int conv_row_slots_of(int Ci, int Co, int per_sm) {
    const size_t w = row_w_bytes(Ci, Co), most = kRowSmemMax / per_sm - (per_sm > 1 ? 1024 : 0);
    if (w >= most) return 0;
    const size_t n = (most - w) / row_slot_bytes(Ci);
    return n < (size_t)kRowSlots ? (int)n : kRowSlots;
}
size_t conv_row_smem_bytes(int Ci, int Co, int slots) {
    return (size_t)slots * row_slot_bytes(Ci) + row_w_bytes(Ci, Co);
}
// tensor-memory columns of the two accumulators (a power of two, at least 32)
__host__ __device__ inline uint32_t row_tmem_cols(int Co) {
    const int need = 2 * Co;
    return need <= 32 ? 32u : (need <= 64 ? 64u : (need <= 128 ? 128u : 256u));
}

template <bool ACT>
__global__ void __launch_bounds__(kRoleThreads, 3)
conv_row_kernel(const bf16* __restrict__ x, int csx, const bf16* __restrict__ w, const float* __restrict__ bias,
                void* __restrict__ y, int csy, int N, int H, int W, int Ci, int Co, int rows_per_cta, int slots,
                int* err) {
    extern __shared__ __align__(1024) unsigned char smem[];
    __shared__ __align__(8) uint64_t bars[kRowSlots + 4];   // full[slot], then done[2], drained[2]
    __shared__ __align__(16) float bias_s[128];
    __shared__ uint32_t tmem_slot;
    __shared__ int failed;
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;   // warp: uniform
    const int segs = W / kRowM;
    const int chunks = (H + rows_per_cta - 1) / rows_per_cta;
    int b = blockIdx.x;
    const int chunk = b % chunks;
    b /= chunks;
    const int seg = b % segs, n = b / segs;
    const int y0 = chunk * rows_per_cta;
    const int y1 = y0 + rows_per_cta < H ? y0 + rows_per_cta : H;
    const int x0 = seg * kRowM;
    const uint32_t wb = smem_u32(smem);                  // weights, then the ring
    const uint32_t sb = wb + row_w_bytes(Ci, Co);
    const uint32_t slot_bytes = row_slot_bytes(Ci), wchunk = row_w_chunk(Co);
    const uint32_t full = smem_u32(&bars[0]), mma_done = full + 8 * kRowSlots, drained = mma_done + 16;
    const uint32_t ncols = row_tmem_cols(Co);
    if (tid < Co) bias_s[tid] = bias ? bias[tid] : 0.0f;
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)),
                     "r"(ncols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid == 0) {
        for (int k = 0; k < slots; ++k) mbar_init(full + 8 * k, kWorkers);
        for (int k = 0; k < 2; ++k) {
            mbar_init(mma_done + 8 * k, 1);
            mbar_init(drained + 8 * k, kWorkers);
        }
        failed = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = tmem_slot;
    const int nch = Ci / 8;
    const int nrows = y1 - y0;
    // row j of the march (row y0 + j) sums in buffer j & 1 over input rows
    // j .. j + 2 (input row k: image row y0 - 1 + k, wrapped, in slot k % slots)
    int issued = 0;
    if (warp < kWorkers / 32) {
        const long long img = (long long)n * H * W;
        // the next input row to copy: its number, slot and image row
        int ck = 0, cs = 0, cy = y0 == 0 ? H - 1 : y0 - 1;
        auto copy_next = [&]() {   // pixels x0 - 1 .. x0 + 128 (wrapped)
            if (ck > nrows + 1) return;
            const uint32_t dst = sb + (uint32_t)cs * slot_bytes;
            const bf16* row = x + (img + (long long)cy * W) * csx;
            for_groups(tid, kRowHalo, nch, [&](int px, int c) {
                int xx = x0 - 1 + px;
                xx = xx < 0 ? xx + W : (xx >= W ? xx - W : xx);
                cp_async16(dst + c * row_plane_bytes() + px * 16, row + (long long)xx * csx + c * 8, 16u);
            });
            mbar_arrive_copies(full + 8 * cs);
            ++ck;
            cs = cs + 1 == slots ? 0 : cs + 1;
            cy = cy + 1 == H ? 0 : cy + 1;
        };
        for_groups(tid, 9 * Co, nch, [&](int row, int c) {   // the weights: landed with row 0
            const int co = row / 9, tap = row - co * 9;
            cp_async16(wb + (uint32_t)(tap * nch + c) * wchunk + co * 16, w + (long long)row * Ci + c * 8, 16u);
        });
        for (int k = 0; k < slots; ++k) copy_next();
        const bool vec = conv_vec<ACT>(y, csy);
        // warps w and w + 4 share a quarter of the lanes
        const uint32_t acc0 = tmem + ((uint32_t)(32 * (warp & 3)) << 16);
        long long at = (img + (long long)y0 * W + x0 + 32 * (warp & 3) + lane) * csy;
        for (int j = 0; j < nrows; ++j, at += (long long)W * csy) {
            // by warps: tcgen05.ld takes all 32 lanes or hangs
            if (!__all_sync(0xffffffffu, mbar_wait_phase(mma_done + 8 * (j & 1), j >> 1, &failed))) break;
            copy_next();   // row j + slots, into the slot of input row j, read last by row j
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            for (int c0 = 16 * (warp >> 2); c0 < Co; c0 += 32) {
                float v[16];
                tc_ld16(acc0 + (uint32_t)((j & 1) * Co + c0), v);
                conv_store16<ACT>(y, at + c0, v, bias_s + c0, vec);
            }
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            mbar_arrive(drained + 8 * (j & 1));
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
    } else {
        const uint32_t idesc = tc_idesc_bf16(kRowM, Co);
        const uint32_t el = tc_elect();
        // slots of input rows j, j + 1, j + 2; phase of the newest
        int s0 = 0, s1 = 1, s2 = 2, ph = 0;
        bool ok = mbar_wait_phase(full, 0, &failed) && mbar_wait_phase(full + 8, 0, &failed);
        const uint64_t a_hi = tc_smem_desc(0, row_plane_bytes(), 128), b0 = tc_smem_desc(wb, wchunk, 128);
        const uint32_t b_tap = (uint32_t)nch * wchunk / 16;
        for (int j = 0; j < nrows && ok; ++j) {
            ok = mbar_wait_phase(full + 8 * s2, ph, &failed);
            if (ok && j >= 2) ok = mbar_wait_phase(drained + 8 * (j & 1), (j >> 1) - 1, &failed);
            if (!__all_sync(0xffffffffu, ok)) break;
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint32_t acc = tmem + (uint32_t)((j & 1) * Co);
#pragma unroll
            for (int dy = 0; dy < 3; ++dy) {
                const uint64_t ad = a_hi + (uint64_t)((sb + (uint32_t)(dy == 0 ? s0 : (dy == 1 ? s1 : s2)) * slot_bytes) >> 4);
#pragma unroll
                for (int dx = 0; dx < 3; ++dx)
                    tc_mma_run(el, acc, ad + (uint64_t)dx, b0 + (uint64_t)((3 * dy + dx) * b_tap),
                               2 * row_plane_bytes() / 16, 2 * wchunk / 16, idesc, nch / 2, dy + dx > 0);
            }
            tc_commit(el, mma_done + 8 * (j & 1));
            issued = j + 1;
            s0 = s1;
            s1 = s2;
            s2 = s2 + 1 == slots ? 0 : s2 + 1;
            ph ^= s2 == 0;
        }
        // the MMAs still running (on the failure path) end before the tensor
        // memory is freed
        if (issued > 0) mbar_wait_bounded(mma_done + 8 * ((issued - 1) & 1), (uint32_t)((issued - 1) >> 1) & 1u, kTcPolls);
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(ncols) : "memory");
    if (tid == 0 && failed) atomicExch(err, 1);
}

// ---------------------------------------------------------------- tcgen05 convolution, flat tiles
// The same convolution for any other width: the image with one halo column on
// each side, read as one flat array of cells with row pitch W + 2.  Output
// position f (row f / (W + 2), column f % (W + 2)) then reads cell f + dy (W + 2)
// + dx for every tap, whatever row it is in, so 128 consecutive positions are
// one MMA tile even where they span several rows; the two positions per row
// that fall on the halo columns are computed and dropped.  A CTA copies the
// 128 + 2 (W + 3) cells its tile reads once, all channels of them (the tap
// kernel copies 9 x 128 pixels, a stage of 64 channels at a time), and the
// weights tap by tap through a ring of `stages` buffers.  Where the tiles leave
// SMs idle (one 256^2 image has 9 at the coarsest level) the output channels are
// split over blockIdx.y, Co of them each.  Taps and channels in the tap kernel's
// order.
constexpr int kFlatStages = 9;

__host__ __device__ inline int flat_cells(int W) { return 128 + 2 * (W + 3); }
__host__ __device__ inline uint32_t flat_plane(int W) { return (uint32_t)(flat_cells(W) | 1) * 16; }
__host__ __device__ inline uint32_t flat_x_bytes(int W, int Ci) { return (uint32_t)(Ci / 8) * flat_plane(W); }
__host__ __device__ inline uint32_t flat_w_bytes(int Ci, int Co) { return (uint32_t)(Ci / 8) * row_w_chunk(Co); }
// weight buffers of a launch: as many as leave room for two CTAs per SM, or
// else for one (below 2: the tiles do not apply)
inline int flat_stages(int W, int Ci, int Co) {
    if (W > 4096 || Ci > 4096) return 0;
    const size_t x = flat_x_bytes(W, Ci), w = flat_w_bytes(Ci, Co);
    size_t n = x + 2 * w <= kRowSmemMax / 2 ? (kRowSmemMax / 2 - x) / w : (x + 2 * w <= kRowSmemMax ? (kRowSmemMax - x) / w : 0);
    return n < (size_t)kFlatStages ? (int)n : kFlatStages;
}

template <bool ACT>
__global__ void __launch_bounds__(kRoleThreads, 3)
conv_flat_kernel(const bf16* __restrict__ x, int csx, const bf16* __restrict__ w, const float* __restrict__ bias,
                 void* y, int csy, int H, int W, int Ci, int Co, int tiles, int stages, int* err) {
    extern __shared__ __align__(1024) unsigned char smem[];
    __shared__ __align__(8) uint64_t bars[2 * kFlatStages];   // full[stage], done[stage]
    __shared__ __align__(16) float bias_s[128];
    __shared__ uint32_t tmem_slot;
    __shared__ int failed;
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;   // warp: uniform
    w += (long long)blockIdx.y * Co * 9 * Ci;
    if (bias) bias += blockIdx.y * Co;
    y = ACT ? (void*)((bf16*)y + blockIdx.y * Co) : (void*)((float*)y + blockIdx.y * Co);
    const int n = blockIdx.x / tiles, f0 = (blockIdx.x - n * tiles) * 128;
    const int Wp = W + 2, nch = Ci / 8, cells = flat_cells(W);
    const uint32_t xs = smem_u32(smem), plane = flat_plane(W);
    const uint32_t ws = xs + flat_x_bytes(W, Ci), wstage = flat_w_bytes(Ci, Co), wchunk = row_w_chunk(Co);
    const uint32_t full = smem_u32(&bars[0]), mma_done = full + 8 * kFlatStages;
    const uint32_t ncols = Co <= 32 ? 32u : (Co <= 64 ? 64u : 128u);
    if (tid < Co) bias_s[tid] = bias ? bias[tid] : 0.0f;
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)),
                     "r"(ncols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid == 0) {
        for (int k = 0; k < stages; ++k) {
            mbar_init(full + 8 * k, kWorkers);
            mbar_init(mma_done + 8 * k, 1);
        }
        failed = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = tmem_slot;
    int issued = 0;
    if (warp < kWorkers / 32) {
        const long long img = (long long)n * H * W;
        auto copy_w = [&](int tap) {   // the tap's weights into buffer tap % stages
            const uint32_t dst = ws + (uint32_t)(tap % stages) * wstage;
            const bf16* src = w + (long long)tap * Ci;
            for_groups(tid, Co, nch, [&](int co, int c) {
                cp_async16(dst + c * wchunk + co * 16, src + (long long)co * 9 * Ci + c * 8, 16u);
            });
            mbar_arrive_copies(full + 8 * (tap % stages));
        };
        // cell k of the tile: padded cell f0 + k, row -1 .. H and column -1 .. W of
        // the image (rows past H, behind the last tile, wrap like the rest);
        // landed with the weights of tap 0
        const bf16* src = x + img * csx;
        for_groups(tid, cells, nch, [&](int k, int c) {
            const int id = f0 + k, row = id / Wp;
            const int yy = (row - 1 + H) % H;
            int xx = id - row * Wp - 1;
            xx = xx < 0 ? W - 1 : (xx >= W ? xx - W : xx);
            cp_async16(xs + c * plane + k * 16, src + ((long long)yy * W + xx) * csx + c * 8, 16u);
        });
        bool ok = true;
        for (int t = 0; t < 9 && ok; ++t) {
            if (t >= stages) ok = mbar_wait_phase(mma_done + 8 * (t % stages), t / stages - 1, &failed);
            if (ok) copy_w(t);
        }
        if (ok) ok = mbar_wait_phase(mma_done + 8 * (8 % stages), 8 / stages, &failed);
        asm volatile("cp.async.wait_all;" ::: "memory");
        if (__all_sync(0xffffffffu, ok)) {
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const int f = f0 + 32 * (warp & 3) + lane, row = f / Wp, col = f - row * Wp;
            const bool in = row < H && col < W;
            const long long pix = img + (long long)row * W + col;
            const bool vec = conv_vec<ACT>(y, csy);
            for (int c0 = 16 * (warp >> 2); c0 < Co; c0 += 32) {
                float v[16];
                tc_ld16(tmem + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)c0, v);
                if (in) conv_store16<ACT>(y, pix * csy + c0, v, bias_s + c0, vec);
            }
        }
    } else {
        const uint32_t idesc = tc_idesc_bf16(128, Co);
        const uint32_t el = tc_elect();
        for (int t = 0; t < 9; ++t) {
            const bool ok = mbar_wait_phase(full + 8 * (t % stages), t / stages, &failed);
            if (!__all_sync(0xffffffffu, ok)) break;
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint64_t ad = tc_smem_desc(xs + (uint32_t)((t / 3) * Wp + t % 3) * 16, plane, 128);
            const uint64_t bd = tc_smem_desc(ws + (uint32_t)(t % stages) * wstage, wchunk, 128);
            tc_mma_run(el, tmem, ad, bd, 2 * plane / 16, 2 * wchunk / 16, idesc, nch / 2, t > 0);
            tc_commit(el, mma_done + 8 * (t % stages));
            issued = t + 1;
        }
        // the MMAs still running (on the failure path) end before the tensor
        // memory is freed
        if (issued > 0)
            mbar_wait_bounded(mma_done + 8 * ((issued - 1) % stages), (uint32_t)((issued - 1) / stages) & 1u, kTcPolls);
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(ncols) : "memory");
    if (tid == 0 && failed) atomicExch(err, 1);
}

// partial[chunk, co, tap, ci] = sum over the chunk's pixels p of gy[p, co] x[shift(p, tap), ci];
// one warp per (chunk, tap, 16 output channels, 8 input channels).
constexpr int kChunk = 1024;   // pixels per partial

__global__ void conv_wgrad_kernel(const bf16* __restrict__ x, int csx, const bf16* __restrict__ gy, int csg,
                                  float* __restrict__ partial, long long M, int H, int W, int Ci, int Co) {
    const long long warp = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    const int nco = Co / 16, nci = Ci / 8;
    const long long per_chunk = 9LL * nco * nci;
    const long long nchunks = (M + kChunk - 1) / kChunk;
    if (warp >= nchunks * per_chunk) return;
    const long long chunk = warp / per_chunk;
    int rem = (int)(warp - chunk * per_chunk);
    const int tap = rem / (nco * nci);
    rem -= tap * nco * nci;
    const int co0 = (rem / nci) * 16, ci0 = (rem % nci) * 8;
    const int dy = tap / 3 - 1, dx = tap % 3 - 1;
    float acc[4] = {0.0f, 0.0f, 0.0f, 0.0f};
    const long long pb = chunk * kChunk;
    const long long pe = pb + kChunk < M ? pb + kChunk : M;
    for (long long pk = pb; pk < pe; pk += 16) {
        // k index = pixel pk + kk; pixel counts are multiples of 16, so no tail
        const long long q0 = pk + 2 * t, q1 = q0 + 1, q8 = q0 + 8, q9 = q0 + 9;
        const uint32_t a[4] = {pack_pair(gy + q0 * csg + co0 + g, gy + q1 * csg + co0 + g),
                               pack_pair(gy + q0 * csg + co0 + g + 8, gy + q1 * csg + co0 + g + 8),
                               pack_pair(gy + q8 * csg + co0 + g, gy + q9 * csg + co0 + g),
                               pack_pair(gy + q8 * csg + co0 + g + 8, gy + q9 * csg + co0 + g + 8)};
        const uint32_t b[2] = {pack_pair(x + shift_pixel(q0, H, W, dy, dx) * csx + ci0 + g,
                                         x + shift_pixel(q1, H, W, dy, dx) * csx + ci0 + g),
                               pack_pair(x + shift_pixel(q8, H, W, dy, dx) * csx + ci0 + g,
                                         x + shift_pixel(q9, H, W, dy, dx) * csx + ci0 + g)};
        mma_bf16(acc, a, b);
    }
    float* out = partial + chunk * (long long)Co * 9 * Ci;
    const int ci = ci0 + 2 * t;
    out[((long long)(co0 + g) * 9 + tap) * Ci + ci] = acc[0];
    out[((long long)(co0 + g) * 9 + tap) * Ci + ci + 1] = acc[1];
    out[((long long)(co0 + g + 8) * 9 + tap) * Ci + ci] = acc[2];
    out[((long long)(co0 + g + 8) * 9 + tap) * Ci + ci + 1] = acc[3];
}

// ---------------------------------------------------------------- tcgen05 weight gradient, row march
// gw[co, tap, ci] = sum_p gy[p, co] x[p + d(tap), ci] as GEMMs over pixels
// on the tensor cores, for images whose width is a multiple of 32: per tap
// D_tap (M x N) += A (M x pixels) B (N x pixels)^T, M the channels of the side
// with more of them, N those of the other, K running over pixels.
//
// Both operands are read where they were copied: a row lies in shared memory as
// planes of 8 channels, 16 bytes per pixel, which is the tensor core's
// no-swizzle MN-major layout (core matrices of 8 pixels x 8 channels, plane
// pitch between channel groups, 128 bytes between groups of 8 pixels).  A tap
// is then the x row of its dy started (1 + dx) pixels in: no transposition
// (transposing both operands through registers into K-major buffers took
// 290 us for the 64 -> 32 layer at 8 x 256^2; this takes 81).  Plane pitches are
// odd multiples of 16 bytes, so the 8 groups of a pixel, copied by neighbouring
// threads, fall into different banks.
//
// A CTA takes a segment of P = 64 (or 32) pixels, one tap row dy, a block of at
// most 128 input channels and a chunk of rows.  It marches groups of rows (256
// pixels' worth) through two or three buffers: the waits and the proxy fence of
// the issuing warp are paid once per group.  The three taps accumulate in tensor
// memory over the whole chunk, rows and pixels in order, and are written out
// once, as the CTA's partial; partials are summed in order (deterministic).
// Chunks are cut by wgrad_row_plan: another cut would change the last bits of
// the gradient, and with them, through Adam's normalised step and the bf16
// rounding of the weights, a training run's course.  M is 64 up to 64 channels,
// else 128 (24 against 40 clk per MMA at N = 32): the rows past a side's
// channels read whatever lies behind its planes and are not written out.
constexpr int kWgCn = 128;            // input channels of one CTA at most
constexpr int kWgPixels = 256;        // pixels of a group of rows
constexpr int kWgBuf = 3;             // buffers at most
constexpr size_t kWgSmemMax = 220 * 1024;   // below the 227 KB per CTA less the kernel's static shared memory

__host__ __device__ inline int wg_m(int channels) { return channels <= 64 ? 64 : 128; }
struct WgLayout {
    uint32_t px, pg;        // plane pitches of x and gy
    uint32_t xrow, grow;    // bytes of one row
    uint32_t rows;          // rows of a group
    uint32_t tail;          // the planes of all M rows an operand reads from the last row
};
// P pixels of a segment, Cn input channels and Co output channels of a CTA
__host__ __device__ inline WgLayout wg_layout(int P, int Cn, int Co) {
    WgLayout L;
    L.px = (uint32_t)((P + 2) | 1) * 16;
    L.pg = (uint32_t)(P | 1) * 16;
    L.xrow = (uint32_t)(Cn / 8) * L.px;
    L.grow = (uint32_t)(Co / 8) * L.pg;
    L.rows = kWgPixels / P;
    while (L.rows > 1 && 2 * L.rows * (L.xrow + L.grow) > kWgSmemMax - 24 * 1024) L.rows /= 2;
    L.tail = Cn >= Co ? (uint32_t)(wg_m(Cn) - Cn) / 8 * L.px : (uint32_t)(wg_m(Co) - Co) / 8 * L.pg;
    return L;
}
__host__ __device__ inline size_t wg_bytes(const WgLayout& L, int bufs) {
    return (size_t)bufs * L.rows * (L.xrow + L.grow) + L.tail;
}
__host__ __device__ inline int wg_n(int Cn, int Co) { return Cn >= Co ? Co : Cn; }   // columns of a tap
__host__ __device__ inline uint32_t wg_tmem_cols(int n) {   // three taps of n columns
    const int need = 3 * n;
    return need <= 64 ? 64u : (need <= 128 ? 128u : (need <= 256 ? 256u : 512u));
}

__global__ void __launch_bounds__(kRoleThreads, 3)
conv_wgrad_row_kernel(const bf16* __restrict__ x, int csx, const bf16* __restrict__ gy, int csg,
                      float* __restrict__ partial, int N, int H, int W, int Ci, int Co, int P, int Cn,
                      int rows_per_cta, int bufs, int* err) {
    extern __shared__ __align__(1024) unsigned char smem[];
    __shared__ __align__(8) uint64_t bars[2 * kWgBuf];   // full[buffer], done[buffer]
    __shared__ uint32_t tmem_slot;
    __shared__ int failed;
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;   // warp: uniform
    const int segs = W / P;
    const int nsplit = Ci / Cn;
    const int chunks = (H + rows_per_cta - 1) / rows_per_cta;
    int b = blockIdx.x;
    const int dy = b % 3 - 1;
    b /= 3;
    const int ci0 = (b % nsplit) * Cn;
    b /= nsplit;
    const int chunk = b % chunks;
    b /= chunks;
    const int seg = b % segs, n = b / segs;
    const int y0 = chunk * rows_per_cta;
    const int S = (y0 + rows_per_cta < H ? y0 + rows_per_cta : H) - y0;   // rows of the march
    const int x0 = seg * P;
    const long long pchunk = ((long long)n * segs + seg) * chunks + chunk;
    const WgLayout Lt = wg_layout(P, Cn, Co);
    const int RG = (int)Lt.rows, groups = (S + RG - 1) / RG;
    const bool x_is_a = Cn >= Co;
    // the buffers of the M side lie last, its tail behind them
    const uint32_t sb = smem_u32(smem);
    const uint32_t xb = x_is_a ? sb + (uint32_t)(bufs * RG) * Lt.grow : sb;
    const uint32_t gb = x_is_a ? sb : sb + (uint32_t)(bufs * RG) * Lt.xrow;
    const uint32_t full = smem_u32(&bars[0]), mma_done = full + 8 * kWgBuf;
    const int Nc = wg_n(Cn, Co);
    const uint32_t ncols = wg_tmem_cols(Nc);
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)),
                     "r"(ncols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid == 0) {
        for (int k = 0; k < bufs; ++k) {
            mbar_init(full + 8 * k, kWorkers);
            mbar_init(mma_done + 8 * k, 1);
        }
        failed = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = tmem_slot;
    bool ok = true;
    if (warp < kWorkers / 32) {
        const int nco8 = Co / 8, nci8 = Cn / 8;
        const long long img = (long long)n * H * W;
        int buf = 0, ph = 0, yx = (y0 + dy + H) % H;   // buffer, its use, image row of x
        for (int g = 0; g < groups && ok; ++g) {
            if (g >= bufs) ok = mbar_wait_phase(mma_done + 8 * buf, ph - 1, &failed);
            if (!ok) break;
            const int r0 = g * RG, r1 = r0 + RG < S ? r0 + RG : S;
            for (int q = r0; q < r1; ++q) {
                const bf16* xrow = x + (img + (long long)yx * W) * csx + ci0;
                const uint32_t xd = xb + (uint32_t)(buf * RG + q - r0) * Lt.xrow;
                for_groups(tid, P + 2, nci8, [&](int p, int c) {   // pixels x0 - 1 .. x0 + P (wrapped)
                    int xx = x0 - 1 + p;
                    xx = xx < 0 ? xx + W : (xx >= W ? xx - W : xx);
                    cp_async16(xd + c * Lt.px + p * 16, xrow + (long long)xx * csx + c * 8, 16u);
                });
                const bf16* grow = gy + (img + (long long)(y0 + q) * W + x0) * csg;
                const uint32_t gd = gb + (uint32_t)(buf * RG + q - r0) * Lt.grow;
                for_groups(tid, P, nco8, [&](int p, int c) {
                    cp_async16(gd + c * Lt.pg + p * 16, grow + (long long)p * csg + c * 8, 16u);
                });
                yx = yx + 1 == H ? 0 : yx + 1;
            }
            mbar_arrive_copies(full + 8 * buf);
            if (++buf == bufs) { buf = 0; ++ph; }
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
        ok = __all_sync(0xffffffffu, ok) != 0;
    } else {
        // both operands MN-major (bits 15 and 16)
        const uint32_t idesc = tc_idesc_bf16(wg_m(x_is_a ? Cn : Co), Nc) | (1u << 15) | (1u << 16);
        const uint32_t el = tc_elect();
        const uint64_t x_hi = tc_smem_desc(0, 128, Lt.px), g_hi = tc_smem_desc(0, 128, Lt.pg);
        int buf = 0, ph = 0, last = 0, last_ph = 0;
        bool any = false;
        for (int g = 0; g < groups; ++g) {
            ok = mbar_wait_phase(full + 8 * buf, ph, &failed);
            ok = __all_sync(0xffffffffu, ok) != 0;
            if (!ok) break;
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const int rows = S - g * RG < RG ? S - g * RG : RG;
            for (int q = 0; q < rows; ++q) {
                const uint64_t gd = g_hi + (uint64_t)((gb + (uint32_t)(buf * RG + q) * Lt.grow) >> 4);
                const uint64_t xd0 = x_hi + (uint64_t)((xb + (uint32_t)(buf * RG + q) * Lt.xrow) >> 4);
#pragma unroll
                for (int dx = 0; dx < 3; ++dx) {
                    const uint64_t xd = xd0 + (uint64_t)dx;
                    tc_mma_run(el, tmem + (uint32_t)(dx * Nc), x_is_a ? xd : gd, x_is_a ? gd : xd, 16, 16, idesc, P / 16,
                               g + q > 0);
                }
            }
            tc_commit(el, mma_done + 8 * buf);
            any = true;
            last = buf;
            last_ph = ph;
            if (++buf == bufs) { buf = 0; ++ph; }
        }
        // the MMAs still running end before the accumulators are read or (on the
        // failure path) the tensor memory is freed
        if (any) ok = mbar_wait_bounded(mma_done + 8 * last, (uint32_t)last_ph & 1u, kTcPolls) && ok;
        if (!ok) failed = 1;
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (!failed && warp < 4) {
        // channel of the M side: row m of an M = 128 accumulator is lane m, of an
        // M = 64 one lane 32 (m / 16) + m % 16
        const bool half = wg_m(x_is_a ? Cn : Co) == 64;
        const int m = half ? (lane < 16 ? 16 * warp + lane : 128) : 32 * warp + lane;
        const int K9 = 9 * Ci;
        float* out = partial + pchunk * Co * (long long)K9;
        for (int t = 0; t < 3; ++t) {
            const int tap = (dy + 1) * 3 + t;
            for (int c0 = 0; c0 < Nc; c0 += 16) {
                float v[16];
                tc_ld16(tmem + ((uint32_t)(32 * warp) << 16) + (uint32_t)(t * Nc + c0), v);
                if (x_is_a) {
                    if (m < Cn) {
#pragma unroll
                        for (int k = 0; k < 16; ++k) out[(long long)(c0 + k) * K9 + tap * Ci + ci0 + m] = v[k];
                    }
                } else if (m < Co) {
                    float* o = out + (long long)m * K9 + tap * Ci + ci0 + c0;
#pragma unroll
                    for (int k = 0; k < 16; k += 4)
                        *reinterpret_cast<float4*>(o + k) = make_float4(v[k], v[k + 1], v[k + 2], v[k + 3]);
                }
            }
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(ncols) : "memory");
    if (tid == 0 && failed) atomicExch(err, 1);
}

// gw[k] = sum over chunks of partial[chunk, k], in chunk order, 16 loads in flight.
// Blocks of one warp while those are few (blocks of 256 threads that waited for
// each load: 18 blocks and 10.3 us for the 4608 values of the 16 -> 32 layer, 5.6
// now), of 256 threads from 2^16 values on (9216 blocks of one warp for the
// 256 -> 128 layer at 8^2: the weight gradient 18.5 us, 14.4 with 1152).
template <int T>
__global__ void __launch_bounds__(T)
sum_chunks_kernel(const float* __restrict__ partial, long long nchunks, long long K, float* __restrict__ gw) {
    const long long k = (long long)blockIdx.x * T + threadIdx.x;
    if (k >= K) return;
    const float* p = partial + k;
    float s = 0.0f;
    long long c = 0;
    for (; c + 16 <= nchunks; c += 16) {
        float v[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) v[i] = p[(c + i) * K];
#pragma unroll
        for (int i = 0; i < 16; ++i) s += v[i];
    }
    for (; c < nchunks; ++c) s += p[c * K];
    gw[k] = s;
}

// wt[ci, 8 - tap, co] = w[co, tap, ci]: the weights of the input-gradient convolution
__global__ void weight_flip_kernel(const bf16* __restrict__ w, bf16* __restrict__ wt, int Ci, int Co) {
    const long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= (long long)Co * 9 * Ci) return;
    const int ci = (int)(k % Ci);
    const int tap = (int)((k / Ci) % 9);
    const int co = (int)(k / (9LL * Ci));
    wt[((long long)ci * 9 + (8 - tap)) * Co + co] = w[k];
}

}  // namespace

namespace {

constexpr int kThreads = 256;
inline unsigned blocks(long long n) { return (unsigned)((n + kThreads - 1) / kThreads); }

// y (bf16) = max(a, 0), channel slices
__global__ void relu_kernel(const float* __restrict__ a, int csa, bf16* __restrict__ y, int csy, long long npix,
                            int C) {
    const long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= npix * C) return;
    const long long p = k / C;
    const int c = (int)(k - p * C);
    y[p * csy + c] = __float2bfloat16_rn(fmaxf(a[p * csa + c], 0.0f));
}

// ga = g where a > 0 else 0 (FP32), and its bf16 copy (optional)
__global__ void relu_bwd_kernel(const float* __restrict__ g, int csg, const float* __restrict__ a, int csa,
                                float* __restrict__ ga, bf16* __restrict__ ga16, long long npix, int C) {
    const long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= npix * C) return;
    const long long p = k / C;
    const int c = (int)(k - p * C);
    const float v = a[p * csa + c] > 0.0f ? g[p * csg + c] : 0.0f;
    ga[k] = v;
    if (ga16) ga16[k] = __float2bfloat16_rn(v);
}

__global__ void to_bf16_kernel(const float* __restrict__ a, int csa, bf16* __restrict__ y, int csy, long long npix,
                               int C) {
    const long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= npix * C) return;
    const long long p = k / C;
    const int c = (int)(k - p * C);
    y[p * csy + c] = __float2bfloat16_rn(a[p * csa + c]);
}

// out = a + b on channel slices
__global__ void add_kernel(const float* __restrict__ a, int csa, const float* __restrict__ b, int csb,
                           float* __restrict__ out, int cso, long long npix, int C) {
    const long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= npix * C) return;
    const long long p = k / C;
    const int c = (int)(k - p * C);
    out[p * cso + c] = a[p * csa + c] + b[p * csb + c];
}

// f x f average pooling, bf16 -> bf16; (N, H, W) the fine grid
__global__ void pool_kernel(const bf16* __restrict__ x, int csx, bf16* __restrict__ y, int csy, int N, int H, int W,
                            int C, int f) {
    const int Hc = H / f, Wc = W / f;
    const long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= (long long)N * Hc * Wc * C) return;
    const int c = (int)(k % C);
    const long long q = k / C;
    const int xc = (int)(q % Wc), yc = (int)((q / Wc) % Hc);
    const long long n = q / ((long long)Hc * Wc);
    float s = 0.0f;
    for (int i = 0; i < f; ++i)
        for (int j = 0; j < f; ++j) {
            const long long p = (n * H + yc * f + i) * W + xc * f + j;
            s += __bfloat162float(x[p * csx + c]);
        }
    y[q * csy + c] = __float2bfloat16_rn(s / (float)(f * f));
}

// 2 x 2 pooling and upsampling on 8 channels (16 bytes) per thread: the
// per-element kernels spend their time on 64-bit index divisions (8 x 256^2 x
// 32 channels: pooling 53 us, upsampling 121 us; these 8 and 11).  The sums are formed in the
// order of pool_kernel.
__device__ __forceinline__ void unpack8(uint4 q, float (&v)[8]) {
    const uint32_t u[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        v[2 * i] = __uint_as_float(u[i] << 16);
        v[2 * i + 1] = __uint_as_float(u[i] & 0xffff0000u);
    }
}

__global__ void pool2_kernel(const bf16* __restrict__ x, int csx, bf16* __restrict__ y, int csy, int nrows, int Wc,
                             int C8) {
    // blockIdx.y: coarse row over all images; its two fine rows are 2 r, 2 r + 1
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= Wc * C8) return;
    const int xc = k / C8, c = (k - xc * C8) * 8;
    for (int r = blockIdx.y; r < nrows; r += gridDim.y) {
        const bf16* p = x + ((long long)(2 * r) * (2 * Wc) + 2 * xc) * csx + c;
        const bf16* q = p + (long long)(2 * Wc) * csx;
        float a[8], b[8], d[8], e[8];
        unpack8(*reinterpret_cast<const uint4*>(p), a);
        unpack8(*reinterpret_cast<const uint4*>(p + csx), b);
        unpack8(*reinterpret_cast<const uint4*>(q), d);
        unpack8(*reinterpret_cast<const uint4*>(q + csx), e);
        __nv_bfloat162 o[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            float s[2];
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                const int m = 2 * i + j;
                s[j] = (((a[m] + b[m]) + d[m]) + e[m]) * 0.25f;
            }
            o[i] = __floats2bfloat162_rn(s[0], s[1]);
        }
        *reinterpret_cast<uint4*>(y + ((long long)r * Wc + xc) * csy + c) = *reinterpret_cast<uint4*>(o);
    }
}

__global__ void upsample2_kernel(const bf16* __restrict__ x, int csx, bf16* __restrict__ y, int csy, int nrows, int Wc,
                                 int C8) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= Wc * C8) return;
    const int xc = k / C8, c = (k - xc * C8) * 8;
    for (int r = blockIdx.y; r < nrows; r += gridDim.y) {
        const uint4 v = *reinterpret_cast<const uint4*>(x + ((long long)r * Wc + xc) * csx + c);
        bf16* p = y + ((long long)(2 * r) * (2 * Wc) + 2 * xc) * csy + c;
        bf16* q = p + (long long)(2 * Wc) * csy;
        *reinterpret_cast<uint4*>(p) = v;
        *reinterpret_cast<uint4*>(p + csy) = v;
        *reinterpret_cast<uint4*>(q) = v;
        *reinterpret_cast<uint4*>(q + csy) = v;
    }
}

// gx[fine] = g[coarse] / f^2
__global__ void pool_bwd_kernel(const float* __restrict__ g, int csg, float* __restrict__ gx, int csx, int N, int H,
                                int W, int C, int f) {
    const long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= (long long)N * H * W * C) return;
    const int c = (int)(k % C);
    const long long p = k / C;
    const int x = (int)(p % W), y = (int)((p / W) % H);
    const long long n = p / ((long long)H * W);
    const int Hc = H / f, Wc = W / f;
    const long long q = (n * Hc + y / f) * Wc + x / f;
    gx[p * csx + c] = g[q * csg + c] / (float)(f * f);
}

// nearest upsampling by f, bf16 -> bf16; (N, H, W) the fine grid
__global__ void upsample_kernel(const bf16* __restrict__ x, int csx, bf16* __restrict__ y, int csy, int N, int H,
                                int W, int C, int f) {
    const long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= (long long)N * H * W * C) return;
    const int c = (int)(k % C);
    const long long p = k / C;
    const int xx = (int)(p % W), yy = (int)((p / W) % H);
    const long long n = p / ((long long)H * W);
    const int Hc = H / f, Wc = W / f;
    const long long q = (n * Hc + yy / f) * Wc + xx / f;
    y[p * csy + c] = x[q * csx + c];
}

// gx[coarse] = sum of g over the f x f block
__global__ void upsample_bwd_kernel(const float* __restrict__ g, int csg, float* __restrict__ gx, int csx, int N,
                                    int H, int W, int C, int f) {
    const int Hc = H / f, Wc = W / f;
    const long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= (long long)N * Hc * Wc * C) return;
    const int c = (int)(k % C);
    const long long q = k / C;
    const int xc = (int)(q % Wc), yc = (int)((q / Wc) % Hc);
    const long long n = q / ((long long)Hc * Wc);
    float s = 0.0f;
    for (int i = 0; i < f; ++i)
        for (int j = 0; j < f; ++j) {
            const long long p = (n * H + yc * f + i) * W + xc * f + j;
            s += g[p * csg + c];
        }
    gx[q * csx + c] = s;
}

// per-block partial sums of column c of g (rows = pixels), fixed order
__global__ void colsum_partial_kernel(const float* __restrict__ g, int csg, long long npix, int C,
                                      float* __restrict__ part) {
    __shared__ float sh[kThreads];
    const int c = blockIdx.y;
    float s = 0.0f;
    for (long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x; p < npix; p += (long long)gridDim.x * blockDim.x)
        s += g[p * csg + c];
    sh[threadIdx.x] = s;
    __syncthreads();
    for (int o = kThreads / 2; o > 0; o >>= 1) {
        if (threadIdx.x < o) sh[threadIdx.x] += sh[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) part[(long long)c * gridDim.x + blockIdx.x] = sh[0];
}

__global__ void colsum_finish_kernel(const float* __restrict__ part, int nb, int C, float* __restrict__ out) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= C) return;
    float s = 0.0f;
    for (int b = 0; b < nb; ++b) s += part[(long long)c * nb + b];
    out[c] = s;
}

// Gradient through a layer's ReLU, fused with what feeds it and with what reads
// it: v = act > 0 ? gradient : 0 as bf16 (the operand of the two gradient
// convolutions), and the bias gradient's block partials from the FP32 v.  The
// gradient of the activation is g (MODE 0), the sum of g over the 2 x 2 fine
// pixels of an upsampling (MODE 1), or g plus a quarter of the pooled path's
// gradient gp (MODE 2); MODE 3 only sums g.  One pass over memory where the
// separate kernels (pooling or upsampling backward, addition, ReLU, column sums)
// took up to seven and an FP32 copy of v in between (the 8 x 256^2 x 32 level:
// 342 us before, 57 now).  A thread takes four channels of two pixels in 256; the sums
// are those of colsum_partial_kernel, in its order (its one channel per block
// reads 4 of every 4 C bytes: 63 us at that level).  H x W the layer's own size.
constexpr int kGradThreads = 512;    // 128 pixels x 16 channels
template <int MODE>
__global__ void __launch_bounds__(kGradThreads)
relu_grad_kernel(const float* __restrict__ g, int csg, const float* __restrict__ gp, int csp,
                 const bf16* __restrict__ act, int csa, bf16* __restrict__ out, int W, int npix, int C,
                 float* __restrict__ part) {
    __shared__ float4 sh[256][4];
    const int quad = threadIdx.x & 3, c = blockIdx.y * 16 + quad * 4, lane = threadIdx.x >> 2;
    float4 sum[2] = {};
    for (int base = blockIdx.x * 256; base < npix && c < C; base += gridDim.x * 256) {
        float4 v[2];
        uint2 m[2];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int p = base + lane + 128 * u;
            v[u] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            if (p >= npix) continue;
            if constexpr (MODE == 0 || MODE == 3) {
                v[u] = *reinterpret_cast<const float4*>(g + (long long)p * csg + c);
            } else {
                const int row = p / W, x = p - row * W;     // row over all images
                if constexpr (MODE == 1) {
                    const float* q = g + ((long long)(2 * row) * (2 * W) + 2 * x) * csg + c;
                    const float4 a = *reinterpret_cast<const float4*>(q);
                    const float4 b = *reinterpret_cast<const float4*>(q + csg);
                    q += (long long)(2 * W) * csg;
                    const float4 d = *reinterpret_cast<const float4*>(q);
                    const float4 e = *reinterpret_cast<const float4*>(q + csg);
                    v[u] = make_float4(((a.x + b.x) + d.x) + e.x, ((a.y + b.y) + d.y) + e.y, ((a.z + b.z) + d.z) + e.z,
                                       ((a.w + b.w) + d.w) + e.w);
                } else {
                    const float4 a = *reinterpret_cast<const float4*>(g + (long long)p * csg + c);
                    const float4 b = *reinterpret_cast<const float4*>(
                        gp + ((long long)(row >> 1) * (W >> 1) + (x >> 1)) * csp + c);
                    v[u] = make_float4(a.x + b.x * 0.25f, a.y + b.y * 0.25f, a.z + b.z * 0.25f, a.w + b.w * 0.25f);
                }
            }
            if constexpr (MODE != 3) m[u] = *reinterpret_cast<const uint2*>(act + (long long)p * csa + c);
        }
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int p = base + lane + 128 * u;
            if (p >= npix) continue;
            if constexpr (MODE != 3) {
                v[u].x = __uint_as_float(m[u].x << 16) > 0.0f ? v[u].x : 0.0f;
                v[u].y = __uint_as_float(m[u].x & 0xffff0000u) > 0.0f ? v[u].y : 0.0f;
                v[u].z = __uint_as_float(m[u].y << 16) > 0.0f ? v[u].z : 0.0f;
                v[u].w = __uint_as_float(m[u].y & 0xffff0000u) > 0.0f ? v[u].w : 0.0f;
                __nv_bfloat162 o[2] = {__floats2bfloat162_rn(v[u].x, v[u].y), __floats2bfloat162_rn(v[u].z, v[u].w)};
                *reinterpret_cast<uint2*>(out + (long long)p * C + c) = *reinterpret_cast<uint2*>(o);
            }
            sum[u].x += v[u].x; sum[u].y += v[u].y; sum[u].z += v[u].z; sum[u].w += v[u].w;
        }
    }
    sh[lane][quad] = sum[0];
    sh[lane + 128][quad] = sum[1];
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
        if (lane < o) {
            float4& a = sh[lane][quad];
            const float4 b = sh[lane + o][quad];
            a.x += b.x; a.y += b.y; a.z += b.z; a.w += b.w;
        }
        __syncthreads();
    }
    if (lane == 0 && c < C) *reinterpret_cast<float4*>(part + (long long)blockIdx.x * C + c) = sh[0][quad];
}

// Sum of v(0) .. v(n - 1) in order, 16 loads in flight; the last group too (loads
// one after the other, 15 of them, cost 2 to 4 us where n is 63 instead of 64).
template <typename F>
__device__ __forceinline__ float ordered_sum(int n, F&& v) {
    float s = 0.0f;
    for (int b = 0; b < n; b += 16) {
        float t[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) t[i] = b + i < n ? v(b + i) : 0.0f;
#pragma unroll
        for (int i = 0; i < 16; ++i)
            if (b + i < n) s += t[i];
    }
    return s;
}

// out[c] = sum of part[b][c] over the blocks, in block order; channels past C of
// `pad` are set to zero
__global__ void channel_finish_kernel(const float* __restrict__ part, int nb, int C, int pad, float* __restrict__ out) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= pad) return;
    out[c] = c < C ? ordered_sum(nb, [&](int b) { return part[(long long)b * C + c]; }) : 0.0f;
}

// Loss of out = x + delta against t over four channels, its gradient in FP32 (g4)
// and as the bf16 operand of the output layer's gradient convolutions (16
// channels, the padded ones zero): one thread per pixel.  part: the block's FP64
// loss sum.
__global__ void __launch_bounds__(kThreads)
mse_grad_kernel(const float4* __restrict__ x, const float* __restrict__ delta, const float* __restrict__ t, bool t_vec,
                bf16* __restrict__ g16, float4* __restrict__ g4, int npix, double inv, double* __restrict__ part) {
    __shared__ double sh[kThreads];
    double s = 0.0;
    for (int p = blockIdx.x * kThreads + threadIdx.x; p < npix; p += gridDim.x * kThreads) {
        const float4 a = x[p], d = *reinterpret_cast<const float4*>(delta + (long long)p * 16);
        const float* tp = t + (long long)p * 4;    // the caller's array: any alignment
        const float4 b = t_vec ? *reinterpret_cast<const float4*>(tp) : make_float4(tp[0], tp[1], tp[2], tp[3]);
        const double e[4] = {(double)a.x + (double)d.x - (double)b.x, (double)a.y + (double)d.y - (double)b.y,
                             (double)a.z + (double)d.z - (double)b.z, (double)a.w + (double)d.w - (double)b.w};
        float g[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            s += e[k] * e[k];
            g[k] = (float)(2.0 * e[k] * inv);
        }
        g4[p] = make_float4(g[0], g[1], g[2], g[3]);
        __nv_bfloat162 o[4] = {__floats2bfloat162_rn(g[0], g[1]), __floats2bfloat162_rn(g[2], g[3]),
                               __floats2bfloat162_rn(0.0f, 0.0f), __floats2bfloat162_rn(0.0f, 0.0f)};
        uint4* q = reinterpret_cast<uint4*>(g16 + (long long)p * 16);
        q[0] = *reinterpret_cast<uint4*>(o);
        q[1] = make_uint4(0u, 0u, 0u, 0u);
    }
    sh[threadIdx.x] = s;
    __syncthreads();
    for (int o = kThreads / 2; o > 0; o >>= 1) {
        if (threadIdx.x < o) sh[threadIdx.x] += sh[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) part[blockIdx.x] = sh[0];
}

// the loss, and the 16 entries of the output layer's bias gradient (4 real) from
// the block partials of g4
__global__ void mse_grad_finish_kernel(const double* __restrict__ part, int nb, const float* __restrict__ gpart, int ngb,
                                       double inv_count, double* __restrict__ loss, float* __restrict__ gb) {
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (w == 0) {
        double s = 0.0;
        for (int b = lane; b < nb; b += 32) s += part[b];
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (lane == 0) loss[0] = s * inv_count;
    } else if (lane < 16) {
        gb[lane] = lane < 4 ? ordered_sum(ngb, [&](int b) { return gpart[4 * b + lane]; }) : 0.0f;
    }
}

// out = x + delta on the first C channels; g = 2 (out - t) / (npix C) (zero beyond C up to csd);
// block partials of sum (out - t)^2 in FP64
__global__ void mse_kernel(const float* __restrict__ x, int csx, const float* __restrict__ delta, int csd,
                           const float* __restrict__ t, int cst, float* __restrict__ g, long long npix, int C,
                           double* __restrict__ part) {
    __shared__ double sh[kThreads];
    double s = 0.0;
    const double inv = 1.0 / ((double)npix * C);
    for (long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x; k < npix * csd;
         k += (long long)gridDim.x * blockDim.x) {
        const long long p = k / csd;
        const int c = (int)(k - p * csd);
        float gv = 0.0f;
        if (c < C) {
            const double e = (double)x[p * csx + c] + (double)delta[k] - (double)t[p * cst + c];
            s += e * e;
            gv = (float)(2.0 * e * inv);
        }
        g[k] = gv;
    }
    sh[threadIdx.x] = s;
    __syncthreads();
    for (int o = kThreads / 2; o > 0; o >>= 1) {
        if (threadIdx.x < o) sh[threadIdx.x] += sh[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) part[blockIdx.x] = sh[0];
}

// Sum of column k of nb rows of `width` partials by the calling warp, fixed
// order, in every lane (a chain of 256 FP64 additions of 65 clk took 8 us).
__device__ __forceinline__ double warp_column(const double* __restrict__ part, int nb, int width, int k) {
    double s = 0.0;
    for (int b = threadIdx.x & 31; b < nb; b += 32) s += part[b * width + k];
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    return s;
}

__global__ void mse_finish_kernel(const double* __restrict__ part, int nb, double inv_count, double* out) {
    const double s = warp_column(part, nb, 1, 0);
    if (threadIdx.x == 0) out[0] = s * inv_count;
}

// Adam on FP32 master values, with the bf16 copy used by the convolutions
__global__ void adam_kernel(float* __restrict__ w, float* __restrict__ m, float* __restrict__ v,
                            const float* __restrict__ g, long long n, float lr, float b1, float b2, float eps,
                            float c1, float c2, bf16* __restrict__ w16) {
    const long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    const float gk = g[k];
    const float mk = b1 * m[k] + (1.0f - b1) * gk;
    const float vk = b2 * v[k] + (1.0f - b2) * gk * gk;
    m[k] = mk;
    v[k] = vk;
    const float wk = w[k] - lr * (mk / c1) / (sqrtf(vk / c2) + eps);
    w[k] = wk;
    if (w16) w16[k] = __float2bfloat16_rn(wk);
}

// Adam on every layer of a network at once: the weights (with their bf16 copy
// and its flipped form, the operand of the input-gradient convolution) and the
// biases.  blockIdx.y is the layer.
constexpr int kMaxLayers = 16;
struct AdamLayers {
    lbm_sg_layer l[kMaxLayers];
};
__device__ __forceinline__ float adam_one(float* w, float* m, float* v, const float* g, long long k, float lr, float b1,
                                          float b2, float eps, float c1, float c2) {
    const float gk = g[k];
    const float mk = b1 * m[k] + (1.0f - b1) * gk;
    const float vk = b2 * v[k] + (1.0f - b2) * gk * gk;
    m[k] = mk;
    v[k] = vk;
    const float wk = w[k] - lr * (mk / c1) / (sqrtf(vk / c2) + eps);
    w[k] = wk;
    return wk;
}
__global__ void adam_layers_kernel(const __grid_constant__ AdamLayers a, float lr, float b1, float b2, float eps,
                                   float c1, float c2) {
    const lbm_sg_layer& l = a.l[blockIdx.y];
    const int n = l.co * 9 * l.ci;
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < n + l.co; k += gridDim.x * blockDim.x) {
        if (k < n) {
            const bf16 h = __float2bfloat16_rn(adam_one(l.w, l.mw, l.vw, l.gw, k, lr, b1, b2, eps, c1, c2));
            ((bf16*)l.w16)[k] = h;
            const int row = k / l.ci, ci = k - row * l.ci, co = row / 9, tap = row - co * 9;
            ((bf16*)l.wt)[((long long)ci * 9 + (8 - tap)) * l.co + co] = h;
        } else {
            adam_one(l.b, l.mb, l.vb, l.gb, k - n, lr, b1, b2, eps, c1, c2);
        }
    }
}

// LB fields (FP64, x fastest: phi, rho u_x, rho u_y, P) -> normalised channels-last input: channel c = field c / scale c
__global__ void pack_kernel(const double* __restrict__ f0, const double* __restrict__ f1, const double* __restrict__ f2,
                            const double* __restrict__ f3, double s0, double s1, double s2, double s3,
                            float* __restrict__ x32, int cs32, bf16* __restrict__ x16, int cs16, long long npix) {
    const long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= npix) return;
    const float v[4] = {(float)(f0[p] / s0), (float)(f1[p] / s1), (float)(f2[p] / s2), (float)(f3[p] / s3)};
    for (int c = 0; c < 4; ++c) x32[p * cs32 + c] = v[c];
    for (int c = 0; c < cs16; ++c) x16[p * cs16 + c] = __float2bfloat16_rn(c < 4 ? v[c] : 0.0f);
}

// (phi, rho u_x, rho u_y, P) = (x + delta) * scale, then u = rho u / rho(phi)
// with phi clipped to [0, 1] inside rho only (a predicted phi a little below
// 0 in the light phase must not make the density vanish or turn negative)
__global__ void unpack_kernel(const float* __restrict__ x32, int cs32, const float* __restrict__ delta, int csd,
                              double* __restrict__ f0, double* __restrict__ f1, double* __restrict__ f2,
                              double* __restrict__ f3, double s0, double s1, double s2, double s3, double rho_L,
                              double rho_dif, const double* __restrict__ phi_rho, long long npix) {
    const long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= npix) return;
    double v[4];
    const double s[4] = {s0, s1, s2, s3};
    for (int c = 0; c < 4; ++c) v[c] = ((double)x32[p * cs32 + c] + (double)delta[p * csd + c]) * s[c];
    const double pr = phi_rho ? phi_rho[p] : v[0];
    const double pc = pr < 0.0 ? 0.0 : (pr > 1.0 ? 1.0 : pr);
    const double rho = rho_L + pc * rho_dif;
    f0[p] = v[0];
    f1[p] = v[1] / rho;
    f2[p] = v[2] / rho;
    f3[p] = v[3];
}

__global__ void shift_kernel(double* __restrict__ a, long long n, double s) {
    const long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (k < n) a[k] += s;
}

// block partials of sum (a - b)^2 and sum a^2 (FP64, fixed order)
__global__ void residual_partial_kernel(const double* __restrict__ a, const double* __restrict__ b, long long n,
                                        double* __restrict__ part) {
    __shared__ double s0[kThreads], s1[kThreads];
    double d2 = 0.0, a2 = 0.0;
    for (long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += (long long)gridDim.x * blockDim.x) {
        const double d = a[k] - b[k];
        d2 += d * d;
        a2 += a[k] * a[k];
    }
    s0[threadIdx.x] = d2;
    s1[threadIdx.x] = a2;
    __syncthreads();
    for (int o = kThreads / 2; o > 0; o >>= 1) {
        if (threadIdx.x < o) { s0[threadIdx.x] += s0[threadIdx.x + o]; s1[threadIdx.x] += s1[threadIdx.x + o]; }
        __syncthreads();
    }
    if (threadIdx.x == 0) { part[2 * blockIdx.x] = s0[0]; part[2 * blockIdx.x + 1] = s1[0]; }
}

__global__ void residual_finish_kernel(const double* __restrict__ part, int nb, double* __restrict__ out) {
    const double v = warp_column(part, nb, 2, threadIdx.x >> 5);   // two warps
    if ((threadIdx.x & 31) == 0) out[threadIdx.x >> 5] = v;
}

// block partials of (sum P, count) over the bulk heavy phase (phi >= 1 - d)
// and over the bulk light phase (phi <= d), FP64, fixed order
__global__ void phase_pressure_partial_kernel(const double* __restrict__ phi, const double* __restrict__ P,
                                              long long n, double d, double* __restrict__ part) {
    __shared__ double sh[4][kThreads];
    double a[4] = {0.0, 0.0, 0.0, 0.0};
    for (long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += (long long)gridDim.x * blockDim.x) {
        const double f = phi[k];
        if (f >= 1.0 - d) { a[0] += P[k]; a[1] += 1.0; }
        if (f <= d) { a[2] += P[k]; a[3] += 1.0; }
    }
    for (int j = 0; j < 4; ++j) sh[j][threadIdx.x] = a[j];
    __syncthreads();
    for (int o = kThreads / 2; o > 0; o >>= 1) {
        if (threadIdx.x < o)
            for (int j = 0; j < 4; ++j) sh[j][threadIdx.x] += sh[j][threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0)
        for (int j = 0; j < 4; ++j) part[4 * blockIdx.x + j] = sh[j][0];
}

__global__ void phase_pressure_finish_kernel(const double* __restrict__ part, int nb, double* __restrict__ out) {
    __shared__ double a[4];
    const double v = warp_column(part, nb, 4, threadIdx.x >> 5);   // four warps
    if ((threadIdx.x & 31) == 0) a[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x != 0) return;
    out[0] = a[1] > 0.0 ? a[0] / a[1] : 0.0;
    out[1] = a[3] > 0.0 ? a[2] / a[3] : 0.0;
    out[2] = a[1];
    out[3] = a[3];
}

// phi <- clip(phi0 + m (phi - phi0), 0, 1), m = 4 phi0 (1 - phi0): the
// predicted change of phi kept inside the interface band of the start and
// none in the bulk phases; block partials of sum phi0, sum phi, sum 4 phi (1 - phi)
__global__ void phi_project_kernel(double* __restrict__ phi, const double* __restrict__ phi0, long long n,
                                   double* __restrict__ part) {
    __shared__ double s0[kThreads], s1[kThreads], s2[kThreads];
    double a0 = 0.0, a1 = 0.0, a2 = 0.0;
    for (long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += (long long)gridDim.x * blockDim.x) {
        const double f0 = phi0[k];
        const double m = 4.0 * f0 * (1.0 - f0);
        double f = f0 + (m > 0.0 ? m : 0.0) * (phi[k] - f0);
        f = f < 0.0 ? 0.0 : (f > 1.0 ? 1.0 : f);
        phi[k] = f;
        a0 += f0;
        a1 += f;
        a2 += 4.0 * f * (1.0 - f);
    }
    s0[threadIdx.x] = a0;
    s1[threadIdx.x] = a1;
    s2[threadIdx.x] = a2;
    __syncthreads();
    for (int o = kThreads / 2; o > 0; o >>= 1) {
        if (threadIdx.x < o) {
            s0[threadIdx.x] += s0[threadIdx.x + o];
            s1[threadIdx.x] += s1[threadIdx.x + o];
            s2[threadIdx.x] += s2[threadIdx.x + o];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        part[3 * blockIdx.x] = s0[0];
        part[3 * blockIdx.x + 1] = s1[0];
        part[3 * blockIdx.x + 2] = s2[0];
    }
}

// c = (sum phi0 - sum phi) / sum 4 phi (1 - phi), into part[3 nb]
__global__ void phi_project_finish_kernel(double* __restrict__ part, int nb) {
    __shared__ double a[3];
    const double v = warp_column(part, nb, 3, threadIdx.x >> 5);   // three warps
    if ((threadIdx.x & 31) == 0) a[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x == 0) part[3 * nb] = a[2] > 0.0 ? (a[0] - a[1]) / a[2] : 0.0;
}

// phi += c 4 phi (1 - phi): the total of phi0 restored by moving the interfaces
__global__ void phi_restore_kernel(double* __restrict__ phi, long long n, const double* __restrict__ c) {
    const long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    const double f = phi[k];
    phi[k] = f + c[0] * 4.0 * f * (1.0 - f);
}

// b = a + k lap(a), five-point Laplacian, periodic in each H x W image
__global__ void smooth_kernel(const double* __restrict__ a, double* __restrict__ b, int N, int H, int W, double k) {
    const long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= (long long)N * H * W) return;
    const int x = (int)(p % W), y = (int)((p / W) % H);
    const long long base = p - (long long)y * W - x;
    const int xm = x == 0 ? W - 1 : x - 1, xp = x == W - 1 ? 0 : x + 1;
    const int ym = y == 0 ? H - 1 : y - 1, yp = y == H - 1 ? 0 : y + 1;
    const double c = a[p];
    const double lap = a[base + (long long)y * W + xm] + a[base + (long long)y * W + xp] + a[base + (long long)ym * W + x] +
                       a[base + (long long)yp * W + x] - 4.0 * c;
    b[p] = c + k * lap;
}

// Shared memory of one SM of the current device (looked up once per device;
// 228 KB, GB300's, if the query fails).
size_t sm_shared_bytes() {
    static int cached[64] = {};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) {
        cudaGetLastError();
        return 228 * 1024;
    }
    if (cached[dev] == 0) {
        int v = 0;
        if (cudaDeviceGetAttribute(&v, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev) != cudaSuccess || v <= 0) {
            cudaGetLastError();
            v = 228 * 1024;
        }
        cached[dev] = v;
    }
    return (size_t)cached[dev];
}

// Dynamic shared memory of a row-march launch: its need, raised if necessary
// so that no more CTAs fit on an SM than its 512 tensor-memory columns serve
// at once (each CTA holds row_tmem_cols(Co) of them for its whole life).
size_t conv_row_launch_smem(size_t need, int Co) {
    const int per_sm = 512 / (int)row_tmem_cols(Co);
    const size_t floor_bytes = sm_shared_bytes() / (size_t)(per_sm + 1) + 1;
    return need > floor_bytes ? need : floor_bytes;
}

// The attribute for large dynamic shared memory of a convolution kernel, once
// per device.
template <typename K>
cudaError_t large_smem(K kernel, bool (&done)[64], int dev) {
    if (dev < 0 || dev >= 64 || !done[dev]) {
        cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kRowSmemMax);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout,
                                     (int)cudaSharedmemCarveoutMaxShared);
        if (e != cudaSuccess) return e;
        if (dev >= 0 && dev < 64) done[dev] = true;
    }
    return cudaSuccess;
}

// Segment width of the weight-gradient row march (0: the width allows none)
// and the input channels of one CTA.
inline int wg_segment(int W) { return W % 64 == 0 ? 64 : (W % 32 == 0 ? 32 : 0); }
inline int wg_block(int Ci) { return Ci <= kWgCn ? Ci : kWgCn; }

// Row chunks of the weight-gradient row march on the current device: rows
// per CTA and chunks per column (0 rows: the march does not apply to these
// sizes).  As many chunks as keep 3 tap rows x channel blocks x N x W / P segments
// x chunks CTAs within what an SM would hold of CTAs with two row buffers in
// both operand layouts (`cta` bytes) and 3 Cn columns of tensor memory.  The
// kernel needs less than that, but the cut fixes the order of the sums.
cudaError_t wgrad_row_plan(int N, int H, int W, int Ci, int Co, int* rows, int* chunks) {
    *rows = 0;
    *chunks = 0;
    const int P = wg_segment(W), Cn = wg_block(Ci);
    if (P == 0 || Ci % Cn || Co > 128 || Ci % 16 || Co % 16 || H < 1) return cudaSuccess;
    const size_t cta = 2 * ((size_t)P * (2 * Co + 16) + (size_t)(P + 2) * (2 * Cn + 16)) +
                       2 * (size_t)(P / 8) * (128 + 3 * (size_t)Cn) * 16;
    if (cta > kWgSmemMax || wg_bytes(wg_layout(P, Cn, Co), 2) > kWgSmemMax) return cudaSuccess;
    static bool attr_set[64] = {};
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = large_smem(conv_wgrad_row_kernel, attr_set, dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    const int by_tmem = 512 / (int)(3 * Cn <= 64 ? 64 : (3 * Cn <= 128 ? 128 : (3 * Cn <= 256 ? 256 : 512)));
    const size_t least = sm_shared_bytes() / (size_t)(by_tmem + 1) + 1;
    int occ = (int)(sm_shared_bytes() / ((cta > least ? cta : least) + 1024));
    if (occ > by_tmem) occ = by_tmem;
    const long long slots = (long long)sms * (occ > 0 ? occ : 1);
    const long long cols = 3LL * (Ci / Cn) * N * (W / P);
    long long c = slots / cols;
    if (c < 1) c = 1;
    if (c > H) c = H;
    const int r = (int)((H + c - 1) / c);
    *rows = r;
    *chunks = (H + r - 1) / r;
    return cudaSuccess;
}

bool conv_dims_ok(long long M, int Ci, int Co) { return M > 0 && M % 16 == 0 && Ci > 0 && Ci % 16 == 0 && Co > 0 && Co % 16 == 0; }

}  // namespace

template <bool ACT>
static int conv3x3(const void* x, int csx, const void* w, const float* bias, void* y, int csy, int N, int H, int W,
                   int Ci, int Co, void* stream) {
    const long long M = (long long)N * H * W;
    if (!x || !w || !y || N < 1 || H < 1 || W < 1 || !conv_dims_ok(M, Ci, Co) || csx < Ci || csx % 2 || csy < Co)
        return LBM_EINVAL;
    if (Co > 128) return LBM_EINVAL;
    // 16-byte copies: channel rows and slices start on 16-byte boundaries
    if (csx % 8 || ((uintptr_t)x & 15) || ((uintptr_t)w & 15)) return LBM_EINVAL;
    cudaStream_t s = (cudaStream_t)stream;
    const size_t smem = conv_tc_smem_bytes(Ci, Co);
    static bool attr_set[64] = {};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return LBM_ECUDA;
    if (dev >= 0 && dev < 64 && !attr_set[dev]) {
        if (cudaFuncSetAttribute(conv_tc_kernel<ACT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)conv_tc_smem_bytes(kTcK, 128)) != cudaSuccess)
            return LBM_ECUDA;
        attr_set[dev] = true;
    }
    int* err = nullptr;
    if (cudaGetSymbolAddress((void**)&err, g_sg_err) != cudaSuccess) return LBM_ECUDA;
    // rows of 128-pixel segments: the row march, when four input rows and the
    // weights of all taps fit in shared memory; else flat tiles, when their
    // cells and two taps' weights do and the image is not too wide, else the tap
    // kernel.  us of the U-Net's
    // layers at 8 x 256^2, tap kernel / this: 128 -> 32 at 128^2 157 / 28 (march),
    // 64 -> 128 at 64^2 42 / 28, 256 -> 64 at 64^2 101 / 49, 128 -> 128 at 32^2 39 / 18
    // (flat).
    int sms = 1;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return LBM_ECUDA;
    // CTAs on an SM: up to three, whose copies, MMAs and stores overlap, as long
    // as each keeps eight rows to spread its weights and halo rows over
    const long long row_segs = W % kRowM ? 0 : (long long)N * H * (W / kRowM);
    int per_sm = row_segs ? 3 : 0;
    while (per_sm > 0 && (per_sm * row_tmem_cols(Co) > 512 || conv_row_slots_of(Ci, Co, per_sm) < 4 ||
                          (per_sm > 1 && row_segs < 8LL * per_sm * sms)))
        --per_sm;
    if (per_sm > 0) {
        const int slots = conv_row_slots_of(Ci, Co, per_sm);
        static bool done[64] = {};
        if (large_smem(conv_row_kernel<ACT>, done, dev) != cudaSuccess) {
            cudaGetLastError();
            return LBM_ECUDA;
        }
        const long long cols = (long long)N * (W / kRowM);
        long long chunks = (long long)sms * per_sm / cols;
        if (chunks < 1) chunks = 1;
        if (chunks > H) chunks = H;
        const int rows = (int)((H + chunks - 1) / chunks);
        const long long nb = cols * ((H + rows - 1) / rows);
        conv_row_kernel<ACT><<<(unsigned)nb, kRoleThreads,
                               conv_row_launch_smem(conv_row_smem_bytes(Ci, Co, slots), Co), s>>>(
            (const bf16*)x, csx, (const bf16*)w, bias, y, csy, N, H, W, Ci, Co, rows, slots, err);
        return check(cudaGetLastError());
    }
    const long long flat = (long long)H * (W + 2), tiles = (flat + 127) / 128;
    int Cs = Co;   // output channels of a CTA: halved while that still fills no more than the SMs
    while (Cs % 32 == 0 && N * tiles * (Co / Cs) * 2 <= sms) Cs /= 2;
    // A tile's cells grow with the width (two rows of halo), the tap kernel's nine
    // copies of 128 pixels do not.  us at 1024 rows, tap kernel / flat tiles: 16 -> 16
    // at W = 392 58 / 49, 450 65 / 60, 500 71 / 67; 32 -> 16 at 392 99 / 92, 450 92 / 109;
    // 48 -> 48 at 392 154 / 143, 500 194 / 272, 900 335 / 593; beyond 64 output
    // channels, where the tap kernel holds one CTA per SM, 64 -> 128 at 560 552 / 442.
    // Tiles of one wave wait for latency, not for copies: 16 rows of 900, 32 -> 64
    // 15 / 13, but of 1200 15 / 17.
    const bool pays = W <= 4096 && (flat_cells(W) <= (Co > 64 ? 1280 : 1024) ||
                                    (flat_cells(W) <= 2048 && N * tiles * (Co / Cs) <= sms));
    const int stages = pays ? flat_stages(W, Ci, Cs) : 0;
    if (stages >= 2 && flat < (1LL << 30) && N * tiles < (1LL << 31)) {
        static bool done[64] = {};
        if (large_smem(conv_flat_kernel<ACT>, done, dev) != cudaSuccess) {
            cudaGetLastError();
            return LBM_ECUDA;
        }
        // no more CTAs on an SM than its tensor memory serves (four of 128 columns)
        const size_t need = flat_x_bytes(W, Ci) + (size_t)stages * flat_w_bytes(Ci, Cs);
        const size_t least = sm_shared_bytes() / 5 + 1;
        conv_flat_kernel<ACT><<<dim3((unsigned)(N * tiles), Co / Cs), kRoleThreads, need > least ? need : least, s>>>(
            (const bf16*)x, csx, (const bf16*)w, bias, y, csy, H, W, Ci, Cs, (int)tiles, stages, err);
        return check(cudaGetLastError());
    }
    const unsigned nb = (unsigned)((M + kTcM - 1) / kTcM);
    conv_tc_kernel<ACT><<<nb, kTcM, smem, s>>>((const bf16*)x, csx, (const bf16*)w, bias, y, csy, M, H, W, Ci, Co, err);
    return check(cudaGetLastError());
}

extern "C" {

int lbm_sg_conv3x3(const void* x, int csx, const void* w, const float* bias, float* y, int csy, int N, int H, int W,
                   int Ci, int Co, void* stream) {
    return conv3x3<false>(x, csx, w, bias, y, csy, N, H, W, Ci, Co, stream);
}

int lbm_sg_conv3x3_relu(const void* x, int csx, const void* w, const float* bias, void* y, int csy, int N, int H,
                        int W, int Ci, int Co, void* stream) {
    return conv3x3<true>(x, csx, w, bias, y, csy, N, H, W, Ci, Co, stream);
}

int lbm_sg_status(void* stream) {
    int* err = nullptr;
    if (cudaGetSymbolAddress((void**)&err, g_sg_err) != cudaSuccess) return LBM_ECUDA;
    int h = 0;
    cudaStream_t s = (cudaStream_t)stream;
    if (cudaMemcpyAsync(&h, err, sizeof(int), cudaMemcpyDeviceToHost, s) != cudaSuccess) return LBM_ECUDA;
    if (cudaStreamSynchronize(s) != cudaSuccess) return LBM_ECUDA;
    if (h) {
        const int zero = 0;
        if (cudaMemcpyAsync(err, &zero, sizeof(int), cudaMemcpyHostToDevice, s) != cudaSuccess) return LBM_ECUDA;
        if (cudaStreamSynchronize(s) != cudaSuccess) return LBM_ECUDA;
        return LBM_ETIMEOUT;
    }
    return LBM_OK;
}

long long lbm_sg_wgrad_scratch_floats(int N, int H, int W, int Ci, int Co) {
    const long long M = (long long)N * H * W;
    long long need = ((M + kChunk - 1) / kChunk) * (long long)Co * 9 * Ci;
    int rows = 0, chunks = 0;
    if (wgrad_row_plan(N, H, W, Ci, Co, &rows, &chunks) == cudaSuccess) {
        if (rows > 0) {
            const long long row_need = (long long)N * (W / wg_segment(W)) * chunks * Co * 9 * Ci;
            if (row_need > need) need = row_need;
        }
    } else {
        cudaGetLastError();   // the plan's failure is reported by lbm_sg_conv3x3_wgrad, not left pending
    }
    return need;
}

static void sum_chunks(const float* partial, long long nchunks, long long K, float* gw, cudaStream_t s) {
    if (K < (1 << 16)) sum_chunks_kernel<32><<<(unsigned)((K + 31) / 32), 32, 0, s>>>(partial, nchunks, K, gw);
    else sum_chunks_kernel<256><<<(unsigned)((K + 255) / 256), 256, 0, s>>>(partial, nchunks, K, gw);
}

int lbm_sg_conv3x3_wgrad(const void* x, int csx, const void* gy, int csg, float* gw, float* scratch,
                         long long scratch_floats, int N, int H, int W, int Ci, int Co, void* stream) {
    const long long M = (long long)N * H * W;
    if (!x || !gy || !gw || !scratch || N < 1 || H < 1 || W < 1 || !conv_dims_ok(M, Ci, Co) || csx < Ci || csg < Co)
        return LBM_EINVAL;
    const long long need = lbm_sg_wgrad_scratch_floats(N, H, W, Ci, Co);
    if (scratch_floats < need) return LBM_EINVAL;
    // rows in segments of 64 or 32 pixels, with 16-byte aligned channel rows: the
    // tcgen05 row march
    int rows = 0, rchunks = 0;
    if (wgrad_row_plan(N, H, W, Ci, Co, &rows, &rchunks) != cudaSuccess) {
        cudaGetLastError();
        return LBM_ECUDA;
    }
    if (rows > 0 && csx % 8 == 0 && csg % 8 == 0 && ((uintptr_t)x & 15) == 0 && ((uintptr_t)gy & 15) == 0 &&
        ((uintptr_t)scratch & 15) == 0) {
        int* err = nullptr;
        if (cudaGetSymbolAddress((void**)&err, g_sg_err) != cudaSuccess) return LBM_ECUDA;
        cudaStream_t s = (cudaStream_t)stream;
        const int P = wg_segment(W), Cn = wg_block(Ci);
        const long long pchunks = (long long)N * (W / P) * rchunks, ctas = 3 * (Ci / Cn) * pchunks;
        const WgLayout Lt = wg_layout(P, Cn, Co);
        // all CTAs on the chip at once where two buffers allow it, a third
        // buffer where it does not cost that; no more than tensor memory serves
        int dev = 0, sms = 1;
        if (cudaGetDevice(&dev) != cudaSuccess ||
            cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
            return LBM_ECUDA;
        const int by_tmem = 512 / (int)wg_tmem_cols(wg_n(Cn, Co));
        long long want = (ctas + sms - 1) / sms;
        if (want > by_tmem) want = by_tmem;
        const int bufs = wg_bytes(Lt, 3) <= kWgSmemMax / (size_t)want - (want > 1 ? 1024 : 0) ? 3 : 2;
        const size_t need = wg_bytes(Lt, bufs), least = sm_shared_bytes() / (size_t)(by_tmem + 1) + 1;
        conv_wgrad_row_kernel<<<(unsigned)ctas, kRoleThreads, need > least ? need : least, s>>>(
            (const bf16*)x, csx, (const bf16*)gy, csg, scratch, N, H, W, Ci, Co, P, Cn, rows, bufs, err);
        const long long K = (long long)Co * 9 * Ci;
        sum_chunks(scratch, pchunks, K, gw, s);
        return check(cudaGetLastError());
    }
    const long long nchunks = (M + kChunk - 1) / kChunk;
    const long long warps = nchunks * 9LL * (Co / 16) * (Ci / 8);
    cudaStream_t s = (cudaStream_t)stream;
    conv_wgrad_kernel<<<(unsigned)((warps * 32 + 127) / 128), 128, 0, s>>>((const bf16*)x, csx, (const bf16*)gy, csg,
                                                                          scratch, M, H, W, Ci, Co);
    const long long K = (long long)Co * 9 * Ci;
    sum_chunks(scratch, nchunks, K, gw, s);
    return check(cudaGetLastError());
}

int lbm_sg_weight_flip(const void* w, void* wt, int Ci, int Co, void* stream) {
    if (!w || !wt || Ci < 1 || Co < 1) return LBM_EINVAL;
    weight_flip_kernel<<<blocks((long long)Co * 9 * Ci), kThreads, 0, (cudaStream_t)stream>>>((const bf16*)w, (bf16*)wt,
                                                                                              Ci, Co);
    return check(cudaGetLastError());
}

// blocks of the sums over pixels, 256 pixels at a time: their number fixes the
// order of the additions
static int sum_blocks(long long npix) {
    return (int)(npix < 64LL * kThreads ? (npix + kThreads - 1) / kThreads : 64);
}

int lbm_sg_bias_grad(const float* g, int csg, float* gb, float* scratch, long long npix, int C, void* stream) {
    if (!g || !gb || !scratch || npix < 1 || C < 1 || csg < C) return LBM_EINVAL;
    const int nb = sum_blocks(npix);
    cudaStream_t s = (cudaStream_t)stream;
    // rows in 16-byte groups, the same sums, from 16 channels on: a block takes 16,
    // and fewer leave its threads idle (10^6 pixels, one channel per block / this: 4
    // channels 12.4 / 20.6 us, 8 20.1 / 20.6, 16 35.7 / 22.6).  Below 32 channels it
    // takes many pixels to pay (16000 pixels of 16: 8.4 / 10.4; 40000: 10.3 either
    // way; 524288: 22.6 / 16.4).
    if ((C >= 32 || (C >= 16 && npix > 32768)) && C % 4 == 0 && csg % 4 == 0 && ((uintptr_t)g & 15) == 0 &&
        ((uintptr_t)scratch & 15) == 0 && npix < (1LL << 30) && (C + 15) / 16 < 65536) {
        relu_grad_kernel<3><<<dim3(nb, (C + 15) / 16), kGradThreads, 0, s>>>(g, csg, nullptr, 0, nullptr, 0, nullptr, 1,
                                                                            (int)npix, C, scratch);
        channel_finish_kernel<<<(C + 31) / 32, 32, 0, s>>>(scratch, nb, C, C, gb);
        return check(cudaGetLastError());
    }
    colsum_partial_kernel<<<dim3(nb, C), kThreads, 0, s>>>(g, csg, npix, C, scratch);
    colsum_finish_kernel<<<blocks(C), kThreads, 0, s>>>(scratch, nb, C, gb);
    return check(cudaGetLastError());
}

int lbm_sg_relu(const float* a, int csa, void* y, int csy, long long npix, int C, void* stream) {
    if (!a || !y || npix < 1 || C < 1 || csa < C || csy < C) return LBM_EINVAL;
    relu_kernel<<<blocks(npix * C), kThreads, 0, (cudaStream_t)stream>>>(a, csa, (bf16*)y, csy, npix, C);
    return check(cudaGetLastError());
}

int lbm_sg_relu_bwd(const float* g, int csg, const float* a, int csa, float* ga, void* ga16, long long npix, int C,
                    void* stream) {
    if (!g || !a || !ga || npix < 1 || C < 1 || csg < C || csa < C) return LBM_EINVAL;
    relu_bwd_kernel<<<blocks(npix * C), kThreads, 0, (cudaStream_t)stream>>>(g, csg, a, csa, ga, (bf16*)ga16, npix, C);
    return check(cudaGetLastError());
}

int lbm_sg_to_bf16(const float* a, int csa, void* y, int csy, long long npix, int C, void* stream) {
    if (!a || !y || npix < 1 || C < 1 || csa < C || csy < C) return LBM_EINVAL;
    to_bf16_kernel<<<blocks(npix * C), kThreads, 0, (cudaStream_t)stream>>>(a, csa, (bf16*)y, csy, npix, C);
    return check(cudaGetLastError());
}

int lbm_sg_add(const float* a, int csa, const float* b, int csb, float* out, int cso, long long npix, int C,
               void* stream) {
    if (!a || !b || !out || npix < 1 || C < 1 || csa < C || csb < C || cso < C) return LBM_EINVAL;
    add_kernel<<<blocks(npix * C), kThreads, 0, (cudaStream_t)stream>>>(a, csa, b, csb, out, cso, npix, C);
    return check(cudaGetLastError());
}

static bool pool_dims_ok(int N, int H, int W, int C, int f) {
    return N >= 1 && f >= 1 && f <= 64 && H >= f && W >= f && H % f == 0 && W % f == 0 && C >= 1;
}

// 2 x 2 blocks of 16-byte channel groups (pool2_kernel, upsample2_kernel), with
// 32-bit row and column counts
static bool wide_ok(const void* x, int csx, const void* y, int csy, int N, int H, int W, int C, int f) {
    return f == 2 && C % 8 == 0 && csx % 8 == 0 && csy % 8 == 0 && ((uintptr_t)x & 15) == 0 && ((uintptr_t)y & 15) == 0 &&
           (long long)N * H < (1LL << 31) && (long long)W * C < (1LL << 31);
}
static dim3 wide_grid(int N, int H, int W, int C) {
    const int rows = N * (H / 2);
    return dim3(blocks((long long)(W / 2) * (C / 8)), rows < 16384 ? rows : 16384);
}

int lbm_sg_relu_grad(const float* g, int csg, int up, const float* gp, int csp, const void* act, int csa, void* ga,
                     float* gb, float* scratch, long long scratch_floats, int N, int H, int W, int C, void* stream) {
    const long long npix = (long long)N * H * W;
    if (!g || !act || !ga || !gb || !scratch || N < 1 || H < 1 || W < 1 || npix >= (1LL << 30)) return LBM_EINVAL;
    if ((up != 1 && up != 2) || (gp && (up != 1 || H % 2 || W % 2 || csp < C || csp % 4))) return LBM_EINVAL;
    if (C < 4 || C % 4 || C > 1024 || csg < C || csg % 4 || csa < C || csa % 4) return LBM_EINVAL;
    if (((uintptr_t)g & 15) || ((uintptr_t)gp & 15) || ((uintptr_t)act & 7) || ((uintptr_t)ga & 7) ||
        ((uintptr_t)scratch & 15))
        return LBM_EINVAL;
    const int nb = sum_blocks(npix);
    if (scratch_floats < (long long)nb * C) return LBM_EINVAL;
    cudaStream_t s = (cudaStream_t)stream;
    const bf16* a = (const bf16*)act;
    bf16* o = (bf16*)ga;
    const dim3 grid(nb, (C + 15) / 16);
    const int np = (int)npix;
    if (gp) relu_grad_kernel<2><<<grid, kGradThreads, 0, s>>>(g, csg, gp, csp, a, csa, o, W, np, C, scratch);
    else if (up == 2) relu_grad_kernel<1><<<grid, kGradThreads, 0, s>>>(g, csg, gp, csp, a, csa, o, W, np, C, scratch);
    else relu_grad_kernel<0><<<grid, kGradThreads, 0, s>>>(g, csg, gp, csp, a, csa, o, W, np, C, scratch);
    channel_finish_kernel<<<(C + 31) / 32, 32, 0, s>>>(scratch, nb, C, C, gb);
    return check(cudaGetLastError());
}

int lbm_sg_mse_grad(const float* x, const float* delta, const float* target, void* g16, float* g4, float* gb,
                    double* scratch, double* loss, long long npix, void* stream) {
    if (!x || !delta || !target || !g16 || !g4 || !gb || !scratch || !loss || npix < 1 || npix >= (1LL << 30))
        return LBM_EINVAL;
    if (((uintptr_t)x & 15) || ((uintptr_t)delta & 15) || ((uintptr_t)g16 & 15) || ((uintptr_t)g4 & 15) ||
        ((uintptr_t)scratch & 15))
        return LBM_EINVAL;
    long long nb = (npix + kThreads - 1) / kThreads;
    if (nb > LBM_SG_LOSS_BLOCKS) nb = LBM_SG_LOSS_BLOCKS;
    const int ngb = sum_blocks(npix);
    cudaStream_t s = (cudaStream_t)stream;
    float* gpart = (float*)(scratch + LBM_SG_LOSS_BLOCKS);
    const double inv = 1.0 / ((double)npix * 4);
    mse_grad_kernel<<<(unsigned)nb, kThreads, 0, s>>>((const float4*)x, delta, target, ((uintptr_t)target & 15) == 0,
                                                      (bf16*)g16, (float4*)g4, (int)npix, inv, scratch);
    relu_grad_kernel<3><<<dim3(ngb, 1), kGradThreads, 0, s>>>(g4, 4, nullptr, 0, nullptr, 0, nullptr, 1, (int)npix, 4,
                                                             gpart);
    mse_grad_finish_kernel<<<1, 64, 0, s>>>(scratch, (int)nb, gpart, ngb, inv, loss, gb);
    return check(cudaGetLastError());
}

int lbm_sg_adam_layers(const lbm_sg_layer* layers, int n, float lr, float b1, float b2, float eps, int step,
                       void* stream) {
    if (!layers || n < 1 || n > kMaxLayers || step < 1 || !(lr > 0) || !(b1 >= 0 && b1 < 1) || !(b2 >= 0 && b2 < 1))
        return LBM_EINVAL;
    AdamLayers a = {};
    int most = 0;
    for (int k = 0; k < n; ++k) {
        const lbm_sg_layer& l = layers[k];
        if (!l.w || !l.mw || !l.vw || !l.gw || !l.b || !l.mb || !l.vb || !l.gb || !l.w16 || !l.wt || l.ci < 1 || l.co < 1 ||
            l.ci > 4096 || l.co > 4096)
            return LBM_EINVAL;
        a.l[k] = l;
        if (l.co * 9 * l.ci + l.co > most) most = l.co * 9 * l.ci + l.co;
    }
    const float c1 = 1.0f - powf(b1, (float)step), c2 = 1.0f - powf(b2, (float)step);
    adam_layers_kernel<<<dim3(blocks(most), n), kThreads, 0, (cudaStream_t)stream>>>(a, lr, b1, b2, eps, c1, c2);
    return check(cudaGetLastError());
}

int lbm_sg_pool(const void* x, int csx, void* y, int csy, int N, int H, int W, int C, int f, void* stream) {
    if (!x || !y || !pool_dims_ok(N, H, W, C, f) || csx < C || csy < C) return LBM_EINVAL;
    const long long n = (long long)N * (H / f) * (W / f) * C;
    if (wide_ok(x, csx, y, csy, N, H, W, C, f)) {
        pool2_kernel<<<wide_grid(N, H, W, C), kThreads, 0, (cudaStream_t)stream>>>((const bf16*)x, csx, (bf16*)y, csy,
                                                                                  N * (H / 2), W / 2, C / 8);
        return check(cudaGetLastError());
    }
    pool_kernel<<<blocks(n), kThreads, 0, (cudaStream_t)stream>>>((const bf16*)x, csx, (bf16*)y, csy, N, H, W, C, f);
    return check(cudaGetLastError());
}

int lbm_sg_pool_bwd(const float* g, int csg, float* gx, int csx, int N, int H, int W, int C, int f, void* stream) {
    if (!g || !gx || !pool_dims_ok(N, H, W, C, f) || csx < C || csg < C) return LBM_EINVAL;
    pool_bwd_kernel<<<blocks((long long)N * H * W * C), kThreads, 0, (cudaStream_t)stream>>>(g, csg, gx, csx, N, H, W,
                                                                                            C, f);
    return check(cudaGetLastError());
}

int lbm_sg_upsample(const void* x, int csx, void* y, int csy, int N, int H, int W, int C, int f, void* stream) {
    if (!x || !y || !pool_dims_ok(N, H, W, C, f) || csx < C || csy < C) return LBM_EINVAL;
    if (wide_ok(x, csx, y, csy, N, H, W, C, f)) {
        upsample2_kernel<<<wide_grid(N, H, W, C), kThreads, 0, (cudaStream_t)stream>>>(
            (const bf16*)x, csx, (bf16*)y, csy, N * (H / 2), W / 2, C / 8);
        return check(cudaGetLastError());
    }
    upsample_kernel<<<blocks((long long)N * H * W * C), kThreads, 0, (cudaStream_t)stream>>>((const bf16*)x, csx,
                                                                                            (bf16*)y, csy, N, H, W, C,
                                                                                            f);
    return check(cudaGetLastError());
}

int lbm_sg_upsample_bwd(const float* g, int csg, float* gx, int csx, int N, int H, int W, int C, int f,
                        void* stream) {
    if (!g || !gx || !pool_dims_ok(N, H, W, C, f) || csx < C || csg < C) return LBM_EINVAL;
    const long long n = (long long)N * (H / f) * (W / f) * C;
    upsample_bwd_kernel<<<blocks(n), kThreads, 0, (cudaStream_t)stream>>>(g, csg, gx, csx, N, H, W, C, f);
    return check(cudaGetLastError());
}

int lbm_sg_mse(const float* x, int csx, const float* delta, int csd, const float* target, int cst, float* g,
               double* scratch, double* loss, long long npix, int C, void* stream) {
    if (!x || !delta || !target || !g || !scratch || !loss || npix < 1 || C < 1 || csd < C || csx < C || cst < C)
        return LBM_EINVAL;
    const int nb = 256;
    cudaStream_t s = (cudaStream_t)stream;
    mse_kernel<<<nb, kThreads, 0, s>>>(x, csx, delta, csd, target, cst, g, npix, C, scratch);
    mse_finish_kernel<<<1, 32, 0, s>>>(scratch, nb, 1.0 / ((double)npix * C), loss);
    return check(cudaGetLastError());
}

int lbm_sg_adam(float* w, float* m, float* v, const float* g, long long n, float lr, float b1, float b2, float eps,
                int step, void* w16, void* stream) {
    if (!w || !m || !v || !g || n < 1 || step < 1 || !(lr > 0) || !(b1 >= 0 && b1 < 1) || !(b2 >= 0 && b2 < 1))
        return LBM_EINVAL;
    const float c1 = 1.0f - powf(b1, (float)step), c2 = 1.0f - powf(b2, (float)step);
    adam_kernel<<<blocks(n), kThreads, 0, (cudaStream_t)stream>>>(w, m, v, g, n, lr, b1, b2, eps, c1, c2, (bf16*)w16);
    return check(cudaGetLastError());
}

int lbm_sg_pack(const double* phi, const double* ux, const double* uy, const double* P, const double scale[4],
                float* x32, int cs32, void* x16, int cs16, long long npix, void* stream) {
    if (!phi || !ux || !uy || !P || !scale || !x32 || !x16 || npix < 1 || cs32 < 4 || cs16 < 4) return LBM_EINVAL;
    for (int c = 0; c < 4; ++c)
        if (!(scale[c] > 0)) return LBM_EINVAL;
    pack_kernel<<<blocks(npix), kThreads, 0, (cudaStream_t)stream>>>(phi, ux, uy, P, scale[0], scale[1], scale[2],
                                                                      scale[3], x32, cs32, (bf16*)x16, cs16, npix);
    return check(cudaGetLastError());
}

int lbm_sg_unpack(const float* x32, int cs32, const float* delta, int csd, double* phi, double* ux, double* uy,
                  double* P, const double scale[4], double rho_L, double rho_dif, const double* phi_rho,
                  long long npix, void* stream) {
    if (!x32 || !delta || !phi || !ux || !uy || !P || !scale || npix < 1 || cs32 < 4 || csd < 4 || !(rho_L > 0))
        return LBM_EINVAL;
    if (phi_rho == phi) return LBM_EINVAL;
    unpack_kernel<<<blocks(npix), kThreads, 0, (cudaStream_t)stream>>>(x32, cs32, delta, csd, phi, ux, uy, P, scale[0],
                                                                        scale[1], scale[2], scale[3], rho_L, rho_dif,
                                                                        phi_rho, npix);
    return check(cudaGetLastError());
}

int lbm_sg_residual(const double* a, const double* b, long long n, double* out, double* scratch, void* stream) {
    if (!a || !b || !out || !scratch || n < 1) return LBM_EINVAL;
    const int nb = 256;
    cudaStream_t s = (cudaStream_t)stream;
    residual_partial_kernel<<<nb, kThreads, 0, s>>>(a, b, n, scratch);
    residual_finish_kernel<<<1, 64, 0, s>>>(scratch, nb, out);
    return check(cudaGetLastError());
}

int lbm_sg_phase_pressure(const double* phi, const double* P, long long n, double d, double* out, double* scratch,
                          void* stream) {
    if (!phi || !P || !out || !scratch || n < 1 || !(d >= 0.0 && d < 0.5)) return LBM_EINVAL;
    const int nb = 256;
    cudaStream_t s = (cudaStream_t)stream;
    phase_pressure_partial_kernel<<<nb, kThreads, 0, s>>>(phi, P, n, d, scratch);
    phase_pressure_finish_kernel<<<1, 128, 0, s>>>(scratch, nb, out);
    return check(cudaGetLastError());
}

int lbm_sg_phi_project(double* phi, const double* phi0, long long n, double* scratch, void* stream) {
    if (!phi || !phi0 || !scratch || n < 1) return LBM_EINVAL;
    const int nb = 256;
    cudaStream_t s = (cudaStream_t)stream;
    phi_project_kernel<<<nb, kThreads, 0, s>>>(phi, phi0, n, scratch);
    phi_project_finish_kernel<<<1, 96, 0, s>>>(scratch, nb);
    phi_restore_kernel<<<blocks(n), kThreads, 0, s>>>(phi, n, scratch + 3 * nb);
    return check(cudaGetLastError());
}

int lbm_sg_smooth(double* a, double* tmp, int N, int H, int W, int iters, double k, void* stream) {
    if (!a || !tmp || N < 1 || H < 1 || W < 1 || iters < 0 || !(k >= 0.0 && k <= 0.25)) return LBM_EINVAL;
    const long long n = (long long)N * H * W;
    cudaStream_t s = (cudaStream_t)stream;
    for (int it = 0; it < iters; ++it) {
        smooth_kernel<<<blocks(n), kThreads, 0, s>>>(a, tmp, N, H, W, k);
        smooth_kernel<<<blocks(n), kThreads, 0, s>>>(tmp, a, N, H, W, k);
    }
    return check(cudaGetLastError());
}

int lbm_sg_shift(double* a, long long n, double s, void* stream) {
    if (!a || n < 1) return LBM_EINVAL;
    shift_kernel<<<blocks(n), kThreads, 0, (cudaStream_t)stream>>>(a, n, s);
    return check(cudaGetLastError());
}

}  // extern "C"
