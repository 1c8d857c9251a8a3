// Tensor-core spectral contractions for the mixed-precision modes (tcgen05, sm_103a).
//
// out[line][i] = scale * sum_j D[i][j] u[line][j] is a GEMM with M = lines (128 per CTA),
// N = output nodes, K = input nodes (the paper's derivative operators as matrices).
//   precision 1 (split BF16 x3): u (FP64 or FP32) and D are each split into three BF16
//     slices, x = x1 + x2 + x3, and the six products with slice-order sum <= 4
//     (a3 D1, a2 D2, a1 D3, a2 D1, a1 D2, a1 D1, smallest first) accumulate in FP32 in
//     tensor memory: about 24 significant bits, the accuracy of an FP32 contraction.
//   precision 2 (TF32): one kind::tf32 product of the FP32 values.
// Operands sit in shared memory in the K-major, non-swizzled core-matrix layout
// (8 rows x 16 bytes per core matrix; leading-byte offset = next core matrix along K,
// stride-byte offset = next 8-row group).  The operator image is prepared once on the
// host in exactly that layout and copied with one cp.async.bulk per CTA; the line tile
// is converted and split by the CTA's threads.  One thread issues the MMAs and commits
// them to an mbarrier; every wait is bounded and reports a timeout through *err.
//
// What bounds it is the latency of each tile's phases (load, convert, multiply, store), not
// HBM (a quarter of its rate) or the tensor pipe.  So a thread takes eight consecutive
// nodes of a line (three 16-byte stores of slices instead of 24 of two bytes, which
// conflicted four ways), all index arithmetic is 32-bit and outside the loops, a CTA
// keeps its tensor memory, barriers and operator over the jobs it walks, and the next
// tile's first loads are issued before the epilogue of the current one.  Several CTAs share
// an SM up to 64 nodes; at 65 .. 128 their operands fill it, so one CTA of 16 warps
// works alone.  Per launch on 4,194,304 nodes (32 x 64 x 128 per element), before and after:
// first derivatives r 473 -> 268, theta 996 -> 356, phi 1,099 -> 572 us; second derivatives
// 458 -> 219, 506 -> 178, 328 -> 195 us (bit-identical results); of that, slices converted in
// pairs and the shorter FP64 -> FP32 conversion gave 292 -> 268, 381 -> 356, 585 -> 572.
#include <stdint.h>

#include "fp_convert.cuh"
#include "grmhd_internal.h"

namespace gk {

namespace {

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ uint64_t smem_desc(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
    uint64_t d = 0;
    d |= (uint64_t)((saddr >> 4) & 0x3FFFu);
    d |= (uint64_t)((lbo >> 4) & 0x3FFFu) << 16;
    d |= (uint64_t)((sbo >> 4) & 0x3FFFu) << 32;
    d |= (uint64_t)1 << 46;  // tcgen05 descriptor version
    return d;                // base offset 0, relative LBO, no swizzle
}

// instruction descriptor: D = F32; A = B = BF16 (kind::f16) or TF32 (kind::tf32); both
// operands K-major; N >> 3 at bit 17, M >> 4 at bit 24
__device__ __forceinline__ uint32_t instr_desc(int tf32, int m, int n) {
    uint32_t ab = tf32 ? 2u : 1u;
    return (1u << 4) | (ab << 7) | (ab << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(m >> 4) << 24);
}

__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t phase) {
    uint32_t done = 0;
    // 2^16 tries, each parking the warp up to 20 us (about 1.3 s in all)
    for (int it = 0; it < (1 << 16) && !done; it++)
        asm volatile("{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n"
                     "selp.u32 %0, 1, 0, p;\n}\n"
                     : "=r"(done) : "r"(smem_u32(bar)), "r"(phase), "r"(20000u) : "memory");
    return done != 0;
}

__device__ __forceinline__ float to_f32(double x) { return d2f_rn(x); }
__device__ __forceinline__ float to_f32(float x) { return x; }

template <bool TF32>
__device__ __forceinline__ void mma_issue(uint32_t tmem, uint64_t da, uint64_t db, uint32_t id, uint32_t acc) {
    if (TF32)
        asm volatile("{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
                     "tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem),
                     "l"(da), "l"(db), "r"(id), "r"(acc));
    else
        asm volatile("{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
                     "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem),
                     "l"(da), "l"(db), "r"(id), "r"(acc));
}

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
    uint32_t r;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
    return r;
}

// eight consecutive values of a line (k >= N and missing lines are zero): 16-byte loads where
// the line's values are contiguous and aligned
template <int DIR>
__device__ __forceinline__ void load8(const double* p, uint32_t stride, int n, bool vec, double* v) {
    if (DIR == 2 && vec && n >= 8) {
#pragma unroll
        for (int u = 0; u < 4; u++) {
            const double2 q = reinterpret_cast<const double2*>(p)[u];
            v[2 * u] = q.x;
            v[2 * u + 1] = q.y;
        }
        return;
    }
#pragma unroll
    for (int u = 0; u < 8; u++) v[u] = u < n ? p[(size_t)u * stride] : 0.0;
}
template <int DIR>
__device__ __forceinline__ void load8(const float* p, uint32_t stride, int n, bool vec, float* v) {
    if (DIR == 2 && vec && n >= 8) {
#pragma unroll
        for (int u = 0; u < 2; u++) {
            const float4 q = reinterpret_cast<const float4*>(p)[u];
            v[4 * u] = q.x;
            v[4 * u + 1] = q.y;
            v[4 * u + 2] = q.z;
            v[4 * u + 3] = q.w;
        }
        return;
    }
#pragma unroll
    for (int u = 0; u < 8; u++) v[u] = u < n ? p[(size_t)u * stride] : 0.f;
}

}  // namespace

// W groups of four warps.  Loads: r and theta, thread = line (tid mod 128) and every W-th
// group of eight nodes; phi, consecutive threads take consecutive groups of a line (coalesced).
// Epilogue: warp w serves tensor-memory lanes 32 (w mod 4) .. and every W-th block of eight
// columns.  Shared memory (bytes): [A slices | B image | 2 mbarriers | tmem address]
//   A: nsl x 128 x Kp x es,  B: nsl x Np x Kp x es  (nsl = 3 for BF16 x3, 1 for TF32)
// CTAs per SM that the registers are cut for
template <typename TIn>
__host__ __device__ constexpr int tc_ctas(int W) { return W == 1 ? (sizeof(TIn) == 4 ? 7 : 5) : (W == 2 ? 3 : 1); }

template <int DIR, typename TIn, bool TF32, int W>
__global__ void __launch_bounds__(128 * W, tc_ctas<TIn>(W))
    k_contract_tc(Dims d, const TcJob* __restrict__ jobs, int njobs, const uint8_t* __restrict__ op_img, int N, int Np,
                  int Kp, int tmem_cols, const double* __restrict__ r_scale, int* __restrict__ err) {
    extern __shared__ __align__(1024) uint8_t sm[];
    constexpr int es = TF32 ? 4 : 2, nsl = TF32 ? 1 : 3, NT = 128 * W;
    constexpr int NB = W == 4 ? 4 : 2;                                // groups of eight per thread and batch
    const int kcores = Kp * es / 16, ngr = Kp / 8;
    const uint32_t a_bytes = 128u * Kp * es;
    const uint32_t b_bytes = (uint32_t)Np * Kp * es;
    uint8_t* sA = sm;
    uint8_t* sB = sm + nsl * a_bytes;
    uint64_t* bars = reinterpret_cast<uint64_t*>(sB + nsl * b_bytes);
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

    // lines of a field (32-bit: a field holds fewer than 2^31 points)
    const uint32_t nlines = DIR == 0 ? (uint32_t)(d.E * d.NtNp)
                                     : (DIR == 1 ? (uint32_t)((long long)d.E * d.Nr * d.Np) : (uint32_t)(d.P / N));
    const uint32_t t0 = blockIdx.x * 128u;
    const uint32_t stride = DIR == 0 ? (uint32_t)d.NtNp : (DIR == 1 ? (uint32_t)d.Np : 1u);
    const auto line_base = [&](uint32_t t, uint32_t* e) -> size_t {
        if (DIR == 0) {
            *e = t / (uint32_t)d.NtNp;
            return (size_t)*e * d.elem + (t - *e * (uint32_t)d.NtNp);
        }
        *e = 0;
        if (DIR == 1) {
            const uint32_t r = t / (uint32_t)d.Np;
            return (size_t)r * d.NtNp + (t - r * (uint32_t)d.Np);
        }
        return (size_t)t * N;
    };
    // epilogue line of this thread
    const int m_out = (warp & 3) * 32 + lane;
    const bool valid = t0 + m_out < nlines;
    uint32_t e_out;
    const size_t base = line_base(min(t0 + m_out, nlines - 1), &e_out);
    const float scale = DIR == 0 && r_scale ? d2f_rn(r_scale[e_out]) : 1.0f;
    // load line of this thread (r, theta: the same line for every group, m = tid mod 128, which is
    // m_out; phi: see below)
    const bool vec = (N * sizeof(TIn)) % 16 == 0;
    const auto group = [&](int i, int* m, int* g) {       // this thread's i-th group of eight
        if (DIR == 2) {
            const uint32_t item = (uint32_t)(i * NT + tid);
            *m = (int)(item / (uint32_t)ngr);
            *g = (int)(item - (uint32_t)*m * ngr);
        } else {
            *m = tid & 127;
            *g = i * W + (tid >> 7);
        }
    };
    const int nmine = DIR == 2 ? (128 * ngr - tid + NT - 1) / NT : (ngr - (tid >> 7) + W - 1) / W;   // its groups
    const auto load_batch = [&](const TIn* src, int b, TIn (*raw)[8]) {
#pragma unroll
        for (int v = 0; v < NB; v++) {
            int m, g;
            group(b * NB + v, &m, &g);
            const uint32_t t = t0 + m;
            const size_t bs = DIR == 2 ? (size_t)t * N : base;
            const bool on = b * NB + v < nmine && t < nlines;
            load8<DIR>(src + bs + (size_t)(8 * g) * stride, stride, on ? N - 8 * g : 0, vec, raw[v]);
        }
    };
    const auto store_batch = [&](int b, const TIn (*raw)[8]) {
#pragma unroll
        for (int v = 0; v < NB; v++) {
            if (b * NB + v >= nmine) continue;
            int m, g;
            group(b * NB + v, &m, &g);
            float x[8];
#pragma unroll
            for (int u = 0; u < 8; u++) x[u] = to_f32(raw[v][u]);
            uint8_t* row = sA + ((uint32_t)(m >> 3) * kcores * 128u + (m & 7) * 16u);
            if (TF32) {
                uint32_t w[8];
#pragma unroll
                for (int u = 0; u < 8; u++) asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(w[u]) : "f"(x[u]));
                *reinterpret_cast<uint4*>(row + 2 * g * 128) = make_uint4(w[0], w[1], w[2], w[3]);
                *reinterpret_cast<uint4*>(row + (2 * g + 1) * 128) = make_uint4(w[4], w[5], w[6], w[7]);
            } else {
                uint32_t w[3][4];
#pragma unroll
                for (int u = 0; u < 4; u++) {
                    // two values at a time: one conversion instruction per slice packs both
                    float f0 = x[2 * u], f1 = x[2 * u + 1];
#pragma unroll
                    for (int l = 0; l < 3; l++) {
                        w[l][u] = pack_bf16(f0, f1);
                        f0 -= __uint_as_float(w[l][u] << 16);
                        f1 -= __uint_as_float(w[l][u] & 0xFFFF0000u);
                    }
                }
#pragma unroll
                for (int l = 0; l < 3; l++)
                    *reinterpret_cast<uint4*>(row + l * a_bytes + g * 128) = make_uint4(w[l][0], w[l][1], w[l][2], w[l][3]);
            }
        }
    };

    if (tid == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&bars[0])));
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&bars[1])));
        asm volatile("fence.mbarrier_init.release.cluster;");
        // operator image: one bulk copy, completion counted in bytes on bars[0]
        const uint32_t bytes = nsl * b_bytes;
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(&bars[0])),
                     "r"(bytes) : "memory");
        asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                         smem_u32(sB)),
                     "l"(op_img), "r"(bytes), "r"(smem_u32(&bars[0]))
                     : "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                     "r"(tmem_cols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    const int nbatch = ((ngr + W - 1) / W + NB - 1) / NB;
    TIn raw[NB][8];
    load_batch(static_cast<const TIn*>(jobs[blockIdx.y].src), 0, raw);
    bool ok = true;
    uint32_t phase = 0;
    for (int j = blockIdx.y; j < njobs; j += gridDim.y, phase ^= 1u) {
        const TcJob job = jobs[j];
        // line tile: convert and split into the K-major layout (zero padding in K and lines)
        for (int b = 0; b < nbatch; b++) {
            if (b > 0) load_batch(static_cast<const TIn*>(job.src), b, raw);
            store_batch(b, raw);
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        asm volatile("tcgen05.fence::before_thread_sync;");
        if (!__syncthreads_and(ok ? 1 : 0)) break;
        asm volatile("tcgen05.fence::after_thread_sync;");
        const uint32_t tmem = *tmem_slot;
        if (tid == 0) {
            ok = phase != 0 || j != (int)blockIdx.y || mbar_wait(&bars[0], 0);
            if (ok) {
                const uint32_t id = instr_desc(TF32, 128, Np);
                const uint32_t lbo = 128u, sbo = (uint32_t)kcores * 128u;
                const int kstep = TF32 ? 8 : 16;                 // K per instruction
                // slice pairs (a, b), smallest contribution first
                const int pa[6] = {2, 1, 0, 1, 0, 0};
                const int pb[6] = {0, 1, 2, 0, 1, 0};
                uint32_t acc = 0;
                for (int q = 0; q < (TF32 ? 1 : 6); q++) {
                    const int ia = TF32 ? 0 : pa[q], ib = TF32 ? 0 : pb[q];
                    for (int c = 0; c < Kp / kstep; c++) {
                        const uint64_t da = smem_desc(smem_u32(sA + ia * a_bytes) + c * 256, lbo, sbo);
                        const uint64_t db = smem_desc(smem_u32(sB + ib * b_bytes) + c * 256, lbo, sbo);
                        mma_issue<TF32>(tmem, da, db, id, acc);
                        acc = 1;
                    }
                }
                asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                    smem_u32(&bars[1])));
            } else {
                atomicExch(err, 1);
                // release bars[1] so that the other threads do not wait in vain
                asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&bars[1])) : "memory");
            }
        }
        __syncwarp();
        // the next tile's first loads, in flight over the multiplication and the epilogue
        if (j + (int)gridDim.y < njobs) load_batch(static_cast<const TIn*>(jobs[j + gridDim.y].src), 0, raw);
        if (!mbar_wait(&bars[1], phase)) {
            ok = false;
            if (lane == 0) atomicExch(err, 1);
        }
        asm volatile("tcgen05.fence::after_thread_sync;");
        // epilogue: eight output columns at a time (the radial Jacobian multiplies in FP32: one
        // rounding more than forming the product in FP64 before the cast, at most 2^-24
        // relative, where the FP64 product kept the FP64 pipe 63-76 % busy)
        for (int cb = (warp >> 2) * 8; cb < Np; cb += 8 * W) {
            uint32_t r[8];
            const uint32_t ta = tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)cb;
            asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                         : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
                           "=r"(r[7])
                         : "r"(ta));
            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
            if (!ok || !valid || cb >= N) continue;
            float o[8];
#pragma unroll
            for (int u = 0; u < 8; u++) o[u] = __fmul_rn(scale, __uint_as_float(r[u]));
            float* p = job.dst + base + (size_t)cb * stride;
            if (DIR == 2 && cb + 8 <= N && (N & 3) == 0) {
                // a line's 8 outputs are contiguous: two 16-byte stores
                float4* p4 = reinterpret_cast<float4*>(p);
                float4 lo = make_float4(o[0], o[1], o[2], o[3]), hi = make_float4(o[4], o[5], o[6], o[7]);
                if (job.accumulate) {
                    const float4 a0 = p4[0], a1 = p4[1];
                    lo.x += a0.x; lo.y += a0.y; lo.z += a0.z; lo.w += a0.w;
                    hi.x += a1.x; hi.y += a1.y; hi.z += a1.z; hi.w += a1.w;
                }
                p4[0] = lo;
                p4[1] = hi;
                continue;
            }
            const int n = min(8, N - cb);
            if (job.accumulate) {
                // all loads before the first store (the compiler cannot reorder them)
                float old[8];
#pragma unroll
                for (int u = 0; u < 8; u++) old[u] = u < n ? p[(size_t)u * stride] : 0.f;
#pragma unroll
                for (int u = 0; u < 8; u++) o[u] += old[u];
            }
#pragma unroll
            for (int u = 0; u < 8; u++)
                if (u < n) p[(size_t)u * stride] = o[u];
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(*tmem_slot), "r"(tmem_cols));
}

size_t tc_smem_bytes(int N, int tf32) {
    const int es = tf32 ? 4 : 2, nsl = tf32 ? 1 : 3;
    const int Kp = (N + 15) / 16 * 16, Np = Kp;
    return (size_t)nsl * (128u * Kp * es + (size_t)Np * Kp * es) + 2 * sizeof(uint64_t) + 16;
}

// groups of four warps per CTA: many small CTAs share an SM up to 32 nodes; above, the
// operands leave room for two or three (64 nodes) or one (128), which get more warps
template <int DIR, typename TIn, bool TF32, int W>
static cudaError_t launch_w(const Dims& d, const TcJob* jobs, int njobs, const uint8_t* img, int N,
                            const double* r_scale, int* err, cudaStream_t s) {
    const int Kp = (N + 15) / 16 * 16, Np = Kp;
    const int cols = Np <= 32 ? 32 : (Np <= 64 ? 64 : (Np <= 128 ? 128 : 256));
    const long long nlines = DIR == 0 ? (long long)d.E * d.NtNp : (DIR == 1 ? (long long)d.E * d.Nr * d.Np : d.P / N);
    if (d.P >= (1LL << 31)) return cudaErrorNotSupported;   // 32-bit line arithmetic
    const long long nb = (nlines + 127) / 128;
    // jobs walked by a CTA: about eight rounds of CTAs in all.  Fewer rounds leave a longer last
    // one, one job per CTA repeats the set-up (4.2M nodes, phi first derivatives: 620 us at two
    // rounds, 618 at four, 585 at eight, 658 at one job each)
    int dev = 0, nsm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    const long long want = tc_ctas<TIn>(W) * (long long)nsm * 8;
    long long gy = (want + nb - 1) / nb;
    if (gy > njobs) gy = njobs;
    if (gy < 1) gy = 1;
    const size_t sm = tc_smem_bytes(N, TF32);
    k_contract_tc<DIR, TIn, TF32, W><<<dim3((unsigned)nb, (unsigned)gy), 128 * W, sm, s>>>(
        d, jobs, njobs, img, N, Np, Kp, cols, r_scale, err);
    return cudaGetLastError();
}

template <int DIR, typename TIn, bool TF32>
static cudaError_t launch_dir(const Dims& d, const TcJob* jobs, int njobs, const uint8_t* img, int N,
                              const double* r_scale, int* err, cudaStream_t s) {
    if (N <= 32) return launch_w<DIR, TIn, TF32, 1>(d, jobs, njobs, img, N, r_scale, err, s);
    if (N <= 64) return launch_w<DIR, TIn, TF32, 2>(d, jobs, njobs, img, N, r_scale, err, s);
    return launch_w<DIR, TIn, TF32, 4>(d, jobs, njobs, img, N, r_scale, err, s);
}

template <int DIR, typename TIn, bool TF32, int W>
static cudaError_t set_attr_w() {
    return cudaFuncSetAttribute(k_contract_tc<DIR, TIn, TF32, W>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)tc_smem_bytes(W == 1 ? 32 : (W == 2 ? 64 : 128), TF32));
}
template <int DIR, typename TIn>
static cudaError_t set_attr() {
    cudaError_t e;
    if ((e = set_attr_w<DIR, TIn, false, 1>()) != cudaSuccess) return e;
    if ((e = set_attr_w<DIR, TIn, false, 2>()) != cudaSuccess) return e;
    if ((e = set_attr_w<DIR, TIn, false, 4>()) != cudaSuccess) return e;
    if ((e = set_attr_w<DIR, TIn, true, 1>()) != cudaSuccess) return e;
    if ((e = set_attr_w<DIR, TIn, true, 2>()) != cudaSuccess) return e;
    return set_attr_w<DIR, TIn, true, 4>();
}

cudaError_t tc_init() {
    cudaError_t e;
    if ((e = set_attr<0, double>()) != cudaSuccess) return e;
    if ((e = set_attr<1, double>()) != cudaSuccess) return e;
    if ((e = set_attr<2, double>()) != cudaSuccess) return e;
    if ((e = set_attr<0, float>()) != cudaSuccess) return e;
    if ((e = set_attr<1, float>()) != cudaSuccess) return e;
    return set_attr<2, float>();
}

template <typename TIn, bool TF32>
static cudaError_t launch_any(int dir, const Dims& d, const TcJob* jobs, int njobs, const uint8_t* img,
                              const double* r_scale, int* err, cudaStream_t s) {
    if (dir == 0) return launch_dir<0, TIn, TF32>(d, jobs, njobs, img, d.Nr, r_scale, err, s);
    if (dir == 1) return launch_dir<1, TIn, TF32>(d, jobs, njobs, img, d.Nt, nullptr, err, s);
    return launch_dir<2, TIn, TF32>(d, jobs, njobs, img, d.Np, nullptr, err, s);
}

cudaError_t launch_contract_tc(int dir, int in_fp32, const Dims& d, const TcJob* jobs, int njobs,
                               const uint8_t* op_img, int tf32, const double* r_scale, int* err,
                               cudaStream_t s) {
    if (njobs <= 0) return cudaSuccess;
    const int N = dir == 0 ? d.Nr : (dir == 1 ? d.Nt : d.Np);
    if (N > 128) return cudaErrorNotSupported;
    if (in_fp32) {
        if (tf32) return launch_any<float, true>(dir, d, jobs, njobs, op_img, r_scale, err, s);
        return launch_any<float, false>(dir, d, jobs, njobs, op_img, r_scale, err, s);
    }
    if (tf32) return launch_any<double, true>(dir, d, jobs, njobs, op_img, r_scale, err, s);
    return launch_any<double, false>(dir, d, jobs, njobs, op_img, r_scale, err, s);
}

}  // namespace gk
