// Spectral derivative / filter contractions on the FP64 units (opts.contraction = 1, and the
// Chebyshev derivatives above 64 nodes): reflection-split products, any size up to 128.
//
// A derivative along direction dir of a field u[E][Nr][Nt][Np] is the 1-D contraction
// (D u)_i = sum_j D_ij u_j along that axis (paper: "The Spectral Derivative Operators"; the
// Chebyshev coefficient route and the Fourier (ik) multiplier are the same linear maps
// written as matrices; r scaled per element, r_scale == nullptr: unscaled).  Every 1-D
// operator of the grid either commutes (modal filters, sign +1) or anticommutes (first
// derivatives, sign -1) with the reflection of its node set: x_j -> -x_j on the Chebyshev
// nodes (j <-> N-1-j) and phi_j -> -phi_j on the Fourier nodes (j <-> N-j, fixed points
// j = 0 and N/2).  Writing a line u as its even and odd parts over the index pairs (j, j'),
// s_j = u_j + u_j',  a_j = u_j - u_j',  gives for an output pair (i, i')
//     out_i  = E s + O a + C u_f,        out_i' = sign (E s - O a + C u_f),
// with E = (D_ij + D_ij')/2, O = (D_ij - D_ij')/2 and C the columns of the fixed points, so
// a pair of outputs costs N fused multiply-adds instead of 2N.
//
// The FP64 pipe (a warp instruction holds a quarter of an SM for 64 cycles) bounds the
// kernel.  A block holds 32 lines (lane = line) as pairs (s, a) in shared memory and the
// operator as pairs (E, O); its four warps share the output pairs, up to four at a time, so
// that one 16-byte read of the line serves eight multiply-adds and eight independent sums hide
// the pipe's latency.  One kernel per direction takes every size
// (a template instance per size, one thread per line, came first, with dense products for
// the sizes without one).  First derivatives, before and after: 8 x 24 x 32 x 64 nodes r 363 ->
// 341, theta 421 -> 406, phi 791 -> 694 us; 5 x 21 x 27 x 40 (dense before) 131 -> 92, 159 ->
// 107, 226 -> 142 us; 96 theta nodes of a 786,432-node grid (dense before) 8,031 -> 2,088 us.
#include "grmhd_internal.h"

namespace gk {

namespace {

// node pairs and fixed points: Chebyshev (directions r, theta; also the theta extension
// operators) or Fourier (phi)
struct SplitSet {
    int np, nf, off;     // pairs (ip + off, N - 1 - ip), fixed points
};
__host__ __device__ __forceinline__ SplitSet split_set(int dir, int N) {
    return dir == 2 ? SplitSet{N / 2 - 1, 2, 1} : SplitSet{N / 2, N % 2, 0};
}
__device__ __forceinline__ int fixed_node(int dir, int N, int f) { return dir == 2 && f == 0 ? 0 : N / 2; }

size_t eo_smem(int dir, int N) {
    const SplitSet s = split_set(dir, N);
    return (size_t)(2 * s.np * s.np + 2 * s.np * s.nf + s.nf * s.nf) * 8 + (size_t)s.np * 32 * 16 + (size_t)s.nf * 32 * 8;
}

// the sums of output pairs ip0 .. ip0 + Q - 1
template <int Q>
__device__ __forceinline__ void pair_sums(const double2* EO, const double2* SA, int np, int ip0, int lane, double* A,
                                          double* B) {
#pragma unroll
    for (int q = 0; q < Q; q++) A[q] = B[q] = 0.0;
    const double2* row = EO + (size_t)ip0 * np;
#pragma unroll 2
    for (int j = 0; j < np; j++) {
        const double2 sa = SA[j * 32 + lane];
#pragma unroll
        for (int q = 0; q < Q; q++) {
            const double2 eo = row[q * np + j];
            A[q] = fma(eo.x, sa.x, A[q]);
            B[q] = fma(eo.y, sa.y, B[q]);
        }
    }
}

}  // namespace

template <int DIR>
__global__ void __launch_bounds__(128) k_deriv_eo(Dims d, const DerivJob* __restrict__ jobs,
                                                  const double* __restrict__ op, int sign,
                                                  const double* __restrict__ r_scale) {
    extern __shared__ __align__(16) double sm[];
    const int N = DIR == 0 ? d.Nr : (DIR == 1 ? d.Nt : d.Np);
    const SplitSet S = split_set(DIR, N);
    const int np = S.np, nf = S.nf, nn = np * np;
    double2* EO = reinterpret_cast<double2*>(sm);
    double2* SA = EO + nn;                             // [np][32]
    double* uf = reinterpret_cast<double*>(SA + np * 32);   // [nf][32]
    double* C = uf + nf * 32;                          // [np][nf]
    double* F = C + np * nf;                           // [nf][np]
    double* G = F + nf * np;                           // [nf][nf]
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int t = threadIdx.x; t < nn; t += 128) EO[t] = make_double2(op[t], op[nn + t]);
    for (int t = threadIdx.x; t < 2 * np * nf + nf * nf; t += 128) C[t] = op[2 * nn + t];
    const DerivJob job = jobs[blockIdx.y];
    const uint32_t nlines = DIR == 0 ? (uint32_t)(d.E * d.NtNp)
                                     : (DIR == 1 ? (uint32_t)((long long)d.E * d.Nr * d.Np) : (uint32_t)(d.P / N));
    const uint32_t t = blockIdx.x * 32u + lane;
    const bool valid = t < nlines;
    const uint32_t tc = valid ? t : nlines - 1;
    size_t base;
    uint32_t stride = 1;
    double scale = 1.0;
    if (DIR == 0) {
        const uint32_t e = tc / (uint32_t)d.NtNp;
        base = (size_t)e * d.elem + (tc - e * (uint32_t)d.NtNp);
        stride = (uint32_t)d.NtNp;
        if (r_scale) scale = r_scale[e];
    } else if (DIR == 1) {
        const uint32_t r = tc / (uint32_t)d.Np;
        base = (size_t)r * d.NtNp + (tc - r * (uint32_t)d.Np);
        stride = (uint32_t)d.Np;
    } else {
        base = (size_t)tc * N;
    }
    const double* src = job.src + base;
    for (int j = warp; j < np; j += 4) {
        const double lo = src[(size_t)(j + S.off) * stride], hi = src[(size_t)(N - 1 - j) * stride];
        SA[j * 32 + lane] = make_double2(lo + hi, lo - hi);
    }
    for (int f = warp; f < nf; f += 4) uf[f * 32 + lane] = src[(size_t)fixed_node(DIR, N, f) * stride];
    __syncthreads();
    double* dst = job.dst + base;
    const auto put = [&](int i, double v) {
        if (!valid) return;
        double* q = dst + (size_t)i * stride;
        *q = job.accumulate ? *q + v : v;
    };
    // pairs per warp and round: the rounds balanced over the four warps
    const int rounds = (np + 15) / 16, Q = rounds ? (np + 4 * rounds - 1) / (4 * rounds) : 1;
    for (int ip0 = warp * Q; ip0 < np; ip0 += 4 * Q) {
        double A[4], B[4];
        const int n = min(Q, np - ip0);
        if (n == 4) pair_sums<4>(EO, SA, np, ip0, lane, A, B);
        else if (n == 3) pair_sums<3>(EO, SA, np, ip0, lane, A, B);
        else if (n == 2) pair_sums<2>(EO, SA, np, ip0, lane, A, B);
        else pair_sums<1>(EO, SA, np, ip0, lane, A, B);
#pragma unroll
        for (int q = 0; q < 4; q++) {
            if (q >= n) break;
            const int ip = ip0 + q;
            double c = 0.0;
            for (int f = 0; f < nf; f++) c = fma(C[ip * nf + f], uf[f * 32 + lane], c);
            put(ip + S.off, (A[q] + B[q] + c) * scale);
            put(N - 1 - ip, sign * (A[q] - B[q] + c) * scale);
        }
    }
    // fixed-point outputs, on the warps that the rounds above leave first
    for (int f = 3 - warp; f < nf; f += 4) {
        double acc = 0.0;
        for (int j = 0; j < np; j++) {
            const double2 sa = SA[j * 32 + lane];
            acc = fma(F[f * np + j], sign < 0 ? sa.y : sa.x, acc);
        }
        for (int g = 0; g < nf; g++) acc = fma(G[f * nf + g], uf[g * 32 + lane], acc);
        put(fixed_node(DIR, N, f), acc * scale);
    }
}

template <int DIR>
static cudaError_t set_attr_eo(int N) {
    return cudaFuncSetAttribute(k_deriv_eo<DIR>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)eo_smem(DIR, N));
}

cudaError_t eo_init() {
    cudaError_t e;
    if ((e = set_attr_eo<0>(128)) != cudaSuccess) return e;
    if ((e = set_attr_eo<1>(128)) != cudaSuccess) return e;
    return set_attr_eo<2>(128);
}

cudaError_t launch_deriv_eo(int dir, const Dims& d, const DerivJob* jobs, int njobs,
                            const double* op_split, int sign, const double* r_scale,
                            cudaStream_t s) {
    if (njobs <= 0 || d.P <= 0) return cudaSuccess;
    const int N = dir == 0 ? d.Nr : (dir == 1 ? d.Nt : d.Np);
    if (N < 2 || N > 128 || (dir == 2 && N % 2) || d.P >= (1LL << 31)) return cudaErrorNotSupported;
    const long long nlines = dir == 0 ? (long long)d.E * d.NtNp : (dir == 1 ? (long long)d.E * d.Nr * d.Np : d.P / N);
    const dim3 grid((unsigned)((nlines + 31) / 32), (unsigned)njobs);
    const size_t sm = eo_smem(dir, N);
    if (dir == 0) k_deriv_eo<0><<<grid, 128, sm, s>>>(d, jobs, op_split, sign, r_scale);
    else if (dir == 1) k_deriv_eo<1><<<grid, 128, sm, s>>>(d, jobs, op_split, sign, nullptr);
    else k_deriv_eo<2><<<grid, 128, sm, s>>>(d, jobs, op_split, sign, nullptr);
    return cudaGetLastError();
}

}  // namespace gk
