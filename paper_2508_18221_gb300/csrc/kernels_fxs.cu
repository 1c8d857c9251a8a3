// Digit-slice contractions of small grids on the integer units.
//
// The same arithmetic as kernels_fx.cu (seven balanced base-256 digits of each line of u and
// row of D, the 28 digit pairs with q + l <= 8, an exact integer sum per digit order, one
// rounding at the end), so the results are the same bits; the products are 4-way 8-bit dot
// products (dp4a) instead of tensor-core tiles.  A tensor-core launch costs 10-15 us however
// small the grid (tensor-memory allocation, operator copy, 128-line tiles that leave most
// SMs idle), and its directions are separate kernels.  Here one launch takes the jobs of
// every direction, with a block of four warps per 32 lines: lane = line, warps share the
// output rows.  Measured on 4,608 nodes (2 x 12 x
// 12 x 16): the derivative chain of a right-hand side (six contractions and four interface
// launches, 92 us) becomes two of 6-13 us and two of 4 us; an SSP-RK3 step 351 -> 224 us
// (172 now).
//
// Work of a block: values to shared memory, line exponents, digit bytes packed four along
// the line (one 32-bit word per digit), then per output row 7 K dot products and the
// conversion of kernels_fx.cu.  Under the Fourier theta basis lanes 0-15 hold the sums and
// lanes 16-31 the differences of 16 phi pairs (fold and unfold of kernels_deriv.cu in
// registers).
#include "fx_digits.cuh"
#include "grmhd_internal.h"

namespace gk {

namespace {

constexpr int NW = 4;           // warps per block
constexpr int LN = 32;          // lines per block (16 phi pairs under the Fourier theta basis)

__host__ __device__ constexpr int fxs_k4(int N) { return (N + 3) / 4; }
// operator image: words[row][k4][8] (digit slice l in word l - 1, four columns per word), then
// the row exponents
__host__ __device__ constexpr int fxs_words(int N) { return N * fxs_k4(N) * 8; }

template <int V>
struct Int {
    static constexpr int value = V;
};

// bytes b of four 64-bit words as one word (b-th byte of z[0] lowest), biased digits made signed
__device__ __forceinline__ uint32_t pack_byte(const unsigned long long z[4], int b) {
    const uint32_t sel = (uint32_t)((b & 3) | ((4 + (b & 3)) << 4));
    const int sh = b >= 4 ? 32 : 0;
    const uint32_t p = __byte_perm((uint32_t)(z[0] >> sh), (uint32_t)(z[1] >> sh), sel);
    const uint32_t q = __byte_perm((uint32_t)(z[2] >> sh), (uint32_t)(z[3] >> sh), sel);
    return __byte_perm(p, q, 0x5410) ^ 0x80808080u;
}

}  // namespace

__global__ void __launch_bounds__(NW * 32) k_contract_small(Dims d, FxsOps ops, const FxsJob* __restrict__ jobs) {
    extern __shared__ __align__(16) uint8_t sm[];
    const FxsJob jb = jobs[blockIdx.y];
    const int dir = jb.dir, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int N = dir == 0 ? d.Nr : (dir == 2 ? d.Np : d.Nt), K4 = fxs_k4(N), words = fxs_words(N);
    const int h = d.Np / 2;
    // tile: first line, lines; radial tiles stay inside an element (its operator)
    int e = 0;
    long long t0, nl;
    if (dir == 0) {
        const int tpe = (int)((d.NtNp + LN - 1) / LN);
        e = blockIdx.x / tpe;
        if (e >= d.E) return;
        t0 = (long long)(blockIdx.x - e * tpe) * LN;
        nl = d.NtNp;
    } else {
        t0 = (long long)blockIdx.x * (dir == 3 ? LN / 2 : LN);
        nl = dir == 1 ? (long long)d.E * d.Nr * d.Np : (dir == 2 ? d.P / N : (long long)d.E * d.Nr * h);
        if (t0 >= nl) return;
    }
    const long long t = t0 + (dir == 3 ? (lane & 15) : lane);
    const bool valid = t < nl;
    long long base = 0, stride = 1;
    if (dir == 0) { base = (long long)e * d.elem + t; stride = d.NtNp; }
    else if (dir == 1) { const long long r = t / d.Np; base = r * d.NtNp + (t - r * d.Np); stride = d.Np; }
    else if (dir == 2) { base = t * N; }
    else { const long long r = t / h; base = r * d.NtNp + (t - r * h); stride = d.Np; }

    // shared memory: operator words (two operators for dir 3) | values [N][33] | digits
    // [K4][7][32] | row exponents (2 N) | partial line exponents
    const int nop = dir == 3 ? 2 : 1;
    uint32_t* sB = reinterpret_cast<uint32_t*>(sm);
    double* sV = reinterpret_cast<double*>(sB + nop * words);
    uint32_t* sA = reinterpret_cast<uint32_t*>(sV + N * 33);
    int* sF = reinterpret_cast<int*>(sA + K4 * 7 * 32);
    int* sE = sF + 2 * N;
    for (int o = 0; o < nop; o++) {
        // dir 3: the sums take the even extension operator when the parity is +1, else the odd
        const uint8_t* img = dir == 3 ? ops.img[(o == 0) == (jb.parity > 0) ? 1 : 3]
                                      : ops.img[dir] + (dir == 0 ? (long long)e * ops.estride : 0);
        const uint4* src = reinterpret_cast<const uint4*>(img);
        uint4* dst = reinterpret_cast<uint4*>(sB + o * words);
        for (int k = threadIdx.x; k < words / 4; k += NW * 32) dst[k] = src[k];
        const int* f = reinterpret_cast<const int*>(img) + words;
        for (int k = threadIdx.x; k < N; k += NW * 32) sF[o * N + k] = f[k];
    }
    // loads in batches of eight: all of a batch in flight
    if (dir == 2) {
        // lines are contiguous: a warp reads its lines along their length
        const int cnt = (int)min((long long)LN, nl - t0);
        for (int k = lane; k < N; k += 32) {
            double v[LN / NW];
#pragma unroll
            for (int q = 0; q < LN / NW; q++) {
                const int l = warp + q * NW;
                v[q] = l < cnt ? jb.src[(t0 + l) * N + k] : 0.0;
            }
#pragma unroll
            for (int q = 0; q < LN / NW; q++) sV[k * 33 + warp + q * NW] = v[q];
        }
    } else {
        for (int k0 = warp; k0 < N; k0 += 8 * NW) {
            double v[8], w[8];
#pragma unroll
            for (int q = 0; q < 8; q++) {
                const int k = k0 + q * NW;
                const bool on = valid && k < N;
                v[q] = on ? jb.src[base + k * stride] : 0.0;
                w[q] = on && dir == 3 ? jb.src[base + h + k * stride] : 0.0;
            }
#pragma unroll
            for (int q = 0; q < 8; q++) {
                const int k = k0 + q * NW;
                if (k < N) sV[k * 33 + lane] = dir == 3 ? (lane < 16 ? v[q] + w[q] : v[q] - w[q]) : v[q];
            }
        }
    }
    __syncthreads();
    int EL = 0;
    for (int k = warp; k < N; k += NW) EL = max(EL, (int)((__double_as_longlong(sV[k * 33 + lane]) >> 52) & 0x7FF));
    sE[warp * 32 + lane] = EL;
    __syncthreads();
#pragma unroll
    for (int w = 0; w < NW; w++) EL = max(EL, sE[w * 32 + lane]);
    for (int g = warp; g < K4; g += NW) {
        unsigned long long z[4];
#pragma unroll
        for (int k = 0; k < 4; k++) z[k] = digit_word(4 * g + k < N ? sV[(4 * g + k) * 33 + lane] : 0.0, EL, 4u);
#pragma unroll
        for (int q = 0; q < 7; q++) sA[(g * 7 + q) * 32 + lane] = pack_byte(z, 6 - q);
    }
    __syncthreads();
    const uint32_t* B = sB + (dir == 3 && lane >= 16 ? words : 0);
    const int* F = sF + (dir == 3 && lane >= 16 ? N : 0);
    const auto finish = [&](const int* acc, int i) {
        // sum_s n_s 2^(8 (7 - s)), the s = 8 term rounded half up: the integer of kernels_fx.cu
        long long R = (long long)acc[0] << 40;
        R += (long long)acc[1] << 32;
        R += (long long)acc[2] << 24;
        R += (long long)acc[3] << 16;
        R += (long long)acc[4] << 8;
        R += (long long)acc[5] + ((acc[6] + 128) >> 8);
        const int X = EL + F[i] - 2096;
        bool ok;
        double v = scale_int_fast(R, X, &ok);
        if (!ok) v = R == 0 ? 0.0 : ldexp_int(R, X);
        if (EL == 0x7FF) v = __longlong_as_double(0x7FF8000000000000ll);
        if (dir == 2) {
            sV[i * 33 + lane] = v;     // (the digits are formed: the values are no longer read)
            return;
        }
        if (dir == 3) {
            const double o = __shfl_xor_sync(0xffffffffu, v, 16);
            v = lane < 16 ? v + o : o - v;
        }
        if (valid) {
            double* q = jb.dst + base + (dir == 3 && lane >= 16 ? h : 0) + i * stride;
            *q = jb.accumulate ? *q + v : v;
        }
    };
    // two output rows at a time share the line's digit words, a last odd one goes alone
    const auto rows = [&](auto nr, int i) {
        constexpr int NR = decltype(nr)::value;
        int acc[NR][7];
#pragma unroll
        for (int r = 0; r < NR; r++)
#pragma unroll
            for (int q = 0; q < 7; q++) acc[r][q] = 0;
#pragma unroll 2
        for (int g = 0; g < K4; g++) {
            uint32_t b[NR][7];
#pragma unroll
            for (int r = 0; r < NR; r++) {
                const uint4* w = reinterpret_cast<const uint4*>(B + ((i + r * NW) * K4 + g) * 8);
                const uint4 b0 = w[0], b1 = w[1];
                b[r][0] = b0.x; b[r][1] = b0.y; b[r][2] = b0.z; b[r][3] = b0.w;
                b[r][4] = b1.x; b[r][5] = b1.y; b[r][6] = b1.z;
            }
#pragma unroll
            for (int q = 0; q < 7; q++) {
                const int a = (int)sA[(g * 7 + q) * 32 + lane];
#pragma unroll
                for (int r = 0; r < NR; r++)
#pragma unroll
                    for (int l = 0; l < 7 - q; l++) acc[r][q + l] = __dp4a(a, (int)b[r][l], acc[r][q + l]);
            }
        }
#pragma unroll
        for (int r = 0; r < NR; r++) finish(acc[r], i + r * NW);
    };
    for (int i = warp; i < N; i += 2 * NW) {
        if (i + NW < N) rows(Int<2>(), i);
        else rows(Int<1>(), i);
    }
    if (dir == 2) {
        // along phi the results go out line by line, as the values came in
        __syncthreads();
        const int cnt = (int)min((long long)LN, nl - t0);
        for (int k = lane; k < N; k += 32)
#pragma unroll
            for (int q = 0; q < LN / NW; q++) {
                const int l = warp + q * NW;
                if (l >= cnt) continue;
                double* o = jb.dst + (t0 + l) * N + k;
                *o = jb.accumulate ? *o + sV[k * 33 + l] : sV[k * 33 + l];
            }
    }
}

bool fxs_supported(int N) { return N >= 2 && N <= 64; }

// the dynamic shared memory of a direction (nop operators of N rows)
static size_t fxs_smem(int N, int nop) {
    return (size_t)nop * fxs_words(N) * 4 + (size_t)N * 33 * 8 + (size_t)fxs_k4(N) * 7 * 32 * 4 + 2 * N * 4 +
           NW * 32 * 4;
}

cudaError_t fxs_init() {
    return cudaFuncSetAttribute(k_contract_small, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)fxs_smem(64, 2));
}

cudaError_t launch_contract_small(const Dims& d, const FxsJob* jobs, int njobs, int dirs, const FxsOps& ops,
                                  cudaStream_t s) {
    if (njobs <= 0 || d.P <= 0) return cudaSuccess;
    long long nb = 0;
    size_t sm = 0;
    const long long blocks[4] = {(long long)d.E * ((d.NtNp + LN - 1) / LN), ((long long)d.E * d.Nr * d.Np + LN - 1) / LN,
                                 (d.P / d.Np + LN - 1) / LN, ((long long)d.E * d.Nr * (d.Np / 2) + LN / 2 - 1) / (LN / 2)};
    const int Ns[4] = {d.Nr, d.Nt, d.Np, d.Nt};
    for (int k = 0; k < 4; k++) {
        if (!(dirs >> k & 1)) continue;
        if (!fxs_supported(Ns[k])) return cudaErrorNotSupported;
        const size_t b = fxs_smem(Ns[k], k == 3 ? 2 : 1);
        sm = b > sm ? b : sm;
        nb = blocks[k] > nb ? blocks[k] : nb;
    }
    k_contract_small<<<dim3((unsigned)nb, (unsigned)njobs), NW * 32, sm, s>>>(d, ops, jobs);
    return cudaGetLastError();
}

}  // namespace gk
