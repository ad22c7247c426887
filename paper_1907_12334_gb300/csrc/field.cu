// field.cu -- xi generation (Philox4x64-10 + Box-Muller) and the truncated KL
// contraction Z = Phi diag(sqrt(lambda)) xi (field law of Sec. 1, Eq. (1.2),
// sampled by a truncated Karhunen-Loeve sum instead of the paper's circulant
// embedding).
#include <cmath>

#include "common.cuh"
#include "kl_tc.cuh"
#include "philox.cuh"
#include "prof.cuh"

namespace msg {

__global__ void k_normals(uint64_t seed, uint64_t s0, int64_t S, int M, double* xi)
{
    const int nb = (M + 3) / 4;
    const int64_t total = S * nb;
    const double two_pi = 6.283185307179586476925286766559;
    const double inv53 = 1.0 / 9007199254740992.0;
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < total; t += (int64_t)gridDim.x * blockDim.x) {
        int64_t i = t / nb;
        int j = (int)(t % nb);
        uint64_t x0 = (uint64_t)j, x1 = s0 + (uint64_t)i, x2 = 0, x3 = 0;
        philox4x64_10(x0, x1, x2, x3, seed, 0);
        uint64_t w[4] = {x0, x1, x2, x3};
        double z[4];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            double ua = (double)(w[2 * h] >> 11) * inv53;
            double ub = (double)(w[2 * h + 1] >> 11) * inv53;
            double rad = sqrt(-2.0 * log(1.0 - ua));
            double sn, cs;
            sincos(two_pi * ub, &sn, &cs);
            z[2 * h] = rad * cs;
            z[2 * h + 1] = rad * sn;
        }
        double* out = xi + i * M + 4 * j;
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (4 * j + k < M) out[k] = z[k];
    }
}

// ---------------------------------------------------------------- SIMT GEMM --
// Z[s][x] = sum_m Phi[x][m] * A[s][m], A = sqrt_lambda[m] * xi[s][m], terms in
// increasing m, one fused multiply-add each: every kernel here gives the same bits.

// A rounded to FP32 once per call, rows padded to a multiple of four terms with zeros.
// (The product is taken in FP64, whose rate is 1/64 of FP32's here: formed again in every
// tile, it costs a large call as much as the contraction.)
__global__ void k_kl_a32(const double* __restrict__ sl, const double* __restrict__ xi, int64_t S, int M, int Mp, float* A)
{
    const int64_t n = S * Mp;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x) {
        const int64_t s = e / Mp;
        const int m = (int)(e - s * Mp);
        A[e] = m < M ? (float)(sl[m] * xi[s * M + m]) : 0.f;
    }
}

// FP32: a tile of 16 TR samples x 128 points per CTA, TR x 8 outputs per thread (samples
// ty TR .. + TR - 1, points tx + 16 b: the half warps of a store write 16 consecutive
// points).  Bound by the FMA pipe: 8 TR FMAs for 8 + TR / 4 shared loads a term; the next
// 16 terms travel to registers meanwhile.  Sample tiles are the fastest grid index, so the
// CTAs that read one tile of Phi run together and find it in L2.  513 x 513 points, 400
// terms, 512 samples: 5.25 ms with the 64 x 64
// tiles of k_kl_simt, 2.35 ms here (46 TFLOP/s).
template <int TR, bool DIRECT, class TZ>
__global__ void __launch_bounds__(256, 2) k_kl_f32(const float* __restrict__ Phi, const float* __restrict__ A,
                                                   const double* __restrict__ sl, const double* __restrict__ xi,
                                                   int64_t npts, int M, int Mp, int64_t S, int64_t stiles, int vec, TZ* __restrict__ Z)
{
    constexpr int TS = 16 * TR, TX = 128, BK = 16, LA = TS + 4, LB = TX + 4;
    __shared__ __align__(16) float sA[2][BK * LA], sB[2][BK * LB];
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    const int64_t s0 = (int64_t)(blockIdx.x % stiles) * TS, x0 = (int64_t)(blockIdx.x / stiles) * TX;
    // loads: four consecutive terms of a row each (rows past the end: the last row, not stored)
    constexpr int NA = (TS * 4 + 255) / 256, NB = TX * 4 / 256;
    const int kq = 4 * (tid & 3), row = tid >> 2;
    // vec: every row of Phi starts on 16 bytes
    float4 ra[NA], rb[NB];
    // this thread's rows relative to the tiles, at its first terms (pointers to them spill at
    // TR 8: 513 x 513 points 2.35 -> 2.50 ms; the caller sees that 128 rows fit 32 bits)
    const float *tA = DIRECT ? nullptr : A + s0 * Mp, *tB = Phi + x0 * M;
    const double* tX = DIRECT ? xi + s0 * M : nullptr;
    int oa[NA], ob[NB];
#pragma unroll
    for (int i = 0; i < NA; ++i) oa[i] = (int)min((int64_t)(row + 64 * i), S - 1 - s0) * (DIRECT ? M : Mp) + kq;
#pragma unroll
    for (int i = 0; i < NB; ++i) ob[i] = (int)min((int64_t)(row + 64 * i), npts - 1 - x0) * M + kq;
    const float4 none = make_float4(0.f, 0.f, 0.f, 0.f);
    auto fetch = [&](int k0) {
        const int k = k0 + kq;
#pragma unroll
        for (int i = 0; i < NA; ++i) {
            if constexpr (DIRECT) {  // A's elements formed here
                ra[i] = none;
                if (row + 64 * i < TS) {
                    const double* x = tX + oa[i] + k0;
                    if (k < M) ra[i].x = (float)(sl[k] * x[0]);
                    if (k + 1 < M) ra[i].y = (float)(sl[k + 1] * x[1]);
                    if (k + 2 < M) ra[i].z = (float)(sl[k + 2] * x[2]);
                    if (k + 3 < M) ra[i].w = (float)(sl[k + 3] * x[3]);
                }
            } else {
                ra[i] = (k < Mp && row + 64 * i < TS) ? *reinterpret_cast<const float4*>(tA + oa[i] + k0) : none;
            }
        }
#pragma unroll
        for (int i = 0; i < NB; ++i) {
            const float* p = tB + ob[i] + k0;
            if (vec) rb[i] = k < M ? *reinterpret_cast<const float4*>(p) : none;
            else
                rb[i] = make_float4(k < M ? p[0] : 0.f, k + 1 < M ? p[1] : 0.f, k + 2 < M ? p[2] : 0.f, k + 3 < M ? p[3] : 0.f);
        }
    };
    auto store = [&](int h) {
#pragma unroll
        for (int i = 0; i < NA; ++i) {
            float* d = &sA[h][kq * LA + row + 64 * i];
            if (row + 64 * i >= TS) continue;
            d[0] = ra[i].x; d[LA] = ra[i].y; d[2 * LA] = ra[i].z; d[3 * LA] = ra[i].w;
        }
#pragma unroll
        for (int i = 0; i < NB; ++i) {
            float* d = &sB[h][kq * LB + row + 64 * i];
            d[0] = rb[i].x; d[LB] = rb[i].y; d[2 * LB] = rb[i].z; d[3 * LB] = rb[i].w;
        }
    };
    float acc[TR][8];
#pragma unroll
    for (int a = 0; a < TR; ++a)
#pragma unroll
        for (int b = 0; b < 8; ++b) acc[a][b] = 0.f;
    fetch(0);
    store(0);
    __syncthreads();
    for (int k0 = 0, h = 0; k0 < Mp; k0 += BK, h ^= 1) {
        if (k0 + BK < Mp) fetch(k0 + BK);
        const float *a0 = sA[h] + ty * TR, *b0 = sB[h] + tx;
#pragma unroll 8
        for (int k = 0; k < BK; ++k) {
            float av[TR], bv[8];
#pragma unroll
            for (int a = 0; a < TR; a += TR < 4 ? TR : 4) {
                if constexpr (TR < 4) {
                    const float2 v = *reinterpret_cast<const float2*>(a0 + k * LA);
                    av[0] = v.x; av[1] = v.y;
                } else {
                    const float4 v = *reinterpret_cast<const float4*>(a0 + k * LA + a);
                    av[a] = v.x; av[a + 1] = v.y; av[a + 2] = v.z; av[a + 3] = v.w;
                }
            }
#pragma unroll
            for (int b = 0; b < 8; ++b) bv[b] = b0[k * LB + 16 * b];
#pragma unroll
            for (int a = 0; a < TR; ++a)
#pragma unroll
                for (int b = 0; b < 8; ++b) acc[a][b] = fmaf(av[a], bv[b], acc[a][b]);
        }
        if (k0 + BK < Mp) store(h ^ 1);  // the other buffer was read before the last barrier
        __syncthreads();
    }
#pragma unroll
    for (int a = 0; a < TR; ++a) {
        const int64_t s = s0 + ty * TR + a;
        if (s >= S) continue;
        const int64_t left = npts - x0 - tx;  // points from this thread's first on
        store_wide<8>(Z + s * npts + x0 + tx, 16, acc[a], (int)min((left + 15) >> 4, (int64_t)8));
    }
}

// FP64: a tile of 8 samples x 32 points per CTA, one output per thread.  Bound by the FP64
// pipe (two FMAs a clock and SM), so what counts is work done for padding and an even
// spread over the SMs: small tiles, with a warp's points consecutive.  129 x 65 points, 64
// terms, 24 samples: 71.8 us with 64 x 64 tiles, 28.7 us here (23 us at
// the FP64 rate).
template <class TZ>
__global__ void __launch_bounds__(256) k_kl_f64(const double* __restrict__ Phi, const double* __restrict__ sl,
                                                const double* __restrict__ xi, int64_t npts, int M, int64_t S, int64_t xtiles,
                                                TZ* __restrict__ Z)
{
    constexpr int BK = 64;
    __shared__ double sA[8][BK], sB[BK][33];
    const int tid = threadIdx.x, tx = tid & 31, ty = tid >> 5;
    const int64_t x0 = (int64_t)(blockIdx.x % xtiles) * 32, s0 = (int64_t)(blockIdx.x / xtiles) * 8;
    double acc = 0.0;
    for (int64_t k0 = 0; k0 < M; k0 += BK) {
        const int nk = (int)min((int64_t)BK, M - k0);
        for (int e = tid; e < 8 * BK; e += 256) {
            const int r = e >> 6, k = e & 63;
            if (k < nk) sA[r][k] = s0 + r < S ? sl[k0 + k] * xi[(s0 + r) * M + k0 + k] : 0.0;
        }
        for (int e = tid; e < 32 * BK; e += 256) {
            const int r = e >> 6, k = e & 63;
            if (k < nk) sB[k][r] = Phi[min(x0 + r, npts - 1) * M + k0 + k];
        }
        __syncthreads();
#pragma unroll 8
        for (int k = 0; k < nk; ++k) acc = fma(sA[ty][k], sB[k][tx], acc);
        __syncthreads();
    }
    const int64_t x = x0 + tx, s = s0 + ty;
    if (x < npts && s < S) Z[s * npts + x] = (TZ)acc;
}

// FP32 for rows of any length: 64x64 tile per CTA, 16-deep K slices staged in shared memory,
// 4x4 outputs per thread.
template <class TZ>
__global__ void __launch_bounds__(256) k_kl_simt(const float* __restrict__ Phi, const double* __restrict__ sl,
                                                 const double* __restrict__ xi, int64_t npts, int M, int64_t S,
                                                 TZ* __restrict__ Z)
{
    __shared__ float sA[16][64 + 1];  // [k][s]
    __shared__ float sB[16][64 + 1];  // [k][x]
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    const int64_t s0 = (int64_t)blockIdx.y * 64, x0 = (int64_t)blockIdx.x * 64;
    float acc[4][4];
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) acc[a][b] = 0.f;
    for (int64_t k0 = 0; k0 < M; k0 += 16) {
        for (int e = threadIdx.x; e < 64 * 16; e += 256) {
            int r = e / 16, k = e % 16;
            int64_t s = s0 + r, x = x0 + r;
            const int64_t m = k0 + k;
            sA[k][r] = (s < S && m < M) ? (float)(sl[m] * xi[s * M + m]) : 0.f;
            sB[k][r] = (x < npts && m < M) ? Phi[x * M + m] : 0.f;
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < 16; ++k) {
            float av[4], bv[4];
#pragma unroll
            for (int a = 0; a < 4; ++a) av[a] = sA[k][ty * 4 + a];
#pragma unroll
            for (int b = 0; b < 4; ++b) bv[b] = sB[k][tx * 4 + b];
#pragma unroll
            for (int a = 0; a < 4; ++a)
#pragma unroll
                for (int b = 0; b < 4; ++b) acc[a][b] = fmaf(av[a], bv[b], acc[a][b]);
        }
        __syncthreads();
    }
#pragma unroll
    for (int a = 0; a < 4; ++a) {
        int64_t s = s0 + ty * 4 + a;
        if (s >= S) continue;
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            int64_t x = x0 + tx * 4 + b;
            if (x < npts) Z[s * npts + x] = (TZ)acc[a][b];
        }
    }
}

__global__ void k_to_float(const double* in, float* out, int64_t n)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        out[i] = (float)in[i];
}

}  // namespace msg

using namespace msg;

extern "C" int32_t msg_normals(uint64_t seed, uint64_t s0, int64_t S, int32_t M, double* xi, void* stream)
{
    clear_error();
    if (S < 0 || M < 1) { set_error("msg_normals: need S >= 0 and M >= 1"); return MSG_ERR_INVALID; }
    if (S == 0) return MSG_OK;
    if (!xi) { set_error("msg_normals: xi is NULL"); return MSG_ERR_INVALID; }
    int64_t total = S * ((M + 3) / 4);
    int blocks = (int)std::min<int64_t>((total + 255) / 256, 152 * 16);
    prof_begin(K_NORMALS, (cudaStream_t)stream);
    k_normals<<<blocks, 256, 0, (cudaStream_t)stream>>>(seed, s0, S, M, xi);
    prof_end(K_NORMALS, (cudaStream_t)stream, 8.0 * S * M, 0.0);
    MSG_CHECK_LAUNCH();
    return MSG_OK;
}

namespace {
size_t align256(size_t x) { return (x + 255) / 256 * 256; }
}

namespace {
// Form of an FP32 call: the sample tile is 16 TR, and DIRECT forms A in the tile.
//
// A wave of one tile an SM takes about 3, 4 and 7 units of time for TR 2, 4 and 8, so the
// widest tile is the cheapest that fills its waves, and the narrowest the fastest of a call
// that gives every SM at most one; a single wave of the widest loses to two of the next one
// by what its start and end cost with few terms (8385 points, 200 samples: 14.4 and 12.4 us at
// 20 terms, even at 150, 47.2 and 49.2 at 300).  Choosing by S alone left most
// SMs without a tile: 400 points, 600 samples, 64 terms 20.5 us with TR 8, 8.3 with TR 2 (the 64 x 64
// tiles of k_kl_simt: 12.8); 4000, 200, 300 47.2 us with TR 8, 30.8 with TR 4 (53.3).
//
// Forming A in the tile costs the FP64 pipe 16 TR M clocks a wave; the launch in front costs
// a call 4 us and its temporary 2 more.  The two are even near 12500 clocks of a single
// wave (2048 points, 200 samples, kernels alone: 8.3 and 12.4 us at 64 terms, 24.7 and 24.7 at
// 300, 30.8 and 28.7 at 400) and near 15000 of several, which overlap them (1175, 1000, 110
// terms: 25.1 and 27.3 us a call).  Every form sums the same terms in the same order.
struct KlForm {
    int TR;
    bool direct;
};
int64_t kl_f32_tiles(int64_t npts, int64_t S, int TR) { return (S + 16 * TR - 1) / (16 * TR) * ((npts + 127) / 128); }
KlForm kl_f32_form(int64_t npts, int32_t M, int64_t S)
{
    auto waves = [&](int TR) { return (kl_f32_tiles(npts, S, TR) + 151) / 152; };
    const int64_t t8 = 14 * waves(8) + (M < 128 && waves(8) == 1 ? 3 : 0), t4 = 8 * waves(4), t2 = 6 * waves(2);
    const int TR = t2 < std::min(t4, t8) ? 2 : t4 < t8 ? 4 : 8;
    return KlForm{TR, 16LL * TR * M * waves(TR) <= (waves(TR) == 1 ? 12500 : 15000)};
}

// Without a temporary for A (none can be had, or the stream is captured: a graph with an
// allocation can neither be instantiated twice nor be part of another) every form is direct:
// 20000 points, 400 terms, 1000 samples 591 us, with the temporary 401, in the 64 x 64
// tiles 799.  Those take what 32-bit offsets into a tile's 128 rows cannot.
template <class TZ>
void kl_fp32(const float* Phi, const double* sl, const double* xi, int64_t npts, int M, int64_t S, TZ* Z, cudaStream_t st)
{
    const KlForm f = kl_f32_form(npts, M, S);
    const int64_t stiles = (S + 16 * f.TR - 1) / (16 * f.TR), tiles = kl_f32_tiles(npts, S, f.TR);
    if (M > 0x7fffffff / 128 - 4 || tiles > 0x7fffffffLL) {
        k_kl_simt<TZ><<<dim3((unsigned)((npts + 63) / 64), (unsigned)((S + 63) / 64)), 256, 0, st>>>(Phi, sl, xi, npts, M, S, Z);
        return;
    }
    const int Mp = (M + 3) & ~3;
    const int vec = M == Mp && (uintptr_t)Phi % 16 == 0;  // (the prepared buffer may have any alignment)
    void* A = nullptr;
    if (!f.direct) {
        cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
        if (cudaStreamIsCapturing(st, &capture) != cudaSuccess) cudaGetLastError();
        if (capture == cudaStreamCaptureStatusNone && temp_alloc(&A, sizeof(float) * S * Mp, st) != cudaSuccess) A = nullptr;
    }
    if (A) {
        k_kl_a32<<<(unsigned)std::min<int64_t>((S * Mp + 255) / 256, 152 * 8), 256, 0, st>>>(sl, xi, S, M, Mp, (float*)A);
        prof_also();
    }
    auto go = [&](auto kernel) { kernel<<<(unsigned)tiles, 256, 0, st>>>(Phi, (const float*)A, sl, xi, npts, M, Mp, S, stiles, vec, Z); };
    if (f.TR == 2) go(A ? k_kl_f32<2, false, TZ> : k_kl_f32<2, true, TZ>);
    else if (f.TR == 4) go(A ? k_kl_f32<4, false, TZ> : k_kl_f32<4, true, TZ>);
    else go(A ? k_kl_f32<8, false, TZ> : k_kl_f32<8, true, TZ>);
    if (A) cudaFreeAsync(A, st);
}
}  // namespace

extern "C" size_t kl_prepared_bytes(int64_t npts, int32_t M, int32_t mode)
{
    clear_error();
    if (npts < 1 || M < 1) return 0;
    switch (mode) {
    case MSG_GEMM_FP64: return align256(sizeof(double) * npts * M) + align256(sizeof(double) * M);
    case MSG_GEMM_FP32: return align256(sizeof(float) * npts * M) + align256(sizeof(double) * M);
    case MSG_GEMM_BF16X3:
    case MSG_GEMM_TF32: return kl_tc_prepared_bytes(npts, M, mode);
    default: return 0;
    }
}

extern "C" int32_t kl_prepare(const double* Phi, const double* sqrt_lambda, int64_t npts, int32_t M, int32_t mode,
                              void* prepared, size_t prepared_bytes, void* stream)
{
    clear_error();
    if (npts < 1 || M < 1 || !Phi || !sqrt_lambda || !prepared) {
        set_error("kl_prepare: invalid arguments");
        return MSG_ERR_INVALID;
    }
    size_t need = kl_prepared_bytes(npts, M, mode);
    if (need == 0) { set_error("kl_prepare: unknown mode"); return MSG_ERR_INVALID; }
    if (prepared_bytes < need) { set_error("kl_prepare: buffer too small"); return MSG_ERR_WORKSPACE; }
    cudaStream_t st = (cudaStream_t)stream;
    char* base = (char*)prepared;
    if (mode == MSG_GEMM_BF16X3 || mode == MSG_GEMM_TF32) {
        if ((uintptr_t)prepared % 256) { set_error("kl_prepare: prepared buffer must be 256-byte aligned"); return MSG_ERR_INVALID; }
        return kl_tc_prepare(Phi, sqrt_lambda, npts, M, mode, prepared, st);
    }
    if (mode == MSG_GEMM_FP64) {
        MSG_CUDA_TRY(cudaMemcpyAsync(base, Phi, sizeof(double) * npts * M, cudaMemcpyDeviceToDevice, st));
        MSG_CUDA_TRY(cudaMemcpyAsync(base + align256(sizeof(double) * npts * M), sqrt_lambda, sizeof(double) * M,
                                     cudaMemcpyDeviceToDevice, st));
    } else {
        prof_begin(K_KL, st);
        k_to_float<<<152 * 8, 256, 0, st>>>(Phi, (float*)base, npts * M);
        prof_end(K_KL, st, 12.0 * npts * M, 0.0);
        MSG_CHECK_LAUNCH();
        MSG_CUDA_TRY(cudaMemcpyAsync(base + align256(sizeof(float) * npts * M), sqrt_lambda, sizeof(double) * M,
                                     cudaMemcpyDeviceToDevice, st));
    }
    return MSG_OK;
}

extern "C" int32_t sample_field(const void* prepared, int64_t npts, int32_t M, int32_t mode, const double* xi,
                                int64_t S, void* Z, int32_t z_fp32, void* stream)
{
    clear_error();
    if (npts < 1 || M < 1 || S < 0) { set_error("sample_field: invalid sizes"); return MSG_ERR_INVALID; }
    if (S == 0) return MSG_OK;
    if (!prepared || !xi || !Z) { set_error("sample_field: NULL pointer"); return MSG_ERR_INVALID; }
    cudaStream_t st = (cudaStream_t)stream;
    if (mode == MSG_GEMM_BF16X3 || mode == MSG_GEMM_TF32) {
        if ((uintptr_t)prepared % 256) { set_error("sample_field: prepared buffer must be 256-byte aligned"); return MSG_ERR_INVALID; }
        return kl_tc_sample(prepared, npts, M, mode, xi, S, Z, z_fp32, st);
    }
    if (S > 65535LL * 64) { set_error("sample_field: too many samples for one call"); return MSG_ERR_INVALID; }
    const char* base = (const char*)prepared;
    const double pe = mode == MSG_GEMM_FP64 ? 8.0 : 4.0, ze = z_fp32 ? 4.0 : 8.0;
    if (mode != MSG_GEMM_FP64 && mode != MSG_GEMM_FP32) {
        set_error("sample_field: unknown mode");
        return MSG_ERR_INVALID;
    }
    prof_begin(K_KL, st);
    if (mode == MSG_GEMM_FP64) {
        const double* Phi = (const double*)base;
        const double* sl = (const double*)(base + align256(sizeof(double) * npts * M));
        const int64_t xt = (npts + 31) / 32, tiles = xt * ((S + 7) / 8);
        if (tiles > 0x7fffffffLL) { set_error("sample_field: too many points and samples for one call"); return MSG_ERR_INVALID; }
        if (z_fp32) k_kl_f64<float><<<(unsigned)tiles, 256, 0, st>>>(Phi, sl, xi, npts, M, S, xt, (float*)Z);
        else k_kl_f64<double><<<(unsigned)tiles, 256, 0, st>>>(Phi, sl, xi, npts, M, S, xt, (double*)Z);
    } else {
        const float* Phi = (const float*)base;
        const double* sl = (const double*)(base + align256(sizeof(float) * npts * M));
        if (z_fp32) kl_fp32<float>(Phi, sl, xi, npts, M, S, (float*)Z, st);
        else kl_fp32<double>(Phi, sl, xi, npts, M, S, (double*)Z, st);
    }
    prof_end(K_KL, st, pe * npts * M + 8.0 * S * M + ze * S * npts, 2.0 * npts * M * S);
    MSG_CHECK_LAUNCH();
    return MSG_OK;
}
