// kl_tc.cu -- KL contraction Z = Phi diag(sqrt(lambda)) xi on the 5th-generation
// tensor cores (tcgen05) with FP32 accumulation, in two operand modes:
//   BF16X3  each operand v is split into bf16 parts v = hi + lo + O(2^-16 |v|) and
//           the product uses hi*hi + hi*lo + lo*hi (kind::f16), about 1e-5 of
//           sum_m |A B| -- the lo*lo term and the remainders are below the FP32
//           accumulation of a 400-term sum of unit-scale products;
//   TF32    both operands rounded to TF32 (10-bit mantissa, round to nearest) and
//           one product per term (kind::tf32), about 1e-3 of sum_m |A B|.
// Neither is the FP64 path; the sampler's error is stated per result in the tests
// and the bench.
//
// Z[s][x] = sum_m A[s][m] B[x][m] with A = sqrt(lambda) * xi (samples x terms)
// and B = Phi (points x terms), as zero-padded [rows][Kp] part arrays: B's are made
// once per basis by kl_tc_prepare, A's once per call in a stream-ordered temporary.
//
// k_kl_tc is persistent, one CTA per SM over tiles of 128 samples x 256 points, with
// a role per warp:
//   warp 0   loads: TMA tiles of both operands, 32 terms a stage (64 bytes of a row in
//            bf16, 128 in TF32) in the swizzled K-major layout the UMMA descriptors
//            expect, through a ring of 4 stages of 48 KB (with 2 stages of 64 terms one
//            load at a time was in flight: 2.11 ms for the BF16X3 size below);
//   warp 1   issues the MMAs of a stage and commits them to its "empty" barrier, and the
//            last of a tile to the accumulator's "full" barrier;
//   warps 4-11  epilogue: 32 x 32 accumulator blocks through a padded shared tile, so that
//            every global store of a warp writes 32 consecutive points of one sample.
// Two accumulators of 256 TMEM columns alternate, so the loads and MMAs of the next tile
// run under the stores of the last.  Bound by the tensor pipe (BF16X3: three products a
// term) and by the Z stores; with the three steps of a tile one after the other in
// 152 x 54 CTAs it took 3.58 ms for 1024 x 1024 points, 400 terms, 1024 samples in
// BF16X3, now 1.90 ms; 257 x 129 points, 300 terms, 777
// samples, FP64 fields in TF32: 113 -> 76 us.
// Sample tiles are the fastest tile index: the CTAs that read one Phi tile run together
// and find it in L2 (A is small and stays there).  Every wait is bounded; one that runs
// out sets a device flag (read by msg_device_status), ends every role and leaves
// the rest of the output unwritten.
#include <cuda.h>

#include <cuda_bf16.h>

#include <algorithm>
#include <type_traits>

#include "common.cuh"
#include "kl_tc.cuh"
#include "prof.cuh"

namespace msg {

namespace {

constexpr int kTM = 128;  // samples per tile (UMMA M)
constexpr int kTN = 256;  // points per tile (UMMA N); the part arrays are padded to whole tiles
constexpr int kSMs = 152;
// tiles of 128 and 64 points: of a call with few tiles
constexpr int kThreadsTC = 384;
template <int TN> constexpr int stages() { return TN == kTN ? 4 : TN == 128 ? 6 : 8; }  // of 48, 32 and 24 KB
constexpr long long kSpinLimit = 1ll << 22;           // bounded mbarrier waits (seconds)

// Operand modes of the tensor-core kernel.
enum { TC_BF16X3 = 0, TC_TF32 = 1 };
template <int MODE> struct TcCfg;
template <> struct TcCfg<TC_BF16X3> {
    typedef __nv_bfloat16 E;
    static constexpr int parts = 2;   // hi, lo
    static constexpr int TK = 32;        // terms a stage
    static constexpr int row_bytes = 64; // one swizzled K row of a stage
    static constexpr int pad = 64;       // rows of the part arrays are padded to this many terms
};
template <> struct TcCfg<TC_TF32> {
    typedef float E;
    static constexpr int parts = 1;
    static constexpr int TK = 32;
    static constexpr int row_bytes = 128;
    static constexpr int pad = 32;
};
template <int MODE> constexpr int a_bytes() { return kTM * TcCfg<MODE>::row_bytes; }  // per part and stage
template <int MODE, int TN> constexpr int b_bytes() { return TN * TcCfg<MODE>::row_bytes; }
template <int MODE, int TN> constexpr int stage_bytes() { return TcCfg<MODE>::parts * (a_bytes<MODE>() + b_bytes<MODE, TN>()); }
constexpr int kEpiBytes = 8 * 32 * 33 * 4;  // a padded 32 x 32 block per epilogue warp
template <int MODE, int TN> constexpr int smem_bytes() { return stages<TN>() * stage_bytes<MODE, TN>() + kEpiBytes + 1024; }  // + alignment slack

__host__ __device__ inline int64_t round_up(int64_t a, int64_t b) { return (a + b - 1) / b * b; }

__device__ int g_tc_error;  // set by a kernel whose mbarrier wait ran out (sticky until msg_device_status)

// tcgen05 shared-memory matrix descriptor: start address >> 4 in bits 0-13,
// leading byte offset >> 4 in 16-29 (unused by swizzled K-major tiles),
// stride byte offset >> 4 in 32-45 (the next atom of 8 rows), descriptor
// version 1 in bits 46-47, swizzle mode in bits 61-63 (2: 128-byte, 4: 64-byte).
template <int MODE>
__device__ __forceinline__ uint64_t smem_desc(uint32_t saddr)
{
    constexpr int row = TcCfg<MODE>::row_bytes;
    return (uint64_t)((saddr >> 4) & 0x3FFF) | ((uint64_t)(16 >> 4) << 16) | ((uint64_t)(8 * row >> 4) << 32) | (1ull << 46) |
           ((row == 128 ? 2ull : 4ull) << 61);
}

// Instruction descriptor: D = F32 (bits 4-5 = 1); A and B formats in bits 7-9
// and 10-12 (kind::f16: 1 = BF16; kind::tf32: 2 = TF32), both K-major;
// N >> 3 in bits 17-22, M >> 4 in bits 24-28.
template <int MODE, int TN>
__host__ __device__ constexpr uint32_t instr_desc()
{
    return (1u << 4) | ((MODE == TC_TF32 ? 2u : 1u) << 7) | ((MODE == TC_TF32 ? 2u : 1u) << 10) |
           ((uint32_t)(TN >> 3) << 17) | ((uint32_t)(kTM >> 4) << 24);
}

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

// Wait until the mbarrier phase with the given parity has completed; false when the
// limit runs out or another role gave up (*dead, which is then set).
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, volatile int* dead)
{
    const uint32_t a = smem_u32(bar);
    for (long long it = 0; it < kSpinLimit; ++it) {
        uint32_t done;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(done)
            : "r"(a), "r"(parity)
            : "memory");
        if (done) return true;
        if ((it & 15) == 15 && *dead) return false;
    }
    *dead = 1;
    return false;
}

// The same for a whole warp, which goes on or gives up as one: its lanes can see the end of
// the phase and the giving up on different sides of each other, and the warp-wide TMEM load
// behind the wait needs every lane.
__device__ __forceinline__ bool warp_wait(uint64_t* bar, uint32_t parity, volatile int* dead)
{
    return __all_sync(0xffffffffu, mbar_wait(bar, parity, dead));
}

__device__ __forceinline__ void mbar_expect(uint64_t* bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

// The box of `map` at element x (a multiple of 64 bytes) and row y into shared memory.
__device__ __forceinline__ void tma_load(uint32_t dst, const CUtensorMap* map, int x, int y, uint64_t* bar)
{
    asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(dst),
                 "l"(map), "r"(x), "r"(y), "r"(smem_u32(bar))
                 : "memory");
}

template <int MODE, int TN>
__device__ __forceinline__ void mma(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t acc)
{
    if constexpr (MODE == TC_TF32)
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "setp.ne.b32 p, %4, 0;\n\t"
            "tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n\t}"
            ::"r"(tmem_d), "l"(adesc), "l"(bdesc), "r"(instr_desc<MODE, TN>()), "r"(acc)
            : "memory");
    else
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "setp.ne.b32 p, %4, 0;\n\t"
            "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
            ::"r"(tmem_d), "l"(adesc), "l"(bdesc), "r"(instr_desc<MODE, TN>()), "r"(acc)
            : "memory");
}

__device__ __forceinline__ void mma_commit(uint64_t* bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
                 : "memory");
}

// 32 consecutive FP32 accumulator columns of this thread's TMEM lane.
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float* v)
{
    uint32_t r[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
        "%15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
          "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
          "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int k = 0; k < 32; ++k) v[k] = __uint_as_float(r[k]);
}

// Split of FP64 values into bf16 hi/lo.
__device__ __forceinline__ void split2(double v, __nv_bfloat16& hi, __nv_bfloat16& lo)
{
    hi = __double2bfloat16(v);
    lo = __double2bfloat16(v - (double)__bfloat162float(hi));
}

// FP64 -> TF32 (round to nearest, ties away), kept in an FP32 container.
__device__ __forceinline__ float to_tf32(double v)
{
    uint32_t r;
    asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"((float)v));
    return __uint_as_float(r);
}

// Operand conversion of 8 consecutive terms into the parts of one 16-byte chunk
// (BF16X3: 8 terms -> 16 bytes per part; TF32: 4 terms -> 16 bytes).
__global__ void k_split_phi(const double* Phi, int64_t npts, int M, int64_t Kp, int64_t Np, __nv_bfloat16* Bhi,
                            __nv_bfloat16* Blo)
{
    const int64_t n = Np * Kp;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x) {
        const int64_t x = e / Kp, m = e % Kp;
        double v = (x < npts && m < M) ? Phi[x * M + m] : 0.0;
        __nv_bfloat16 h, l;
        split2(v, h, l);
        Bhi[e] = h;
        Blo[e] = l;
    }
}

__global__ void k_tf32_phi(const double* Phi, int64_t npts, int M, int64_t Kp, int64_t Np, float* B)
{
    const int64_t n = Np * Kp;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x) {
        const int64_t x = e / Kp, m = e % Kp;
        B[e] = (x < npts && m < M) ? to_tf32(Phi[x * M + m]) : 0.f;
    }
}

// A = sqrt(lambda) * xi converted once per call into zero-padded [Sp][Kp] part
// arrays in the operand format (the main loop then only copies); a warp per row.
template <int MODE>
__global__ void k_prep_a(const double* sl, const double* xi, int64_t S, int M, int Kp, int64_t Sp,
                         typename TcCfg<MODE>::E* A0, typename TcCfg<MODE>::E* A1)
{
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int64_t s = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (s >= Sp) return;
    for (int m = threadIdx.x & 31; m < Kp; m += 32) {
        const double v = (s < S && m < M) ? sl[m] * xi[s * M + m] : 0.0;
        const int64_t e = s * Kp + m;
        if constexpr (MODE == TC_TF32) {
            A0[e] = to_tf32(v);
        } else {
            __nv_bfloat16 h, l;
            split2(v, h, l);
            A0[e] = h;
            A1[e] = l;
        }
    }
}

// tile t: samples 128 (t mod stiles) .., points TN (t / stiles) ..; the second part of an
// operand follows the first, so one map covers both
template <int MODE, int TN, class TZ>
__global__ void __launch_bounds__(kThreadsTC, 1)
    k_kl_tc(const __grid_constant__ CUtensorMap mA, const __grid_constant__ CUtensorMap mB, int64_t npts, int nchunks,
            int64_t S, int stiles, int xtiles, int Np, TZ* __restrict__ Z)
{
    constexpr int parts = TcCfg<MODE>::parts, TK = TcCfg<MODE>::TK, NST = stages<TN>(), kAbytes = a_bytes<MODE>(),
                  kBbytes = b_bytes<MODE, TN>(), kStage = stage_bytes<MODE, TN>();
    extern __shared__ unsigned char smem_raw[];
    __shared__ __align__(8) uint64_t full[NST], empty[NST], acc_full[2], acc_empty[2];
    __shared__ uint32_t tmem_base_slot;
    __shared__ volatile int dead;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, ntiles = stiles * xtiles;
    // 1024-aligned stage buffers (swizzle atoms must start on 1024 bytes)
    const uint32_t raw = smem_u32(smem_raw);
    unsigned char* base = smem_raw + (((raw + 1023) & ~1023u) - raw);

    if (warp == 0) {  // TMEM: 128 lanes x 2 TN FP32 columns, two accumulators
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_slot)),
                     "r"(2 * TN)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid == 0) {
        for (int k = 0; k < NST; ++k) {
            mbar_init(&full[k], 1);
            mbar_init(&empty[k], 1);
        }
        for (int k = 0; k < 2; ++k) {
            mbar_init(&acc_full[k], 1);
            mbar_init(&acc_empty[k], 8);
        }
        dead = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = tmem_base_slot;
    auto stage = [&](int n) { return smem_u32(base + (n % NST) * kStage); };  // A parts, then B parts

    if (warp == 0 && lane == 0) {  // ---- loads
        int n = 0;  // stages filled
        bool ok = true;
        // this kernel starts under k_prep_a, which writes A: its barriers and TMEM are ready by
        // then (2 to 3 us of a call: 256 x 100 points, 300 terms, FP32 fields 19.9 -> 16.8 us)
        asm volatile("griddepcontrol.wait;" ::: "memory");
        for (int t = blockIdx.x; t < ntiles && ok; t += gridDim.x) {
            const int s0 = (t % stiles) * kTM, x0 = (t / stiles) * TN;
            for (int kc = 0; kc < nchunks; ++kc, ++n) {
                if (n >= NST && !(ok = mbar_wait(&empty[n % NST], ((n / NST) - 1) & 1, &dead))) break;
                uint64_t* bar = &full[n % NST];
                const uint32_t d = stage(n);
                mbar_expect(bar, kStage);
                tma_load(d, &mA, kc * TK, s0, bar);
                if constexpr (parts == 2) tma_load(d + kAbytes, &mA, kc * TK, stiles * kTM + s0, bar);
                tma_load(d + parts * kAbytes, &mB, kc * TK, x0, bar);
                if constexpr (parts == 2) tma_load(d + parts * kAbytes + kBbytes, &mB, kc * TK, Np + x0, bar);
            }
        }
        // copies in flight end before the CTA does (normally the MMAs have waited for them)
        for (int k = n > NST ? n - NST : 0; k < n; ++k) {
            int none = 0;
            mbar_wait(&full[k % NST], (k / NST) & 1, &none);
        }
    } else if (warp == 1 && lane == 0) {  // ---- MMAs
        int n = 0, w = 0;  // stages read, tiles done
        bool ok = true;
        for (int t = blockIdx.x; t < ntiles && ok; t += gridDim.x, ++w) {
            const uint32_t acc = tmem + (uint32_t)((w & 1) * TN);
            if (w >= 2 && !(ok = mbar_wait(&acc_empty[w & 1], ((w >> 1) - 1) & 1, &dead))) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            for (int kc = 0; kc < nchunks; ++kc, ++n) {
                if (!(ok = mbar_wait(&full[n % NST], (n / NST) & 1, &dead))) break;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint32_t a0 = stage(n), b0 = a0 + parts * kAbytes;
#pragma unroll
                for (int ks = 0; ks < TcCfg<MODE>::row_bytes / 32; ++ks) {  // MMA K steps of 32 bytes
                    const uint32_t ko = ks * 32;
                    const uint32_t first = (kc == 0 && ks == 0) ? 0u : 1u;
                    mma<MODE, TN>(acc, smem_desc<MODE>(a0 + ko), smem_desc<MODE>(b0 + ko), first);
                    if constexpr (MODE == TC_BF16X3) {
                        mma<MODE, TN>(acc, smem_desc<MODE>(a0 + ko), smem_desc<MODE>(b0 + kBbytes + ko), 1u);  // hi * lo
                        mma<MODE, TN>(acc, smem_desc<MODE>(a0 + kAbytes + ko), smem_desc<MODE>(b0 + ko), 1u);  // lo * hi
                    }
                }
                mma_commit(&empty[n % NST]);
            }
            if (ok) mma_commit(&acc_full[w & 1]);
        }
        // MMAs in flight end before the memory they use is given back (normally the epilogue
        // has waited for them)
        if (!ok && n > 0) {
            int none = 0;
            mbar_wait(&empty[(n - 1) % NST], ((n - 1) / NST) & 1, &none);
        }
    } else if (warp >= 4) {  // ---- epilogue
        // warp w reads TMEM lanes 32 (w % 4) .. + 31 (samples), columns TN / 2 ((w - 4) / 4) .. (points)
        const int lane_base = 32 * (warp & 3), col_base = TN / 2 * ((warp - 4) >> 2);
        const uint32_t tile = smem_u32(base + NST * kStage) + (warp - 4) * 32 * 33 * 4;
        const uint32_t mine = tile + lane * 33 * 4, column = tile + lane * 4;
        int w = 0;
        for (int t = blockIdx.x; t < ntiles; t += gridDim.x, ++w) {
            const int64_t s0 = (int64_t)(t % stiles) * kTM + lane_base, x0 = (int64_t)(t / stiles) * TN + col_base;
            if (!warp_wait(&acc_full[w & 1], (w >> 1) & 1, &dead)) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint32_t acc = tmem + ((uint32_t)lane_base << 16) + (uint32_t)((w & 1) * TN + col_base);
            const int rows = (int)min((int64_t)32, S - s0);  // may be <= 0
            for (int cb = 0; cb < TN / 2; cb += 32) {
                float v[32];
                tmem_ld32(acc + (uint32_t)cb, v);
                if (cb == TN / 2 - 32) {  // the accumulator is in registers: the MMAs may have it back
                    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&acc_empty[w & 1]);
                }
#pragma unroll
                for (int k = 0; k < 32; ++k) asm volatile("st.shared.f32 [%0], %1;" ::"r"(mine + 4 * k), "f"(v[k]) : "memory");
                __syncwarp();
                const int64_t x = x0 + cb + lane;
                TZ* z = Z + s0 * npts + x;
                if (x < npts) {
#pragma unroll
                    for (int r0 = 0; r0 < 32; r0 += 16) {  // 16 loads in flight, then their stores
                        float o[16];
#pragma unroll
                        for (int k = 0; k < 16; ++k)
                            asm volatile("ld.shared.f32 %0, [%1];" : "=f"(o[k]) : "r"(column + (r0 + k) * 33 * 4) : "memory");
                        store_wide<16>(z + r0 * npts, npts, o, rows - r0);
                    }
                }
                __syncwarp();
            }
        }
    }
    __syncwarp();
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (tid == 0 && dead) atomicExch(&g_tc_error, 1);
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(2 * TN) : "memory");
}

struct TcLayout {
    int64_t Kp, Np;
    size_t p0, p1, sl, total;
};

TcLayout tc_layout(int64_t npts, int32_t M, int mode)
{
    TcLayout L{};
    const bool tf = mode == TC_TF32;
    L.Kp = round_up(M, tf ? TcCfg<TC_TF32>::pad : TcCfg<TC_BF16X3>::pad);
    L.Np = round_up(npts, kTN);
    const size_t part = (size_t)L.Np * L.Kp * (tf ? sizeof(float) : sizeof(__nv_bfloat16));
    L.p0 = 0;
    L.p1 = (part + 255) / 256 * 256;
    L.sl = tf ? L.p1 : 2 * L.p1;
    L.total = L.sl + ((sizeof(double) * M + 255) / 256 * 256);
    return L;
}

int tc_mode(int32_t gemm_mode) { return gemm_mode == MSG_GEMM_TF32 ? TC_TF32 : TC_BF16X3; }

// cuTensorMapEncodeTiled through the runtime (no link against the driver library).
typedef CUresult (*EncodeFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                             const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                             CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
EncodeFn encode_fn()
{
    static const EncodeFn fn = [] {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) != cudaSuccess ||
            q != cudaDriverEntryPointSuccess)
            p = nullptr;
        return (EncodeFn)p;
    }();
    return fn;
}

// Map of a [rows][Kp] part array in boxes of one stage's terms x box_rows.
template <int MODE>
bool part_map(CUtensorMap* m, const void* p, int64_t rows, int64_t Kp, int box_rows)
{
    typedef typename TcCfg<MODE>::E E;
    const cuuint64_t dim[2] = {(cuuint64_t)Kp, (cuuint64_t)rows}, stride[1] = {(cuuint64_t)(Kp * sizeof(E))};
    const cuuint32_t box[2] = {(cuuint32_t)TcCfg<MODE>::TK, (cuuint32_t)box_rows}, es[2] = {1, 1};
    return encode_fn()(m, MODE == TC_TF32 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2,
                       const_cast<void*>(p), dim, stride, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
                       TcCfg<MODE>::row_bytes == 128 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B,
                       CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <int MODE, int TN, class TZ>
int tc_launch(const TcLayout& L, const char* b, int64_t npts, int32_t M, const double* xi, int64_t S, void* Z,
              cudaStream_t st)
{
    typedef typename TcCfg<MODE>::E E;
    constexpr int parts = TcCfg<MODE>::parts;
    const int64_t Sp = round_up(S, kTM), stiles = Sp / kTM, xtiles = (npts + TN - 1) / TN;
    if (stiles * xtiles > 0x7fffffffLL || 2 * Sp > 0x7fffffffLL || 2 * L.Np > 0x7fffffffLL) {
        set_error("sample_field: too many samples for one call");
        return MSG_ERR_INVALID;
    }
    const size_t apart = (size_t)Sp * L.Kp * sizeof(E);
    if (!encode_fn()) { set_error("cuTensorMapEncodeTiled is not available"); return MSG_ERR_UNSUPPORTED; }
    // the converted A lives in a stream-ordered temporary, freed after the contraction
    char* abuf = nullptr;
    MSG_CUDA_TRY(temp_alloc((void**)&abuf, parts * apart, st));
    E* A0 = (E*)abuf;
    E* A1 = parts == 2 ? (E*)(abuf + apart) : A0;
    // (a part of B is whole tiles of whole 128-byte rows: the next starts right behind it)
    CUtensorMap mA, mB;
    const bool mapped = part_map<MODE>(&mA, A0, parts * Sp, L.Kp, kTM) && part_map<MODE>(&mB, b + L.p0, parts * L.Np, L.Kp, TN);
    cudaError_t e = mapped ? cudaSuccess : cudaErrorInvalidValue;
    if (e == cudaSuccess) {
        k_prep_a<MODE><<<(unsigned)((Sp + 7) / 8), 256, 0, st>>>((const double*)(b + L.sl), xi, S, M, (int)L.Kp, Sp, A0, A1);
        prof_also();
        e = cudaGetLastError();
    }
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_kl_tc<MODE, TN, TZ>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_bytes<MODE, TN>());
    if (e == cudaSuccess) {
        cudaLaunchConfig_t cfg{};
        cudaLaunchAttribute at{};
        at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
        at.val.programmaticStreamSerializationAllowed = 1;
        cfg.gridDim = dim3((unsigned)std::min<int64_t>(stiles * xtiles, kSMs));
        cfg.blockDim = dim3(kThreadsTC);
        cfg.dynamicSmemBytes = smem_bytes<MODE, TN>();
        cfg.stream = st;
        cfg.attrs = &at;
        cfg.numAttrs = 1;
        e = cudaLaunchKernelEx(&cfg, k_kl_tc<MODE, TN, TZ>, mA, mB, npts, (M + TcCfg<MODE>::TK - 1) / TcCfg<MODE>::TK, S,
                               (int)stiles, (int)xtiles, (int)L.Np, (TZ*)Z);
    }
    cudaFreeAsync(abuf, st);
    if (e != cudaSuccess) { set_error(std::string("sample_field: ") + cudaGetErrorString(e)); return MSG_ERR_CUDA; }
    return MSG_OK;
}

}  // namespace

size_t kl_tc_prepared_bytes(int64_t npts, int32_t M, int32_t mode) { return tc_layout(npts, M, tc_mode(mode)).total; }

int32_t kl_tc_prepare(const double* Phi, const double* sqrt_lambda, int64_t npts, int32_t M, int32_t mode,
                      void* prepared, cudaStream_t st)
{
    const int tm = tc_mode(mode);
    const TcLayout L = tc_layout(npts, M, tm);
    char* b = (char*)prepared;
    prof_begin(K_KL, st);
    if (tm == TC_TF32)
        k_tf32_phi<<<152 * 8, 256, 0, st>>>(Phi, npts, M, L.Kp, L.Np, (float*)(b + L.p0));
    else
        k_split_phi<<<152 * 8, 256, 0, st>>>(Phi, npts, M, L.Kp, L.Np, (__nv_bfloat16*)(b + L.p0),
                                              (__nv_bfloat16*)(b + L.p1));
    prof_end(K_KL, st, 8.0 * npts * M + 4.0 * L.Np * L.Kp, 0.0);
    MSG_CHECK_LAUNCH();
    MSG_CUDA_TRY(cudaMemcpyAsync(b + L.sl, sqrt_lambda, sizeof(double) * M, cudaMemcpyDeviceToDevice, st));
    return MSG_OK;
}

int32_t kl_tc_sample(const void* prepared, int64_t npts, int32_t M, int32_t mode, const double* xi, int64_t S, void* Z,
                     int32_t z_fp32, cudaStream_t st)
{
    const int tm = tc_mode(mode);
    const TcLayout L = tc_layout(npts, M, tm);
    if ((npts + kTN - 1) / kTN > 65535) { set_error("sample_field: too many points for one call"); return MSG_ERR_INVALID; }
    const char* b = (const char*)prepared;
    prof_begin(K_KL, st);
    // The widest tiles, unless narrower ones still give every tile an SM of its own: up to four
    // times the CTAs, each with a fraction of the loads and stores (100 x 60 points, 400
    // terms, 100 samples: BF16X3 28.7 -> 18.5 us a call, TF32 23.2 -> 15.2; 256 x 50 points, 300
    // terms, FP32 fields: 15.9 us in tiles of 128, 20.5 in twice as many of 64 (2 us of it
    // the start under k_prep_a); 256 x 100: 16.8 us in tiles of 256).
    // The sums are the same, term by term.
    const int64_t tiles = ((npts + kTN - 1) / kTN) * ((S + kTM - 1) / kTM);
    int rc;
    auto go = [&](auto mode, auto tn) {
        constexpr int MD = decltype(mode)::value, TN = decltype(tn)::value;
        return z_fp32 ? tc_launch<MD, TN, float>(L, b, npts, M, xi, S, Z, st) : tc_launch<MD, TN, double>(L, b, npts, M, xi, S, Z, st);
    };
    auto pick = [&](auto mode) {
        if (4 * tiles <= kSMs) return go(mode, std::integral_constant<int, 64>());
        if (2 * tiles <= kSMs) return go(mode, std::integral_constant<int, 128>());
        return go(mode, std::integral_constant<int, kTN>());
    };
    if (tm == TC_TF32) rc = pick(std::integral_constant<int, TC_TF32>());
    else rc = pick(std::integral_constant<int, TC_BF16X3>());
    if (rc != MSG_OK) return rc;
    // algorithmic work: (3 split products or 1) of 2 npts M S flops; bytes: Phi parts, xi, Z
    const double parts = tm == TC_TF32 ? 1.0 : 3.0, pbytes = tm == TC_TF32 ? 4.0 : 4.0;
    prof_end(K_KL, st, pbytes * npts * M + 8.0 * S * M + (z_fp32 ? 4.0 : 8.0) * S * npts, 2.0 * parts * npts * M * S);
    MSG_CHECK_LAUNCH();
    // a bounded wait that runs out sets g_tc_error (reported by msg_device_status)
    return MSG_OK;
}

}  // namespace msg

extern "C" int32_t msg_device_status(void)
{
    msg::clear_error();
    MSG_CUDA_TRY(cudaDeviceSynchronize());
    int err = 0, zero = 0;
    MSG_CUDA_TRY(cudaMemcpyFromSymbol(&err, msg::g_tc_error, sizeof(int)));
    MSG_CUDA_TRY(cudaMemcpyToSymbol(msg::g_tc_error, &zero, sizeof(int)));
    if (err) {
        msg::set_error("a bounded wait in a tensor-core kernel ran out; its output is incomplete");
        return MSG_ERR_TIMEOUT;
    }
    return MSG_OK;
}
