// Dense contractions of blocked large-chi networks on the tensor cores
// (tcgen05), and the exact contraction of 2D grid networks built on them.
//
// The paper's own benchmarks group patches of the lattice into single tensors
// of bond dimension chi = 16 or 64 (App. A) and contract the resulting small
// networks exactly (Sec. III, IV.A).  At such bond dimensions the exact
// contraction is a chain of dense matrix products: a 2D grid contracted row
// by row keeps a running tensor over the open legs, and absorbing one site is
//     out[rest][d][h'] = sum_{u,h} in[u][rest][h] * T[h, u, h', d],
// a GEMM with M = |rest| (up to chi^(w-1) for width w), K = chi_u chi_h and
// N = chi_d chi_h' (256 each at chi = 16).  The running tensor is kept in a
// "ring" order -- the legs still to be contracted from above first, then the
// legs already produced, then the horizontal leg -- so the site's two input
// legs sit at the two ends and its two output legs are appended at the end:
// the next site finds its own legs at the ends again, across rows too.
//
// The large products run on one persistent kernel (tc_stream_kernel: operand
// stages filled by the Tensor Memory Accelerator, tcgen05.mma with M = 128,
// N <= 256 and FP32 accumulation in tensor memory, a finished tile stored while
// the next accumulates); products whose A is not on 16-byte boundaries get there
// behind a padded copy of A where many columns repay it (launch_padded_stream).
// Small products of pne_dense_gemm, and the unaligned ones that are shallow or
// narrow (launch_tc has the rule), take tc_gemm_kernel: one CTA per tile, K staged
// 128 bytes per row at a time in two shared-memory stages written by all
// threads in the canonical no-swizzle K-major layout (8-row x 16-byte core
// matrices, the two core matrices of one MMA K step 128 bytes apart, 8-row
// groups 1024 bytes apart), each stage committed to an mbarrier on which the
// loaders wait (bounded) before refilling it.  Both add a K step of 32 bytes at
// a time in the same order, so their results are the same bit for bit.  The
// grid's steps record the largest |entry| per set, from which the next step
// takes a power-of-two scale (kept exactly in a log-2 counter).  The FP64 form
// (f64_gemm_kernel) does the same products on the CUDA cores: the reference the
// reduced-precision forms are stated against.
#include <cuda.h>
#include <cuda_runtime.h>
#include <cooperative_groups.h>
#include <cuda_bf16.h>
#include <cudaTypedefs.h>

#include <mutex>

#include <algorithm>
#include <cmath>
#include <cstdlib>
#include <cstring>
#include <string>
#include <type_traits>
#include <vector>

#include "pne_internal.h"

namespace pne {
namespace cg = cooperative_groups;
namespace {

constexpr int kTcThreads = 128;
constexpr int kTcBM = 128;
constexpr int kChunk = 128;                   // K bytes per row per stage
constexpr int kATileBytes = kTcBM * kChunk;   // 16 KB
constexpr uint64_t kWaitNs = 2000000000ull;   // bounded mbarrier waits: 2 s

// ---------------------------------------------------------------- PTX wrappers
__device__ __forceinline__ uint32_t smem_addr(const void *p)
{
    return (uint32_t)__cvta_generic_to_shared(p);
}

// shared-memory matrix descriptor: start address, leading (K) and stride (M/N)
// byte offsets between core matrices, descriptor version 1, no swizzle
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr, uint32_t lbo, uint32_t sbo)
{
    uint64_t d = 0;
    d |= (uint64_t)((addr & 0x3FFFFu) >> 4);
    d |= (uint64_t)((lbo >> 4) & 0x3FFFu) << 16;
    d |= (uint64_t)((sbo >> 4) & 0x3FFFu) << 32;
    d |= (uint64_t)1 << 46;
    return d;
}

// instruction descriptor: FP32 accumulator, A and B of one format (2 = TF32
// for kind::tf32, 1 = BF16 for kind::f16), both K-major, M and N
__host__ __device__ constexpr uint32_t instr_desc(uint32_t fmt, uint32_t M, uint32_t N)
{
    return (1u << 4) | (fmt << 7) | (fmt << 10) | ((N >> 3) << 17) | ((M >> 4) << 24);
}

__device__ __forceinline__ void tmem_alloc(uint32_t dst_smem, uint32_t ncols)
{
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(dst_smem), "r"(ncols)
                 : "memory");
}
__device__ __forceinline__ void tmem_relinquish()
{
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols)
{
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
__device__ __forceinline__ void tc_fence_after()
{
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_before()
{
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void fence_proxy_async()
{
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
template <int EB>
__device__ __forceinline__ void tc_mma(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc)
{
    if (EB == 4)
        asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                     "tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(d),
                     "l"(a), "l"(b), "r"(idesc), "r"(acc)
                     : "memory");
    else
        asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                     "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(d),
                     "l"(a), "l"(b), "r"(idesc), "r"(acc)
                     : "memory");
}
__device__ __forceinline__ void tc_commit(uint32_t mbar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(mbar)
                 : "memory");
}
__device__ __forceinline__ void mbar_init(uint32_t addr, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(addr), "r"(count) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t addr, uint32_t parity)
{
    uint32_t ok;
    asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
                 "selp.u32 %0, 1, 0, p;\n\t}\n"
                 : "=r"(ok)
                 : "r"(addr), "r"(parity)
                 : "memory");
    return ok != 0;
}
__device__ __forceinline__ uint64_t global_ns()
{
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}
// bounded wait (about two seconds of the global timer); false when it gave up
__device__ __forceinline__ bool mbar_wait(uint32_t addr, uint32_t parity)
{
    // reading the timer costs more than most waits: not before a few tries
    for (int i = 0; i < 32; ++i)
        if (mbar_try_wait(addr, parity)) return true;
    const uint64_t t0 = global_ns();
    for (;;) {
        if (mbar_try_wait(addr, parity)) return true;
        if (global_ns() - t0 > kWaitNs) return false;
    }
}
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&r)[16])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, "
                 "%13, %14, %15}, [%16];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
                   "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]),
                   "=r"(r[15])
                 : "r"(taddr)
                 : "memory");
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t to_tf32(float x)
{
    uint32_t r;
    asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
    return r;
}

// ---------------------------------------------------------------- the GEMMs
// C[b][m][n] = sum_k A[b][m][k] B[b][n][k]  (A and B K-major, C row-major)
struct GemmParams {
    const float *A;
    int64_t lda, strideA;
    const float *B;
    int64_t ldb, strideB;
    float *C;
    int64_t ldc, strideC;
    int M, N, K;
    int *err;   // set to 1 when a bounded wait gave up
};

// 16 bytes of one row of a stage: EB = 4 -> 4 TF32 values, EB = 2 -> 8 BF16 values
template <int EB>
__device__ __forceinline__ uint4 load_unit(const float *row, int k0, int K, bool row_ok)
{
    uint4 v = make_uint4(0, 0, 0, 0);
    if (!row_ok) return v;
    if (EB == 4) {
        uint32_t w[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) w[j] = (k0 + j < K) ? to_tf32(__ldg(row + k0 + j)) : 0u;
        v = make_uint4(w[0], w[1], w[2], w[3]);
    } else {
        uint32_t w[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const float a = (k0 + 2 * j < K) ? __ldg(row + k0 + 2 * j) : 0.f;
            const float c = (k0 + 2 * j + 1 < K) ? __ldg(row + k0 + 2 * j + 1) : 0.f;
            const __nv_bfloat162 h = __floats2bfloat162_rn(a, c);
            w[j] = *reinterpret_cast<const uint32_t *>(&h);
        }
        v = make_uint4(w[0], w[1], w[2], w[3]);
    }
    return v;
}

// offset of (row r, 16-byte unit c) in a stage tile: 8-row groups 1024 bytes
// apart, units of one group 128 bytes apart, rows 16 bytes apart
__device__ __forceinline__ uint32_t tile_off(int r, int c)
{
    return (uint32_t)((r >> 3) * 1024 + c * 128 + (r & 7) * 16);
}

template <int EB>
__global__ void __launch_bounds__(kTcThreads, 1) tc_gemm_kernel(GemmParams p, int BN)
{
    extern __shared__ uint8_t smem_raw[];
    __shared__ __align__(8) uint64_t mbar[2];
    __shared__ uint32_t tmem_base_sh;
    uint8_t *base = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    const int b_tile_bytes = BN * kChunk;
    const int stage_bytes = kATileBytes + b_tile_bytes;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int set = blockIdx.z;
    const int m0 = blockIdx.x * kTcBM, n0 = blockIdx.y * BN;
    const float *A = p.A + set * p.strideA;
    const float *B = p.B + set * p.strideB;
    float *C = p.C + set * p.strideC;
    const uint32_t tcols = BN <= 32 ? 32u : (BN <= 64 ? 64u : (BN <= 128 ? 128u : 256u));

    if (warp == 0) {
        tmem_alloc(smem_addr(&tmem_base_sh), tcols);
        tmem_relinquish();
    }
    if (tid == 0) {
        mbar_init(smem_addr(&mbar[0]), 1);
        mbar_init(smem_addr(&mbar[1]), 1);
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_base_sh;

    constexpr int EPU = 16 / EB;                  // values per 16-byte unit
    constexpr int KC = kChunk / EB;               // values per stage row
    const int nchunks = (p.K + KC - 1) / KC;
    const uint32_t idesc = instr_desc(EB == 4 ? 2u : 1u, kTcBM, (uint32_t)BN);
    bool ok = true;
    for (int c = 0; c < nchunks; ++c) {
        const int s = c & 1;
        if (c >= 2) {
            bool w = ok ? mbar_wait(smem_addr(&mbar[s]), (uint32_t)((c - 2) >> 1) & 1u) : false;
            ok = __syncthreads_and(w) != 0;     // one decision for the whole block
        }
        uint8_t *sa = base + s * stage_bytes;
        uint8_t *sb = sa + kATileBytes;
        const int kbase = c * KC;
        for (int u = tid; u < kTcBM * 8; u += kTcThreads) {
            const int r = u >> 3, cu = u & 7;
            const int m = m0 + r;
            const uint4 v = load_unit<EB>(A + (int64_t)(m < p.M ? m : 0) * p.lda, kbase + cu * EPU, p.K, m < p.M);
            *reinterpret_cast<uint4 *>(sa + tile_off(r, cu)) = v;
        }
        for (int u = tid; u < BN * 8; u += kTcThreads) {
            const int r = u >> 3, cu = u & 7;
            const int n = n0 + r;
            const uint4 v = load_unit<EB>(B + (int64_t)(n < p.N ? n : 0) * p.ldb, kbase + cu * EPU, p.K, n < p.N);
            *reinterpret_cast<uint4 *>(sb + tile_off(r, cu)) = v;
        }
        fence_proxy_async();
        __syncthreads();
        if (tid == 0 && ok) {
            tc_fence_after();
#pragma unroll
            for (int ks = 0; ks < 4; ++ks) {
                const uint64_t ad = smem_desc(smem_addr(sa) + ks * 256, 128, 1024);
                const uint64_t bd = smem_desc(smem_addr(sb) + ks * 256, 128, 1024);
                tc_mma<EB>(tmem, ad, bd, idesc, (c > 0 || ks > 0) ? 1u : 0u);
            }
            tc_commit(smem_addr(&mbar[s]));
        }
    }
    {
        bool w = ok ? mbar_wait(smem_addr(&mbar[(nchunks - 1) & 1]), (uint32_t)((nchunks - 1) >> 1) & 1u) : false;
        ok = __syncthreads_and(w) != 0;
    }
    tc_fence_after();
    const int row = m0 + warp * 32 + lane;
    if (ok) {
        for (int c0 = 0; c0 < BN; c0 += 16) {
            uint32_t r[16];
            tmem_ld16(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)c0, r);
            if (row < p.M) {
                float *dst = C + (int64_t)row * p.ldc + n0 + c0;
#pragma unroll
                for (int j = 0; j < 16; ++j) {
                    if (n0 + c0 + j < p.N) dst[j] = __uint_as_float(r[j]);
                }
            }
        }
    } else if (tid == 0) {
        *(volatile int *)p.err = 1;
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, tcols);
}

// ---------------------------------------------------------------- FP64 products
// C = A B^T in FP64, and (RING) one site absorption of the grid contraction
// with A read in the running tensor's ring order and scaled by 2^-e as the
// tensor-core form does.  Bound by the FP64 pipes alone: a scheduler needs 64
// clocks for one FP64 instruction of a warp, so the questions are how many of
// its lanes do useful work, how evenly the instructions spread over the
// schedulers, and that operand loads, which share the pipes' queue, are few.
// The unit of work is 16 rows x 4 columns of C, two entries per lane (121
// columns pad to 124), whose operands for two k are three 16-byte loads per
// lane, two of them shared with the next unit of the same rows.  A block takes
// a run of consecutive units of a block of up to 128 columns, its 16 warps (four
// per scheduler) G units each, in registers; the host chooses the run so that
// the SMs come out even.  64 x 64 tiles with 4 x 4 entries a thread, before,
// padded 121 columns to 128 and left 458 tiles to 152 SMs: 15.1 ms for the 25
// steps of a 5 x 5 grid of chi 11, now 11.0 (the FP64 pipes' own time 9.8 ms);
// and gave 16 SMs work at M = N = K = 256: 305 us a call, now 72.
// K goes in slabs, the next one copied while one is multiplied: of 32 where a
// block has an SM to itself anyway, for fewer barriers, else of 16, so that two
// fit.  Each entry is accumulated in the order of k.
constexpr int kF64Threads = 512, kF64Warps = kF64Threads / 32;
constexpr int kF64Rows = 256, kF64Cols = 128;            // staged rows of A and B
constexpr int kF64MaxUnits = 12;                         // per warp
constexpr int f64_slab(int G) { return G > 4 ? 32 : 16; }
constexpr int f64_pitch(int G) { return f64_slab(G) + 2; }   // 16-byte loads of 8 rows on different banks
constexpr int f64_stage(int G) { return (kF64Rows + kF64Cols) * f64_pitch(G); }

struct F64Params {
    const double *A;
    int64_t lda, strideA;
    const double *B;
    int64_t ldb, strideB;
    double *C;
    int64_t ldc, strideC;
    int M, N, K;
    int cub;                             // units (4 columns) per column block
    int run;                             // units per block, <= kF64Warps * G
    int64_t R;                           // RING: A[m][u Kh + h] = S[(u R + m) Kh + h]
    int Kh;
    const unsigned long long *max_in;    // [set] largest |S| (its bits)
    unsigned long long *max_out;         // [set] largest |C|, atomicMax
    unsigned long long *max_clear;       // [set] cleared for the next step
    long long *log2s;                    // [set] += e
};

// 8 bytes into shared memory, zero when !ok (src is then not read)
__device__ __forceinline__ void copy8_async(const double *dst, const double *src, bool ok)
{
    const int n = ok ? 8 : 0;
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(smem_addr(dst)), "l"(src), "r"(n) : "memory");
}

template <int G, bool RING>
__global__ void __launch_bounds__(kF64Threads, G > 4 ? 1 : 2) f64_gemm_kernel(F64Params p)
{
    constexpr int kSlab = f64_slab(G), kPitch = f64_pitch(G), kStage = f64_stage(G);
    extern __shared__ __align__(16) double f64_smem[];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, set = blockIdx.z;
    double sc = 1.0;
    int e = 0;
    if (RING) {
        const double mx = __longlong_as_double((long long)p.max_in[set]);
        if (mx > 0.0) e = ilogb(mx);
        if (e) sc = ldexp(1.0, -e);
        if (blockIdx.x == 0 && blockIdx.y == 0 && tid == 0) {
            p.max_clear[set] = 0ull;
            p.log2s[set] += e;
        }
    }
    // the block's run of units (row group major) and the warp's part of it
    const int c0 = blockIdx.y * p.cub, cub = min(p.cub, ((p.N - 1) >> 2) + 1 - c0);
    const int64_t units = (int64_t)(((p.M - 1) >> 4) + 1) * cub, first = (int64_t)blockIdx.x * p.run;
    if (first >= units) return;
    const int run = (int)min((int64_t)p.run, units - first);
    const int group0 = (int)(first / cub), skip = (int)(first - (int64_t)group0 * cub);
    const int rows = 16 * ((skip + run - 1) / cub + 1);      // <= kF64Rows
    const int cols = 4 * cub, m0 = 16 * group0, n0 = 4 * c0;
    // warps w and w + 4 share a scheduler, so the odd units of a run go round them
    const int share = run / kF64Warps, odd = run % kF64Warps;
    const int u0 = skip + warp * share + min(warp, odd), g = share + (warp < odd ? 1 : 0);
    const int r0 = u0 / cub, col0 = u0 - r0 * cub;
    double acc[G][2];
#pragma unroll
    for (int i = 0; i < G; ++i) acc[i][0] = acc[i][1] = 0.0;
    const double *A = p.A + set * p.strideA, *B = p.B + set * p.strideB;
    const int kk = tid & (kSlab - 1), row0 = tid / kSlab;
    constexpr int kRowStep = kF64Threads / kSlab;
    auto load = [&](int k0, double *st) {
        const int k = k0 + kk;
        int64_t a_off = k, a_row = p.lda;
        if (RING) {
            const int u = k / p.Kh;
            a_off = (int64_t)u * p.R * p.Kh + (k - u * p.Kh);
            a_row = p.Kh;
        }
        for (int r = row0; r < rows; r += kRowStep) {
            const bool ok = k < p.K && m0 + r < p.M;
            copy8_async(st + r * kPitch + kk, ok ? A + a_off + (m0 + r) * a_row : A, ok);
        }
        for (int r = row0; r < cols; r += kRowStep) {
            const bool ok = k < p.K && n0 + r < p.N;
            copy8_async(st + (kF64Rows + r) * kPitch + kk, ok ? B + (int64_t)(n0 + r) * p.ldb + k : B, ok);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    load(0, f64_smem);
    for (int k0 = 0, b = 0; k0 < p.K; k0 += kSlab, b ^= 1) {
        double *st = f64_smem + b * kStage;
        if (k0 + kSlab < p.K) {
            load(k0 + kSlab, f64_smem + (b ^ 1) * kStage);
            asm volatile("cp.async.wait_group 1;" ::: "memory");
        } else {
            asm volatile("cp.async.wait_group 0;" ::: "memory");
        }
        if (RING && e && k0 + kk < p.K) {                    // each thread the entries that it copied
            for (int r = row0; r < rows; r += kRowStep) st[r * kPitch + kk] *= sc;
        }
        __syncthreads();
        if (g > 0) {
            const double *arow = st + (16 * r0 + (lane >> 2)) * kPitch;
            const double *bcol = st + (kF64Rows + (lane & 3)) * kPitch;
            const int kn = min(kSlab, p.K - k0);
            for (int q = 0; q < kn; q += 2) {                // an odd K's last column is staged as zeros
                const double *ar = arow + q;
                int col = col0;
                double2 a0 = *reinterpret_cast<const double2 *>(ar);
                double2 a1 = *reinterpret_cast<const double2 *>(ar + 8 * kPitch);
#pragma unroll
                for (int i = 0; i < G; ++i) {
                    if (i == G - 1 && i >= g) break;         // g is G or G - 1 but in a block's last run
                    if (col == cub) {                        // the next row group
                        col = 0;
                        if (i < g) {
                            ar += 16 * kPitch;
                            a0 = *reinterpret_cast<const double2 *>(ar);
                            a1 = *reinterpret_cast<const double2 *>(ar + 8 * kPitch);
                        }
                    }
                    const double2 bv = *reinterpret_cast<const double2 *>(bcol + 4 * col * kPitch + q);
                    acc[i][0] = fma(a0.x, bv.x, acc[i][0]);
                    acc[i][1] = fma(a1.x, bv.x, acc[i][1]);
                    acc[i][0] = fma(a0.y, bv.y, acc[i][0]);
                    acc[i][1] = fma(a1.y, bv.y, acc[i][1]);
                    ++col;
                }
            }
        }
        __syncthreads();
    }
    double *C = p.C + set * p.strideC;
    unsigned long long mx = 0;
#pragma unroll
    for (int i = 0; i < G; ++i) {
        if (i >= g) continue;
        const int r = (u0 + i) / cub;
        const int m = m0 + 16 * r + (lane >> 2), n = n0 + 4 * (u0 + i - r * cub) + (lane & 3);
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            if (m + 8 * j >= p.M || n >= p.N) continue;
            C[(int64_t)(m + 8 * j) * p.ldc + n] = acc[i][j];
            if (RING) {                                      // largest |C| by its bits, a NaN passed over
                const unsigned long long bits =
                    (unsigned long long)__double_as_longlong(acc[i][j]) & 0x7fffffffffffffffull;
                if (bits <= 0x7ff0000000000000ull && bits > mx) mx = bits;
            }
        }
    }
    if (RING) {
        for (int off = 16; off > 0; off >>= 1) {
            const unsigned long long o = __shfl_xor_sync(0xffffffffu, mx, off);
            if (o > mx) mx = o;
        }
        if (lane == 0 && mx) atomicMax(p.max_out + set, mx);
    }
}

// ---------------------------------------------------------------- grid contraction
// Site matrices B_v[n = d Nh + h'][k = u Kh + h] = 2^-s_v T_v[l = h, u, r = h', d]
// per (set, site), rows zero-padded to ldb, in the product's operand type; s_v
// is the exponent of the tensor's largest |entry|.  gridDim.z blocks per tensor
// (a cluster when more than one), each searching its part of it and writing its
// part of the rows, a warp per row; see site_blocks.
constexpr int kSiteBlocks = 8;                  // most blocks per tensor

template <typename E>
__device__ __forceinline__ E site_elem(double x);
template <>
__device__ __forceinline__ double site_elem<double>(double x) { return x; }
template <>
__device__ __forceinline__ float site_elem<float>(double x) { return __uint_as_float(to_tf32((float)x)); }
template <>
__device__ __forceinline__ __nv_bfloat16 site_elem<__nv_bfloat16>(double x) { return __float2bfloat16_rn((float)x); }

template <typename E>
__global__ void __launch_bounds__(256)
    grid_sites_kernel(const double *data, int64_t set_stride, const SiteMap *sites, E *Bm, int64_t b_stride,
                      const int64_t *ldb, long long *log2s)
{
    const int v = blockIdx.x, set = blockIdx.y, part = blockIdx.z, parts = gridDim.z;
    const SiteMap sm = sites[v];
    const double *t = data + set * set_stride + sm.t_off;
    const int Kh = sm.dim[0], Ku = sm.dim[1], Nh = sm.dim[2], Nd = sm.dim[3];
    const int K = Ku * Kh, N = Nd * Nh;
    const int64_t n_ent = (int64_t)N * K;
    __shared__ unsigned long long largest[8];   // of each warp
    cg::cluster_group cluster = cg::this_cluster();
    // the largest |entry| by its bits (comparing doubles costs FP64 time), a NaN passed over
    unsigned long long mx = 0;
    for (int64_t i = part * 256 + threadIdx.x; i < n_ent; i += 256 * parts) {
        const unsigned long long bits = (unsigned long long)__double_as_longlong(t[i]) & 0x7fffffffffffffffull;
        if (bits <= 0x7ff0000000000000ull && bits > mx) mx = bits;
    }
    for (int off = 16; off > 0; off >>= 1) {
        const unsigned long long o = __shfl_xor_sync(0xffffffffu, mx, off);
        if (o > mx) mx = o;
    }
    if ((threadIdx.x & 31) == 0) largest[threadIdx.x >> 5] = mx;
    if (parts > 1) cluster.sync();
    else __syncthreads();
    mx = 0;
    for (int i = threadIdx.x & 31; i < 8 * parts; i += 32) {
        const unsigned long long o = parts > 1 ? cluster.map_shared_rank(largest, i >> 3)[i & 7] : largest[i];
        if (o > mx) mx = o;
    }
    for (int off = 16; off > 0; off >>= 1) {
        const unsigned long long o = __shfl_xor_sync(0xffffffffu, mx, off);
        if (o > mx) mx = o;
    }
    if (parts > 1) cluster.sync();              // no block leaves while its maxima are read
    const double top = __longlong_as_double((long long)mx);
    const int e = top > 0.0 ? ilogb(top) : 0;
    const double sc = ldexp(1.0, -e);
    const int ld = (int)ldb[v];
    E *out = Bm + set * b_stride + sm.b_off;
    for (int n = part * 8 + (threadIdx.x >> 5); n < N; n += 8 * parts) {
        const int d = n / Nh, hp = n - d * Nh;
        const double *row = t + (int64_t)hp * sm.stride[2] + (int64_t)d * sm.stride[3];
        for (int k = threadIdx.x & 31; k < ld; k += 32) {
            const int u = k / Kh, h = k - u * Kh;
            out[(int64_t)n * ld + k] =
                site_elem<E>(k < K ? row[(int64_t)h * sm.stride[0] + (int64_t)u * sm.stride[1]] * sc : 0.0);
        }
    }
    if (part == 0 && threadIdx.x == 0)
        atomicAdd(reinterpret_cast<unsigned long long *>(log2s + set), (unsigned long long)(long long)e);
}

template <typename E>
__global__ void grid_init_kernel(E *S, int64_t stride, unsigned long long *maxbits, long long *log2s, int n_sets)
{
    const int set = blockIdx.x * blockDim.x + threadIdx.x;
    if (set >= n_sets) return;
    S[set * stride] = site_elem<E>(1.0);
    maxbits[set] = sizeof(E) == 8 ? (unsigned long long)__double_as_longlong(1.0)
                                  : (unsigned long long)__float_as_uint(1.0f);
    log2s[set] = 0;
}

template <typename E>
__global__ void grid_final_kernel(const E *S, int64_t stride, const long long *log2s, int n_sets, double *out)
{
    const int set = blockIdx.x * blockDim.x + threadIdx.x;
    if (set >= n_sets) return;
    out[2 * set] = (double)S[set * stride];
    out[2 * set + 1] = (double)log2s[set];
}

// ---------------------------------------------------------------- the grid's GEMM step
// One site absorption of the grid contraction on the tensor cores, with the
// running tensor S read in its ring order directly (no packing pass):
//     out[m][n] = 2^-e_in * sum_{u,h} S[u][m][h] * Bm[n][u Kh + h],
// the result rounded to the operand type (TF32 kept in FP32 words, or BF16) as
// the next step's running tensor, its largest |entry| recorded per set.
template <typename E>
struct RingParams {
    const E *S;              // [set][stride] running tensor [Ku][R][Kh]
    const E *B;              // site matrix [N][ldb] (rows zero-padded to ldb)
    E *out;                  // [set][stride] next running tensor [R][N]
    int64_t stride;          // running-tensor elements per set
    int64_t b_stride;        // site-matrix elements per set
    int64_t ldb;
    int64_t R;
    int Ku, Kh, N, K;
    const unsigned long long *max_in;   // [set] largest |S| (float bits)
    unsigned long long *max_out;        // [set] largest |out|, atomicMax
    unsigned long long *max_clear;      // [set] cleared for the next step
    long long *log2s;                   // [set] += e_in
    int *err;
};

// ---------------------------------------------------------------- the persistent GEMM
// One kernel for the large products, by where A comes from:
//   kBoxes   a site absorption of the grid contraction: A is the running
//            tensor S[u][m][h] (k = u Kh + h), already in the MMA's type,
//            copied by the Tensor Memory Accelerator; the result is scaled,
//            rounded to that type and stored as the next running tensor, its
//            largest |entry| recorded.
//   kGather  the same where no 16-byte unit of k is contiguous in S (a left
//            boundary site, Kh = 1, whose m runs fastest, or an odd Kh): eight
//            warps load it, lanes along m, and write the operand stages.  At
//            Kh = 1 the loads are whole lines; S is small beside the result.
//   kRound   pne_dense_gemm: A is FP32; eight warps round each box to the
//            MMA's type on its way from the landing buffer to the operand
//            stage (the rounding of B, read by every row tile, is done once by
//            round_rows_kernel); the result is stored as FP32.
// Both are bound by HBM at the sizes they are for (K, N = 256: 64 flops per
// byte of A and C against 140 at the TF32 and 290 at the BF16 tensor rate), so
// the split is chosen to keep loads in flight: one block per SM walks the
// tiles; one thread issues the loads (64 KB of A in flight per SM), one the
// MMAs, eight warps (four where A is rounded, see store_warps) store a finished
// tile from tensor memory while the next one accumulates in its other half; the
// stages fill the shared memory, up to 12 (with four, the N = 16 steps of the last
// column read 4.1 TB/s).  An operand row of a stage is 128 bytes, copied
// in boxes of the widest swizzle whose bytes are contiguous in A (128, 64 or
// 32; 16 without one): boxes of 16 bytes, which every stage used before, cost
// the copy engine one request per 16 bytes and bound the kernel.
// Measured, before -> after (HBM 6.7 TB/s): 4 x 32768 x 256 x 256 with B's
// rounding, BF16 340.6 -> 54.8 us (4.9 TB/s), TF32 507 -> 57 us; 20000 x 2000 x
// 1000 BF16 1241 -> 131 us (612 TFLOP/s); 32 5 x 4 networks of chi = 16, whole
// calls: TF32 14.97 -> 6.30 ms (a step with K = N = 256 moves 4.25 GB in 0.64 to
// 0.66 ms, 6.5 TB/s), BF16 13.58 -> 4.24 ms; 16 5 x 5 networks of chi = 11,
// gathered: TF32 3.28 -> 1.66 ms.
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void tma_load4(uint32_t dst, const CUtensorMap *map, int c0, int c1, int c2, int c3,
                                          uint32_t bar)
{
    asm volatile("cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], [%6];"
                 ::"r"(dst), "l"((uint64_t)map), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(bar)
                 : "memory");
}
__device__ __forceinline__ void tma_load3(uint32_t dst, const CUtensorMap *map, int c0, int c1, int c2, uint32_t bar)
{
    asm volatile("cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
                 ::"r"(dst), "l"((uint64_t)map), "r"(c0), "r"(c1), "r"(c2), "r"(bar)
                 : "memory");
}
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&r)[32])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, "
                 "%14, %15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
                   "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]),
                   "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]),
                   "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]),
                   "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
                 : "r"(taddr)
                 : "memory");
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

// shared-memory matrix descriptor of a K-major tile whose rows are `w` bytes
// wide: swizzled over w = 128, 64 or 32 bytes (8-row groups 8 w apart), or
// w = 16, unswizzled 16-byte columns of 128 rows
__device__ __forceinline__ uint64_t tile_desc(uint32_t addr, int w)
{
    if (w == 16) return smem_desc(addr, kTcBM * 16, 128);
    const uint64_t layout = w == 128 ? 2 : (w == 64 ? 4 : 6);
    return smem_desc(addr, 16, (uint32_t)(8 * w)) | (layout << 61);
}

struct StreamParams {
    int64_t M;                          // rows of A and of the result
    int N, K, BN;                       // BN: columns per tile, a multiple of 16
    int mt, nt, batch;                  // tiles down, across, tensor sets
    int stages;                         // operand stages in shared memory
    int w, Kh;                          // kBoxes: bytes of a box of A; h range of one u
    const void *S;                      // kGather: running tensor [set][Ku][M][Kh], sets strideC apart
    void *out;                          // [batch][M][ldc]
    int64_t ldc, strideC;
    int vec;                            // rows of the result on 16-byte boundaries
    const unsigned long long *max_in;   // the grid's sources: as RingParams
    unsigned long long *max_out, *max_clear;
    long long *log2s;
    int *err;
};

// The tiles of one block, every gridDim.x-th, columns fastest, then rows, then
// sets: advanced by adding (a 64-bit division per tile and role took a third
// of the time of the steps whose tiles are short).
struct TileWalk {
    int n, m, set, dn, dm, ds, nt, mt, batch;
    __device__ explicit TileWalk(const StreamParams &p) : nt(p.nt), mt(p.mt), batch(p.batch)
    {
        const unsigned b = blockIdx.x, g = gridDim.x;
        n = (int)(b % nt); m = (int)(b / nt % mt); set = (int)(b / nt / mt);
        dn = (int)(g % nt); dm = (int)(g / nt % mt); ds = (int)(g / nt / mt);
    }
    __device__ __forceinline__ bool more() const { return set < batch; }
    __device__ __forceinline__ void next()
    {
        n += dn;
        int c = n >= nt;
        n -= c ? nt : 0;
        m += dm + c;
        c = m >= mt;
        m -= c ? mt : 0;
        set += ds + c;
    }
};

constexpr int kStreamStages = 12, kRawBoxes = 4;   // most operand stages; landing boxes
constexpr int kBoxBytes = kTcBM * 128;
constexpr int kConvertWarps = 8;
enum StreamSource { kBoxes = 0, kRound = 1, kGather = 2 };
// Storing warps, one or two per 32 rows.  The grid's short tiles are bound by
// four (N = 256, K = 16: 630 us a step with four, 454 with eight); where A is
// rounded the second four would take the fourth landing box's shared memory
// (4 x 32768 x 256 x 256 TF32: 57.5 us with four, 61.5 with eight and three boxes).
constexpr int store_warps(int src) { return src == kRound ? 4 : 8; }
constexpr int stream_threads(int src) { return 32 * (4 + store_warps(src) + (src == kBoxes ? 0 : kConvertWarps)); }

template <int EB, int SRC>
__global__ void __launch_bounds__(stream_threads(SRC), 1) tc_stream_kernel(const __grid_constant__ CUtensorMap tmA,
                                                                           const __grid_constant__ CUtensorMap tmB,
                                                                           StreamParams p)
{
    constexpr bool RAW = SRC == kRound;
    constexpr int kStoreWarps = store_warps(SRC), kConvert0 = 4 + kStoreWarps;   // first converting warp
    constexpr bool FILL = SRC != kBoxes;           // warps kConvert0.. write A's operand stages
    const int NST = p.stages;
    constexpr int KC = 128 / EB;                   // k values per stage
    constexpr int OB = RAW ? 4 : EB;               // bytes of a stored value
    constexpr int RPC = RAW ? 4 / EB : 1;          // landing boxes per operand stage
    extern __shared__ uint8_t smem_raw[];
    __shared__ __align__(8) uint64_t full[kStreamStages], empty[kStreamStages], rfull[kRawBoxes], rempty[kRawBoxes], afull[2], aempty[2];
    __shared__ uint32_t tmem_base_sh;
    uint8_t *base = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    const int b_bytes = p.BN * 128;
    const int stage_bytes = kBoxBytes + b_bytes;   // 1024-byte multiples: BN is a multiple of 16
    uint8_t *epi = base + NST * stage_bytes;
    uint8_t *raw = epi + kStoreWarps * 4096;       // a storing warp holds 32 rows of 128 bytes
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t acols = p.BN <= 32 ? 32u : (p.BN <= 64 ? 64u : (p.BN <= 128 ? 128u : 256u));
    if (warp == 3) {
        tmem_alloc(smem_addr(&tmem_base_sh), 2 * acols);
        tmem_relinquish();
    }
    if (tid == 0) {
        for (int i = 0; i < NST; ++i) {
            mbar_init(smem_addr(&full[i]), FILL ? 1 + kConvertWarps : 1);
            mbar_init(smem_addr(&empty[i]), 1);
        }
        for (int i = 0; i < kRawBoxes; ++i) {
            mbar_init(smem_addr(&rfull[i]), 1);
            mbar_init(smem_addr(&rempty[i]), kConvertWarps);
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(smem_addr(&afull[i]), 1);
            mbar_init(smem_addr(&aempty[i]), kStoreWarps);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_base_sh;
    const int nch = (p.K + KC - 1) / KC;
    // a wait that gives up ends its role; the others give up on their own waits
    auto failed = [&] { *(volatile int *)p.err = 1; };
    auto stage_a = [&](int s) { return smem_addr(base + s * stage_bytes); };

    if (tid == 0 || (RAW && tid == 64)) {
        // loads: thread 0 fills the stages, A's boxes and B's; when A is
        // rounded it fills the landing boxes and thread 64 the B of the stages
        const bool do_raw = RAW && tid == 0;
        int s = 0, n_issued = 0;
        uint32_t ph = 0;
        bool ok = true;
        const int step = FILL ? 0 : p.w / EB, boxes = FILL ? 0 : 128 / p.w;
        const int steps = do_raw ? nch * RPC : nch;
        for (TileWalk t(p); t.more() && ok; t.next()) {
            const int m0 = t.m * kTcBM, n0 = t.n * p.BN, set = t.set;
            int u = 0, h = 0;
            for (int c = 0; c < steps && ok; ++c) {
                if (do_raw) {
                    ok = mbar_wait(smem_addr(&rempty[s]), ph ^ 1);
                    if (!ok) break;
                    const uint32_t fb = smem_addr(&rfull[s]);
                    mbar_expect_tx(fb, kBoxBytes);
                    tma_load3(smem_addr(raw + s * kBoxBytes), &tmA, c * 32, m0, set, fb);
                    if (++s == kRawBoxes) { s = 0; ph ^= 1; }
                } else {
                    ok = mbar_wait(smem_addr(&empty[s]), ph ^ 1);
                    if (!ok) break;
                    const uint32_t fb = smem_addr(&full[s]);
                    mbar_expect_tx(fb, (uint32_t)(FILL ? b_bytes : stage_bytes));
                    const uint32_t sa = stage_a(s);
                    for (int b = 0; b < boxes; ++b) {
                        tma_load4(sa + (uint32_t)(b * p.w * kTcBM), &tmA, h, m0, u, set, fb);
                        h += step;
                        if (h >= p.Kh) { h = 0; ++u; }
                    }
                    tma_load3(sa + kBoxBytes, &tmB, c * KC, n0, set, fb);
                    if (++s == NST) { s = 0; ph ^= 1; }
                }
                ++n_issued;
            }
        }
        if (!ok) {
            failed();
            // the copies in flight land before the block may end
            const int slots = do_raw ? kRawBoxes : NST;
            for (int i = 0; i < slots && i < n_issued; ++i) {
                if (--s < 0) { s = slots - 1; ph ^= 1; }
                mbar_wait(smem_addr(do_raw ? &rfull[s] : &full[s]), ph);
            }
        }
    } else if (tid == 32) {
        // MMAs
        const uint32_t idesc = instr_desc(EB == 4 ? 2u : 1u, kTcBM, (uint32_t)p.BN);
        const int w = FILL ? 128 : p.w;
        uint64_t ad[4], bd[4];                     // descriptors of the four K steps in stage 0
#pragma unroll
        for (int ks = 0; ks < 4; ++ks) {
            const int o = ks * 32;
            const uint32_t at = w == 16 ? (uint32_t)(o * kTcBM) : (uint32_t)(o / w * w * kTcBM + o % w);
            ad[ks] = tile_desc(stage_a(0) + at, w);
            bd[ks] = tile_desc(stage_a(0) + kBoxBytes + o, 128);
        }
        int s = 0;
        uint32_t ph = 0, it = 0;
        bool ok = true;
        for (TileWalk t(p); t.more() && ok; t.next(), ++it) {
            const uint32_t acc = tmem + (it & 1) * acols;
            ok = mbar_wait(smem_addr(&aempty[it & 1]), ((it >> 1) & 1) ^ 1);
            for (int c = 0; c < nch && ok; ++c) {
                ok = mbar_wait(smem_addr(&full[s]), ph);
                if (!ok) break;
                tc_fence_after();
                const uint64_t so = (uint64_t)((s * stage_bytes) >> 4);
#pragma unroll
                for (int ks = 0; ks < 4; ++ks)
                    tc_mma<EB>(acc, ad[ks] + so, bd[ks] + so, idesc, (c > 0 || ks > 0) ? 1u : 0u);
                tc_commit(smem_addr(&empty[s]));
                if (++s == NST) { s = 0; ph ^= 1; }
            }
            if (ok) tc_commit(smem_addr(&afull[it & 1]));
        }
        if (!ok) failed();
    } else if (warp >= 4 && warp < kConvert0) {
        // results: tensor memory -> registers -> this warp's 32 x 128-byte
        // buffer (16-byte units swizzled by the row) -> whole row segments
        constexpr int CW = 128 / OB;               // columns per round
        uint8_t *buf = epi + (warp - 4) * 4096;
        const int rows0 = (warp & 3) * 32;         // the tensor-memory lanes of this warp
        uint32_t it = 0;
        bool ok = true;
        int e_in = 0, scaled_set = -1;
        float sc = 1.f;
        for (TileWalk t(p); t.more(); t.next(), ++it) {
            const int n = t.n, set = t.set;
            const int64_t m0 = (int64_t)t.m * kTcBM + rows0;
            float mx = 0.f;
            if (!RAW) {
                // the scale of this step: 2^-e_in, e_in the exponent of the input's largest |entry|
                if (set != scaled_set) {
                    const float mx_in = __uint_as_float((unsigned)p.max_in[set]);
                    e_in = mx_in > 0.f ? ilogbf(mx_in) : 0;
                    sc = ldexpf(1.f, -e_in);
                    scaled_set = set;
                }
                if (n == 0 && t.m == 0 && tid == 128) {
                    p.log2s[set] += e_in;
                    p.max_clear[set] = 0ull;
                }
            }
            ok = mbar_wait(smem_addr(&afull[it & 1]), (it >> 1) & 1);
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) break;
            tc_fence_after();
            const uint32_t acc = tmem + (it & 1) * acols + ((uint32_t)rows0 << 16);
            uint8_t *out = static_cast<uint8_t *>(p.out) + ((int64_t)set * p.strideC) * OB;
            for (int c0 = (warp - 4) / 4 * CW; c0 < p.BN; c0 += kStoreWarps / 4 * CW) {
#pragma unroll
                for (int h = 0; h < CW; h += 32) {
                    if (h > 0 && c0 + h >= (int)acols) break;
                    uint32_t v[32];
                    tmem_ld32(acc + (uint32_t)(c0 + h), v);
                    const bool whole = c0 + h + 32 <= p.BN;    // else 16 columns: BN is a multiple of 16
                    if (OB == 4) {
                        if (!RAW) {
#pragma unroll
                            for (int j = 0; j < 32; ++j) {
                                v[j] = to_tf32(__uint_as_float(v[j]) * sc);
                                if (j < 16 || whole) mx = fmaxf(mx, fabsf(__uint_as_float(v[j])));
                            }
                        }
#pragma unroll
                        for (int q = 0; q < 8; ++q)
                            *reinterpret_cast<uint4 *>(buf + lane * 128 + ((q ^ (lane & 7)) * 16)) =
                                make_uint4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
                    } else {
                        uint32_t x[16];
#pragma unroll
                        for (int j = 0; j < 16; ++j) {
                            const __nv_bfloat162 b2 = __floats2bfloat162_rn(__uint_as_float(v[2 * j]) * sc,
                                                                            __uint_as_float(v[2 * j + 1]) * sc);
                            if (j < 8 || whole)
                                mx = fmaxf(mx, fmaxf(fabsf(__low2float(b2)), fabsf(__high2float(b2))));
                            x[j] = *reinterpret_cast<const uint32_t *>(&b2);
                        }
#pragma unroll
                        for (int q = 0; q < 4; ++q)
                            *reinterpret_cast<uint4 *>(buf + lane * 128 + (((h / 8 + q) ^ (lane & 7)) * 16)) =
                                make_uint4(x[4 * q], x[4 * q + 1], x[4 * q + 2], x[4 * q + 3]);
                    }
                }
                __syncwarp();
                constexpr int EPO = 16 / OB;
                const int unit = lane & 7;
                const int col = n * p.BN + c0 + unit * EPO;
                const int left = min(p.N, (n + 1) * p.BN) - col;
                const int row1 = lane >> 3;                     // rows row1, row1 + 4, ...
                uint8_t *dst = out + ((m0 + row1) * p.ldc + col) * OB;
                const int64_t hop = 4 * p.ldc * OB;
                const int rows = (int)min((int64_t)32, p.M - m0);
                if (RAW && !p.vec) {                            // unaligned rows of FP32: a line of one row at a time
                    const int cc = n * p.BN + c0 + lane;
                    const bool in = cc < min(p.N, (n + 1) * p.BN);
                    uint32_t *line = reinterpret_cast<uint32_t *>(out) + m0 * p.ldc + cc;
#pragma unroll 8
                    for (int rr = 0; rr < 32; ++rr) {
                        const uint32_t v = *reinterpret_cast<const uint32_t *>(
                            buf + rr * 128 + (((lane >> 2) ^ (rr & 7)) * 16) + (lane & 3) * 4);
                        if (in && rr < rows) line[rr * p.ldc] = v;
                    }
                } else if (p.vec && left >= EPO) {
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        const int rr = i * 4 + row1;
                        const uint4 v = *reinterpret_cast<const uint4 *>(buf + rr * 128 + ((unit ^ (rr & 7)) * 16));
                        if (rr < rows) *reinterpret_cast<uint4 *>(dst + i * hop) = v;
                    }
                } else {
                    for (int i = 0; i < 8; ++i) {
                        const int rr = i * 4 + row1;
                        if (rr >= rows) break;
                        const uint8_t *src = buf + rr * 128 + ((unit ^ (rr & 7)) * 16);
                        for (int j = 0; j < EPO && j < left; ++j) {
                            if (OB == 4) reinterpret_cast<uint32_t *>(dst + i * hop)[j] = reinterpret_cast<const uint32_t *>(src)[j];
                            else reinterpret_cast<uint16_t *>(dst + i * hop)[j] = reinterpret_cast<const uint16_t *>(src)[j];
                        }
                    }
                }
                __syncwarp();
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_addr(&aempty[it & 1]));
            if (!RAW) {
                for (int off = 16; off > 0; off >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, off));
                if (lane == 0 && mx > 0.f) atomicMax(p.max_out + set, (unsigned long long)__float_as_uint(mx));
            }
        }
        if (!ok && lane == 0) failed();
    } else if (SRC == kGather && warp >= kConvert0) {
        // running tensor -> operand stage: a row per lane, four of the eight
        // 16-byte units of its 128 bytes per thread
        using E = typename std::conditional<EB == 4, uint32_t, uint16_t>::type;
        constexpr int EPU = 16 / EB;
        const int cw = warp - kConvert0, row = (cw & 3) * 32 + lane, u0 = (cw >> 2) * 4;
        int s = 0;
        uint32_t ph = 0;
        bool ok = true;
        // the values of one chunk of one tile; zeros past the rows and past K
        auto load = [&](const TileWalk &t, int c, E (&v)[4][EPU]) {
            const int64_t m = (int64_t)t.m * kTcBM + row;
            const E *S = static_cast<const E *>(p.S) + t.set * p.strideC + m * p.Kh;
            int k = c * KC + u0 * EPU;
            int u = k / p.Kh, h = k - u * p.Kh;
            const E *at = S + (int64_t)u * p.M * p.Kh;
            const int64_t hop = p.M * p.Kh;
#pragma unroll
            for (int q = 0; q < 4; ++q)
#pragma unroll
                for (int j = 0; j < EPU; ++j) {
                    v[q][j] = (m < p.M && k < p.K) ? __ldg(at + h) : (E)0;
                    ++k;
                    if (++h == p.Kh) { h = 0; at += hop; }
                }
        };
        TileWalk t(p);
        int c = 0;
        __align__(16) E v[4][EPU], w[4][EPU];
        if (t.more()) load(t, 0, v);
        while (t.more()) {
            // the next chunk's loads run while this one waits for its stage
            TileWalk t1 = t;
            int c1 = c + 1;
            if (c1 == nch) { c1 = 0; t1.next(); }
            if (t1.more()) load(t1, c1, w);
            ok = __all_sync(0xffffffffu, mbar_wait(smem_addr(&empty[s]), ph ^ 1));
            if (!ok) break;
            uint8_t *op = base + s * stage_bytes + row * 128;
#pragma unroll
            for (int q = 0; q < 4; ++q)
                *reinterpret_cast<uint4 *>(op + (((u0 + q) ^ (row & 7)) * 16)) = *reinterpret_cast<const uint4 *>(v[q]);
            fence_proxy_async();
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_addr(&full[s]));
            if (++s == NST) { s = 0; ph ^= 1; }
            t = t1;
            c = c1;
#pragma unroll
            for (int q = 0; q < 4; ++q)
#pragma unroll
                for (int j = 0; j < EPU; ++j) v[q][j] = w[q][j];
        }
        if (!ok && lane == 0) failed();
    } else if (RAW && warp >= kConvert0) {
        // rounding: landing box -> operand stage, both 128-byte rows with the
        // copy engine's swizzle (16-byte unit c of row r at c ^ (r & 7))
        const int cw = warp - kConvert0;
        int s = 0, rs = 0;
        uint32_t ph = 0, rph = 0;
        bool ok = true;
        for (TileWalk t(p); t.more() && ok; t.next()) {
            for (int c = 0; c < nch && ok; ++c) {
                ok = __all_sync(0xffffffffu, mbar_wait(smem_addr(&empty[s]), ph ^ 1));
                if (!ok) break;
                uint8_t *op = base + s * stage_bytes;
#pragma unroll
                for (int bx = 0; bx < RPC; ++bx) {
                    ok = __all_sync(0xffffffffu, mbar_wait(smem_addr(&rfull[rs]), rph));
                    if (!ok) break;
                    const uint8_t *src = raw + rs * kBoxBytes;
                    if (EB == 4) {
                        // the same unit of the same row: the same offset
                        for (int o = (cw * 32 + lane) * 16; o < kBoxBytes; o += kConvertWarps * 512) {
                            const float4 f = *reinterpret_cast<const float4 *>(src + o);
                            *reinterpret_cast<uint4 *>(op + o) =
                                make_uint4(to_tf32(f.x), to_tf32(f.y), to_tf32(f.z), to_tf32(f.w));
                        }
                    } else {
                        // eight values (two units of the box) to one unit; the rows of
                        // a quarter warp differ by 5 mod 8, so that neither the reads
                        // nor the writes meet in a bank
                        const int k4 = lane & 3, r8 = (lane >> 3) ^ ((lane & 4) ? 5 : 0);
                        for (int g = cw; g < kTcBM / 8; g += kConvertWarps) {
                            const int r = g * 8 + r8;
                            const float4 f = *reinterpret_cast<const float4 *>(src + r * 128 + (((2 * k4) ^ r8) * 16));
                            const float4 h = *reinterpret_cast<const float4 *>(src + r * 128 + (((2 * k4 + 1) ^ r8) * 16));
                            const __nv_bfloat162 a = __floats2bfloat162_rn(f.x, f.y), b = __floats2bfloat162_rn(f.z, f.w);
                            const __nv_bfloat162 d = __floats2bfloat162_rn(h.x, h.y), e = __floats2bfloat162_rn(h.z, h.w);
                            *reinterpret_cast<uint4 *>(op + r * 128 + (((bx * 4 + k4) ^ r8) * 16)) =
                                make_uint4(*reinterpret_cast<const uint32_t *>(&a), *reinterpret_cast<const uint32_t *>(&b),
                                           *reinterpret_cast<const uint32_t *>(&d), *reinterpret_cast<const uint32_t *>(&e));
                        }
                    }
                    __syncwarp();
                    if (lane == 0) mbar_arrive(smem_addr(&rempty[rs]));
                    if (++rs == kRawBoxes) { rs = 0; rph ^= 1; }
                }
                if (!ok) break;
                fence_proxy_async();
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_addr(&full[s]));
                if (++s == NST) { s = 0; ph ^= 1; }
            }
        }
        if (!ok && lane == 0) failed();
    }
    __syncwarp();
    tc_fence_before();
    __syncthreads();
    if (warp == 3) tmem_dealloc(tmem, 2 * acols);
}

// B of pne_dense_gemm rounded to the operand type once, rows padded with zeros
// to 16-byte units: W[b][n][ldw].  Each value is read again by every row tile,
// so rounding it there would cost M / 128 times the work.
template <int EB>
__global__ void round_rows_kernel(const float *B, int64_t ldb, int64_t strideB, int N, int K, int ldw, void *W,
                                  int64_t total)
{
    constexpr int EPU = 16 / EB;
    const int units = ldw / EPU;
    for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < total; q += (int64_t)gridDim.x * blockDim.x) {
        const int u = (int)(q % units);
        const int64_t r = q / units;
        const float *row = B + r / N * strideB + r % N * ldb;
        static_cast<uint4 *>(W)[q] = load_unit<EB>(row, u * EPU, K, true);
    }
}

PFN_cuTensorMapEncodeTiled_v12000 tensor_map_encoder()
{
    static std::once_flag once;
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    std::call_once(once, [] {
        void *f = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = (PFN_cuTensorMapEncodeTiled_v12000)f;
    });
    return fn;
}

// tiles of BN <= 256 columns of equal width; narrower ones while the tiles
// do not reach every SM (128 x 2048 x 256 TF32: 75 -> 18 us)
void stream_tiles(StreamParams &p, int n_sm)
{
    p.mt = (int)((p.M + kTcBM - 1) / kTcBM);
    p.nt = (p.N + 255) / 256;
    auto width = [&] { return ((p.N + p.nt - 1) / p.nt + 15) / 16 * 16; };
    while ((int64_t)p.mt * p.nt * p.batch < n_sm && width() > 64) p.nt *= 2;
    p.BN = width();
    p.nt = (p.N + p.BN - 1) / p.BN;
}

template <int EB, int SRC>
cudaError_t launch_stream(const CUtensorMap &ma, const CUtensorMap &mb, StreamParams p, int n_sm, cudaStream_t s)
{
    const int fixed = store_warps(SRC) * 4096 + (SRC == kRound ? kRawBoxes * kBoxBytes : 0) + 1024;
    const int stage = kBoxBytes + p.BN * 128;
    p.stages = std::min(kStreamStages, (226 * 1024 - fixed) / stage);   // 227 KB less the barriers
    const size_t smem = (size_t)p.stages * stage + fixed;
    cudaError_t e = grant_dynamic_smem((const void *)tc_stream_kernel<EB, SRC>, smem);
    if (e != cudaSuccess) return e;
    const int64_t tiles = (int64_t)p.mt * p.nt * p.batch;
    tc_stream_kernel<EB, SRC><<<(unsigned)std::min<int64_t>(tiles, n_sm), stream_threads(SRC), smem, s>>>(ma, mb, p);
    return cudaGetLastError();
}

// operand boxes of 128 bytes by `rows` rows over [batch][rows][ld]
bool encode_rows(CUtensorMap *m, int eb, const void *ptr, int64_t ld, int64_t cols, int64_t rows, int64_t stride,
                 int batch, int box_rows)
{
    auto enc = tensor_map_encoder();
    if (!enc) return false;
    const CUtensorMapDataType dt = eb == 4 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16;
    const cuuint64_t dim[3] = {(cuuint64_t)cols, (cuuint64_t)rows, (cuuint64_t)batch};
    const cuuint64_t str[2] = {(cuuint64_t)ld * eb, (cuuint64_t)(batch > 1 ? stride : ld * rows) * eb};
    const cuuint32_t box[3] = {(cuuint32_t)(128 / eb), (cuuint32_t)box_rows, 1};
    const cuuint32_t one[3] = {1, 1, 1};
    return enc(m, dt, 3, const_cast<void *>(ptr), dim, str, box, one, CU_TENSOR_MAP_INTERLEAVE_NONE,
               CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) ==
           CUDA_SUCCESS;
}

// A site absorption on the persistent kernel.  The copy engine takes A where
// every 16-byte unit of k is contiguous in the running tensor; the other sites
// gather it.  The site matrix is padded to 16-byte rows (grid_plan).
template <typename E>
cudaError_t launch_grid_stream(const RingParams<E> &p, int batch, int n_sm, cudaStream_t s)
{
    auto enc = tensor_map_encoder();
    if (!enc) return cudaErrorSymbolNotFound;
    constexpr int EB = (int)sizeof(E);
    StreamParams q{};
    q.M = p.R;
    q.N = p.N;
    q.K = p.K;
    q.batch = batch;
    stream_tiles(q, n_sm);
    q.Kh = p.Kh;
    q.w = 128;
    while (q.w > 16 && (p.Kh * EB) % q.w != 0) q.w /= 2;
    q.out = p.out;
    q.ldc = p.N;
    q.strideC = p.stride;
    q.vec = (p.N * EB) % 16 == 0 && (p.stride * EB) % 16 == 0 && (reinterpret_cast<uintptr_t>(p.out) & 15) == 0;
    q.max_in = p.max_in;
    q.max_out = p.max_out;
    q.max_clear = p.max_clear;
    q.log2s = p.log2s;
    q.err = p.err;
    q.S = p.S;
    CUtensorMap ma{}, mb;
    if (!encode_rows(&mb, EB, p.B, p.ldb, p.ldb, p.N, p.b_stride, batch, q.BN)) return cudaErrorInvalidValue;
    if ((p.Kh * EB) % 16 != 0) return launch_stream<EB, kGather>(ma, mb, q, n_sm, s);
    const CUtensorMapDataType dt = EB == 4 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16;
    const CUtensorMapSwizzle sw = q.w == 128  ? CU_TENSOR_MAP_SWIZZLE_128B
                                  : q.w == 64 ? CU_TENSOR_MAP_SWIZZLE_64B
                                  : q.w == 32 ? CU_TENSOR_MAP_SWIZZLE_32B
                                              : CU_TENSOR_MAP_SWIZZLE_NONE;
    // A: [set][Ku][R][Kh], innermost first
    const cuuint64_t adim[4] = {(cuuint64_t)p.Kh, (cuuint64_t)p.R, (cuuint64_t)p.Ku, (cuuint64_t)batch};
    const cuuint64_t astr[3] = {(cuuint64_t)p.Kh * EB, (cuuint64_t)p.R * p.Kh * EB, (cuuint64_t)p.stride * EB};
    const cuuint32_t abox[4] = {(cuuint32_t)(q.w / EB), (cuuint32_t)kTcBM, 1, 1};
    const cuuint32_t one4[4] = {1, 1, 1, 1};
    if (enc(&ma, dt, 4, (void *)p.S, adim, astr, abox, one4, CU_TENSOR_MAP_INTERLEAVE_NONE, sw,
            CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
        return cudaErrorInvalidValue;
    return launch_stream<EB, kBoxes>(ma, mb, q, n_sm, s);
}

// Blocks per tensor of grid_sites_kernel.  One of them works through n entries in
// about 1.6 ns each, a launch of T tensors takes about 5 ns per block: P blocks a
// tensor are best near P^2 = n / (3 T).  us of the FP64 launch, 3 x 3 networks, with
// 1, 2, 4 and 8 blocks: chi 2, 1000 sets 39, 96, 178, 364; chi 7, 1000 sets 74, 142,
// 240, 445; chi 11, 1 set 32, 33, 22, 16, 300 sets 92, 103, 127, 191; chi 16, 1 set
// 104, 58, 34, 25, 64 sets 133, 85, 76, 77, 200 sets 292, 157, 150, 190 (one block
// with a division per entry took 63, 85, 34, 90, 140, 181 and 325).
int site_blocks(const GridPlan &plan, int nb)
{
    int64_t n = 1;
    for (const GridStep &sd : plan.steps) n = std::max(n, (int64_t)sd.Ku * sd.Kh * sd.Nd * sd.Nh);
    int P = 1;
    while (P < kSiteBlocks && n >= 3 * (int64_t)(2 * P) * (2 * P) * plan.n * nb) P *= 2;
    return P;
}

template <typename E>
cudaError_t launch_grid_sites(const GridPlan &plan, int nb, const double *data, int64_t set_stride, const SiteMap *maps,
                              E *Bm, const int64_t *ldb, long long *lg, cudaStream_t s)
{
    const int blocks = site_blocks(plan, nb);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)plan.n, (unsigned)nb, (unsigned)blocks);
    cfg.blockDim = dim3(256, 1, 1);
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 1;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = (unsigned)blocks;
    cfg.attrs = attr;
    cfg.numAttrs = blocks > 1 ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, grid_sites_kernel<E>, data, set_stride, maps, Bm, plan.b_total, ldb, lg);
}

size_t tc_smem_bytes(int BN)
{
    return (size_t)2 * (kATileBytes + BN * kChunk) + 1024;
}

// pne_dense_gemm on the persistent kernel, B rounded into `W` first; used =
// false when A cannot be described to the copy engine
template <int EB>
cudaError_t launch_dense_stream(const GemmParams &p, int batch, int n_sm, void *W, int64_t ldw, cudaStream_t s,
                                bool &used)
{
    used = false;
    StreamParams q{};
    q.M = p.M;
    q.N = p.N;
    q.K = p.K;
    q.batch = batch;
    stream_tiles(q, n_sm);
    q.w = 128;
    q.out = p.C;
    q.ldc = p.ldc;
    q.strideC = p.strideC;
    q.vec = p.ldc % 4 == 0 && (batch == 1 || p.strideC % 4 == 0) && (reinterpret_cast<uintptr_t>(p.C) & 15) == 0;
    q.err = p.err;
    CUtensorMap ma, mb;
    if (!encode_rows(&ma, 4, p.A, p.lda, p.K, p.M, p.strideA, batch, kTcBM) ||
        !encode_rows(&mb, EB, W, ldw, ldw, p.N, ldw * p.N, batch, q.BN))
        return cudaSuccess;
    used = true;
    const int64_t units = (int64_t)batch * p.N * (ldw / (16 / EB));
    round_rows_kernel<EB><<<(unsigned)std::min<int64_t>((units + 255) / 256, (int64_t)n_sm * 16), 256, 0, s>>>(
        p.B, p.ldb, p.strideB, p.N, p.K, (int)ldw, W, units);
    const cudaError_t e = cudaGetLastError();
    return e != cudaSuccess ? e : launch_stream<EB, kRound>(ma, mb, q, n_sm, s);
}

// Rows of A that the copy engine cannot address, one warp per row, to rows of
// ldp values (a multiple of four; the padding is never read)
__global__ void pad_rows_kernel(const float *A, int64_t lda, int64_t strideA, int M, int K, int64_t rows, int64_t ldp,
                                float *P)
{
    const int lane = threadIdx.x & 31;
    for (int64_t r = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); r < rows;
         r += (int64_t)gridDim.x * (blockDim.x >> 5)) {
        const int64_t b = r / M;
        const float *src = A + b * strideA + (r - b * M) * lda;
        float *dst = P + r * ldp;
#pragma unroll 4
        for (int k = lane; k < K; k += 32) dst[k] = __ldg(src + k);
    }
}

// The persistent kernel behind a padded copy of A, a piece of at most kPadBytes
// at a time: several whole sets, or a range of one set's rows.
constexpr int64_t kPadBytes = (int64_t)96 << 20;

template <int EB>
cudaError_t launch_padded_stream(const GemmParams &p, int batch, int n_sm, float *P, int64_t ldp, void *W,
                                 int64_t ldw, cudaStream_t s, bool &used)
{
    const int64_t most = std::max<int64_t>(kPadBytes / (ldp * 4) / kTcBM * kTcBM, kTcBM);
    const int sets = (int)std::min<int64_t>(batch, std::max<int64_t>(1, most / p.M));
    const int64_t rows = std::min<int64_t>(p.M, most);
    for (int b = 0; b < batch; b += sets)
        for (int64_t m = 0; m < p.M; m += rows) {
            const int nb = std::min(sets, batch - b);
            GemmParams q = p;
            q.M = (int)std::min<int64_t>(rows, p.M - m);
            q.A = P;
            q.lda = ldp;
            q.strideA = ldp * q.M;
            q.B = p.B + b * p.strideB;
            q.C = p.C + b * p.strideC + m * p.ldc;
            const int64_t n = (int64_t)nb * q.M;
            pad_rows_kernel<<<(unsigned)std::min<int64_t>((n + 7) / 8, (int64_t)n_sm * 16), 256, 0, s>>>(
                p.A + b * p.strideA + m * p.lda, p.lda, p.strideA, q.M, p.K, n, ldp, P);
            cudaError_t e = cudaGetLastError();
            if (e == cudaSuccess) e = launch_dense_stream<EB>(q, nb, n_sm, W, ldw, s, used);
            if (e != cudaSuccess || !used) return e;
        }
    return cudaSuccess;
}

template <int EB>
cudaError_t launch_tc(pne_ctx *ctx, const GemmParams &p, int batch, cudaStream_t s)
{
    const bool aligned = (reinterpret_cast<uintptr_t>(p.A) & 15) == 0 && p.lda % 4 == 0 &&
                         (batch == 1 || (p.strideA % 4 == 0 && p.strideA > 0));
    const int BN = std::min(256, ((p.N + 15) / 16) * 16);
    // The copying kernel takes about K (128 + BN) loads per block, one by one;
    // the persistent one costs a launch and a workspace more.  Whole calls
    // cross between 64 x 64 x 64 (34.0 against 35.1 us TF32, 33.5 against 34.8
    // BF16) and 512 x 128 x 128 (50.4 against 36.9, 46.4 against 35.2), BF16
    // the later (16 x 640 x 64 x 100: 45.9 against 36.2 TF32, 34.6 against 35.8
    // BF16); many blocks take it at any K.
    const int64_t blocks = (int64_t)((p.M + kTcBM - 1) / kTcBM) * ((p.N + BN - 1) / BN) * batch;
    // Rows of A off the 16-byte boundaries are copied to a padded piece first,
    // which many columns repay: 2 x 22748 x 995 x 125 in BF16 327 -> 127 us, 2000 x
    // 300 x 77 47 -> 30, 512 x 128 x 127 31.4 -> 29.9; but 65536 x 16 x 131 35 -> 49,
    // and 16 x 640 x 64 x 99 26 -> 27.
    const bool deep = (int64_t)p.K * (kTcBM + BN) >= (EB == 4 ? 14000 : 20000);
    if (aligned ? deep || blocks >= 2 * ctx->n_sm : deep && p.N >= 96) {
        const int64_t ldw = ((int64_t)p.K * EB + 15) / 16 * 16 / EB, ldp = ((int64_t)p.K + 3) / 4 * 4;
        const int64_t pad = aligned ? 0
                                    : std::min<int64_t>((int64_t)batch * p.M * ldp * 4,
                                                        std::max(kPadBytes, (int64_t)kTcBM * ldp * 4));
        const int64_t w_bytes = ((int64_t)batch * p.N * ldw * EB + 15) / 16 * 16;
        DevBuf W;
        if (dev_alloc(ctx, W, (size_t)(w_bytes + pad), s) == PNE_OK) {
            bool used = false;
            const cudaError_t e =
                aligned ? launch_dense_stream<EB>(p, batch, ctx->n_sm, W.ptr, ldw, s, used)
                        : launch_padded_stream<EB>(p, batch, ctx->n_sm, (float *)((char *)W.ptr + w_bytes), ldp, W.ptr,
                                                   ldw, s, used);
            dev_free(ctx, W, s);
            if (e != cudaSuccess || used) return e;
        } else {
            (void)cudaGetLastError();     // no room for the workspace: the copying kernel needs none
        }
    }
    const size_t smem = tc_smem_bytes(BN);
    cudaError_t e = grant_dynamic_smem((const void *)tc_gemm_kernel<EB>, smem);
    if (e != cudaSuccess) return e;
    const dim3 grid((unsigned)((p.M + kTcBM - 1) / kTcBM), (unsigned)((p.N + BN - 1) / BN), (unsigned)batch);
    tc_gemm_kernel<EB><<<grid, kTcThreads, smem, s>>>(p, BN);
    return cudaGetLastError();
}

template <int G, bool RING>
cudaError_t launch_f64_units(const F64Params &p, dim3 grid, cudaStream_t s)
{
    const size_t smem = 2 * f64_stage(G) * sizeof(double);
    const cudaError_t e = grant_dynamic_smem((const void *)f64_gemm_kernel<G, RING>, smem);
    if (e != cudaSuccess) return e;
    f64_gemm_kernel<G, RING><<<grid, kF64Threads, smem, s>>>(p);
    return cudaGetLastError();
}

// A block's run of f64_gemm_kernel: for the fewest waves of one block per SM that
// 12 units a warp allow, and three more, as many blocks as the waves hold; of
// these the run that ends first, a wave taking its units per scheduler and two
// more for filling and storing; or four units a warp, whose blocks share an SM
// by twos and so hide that (M = N = 4096, K = 512, 13.7 ms on the pipes alone:
// 13.88 ms, 14.15 as waves of single blocks).  A run of n units may touch
// (n - 2) / columns + 2 row groups, of which 16 are staged, so few columns take
// short runs; four units are one per scheduler.
template <bool RING>
cudaError_t launch_f64(F64Params p, int batch, int n_sm, cudaStream_t s)
{
    const int64_t groups = (p.M - 1) / 16 + 1, cu = (p.N - 1) / 4 + 1;
    const int64_t cblocks = (cu + kF64Cols / 4 - 1) / (kF64Cols / 4);
    p.cub = (int)((cu + cblocks - 1) / cblocks);
    const int64_t units = groups * p.cub, P = cblocks * batch;
    const int64_t narrow = cu - (cblocks - 1) * p.cub;       // units across the last column block
    const int64_t most = std::min<int64_t>(kF64Warps * kF64MaxUnits, (kF64Rows / 16 - 1) * narrow + 1);
    const int64_t least = (units + most - 1) / most, w0 = (P * least + n_sm - 1) / n_sm;
    int64_t cost = INT64_MAX;
    for (int64_t w = w0; w < w0 + 4; ++w) {
        const int64_t b = w * n_sm / P;
        const int64_t run = std::max<int64_t>((units + b - 1) / b, 4);
        if (w * ((run + 3) / 4 + 2) >= cost) continue;
        cost = w * ((run + 3) / 4 + 2);
        p.run = (int)run;
    }
    const int64_t pair = std::min<int64_t>(kF64Warps * 4, most);
    if (((units + pair - 1) / pair * P + n_sm - 1) / n_sm * ((pair + 3) / 4) + 2 < cost) p.run = (int)pair;
    const dim3 grid((unsigned)((units + p.run - 1) / p.run), (unsigned)cblocks, (unsigned)batch);
    switch ((p.run + kF64Warps - 1) / kF64Warps) {
    case 1: return launch_f64_units<1, RING>(p, grid, s);
    case 2: return launch_f64_units<2, RING>(p, grid, s);
    case 3: return launch_f64_units<3, RING>(p, grid, s);
    case 4: return launch_f64_units<4, RING>(p, grid, s);
    case 5: return launch_f64_units<5, RING>(p, grid, s);
    case 6: return launch_f64_units<6, RING>(p, grid, s);
    case 7: return launch_f64_units<7, RING>(p, grid, s);
    case 8: return launch_f64_units<8, RING>(p, grid, s);
    case 9: return launch_f64_units<9, RING>(p, grid, s);
    case 10: return launch_f64_units<10, RING>(p, grid, s);
    case 11: return launch_f64_units<11, RING>(p, grid, s);
    default: return launch_f64_units<kF64MaxUnits, RING>(p, grid, s);
    }
}

}  // namespace

pne_status grid_plan(pne_ctx *ctx, int lx, int ly, int n_bonds, const int32_t *bond_site, const int32_t *bond_dim,
                     const int32_t *site_ptr, const int32_t *site_bonds, const int64_t *data_off, pne_dtype dtype,
                     int nb, GridPlan &plan)
{
    auto bad = [&](const std::string &m) { set_error(ctx, PNE_EINVAL, m); return PNE_EINVAL; };
    const int n = lx * ly;
    // bond between grid neighbours: horizontal hb[v] (x, y)-(x+1, y), vertical vb[v] (x, y)-(x, y+1)
    std::vector<int> hb((size_t)n, -1), vb((size_t)n, -1);
    for (int b = 0; b < n_bonds; ++b) {
        int s0 = bond_site[2 * b], s1 = bond_site[2 * b + 1];
        if (s0 < 0 || s1 < 0 || s0 >= n || s1 >= n) return bad("grid networks have no open indices");
        if (s0 > s1) std::swap(s0, s1);
        const int x0 = s0 % lx, y0 = s0 / lx, x1 = s1 % lx, y1 = s1 / lx;
        const int d = bond_dim[b];
        if (d < 1 || d > 4096) return bad("bond dimension out of range");
        if (y0 == y1 && x1 == x0 + 1) {
            if (hb[s0] >= 0) return bad("two bonds join the same grid neighbours");
            hb[s0] = b;
        } else if (x0 == x1 && y1 == y0 + 1) {
            if (vb[s0] >= 0) return bad("two bonds join the same grid neighbours");
            vb[s0] = b;
        } else {
            return bad("a bond does not join grid neighbours (site id = y * lx + x)");
        }
    }
    for (int y = 0; y < ly; ++y)
        for (int x = 0; x < lx; ++x) {
            const int v = y * lx + x;
            if ((x + 1 < lx && hb[v] < 0) || (y + 1 < ly && vb[v] < 0)) return bad("a grid bond is missing");
        }
    plan.n = n;
    plan.maps.assign((size_t)n, SiteMap{});
    plan.steps.assign((size_t)n, GridStep{});
    plan.ldb.assign((size_t)n, 0);
    const size_t esz = dtype == PNE_F64 ? 8 : (dtype == PNE_TF32 ? 4 : 2);
    const int epu = dtype == PNE_F64 ? 1 : (int)(16 / esz);
    int64_t b_total = 0, state = 1, max_state = 1;
    for (int y = 0; y < ly; ++y)
        for (int x = 0; x < lx; ++x) {
            const int v = y * lx + x;
            const int legb[4] = {x > 0 ? hb[v - 1] : -1, y > 0 ? vb[v - lx] : -1, x + 1 < lx ? hb[v] : -1,
                                 y + 1 < ly ? vb[v] : -1};
            SiteMap &sm = plan.maps[(size_t)v];
            const int p0 = site_ptr[v], p1 = site_ptr[v + 1];
            int nlegs = 0;
            for (int i = 0; i < 4; ++i) nlegs += legb[i] >= 0;
            if (p1 - p0 != nlegs) return bad("a site's legs are not its grid bonds");
            for (int i = 0; i < 4; ++i) {
                sm.dim[i] = legb[i] >= 0 ? bond_dim[legb[i]] : 1;
                sm.stride[i] = 0;
            }
            // strides: legs in the order of site_bonds, row-major
            int64_t stride = 1;
            for (int q = p1 - 1; q >= p0; --q) {
                const int b = site_bonds[q];
                int which = -1;
                for (int i = 0; i < 4; ++i)
                    if (legb[i] == b) which = i;
                if (which < 0) return bad("a site's legs are not its grid bonds");
                if (stride > INT32_MAX) return bad("site tensor too large");
                sm.stride[which] = (int)stride;
                stride *= bond_dim[b];
            }
            if (data_off[v + 1] - data_off[v] != stride) return bad("data_off does not match the bond dims");
            sm.t_off = data_off[v];
            GridStep sd{sm.dim[1], sm.dim[0], sm.dim[3], sm.dim[2], 0};
            const int64_t K = (int64_t)sd.Ku * sd.Kh;
            if (state % K != 0) return bad("internal: running tensor does not split");
            sd.R = state / K;
            if (sd.R > INT32_MAX || (int64_t)sd.Nd * sd.Nh > INT32_MAX || K > INT32_MAX)
                return bad("a step's matrix is too large");
            plan.ldb[(size_t)v] = (K + epu - 1) / epu * epu;
            sm.b_off = b_total;
            b_total += plan.ldb[(size_t)v] * sd.Nd * sd.Nh;
            state = sd.R * sd.Nd * sd.Nh;
            max_state = std::max(max_state, std::max(state, sd.R * K));
            plan.steps[(size_t)v] = sd;
        }
    if (state != 1) return bad("internal: the contraction did not close");
    plan.b_total = b_total;
    plan.max_state = (max_state + 63) / 64 * 64;
    if ((double)plan.max_state * esz * 2 * nb > 64e9) return bad("running tensors exceed 64 GB for this batch");
    return PNE_OK;
}

pne_status grid_run(pne_ctx *ctx, const GridPlan &plan, const double *data, int64_t set_stride, int nb,
                    pne_dtype dtype, cudaStream_t s, std::vector<double> &h, double &bound)
{
    const int n = plan.n;
    const size_t esz = dtype == PNE_F64 ? 8 : (dtype == PNE_TF32 ? 4 : 2);
    const int64_t max_state = plan.max_state, b_total = plan.b_total;
    DevBuf dMaps, dB, dS, dA, dMax, dLog, dOut, dErr, dLdb;
    auto cleanup = [&]() {
        for (DevBuf *b : {&dMaps, &dB, &dS, &dA, &dMax, &dLog, &dOut, &dErr, &dLdb}) dev_free(ctx, *b, s);
    };
    pne_status st;
    if ((st = dev_alloc(ctx, dMaps, plan.maps.size() * sizeof(SiteMap), s)) ||
        (st = dev_alloc(ctx, dB, (size_t)nb * b_total * esz, s)) ||
        (st = dev_alloc(ctx, dS, (size_t)nb * max_state * esz, s)) ||
        (st = dev_alloc(ctx, dA, (size_t)nb * max_state * esz, s)) || (st = dev_alloc(ctx, dMax, (size_t)nb * 24, s)) ||
        (st = dev_alloc(ctx, dLog, (size_t)nb * 8, s)) || (st = dev_alloc(ctx, dOut, (size_t)nb * 16, s)) ||
        (st = dev_alloc(ctx, dErr, 16, s)) || (st = dev_alloc(ctx, dLdb, (size_t)n * 8, s))) {
        cleanup();
        return st;
    }
    auto fail = [&](cudaError_t e, const char *what) {
        set_error(ctx, PNE_ECUDA, std::string(what) + ": " + cudaGetErrorString(e));
        cleanup();
        return PNE_ECUDA;
    };
    cudaError_t e = cudaMemcpyAsync(dMaps.ptr, plan.maps.data(), plan.maps.size() * sizeof(SiteMap),
                                    cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(dLdb.ptr, plan.ldb.data(), (size_t)n * 8, cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) e = cudaMemsetAsync(dErr.ptr, 0, 16, s);
    if (e == cudaSuccess) e = cudaMemsetAsync(dMax.ptr, 0, (size_t)nb * 24, s);
    if (e != cudaSuccess) return fail(e, "grid upload");
    unsigned long long *mb = (unsigned long long *)dMax.ptr;
    long long *lg = (long long *)dLog.ptr;
    const int ib = (nb + 127) / 128;
    bound = 0.0;
    const double u_in = dtype == PNE_TF32 ? std::ldexp(1.0, -11) : (dtype == PNE_BF16 ? std::ldexp(1.0, -8) : 0.0);
    if (dtype != PNE_F64) {
        // running tensors ping-pong between dS and dA; largest |entry| in three rotating slots
        auto run_tc = [&](auto tag) -> cudaError_t {
            using E = decltype(tag);
            E *S0 = (E *)dS.ptr, *S1 = (E *)dA.ptr;
            cudaError_t ee;
            {
                ProfScope ps(ctx, s, "grid_sites");
                grid_init_kernel<E><<<ib, 128, 0, s>>>(S0, max_state, mb, lg, nb);
                ee = cudaGetLastError();
                if (ee == cudaSuccess)
                    ee = launch_grid_sites<E>(plan, nb, data, set_stride, (const SiteMap *)dMaps.ptr, (E *)dB.ptr,
                                              (const int64_t *)dLdb.ptr, lg, s);
            }
            if (ee != cudaSuccess) return ee;
            for (int v = 0; v < n; ++v) {
                const GridStep &sd = plan.steps[(size_t)v];
                RingParams<E> rp;
                rp.S = (v & 1) ? S1 : S0;
                rp.out = (v & 1) ? S0 : S1;
                rp.B = (const E *)dB.ptr + plan.maps[(size_t)v].b_off;
                rp.stride = max_state;
                rp.b_stride = b_total;
                rp.ldb = plan.ldb[(size_t)v];
                rp.R = sd.R;
                rp.Ku = sd.Ku;
                rp.Kh = sd.Kh;
                rp.N = sd.Nd * sd.Nh;
                rp.K = sd.Ku * sd.Kh;
                rp.max_in = mb + (size_t)(v % 3) * nb;
                rp.max_out = mb + (size_t)((v + 1) % 3) * nb;
                rp.max_clear = mb + (size_t)((v + 2) % 3) * nb;
                rp.log2s = lg;
                rp.err = (int *)dErr.ptr;
                ProfScope ps(ctx, s, "grid_gemm_tc");
                if ((ee = launch_grid_stream<E>(rp, nb, ctx->n_sm, s)) != cudaSuccess) return ee;
                bound += 2.0 * u_in + (double)rp.K * std::ldexp(1.0, -24);
            }
            {
                ProfScope ps(ctx, s, "grid_final");
                grid_final_kernel<E><<<ib, 128, 0, s>>>((n & 1) ? S1 : S0, max_state, lg, nb, (double *)dOut.ptr);
            }
            return cudaGetLastError();
        };
        e = dtype == PNE_TF32 ? run_tc(float(0)) : run_tc(__nv_bfloat16());
        if (e != cudaSuccess) return fail(e, "grid contraction (tensor cores)");
    } else {
        double *S0 = (double *)dS.ptr, *S1 = (double *)dA.ptr;
        {
            ProfScope ps(ctx, s, "grid_sites");
            grid_init_kernel<double><<<ib, 128, 0, s>>>(S0, max_state, mb, lg, nb);
            e = cudaGetLastError();
            if (e == cudaSuccess)
                e = launch_grid_sites<double>(plan, nb, data, set_stride, (const SiteMap *)dMaps.ptr, (double *)dB.ptr,
                                              (const int64_t *)dLdb.ptr, lg, s);
        }
        if (e != cudaSuccess) return fail(e, "grid site matrices");
        for (int v = 0; v < n; ++v) {
            const GridStep &sd = plan.steps[(size_t)v];
            F64Params p{};
            p.A = (v & 1) ? S1 : S0;
            p.strideA = max_state;
            p.B = (const double *)dB.ptr + plan.maps[(size_t)v].b_off;
            p.ldb = plan.ldb[(size_t)v];
            p.strideB = b_total;
            p.C = (v & 1) ? S0 : S1;
            p.strideC = max_state;
            p.M = (int)sd.R;
            p.N = sd.Nd * sd.Nh;
            p.K = sd.Ku * sd.Kh;
            p.ldc = p.N;
            p.R = sd.R;
            p.Kh = sd.Kh;
            p.max_in = mb + (size_t)(v % 3) * nb;
            p.max_out = mb + (size_t)((v + 1) % 3) * nb;
            p.max_clear = mb + (size_t)((v + 2) % 3) * nb;
            p.log2s = lg;
            {
                ProfScope ps(ctx, s, "grid_gemm_f64");
                e = launch_f64<true>(p, nb, ctx->n_sm, s);
            }
            if (e != cudaSuccess) return fail(e, "grid GEMM");
            bound += (double)p.K * std::ldexp(1.0, -53);
        }
        {
            ProfScope ps(ctx, s, "grid_final");
            grid_final_kernel<double><<<ib, 128, 0, s>>>((n & 1) ? S1 : S0, max_state, lg, nb, (double *)dOut.ptr);
        }
        if ((e = cudaGetLastError()) != cudaSuccess) return fail(e, "grid_final_kernel");
    }
    h.assign((size_t)nb * 2, 0.0);
    int herr = 0;
    if ((e = cudaMemcpyAsync(h.data(), dOut.ptr, h.size() * 8, cudaMemcpyDeviceToHost, s)) != cudaSuccess ||
        (e = cudaMemcpyAsync(&herr, dErr.ptr, 4, cudaMemcpyDeviceToHost, s)) != cudaSuccess ||
        (e = cudaStreamSynchronize(s)) != cudaSuccess)
        return fail(e, "grid results");
    cleanup();
    if (herr) {
        set_error(ctx, PNE_ETIMEOUT, "grid contraction: a tensor-core stage wait gave up");
        return PNE_ETIMEOUT;
    }
    return PNE_OK;
}

}  // namespace pne

using namespace pne;

extern "C" {

pne_status pne_dense_gemm(pne_ctx *ctx, pne_dtype dtype, int32_t batch, int32_t M, int32_t N, int32_t K,
                          const void *A, int64_t lda, int64_t strideA, const void *B, int64_t ldb, int64_t strideB,
                          void *C, int64_t ldc, int64_t strideC, void *stream)
{
    HostScope hs__(ctx, "dense_gemm");
    if (!ctx || !A || !B || !C) return PNE_EINVAL;
    auto bad = [&](const std::string &m) { set_error(ctx, PNE_EINVAL, m); return PNE_EINVAL; };
    if (batch < 1 || batch > 65535 || M < 1 || N < 1 || K < 1) return bad("batch in 1..65535, M, N, K >= 1");
    if (lda < K || ldb < K || ldc < N) return bad("leading dimensions below K (A, B) or N (C)");
    if (dtype == PNE_F32) return bad("dense_gemm takes PNE_F64, PNE_TF32 or PNE_BF16");
    cudaStream_t s = (cudaStream_t)stream;
    // A wait of the tensor-core kernels that gave up is told in host memory where
    // the kernel can write it: a word on the device takes a clear before and a copy
    // after the product (BF16: 4 x 32768 x 256 x 256 80 us a call with them, 73 to
    // 77 without; 128 x 16 x 16 31 and 17).  The word is the call's own, from the
    // context's pool.
    size_t flag_bytes = 0;
    int *flag = dtype == PNE_F64 ? nullptr : (int *)take_pinned(ctx, sizeof(int), &flag_bytes);
    DevBuf err;
    cudaError_t e = cudaSuccess;
    if (flag) {
        *(volatile int *)flag = 0;
    } else if (dtype != PNE_F64) {
        (void)cudaGetLastError();
        const pne_status st = dev_alloc(ctx, err, 16, s);
        if (st) return st;
        e = cudaMemsetAsync(err.ptr, 0, 16, s);
    }
    if (e == cudaSuccess) {
        ProfScope ps(ctx, s, dtype == PNE_F64 ? "dense_gemm_f64" : "dense_gemm_tc");
        if (dtype == PNE_F64) {
            F64Params p{};
            p.A = (const double *)A;
            p.lda = lda;
            p.strideA = strideA;
            p.B = (const double *)B;
            p.ldb = ldb;
            p.strideB = strideB;
            p.C = (double *)C;
            p.ldc = ldc;
            p.strideC = strideC;
            p.M = M;
            p.N = N;
            p.K = K;
            e = launch_f64<false>(p, batch, ctx->n_sm, s);
        } else {
            GemmParams p{(const float *)A, lda, strideA, (const float *)B, ldb, strideB, (float *)C, ldc,
                                strideC, M, N, K, flag ? flag : (int *)err.ptr};
            e = dtype == PNE_TF32 ? launch_tc<4>(ctx, p, batch, s) : launch_tc<2>(ctx, p, batch, s);
        }
    }
    int herr = 0;
    if (e == cudaSuccess && err.ptr) e = cudaMemcpyAsync(&herr, err.ptr, 4, cudaMemcpyDeviceToHost, s);
    const cudaError_t done = cudaStreamSynchronize(s);       // no kernel may write the word after the call
    if (e == cudaSuccess) e = done;
    if (flag) herr = *(volatile int *)flag;
    give_pinned(ctx, flag, flag_bytes);
    dev_free(ctx, err, s);
    if (e != cudaSuccess) {
        set_error(ctx, PNE_ECUDA, std::string("dense_gemm: ") + cudaGetErrorString(e));
        return PNE_ECUDA;
    }
    if (herr) {
        set_error(ctx, PNE_ETIMEOUT, "dense_gemm: a tensor-core stage wait gave up");
        return PNE_ETIMEOUT;
    }
    return PNE_OK;
}

pne_status pne_grid_contract(pne_ctx *ctx, const pne_network *net, int32_t lx, int32_t ly, pne_dtype dtype,
                             void *stream, pne_result *out)
{
    HostScope hs__(ctx, "grid_contract");
    if (!ctx || !net || !out) return PNE_EINVAL;
    auto bad = [&](const std::string &m) { set_error(ctx, PNE_EINVAL, m); return PNE_EINVAL; };
    if (dtype == PNE_F32) return bad("grid_contract takes PNE_F64, PNE_TF32 or PNE_BF16");
    const int nb = net->n_batch;
    if (nb < 1 || nb > 65535) return bad("n_batch in 1..65535");
    if (!net->bond_site || !net->bond_dim || !net->site_ptr || !net->site_bonds || !net->data || !net->data_off)
        return bad("null network array");
    if (lx < 1 || ly < 1 || (int64_t)lx * ly != net->n_sites) return bad("n_sites must be lx * ly");
    GridPlan plan;
    pne_status st = grid_plan(ctx, lx, ly, net->n_bonds, net->bond_site, net->bond_dim, net->site_ptr,
                              net->site_bonds, net->data_off, dtype, nb, plan);
    if (st) return st;
    cudaStream_t s = (cudaStream_t)stream;
    const int64_t set_stride = net->data_off[net->n_sites];
    DevBuf dData;
    const double *data = net->data;
    if (!net->data_on_device) {
        if ((st = dev_alloc(ctx, dData, (size_t)nb * set_stride * 8, s))) return st;
        if ((st = upload(ctx, dData.ptr, net->data, (size_t)nb * set_stride * 8, s))) {
            dev_free(ctx, dData, s);
            return st;
        }
        data = (const double *)dData.ptr;
    }
    std::vector<double> h;
    double bound = 0.0;
    st = grid_run(ctx, plan, data, set_stride, nb, dtype, s, h, bound);
    dev_free(ctx, dData, s);
    if (st != PNE_OK && st != PNE_ETIMEOUT) return st;
    for (int b = 0; b < nb; ++b) {
        pne_result &r = out[b];
        std::memset(&r, 0, sizeof(r));
        const double m = h[2 * b], l2 = h[2 * b + 1];
        r.sign = m > 0 ? 1 : (m < 0 ? -1 : 0);
        r.log_abs = m != 0 ? std::log(std::fabs(m)) + l2 * std::log(2.0) : -INFINITY;
        r.value = m != 0 ? (double)r.sign * std::exp(r.log_abs) : 0.0;
        r.n_orders = 1;
        r.c[0] = 1.0;
        r.abs_c[0] = 1.0;
        r.log_abs_zref = r.log_abs;
        r.sign_zref = r.sign;
        r.log_series = r.log_abs;
        r.err_bound = bound;
        r.n_terms = 1;
    }
    return st;
}

}  // extern "C"
