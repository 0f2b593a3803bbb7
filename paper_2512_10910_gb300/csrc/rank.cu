// Rank-r projectors by weight passing (App. C) and the expansions built on
// them (Sec. V.A).
//
// Weight passing keeps a diagonal weight matrix S_i on every bond.  An update
// of bond i between tensors A and B (Eq. weight1-3) absorbs the weights of the
// other legs into A and B, takes the SVD of each (as a matrix between index i
// and the rest), then of S_A V_A^T S_i U_B S_B = U_C S_C V_C^T, and re-gauges
//     A <- A V_A S_A^{-1} U_C S_C^{(1-alpha)/2},
//     B <- S_C^{(1-alpha)/2} V_C^T S_B^{-1} U_B^T B,    S_i <- S_C^alpha,
// which leaves the network (with the weights inserted) unchanged.  Only the
// right singular vectors and values of the matricised tensors are needed: a
// Householder QR reduces each to a d x d triangle, whose SVD (and that of the
// d x d core) is taken by one-sided Jacobi rotations (Hestenes), in FP64.
// A cluster of up to eight thread blocks per tensor set runs the sweeps over
// the bonds in id order.
//
// The rank-r expansion restricts, per term, each bond's index to the P range
// [0, r) of the r largest weights, to the Q range [r, d), or leaves it whole,
// and contracts the weighted network exactly: a block per (term, tensor set)
// absorbs the sites one by one into a dense running tensor over the open
// frontier (FP64 multiply-adds).
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <limits>
#include <string>
#include <vector>

#include "jacobi.h"
#include "pne_internal.h"

struct pne_weights {
    pne_ctx *ctx = nullptr;
    std::shared_ptr<pne::GeomPair> geo;
    int n_sets = 1;
    pne::DevBuf T;           // [n_sets][stride] weighted network (sqrt(S) absorbed)
    pne::DevBuf S;           // [n_sets][n_bonds][16]
    std::vector<double> log_scale;
    std::vector<int32_t> sweeps;
    cudaStream_t last_stream = nullptr;
};

namespace pne {

// the geometry of a validated network through the context's cache (pne_api.cu)
pne_status geometry_for(pne_ctx *ctx, const pne_network *net, cudaStream_t s, std::shared_ptr<GeomPair> &out,
                        int max_dim, int64_t max_size);

namespace {

constexpr int kWpDim = kJacobiDim;      // largest bond dimension of weight passing
constexpr int kWpThreads = kJacobiThreads;
constexpr int kWpWarps = kWpThreads / 32;
constexpr int kWpRows = 4;              // rows a thread holds during the QR
constexpr int kWpPanel = kWpThreads * kWpRows;
constexpr int kWpCluster = 8;           // most blocks per tensor set (portable cluster size)
constexpr int kWpParts = kWpCluster;    // most parts of a matrix's rows
constexpr int kWpLd = kJacobiLd;

// What the blocks of one set pass to each other, in global memory (read past
// L1), each field written between two cluster barriers and read after them.
struct WPShare {
    double R[kWpParts][kWpDim * kWpDim];        // triangles of each part of the rows, side A then side B
    double RB[kWpParts][kWpDim * kWpDim];
    double WB[kWpDim * kWpDim], sB[kWpDim];     // U_B (column c at c * kWpDim) and S_B
    double XL[kWpDim * kWpDim], XR[kWpDim * kWpDim];   // leg transforms [in][out]
    int code;                                   // 0 next bond, 1 a bad singular value, 2 converged
};

struct WPParams {
    int n_sets, n_sites, n_bonds;
    const int32_t *site_ptr, *site_bonds, *bond_dim, *bond_site, *bond_leg;
    const int64_t *tens_off;
    int64_t set_stride;
    double *T;                 // [n_sets][stride]: re-gauged in place, weighted at the end
    double *S;                 // [n_sets][n_bonds][kWpDim]
    WPShare *share;            // [n_sets]
    double alpha, tol;
    int max_sweeps;
    double *log_scale;         // [n_sets]
    int32_t *sweeps;           // [n_sets] (0: not converged)
    int32_t *flags;            // [n_sets] 1: a zero singular value, or one that is not finite
};

__device__ __forceinline__ void wp_barrier(int blocks)
{
    if (blocks == 1) __syncthreads();
    else asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}

// Sums of NV values over the warp, one per group of 32 / NV lanes: value
// lane / (32 / NV) is returned.  Halving the list at each exchange takes NV
// additions instead of 5 NV; FP64 additions are what the QR's reductions cost
// (an SM retires two lanes per clock).
template <int NV>
__device__ __forceinline__ double warp_sums(double (&v)[NV])
{
    const int lane = threadIdx.x & 31;
    int off = 16;
#pragma unroll
    for (int h = NV / 2; h >= 1; h >>= 1, off >>= 1) {
        const bool up = lane & off;
#pragma unroll
        for (int k = 0; k < h; ++k) {
            const double give = up ? v[k] : v[k + h], keep = up ? v[k + h] : v[k];
            v[k] = keep + __shfl_xor_sync(0xffffffffu, give, off);
        }
    }
    double t = v[0];
#pragma unroll
    for (; off >= 1; off >>= 1) t += __shfl_xor_sync(0xffffffffu, t, off);
    return t;
}

struct QrShared {
    double R[kWpDim][kWpDim];           // the triangle so far
    double part[kWpWarps][kWpDim];      // per-warp sums of one column step
    double f[kWpDim];
};

// One column step of the QR of [R; panel]: the reflection with head R[J][J]
// and tail column J of the panel zeroes that column.  All inner products of
// column J with columns J.. are formed in one pass over the registers and one
// reduction; one warp turns them into the factors.
template <int DM, int J>
__device__ __forceinline__ void qr_column(double (&x)[kWpRows][DM], int nr, QrShared &q, int d)
{
    constexpr int N = DM - J;
    constexpr int NV = N > 8 ? 16 : (N > 4 ? 8 : (N > 2 ? 4 : (N > 1 ? 2 : 1)));
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (nr > 0) {
        double g[NV];
#pragma unroll
        for (int c = 0; c < NV; ++c) g[c] = c < N ? x[0][J] * x[0][J + c < DM ? J + c : J] : 0.0;
#pragma unroll
        for (int r = 1; r < kWpRows; ++r)
            if (r < nr) {
#pragma unroll
                for (int c = 0; c < N; ++c) g[c] = fma(x[r][J], x[r][J + c], g[c]);
            }
        const double t = warp_sums<NV>(g);
        constexpr int per = 32 / NV;
        if (lane % per == 0) q.part[warp][lane / per] = t;
    } else if (lane < NV) {
        q.part[warp][lane] = 0.0;
    }
    __syncthreads();
    if (warp == 0) {
        const int c = lane & 15;
        double s = 0.0;
        if (c < N)
            for (int w = lane >> 4; w < kWpWarps; w += 2) s += q.part[w][c];
        s += __shfl_xor_sync(0xffffffffu, s, 16);       // lane c: sum over the panel of column J times column J + c
        const double s0 = __shfl_sync(0xffffffffu, s, 0);
        const double head = q.R[J][J];
        const double nrm = sqrt(fma(head, head, s0));
        const double diag = head >= 0.0 ? -nrm : nrm, vj = head - diag;
        const double vn2 = fma(vj, vj, s0);
        const double beta = (s0 > 0.0 && vn2 > 0.0) ? 2.0 / vn2 : 0.0;
        if (lane < N) {
            if (lane == 0) {
                if (beta != 0.0) q.R[J][J] = diag;
                q.f[J] = 0.0;
            } else {
                const double old = q.R[J][J + lane];
                const double f = beta * fma(vj, old, s);
                q.R[J][J + lane] = fma(-f, vj, old);
                q.f[J + lane] = f;
            }
        }
    }
    __syncthreads();
#pragma unroll
    for (int c = J + 1; c < DM; ++c) {
        if (c >= d) break;
        const double f = q.f[c];
#pragma unroll
        for (int r = 0; r < kWpRows; ++r)
            if (r < nr) x[r][c] = fma(-f, x[r][J], x[r][c]);
    }
}

template <int DM, int J>
__device__ __forceinline__ void qr_columns(double (&x)[kWpRows][DM], int nr, QrShared &q, int d)
{
    if constexpr (J < DM) {
        if (J < d) {
            qr_column<DM, J>(x, nr, q, d);
            qr_columns<DM, J + 1>(x, nr, q, d);
        }
    }
}

// The triangle of the QR of `rows` rows of d values, load(row, x) giving one,
// into q.R.  A thread holds four rows of a panel in registers for all d column
// steps (the panel is read once; the column-by-column form walked the matrix
// 2 d times through L2), and each panel is stacked under the triangle so far.
template <int DM, class Load>
__device__ void qr_rows(const Load &load, int rows, int d, QrShared &q)
{
    const int warp = threadIdx.x >> 5;
    __syncthreads();
    for (int e = threadIdx.x; e < kWpDim * kWpDim; e += kWpThreads) q.R[e / kWpDim][e % kWpDim] = 0.0;
    __syncthreads();
    for (int p0 = 0; p0 < rows; p0 += kWpPanel) {
        double x[kWpRows][DM];
        int nr = 0;
#pragma unroll
        for (int r = 0; r < kWpRows; ++r) {
            const int row = p0 + r * kWpThreads + (int)threadIdx.x;
            if (p0 + r * kWpThreads + warp * 32 < rows) nr = r + 1;
#pragma unroll
            for (int c = 0; c < DM; ++c) x[r][c] = 0.0;
            if (row < rows) load(row, x[r]);
        }
        qr_columns<DM, 0>(x, nr, q, d);
    }
    __syncthreads();
}

// A site's legs as one bond update needs them
struct WPSite {
    const double *T;
    int64_t T_off;
    int k, l, d, rest;
    int dims[kMaxDeg], stride[kMaxDeg], bond[kMaxDeg];
};

__device__ WPSite wp_site(const WPParams &p, const double *Tset, int v, int l)
{
    WPSite s;
    const int l0 = p.site_ptr[v];
    s.k = p.site_ptr[v + 1] - l0;
    s.l = l;
    s.T_off = p.tens_off[v];
    s.T = Tset + s.T_off;
    int stride = 1;
    for (int i = s.k - 1; i >= 0; --i) {
        s.bond[i] = p.site_bonds[l0 + i];
        s.dims[i] = p.bond_dim[s.bond[i]];
        s.stride[i] = stride;
        stride *= s.dims[i];
    }
    s.d = s.dims[l];
    s.rest = stride / s.d;
    return s;
}

// Start of row `row` (the other legs row-major) in the site's tensor; the
// product of those legs' weights (Sset, read past L1) in *wgt when asked for
__device__ __forceinline__ int wp_row(const WPSite &s, int row, const double *Sset, double *wgt)
{
    int off = 0;
    double w = 1.0;
    for (int i = s.k - 1; i >= 0; --i) {
        if (i == s.l) continue;
        const int q = row / s.dims[i], dg = row - q * s.dims[i];
        row = q;
        off += dg * s.stride[i];
        if (wgt) w *= __ldcg(Sset + (int64_t)s.bond[i] * kWpDim + dg);
    }
    if (wgt) *wgt = w;
    return off;
}

// Parts of the rows of a matricised tensor above one panel: a panel each, up to
// eight.  It follows from the tensor alone, so that a set gets the same bits with any
// number of blocks, that is in any batch.  3 x 3, D = 9 (729 rows), 1, 30, 60 and 100
// sets: 70.0, 81.5, 93.0, 144 ms; with parts of 128 rows 69.2, 85.1, 102, 162.
__device__ __forceinline__ int wp_parts(int rest) { return min(kWpParts, (rest + kWpPanel - 1) / kWpPanel); }

// The updates of one tensor set by a cluster of blocks.  Per bond: the rows of
// a matricised tensor above one panel are split into parts, dealt to the blocks
// and each reduced to a triangle; block 0 takes A (stacking the triangles, or the
// whole of a small tensor) to its SVD while block 1 takes B; block 0 forms the
// core, its SVD, the weights and the leg transforms; every block multiplies
// its rows.  FP64 multiply-adds bound the large tensors (two per clock and
// SM: 2 x 1.05 M for a 16^4 tensor, so the split over SMs is what pays), the
// chain of column steps and Jacobi rounds the small ones.
// Measured, blocked Ising 3 x 3, 8 sets, 0.65 to 0.8 T_c: chi = 16 933 -> 99 ms
// (one block of 256 threads per set walked each matrix column by column in L2
// and rotated one pair of columns at a time), chi = 8 264 -> 52, chi = 4 97 -> 31.
template <int DM>
__global__ void __launch_bounds__(kWpThreads) weight_passing_kernel(WPParams p, int blocks)
{
    __shared__ QrShared q;
    __shared__ double WA[kWpDim * kWpLd], WBs[kWpDim * kWpLd], WC[kWpDim * kWpLd], VC[kWpDim * kWpLd];
    __shared__ double X[2][kWpDim * kWpDim];
    __shared__ double sA[kWpDim], sB[kWpDim], sC[kWpDim], gC[kWpDim];
    __shared__ int bad_sh;
    const int set = blockIdx.x / blocks, rank = blockIdx.x % blocks, tid = threadIdx.x;
    double *Tset = p.T + (int64_t)set * p.set_stride;
    double *Sset = p.S + (int64_t)set * p.n_bonds * kWpDim;
    WPShare &sh = p.share[set];
    for (int64_t i = rank * kWpThreads + tid; i < (int64_t)p.n_bonds * kWpDim; i += blocks * kWpThreads)
        Sset[i] = ((int)(i % kWpDim) < p.bond_dim[i / kWpDim]) ? 1.0 : 0.0;
    double scale = 0.0, change = 0.0;      // kept by block 0's first warp
    int code = 0, sweep = 0;               // without a bond the first sweep changes nothing
    wp_barrier(blocks);
    while (code == 0 && sweep < p.max_sweeps) {
        ++sweep;
        change = 0.0;
        if (p.n_bonds == 0) code = 2;
        for (int b = 0; b < p.n_bonds && code != 1; ++b) {
            const WPSite sa = wp_site(p, Tset, p.bond_site[2 * b], p.bond_leg[2 * b]);
            const WPSite sb = wp_site(p, Tset, p.bond_site[2 * b + 1], p.bond_leg[2 * b + 1]);
            const int d = sa.d;
            const bool split_a = sa.rest > kWpPanel, split_b = sb.rest > kWpPanel;
            auto rows_of = [&](const WPSite &s, int lo) {
                return [&s, lo, Sset](int row, double (&x)[DM]) {
                    double w;
                    const double *t = s.T + wp_row(s, lo + row, Sset, &w);
#pragma unroll
                    for (int c = 0; c < DM; ++c)
                        if (c < s.d) x[c] = __ldcg(t + (int64_t)c * s.stride[s.l]) * w;
                };
            };
            auto share_rows = [&](const WPSite &s, double (*R)[kWpDim * kWpDim]) {
                const int parts = wp_parts(s.rest), per = (s.rest + parts - 1) / parts;
                for (int part = rank; part < parts; part += blocks) {
                    const int lo = min(s.rest, part * per);
                    qr_rows<DM>(rows_of(s, lo), min(s.rest, lo + per) - lo, d, q);
                    for (int e = tid; e < kWpDim * kWpDim; e += kWpThreads)
                        __stcg(&R[part][e], q.R[e / kWpDim][e % kWpDim]);
                }
            };
            if (split_a) share_rows(sa, sh.R);
            if (split_b) share_rows(sb, sh.RB);
            if (split_a || split_b) wp_barrier(blocks);
            // The right vectors V and singular values of one side's triangle.  V is the product of
            // the rotations: its small entries are right to their own size, which the columns of
            // R^T Q / S = V are not, and the leg transforms divide them by weights as small.
            auto side = [&](const WPSite &s, bool split, const double (*R)[kWpDim * kWpDim], double *V, double *sig) {
                if (split)
                    qr_rows<DM>([&](int row, double (&x)[DM]) {
#pragma unroll
                        for (int c = 0; c < DM; ++c)
                            if (c < d) x[c] = __ldcg(&R[row / d][row % d * kWpDim + c]);
                    }, wp_parts(s.rest) * d, d, q);
                else
                    qr_rows<DM>(rows_of(s, 0), s.rest, d, q);
                for (int e = tid; e < d * d; e += kWpThreads) {
                    WC[e % d * kWpLd + e / d] = q.R[e / d][e % d];
                    V[e / d * kWpLd + e % d] = e / d == e % d ? 1.0 : 0.0;
                }
                __syncthreads();
                jacobi_columns(WC, V, sig, d);
                __syncthreads();
            };
            const int rank_b = blocks > 1 ? 1 : 0;
            if (rank == 0) side(sa, split_a, sh.R, WA, sA);
            if (rank == rank_b) {
                side(sb, split_b, sh.RB, WBs, sB);
                if (blocks > 1) {
                    for (int e = tid; e < d * d; e += kWpThreads) __stcg(&sh.WB[e / d * kWpDim + e % d], WBs[e / d * kWpLd + e % d]);
                    if (tid < d) __stcg(&sh.sB[tid], sB[tid]);
                }
            }
            if (blocks > 1) wp_barrier(blocks);
            if (rank == 0) {
                if (blocks > 1) {
                    for (int e = tid; e < d * d; e += kWpThreads) WBs[e / d * kWpLd + e % d] = __ldcg(&sh.WB[e / d * kWpDim + e % d]);
                    if (tid < d) sB[tid] = __ldcg(&sh.sB[tid]);
                }
                __syncthreads();
                const bool bad_side = tid < d && (!(sA[tid] > 1e-300) || !(sB[tid] > 1e-300));
                // core M = S_A V_A^T S_i U_B S_B and its SVD
                double *Si = Sset + (int64_t)b * kWpDim;
                for (int e = tid; e < d * d; e += kWpThreads) {
                    const int a = e / d, c = e % d;
                    double acc = 0.0;
                    for (int x = 0; x < d; ++x) acc = fma(WA[a * kWpLd + x] * __ldcg(Si + x), WBs[c * kWpLd + x], acc);
                    WC[c * kWpLd + a] = sA[a] * acc * sB[c];
                    VC[c * kWpLd + a] = a == c ? 1.0 : 0.0;
                }
                const bool sides_ok = !__syncthreads_or(bad_side);
                if (sides_ok) jacobi_columns(WC, VC, sC, d);         // WC -> U_C S_C, VC = V_C
                if (sides_ok && tid < 32) {
                    const double s = tid < d ? sC[tid] : 0.0;
                    const double w = tid < d ? pow(s, p.alpha) : 0.0;
                    if (tid < d) gC[tid] = pow(s, 0.5 * (1.0 - p.alpha));
                    double mx = w;
                    for (int off = 16; off > 0; off >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, off));
                    scale += log(mx);
                    const double nw = w / mx;
                    // a zero singular value, or one that overflowed (fmax passes a NaN over)
                    const bool bad = __any_sync(0xffffffffu, tid < d && (!(s > 1e-300) || nw != nw));
                    if (tid == 0) bad_sh = bad;
                    double ch = tid < d ? fabs(nw - __ldcg(Si + tid)) : 0.0;
                    for (int off = 16; off > 0; off >>= 1) ch = fmax(ch, __shfl_xor_sync(0xffffffffu, ch, off));
                    change = fmax(change, ch);
                    if (tid < d) __stcg(Si + tid, nw);
                }
                __syncthreads();
                const bool ok = sides_ok && !bad_sh;
                if (ok) {
                    // left = V_A S_A^{-1} U_C S_C^{(1-alpha)/2} on A's leg,
                    // right = S_C^{(1-alpha)/2} V_C^T S_B^{-1} U_B^T on B's, as [in][out]
                    for (int e = tid; e < d * d; e += kWpThreads) {
                        const int c = e / d, at = c * kWpLd + e % d;
                        WA[at] = WA[at] / sA[c];
                        WBs[at] = WBs[at] / sB[c];
                        WC[at] = WC[at] / sC[c];
                    }
                    __syncthreads();
                    for (int e = tid; e < 2 * d * d; e += kWpThreads) {
                        const int side_b = e >= d * d, f = e - side_b * d * d, a = f / d, c = f % d;
                        const double *L = (side_b ? WBs : WA) + a, *R = (side_b ? VC : WC) + c * kWpLd;
                        double acc = 0.0;
                        for (int x = 0; x < d; ++x) acc = fma(L[x * kWpLd], R[x], acc);
                        __stcg((side_b ? sh.XR : sh.XL) + a * kWpDim + c, acc * gC[c]);
                    }
                }
                if (tid == 0) __stcg(&sh.code, !ok ? 1 : (b == p.n_bonds - 1 && change < p.tol ? 2 : 0));
            }
            wp_barrier(blocks);
            code = __ldcg(&sh.code);
            if (code != 1) {
                for (int e = tid; e < d * d; e += kWpThreads) {
                    X[0][e / d * kWpDim + e % d] = __ldcg(sh.XL + e / d * kWpDim + e % d);
                    X[1][e / d * kWpDim + e % d] = __ldcg(sh.XR + e / d * kWpDim + e % d);
                }
                __syncthreads();
                // rows of both tensors times their transform, a row per thread
                for (int side_b = 0; side_b < 2; ++side_b) {
                    const WPSite &s = side_b ? sb : sa;
                    const double *Xs = X[side_b];
                    const int st = s.stride[s.l];
                    for (int row = rank * kWpThreads + tid; row < s.rest; row += blocks * kWpThreads) {
                        double *t = Tset + s.T_off + wp_row(s, row, nullptr, nullptr);
                        double in[DM], out[DM];
#pragma unroll
                        for (int c = 0; c < DM; ++c) {
                            in[c] = c < d ? __ldcg(t + (int64_t)c * st) : 0.0;
                            out[c] = 0.0;
                        }
#pragma unroll
                        for (int a = 0; a < DM; ++a) {
                            if (a >= d) break;
#pragma unroll
                            for (int c = 0; c < DM; ++c)
                                if (c < d) out[c] = fma(in[a], Xs[a * kWpDim + c], out[c]);
                        }
#pragma unroll
                        for (int c = 0; c < DM; ++c)
                            if (c < d) __stcg(t + (int64_t)c * st, out[c]);
                    }
                }
            }
            wp_barrier(blocks);
        }
    }
    if (rank == 0 && tid == 0) {
        p.sweeps[set] = code == 2 ? sweep : 0;
        p.flags[set] = code == 1;
        p.log_scale[set] = scale;
    }
    // the weighted network: sqrt(S) into both ends of every bond
    for (int v = 0; v < p.n_sites; ++v) {
        const int l0 = p.site_ptr[v], k = p.site_ptr[v + 1] - l0;
        const int n = (int)(p.tens_off[v + 1] - p.tens_off[v]);
        double *T = Tset + p.tens_off[v];
        for (int e = rank * kWpThreads + tid; e < n; e += blocks * kWpThreads) {
            int r = e;
            double w = 1.0;
            for (int i = k - 1; i >= 0; --i) {
                const int bd = p.site_bonds[l0 + i], dim = p.bond_dim[bd], dg = r % dim;
                r /= dim;
                w *= sqrt(__ldcg(Sset + (int64_t)bd * kWpDim + dg));
            }
            __stcg(T + e, __ldcg(T + e) * w);
        }
    }
}

template <int DM>
cudaError_t launch_weight_passing(const WPParams &p, int blocks, cudaStream_t s)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(p.n_sets * blocks), 1, 1);
    cfg.blockDim = dim3(kWpThreads, 1, 1);
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)blocks;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = blocks > 1 ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, weight_passing_kernel<DM>, p, blocks);
}

// ---------------------------------------------------------------- dense terms
constexpr int kDtThreads = 256;
constexpr int64_t kDtMaxFront = 1 << 18;      // entries of a running tensor
constexpr int kDtMaxLegs = 20;                // bonds of a frontier
constexpr int kDtMaxBonds = 1024;             // bonds of a network

// One step of the site-by-site contraction: the site absorbed, the frontier
// before (bond ids, in order) and after, and for each leg of the site its
// position in the old frontier (closing) or the new one (opening).
struct DtStep {
    int site, k, nf0, nf1;
    int f0[kDtMaxLegs];
    int f1[kDtMaxLegs];
    int leg_bond[kMaxDeg];
    int leg_old[kMaxDeg];       // position in f0, or -1
    int leg_new[kMaxDeg];       // position in f1, or -1
    int keep_new[kDtMaxLegs];   // for each position of f1: position in f0 (kept) or -1 (a new leg)
};

struct DtParams {
    const DtStep *steps;
    int n_steps, n_bonds, n_terms, n_sets;
    const int8_t *kind;          // [n_terms][n_bonds]: 0 whole, 1 P range, 2 Q range
    const int32_t *bond_dim;
    int rank;
    const double *T;             // [n_sets][stride] weighted network
    const int64_t *tens_off;
    int64_t set_stride;
    double *scratch;             // [grid][2][kDtMaxFront]
    double *value;               // [n_sets][n_terms]
};

__global__ void __launch_bounds__(kDtThreads) dense_term_kernel(DtParams p)
{
    __shared__ int lo[kDtMaxBonds], len[kDtMaxBonds];
    double *X = p.scratch + (int64_t)blockIdx.x * 2 * kDtMaxFront;
    double *Y = X + kDtMaxFront;
    const int64_t items = (int64_t)p.n_terms * p.n_sets;
    for (int64_t item = blockIdx.x; item < items; item += gridDim.x) {
        const int term = (int)(item % p.n_terms), set = (int)(item / p.n_terms);
        for (int b = threadIdx.x; b < p.n_bonds; b += blockDim.x) {
            const int kd = p.kind[(int64_t)term * p.n_bonds + b], d = p.bond_dim[b];
            lo[b] = (kd == 2) ? p.rank : 0;
            len[b] = (kd == 0) ? d : (kd == 1 ? p.rank : d - p.rank);
        }
        if (threadIdx.x == 0) X[0] = 1.0;
        __syncthreads();
        const double *Tset = p.T + (int64_t)set * p.set_stride;
        for (int s = 0; s < p.n_steps; ++s) {
            const DtStep &st = p.steps[s];
            // sizes and row-major strides of the old and new frontiers
            int64_t n1 = 1;
            for (int i = 0; i < st.nf1; ++i) n1 *= len[st.f1[i]];
            int64_t str0[kDtMaxLegs];
            {
                int64_t m = 1;
                for (int i = st.nf0 - 1; i >= 0; --i) { str0[i] = m; m *= len[st.f0[i]]; }
            }
            int cl_len[kMaxDeg], cl_pos[kMaxDeg], nc = 0;
            int64_t ncomb = 1;
            for (int l = 0; l < st.k; ++l)
                if (st.leg_old[l] >= 0) { cl_pos[nc] = l; cl_len[nc] = len[st.leg_bond[l]]; ncomb *= cl_len[nc]; ++nc; }
            int dims[kMaxDeg];
            for (int l = 0; l < st.k; ++l) dims[l] = p.bond_dim[st.leg_bond[l]];
            const double *Tv = Tset + p.tens_off[st.site];
            for (int64_t o = threadIdx.x; o < n1; o += blockDim.x) {
                // digits of the new frontier (last fastest)
                int dg1[kDtMaxLegs];
                int64_t r = o;
                for (int i = st.nf1 - 1; i >= 0; --i) { const int L = len[st.f1[i]]; dg1[i] = (int)(r % L); r /= L; }
                int64_t xbase = 0;
                for (int i = 0; i < st.nf1; ++i)
                    if (st.keep_new[i] >= 0) xbase += dg1[i] * str0[st.keep_new[i]];
                int tdg[kMaxDeg];
                for (int l = 0; l < st.k; ++l)
                    tdg[l] = (st.leg_new[l] >= 0) ? lo[st.leg_bond[l]] + dg1[st.leg_new[l]] : 0;
                double acc = 0.0;
                for (int64_t c = 0; c < ncomb; ++c) {
                    int64_t rc = c, xo = xbase;
                    for (int j = nc - 1; j >= 0; --j) {
                        const int l = cl_pos[j];
                        const int dg = (int)(rc % cl_len[j]);
                        rc /= cl_len[j];
                        xo += dg * str0[st.leg_old[l]];
                        tdg[l] = lo[st.leg_bond[l]] + dg;
                    }
                    int64_t to = 0;
                    for (int l = 0; l < st.k; ++l) to = to * dims[l] + tdg[l];
                    acc = fma(X[xo], Tv[to], acc);
                }
                Y[o] = acc;
            }
            __syncthreads();
            double *t = X; X = Y; Y = t;
        }
        if (threadIdx.x == 0) p.value[(int64_t)set * p.n_terms + term] = X[0];
        __syncthreads();
        // X, Y alternate per step: restore the block's buffer order
        X = p.scratch + (int64_t)blockIdx.x * 2 * kDtMaxFront;
        Y = X + kDtMaxFront;
    }
}

// One term's tensors with every bond's index restricted to [lo_b, lo_b + len_b):
// block per (site, set), row-major over the site's legs in ascending bond id.
__global__ void restrict_kernel(const double *__restrict__ T, int64_t set_stride, const int64_t *tens_off,
                                const int32_t *site_ptr, const int32_t *site_bonds, const int32_t *bond_dim,
                                const int32_t *lo, const int32_t *len, const int64_t *new_off, int64_t new_stride,
                                double *out)
{
    const int v = blockIdx.x, set = blockIdx.y;
    const int p0 = site_ptr[v], p1 = site_ptr[v + 1];
    const int64_t n_out = new_off[v + 1] - new_off[v];
    const double *src = T + set * set_stride + tens_off[v];
    double *dst = out + set * new_stride + new_off[v];
    for (int64_t q = threadIdx.x; q < n_out; q += blockDim.x) {
        int64_t r = q, off = 0, stride = 1;
        for (int i = p1 - 1; i >= p0; --i) {
            const int b = site_bonds[i];
            const int64_t digit = r % len[b];
            r /= len[b];
            off += (lo[b] + digit) * stride;
            stride *= bond_dim[b];
        }
        dst[q] = src[off];
    }
}

struct RankTerms {
    std::vector<int8_t> kind;       // [n_terms][n_bonds]: 0 whole, 1 P range, 2 Q range
    std::vector<int> order, sign;
    int M = 0;
};

pne_status rank_terms(pne_ctx *ctx, const Geometry &g, int32_t rank, int32_t form, int32_t n_partitions,
                      const int32_t *partition_ptr, const int32_t *partition_bonds, RankTerms &t)
{
    auto bad = [&](const std::string &m) { set_error(ctx, PNE_EINVAL, m); return PNE_EINVAL; };
    const int M = n_partitions, NB = g.n_bonds;
    if (M < 1 || M > 20) return bad("1..20 partitions");
    if (form != 0 && form != 1) return bad("form is 0 (linear) or 1 (combinatorial)");
    if (partition_ptr[0] != 0) return bad("partition_ptr[0] must be 0");
    std::vector<std::vector<int>> parts(M);
    for (int p = 0; p < M; ++p) {
        if (partition_ptr[p + 1] <= partition_ptr[p]) return bad("every partition needs at least one bond");
        for (int i = partition_ptr[p]; i < partition_ptr[p + 1]; ++i) {
            const int b = partition_bonds[i];
            if (b < 0 || b >= NB) return bad("partition bond out of range");
            if (rank < 1 || rank >= g.bond_dim[b]) return bad("rank must be in 1 .. d - 1 on every partitioned bond");
            parts[p].push_back(b);
        }
        if (form == 0 && parts[p].size() != 1) return bad("the linear form takes single-index partitions");
    }
    if (form == 0)
        for (int p = 0; p < M; ++p)
            for (int q = p + 1; q < M; ++q)
                if (parts[p][0] == parts[q][0]) return bad("the linear form takes distinct bonds");
    t.M = M;
    t.kind.clear();
    t.order.clear();
    t.sign.clear();
    if (form == 0) {
        for (int k = 0; k < M; ++k) {
            std::vector<int8_t> row(NB, 0);
            for (int p = 0; p < k; ++p) row[parts[p][0]] = 2;
            row[parts[k][0]] = 1;
            t.kind.insert(t.kind.end(), row.begin(), row.end());
            t.order.push_back(k);
            t.sign.push_back(1);
        }
    } else {
        for (uint32_t x = 1; x < (1u << M); ++x) {
            std::vector<int8_t> row(NB, 0);
            int k = 0;
            for (int p = 0; p < M; ++p)
                if (x >> p & 1) { ++k; for (int b : parts[p]) row[b] = 1; }
            t.kind.insert(t.kind.end(), row.begin(), row.end());
            t.order.push_back(k);
            t.sign.push_back((k % 2 == 1) ? 1 : -1);
        }
    }
    return PNE_OK;
}

// per set: c[k], abs_c[k], the signed Neumaier sum of the term values (in the
// weighted network's scale), log_abs with the weights' log scale, and the
// a-priori bound: FP64 rounding of nops operations per term plus, for a
// reduced-precision contraction, bound_abs[set][term] = the contraction's
// relative bound x |value| (relative to each term's absolute contraction,
// which equals |value| for a term of non-negative tensors)
void rank_results(const pne_weights *w, int form, const RankTerms &t, const std::vector<double> &vals,
                  const std::vector<double> &bound_abs, int nops, pne_result *out)
{
    const int n_terms = (int)t.order.size();
    for (int set = 0; set < w->n_sets; ++set) {
        pne_result &r = out[set];
        std::memset(&r, 0, sizeof r);
        const int K = form == 0 ? t.M - 1 : t.M;
        r.n_orders = K + 1;
        double sum = 0.0, comp = 0.0, asum = 0.0, rb = 0.0;
        for (int q = 0; q < n_terms; ++q) {
            const double v = vals[(size_t)set * n_terms + q];
            r.c[t.order[q]] += v;
            r.abs_c[t.order[q]] += std::fabs(v);
        }
        for (int q = 0; q < n_terms; ++q) {            // Neumaier over the terms, in term order
            const double x = t.sign[q] * vals[(size_t)set * n_terms + q], tt = sum + x;
            comp += (std::fabs(sum) >= std::fabs(x)) ? (sum - tt) + x : (x - tt) + sum;
            sum = tt;
            asum += std::fabs(x);
            if (!bound_abs.empty()) rb += bound_abs[(size_t)set * n_terms + q];
        }
        sum += comp;
        const double ls = w->log_scale[set];
        r.log_abs_zref = ls;
        r.sign_zref = 1;
        r.sign = sum < 0 ? -1 : 1;
        r.log_abs = (sum != 0.0) ? ls + std::log(std::fabs(sum)) : -std::numeric_limits<double>::infinity();
        r.value = (sum == 0.0) ? 0.0 : (r.log_abs > 709.7 ? r.sign * std::numeric_limits<double>::infinity()
                                                           : r.sign * std::exp(r.log_abs));
        r.log_series = std::numeric_limits<double>::quiet_NaN();
        const double u = 0x1p-53;
        r.err_bound = (sum != 0.0) ? ((nops * u / (1 - nops * u)) * asum + rb) / std::fabs(sum)
                                   : std::numeric_limits<double>::infinity();
        r.n_terms = (uint64_t)n_terms;
        r.bp_iters = w->sweeps[set];
    }
}

// Every term network (bond kinds per term: 0 whole, 1 P range [0, rank), 2 Q
// range [rank, d)) contracted as a grid: the restricted tensors gathered per
// term, then the row-by-row GEMMs.  vals / bound_abs [set][term].
pne_status grid_term_values(pne_ctx *ctx, const pne_weights *w, const std::vector<int8_t> &kind, int n_terms,
                            int32_t rank, int32_t lx, int32_t ly, pne_dtype dtype, cudaStream_t s,
                            std::vector<double> &vals, std::vector<double> &bound_abs)
{
    const Geometry &g = w->geo->full;
    const int NB = g.n_bonds, ns = w->n_sets;
    vals.assign((size_t)ns * n_terms, 0.0);
    bound_abs.assign((size_t)ns * n_terms, 0.0);
    std::vector<int32_t> lo((size_t)NB), len((size_t)NB);
    std::vector<int64_t> off((size_t)g.n_sites + 1);
    DevBuf dlo, dlen, doff, ddata;
    auto cleanup = [&]() { dev_free(ctx, dlo, s); dev_free(ctx, dlen, s); dev_free(ctx, doff, s); dev_free(ctx, ddata, s); };
    pne_status st;
    if ((st = dev_alloc(ctx, dlo, (size_t)NB * 4, s)) || (st = dev_alloc(ctx, dlen, (size_t)NB * 4, s)) ||
        (st = dev_alloc(ctx, doff, off.size() * 8, s)) ||
        (st = dev_alloc(ctx, ddata, (size_t)ns * g.tens_off[g.n_sites] * 8, s))) {
        cleanup();
        return st;
    }
    for (int q = 0; q < n_terms; ++q) {
        for (int b = 0; b < NB; ++b) {
            const int kd = kind[(size_t)q * NB + b], d = g.bond_dim[b];
            lo[(size_t)b] = kd == 2 ? rank : 0;
            len[(size_t)b] = kd == 0 ? d : (kd == 1 ? rank : d - rank);
        }
        off[0] = 0;
        for (int v = 0; v < g.n_sites; ++v) {
            int64_t sz = 1;
            for (int i = g.site_ptr[v]; i < g.site_ptr[v + 1]; ++i) sz *= len[(size_t)g.site_bonds[i]];
            off[(size_t)v + 1] = off[(size_t)v] + sz;
        }
        GridPlan plan;
        if ((st = grid_plan(ctx, lx, ly, NB, g.bond_site.data(), len.data(), g.site_ptr.data(), g.site_bonds.data(),
                            off.data(), dtype, ns, plan)) ||
            (st = upload(ctx, dlo.ptr, lo.data(), (size_t)NB * 4, s)) ||
            (st = upload(ctx, dlen.ptr, len.data(), (size_t)NB * 4, s)) ||
            (st = upload(ctx, doff.ptr, off.data(), off.size() * 8, s))) {
            cleanup();
            return st;
        }
        {
            ProfScope ps(ctx, s, "rank_restrict");
            restrict_kernel<<<dim3(g.n_sites, ns), 256, 0, s>>>((const double *)w->T.ptr, g.tens_off[g.n_sites],
                                                                g.d_tens_off, g.d_site_ptr, g.d_site_bonds,
                                                                g.d_bond_dim, (const int32_t *)dlo.ptr,
                                                                (const int32_t *)dlen.ptr, (const int64_t *)doff.ptr,
                                                                off[(size_t)g.n_sites], (double *)ddata.ptr);
        }
        if (cudaGetLastError() != cudaSuccess) {
            cleanup();
            set_error(ctx, PNE_ECUDA, "restrict_kernel launch failed");
            return PNE_ECUDA;
        }
        std::vector<double> h;
        double bound = 0.0;
        if ((st = grid_run(ctx, plan, (const double *)ddata.ptr, off[(size_t)g.n_sites], ns, dtype, s, h, bound))) {
            cleanup();
            return st;
        }
        for (int set = 0; set < ns; ++set) {
            const double v = std::ldexp(h[2 * (size_t)set], (int)h[2 * (size_t)set + 1]);
            vals[(size_t)set * n_terms + q] = v;
            bound_abs[(size_t)set * n_terms + q] = dtype == PNE_F64 ? 0.0 : bound * std::fabs(v);
        }
    }
    cleanup();
    return PNE_OK;
}

}  // namespace
}  // namespace pne

// ======================================================================= host
using namespace pne;

namespace {

// Site order of the dense contraction: from site 0, repeatedly the site whose
// absorption leaves the smallest frontier (whole dimensions), ties by id; the
// steps record the frontiers before and after and where each leg goes.
pne_status dense_plan(pne_ctx *ctx, const Geometry &g, std::vector<DtStep> &steps, int64_t &max_front)
{
    const int N = g.n_sites;
    std::vector<char> in(N, 0);
    std::vector<int> front;                 // frontier bonds, in order
    max_front = 1;
    for (int s = 0; s < N; ++s) {
        int best = -1;
        double best_size = 0.0;
        for (int v = 0; v < N; ++v) {
            if (in[v]) continue;
            double size = 1.0;
            for (int b : front) {
                const bool closes = g.bond_site[2 * b] == v || g.bond_site[2 * b + 1] == v;
                if (!closes) size *= g.bond_dim[b];
            }
            for (int i = g.site_ptr[v]; i < g.site_ptr[v + 1]; ++i) {
                const int b = g.site_bonds[i];
                const int o = g.bond_site[2 * b] == v ? g.bond_site[2 * b + 1] : g.bond_site[2 * b];
                if (!in[o]) size *= g.bond_dim[b];
            }
            // prefer a site that touches the frontier (keeps components together)
            bool touches = front.empty();
            for (int b : front)
                if (g.bond_site[2 * b] == v || g.bond_site[2 * b + 1] == v) touches = true;
            const double key = touches ? size : size * 1e30;
            if (best < 0 || key < best_size) { best = v; best_size = key; }
        }
        const int v = best;
        DtStep st;
        std::memset(&st, 0, sizeof st);
        st.site = v;
        st.k = g.site_ptr[v + 1] - g.site_ptr[v];
        st.nf0 = (int)front.size();
        if (st.nf0 > kDtMaxLegs) { set_error(ctx, PNE_EINVAL, "frontier of the dense contraction too wide"); return PNE_EINVAL; }
        for (int i = 0; i < st.nf0; ++i) st.f0[i] = front[i];
        std::vector<int> nf;
        std::vector<int> keep;
        for (int i = 0; i < st.nf0; ++i) {
            const int b = front[i];
            if (g.bond_site[2 * b] == v || g.bond_site[2 * b + 1] == v) continue;
            nf.push_back(b);
            keep.push_back(i);
        }
        for (int l = 0; l < st.k; ++l) {
            const int b = g.site_bonds[g.site_ptr[v] + l];
            st.leg_bond[l] = b;
            st.leg_old[l] = -1;
            st.leg_new[l] = -1;
            for (int i = 0; i < st.nf0; ++i) if (front[i] == b) st.leg_old[l] = i;
            if (st.leg_old[l] < 0) {
                const int o = g.bond_site[2 * b] == v ? g.bond_site[2 * b + 1] : g.bond_site[2 * b];
                if (!in[o]) { st.leg_new[l] = (int)nf.size(); nf.push_back(b); keep.push_back(-1); }
            }
        }
        st.nf1 = (int)nf.size();
        if (st.nf1 > kDtMaxLegs) { set_error(ctx, PNE_EINVAL, "frontier of the dense contraction too wide"); return PNE_EINVAL; }
        int64_t size = 1;
        for (int i = 0; i < st.nf1; ++i) { st.f1[i] = nf[i]; st.keep_new[i] = keep[i]; size *= g.bond_dim[nf[i]]; }
        max_front = std::max(max_front, size);
        if (size > kDtMaxFront) {
            set_error(ctx, PNE_EINVAL, "an intermediate tensor of the dense contraction exceeds 2^18 entries");
            return PNE_EINVAL;
        }
        in[v] = 1;
        front = nf;
        steps.push_back(st);
    }
    return PNE_OK;
}

}  // namespace

extern "C" {

pne_status pne_weight_passing(pne_ctx *ctx, const pne_network *net, double alpha, double tol, int32_t max_sweeps,
                              void *stream, pne_weights **out)
{
    HostScope hs__(ctx, "weight_passing");
    if (!ctx || !net || !out) return PNE_EINVAL;
    *out = nullptr;
    auto bad = [&](const std::string &m) { set_error(ctx, PNE_EINVAL, m); return PNE_EINVAL; };
    if (!(alpha > 0.0 && alpha <= 1.0) || !(tol > 0.0) || max_sweeps < 1) return bad("alpha in (0, 1], tol > 0, max_sweeps > 0");
    cudaStream_t s = (cudaStream_t)stream;
    auto w = new pne_weights();
    w->ctx = ctx;
    // bond dimensions up to 16 and site tensors up to 2^20 entries here
    pne_status st = geometry_for(ctx, net, s, w->geo, kWpDim, (int64_t)1 << 20);
    if (st) { delete w; return st; }
    const Geometry &g = w->geo->full;
    if (!w->geo->open_bonds.empty()) { delete w; return bad("weight passing takes closed networks"); }
    for (int b = 0; b < g.n_bonds; ++b) {
        if (g.bond_dim[b] > kWpDim) { delete w; return bad("weight passing needs bond dimensions <= 16"); }
        for (int side = 0; side < 2; ++side) {
            const int v = g.bond_site[2 * b + side];
            const int64_t n = g.tens_off[v + 1] - g.tens_off[v];
            if (n / g.bond_dim[b] < g.bond_dim[b]) {
                delete w;
                return bad("a bond dimension exceeds the product of the other dimensions of its tensor");
            }
        }
    }
    const int B = net->n_batch;
    w->n_sets = B;
    const int64_t stride = g.tens_off[g.n_sites];
    int64_t tmax = 1;
    int dmax = 1;
    for (int v = 0; v < g.n_sites; ++v) tmax = std::max<int64_t>(tmax, g.tens_off[v + 1] - g.tens_off[v]);
    for (int b = 0; b < g.n_bonds; ++b) dmax = std::max(dmax, (int)g.bond_dim[b]);
    // Blocks per set: two take the two sides of a bond, more share the rows of
    // tensors above one panel, while every set's cluster fits the GPU at once.
    // 3 x 3, chi = 16, 8 sets: 212, 132, 110 and 99 ms with 1, 2, 4 and 8 blocks;
    // chi = 8 (512 rows, one panel): 73 and 52 with 1 and 2.
    int blocks = 1;
    const int most = tmax / dmax > kWpPanel ? kWpCluster : 2;
    while (2 * blocks <= most && 2 * blocks * B <= ctx->n_sm) blocks *= 2;
    DevBuf scratch, rec;
    if ((st = dev_alloc(ctx, w->T, (size_t)B * stride * 8, s)) ||
        (st = dev_alloc(ctx, w->S, (size_t)B * std::max(g.n_bonds, 1) * kWpDim * 8, s)) ||
        (st = dev_alloc(ctx, scratch, (size_t)B * sizeof(WPShare), s)) || (st = dev_alloc(ctx, rec, (size_t)B * 16, s))) {
        dev_free(ctx, scratch, s); dev_free(ctx, rec, s); pne_weights_destroy(w);
        return st;
    }
    PNE_CUDA_TRY(ctx, cudaMemcpyAsync(w->T.ptr, net->data, (size_t)B * stride * 8,
                                      net->data_on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice, s));
    WPParams p;
    p.n_sets = B; p.n_sites = g.n_sites; p.n_bonds = g.n_bonds;
    p.site_ptr = g.d_site_ptr; p.site_bonds = g.d_site_bonds; p.bond_dim = g.d_bond_dim; p.bond_site = g.d_bond_site;
    p.bond_leg = g.d_bond_leg; p.tens_off = g.d_tens_off; p.set_stride = stride;
    p.T = (double *)w->T.ptr; p.S = (double *)w->S.ptr;
    p.share = (WPShare *)scratch.ptr;
    p.alpha = alpha; p.tol = tol; p.max_sweeps = max_sweeps;
    p.log_scale = (double *)rec.ptr;
    p.sweeps = (int32_t *)((char *)rec.ptr + (size_t)B * 8);
    p.flags = p.sweeps + B;
    {
        ProfScope ps(ctx, s, "weight_passing");
        const cudaError_t e = dmax <= 4   ? launch_weight_passing<4>(p, blocks, s)
                              : dmax <= 8 ? launch_weight_passing<8>(p, blocks, s)
                                          : launch_weight_passing<16>(p, blocks, s);
        if (e != cudaSuccess) set_error(ctx, PNE_ECUDA, std::string("weight passing: ") + cudaGetErrorString(e));
    }
    PNE_LAUNCH_CHECK(ctx);
    std::vector<char> h((size_t)B * 16);
    PNE_CUDA_TRY(ctx, cudaMemcpyAsync(h.data(), rec.ptr, h.size(), cudaMemcpyDeviceToHost, s));
    dev_free(ctx, scratch, s);
    dev_free(ctx, rec, s);
    PNE_CUDA_TRY(ctx, cudaStreamSynchronize(s));
    w->log_scale.assign((const double *)h.data(), (const double *)h.data() + B);
    const int32_t *sw = (const int32_t *)(h.data() + (size_t)B * 8);
    w->sweeps.assign(sw, sw + B);
    w->last_stream = s;
    *out = w;
    for (int b = 0; b < B; ++b)
        if (sw[B + b]) { set_error(ctx, PNE_EDEGENERATE, "a singular value in weight passing is zero or not finite"); return PNE_EDEGENERATE; }
    for (int b = 0; b < B; ++b)
        if (sw[b] == 0) { set_error(ctx, PNE_ENOCONV, "weight passing did not converge for a tensor set"); return PNE_ENOCONV; }
    return PNE_OK;
}

pne_status pne_weights_read(pne_ctx *ctx, const pne_weights *w, void *stream, double *weights, int32_t *sweeps,
                            double *log_scale)
{
    if (!ctx || !w) return PNE_EINVAL;
    cudaStream_t s = (cudaStream_t)stream;
    if (weights) {
        const size_t n = (size_t)w->n_sets * std::max(w->geo->full.n_bonds, 1) * kWpDim;
        PNE_CUDA_TRY(ctx, cudaMemcpyAsync(weights, w->S.ptr, n * 8, cudaMemcpyDeviceToHost, s));
        PNE_CUDA_TRY(ctx, cudaStreamSynchronize(s));
    }
    if (sweeps) std::copy(w->sweeps.begin(), w->sweeps.end(), sweeps);
    if (log_scale) std::copy(w->log_scale.begin(), w->log_scale.end(), log_scale);
    return PNE_OK;
}

void pne_weights_destroy(pne_weights *w)
{
    if (!w) return;
    dev_free(w->ctx, w->T, w->last_stream);
    dev_free(w->ctx, w->S, w->last_stream);
    if (w->geo) w->geo->uses.note(w->ctx, w->last_stream);
    delete w;
}

pne_status pne_rank_r_expand(pne_ctx *ctx, const pne_weights *w, int32_t rank, int32_t form, int32_t n_partitions,
                             const int32_t *partition_ptr, const int32_t *partition_bonds, void *stream,
                             pne_result *out)
{
    HostScope hs__(ctx, "rank_r_expand");
    if (!ctx || !w || !out || !partition_ptr || !partition_bonds) return PNE_EINVAL;
    const Geometry &g = w->geo->full;
    const int NB = g.n_bonds;
    if (NB > kDtMaxBonds) {
        set_error(ctx, PNE_EINVAL, "too many bonds for the dense contraction");
        return PNE_EINVAL;
    }
    RankTerms t;
    pne_status st = rank_terms(ctx, g, rank, form, n_partitions, partition_ptr, partition_bonds, t);
    if (st) return st;
    const int n_terms = (int)t.order.size();
    std::vector<DtStep> steps;
    int64_t max_front = 1;
    st = dense_plan(ctx, g, steps, max_front);
    if (st) return st;
    cudaStream_t s = (cudaStream_t)stream;
    const int64_t items = (int64_t)n_terms * w->n_sets;
    const int grid = (int)std::max<int64_t>(1, std::min<int64_t>(items, 2 * (int64_t)ctx->n_sm));
    DevBuf dsteps, dkind, dscr, dval;
    if ((st = dev_alloc(ctx, dsteps, steps.size() * sizeof(DtStep), s)) || (st = dev_alloc(ctx, dkind, t.kind.size(), s)) ||
        (st = dev_alloc(ctx, dscr, (size_t)grid * 2 * kDtMaxFront * 8, s)) ||
        (st = dev_alloc(ctx, dval, (size_t)items * 8, s)) ||
        (st = upload(ctx, dsteps.ptr, steps.data(), steps.size() * sizeof(DtStep), s)) ||
        (st = upload(ctx, dkind.ptr, t.kind.data(), t.kind.size(), s))) {
        dev_free(ctx, dsteps, s); dev_free(ctx, dkind, s); dev_free(ctx, dscr, s); dev_free(ctx, dval, s);
        return st;
    }
    DtParams p;
    p.steps = (const DtStep *)dsteps.ptr; p.n_steps = (int)steps.size(); p.n_bonds = NB; p.n_terms = n_terms;
    p.n_sets = w->n_sets; p.kind = (const int8_t *)dkind.ptr; p.bond_dim = g.d_bond_dim; p.rank = rank;
    p.T = (const double *)w->T.ptr; p.tens_off = g.d_tens_off; p.set_stride = g.tens_off[g.n_sites];
    p.scratch = (double *)dscr.ptr; p.value = (double *)dval.ptr;
    {
        ProfScope ps(ctx, s, "dense_terms");
        dense_term_kernel<<<grid, kDtThreads, 0, s>>>(p);
    }
    if (cudaGetLastError() != cudaSuccess) {
        dev_free(ctx, dsteps, s); dev_free(ctx, dkind, s); dev_free(ctx, dscr, s); dev_free(ctx, dval, s);
        set_error(ctx, PNE_ECUDA, "dense_term_kernel launch failed");
        return PNE_ECUDA;
    }
    std::vector<double> vals((size_t)items);
    PNE_CUDA_TRY(ctx, cudaMemcpyAsync(vals.data(), dval.ptr, vals.size() * 8, cudaMemcpyDeviceToHost, s));
    dev_free(ctx, dsteps, s); dev_free(ctx, dkind, s); dev_free(ctx, dscr, s); dev_free(ctx, dval, s);
    PNE_CUDA_TRY(ctx, cudaStreamSynchronize(s));
    const_cast<pne_weights *>(w)->last_stream = s;
    const int nops = 2 * g.n_sites + (int)std::ceil(std::log2((double)std::max<int64_t>(max_front, 2))) + t.M + 2;
    rank_results(w, form, t, vals, {}, nops, out);
    return PNE_OK;
}

pne_status pne_rank_r_expand_grid(pne_ctx *ctx, const pne_weights *w, int32_t rank, int32_t form,
                                  int32_t n_partitions, const int32_t *partition_ptr, const int32_t *partition_bonds,
                                  int32_t lx, int32_t ly, pne_dtype dtype, void *stream, pne_result *out)
{
    HostScope hs__(ctx, "rank_r_expand_grid");
    if (!ctx || !w || !out || !partition_ptr || !partition_bonds) return PNE_EINVAL;
    auto bad = [&](const std::string &m) { set_error(ctx, PNE_EINVAL, m); return PNE_EINVAL; };
    const Geometry &g = w->geo->full;
    if (dtype == PNE_F32) return bad("rank_r_expand_grid takes PNE_F64, PNE_TF32 or PNE_BF16");
    if (lx < 1 || ly < 1 || (int64_t)lx * ly != g.n_sites) return bad("n_sites must be lx * ly");
    RankTerms t;
    pne_status st = rank_terms(ctx, g, rank, form, n_partitions, partition_ptr, partition_bonds, t);
    if (st) return st;
    cudaStream_t s = (cudaStream_t)stream;
    std::vector<double> vals, babs;
    if ((st = grid_term_values(ctx, w, t.kind, (int)t.order.size(), rank, lx, ly, dtype, s, vals, babs))) return st;
    const_cast<pne_weights *>(w)->last_stream = s;
    const int nops = 2 * g.n_sites + 4 * std::max(lx, ly) + t.M + 2;
    rank_results(w, form, t, vals, babs, nops, out);
    return PNE_OK;
}

pne_status pne_recursive_expand_grid(pne_ctx *ctx, const pne_weights *w, int32_t rank, int32_t n_partitions,
                                     const int32_t *partition_ptr, const int32_t *partition_bonds,
                                     int32_t n_sub_partitions, const int32_t *sub_ptr, const int32_t *sub_bonds,
                                     int32_t max_side, int32_t lx, int32_t ly, pne_dtype dtype, void *stream,
                                     pne_result *out, uint64_t *n_contractions)
{
    HostScope hs__(ctx, "recursive_expand_grid");
    if (!ctx || !w || !out || !partition_ptr || !partition_bonds || (n_sub_partitions > 0 && (!sub_ptr || !sub_bonds)))
        return PNE_EINVAL;
    auto bad = [&](const std::string &m) { set_error(ctx, PNE_EINVAL, m); return PNE_EINVAL; };
    const Geometry &g = w->geo->full;
    const int NB = g.n_bonds, N = g.n_sites;
    if (dtype == PNE_F32) return bad("recursive_expand_grid takes PNE_F64, PNE_TF32 or PNE_BF16");
    if (lx < 1 || ly < 1 || (int64_t)lx * ly != N) return bad("n_sites must be lx * ly");
    if (max_side < 1) return bad("max_side must be positive");
    if (n_partitions > 16) return bad("at most 16 first-level partitions");
    if (n_sub_partitions < 0 || n_sub_partitions > 64) return bad("0..64 second-level partitions");
    RankTerms t1;
    pne_status st = rank_terms(ctx, g, rank, 1, n_partitions, partition_ptr, partition_bonds, t1);
    if (st) return st;
    std::vector<std::vector<int>> sub((size_t)n_sub_partitions);
    for (int p = 0; p < n_sub_partitions; ++p) {
        if (sub_ptr[p + 1] <= sub_ptr[p] || (p == 0 && sub_ptr[0] != 0)) return bad("malformed second-level partitions");
        for (int i = sub_ptr[p]; i < sub_ptr[p + 1]; ++i) {
            const int b = sub_bonds[i];
            if (b < 0 || b >= NB) return bad("second-level partition bond out of range");
            if (rank >= g.bond_dim[b]) return bad("rank must be below every partitioned bond's dimension");
            sub[(size_t)p].push_back(b);
        }
    }
    // every first-level subset x: the cut bonds, the components left, and
    // either the sub-network itself or its expansion over the second-level
    // partitions that fit inside its too-large components
    const int n1 = (int)t1.order.size();
    std::vector<int8_t> kind;            // every network to contract
    std::vector<int> owner, sign2;       // its first-level term and second-level sign
    std::vector<int> parent((size_t)N);
    auto find = [&](int a) {
        while (parent[(size_t)a] != a) a = parent[(size_t)a] = parent[(size_t)parent[(size_t)a]];
        return a;
    };
    for (int q = 0; q < n1; ++q) {
        const int8_t *row = t1.kind.data() + (size_t)q * NB;
        for (int v = 0; v < N; ++v) parent[(size_t)v] = v;
        for (int b = 0; b < NB; ++b) {
            if (row[b] == 1) continue;
            const int ra = find(g.bond_site[2 * b]), rb = find(g.bond_site[2 * b + 1]);
            if (ra != rb) parent[(size_t)std::max(ra, rb)] = std::min(ra, rb);
        }
        // a component is too costly when both sides of its bounding box exceed max_side
        std::vector<int> x0((size_t)N, INT32_MAX), x1((size_t)N, -1), y0((size_t)N, INT32_MAX), y1((size_t)N, -1);
        for (int v = 0; v < N; ++v) {
            const size_t r = (size_t)find(v);
            x0[r] = std::min(x0[r], v % lx); x1[r] = std::max(x1[r], v % lx);
            y0[r] = std::min(y0[r], v / lx); y1[r] = std::max(y1[r], v / lx);
        }
        auto big = [&](int v) {
            const size_t r = (size_t)find(v);
            return std::min(x1[r] - x0[r] + 1, y1[r] - y0[r] + 1) > max_side;
        };
        std::vector<int> fit;
        for (int p = 0; p < n_sub_partitions; ++p) {
            bool ok = true;
            for (int b : sub[(size_t)p]) {
                const int s0 = g.bond_site[2 * b], s1 = g.bond_site[2 * b + 1];
                if (row[b] == 1 || !big(s0) || find(s0) != find(s1)) { ok = false; break; }
            }
            if (ok) fit.push_back(p);
        }
        if (fit.size() > 16) return bad("more than 16 second-level partitions fit one sub-network");
        if (fit.empty()) {
            kind.insert(kind.end(), row, row + NB);
            owner.push_back(q);
            sign2.push_back(1);
            continue;
        }
        for (uint32_t y = 1; y < (1u << fit.size()); ++y) {
            std::vector<int8_t> r2(row, row + NB);
            int k = 0;
            for (size_t i = 0; i < fit.size(); ++i)
                if (y >> i & 1) { ++k; for (int b : sub[(size_t)fit[i]]) r2[(size_t)b] = 1; }
            kind.insert(kind.end(), r2.begin(), r2.end());
            owner.push_back(q);
            sign2.push_back(k % 2 == 1 ? 1 : -1);
        }
    }
    const int nt = (int)owner.size();
    cudaStream_t s = (cudaStream_t)stream;
    std::vector<double> vals, babs;
    if ((st = grid_term_values(ctx, w, kind, nt, rank, lx, ly, dtype, s, vals, babs))) return st;
    const_cast<pne_weights *>(w)->last_stream = s;
    // first-level values: the second-level sums (Neumaier, in network order)
    const int ns = w->n_sets;
    std::vector<double> v1((size_t)ns * n1, 0.0), b1((size_t)ns * n1, 0.0), c1((size_t)ns * n1, 0.0);
    for (int set = 0; set < ns; ++set)
        for (int i = 0; i < nt; ++i) {
            const size_t a = (size_t)set * n1 + owner[(size_t)i];
            const double x = sign2[(size_t)i] * vals[(size_t)set * nt + i], tt = v1[a] + x;
            c1[a] += (std::fabs(v1[a]) >= std::fabs(x)) ? (v1[a] - tt) + x : (x - tt) + v1[a];
            v1[a] = tt;
            b1[a] += babs[(size_t)set * nt + i];
        }
    for (size_t a = 0; a < v1.size(); ++a) v1[a] += c1[a];
    const int nops = 2 * N + 4 * std::max(lx, ly) + t1.M + 2 + 20;
    rank_results(w, 1, t1, v1, b1, nops, out);
    for (int set = 0; set < ns; ++set) out[set].n_terms = (uint64_t)nt;
    if (n_contractions) *n_contractions = (uint64_t)nt;
    return PNE_OK;
}

}  // extern "C"
