// lu.cu -- blocked, partially pivoted LU in FP64 for the recompute (Sec. II.C, Eq. GrFMatNew).
//
// The re-orthonormalisation of the propagated factor U (N x Nsigma) and the solve
// (U_L U_R) Z = U_L both rest on an LU factorisation with partial pivoting.  GB300 runs FP64
// at a small fraction of its FP32 rate and every pivot is a grid-wide dependency, so the
// factorisation is blocked:
//   * a panel of LU_NB columns is factored by one thread-block cluster per matrix: each CTA
//     keeps its share of the rows in shared memory and the CTAs agree on every pivot by sending one
//     another their best rows through distributed shared memory;
//   * the pivot rows' trailing part U12 = L11^{-1} A12 and the trailing update A22 -= L21 U12 of the
//     unpivoted rows run over the whole GPU.
// Rows are not swapped: a pivoted row is flagged, keeps its multipliers left of its pivot
// column and its U entries from there on, and perm[j] names the pivot row of column j.  Both
// spins go through every launch (two independent matrices).
#include <cooperative_groups.h>
#include <limits.h>

#include <algorithm>

#include "internal.h"
#include "lu_cluster.h"

namespace afq {
namespace cg = cooperative_groups;

__device__ __forceinline__ double* lu_A(const LuArgs& a, int b) {
    return a.A0 + (long)(b / a.ng) * a.wstride + (long)(b % a.ng) * a.sstride;
}

constexpr int LU_NB = 32;
constexpr int LU_NBP = LU_NB + 1;

// A pivoted row's flag: its panel's number from 1 (a trailing update that runs beside the next panel tells
// the rows of that panel, which it still updates, from the earlier ones).
constexpr int LU_PANELS_MAX = 254;
__device__ __forceinline__ int8_t lu_flag(int j0) { return (int8_t)min(j0 / LU_NB + 1, LU_PANELS_MAX + 1); }

// One cluster of CS CTAs per matrix (blockIdx.x / CS = matrix).  Factors columns
// [j0, j0 + nbk) over the rows not yet pivoted.
// Pivot candidates compare |a| through the bit pattern of the double with the sign cleared:
// for finite non-negative doubles the integer order is the numeric order, and integer compares
// avoid the long FP64 latency on the pivot search's critical path.  Ties go to the lower row.
__device__ __forceinline__ unsigned long long lu_key(double x) {
    return (unsigned long long)__double_as_longlong(x) & 0x7fffffffffffffffULL;
}
__device__ __forceinline__ void lu_pick(unsigned long long& k, int& r, unsigned long long ok, int orr) {
    if (ok > k || (ok == k && orr < r)) {
        k = ok;
        r = orr;
    }
}

// The best candidate of a warp in every lane: largest key, ties to the lower row.  Three integer reductions.
// Returns the lane that holds it.
__device__ __forceinline__ int lu_warp_best(unsigned long long& k, int& r) {
    const unsigned hi = (unsigned)(k >> 32), lo = (unsigned)k;
    const unsigned mh = __reduce_max_sync(0xffffffffu, hi);
    const unsigned ml = __reduce_max_sync(0xffffffffu, hi == mh ? lo : 0u);
    const bool best = hi == mh && lo == ml;
    const unsigned mr = __reduce_min_sync(0xffffffffu, best ? (unsigned)r : 0xffffffffu);
    const int src = __ffs(__ballot_sync(0xffffffffu, best && (unsigned)r == mr)) - 1;
    k = ((unsigned long long)mh << 32) | ml;
    r = (int)mr;
    return src;
}

// ---- asynchronous stores between the CTAs of a cluster, counted by an mbarrier of the receiver ----
__device__ __forceinline__ unsigned lu_smem_u32(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }
__device__ __forceinline__ unsigned lu_mapa(unsigned addr, int rank) {
    unsigned r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
__device__ __forceinline__ void lu_st_async(unsigned dst, double v, unsigned bar) {
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.b64 [%0], %1, [%2];" ::"r"(dst),
                 "l"(__double_as_longlong(v)), "r"(bar)
                 : "memory");
}
__device__ __forceinline__ void lu_st_async(unsigned dst, int v, unsigned bar) {
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.b32 [%0], %1, [%2];" ::"r"(dst), "r"(v),
                 "r"(bar)
                 : "memory");
}
// Wait for phase `parity` of the mbarrier; false after two seconds of %globaltimer.
__device__ __forceinline__ bool lu_bar_wait(unsigned bar, unsigned parity) {
    unsigned long long t0 = 0;
    for (unsigned polls = 0;; ++polls) {
        unsigned ok;
        asm volatile(
            "{\n.reg .pred p;\nmbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n"
            "selp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(ok)
            : "r"(bar), "r"(parity)
            : "memory");
        if (ok) return true;
        if ((polls & 63u) == 63u) {
            unsigned long long t;
            asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
            if (t0 == 0) t0 = t;
            else if (t - t0 > 2000000000ULL) return false;
        }
    }
}

// tpr threads per row (a power of two up to 8).  Per column: every warp's candidate, one block barrier, and
// warp 0 sends the CTA's best row to all CTAs of the cluster (asynchronous stores counted by the receiver's
// mbarrier, double-buffered by step parity: no cluster barrier and no memory fence per step); when the CS rows
// have arrived, every warp picks the winner by itself, takes the reciprocal of the pivot, and updates its
// rows, the next column first for the next candidates.  A CTA sends its row of step j + 1 after all its warps
// are done with the rows of step j, so a buffer is free again when the rows of step j + 2 arrive.  Bound by
// that chain.  First panel of the 1600 x 700 factor: 128 us with one thread per row, the FP64 division and
// candidates read back through distributed shared memory behind a cluster barrier; 77 us with the
// candidates pushed before the cluster barrier and the pivot row read after it.
template <int CS>
__device__ __forceinline__ void lu_panel(const LuArgs& a, int j0, int nbk, int tpr) {
    cg::cluster_group cl = cg::this_cluster();
    const int rank = (int)cl.block_rank();
    const int mat = blockIdx.x / CS;
    double* A = lu_A(a, mat);
    int* perm = a.perm0 + (long)mat * a.pstride;
    int8_t* flag = a.flag0 + (long)mat * a.pstride;
    const int m = a.m;
    const long lda = a.lda;
    const int r0 = (int)((long)m * rank / CS), r1 = (int)((long)m * (rank + 1) / CS), nr = r1 - r0;
    const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, wid = tid >> 5;
    extern __shared__ __align__(16) double lu_smem[];
    double* Pn = lu_smem;                    // [nr][LU_NBP] own rows of the panel
    int8_t* fl = (int8_t*)(Pn + (size_t)nr * LU_NBP);
    __shared__ __align__(16) double rowb[2][CS][LU_NB];  // every CTA's best row (by step parity)
    __shared__ int rowi[2][CS];                          // its index in the matrix, INT_MAX: none left
    __shared__ __align__(8) unsigned long long mbar[2];
    __shared__ unsigned long long ck[8];
    __shared__ int cr[8];
    bool any_bad = false, late = false;
    if (tid == 0) {
        for (int q = 0; q < 2; ++q)
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(lu_smem_u32(&mbar[q])) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    for (int e = tid; e < nr * nbk; e += nt) {
        const int q = e / nbk, c = e - q * nbk;
        Pn[q * LU_NBP + c] = A[(long)(r0 + q) * lda + j0 + c];
    }
    for (int q = tid; q < nr; q += nt) fl[q] = flag[r0 + q];
    cl.sync();  // every CTA of the cluster runs and its mbarriers are set up
    const int h = tid & (tpr - 1), rows = nt / tpr, q0 = tid / tpr;
    // candidate of column 0 (later columns: found during the previous step's row update)
    unsigned long long bk = 0;
    int br = INT_MAX;
    if (h == 0)
        for (int q = q0; q < nr; q += rows)
            if (!fl[q]) lu_pick(bk, br, lu_key(Pn[q * LU_NBP]), r0 + q);
    for (int jj = 0; jj < nbk; ++jj) {
        const int par = jj & 1;
        const unsigned bar = lu_smem_u32(&mbar[par]);
        lu_warp_best(bk, br);
        if (lane == 0) {
            ck[wid] = bk;
            cr[wid] = br;
        }
        __syncthreads();  // the candidates are there, and every row update of the last step is done
        if (wid == 0) {
            unsigned long long k = lane < 8 ? ck[lane] : 0ULL;
            int r = lane < 8 ? cr[lane] : INT_MAX;
            lu_warp_best(k, r);
            const double v = (r != INT_MAX && lane < nbk) ? Pn[(r - r0) * LU_NBP + lane] : 0.0;
            if (lane == 0)
                asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar),
                             "r"(CS * (LU_NB * 8 + 4))
                             : "memory");
            const unsigned dv = lu_smem_u32(&rowb[par][rank][lane]), di = lu_smem_u32(&rowi[par][rank]);
#pragma unroll 4
            for (int d = 0; d < CS; ++d) {
                const unsigned rb = lu_mapa(bar, d);
                lu_st_async(lu_mapa(dv, d), v, rb);
                if (lane == 0) lu_st_async(lu_mapa(di, d), r, rb);
            }
        }
        if (!late && !lu_bar_wait(bar, (unsigned)(jj >> 1) & 1u)) late = true;
        // the winner over the cluster's CTAs
        int r = lane < CS ? rowi[par][lane] : INT_MAX;
        unsigned long long k = (lane < CS && r != INT_MAX) ? lu_key(rowb[par][lane < CS ? lane : 0][jj]) : 0ULL;
        const int win = lu_warp_best(k, r) & (CS - 1);
        const double* urow = rowb[par][win];
        const bool bad = late || (k == 0ULL) || (k >= 0x7ff0000000000000ULL) || r >= m || r < 0;
        const int p = (late || r >= m || r < 0) ? 0 : r;  // with a zero pivot too: perm stays a permutation
        const double pinv = bad ? 0.0 : fast_rcp(urow[jj]);
        any_bad = any_bad || bad;
        if (tid == 0) {
            if (p >= r0 && p < r1) fl[p - r0] = lu_flag(j0);
            if (rank == 0) perm[j0 + jj] = p;
        }
        // own unpivoted rows: multiplier into column jj, rank-1 step on the later panel columns, and the
        // candidate for column jj + 1
        bk = 0;
        br = INT_MAX;
        const int hj = jj & (tpr - 1), c0 = jj + 1 + ((h - (jj + 1)) & (tpr - 1));
        for (int qb = 0; qb < nr; qb += rows) {
            const int q = qb + q0;
            const bool act = q < nr && r0 + q != p && !fl[q];
            double* __restrict__ row = Pn + (act ? q : 0) * LU_NBP;
            double l = 0.0;
            if (act && h == hj) {
                l = row[jj] * pinv;
                row[jj] = l;
            }
            l = __shfl_sync(0xffffffffu, l, (lane & ~(tpr - 1)) | hj);
            if (!act) continue;
            int c = c0;
            if (c < nbk) {
                const double x = row[c] - l * urow[c];
                row[c] = x;
                if (c == jj + 1) lu_pick(bk, br, lu_key(x), r0 + q);
                c += tpr;
            }
            for (; c + 3 * tpr < nbk; c += 4 * tpr) {
                const double u0 = urow[c], u1 = urow[c + tpr], u2 = urow[c + 2 * tpr], u3 = urow[c + 3 * tpr];
                const double v0 = row[c], v1 = row[c + tpr], v2 = row[c + 2 * tpr], v3 = row[c + 3 * tpr];
                row[c] = v0 - l * u0;
                row[c + tpr] = v1 - l * u1;
                row[c + 2 * tpr] = v2 - l * u2;
                row[c + 3 * tpr] = v3 - l * u3;
            }
            for (; c < nbk; c += tpr) row[c] -= l * urow[c];
        }
        __syncwarp();
    }
    cl.sync();  // no CTA leaves while a store to another may still be in flight
    if (late && lane == 0) set_err(a.err, DEV_TIMEOUT);
    if (tid == 0 && rank == 0 && any_bad) set_err(a.err, DEV_NUMERIC);
    for (int e = tid; e < nr * nbk; e += nt) {
        const int q = e / nbk, c = e - q * nbk;
        A[(long)(r0 + q) * lda + j0 + c] = Pn[q * LU_NBP + c];
    }
    for (int q = tid; q < nr; q += nt) flag[r0 + q] = fl[q];
}

template <int CS>
__global__ void __launch_bounds__(256) lu_panel_kernel(LuArgs a, int j0, int nbk, int tpr) {
    lu_panel<CS>(a, j0, nbk, tpr);
}

// U12 = L11^{-1} A12 on the pivot rows of a panel, columns [j0 + nbk, n): eight lanes per column, lane h
// holds the entries h, h + 8, ... (the FP64 work of a column is sequential, so a column spreads over lanes
// and the columns over the whole GPU).  Grid (16-column blocks, matrix).
constexpr int LU_UC = 16;
__global__ void __launch_bounds__(8 * LU_UC) lu_u12_kernel(LuArgs a, int j0, int nbk) {
    const int mat = blockIdx.y, tid = threadIdx.x, h = tid >> 4, cl = tid & 15;
    double* A = lu_A(a, mat);
    const int* perm = a.perm0 + (long)mat * a.pstride + j0;
    const long lda = a.lda;
    const int c = j0 + nbk + blockIdx.x * LU_UC + cl, cc = min(c, a.n - 1);
    __shared__ double L11[LU_NB][LU_NBP];
    __shared__ double xs[LU_NB][LU_UC];  // finished entries
    for (int e = tid; e < LU_NB * LU_NB; e += 8 * LU_UC) {
        const int k = e / LU_NB, kp = e % LU_NB;
        L11[k][kp] = (k < nbk && kp < k) ? A[(long)perm[k] * lda + j0 + kp] : 0.0;
    }
    double v[4];
#pragma unroll
    for (int t = 0; t < 4; ++t) v[t] = (h + 8 * t < nbk) ? A[(long)perm[h + 8 * t] * lda + cc] : 0.0;
    __syncthreads();
#pragma unroll
    for (int kp = 0; kp < LU_NB; ++kp) {
        if (kp < nbk) {
            if (h == (kp & 7)) xs[kp][cl] = v[kp >> 3];
            __syncthreads();
            const double x = xs[kp][cl];
#pragma unroll
            for (int t = 0; t < 4; ++t)
                if (8 * t + 7 > kp) v[t] -= L11[h + 8 * t][kp] * x;  // zero at and before kp
        }
    }
    if (c < a.n)
#pragma unroll
        for (int t = 0; t < 4; ++t)
            if (h + 8 * t < nbk && h + 8 * t > 0) A[(long)perm[h + 8 * t] * lda + c] = v[t];
}

// A[r][c] -= sum_k A[r][j0 + k] U12[k][c] for the rows r that were unpivoted after the panel at j0 and c in
// [ca, cb), with U12[k] the pivot row perm[j0 + k]: tile (bx, by) of BM of these rows x BN columns, BM / 16 x
// BN / 16 outputs per thread.  A block finds its rows by counting the flags, so no multiply-add goes to a
// pivoted row (they are the bound: 2 a clock and SM).
template <int BM, int BN>
__device__ __forceinline__ void lu_update(const LuArgs& a, int j0, int nbk, int ca, int cb, int bx, int by, int mat) {
    constexpr int TM = BM / 16, TN = BN / 16;
    double* A = lu_A(a, mat);
    const int* perm = a.perm0 + (long)mat * a.pstride;
    const int8_t* flag = a.flag0 + (long)mat * a.pstride;
    const long lda = a.lda;
    const int m = a.m, n = cb, closed = (uint8_t)lu_flag(j0);
    const int f0 = bx * BM, c0 = ca + by * BN;
    __shared__ double Ls[BM][LU_NBP];
    __shared__ double Us[LU_NB][BN + 1];
    __shared__ int rid[BM];
    __shared__ int wsum[8];
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    for (int q = tid; q < BM; q += 256) rid[q] = -1;
    for (int base = 0, seen = 0; base < m && seen < f0 + BM; base += 256) {
        const int r = base + tid;
        const int f = r < m ? (int)(uint8_t)flag[r] : closed;
        const bool open = f == 0 || f > closed;
        const unsigned ball = __ballot_sync(0xffffffffu, open);
        if (lane == 0) wsum[wid] = __popc(ball);
        __syncthreads();
        int before = seen, all = 0;
        for (int w = 0; w < 8; ++w) {
            if (w < wid) before += wsum[w];
            all += wsum[w];
        }
        const int pos = before + __popc(ball & ((1u << lane) - 1u)) - f0;
        if (open && pos >= 0 && pos < BM) rid[pos] = r;
        seen += all;
        __syncthreads();
    }
    for (int e = tid; e < BM * LU_NB; e += 256) {
        const int q = e / LU_NB, k = e - q * LU_NB;
        Ls[q][k] = (k < nbk && rid[q] >= 0) ? A[(long)rid[q] * lda + j0 + k] : 0.0;
    }
    for (int e = tid; e < LU_NB * BN; e += 256) {
        const int k = e / BN, c = e % BN;
        Us[k][c] = (k < nbk && c0 + c < n) ? A[(long)perm[j0 + k] * lda + c0 + c] : 0.0;
    }
    __syncthreads();
    const int tx = tid & 15, ty = tid >> 4;
    double acc[TM][TN];
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TN; ++j) acc[i][j] = 0.0;
    for (int k = 0; k < nbk; ++k) {
        double lv[TM], uv[TN];
#pragma unroll
        for (int i = 0; i < TM; ++i) lv[i] = Ls[ty + 16 * i][k];
#pragma unroll
        for (int j = 0; j < TN; ++j) uv[j] = Us[k][tx + 16 * j];
#pragma unroll
        for (int i = 0; i < TM; ++i)
#pragma unroll
            for (int j = 0; j < TN; ++j) acc[i][j] += lv[i] * uv[j];
    }
#pragma unroll
    for (int i = 0; i < TM; ++i) {
        const int r = rid[ty + 16 * i];
        if (r < 0) continue;
#pragma unroll
        for (int j = 0; j < TN; ++j) {
            const int c = c0 + tx + 16 * j;
            if (c < n) A[(long)r * lda + c] -= acc[i][j];
        }
    }
}

// Grid (tiles of the unpivoted rows, column tiles, matrix).
template <int BM, int BN>
__global__ void __launch_bounds__(256) lu_update_kernel(LuArgs a, int j0, int nbk, int ca, int cb) {
    lu_update<BM, BN>(a, j0, nbk, ca, cb, blockIdx.x, blockIdx.y, blockIdx.z);
}

// The panel at j0 on the first CS nmat blocks and, on the others, the trailing update of the panel before it
// on the columns right of this one (their tiles: nx x ny per matrix).  The two touch different columns, and
// no block waits for one outside its cluster.  Against the update in a launch of its own: the 24 x 24 spin-coupled
// pass 52.1 -> 50.0 ms, 40 x 40 62.8 -> 61.7 ms, eight 20 x 20 pairing walkers 204.9 -> 202.6 ms.
template <int CS, int BM, int BN>
__global__ void __launch_bounds__(256) lu_step_kernel(LuArgs a, int j0, int nbk, int tpr, int nx, int ny) {
    const int b = (int)blockIdx.x - CS * a.nmat;
    if (b < 0) {
        lu_panel<CS>(a, j0, nbk, tpr);
    } else if (b < nx * ny * a.nmat) {
        const int t = b % (nx * ny);
        lu_update<BM, BN>(a, j0 - LU_NB, LU_NB, j0 + nbk, a.n, t % nx, t / nx, b / (nx * ny));
    }
}

template <int BM, int BN>
static cudaError_t launch_update(cudaStream_t st, const LuArgs& a, int j0, int nbk, int mr, int ca, int cb) {
    count_launch();
    lu_update_kernel<BM, BN><<<dim3((mr + BM - 1) / BM, (cb - ca + BN - 1) / BN, a.nmat), 256, 0, st>>>(a, j0, nbk, ca,
                                                                                                      cb);
    return cudaGetLastError();
}

// Pivot rows of the factored tall matrix become unit rows: A[perm[j]][c] = (c == j) for c >= j,
// so A = P L (unit lower trapezoidal, rows in the original order) spans the same columns.
__global__ void lu_unit_rows_kernel(LuArgs a) {
    const int mat = blockIdx.y;
    double* A = lu_A(a, mat);
    const int* perm = a.perm0 + (long)mat * a.pstride;
    const int n = a.n;
    for (long e = (long)blockIdx.x * blockDim.x + threadIdx.x; e < (long)n * n; e += (long)gridDim.x * blockDim.x) {
        const int j = (int)(e / n), c = (int)(e % n);
        if (c >= j) A[(long)perm[j] * a.lda + c] = (c == j) ? 1.0 : 0.0;
    }
}

// sign_out[w] *= the sign of the product of the pivots of walker w's ng matrices (times each permutation's
// parity when `parity`): the sign of det(A) for square A.  One block per walker.  The parity of a permutation
// of m rows is that of m minus its number of cycles; the smallest row of every cycle comes from pointer
// jumping (log2 m rounds in shared memory), and the rows that are their own smallest are counted.  Bound by
// the latency of the scattered pivots and of the rounds.  One thread that followed the cycles through global
// memory took 445 us for two 700 x 700 matrices; with the block the constrained-path pass (16 x 16, 32 walkers,
// five steps) went from 27.5 to 26.4 ms.
constexpr int LS_THREADS = 256;
__global__ void __launch_bounds__(LS_THREADS) lu_sign_kernel(LuArgs a, int parity, double* sign_out) {
    extern __shared__ int ls_smem[];
    const int wk = blockIdx.x, tid = threadIdx.x, m = a.m;
    int *lab = ls_smem, *nxt = lab + m, *lab2 = nxt + m, *nxt2 = lab2 + m;  // smallest row seen, row reached
    int odd = 0;
    for (int q = 0; q < a.ng; ++q) {
        const int mat = wk * a.ng + q;
        const double* A = lu_A(a, mat);
        const int* perm = a.perm0 + (long)mat * a.pstride;
        for (int j = tid; j < a.n; j += LS_THREADS) odd ^= A[(long)perm[j] * a.lda + j] < 0.0 ? 1 : 0;
        if (!parity) continue;
        if (tid == 0) odd ^= m & 1;
        for (int r = tid; r < m; r += LS_THREADS) {
            lab[r] = r;
            nxt[r] = perm[r];
        }
        __syncthreads();
        for (int span = 1; span < m; span *= 2) {
            for (int r = tid; r < m; r += LS_THREADS) {
                const int t = nxt[r];
                lab2[r] = min(lab[r], lab[t]);
                nxt2[r] = nxt[t];
            }
            __syncthreads();
            int* t0 = lab; lab = lab2; lab2 = t0;
            t0 = nxt; nxt = nxt2; nxt2 = t0;
        }
        for (int r = tid; r < m; r += LS_THREADS) odd ^= lab[r] == r ? 1 : 0;
        __syncthreads();
    }
    if ((__syncthreads_count(odd) & 1) && tid == 0) sign_out[wk] = -sign_out[wk];
}

// Dynamic shared memory of a panel's CTA, the most of it, and the most beside the trailing update's static tiles.
static size_t lu_panel_smem(int m, int cs) {
    const size_t rpc = (m + cs - 1) / cs;
    return rpc * LU_NBP * sizeof(double) + rpc + 16;
}
constexpr size_t LU_PANEL_SMEM = 227 * 1024 - 16 * 1024, LU_STEP_SMEM = 144 * 1024;

// mr > 0: with the update of the mr rows unpivoted after the panel before, on the columns right of this one.
template <int CS>
static cudaError_t launch_panel(cudaStream_t st, const LuArgs& a, int j0, int nbk, int mr) {
    const int rpc = (a.m + CS - 1) / CS;
    const size_t shm = lu_panel_smem(a.m, CS);
    {
        cudaError_t e = ensure_smem_attr((const void*)lu_panel_kernel<CS>, LU_PANEL_SMEM);
        if (e != cudaSuccess) return e;
        if (CS > 8) {
            e = ensure_func_attr((const void*)lu_panel_kernel<CS>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
            if (e != cudaSuccess) return e;
        }
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(CS * a.nmat);
    cfg.blockDim = dim3(256);
    cfg.dynamicSmemBytes = shm;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = CS;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    int tpr = 8;  // threads per row: all 256 threads busy
    while (tpr > 1 && rpc * tpr > 256) tpr /= 2;
    count_launch();
    if (mr == 0) return cudaLaunchKernelEx(&cfg, lu_panel_kernel<CS>, a, j0, nbk, tpr);
    // with the previous panel's update: the tile whose busiest SM issues the fewest multiply-adds
    const int nc = a.n - j0 - nbk;
    auto tiles = [&](int b) { return (long)((mr + b - 1) / b) * ((nc + b - 1) / b) * a.nmat; };
    const bool big = (tiles(64) + 151) / 152 * (64 * 64 + 128) <= (tiles(32) + 151) / 152 * (32 * 32 + 128);
    const int b = big ? 64 : 32, nx = (mr + b - 1) / b, ny = (nc + b - 1) / b;
    auto kern = big ? lu_step_kernel<CS, 64, 64> : lu_step_kernel<CS, 32, 32>;
    cudaError_t e = ensure_smem_attr((const void*)kern, LU_STEP_SMEM);
    if (e == cudaSuccess && CS > 8) e = ensure_func_attr((const void*)kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
    cfg.gridDim = dim3((unsigned)(CS * a.nmat + (tiles(b) + CS - 1) / CS * CS));
    return cudaLaunchKernelEx(&cfg, kern, a, j0, nbk, tpr, nx, ny);
}

// Resident 16-CTA clusters of a kernel with shm bytes of dynamic shared memory, -1 if that cannot be told.
static int lu_resident16(const void* fn, size_t attr_bytes, size_t shm) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(32);
    cfg.blockDim = dim3(256);
    cfg.dynamicSmemBytes = shm;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = 16;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    int ncl = 0;
    if (ensure_func_attr(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess &&
        ensure_smem_attr(fn, attr_bytes) == cudaSuccess &&
        cudaOccupancyMaxActiveClusters(&ncl, fn, &cfg) == cudaSuccess)
        return ncl;
    cudaGetLastError();
    return -1;
}

// Cluster size: enough CTAs per matrix that a panel step's FP64 work per SM stays small, few
// enough that all nmat clusters of a batch are resident together (about two CTAs per SM).
// Rows per CTA stay at or below 512 (shared memory); 16-CTA clusters are used only if two of
// them fit on the device at once (else 8), of the panel kernel and of the step kernel with its update tiles.
static int lu_cluster_size(const LuArgs& a) {
    static BigClusterCache big;
    int nsm = 152, dev = 0;
    if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    int cs = 1;
    while (cs < 16 && (a.m + cs - 1) / cs > 64 && cs * a.nmat <= nsm) cs *= 2;  // spread rows
    while (cs < 16 && (a.m + cs - 1) / cs > 512) cs *= 2;                              // shared memory
    if (cs == 16) {
        const size_t shm = lu_panel_smem(a.m, 16);
        const bool fits = big.fits(dev, shm, [&] {
            const int panel = lu_resident16((const void*)lu_panel_kernel<16>, LU_PANEL_SMEM, shm);
            if (shm > LU_STEP_SMEM) return panel;  // no look-ahead
            return std::min(panel, lu_resident16((const void*)lu_step_kernel<16, 64, 64>, LU_STEP_SMEM, shm));
        });
        if (!fits) cs = 8;
    }
    return cs;
}

cudaError_t launch_lu(cudaStream_t st, const LuArgs& a) {
    if (a.m < a.n || a.n < 1 || a.nmat < 1 || a.pstride < a.m) return cudaErrorInvalidValue;
    const int cs = lu_cluster_size(a);
    if ((a.m + cs - 1) / cs * (LU_NBP * sizeof(double) + 1) > 200 * 1024) return cudaErrorInvalidValue;
    cudaError_t e;
    if ((e = cudaMemsetAsync(a.flag0, 0, (size_t)(a.nmat - 1) * a.pstride + a.m, st)) != cudaSuccess) return e;
    // Look-ahead: a panel's update goes to the next panel's columns first (a launch of its own), the rest of it
    // beside the next panel, whose chain leaves most of the FP64 units idle; only where that rest is more than
    // two 32 x 32 tiles an SM (below, the extra launch costs what it hides: four 441 x 138 factors 32.3 ms a
    // pass without, 32.4 with it).
    const bool ahead = a.n <= LU_PANELS_MAX * LU_NB && lu_panel_smem(a.m, cs) <= LU_STEP_SMEM;
    int mr_open = 0;  // rows of the update that goes with the next panel, 0: none
    for (int j0 = 0; j0 < a.n; j0 += LU_NB) {
        const int nbk = (a.n - j0 < LU_NB) ? a.n - j0 : LU_NB;
        switch (cs) {
            case 1: e = launch_panel<1>(st, a, j0, nbk, mr_open); break;
            case 2: e = launch_panel<2>(st, a, j0, nbk, mr_open); break;
            case 4: e = launch_panel<4>(st, a, j0, nbk, mr_open); break;
            case 8: e = launch_panel<8>(st, a, j0, nbk, mr_open); break;
            default: e = launch_panel<16>(st, a, j0, nbk, mr_open); break;
        }
        if (e != cudaSuccess) return e;
        const int ca = j0 + nbk, nc = a.n - ca, mr = a.m - ca;
        if (nc <= 0) break;
        count_launch();
        lu_u12_kernel<<<dim3((nc + LU_UC - 1) / LU_UC, a.nmat), 8 * LU_UC, 0, st>>>(a, j0, nbk);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        mr_open = 0;
        if (mr <= 0) continue;
        if (ahead && (long)((mr + 31) / 32) * ((nc - 1) / 32) * a.nmat > 304) {
            if ((e = launch_update<32, 16>(st, a, j0, nbk, mr, ca, ca + LU_NB)) != cudaSuccess) return e;
            mr_open = mr;
            continue;
        }
        // the tile whose busiest SM issues the fewest multiply-adds (plus a fixed cost per tile)
        auto cost = [&](int bm, int bn) {
            const long t = (long)((mr + bm - 1) / bm) * ((nc + bn - 1) / bn) * a.nmat;
            return (t + 151) / 152 * (bm * bn + 128);
        };
        const long c64 = cost(64, 64), c33 = cost(32, 32);
        if (c64 <= c33) e = launch_update<64, 64>(st, a, j0, nbk, mr, ca, a.n);
        else e = launch_update<32, 32>(st, a, j0, nbk, mr, ca, a.n);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

cudaError_t launch_lu_unit_rows(cudaStream_t st, const LuArgs& a) {
    count_launch();
    lu_unit_rows_kernel<<<dim3(256, a.nmat), 256, 0, st>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_lu_sign(cudaStream_t st, const LuArgs& a, int parity, double* sign_out) {
    if (!sign_out) return cudaSuccess;
    const size_t shm = parity ? 4 * (size_t)a.m * sizeof(int) : 0;
    cudaError_t e = ensure_smem_attr((const void*)lu_sign_kernel, shm);
    if (e != cudaSuccess) return e;
    count_launch();
    lu_sign_kernel<<<a.nmat / a.ng, LS_THREADS, shm, st>>>(a, parity, sign_out);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Z = O^{-1} B for a factored square O (ns x ns, no-swap form: row perm[j] holds L[j][0..j)
// and U[j][j..ns)) and B (ns x N), both matrices of the batch:
//   forward  y_j = B[perm[j]] - sum_{k<j} L[j][k] y_k,
//   backward z_j = (y_j - sum_{k>j} U[j][k] z_k) / U[j][j],   Z[j] = z_j.
// The right-hand sides are independent: one warp per column.  The column lives in shared memory; a block of
// 32 rows is one row per lane: the products with the finished rows (coefficients staged for the whole CTA in
// 32 x SV_KB tiles, the next one copied asynchronously under the current one), then the 32 x 32 diagonal block
// by shuffles.  Bound by the FP64 multiply-adds (2 a clock and SM), so what counts is that every partition of
// the SM has the same work: with the pivot-ordered identity column c costs its forward substitution from row
// c on, and a CTA takes as many columns from the front as from the back.  (With ten contiguous columns per CTA,
// ten columns of one row block dealt over eight warps, the inverse of two 700 x 700 matrices took 2.43 ms.)
// Grid (column blocks, matrix).
// ---------------------------------------------------------------------------
constexpr int SV_KB = 64, SV_LP = SV_KB + 1;

__device__ __forceinline__ void sv_cp_async(double* dst, const double* src, bool in) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    const int sz = in ? 8 : 0;
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(d), "l"(src), "r"(sz) : "memory");
}

__global__ void __launch_bounds__(320) lu_solve_kernel(SolveArgs a) {
    const int mat = blockIdx.y;
    const double* LU = a.LU0 + (long)mat * a.ostride;
    const int* perm = a.perm0 + (long)mat * a.pstride;
    const double* B = a.B0 + (long)(mat / a.ng) * a.wstride + (long)(mat % a.ng) * a.sstride;
    double* Z = a.Z0 + (long)mat * a.zstride;
    const int ns = a.ns, N = a.N;
    const long ldl = a.ldl, ldb = a.ldb ? a.ldb : N;
    const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, w = tid >> 5, nc = nt >> 5;
    const bool eye = a.eye != 0;
    // this warp's column: contiguous, or (identity) half from the front and half from the back
    const int half = nc / 2;
    int c = blockIdx.x * nc + w;
    bool own = c < N;
    if (eye) {
        const int f = blockIdx.x * half + (w < half ? w : w - half);
        c = w < half ? f : N - 1 - f;
        own = w < half ? f < (N + 1) / 2 : f < N / 2;
    }
    extern __shared__ __align__(16) double sv_smem[];
    double* Lt = sv_smem;                       // [2][32][SV_LP] coefficient tiles
    double* rinv = Lt + 2 * 32 * SV_LP;         // [ns]
    double* y = rinv + ns + (size_t)w * ns;     // [ns] the column
    int* sp = (int*)(rinv + ns + (size_t)nc * ns);  // [ns]
    for (int j = tid; j < ns; j += nt) sp[j] = perm[j];
    __syncthreads();
    for (int j = tid; j < ns; j += nt) rinv[j] = 1.0 / LU[(long)sp[j] * ldl + j];
    if (eye) {
        for (int j = lane; j < ns; j += 32) y[j] = j == c ? 1.0 : 0.0;
    } else {  // rows by warps, the CTA's columns by lanes
        double* y0 = rinv + ns;
        const int cb = blockIdx.x * nc;
        for (int j = w; j < ns; j += nc)
            if (lane < nc) y0[(size_t)lane * ns + j] = cb + lane < N ? B[(long)sp[j] * ldb + cb + lane] : 0.0;
    }
    const int nb = (ns + 31) / 32;
    const int first = eye ? (blockIdx.x * half) / 32 : 0;         // first block any column of the CTA needs
    const int mine = !own ? nb : (eye ? c / 32 : 0);              // first block this column needs
    // tile (rows J0.., columns k0 ..): coefficient rows are the pivot rows
    auto fetch = [&](int buf, int J0, int k0) {
        for (int r = w; r < 32; r += nc)
            for (int k = lane; k < SV_KB; k += 32) {
                const bool in = J0 + r < ns && k0 + k < ns;
                sv_cp_async(Lt + (buf * 32 + r) * SV_LP + k, in ? LU + (long)sp[J0 + r] * ldl + k0 + k : LU, in);
            }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    auto arrived = [&] {
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncthreads();
    };
    __syncthreads();
    int buf = 0;
    // forward substitution (unit lower L), then backward (U): block rows jb, coefficient tiles of the finished
    // columns, then the diagonal block
    for (int dir = 0; dir < 2; ++dir) {
        const int b0 = dir ? nb - 1 : first, b1 = dir ? -1 : nb, step = dir ? -1 : 1;
        for (int jb = b0; jb != b1; jb += step) {
            const int J0 = jb * 32, row = J0 + lane;
            // finished columns: [first block, J0) forward, [J0 + 32, ns) backward, in SV_KB steps
            const int ks = dir ? J0 + 32 : first * 32, ke = dir ? ns : J0;
            const bool work = own && (dir || jb >= mine);
            double v = (work && row < ns) ? y[row] : 0.0;
            fetch(buf, J0, ks < ke ? ks : J0);
            for (int k0 = ks; k0 < ke; k0 += SV_KB) {
                arrived();
                const double* Lc = Lt + (buf * 32 + lane) * SV_LP;
                buf ^= 1;
                fetch(buf, J0, k0 + SV_KB < ke ? k0 + SV_KB : J0);  // the next tile, at last the diagonal block
                const int kb = min(SV_KB, ke - k0);
                if (work && (dir || k0 + kb > mine * 32)) {
                    double a0 = 0.0, a1 = 0.0, a2 = 0.0, a3 = 0.0;  // independent chains (FP64 latency)
                    int k = 0;
                    for (; k + 3 < kb; k += 4) {
                        a0 += Lc[k] * y[k0 + k];
                        a1 += Lc[k + 1] * y[k0 + k + 1];
                        a2 += Lc[k + 2] * y[k0 + k + 2];
                        a3 += Lc[k + 3] * y[k0 + k + 3];
                    }
                    for (; k < kb; ++k) a0 += Lc[k] * y[k0 + k];
                    v -= (a0 + a1) + (a2 + a3);
                }
            }
            arrived();
            const double* Ld = Lt + (buf * 32 + lane) * SV_LP;  // row `lane` of the diagonal block
            const int jn = min(32, ns - J0);
            if (work) {
                if (dir == 0) {
                    for (int k = 0; k + 1 < jn; ++k) {
                        const double x = __shfl_sync(0xffffffffu, v, k);
                        if (lane > k && lane < jn) v -= Ld[k] * x;
                    }
                } else {
                    const double ri = lane < jn ? rinv[row] : 0.0;
                    for (int k = jn - 1; k >= 0; --k) {
                        if (lane == k) v *= ri;
                        const double x = __shfl_sync(0xffffffffu, v, k);
                        if (lane < k) v -= Ld[k] * x;
                    }
                }
                if (lane < jn) y[row] = v;
            }
            buf ^= 1;
        }
        __syncwarp();
    }
    __syncthreads();
    if (eye) {
        if (own)
            for (int j = lane; j < ns; j += 32) Z[(long)j * N + sp[c]] = y[j];
    } else {
        const double* y0 = rinv + ns;
        const int cb = blockIdx.x * nc;
        for (int j = w; j < ns; j += nc)
            if (lane < nc && cb + lane < N) Z[(long)j * N + cb + lane] = y0[(size_t)lane * ns + j];
    }
}

cudaError_t launch_lu_solve(cudaStream_t st, const SolveArgs& a) {
    auto smem = [&](int nc) {
        return ((size_t)2 * 32 * SV_LP + (size_t)a.ns * (nc + 1)) * sizeof(double) + (size_t)a.ns * sizeof(int);
    };
    // columns (warps) per CTA, an even number (the identity's columns come from both ends): the one whose
    // busiest SM partition has the fewest columns, the larger on a tie (tiles shared by more columns)
    int nc = 2;
    long best = 0;
    for (int k = 10; k >= 2; k -= 2) {
        if (smem(k) > 220 * 1024) continue;
        const long t = (((long)((a.N + k - 1) / k) * a.nmat + 151) / 152) * ((k + 3) / 4);
        if (best == 0 || t < best) {
            best = t;
            nc = k;
        }
    }
    if (smem(nc) > 220 * 1024) return cudaErrorInvalidValue;
    {
        cudaError_t e = ensure_smem_attr((const void*)lu_solve_kernel, 220 * 1024);
        if (e != cudaSuccess) return e;
    }
    count_launch();
    lu_solve_kernel<<<dim3((a.N + nc - 1) / nc, a.nmat), 32 * nc, smem(nc), st>>>(a);
    return cudaGetLastError();
}

}  // namespace afq
