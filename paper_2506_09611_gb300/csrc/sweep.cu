// sweep.cu -- the per-slice site loop of the PQMC update sweep in G form.
//
//   local   : persistent cooperative kernel, one grid barrier per site, the
//             rank-1 update G <- G - (d/r) G_{:,i} (e_i^T - G_{i,:}) applied to
//             the whole of G on every accepted flip (Eqs. DetRatiolocal,
//             UpdateLTRlocal restated for G).
//   delayed : a window of n consecutive sites is decided by ONE CTA on the
//   blockfb   n x n diagonal block of G held in shared memory; the accepted
//             flips I are then applied to the full G as one rank-|I| product
//                 G <- G - G[:, I] W (E_I^T - G[I, :]),  W = D_I (1 + A0_II D_I)^{-1}
//             which equals the buffered sum of the paper's delayed vectors
//             (Eqs. DelayTMat00, DelayRgenk, FinalDelay) and the block
//             force-bias upgrade (Eq. BlkFrcBsTnew2).
#include <math.h>

#include "internal.h"

namespace afq {

// ---------------------------------------------------------------------------
// uniforms of one slice visit
// ---------------------------------------------------------------------------
// The visit counter lives on the device so that a captured slice replays with fresh uniforms.
__global__ void uniforms_kernel(uint64_t seed, const int* gid, const unsigned long long* visit, int count, double* u) {
    int j = blockIdx.x * blockDim.x + threadIdx.x;
    const int w = blockIdx.y;
    if (j < count) u[(size_t)w * count + j] = philox_uniform(seed, (uint64_t)gid[w], (uint64_t)*visit, (uint64_t)j);
}

__global__ void bump_kernel(unsigned long long* visit) { *visit += 1ULL; }

cudaError_t launch_uniforms(cudaStream_t st, uint64_t seed, const int* gid, const unsigned long long* visit, int count,
                            double* u, int nwk) {
    count_launch();
    uniforms_kernel<<<dim3((count + 255) / 256, nwk), 256, 0, st>>>(seed, gid, visit, count, u);
    return cudaGetLastError();
}

cudaError_t launch_bump(cudaStream_t st, unsigned long long* visit) {
    count_launch();
    bump_kernel<<<1, 1, 0, st>>>(visit);
    return cudaGetLastError();
}

// Buffers of walker j of a group (see Batch).
template <typename T>
__device__ __forceinline__ WindowBufs wb_walker(WindowBufs wb, int j, int N);
__device__ __forceinline__ SliceOut so_walker(SliceOut so, int j, int N) {
    so.dec += (size_t)j * 2 * N;
    so.ratio += (size_t)j * 2 * N;
    so.stats += (size_t)j * 8;
    so.maxr += j;
    if (so.sign) so.sign += j;
    if (so.cp) so.cp += (size_t)j * 4;
    return so;
}

__device__ __forceinline__ double hs_log_scalar(const SiteParams& sp, int x) {
    return sp.hs == AFQMC_HS_CHARGE_REAL ? -sp.lam * (double)x : 0.0;
}

// ---------------------------------------------------------------------------
// local update: persistent cooperative kernel, one grid barrier per ACCEPT
// ---------------------------------------------------------------------------
// CTA b owns the rows [r0, r1) of both spins.  A phase handles one accepted site:
//   1. thread 0 of every CTA passes the grid barrier (one release reduction on an arrival counter,
//      then polling), and warp 0 at once scans the sites after the last accept (32 sites per round;
//      a ballot finds the first acceptance) from a copy of the two diagonals in global memory.
//      Every CTA reads the same values and runs the same arithmetic, so all reach the same site b;
//   2. every CTA reads row b of both spins (e_b^T - G[b, :]) and column b of its own rows;
//   3. every CTA applies G_s[r, c] -= f_s G_s[r, b] (delta_bc - G_s[b, c]) to its own rows with
//      16-byte accesses and several loads in flight per thread, and writes the new diagonal of its
//      rows to the other diagonal buffer.
// A rejected site leaves G unchanged, so it costs a diagonal read and no barrier.  Two cross-CTA
// hazards inside a phase are avoided without a second grid barrier:
//   * the diagonals are double-buffered by phase parity: the scan reads the buffer the previous
//     phase wrote, and the update writes the other one;
//   * every CTA reads row b while its owner updates its rows, so the owner keeps its new row b in
//     shared memory and stores it to G in the next phase, after the barrier (no CTA reads row b
//     again in this slice).
// The diagonal copy is computed with the same fused multiply-add as the element of G, so the two
// stay bit-identical.  diag: [2 buffers][2 spins][N].
template <typename T> struct Vec16;
template <> struct Vec16<float> { using V = float4; static constexpr int W = 4; };
template <> struct Vec16<double> { using V = double2; static constexpr int W = 2; };

template <typename T>
__device__ __forceinline__ void vfma_rank1(typename Vec16<T>::V& g, T a, const typename Vec16<T>::V& r);
template <>
__device__ __forceinline__ void vfma_rank1<float>(float4& g, float a, const float4& r) {
    g.x = fmaf(a, r.x, g.x); g.y = fmaf(a, r.y, g.y); g.z = fmaf(a, r.z, g.z); g.w = fmaf(a, r.w, g.w);
}
template <>
__device__ __forceinline__ void vfma_rank1<double>(double2& g, double a, const double2& r) {
    g.x = fma(a, r.x, g.x); g.y = fma(a, r.y, g.y);
}

constexpr int LOCAL_THREADS = 1024;
// Loads in flight per thread in the row update (the largest count that fits 64 registers)
template <typename T> struct LocalUnroll { static constexpr int U = sizeof(T) == 4 ? 6 : 4; };

// Shared-memory layout of local_kernel (byte offsets, 16-byte aligned where vectors are read).
struct LocalSmem {
    size_t us, rowb, patch, colb, xs, rp, total;
};
template <typename T>
__host__ __device__ inline LocalSmem local_smem(int N, long ld, int nrmax) {
    auto al = [](size_t b) { return (b + 15) & ~(size_t)15; };
    LocalSmem s;
    s.us = 0;                                              // double us[N]: the site uniforms
    s.rowb = al(s.us + (size_t)N * sizeof(double));        // T rowb[2][ld]: e_b^T - G_s[b, :], 0 beyond N
    s.patch = al(s.rowb + 2 * (size_t)ld * sizeof(T));     // T patch[2][ld]: the owner's new row b
    s.colb = al(s.patch + 2 * (size_t)ld * sizeof(T));     // T colb[2][nrmax]: G_s[r, b] of the own rows
    s.xs = al(s.colb + 2 * (size_t)nrmax * sizeof(T));     // int8 xs[N]: fields of the slice
    s.rp = s.xs + (size_t)N;                               // uint8 rp[N]: forced decisions
    s.total = al(s.rp + (size_t)N);
    return s;
}

template <typename T>
__global__ void __launch_bounds__(LOCAL_THREADS, 1) local_kernel(T* Gu, T* Gd, int8_t* xl_g, const double* u,
                                                                 const uint8_t* replay, SiteParams sp, SliceOut so,
                                                                 T* diag, GridBar* bar, int* err, int nrmax) {
    using V = typename Vec16<T>::V;
    constexpr int VW = Vec16<T>::W;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int N = sp.N;
    const long ld = sp.ld;
    const int nblk = gridDim.x, b = blockIdx.x, tid = threadIdx.x, nt = blockDim.x;
    const int r0 = (int)((long)N * b / nblk), r1 = (int)((long)N * (b + 1) / nblk);
    const int nr = r1 - r0;
    const int nv = (N + VW - 1) / VW;  // 16-byte vectors per row; VW nv <= ld (ld is padded to 32)
    const LocalSmem L = local_smem<T>(N, ld, nrmax);
    double* us = (double*)(smem_raw + L.us);
    T* rowb = (T*)(smem_raw + L.rowb);
    T* patch = (T*)(smem_raw + L.patch);
    T* colb = (T*)(smem_raw + L.colb);
    int8_t* xs = (int8_t*)(smem_raw + L.xs);
    uint8_t* rp = (uint8_t*)(smem_raw + L.rp);
    __shared__ int s_b, s_nneg;
    __shared__ T s_f[2];
    __shared__ double s_maxr;
    for (int i = tid; i < N; i += nt) {
        us[i] = u[i];
        xs[i] = xl_g[i];
        rp[i] = replay ? replay[i] : 0;
    }
    if (tid == 0) {
        s_nneg = 0;
        s_maxr = 0.0;
    }
    for (int e = tid; e < 2 * nr; e += nt) {  // diagonals of the own rows into buffer 0
        const int s = e >= nr ? 1 : 0, r = r0 + e - s * nr;
        diag[(0 * 2 + s) * N + r] = (s ? Gd : Gu)[(long)r * ld + r];
    }
    // This thread's part of the own rows: the 16-byte column vectors v = vt, vt + vstep, ... of the
    // rows r = g, g + ng, ... of each spin.  With fewer vectors per row than threads the block splits
    // into ng = nt / nv row groups (one vector per thread, threads beyond ng nv idle); otherwise a
    // single group whose threads stride over the vectors.
    const int ng = nv >= nt ? 1 : nt / nv;
    const int g = nv >= nt ? 0 : tid / nv;
    const int vt = nv >= nt ? tid : tid - g * nv;
    const int vstep = nv >= nt ? nt : nv;
    unsigned int* ctr = &bar->count;
    unsigned int nbar = 0;  // grid barriers passed (thread 0)

    // flip constants in T (x = +1: index 0, x = -1: index 1), selected without local-memory indexing
    const T df00 = (T)sp.dflip[0][0], df01 = (T)sp.dflip[0][1], df10 = (T)sp.dflip[1][0],
            df11 = (T)sp.dflip[1][1], sf0 = (T)sp.sflip[0], sf1 = (T)sp.sflip[1];
    int n_acc = 0;
    int p = 0;      // next site to test (warp 0)
    int cur = 0;    // diagonal buffer the scan reads
    int pend = -1;  // own row whose new values wait in `patch`
    __syncthreads();
    for (;;) {
        // grid barrier (thread 0), then the scan for the next accept (warp 0); the other warps wait
        // at the block barrier below
        if (tid < 32) {
            int ok = 1;
            if (tid == 0) ok = grid_arrive_wait(ctr, (++nbar) * (unsigned int)nblk, err) ? 1 : 0;
            __syncwarp();
            ok = __shfl_sync(0xffffffffu, ok, 0);
            int bsel = ok ? N : -1;
            const T* d0 = diag + (cur * 2 + 0) * N;
            const T* d1 = diag + (cur * 2 + 1) * N;
            while (ok && p < N) {
                const int q = p + tid;
                bool acc = false;
                T R = T(0), rr0 = T(1), rr1 = T(1), del0 = df00, del1 = df10;
                if (q < N) {
                    // ratio arithmetic in the bulk precision T (no FP64 division on the FP32 path);
                    // the diagonals were written by other CTAs: read past L1
                    const int xi = xs[q] > 0 ? 0 : 1;
                    del0 = xi ? df01 : df00;
                    del1 = xi ? df11 : df10;
                    rr0 = T(1) + del0 * (T(1) - __ldcg(d0 + q));
                    rr1 = T(1) + del1 * (T(1) - __ldcg(d1 + q));
                    R = (xi ? sf1 : sf0) * rr0 * rr1;
                    acc = replay ? (rp[q] != 0) : (us[q] < (double)fabs(R));
                    if (!isfinite(R)) {
                        if (b == 0) set_err(err, DEV_NUMERIC);
                        acc = false;
                    }
                }
                const unsigned ball = __ballot_sync(0xffffffffu, acc);
                const int first = ball ? __ffs(ball) - 1 : 32;
                if (b == 0 && q < N && tid <= first) {
                    so.dec[q] = (tid == first) ? 1 : 0;
                    so.ratio[q] = (double)R;
                }
                if (tid == first) {
                    s_f[0] = del0 / rr0;
                    s_f[1] = del1 / rr1;
                    if (b == 0) {
                        xl_g[q] = (int8_t)(-xs[q]);
                        if (R < T(0)) s_nneg += 1;
                        s_maxr = fmax(s_maxr, (double)fabs(R));
                    }
                }
                __syncwarp();
                if (first < 32) {
                    bsel = p + first;
                    p = bsel + 1;
                    break;
                }
                p += 32;
            }
            if (tid == 0) s_b = bsel;
        }
        __syncthreads();
        const int bs = s_b;
        if (bs < 0) return;  // a bounded wait expired, or another CTA recorded an error
        if (pend >= 0) {     // every CTA has read row pend in the previous phase: store its new values
            for (int e = tid; e < 2 * nv; e += nt) {
                const int s = e >= nv ? 1 : 0, v = e - s * nv;
                *(V*)((s ? Gd : Gu) + (long)pend * ld + (long)v * VW) = *(const V*)(patch + (long)s * ld + (long)v * VW);
            }
        }
        if (bs >= N) break;
        ++n_acc;
        // row b of both spins (e_b^T - G[b, :], zero beyond N; written by another CTA: read past L1)
        // and column b of the own rows (row pend from `patch`, whose store above may be in flight)
        for (int e = tid; e < 2 * nv; e += nt) {
            const int s = e >= nv ? 1 : 0, v = e - s * nv;
            T gv[VW];
            *(V*)gv = __ldcg((const V*)((s ? Gd : Gu) + (long)bs * ld + (long)v * VW));
            T* o = rowb + (long)s * ld + (long)v * VW;
#pragma unroll
            for (int l = 0; l < VW; ++l) {
                const int c = v * VW + l;
                o[l] = c < N ? ((c == bs ? T(1) : T(0)) - gv[l]) : T(0);
            }
        }
        for (int e = tid; e < 2 * nr; e += nt) {
            const int s = e >= nr ? 1 : 0, r = e - s * nr;
            colb[s * nrmax + r] = (r0 + r == pend) ? patch[(long)s * ld + bs] : (s ? Gd : Gu)[(long)(r0 + r) * ld + bs];
        }
        pend = -1;
        __syncthreads();
        // G_s[r, :] += (-f_s G_s[r, b]) (e_b^T - G_s[b, :]) on the own rows: 16-byte accesses, all
        // LocalUnroll<T>::U loads of a thread issued before its stores.  The owner's row b goes to `patch`.
        const T nf0 = -s_f[0], nf1 = -s_f[1];
        constexpr int U = LocalUnroll<T>::U;
        for (int v = vt; g < ng && v < nv; v += vstep) {
            for (int sp_ = 0; sp_ < 2; ++sp_) {
                const V rv = *(const V*)(rowb + (long)sp_ * ld + (long)v * VW);  // e_b^T - G[b, :] here
                const T nf = sp_ ? nf1 : nf0;
                const T* cb = colb + sp_ * nrmax;
                T* base = (sp_ ? Gd : Gu) + (long)r0 * ld + (long)v * VW;
                T* pb = patch + (long)sp_ * ld + (long)v * VW;
                for (int r = g; r < nr; r += ng * U) {
                    V gv[U];
#pragma unroll
                    for (int q = 0; q < U; ++q) {
                        const int rr = r + q * ng;
                        if (rr < nr) gv[q] = *(const V*)(base + (long)rr * ld);
                    }
#pragma unroll
                    for (int q = 0; q < U; ++q) {
                        const int rr = r + q * ng;
                        if (rr < nr) {
                            vfma_rank1<T>(gv[q], nf * cb[rr], rv);
                            *(V*)((r0 + rr == bs) ? pb : base + (long)rr * ld) = gv[q];
                        }
                    }
                }
            }
        }
        // the new diagonals of the own rows (the same fused multiply-add as the element of G)
        for (int e = tid; e < 2 * nr; e += nt) {
            const int s = e >= nr ? 1 : 0, r = e - s * nr, gr = r0 + r;
            const T a = (s ? nf1 : nf0) * colb[s * nrmax + r];
            diag[((cur ^ 1) * 2 + s) * N + gr] = fma(a, rowb[(long)s * ld + gr], diag[(cur * 2 + s) * N + gr]);
        }
        if (bs >= r0 && bs < r1) pend = bs;
        cur ^= 1;
        __syncthreads();  // every write of the CTA precedes thread 0's arrival at the next barrier
    }
    if (b == 0 && tid == 0) {
        if (so.sign && (s_nneg & 1)) *so.sign = -*so.sign;
        so.stats[0] += N;
        so.stats[1] += n_acc;
        so.stats[2] += n_acc;
        *so.maxr = fmax(*so.maxr, s_maxr);
    }
}

// Grid size of the local kernel: at most max_blocks CTAs (one per SM) and at least one row each.
template <typename T>
cudaError_t launch_local(cudaStream_t st, T* Gu, T* Gd, int8_t* xl, const double* u, const uint8_t* replay,
                         const SiteParams& sp, SliceOut so, T* colbuf, T* rowbuf, GridBar* bar, int* err,
                         int max_blocks) {
    (void)rowbuf;
    const int nblk = max_blocks < sp.N ? max_blocks : sp.N;
    if (nblk < 1) return cudaErrorInvalidValue;
    const int nrmax = (sp.N + nblk - 1) / nblk;
    const size_t shm = local_smem<T>(sp.N, sp.ld, nrmax).total;
    cudaError_t e = ensure_smem_attr((const void*)local_kernel<T>, shm);
    if (e != cudaSuccess) return e;
    SiteParams spc = sp;
    int nrm = nrmax;
    void* args[] = {&Gu, &Gd, &xl, &u, &replay, &spc, &so, &colbuf, &bar, &err, &nrm};
    count_launch();
    return cudaLaunchCooperativeKernel((void*)local_kernel<T>, dim3(nblk), dim3(LOCAL_THREADS), args, shm, st);
}
// ---------------------------------------------------------------------------
// window chain: delayed (MODE 1) and block force-bias (MODE 2)
// ---------------------------------------------------------------------------
template <typename T> struct WinCap;
template <> struct WinCap<float> { static constexpr int NW = 128; };
template <> struct WinCap<double> { static constexpr int NW = 64; };
constexpr int NBMAX = 32;
constexpr int WIN_THREADS = 1024;  // 32 warps: the tail's W solve assigns 16 warps to each spin

template <typename T>
int window_max() { return WinCap<T>::NW; }
template int window_max<float>();
template int window_max<double>();

template <typename T>
__device__ __forceinline__ WindowBufs wb_walker(WindowBufs wb, int j, int N) {
    constexpr int NW = WinCap<T>::NW;
    wb.m += j;
    wb.idx += (size_t)j * NW;
    wb.Wm = (T*)wb.Wm + (size_t)j * 2 * NW * NW;
    if (wb.Wx) wb.Wx = (T*)wb.Wx + (size_t)j * 2 * NW * NW;
    wb.X = (T*)wb.X + (size_t)j * 2 * N * NW;
    wb.Y = (T*)wb.Y + (size_t)j * 2 * NW * N;  // this walker's Yraw (the products follow all walkers' Yraw)
    return wb;
}

// Sites per sub-block of the window (window_sub_sites): what one warp keeps in registers for both
// spins, 16 FP32 or 4 FP64 elements a lane.
template <typename T> struct WinSub { static constexpr int B = sizeof(T) == 4 ? 16 : 8; };

template <typename T>
static size_t window_smem(int n) {
    constexpr size_t B = WinSub<T>::B;
    size_t P = (size_t)n + 1;
    size_t g = 2 * (size_t)n * P * sizeof(T);            // Gs[2][n][n+1]
    size_t pan = 4 * B * (B + (size_t)n) * sizeof(T);    // sub-block coefficients and panels
    size_t s1 = 2 * (size_t)NBMAX * (NBMAX + 1) * sizeof(T);
    size_t vec = 4 * (size_t)n * sizeof(T) + 2 * (size_t)NBMAX * sizeof(T);  // staging vectors
    size_t misc = (size_t)n * (sizeof(int) + 1) + 8 * (size_t)NBMAX * sizeof(double) + 256;
    return g + pan + s1 + vec + misc;
}

// G_s[r][c] += f_s * G_s[r][a] * G_s[a][c] for r, c in (a, n), both spins; 32 x 32 thread tiles.
template <typename T>
__device__ __forceinline__ void trailing_update(T* Gs, int n, int P, int a, T f0, T f1, int tid, int nt) {
    const int tx = tid & 31, ty = tid >> 5, ny = nt >> 5;
    for (int s = 0; s < 2; ++s) {
        T* Gb = Gs + (size_t)s * n * P;
        const T f = s ? f1 : f0;
        for (int r = a + 1 + ty; r < n; r += ny) {
            const T g = f * Gb[r * P + a];
            for (int c = a + 1 + tx; c < n; c += 32) Gb[r * P + c] = fma(g, Gb[a * P + c], Gb[r * P + c]);
        }
    }
}

// W = -F U1^{-1} L1^{-1} of the window (see the window kernel's tail); written to Wx[s][k][j] (pitch
// NW).  Cc[s][k][k'] (pitch P, spin stride n P) holds C[k][k'] f_k'.  32 warps: spin = warp / 16,
// columns (warp % 16) WC + c; lane l holds rows l + 32 r, r < RPL (RPL >= ceil(m / 32)).  WC is the
// least count that covers m columns with 16 warps, so all of them work; the next step's coefficient
// is fetched while the current one is applied, and the forward pass of a warp starts at its first
// column (identity columns are zero above the diagonal).
template <typename T, int RPL, int WC>
__device__ __forceinline__ void window_w_rpl(const T* Cc, int n, int P, const T (*fk)[WinCap<T>::NW], int m, T* Wx,
                                             int lane, int w) {
    constexpr int NW = WinCap<T>::NW;
    const int s = w >> 4, j0 = (w & 15) * WC;
    if (j0 >= m) return;
    const T* Cb = Cc + (size_t)s * n * P;
    T y[RPL][WC];
#pragma unroll
    for (int r = 0; r < RPL; ++r)
#pragma unroll
        for (int c = 0; c < WC; ++c) y[r][c] = (lane + 32 * r == j0 + c) ? T(1) : T(0);
    auto coef = [&](int kp, T* cf) {  // C[k][kp] f_kp of this lane's rows
#pragma unroll
        for (int r = 0; r < RPL; ++r) {
            const int k = lane + 32 * r;
            cf[r] = k < m ? Cb[k * P + kp] : T(0);
        }
    };
    auto bcast = [&](int kp, T* v) {  // row kp of y from the lane that holds it
        const int ro = kp >> 5, lo = kp & 31;
#pragma unroll
        for (int c = 0; c < WC; ++c) {
            T src = y[0][c];
#pragma unroll
            for (int r = 1; r < RPL; ++r)
                if (ro == r) src = y[r][c];
            v[c] = __shfl_sync(0xffffffffu, src, lo);
        }
    };
    T cf[RPL], cfn[RPL], v[WC];
    // forward: rows k > kp
    if (j0 + 1 < m) coef(j0, cf);
    for (int kp = j0; kp + 1 < m; ++kp) {
        if (kp + 2 < m) coef(kp + 1, cfn);
        bcast(kp, v);
#pragma unroll
        for (int r = 0; r < RPL; ++r) {
            const int k = lane + 32 * r;
            if (k > kp && k < m) {
#pragma unroll
                for (int c = 0; c < WC; ++c) y[r][c] -= cf[r] * v[c];
            }
        }
#pragma unroll
        for (int r = 0; r < RPL; ++r) cf[r] = cfn[r];
    }
    // backward: rows k < kp
    if (m >= 2) coef(m - 1, cf);
    for (int kp = m - 1; kp >= 1; --kp) {
        if (kp >= 2) coef(kp - 1, cfn);
        bcast(kp, v);
#pragma unroll
        for (int r = 0; r < RPL; ++r) {
            const int k = lane + 32 * r;
            if (k < kp) {
#pragma unroll
                for (int c = 0; c < WC; ++c) y[r][c] -= cf[r] * v[c];
            }
        }
#pragma unroll
        for (int r = 0; r < RPL; ++r) cf[r] = cfn[r];
    }
    T* Wd = Wx + (size_t)s * NW * NW;
#pragma unroll
    for (int r = 0; r < RPL; ++r) {
        const int k = lane + 32 * r;
        if (k < m) {
            const T fkk = -fk[s][k];
#pragma unroll
            for (int c = 0; c < WC; ++c)
                if (j0 + c < m) Wd[k * NW + j0 + c] = fkk * y[r][c];
        }
    }
}

// Cc[s][k][k'] = C[k][k'] f_k' in place over the block: every element of the accepted rows and columns
// is read (RU x CU registers a thread; warps over rows, lanes over columns) before any is written.  The
// block itself is not needed any more.
template <typename T, int RU, int CU>
__device__ __forceinline__ void window_compact(T* Gs, int n, int P, const int* idx, const T (*fk)[WinCap<T>::NW],
                                               int m, int tid) {
    const int lane = tid & 31, w = tid >> 5;
    T v[RU][CU];
#pragma unroll
    for (int a = 0; a < RU; ++a) {
        const int row = w + 32 * a, s = row >= m ? 1 : 0, k = row - s * m;
#pragma unroll
        for (int c = 0; c < CU; ++c) {
            const int kp = lane + 32 * c;
            if (k < m && kp < m) v[a][c] = Gs[(s * n + idx[k]) * P + idx[kp]] * fk[s][kp];
        }
    }
    __syncthreads();
#pragma unroll
    for (int a = 0; a < RU; ++a) {
        const int row = w + 32 * a, s = row >= m ? 1 : 0, k = row - s * m;
#pragma unroll
        for (int c = 0; c < CU; ++c) {
            const int kp = lane + 32 * c;
            if (k < m && kp < m) Gs[(s * n + k) * P + kp] = v[a][c];
        }
    }
    __syncthreads();
}

template <typename T>
__device__ __forceinline__ void window_w(T* Gs, int n, int P, const int* idx, const T (*fk)[WinCap<T>::NW], int m,
                                         T* Wx, int tid) {
    constexpr bool BIG = WinCap<T>::NW > 64;
    const int lane = tid & 31, w = tid >> 5;
    if (m <= 64) window_compact<T, 4, 2>(Gs, n, P, idx, fk, m, tid);
    else window_compact<T, WinCap<T>::NW / 16, WinCap<T>::NW / 32>(Gs, n, P, idx, fk, m, tid);
    if (m <= 16) window_w_rpl<T, 1, 1>(Gs, n, P, fk, m, Wx, lane, w);
    else if (m <= 32) window_w_rpl<T, 1, 2>(Gs, n, P, fk, m, Wx, lane, w);
    else if (m <= 48) window_w_rpl<T, 2, 3>(Gs, n, P, fk, m, Wx, lane, w);
    else if (m <= 64) window_w_rpl<T, 2, 4>(Gs, n, P, fk, m, Wx, lane, w);
    else if (BIG && m <= 96) window_w_rpl<T, BIG ? 3 : 2, BIG ? 6 : 4>(Gs, n, P, fk, m, Wx, lane, w);
    else window_w_rpl<T, BIG ? 4 : 2, BIG ? 8 : 4>(Gs, n, P, fk, m, Wx, lane, w);
}

// What warp 0 carries through a window's decisions (the same in every lane).
template <typename T>
struct WinScan {
    int m = 0;        // accepts so far
    int nneg = 0;     // accepted negative ratios (sign parity)
    T maxr = T(0);    // largest |R| of an accept
    bool alive = true;  // constrained path: the walker has not been removed
    bool bad = false;   // a non-finite ratio was met
    int done = 0;       // sites decided
};

// The decisions of the sites [b0, b0 + nbk) of the window, one warp for both spins: lane
// 16 s + r CG + cg holds row r, columns j CG + cg of spin s's sub-block in registers (CG = 16 / B), so
// a site costs its ratio (one shuffle for the diagonal, one to pair the spins) and an accept B shuffles
// of its row and as many multiply-adds, with no barrier.  Every lane takes the decision redundantly.
// An accept a updates the rows and columns after a only, with the products
// G[r][c] += (Delta/r G[r][a]) G[a][c] (f = -Delta/r) in accept order; row a and column a keep their values of that moment (the frozen coefficients).
//   Metropolis (AFQMC_MODE_DELAYED): R = s(-x)/s(x) r_up r_dn, r_s = 1 + Delta_s (1 - G_s[q][q]).
//   Constrained-path heat bath (WIN_MODE_CP, Sec. IV.D, Eq. ptilde): lambda(x) = p(x) s(x) r_up(x) r_dn(x),
//   negative lambda clamped to zero, x = +1 iff u (lambda(+1) + lambda(-1)) < lambda(+1); the walker is
//   removed when both vanish; every site is an accept.
template <typename T, int MODE>
__device__ __forceinline__ void window_sub_sites(T* Gs, int n, int P, int b0, int nbk, const int8_t* xw, const T* s_u,
                                                 const uint8_t* s_rep, bool forced, const T (*dflip)[2],
                                                 const T* sflip, T* s_rat, T* s_det, uint8_t* s_dec, int8_t* s_xch,
                                                 T (*s_fk)[WinCap<T>::NW], int* idx, WinScan<T>& sc, int lane) {
    constexpr int B = WinSub<T>::B, CG = 16 / B, CW = B / CG;
    constexpr unsigned FULL = 0xffffffffu;
    const int s = lane >> 4, r = (lane & 15) / CG, cg = lane % CG, half = lane & 16;
    T g[CW];  // columns q0 + j CG + cg of row r, q0 the site the loop is at
#pragma unroll
    for (int j = 0; j < CW; ++j) {
        const int c = j * CG + cg;
        g[j] = (r < nbk && c < nbk) ? Gs[(s * n + b0 + r) * P + b0 + c] : T(0);
    }
    T* col = Gs + (size_t)(s * n + b0 + (r < nbk ? r : 0)) * P + b0 + cg;
    const int ls = lane < nbk ? lane : 0;  // lane l < nbk keeps the inputs and outputs of site l
    const T u_l = s_u[b0 + ls];
    const int x_l = xw[b0 + ls], rep_l = s_rep[b0 + ls];
    const T d0 = dflip[s][0], d1 = dflip[s][1], sf0 = sflip[0], sf1 = sflip[1];
    unsigned mask = 0, plus = 0;
    T rat_l = T(0), det_l = T(0), f_l = T(0);
    const int m0 = sc.m;
#pragma unroll 1
    for (int q0 = 0; q0 < nbk && sc.alive; q0 += CG) {
#pragma unroll
        for (int t = 0; t < CG; ++t) {  // the current column sits in g[0] of the lanes cg == t
            const int q = q0 + t, src = half + q * CG;
            if (t > 0 && (q >= nbk || !sc.alive)) break;
            const T a = T(1) - __shfl_sync(FULL, g[0], src + t);
            const T u = __shfl_sync(FULL, u_l, q);
            const bool rep = __shfl_sync(FULL, rep_l, q) != 0;
            bool acc;
            T f;
            if (MODE == WIN_MODE_CP) {
                const T rp = T(1) + d0 * a, rm = T(1) + d1 * a;
                const T rpo = __shfl_xor_sync(FULL, rp, 16), rmo = __shfl_xor_sync(FULL, rm, 16);
                const T lp = fmax(sf0 * (s ? rpo : rp) * (s ? rp : rpo), T(0));
                const T lm = fmax(sf1 * (s ? rmo : rm) * (s ? rm : rmo), T(0));
                const T nrm = lp + lm;
                acc = nrm > T(0) && isfinite(nrm);
                if (!acc) {
                    sc.alive = false;
                    if (!isfinite(nrm)) sc.bad = true;
                }
                const bool up = forced ? rep : u * nrm < lp;
                f = -((up ? d0 : d1) / (up ? rp : rm));
                if (acc && up) plus |= 1u << q;
                if (lane == q) {
                    rat_l = nrm;
                    det_l = up ? rp * rpo : rm * rmo;
                }
            } else {
                const int xi = __shfl_sync(FULL, x_l, q) > 0 ? 0 : 1;
                const T dl = xi ? d1 : d0;
                const T rr = T(1) + dl * a, ro = __shfl_xor_sync(FULL, rr, 16);
                const T R = (xi ? sf1 : sf0) * (s ? ro : rr) * (s ? rr : ro);
                acc = forced ? rep : u < fabs(R);
                if (!isfinite(R)) {
                    acc = false;
                    sc.bad = true;
                }
                f = -(dl / rr);
                if (lane == q) rat_l = R;
                if (acc) {
                    if (R < T(0)) ++sc.nneg;
                    sc.maxr = fmax(sc.maxr, fabs(R));
                }
            }
            ++sc.done;
            if (acc) {
                mask |= 1u << q;
                if ((lane & 15) == q) f_l = f;
                const T fc = -f * (CG == 1 ? g[0] : __shfl_sync(FULL, g[0], half + r * CG + t));
#pragma unroll
                for (int j = t == CG - 1 ? 1 : 0; j < CW; ++j) {
                    const T rv = __shfl_sync(FULL, g[j], src + cg);
                    if (r > q && (j > 0 || cg > t)) g[j] = fma(fc, rv, g[j]);
                }
            }
        }
        if (r < nbk && q0 + cg < nbk) col[q0] = g[0];  // these columns are never written again
#pragma unroll
        for (int j = 0; j + 1 < CW; ++j) g[j] = g[j + 1];
    }
    sc.m = m0 + __popc(mask);
    if (lane < nbk) {
        s_dec[b0 + lane] = MODE == WIN_MODE_CP ? (plus >> lane) & 1u : (mask >> lane) & 1u;
        s_rat[b0 + lane] = rat_l;
        if (MODE == WIN_MODE_CP) s_det[b0 + lane] = det_l;
    }
    if ((mask >> (lane & 15)) & 1u) {
        const int k = m0 + __popc(mask & ((1u << (lane & 15)) - 1u));
        s_fk[s][k] = f_l;
        if (s == 0) {
            idx[k] = b0 + lane;
            if (MODE == WIN_MODE_CP) s_xch[k] = (plus >> lane) & 1u ? 1 : -1;
        }
    }
}

// The accepts k = 0 .. mk - 1 of the sub-block that ends before site b1 (sites ia[k], factors fa[s][k])
// applied to the rows and columns [b1, n) of both spins, all threads of the block:
//   1. the coefficient triangles of the sub-block, shifted to start after the diagonal:
//      D[0][s][k'][j] = G[a_k'][a_k] and D[1][s][k'][j] = -f_k' G[a_k][a_k'], k = k' + 1 + j (f = -Delta/r);
//   2. one thread per row (or column) of the panels: column a_k of the rows after the sub-block, and
//      row a_k of the columns after it, as they stood when a_k was accepted, by the recursion over the
//      earlier accepts; stored in place (the frozen coefficients) and as pw[s][r][k] = -f_k G[r][a_k],
//      qv[s][k][c] = G[a_k][c], zero-padded to whole 16-byte vectors;
//   3. G[r][c] += sum_k pw qv, in accept order, one column and a few rows a thread.
// The arithmetic is that of one trailing rank-1 update per accept, in the same order.
template <typename T>
__device__ __forceinline__ void window_sub_update(T* Gs, int n, int P, int b1, int mk, const int* ia, const T* fu,
                                                  const T* fd, T* D, T* pw, T* qv, int tid, int nt) {
    constexpr int B = WinSub<T>::B, VW = Vec16<T>::W;
    using V = typename Vec16<T>::V;
    const int rem = n - b1;
    for (int e = tid; e < 4 * B * B; e += nt) {
        const int j = e % B, kp = (e / B) % B, s = (e / (B * B)) & 1, kind = e / (2 * B * B), k = kp + 1 + j;
        T v = T(0);
        if (k < mk) {
            const T* Gb = Gs + (size_t)s * n * P;
            v = kind ? -(s ? fd : fu)[kp] * Gb[ia[k] * P + ia[kp]] : Gb[ia[kp] * P + ia[k]];
        }
        D[e] = v;
    }
    __syncthreads();
    for (int e = tid; e < 4 * rem; e += nt) {
        const int kind = e >= 2 * rem ? 1 : 0, e2 = e - kind * 2 * rem, s = e2 >= rem ? 1 : 0, i = e2 - s * rem;
        T* line = Gs + (size_t)s * n * P + (kind ? b1 + i : (b1 + i) * P);
        const int step = kind ? P : 1;
        const T* Dm = D + (kind * 2 + s) * B * B;
        const T* f = s ? fd : fu;
        T* out = kind ? qv + s * B * n + i : pw + (s * n + i) * B;
        const int ostep = kind ? n : 1;
        T v[B];  // v[j]: entry kp + j of the line, kp the accept the loop is at
#pragma unroll
        for (int k = 0; k < B; ++k) v[k] = k < mk ? line[ia[k] * step] : T(0);
#pragma unroll 1
        for (int kp = 0; kp < mk; ++kp) {
            const T w = kind ? v[0] : -f[kp] * v[0];
            line[ia[kp] * step] = v[0];
            out[kp * ostep] = w;
#pragma unroll
            for (int j0 = 0; j0 < B; j0 += VW) {
                T d[VW];
                *(V*)d = *(const V*)(Dm + kp * B + j0);
#pragma unroll
                for (int l = 0; l < VW; ++l)
                    if (j0 + l + 1 < B) v[j0 + l] = fma(w, d[l], v[j0 + l + 1]);
            }
        }
        for (int kp = mk; kp < (mk + VW - 1) / VW * VW; ++kp) out[kp * ostep] = T(0);
    }
    __syncthreads();
    const int rt = (2 * rem * rem + nt - 1) / nt, ngr = (rem + rt - 1) / rt, tot = 2 * rem * ngr;
    for (int e = tid; e < tot; e += nt) {
        const int s = e >= rem * ngr ? 1 : 0, e2 = e - s * rem * ngr, rg = e2 / rem, c = e2 - rg * rem;
        T q[B];
#pragma unroll
        for (int k0 = 0; k0 < B; k0 += VW)
#pragma unroll
            for (int l = 0; l < VW; ++l) q[k0 + l] = k0 < mk ? qv[(s * B + k0 + l) * n + c] : T(0);
        const int rlo = rg * rt, rhi = min(rem, rlo + rt);
        T* out = Gs + ((size_t)s * n + b1 + rlo) * P + b1 + c;
        const T* pr = pw + (size_t)(s * n + rlo) * B;
        for (int r = rlo; r < rhi; ++r, out += P, pr += B) {
            T acc = *out;
#pragma unroll
            for (int k0 = 0; k0 < B; k0 += VW) {
                if (k0 < mk) {
                    T w[VW];
                    *(V*)w = *(const V*)(pr + k0);
#pragma unroll
                    for (int l = 0; l < VW; ++l) acc = fma(w[l], q[k0 + l], acc);
                }
            }
            *out = acc;
        }
    }
    __syncthreads();
}

template <typename T, int MODE>
__global__ void __launch_bounds__(WIN_THREADS) window_kernel(const T* __restrict__ Gu0, int8_t* xl0, const double* u0,
                                                             const uint8_t* replay0, SiteParams sp, SliceOut so0,
                                                             int s0, int n, int nb, WindowBufs wb0, const T* blk0,
                                                             int* err, Batch bt) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int P = n + 1;
    const int tid = threadIdx.x, nt = blockDim.x;
    const int N = sp.N;
    const long ld = sp.ld;
    // walker blockIdx.x of the group
    const int wk = blockIdx.x;
    const T* __restrict__ Gu = Gu0 + (size_t)wk * bt.gstride;
    const T* __restrict__ Gd = Gu + (size_t)N * ld;
    int8_t* xl_g = xl0 + (size_t)wk * bt.xstride;
    const double* u = u0 + (size_t)wk * 2 * N;
    const uint8_t* replay = replay0 ? replay0 + (size_t)wk * 2 * N : nullptr;
    const SliceOut so = so_walker(so0, wk, N);
    const WindowBufs wb = wb_walker<T>(wb0, wk, N);
    const T* blk = blk0 ? blk0 + (size_t)wk * 2 * WinCap<T>::NW * WinCap<T>::NW : nullptr;
    T* Gs = (T*)smem_raw;  // [2][n][P]
    size_t off = 2 * (size_t)n * P * sizeof(T);  // a multiple of 16: n (n + 1) is even
    constexpr int SB = WinSub<T>::B;
    T* Dsub = (T*)(smem_raw + off);    // [2][2][SB][SB] sub-block coefficients (window_sub_update)
    T* pwsub = Dsub + 4 * SB * SB;     // [2][n][SB]
    T* qvsub = pwsub + 2 * n * SB;     // [2][SB][n]
    off += 4 * (size_t)SB * (SB + n) * sizeof(T);
    T* S1 = (T*)(smem_raw + off);  // [2][NBMAX][NBMAX+1]
    off += 2 * (size_t)NBMAX * (NBMAX + 1) * sizeof(T);
    T* stc = (T*)(smem_raw + off);  // staging: col[2][n], row[2][n]
    off += 4 * (size_t)n * sizeof(T);
    T* stb = (T*)(smem_raw + off);  // small staging [2][NBMAX]
    off += 2 * (size_t)NBMAX * sizeof(T);
    off = (off + 7) & ~(size_t)7;
    double* fb = (double*)(smem_raw + off);  // block-FB scalars [8][NBMAX]
    off += 8 * (size_t)NBMAX * sizeof(double);
    int* idx = (int*)(smem_raw + off);  // accepted positions [n]
    off += (size_t)n * sizeof(int);
    int8_t* xw = (int8_t*)(smem_raw + off);  // window fields [n]
    off += (size_t)n;
    __shared__ int s_m, s_nF;
    __shared__ int s_F[NBMAX];
    __shared__ double s_R;
    constexpr int NWC = WinCap<T>::NW;
    __shared__ T s_fk[2][NWC];  // f_k = -Delta_k / r_k of accept k, both spins

    const T* G[2] = {Gu, Gd};
    // the n x n diagonal block of both spins: from G, or from the corrected snapshot the
    // previous window's flush prepared (pitch NW, spin stride NW^2)
    {  // warps over rows, lanes over columns; four rows' loads in flight per thread before their stores
        const int lane = tid & 31;
        for (int c = lane; c < n; c += 32)
            for (int row0 = tid >> 5; row0 < 2 * n; row0 += 4 * (nt >> 5)) {
                T v[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const int row = row0 + q * (nt >> 5), s = row >= n ? 1 : 0, a = row - s * n;
                    if (row < 2 * n)
                        v[q] = blk ? blk[((size_t)s * WinCap<T>::NW + a) * WinCap<T>::NW + c]
                                   : G[s][(long)(s0 + a) * ld + (s0 + c)];
                }
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const int row = row0 + q * (nt >> 5);
                    if (row < 2 * n) Gs[row * P + c] = v[q];
                }
            }
    }
    for (int p = tid; p < n; p += nt) xw[p] = xl_g[s0 + p];
    // the window's site uniforms (and forced decisions) live in shared memory: the scan reads
    // them on its critical path
    // (in the bulk precision: the delayed scan compares them with ratios computed in T)
    __shared__ T s_u[WinCap<float>::NW];
    __shared__ uint8_t s_rep[WinCap<float>::NW];
    __shared__ T s_rat[WinCap<float>::NW];    // ratio of every decided site, written out after the decisions
    __shared__ uint8_t s_dec[WinCap<float>::NW];
    for (int p = tid; p < n; p += nt) {
        s_u[p] = (T)u[s0 + p];
        s_rep[p] = replay ? replay[s0 + p] : 0;
    }
    __shared__ double c_dflip[2][2], c_dstrip[2][2], c_sflip[2];
    __shared__ T c_dflipT[2][2], c_sflipT[2];  // the same in T for the scan's critical path
    if (tid < 4) {
        c_dflip[tid >> 1][tid & 1] = sp.dflip[tid >> 1][tid & 1];
        c_dstrip[tid >> 1][tid & 1] = sp.dstrip[tid >> 1][tid & 1];
    }
    if (tid < 2) c_sflip[tid] = sp.sflip[tid];
    if (tid < 4) c_dflipT[tid >> 1][tid & 1] = (T)sp.dflip[tid >> 1][tid & 1];
    if (tid < 2) c_sflipT[tid] = (T)sp.sflip[tid];
    if (tid == 0) s_m = 0;
    __syncthreads();

    __shared__ double s_sign, s_maxr;  // walker sign and max |R|, owned by one thread at a time
    if (tid == 0) {
        s_sign = so.sign ? *so.sign : 1.0;
        s_maxr = 0.0;
    }
    __syncthreads();
    int n_prop = 0, n_acc = 0, n_flip = 0;

    __shared__ int8_t s_xch[WinCap<float>::NW];  // constrained path: the field chosen at each site
    __shared__ double s_cpl[2];                  // constrained path: sum ln N_i, sum ln |r_up r_dn|
    __shared__ int s_dead;
    if ((MODE == WIN_MODE_CP || MODE == WIN_MODE_CPB) && tid == 0) {
        s_cpl[0] = 0.0;
        s_cpl[1] = 0.0;
        s_dead = so.cp ? (so.cp[2] != 0.0) : 0;
    }
    __syncthreads();
    if (MODE == AFQMC_MODE_DELAYED || MODE == WIN_MODE_CP) {
        // Two levels: warp 0 decides a sub-block of SB sites in registers (no barrier per accept), then
        // all warps bring the rest of the window's block up to date with the sub-block's accepts.
        __shared__ int s_mk[2];
        __shared__ T s_det[WinCap<float>::NW];  // constrained path: r_up r_dn of every site
        WinScan<T> sc;
        sc.alive = !((MODE == WIN_MODE_CP) && s_dead);
        int m_all = 0;
        for (int b0 = 0, it = 0; b0 < n; b0 += SB, ++it) {
            const int b1 = min(n, b0 + SB);
            if (tid < 32) {
                window_sub_sites<T, MODE>(Gs, n, P, b0, b1 - b0, xw, s_u, s_rep, replay != nullptr, c_dflipT,
                                          c_sflipT, s_rat, s_det, s_dec, s_xch, s_fk, idx, sc, tid);
                if (tid == 0) s_mk[it & 1] = sc.m;
            }
            __syncthreads();
            const int mk = s_mk[it & 1] - m_all;
            if (mk > 0 && b1 < n)
                window_sub_update<T>(Gs, n, P, b1, mk, idx + m_all, s_fk[0] + m_all, s_fk[1] + m_all, Dsub, pwsub,
                                     qvsub, tid, nt);
            m_all += mk;
        }
        if (tid == 0) {
            s_m = sc.m;
            if (sc.bad) set_err(err, DEV_NUMERIC);
            if (sc.nneg & 1) s_sign = -s_sign;
            s_maxr = fmax(s_maxr, (double)sc.maxr);
            n_prop = sc.done;
            n_acc = n_flip = sc.m;
            if (MODE == WIN_MODE_CP && !sc.alive) s_dead = 1;
        }
        __syncthreads();
        // decisions and ratios in their ABI types; the walker's weight factors as sums over its sites
        for (int q = tid; q < n; q += nt) {
            so.dec[s0 + q] = s_dec[q];
            so.ratio[s0 + q] = (double)s_rat[q];
        }
        if (MODE == WIN_MODE_CP && tid < 32) {
            double a0 = 0.0, a1 = 0.0;
            for (int q = tid; q < s_m; q += 32) {
                a0 += log((double)s_rat[idx[q]]);
                a1 += log(fabs((double)s_det[idx[q]]));
            }
            for (int o = 16; o > 0; o >>= 1) {
                a0 += __shfl_xor_sync(0xffffffffu, a0, o);
                a1 += __shfl_xor_sync(0xffffffffu, a1, o);
            }
            if (tid == 0) {
                s_cpl[0] = a0;
                s_cpl[1] = a1;
            }
        }
        __syncthreads();
    } else if (MODE == WIN_MODE_CPB) {
        // ---- constrained-path block force bias (Sec. IV.D) ----
        // Per block S of nb sites (no field set yet): the force bias F_i of the current block's
        // diagonal (spin channel sum_s c_s A_s[i][i], charge channel lam (A_up + A_dn - 1)[i][i]),
        // each x_i from q(x_i) = e^{x_i F_i} / (2 cosh F_i); the weight factor
        // prod_i s(x_i) cosh F_i e^{-x_i F_i} prod_s det(1 + Delta_s A_s[S][S]) (the determinant as the
        // product of the sequential rank-1 ratios on a copy of the block); a factor <= 0 removes the
        // walker; the fields are then applied as accepts of the delayed update.
        __shared__ T s_phi2[2][NBMAX];
        __shared__ double s_rs2[2];
        T* strow = stc + 2 * n;  // [2][n]
        for (int p0 = 0; p0 < n && !s_dead; p0 += nb) {
            const int nbk = min(nb, n - p0);
            if (tid < nbk) {
                const int a = tid, i = s0 + p0 + a;
                const double a0 = 1.0 - (double)Gs[(0 * n + p0 + a) * P + p0 + a];
                const double a1 = 1.0 - (double)Gs[(1 * n + p0 + a) * P + p0 + a];
                const double F = sp.hs == AFQMC_HS_CHARGE_REAL ? sp.lam * (a0 + a1 - 1.0) : sp.c[0] * a0 + sp.c[1] * a1;
                const double lamp = 1.0 / (1.0 + exp(-2.0 * F));
                const int xp = replay ? (replay[i] ? 1 : -1) : (u[i] < lamp ? 1 : -1);
                so.dec[i] = xp > 0 ? 1 : 0;
                so.ratio[i] = lamp;
                fb[0 * NBMAX + a] = hs_log_scalar(sp, xp) + log(cosh(F)) - xp * F;
                s_xch[s_m + a] = (int8_t)xp;
            }
            for (int e = tid; e < 2 * nbk * nbk; e += nt) {
                int sp2 = e / (nbk * nbk), rem = e % (nbk * nbk), a = rem / nbk, c = rem % nbk;
                S1[(sp2 * NBMAX + a) * (NBMAX + 1) + c] = Gs[(sp2 * n + p0 + a) * P + p0 + c];
            }
            if (tid == 0) {
                s_rs2[0] = 1.0;
                s_rs2[1] = 1.0;
            }
            __syncthreads();
            const int mb = s_m;
            for (int q = 0; q < nbk; ++q) {
                for (int e = tid; e < 2 * nbk; e += nt) {
                    int sp2 = e / nbk, c = e % nbk;
                    T* Sb = S1 + sp2 * NBMAX * (NBMAX + 1);
                    stb[sp2 * NBMAX + c] = Sb[c * (NBMAX + 1) + q];
                    strow[sp2 * n + c] = (c == q ? T(1) : T(0)) - Sb[q * (NBMAX + 1) + c];
                }
                if (tid < 2) {
                    const int xi = s_xch[mb + q] > 0 ? 0 : 1;
                    const T dd = c_dflipT[tid][xi];
                    const T rr = T(1) + dd * (T(1) - S1[(tid * NBMAX + q) * (NBMAX + 1) + q]);
                    s_rs2[tid] *= (double)rr;
                    s_phi2[tid][q] = dd / rr;
                }
                __syncthreads();
                for (int e = tid; e < 2 * nbk * nbk; e += nt) {
                    int sp2 = e / (nbk * nbk), rem = e % (nbk * nbk), r = rem / nbk, c = rem % nbk;
                    T* Sb = S1 + sp2 * NBMAX * (NBMAX + 1);
                    Sb[r * (NBMAX + 1) + c] -= s_phi2[sp2][q] * stb[sp2 * NBMAX + r] * strow[sp2 * n + c];
                }
                __syncthreads();
            }
            if (tid == 0) {
                double lw = 0.0;
                for (int a = 0; a < nbk; ++a) lw += fb[0 * NBMAX + a];
                const double det = s_rs2[0] * s_rs2[1];
                const int blk = (s0 + p0) / nb;
                so.ratio[N + blk] = det;
                if (!(det > 0.0) || !isfinite(det)) {
                    s_dead = 1;
                    if (!isfinite(det)) set_err(err, DEV_NUMERIC);
                } else {
                    s_cpl[0] += lw + log(det);
                    s_cpl[1] += log(det);
                }
                so.dec[N + blk] = s_dead ? 0 : 1;
            }
            __syncthreads();
            if (s_dead) break;
            ++n_prop;
            ++n_acc;
            n_flip += nbk;
            for (int q = 0; q < nbk; ++q) {
                const int a = p0 + q, k = mb + q;
                if (tid == 0) {
                    idx[k] = a;
                    s_fk[0][k] = -s_phi2[0][q];
                    s_fk[1][k] = -s_phi2[1][q];
                }
                trailing_update(Gs, n, P, a, s_phi2[0][q], s_phi2[1][q], tid, nt);
                __syncthreads();
            }
            if (tid == 0) s_m = mb + nbk;
            __syncthreads();
        }
    } else {
        // ---- block force-bias (Sec. III.B) ----
        __shared__ T s_fs[2];
        __shared__ double s_rs[2];
        __shared__ int s_accb;
        __shared__ T s_phi[2][NBMAX];
        T* strow = stc + 2 * n;  // [2][n]
        for (int p0 = 0; p0 < n; p0 += nb) {
            const int nbk = min(nb, n - p0);
            const int blk = (s0 + p0) / nb;
            // (a) stripped force bias (Eq. BlkFrcBsTnew1): remove the block's fields one site at a time,
            //     each a rank-1 step G <- G - (d/r) G_{:,a} (e_a^T - G_{a,:}) with d = exp(-c x_a) - 1
            for (int e = tid; e < 2 * nbk * nbk; e += nt) {
                int s = e / (nbk * nbk), rem = e % (nbk * nbk), a = rem / nbk, c = rem % nbk;
                S1[(s * NBMAX + a) * (NBMAX + 1) + c] = Gs[(s * n + p0 + a) * P + p0 + c];
            }
            __syncthreads();
            for (int a = 0; a < nbk; ++a) {
                for (int e = tid; e < 2 * nbk; e += nt) {
                    int s = e / nbk, c = e % nbk;
                    T* Sb = S1 + s * NBMAX * (NBMAX + 1);
                    stb[s * NBMAX + c] = Sb[c * (NBMAX + 1) + a];                       // column a
                    strow[s * n + c] = (c == a ? T(1) : T(0)) - Sb[a * (NBMAX + 1) + c];  // e_a^T - row a
                }
                if (tid < 2) {
                    const int xi = xw[p0 + a] > 0 ? 0 : 1;
                    const T db = (T)c_dstrip[tid][xi];
                    const T rr = T(1) + db * (T(1) - S1[(tid * NBMAX + a) * (NBMAX + 1) + a]);
                    s_fs[tid] = db / rr;
                }
                __syncthreads();
                for (int e = tid; e < 2 * nbk * nbk; e += nt) {
                    int s = e / (nbk * nbk), rem = e % (nbk * nbk), r = rem / nbk, c = rem % nbk;
                    T* Sb = S1 + s * NBMAX * (NBMAX + 1);
                    Sb[r * (NBMAX + 1) + c] -= s_fs[s] * stb[s * NBMAX + r] * strow[s * n + c];
                }
                __syncthreads();
            }
            // (b) proposals from lambda(x') = bbar(x') / sum bbar, bbar(x) = s(x) e^{x h}
            if (tid < nbk) {
                const int a = tid, i = s0 + p0 + a;
                const double nb0 = 1.0 - (double)S1[(0 * NBMAX + a) * (NBMAX + 1) + a];
                const double nb1 = 1.0 - (double)S1[(1 * NBMAX + a) * (NBMAX + 1) + a];
                const double h = sp.c[0] * nb0 + sp.c[1] * nb1;
                const double lp = hs_log_scalar(sp, +1) + h, lm = hs_log_scalar(sp, -1) - h;
                const double lamp = 1.0 / (1.0 + exp(lm - lp));
                const int x = xw[p0 + a];
                const int xp = replay ? (replay[i] ? 1 : -1) : (u[i] < lamp ? 1 : -1);
                so.dec[i] = xp > 0 ? 1 : 0;
                so.ratio[i] = lamp;
                double lpr = 0.0;
                if (xp != x) {
                    double lbx = hs_log_scalar(sp, x) + x * h, lbxp = hs_log_scalar(sp, xp) + xp * h;
                    lpr = (hs_log_scalar(sp, xp) - hs_log_scalar(sp, x)) + (lbx - lbxp);
                }
                fb[0 * NBMAX + a] = lpr;
                fb[1 * NBMAX + a] = (xp != x) ? 1.0 : 0.0;
            }
            __syncthreads();
            if (tid == 0) {
                int nF = 0;
                double lpr = 0.0;
                for (int a = 0; a < nbk; ++a)
                    if (fb[1 * NBMAX + a] != 0.0) {
                        s_F[nF++] = a;
                        lpr += fb[0 * NBMAX + a];
                    }
                s_nF = nF;
                s_R = exp(lpr);
                s_rs[0] = 1.0;
                s_rs[1] = 1.0;
            }
            __syncthreads();
            const int nF = s_nF;
            ++n_prop;
            if (nF == 0) {
                if (tid == 0) {
                    so.dec[N + blk] = 1;
                    so.ratio[N + blk] = 1.0;
                }
                ++n_acc;
                continue;
            }
            // (c) det(1 + D_F A_FF) (Eq. BlkFrcBsTnew2's ratio) as the product of sequential rank-1 ratios
            for (int e = tid; e < 2 * nbk * nbk; e += nt) {
                int s = e / (nbk * nbk), rem = e % (nbk * nbk), a = rem / nbk, c = rem % nbk;
                S1[(s * NBMAX + a) * (NBMAX + 1) + c] = Gs[(s * n + p0 + a) * P + p0 + c];
            }
            __syncthreads();
            for (int q = 0; q < nF; ++q) {
                const int a = s_F[q];
                for (int e = tid; e < 2 * nbk; e += nt) {
                    int s = e / nbk, c = e % nbk;
                    T* Sb = S1 + s * NBMAX * (NBMAX + 1);
                    stb[s * NBMAX + c] = Sb[c * (NBMAX + 1) + a];
                    strow[s * n + c] = (c == a ? T(1) : T(0)) - Sb[a * (NBMAX + 1) + c];
                }
                if (tid < 2) {
                    const int xi = xw[p0 + a] > 0 ? 0 : 1;
                    const T dd = (T)c_dflip[tid][xi];
                    const T rr = T(1) + dd * (T(1) - S1[(tid * NBMAX + a) * (NBMAX + 1) + a]);
                    s_rs[tid] *= (double)rr;
                    s_phi[tid][q] = dd / rr;
                    fb[(4 + tid) * NBMAX + q] = (double)dd;
                }
                __syncthreads();
                for (int e = tid; e < 2 * nbk * nbk; e += nt) {
                    int s = e / (nbk * nbk), rem = e % (nbk * nbk), r = rem / nbk, c = rem % nbk;
                    T* Sb = S1 + s * NBMAX * (NBMAX + 1);
                    Sb[r * (NBMAX + 1) + c] -= s_phi[s][q] * stb[s * NBMAX + r] * strow[s * n + c];
                }
                __syncthreads();
            }
            if (tid == 0) {
                const double R = s_R * s_rs[0] * s_rs[1];
                bool acc = replay ? (replay[N + blk] != 0) : (u[N + blk] < fabs(R));
                if (!isfinite(R)) {
                    acc = false;
                    set_err(err, DEV_NUMERIC);
                }
                so.dec[N + blk] = acc ? 1 : 0;
                so.ratio[N + blk] = R;
                s_accb = acc ? 1 : 0;
                if (acc) {
                    if (R < 0) s_sign = -s_sign;
                    s_maxr = fmax(s_maxr, fabs(R));
                }
            }
            __syncthreads();
            if (!s_accb) continue;
            ++n_acc;
            n_flip += nF;
            // (d) apply the flips in increasing site order, each as the trailing rank-1 step of the
            //     delayed update (rows / columns after the flipped site): the same product of
            //     rank-1 factors as Eq. BlkFrcBsTnew2, and the frozen rows / columns feed the flush
            const int mb = s_m;
            for (int q = 0; q < nF; ++q) {
                const int a = p0 + s_F[q], k = mb + q;
                if (tid == 0) {
                    idx[k] = a;
                    s_fk[0][k] = -s_phi[0][q];
                    s_fk[1][k] = -s_phi[1][q];
                    xw[a] = (int8_t)(-xw[a]);
                }
                trailing_update(Gs, n, P, a, s_phi[0][q], s_phi[1][q], tid, nt);
                __syncthreads();
            }
            if (tid == 0) s_m = mb + nF;
            __syncthreads();
        }
    }
    __syncthreads();
    const int m = s_m;
    if (MODE == AFQMC_MODE_DELAYED) {  // apply the accepted flips (deferred: xw[p] was read by every thread)
        for (int q = tid; q < m; q += nt) xw[idx[q]] = (int8_t)(-xw[idx[q]]);
        __syncthreads();
    }
    if (MODE == WIN_MODE_CP || MODE == WIN_MODE_CPB) {  // the chosen fields, and the walker's weight factors
        for (int q = tid; q < m; q += nt) xw[idx[q]] = s_xch[q];
        if (tid == 0 && so.cp) {
            so.cp[0] += s_cpl[0];
            so.cp[1] += s_cpl[1];
            if (s_dead) so.cp[2] = 1.0;
        }
        __syncthreads();
    }
    for (int p = tid; p < n; p += nt) xl_g[s0 + p] = xw[p];
    for (int q = tid; q < m; q += nt) wb.idx[q] = s0 + idx[q];
    // The window's update matrix W (Eq. DelayRgenk in G form).  With C[k][k'] = Gs[idx[k]][idx[k']]
    // the block entries frozen at acceptance time (rows and columns at or before an accepted site
    // are never touched again), f_k = -Delta_k / r_k, L1 = I + Cl F and U1 = I + Cu F (Cl, Cu the
    // strictly lower / upper parts of C, F = diag f), the delayed-update recursions give
    // W = -F U1^{-1} L1^{-1}: per column of the identity a forward and a backward substitution,
    //   y_k = b_k - sum_{k'<k} C[k][k'] f_k' y_k',   z_k = y_k - sum_{k'>k} C[k][k'] f_k' z_k',
    //   W_k = -f_k z_k.
    // The coefficients are gathered into a dense m x m matrix first; then each warp owns a few columns
    // of one spin in registers (lane l holds rows l, l + 32, ...) and broadcasts the finished row of
    // every step with a shuffle: no block-wide barrier per step.
    window_w<T>(Gs, n, P, idx, s_fk, m, (T*)wb.Wx, tid);
    if (tid == 0) {
        *wb.m = m;
        if (so.sign) *so.sign = s_sign;
        so.stats[0] += n_prop;
        so.stats[1] += n_acc;
        so.stats[2] += n_flip;
        so.stats[3] += (m > 0) ? 1 : 0;
        *so.maxr = fmax(*so.maxr, s_maxr);
    }
}

template <typename T>
cudaError_t launch_window_chain(cudaStream_t st, int mode, const T* Gu, const T* Gd, int8_t* xl,
                                const double* u, const uint8_t* replay, const SiteParams& sp, SliceOut so,
                                int s0, int n, int nb, WindowBufs wb, const T* blk, int* err, Batch bt) {
    (void)Gd;  // spin down follows spin up (N x ld) in every walker's G
    size_t shm = window_smem<T>(n);
    auto kfn = (mode == AFQMC_MODE_DELAYED) ? (const void*)window_kernel<T, AFQMC_MODE_DELAYED>
               : (mode == WIN_MODE_CP)     ? (const void*)window_kernel<T, WIN_MODE_CP>
               : (mode == WIN_MODE_CPB)    ? (const void*)window_kernel<T, WIN_MODE_CPB>
                                            : (const void*)window_kernel<T, AFQMC_MODE_BLOCKFB>;
    {
        cudaError_t e = ensure_smem_attr(kfn, window_smem<T>(WinCap<T>::NW));
        if (e != cudaSuccess) return e;
    }
    if (bt.nwk < 1) bt.nwk = 1;
    count_launch();
    if (mode == AFQMC_MODE_DELAYED)
        window_kernel<T, AFQMC_MODE_DELAYED><<<bt.nwk, WIN_THREADS, shm, st>>>(Gu, xl, u, replay, sp, so, s0, n, nb,
                                                                              wb, blk, err, bt);
    else if (mode == WIN_MODE_CP)
        window_kernel<T, WIN_MODE_CP><<<bt.nwk, WIN_THREADS, shm, st>>>(Gu, xl, u, replay, sp, so, s0, n, nb, wb,
                                                                       blk, err, bt);
    else if (mode == WIN_MODE_CPB)
        window_kernel<T, WIN_MODE_CPB><<<bt.nwk, WIN_THREADS, shm, st>>>(Gu, xl, u, replay, sp, so, s0, n, nb, wb,
                                                                        blk, err, bt);
    else
        window_kernel<T, AFQMC_MODE_BLOCKFB><<<bt.nwk, WIN_THREADS, shm, st>>>(Gu, xl, u, replay, sp, so, s0, n, nb,
                                                                              wb, blk, err, bt);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// flush: X = G[:, I], Yraw = E_I^T - G[I, :], Y = W Yraw, G <- G - X Y
// ---------------------------------------------------------------------------
template <typename T>
__global__ void gather_kernel(const T* __restrict__ Gu0, long ld, int N, WindowBufs wb0, int NW, long gstride,
                              long sstride) {
    const int wk = blockIdx.z;
    const WindowBufs wb = wb_walker<T>(wb0, wk, N);
    const int m = *wb.m;
    const int s = blockIdx.y;
    const T* G = Gu0 + (size_t)wk * gstride + (long)s * sstride;
    T* X = (T*)wb.X + (size_t)s * N * NW;
    T* Y = (T*)wb.Y + (size_t)s * NW * N;  // Yraw here; the product with W comes after
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < m * N; e += gridDim.x * blockDim.x) {
        int a = e / N, j = e % N;
        int I = wb.idx[a];
        Y[(size_t)a * N + j] = (j == I ? T(1) : T(0)) - G[(long)I * ld + j];
        int r = e / m, q = e % m;  // X row r, column q (coalesced over q is poor; rows are short)
        X[(size_t)r * NW + q] = G[(long)r * ld + wb.idx[q]];
    }
}

template <typename T>
cudaError_t launch_flush(cudaStream_t st, T* Gu, T* Gd, const SiteParams& sp, WindowBufs wb, int nw) {
    const int N = sp.N;
    const int NWC = WinCap<T>::NW;
    count_launch();
    gather_kernel<T><<<dim3(256, 2, 1), 256, 0, st>>>(Gu, sp.ld, N, wb, NWC, 0, (long)(Gd - Gu));
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    // Y <- W * Yraw  (rows >= m are never read); written into the X buffer's tail? use a separate pass:
    // compute in place is unsafe, so the product goes to the second half of the Y buffer.
    GemmArgs<T> g;
    g.M = nw; g.N = N; g.K = nw; g.Kdev = wb.m;
    g.A = (const T*)wb.Wm; g.lda = NWC; g.sA = (long)NWC * NWC;
    g.B = (const T*)wb.Y; g.ldb = N; g.sB = (long)NWC * N;
    g.C = (T*)wb.Y + (size_t)2 * NWC * N; g.ldc = N; g.sC = (long)NWC * N;
    g.alpha = T(1); g.beta = T(0);
    g.batch = 2;
    e = gemm<T>(st, g);
    if (e != cudaSuccess) return e;
    // G <- G - X Y
    GemmArgs<T> h;
    h.M = N; h.N = N; h.K = nw; h.Kdev = wb.m;
    h.A = (const T*)wb.X; h.lda = NWC; h.sA = (long)N * NWC;
    h.B = (const T*)wb.Y + (size_t)2 * NWC * N; h.ldb = N; h.sB = (long)NWC * N;
    h.C = Gu; h.ldc = sp.ld; h.sC = (long)(Gd - Gu);
    h.alpha = T(-1); h.beta = T(1);
    h.batch = 2;
    return gemm<T>(st, h);
}

template cudaError_t launch_local<float>(cudaStream_t, float*, float*, int8_t*, const double*, const uint8_t*,
                                         const SiteParams&, SliceOut, float*, float*, GridBar*, int*, int);
template cudaError_t launch_local<double>(cudaStream_t, double*, double*, int8_t*, const double*, const uint8_t*,
                                          const SiteParams&, SliceOut, double*, double*, GridBar*, int*, int);
template cudaError_t launch_window_chain<float>(cudaStream_t, int, const float*, const float*, int8_t*,
                                                const double*, const uint8_t*, const SiteParams&, SliceOut, int,
                                                int, int, WindowBufs, const float*, int*, Batch);
template cudaError_t launch_window_chain<double>(cudaStream_t, int, const double*, const double*, int8_t*,
                                                 const double*, const uint8_t*, const SiteParams&, SliceOut, int,
                                                 int, int, WindowBufs, const double*, int*, Batch);
// ---------------------------------------------------------------------------
// Pipelined flush of one window.
//
// The window kernel leaves W (m x m) in wb.Wm: the accumulated update of the window is
// G <- G - X W Yraw with X = G[:, I] and Yraw = E_I^T - G[I, :] (I the accepted sites).
//   * next_block_kernel (main stream, right after the window): the next window's n' x n' block
//     of G as it will be after this window's update, from three small gathers of G and two
//     small products in shared memory.  The next window starts from it at once.
//   * launch_flush_panels + launch_flush_gemm (flush stream): the panel gathers, Y' = W Yraw
//     and the rank-m product over all of G, overlapping the next window's decisions.
// ---------------------------------------------------------------------------

// snap[s][a][c] = G[sn + a][sn + c] - sum_k X[sn + a][k] Y'[k][sn + c], with X = G[:, I],
// Y' = W Yraw and Yraw[l][sn + c] = -G[I_l][sn + c] (the next window's sites are not in I): the
// block of the next window as it will be after this window's product.  Grid (row blocks of
// NB_ROWS, spin); each CTA forms (X_blk W) and then (X_blk W) Yraw_n for its rows.
constexpr int NB_ROWS = 4;
constexpr int NB_THREADS = 512;
// One CTA per (row block of NB_ROWS rows, spin, walker).  The gathers depend on the accepted sites,
// so the kernel takes two rounds of global loads: the sites, then W, Yraw_n, X_blk and the block's
// own rows of G, each mapped as warps over rows and lanes over columns (no index divisions, every
// load of a thread in flight before its shared-memory stores).  The two products split each
// output's sum over four consecutive lanes (strided partial sums, combined by shuffles), so every
// warp works on them.
template <typename T>
__global__ void __launch_bounds__(NB_THREADS) next_block_kernel(const T* __restrict__ Gu0, long ld, int N,
                                                                WindowBufs wb0, int sn, int nn, T* snap0,
                                                                long gstride) {
    constexpr int NW = WinCap<T>::NW, PP = NW + 1;
    const int wk = blockIdx.z;
    const WindowBufs wb = wb_walker<T>(wb0, wk, N);
    const int m = *wb.m;
    const int s = blockIdx.y, a0 = blockIdx.x * NB_ROWS, tid = threadIdx.x, nt = blockDim.x;
    const int ra = min(NB_ROWS, nn - a0);
    const T* G = Gu0 + (size_t)wk * gstride + (size_t)s * N * ld;
    T* out = snap0 + (size_t)wk * 2 * NW * NW + (size_t)s * NW * NW;
    extern __shared__ __align__(16) unsigned char nb_smem[];
    T* Ws = (T*)nb_smem;         // [m][PP]
    T* Ys = Ws + NW * PP;        // [m][PP]   Yraw_n
    T* Xs = Ys + NW * PP;        // [NB_ROWS][PP]
    T* Ts = Xs + NB_ROWS * PP;   // [NB_ROWS][PP]  X_blk W
    T* Gr = Ts + NB_ROWS * PP;   // [NB_ROWS][PP]  G[sn + a0 + a][sn + c]
    constexpr int CS = NW / 32;
    const int lane = tid & 31, warp = tid >> 5, nwarp = nt >> 5;
    __shared__ int sidx[NW];
    for (int q = tid; q < m; q += nt) sidx[q] = wb.idx[q];
    __syncthreads();
    const T* W = (const T*)wb.Wx + (size_t)s * NW * NW;
    // rows r of W and Yraw_n (r < m), of X_blk and of the block's own rows (r < ra) by warps,
    // columns by lanes
    for (int r = warp; r < m; r += nwarp) {
        const T* wrow = W + (size_t)r * NW;
        const T* grow = G + (long)sidx[r] * ld + sn;
        T vw[CS], vy[CS];
#pragma unroll
        for (int j = 0; j < CS; ++j) {
            const int c = lane + 32 * j;
            vw[j] = c < m ? wrow[c] : T(0);
            vy[j] = c < nn ? grow[c] : T(0);
        }
#pragma unroll
        for (int j = 0; j < CS; ++j) {
            const int c = lane + 32 * j;
            if (c < m) Ws[r * PP + c] = vw[j];
            if (c < nn) Ys[r * PP + c] = -vy[j];
        }
    }
    for (int a = warp; a < ra; a += nwarp) {
        const T* grow = G + (long)(sn + a0 + a) * ld;
        T vx[CS], vg[CS];
#pragma unroll
        for (int j = 0; j < CS; ++j) {
            const int k = lane + 32 * j;
            vx[j] = k < m ? grow[sidx[k]] : T(0);
            vg[j] = k < nn ? grow[sn + k] : T(0);
        }
#pragma unroll
        for (int j = 0; j < CS; ++j) {
            const int k = lane + 32 * j;
            if (k < m) Xs[a * PP + k] = vx[j];
            if (k < nn) Gr[a * PP + k] = vg[j];
        }
    }
    __syncthreads();
    // Ts = X_blk W: output (a, k) summed over l = part, part + 4, ... by lanes 4 g + part
    {
        const int nout = ra * m, iters = (4 * nout + nt - 1) / nt;
        for (int it = 0; it < iters; ++it) {
            const int o4 = tid + it * nt, g = o4 >> 2, part = o4 & 3;
            T acc = T(0);
            if (g < nout) {
                const int a = g / m, k = g - a * m;
                for (int l = part; l < m; l += 4) acc += Xs[a * PP + l] * Ws[l * PP + k];
            }
            acc += __shfl_xor_sync(0xffffffffu, acc, 1);
            acc += __shfl_xor_sync(0xffffffffu, acc, 2);
            if (g < nout && part == 0) Ts[(g / m) * PP + g % m] = acc;
        }
    }
    __syncthreads();
    // snap rows = G[rows, J] - Ts Yraw_n, the same split
    {
        const int nout = ra * nn, iters = (4 * nout + nt - 1) / nt;
        for (int it = 0; it < iters; ++it) {
            const int o4 = tid + it * nt, g = o4 >> 2, part = o4 & 3;
            T acc = T(0);
            int a = 0, c = 0;
            if (g < nout) {
                a = g / nn;
                c = g - a * nn;
                for (int l = part; l < m; l += 4) acc += Ts[a * PP + l] * Ys[l * PP + c];
            }
            acc += __shfl_xor_sync(0xffffffffu, acc, 1);
            acc += __shfl_xor_sync(0xffffffffu, acc, 2);
            if (g < nout && part == 0) out[(a0 + a) * NW + c] = Gr[a * PP + c] - acc;
        }
    }
}

template <typename T>
cudaError_t launch_next_block(cudaStream_t st, const T* Gu, const T* Gd, const SiteParams& sp, WindowBufs wb, int sn,
                              int nn, T* snap, Batch bt) {
    (void)Gd;
    constexpr int NW = WinCap<T>::NW;
    const size_t shm = (2 * (size_t)NW + 3 * NB_ROWS) * (NW + 1) * sizeof(T);
    {
        cudaError_t ea = ensure_smem_attr((const void*)next_block_kernel<T>, shm);
        if (ea != cudaSuccess) return ea;
    }
    count_launch();
    const int nbx = (nn + NB_ROWS - 1) / NB_ROWS;
    next_block_kernel<T><<<dim3(nbx, 2, bt.nwk), NB_THREADS, shm, st>>>(Gu, sp.ld, sp.N, wb, sn, nn, snap,
                                                                         bt.gstride);
    return cudaGetLastError();
}

// The panel gathers X = G[:, I], Yraw = E_I^T - G[I, :] and Y' = W Yraw of one window.
template <typename T>
cudaError_t launch_flush_panels(cudaStream_t sf, T* Gu, T* Gd, const SiteParams& sp, WindowBufs wb, int nw, Batch bt) {
    (void)Gd;
    constexpr int NW = WinCap<T>::NW;
    const int N = sp.N;
    count_launch();
    gather_kernel<T><<<dim3(256, 2, bt.nwk), 256, 0, sf>>>(Gu, sp.ld, N, wb, NW, bt.gstride, (long)N * sp.ld);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    GemmArgs<T> g;  // Y' = W Yraw, batch (walker, spin)
    g.M = nw; g.N = N; g.K = nw; g.Kdev = wb.m; g.kdiv = 2;
    g.A = (const T*)wb.Wx; g.lda = NW; g.sA = (long)NW * NW;
    g.B = (const T*)wb.Y; g.ldb = N; g.sB = (long)NW * N;
    g.C = (T*)wb.Y + (size_t)2 * bt.nwk * NW * N; g.ldc = N; g.sC = (long)NW * N;
    g.batch = 2 * bt.nwk;
    return gemm<T>(sf, g);
}

// G <- G - X Y' (the N x N rank-m product, after launch_flush_panels on the same stream).
template <typename T>
cudaError_t launch_flush_gemm(cudaStream_t sf, T* Gu, T* Gd, const SiteParams& sp, WindowBufs wb, int nw, Batch bt) {
    (void)Gd;
    constexpr int NW = WinCap<T>::NW;
    const int N = sp.N;
    GemmArgs<T> h;
    h.M = N; h.N = N; h.K = nw; h.Kdev = wb.m; h.kdiv = 2;
    h.A = (const T*)wb.X; h.lda = NW; h.sA = (long)N * NW;
    h.B = (const T*)wb.Y + (size_t)2 * bt.nwk * NW * N; h.ldb = N; h.sB = (long)NW * N;
    h.C = Gu; h.ldc = sp.ld; h.sC = (long)N * sp.ld;
    h.alpha = T(-1); h.beta = T(1);
    h.batch = 2 * bt.nwk;
    return gemm<T>(sf, h);
}
// ---------------------------------------------------------------------------
// T form (the paper's walker state: U_R, U_L, T = (U_L U_R)^{-1}; G = 1 - U_R T U_L)
// ---------------------------------------------------------------------------
// For every (walker, spin) z of the batch, with the window's accepted sites I (wb.idx, m = wb.m):
//   ULI[z][a][k] = UL[z][a][I_k]   (ns x m, pitch NW)      URI[z][k][a] = UR[z][I_k][a]   (m x ns, pitch ldr)
// UR: N x ns (leading dimension ldr), UL: ns x N (leading dimension N); batch strides sr, sl.
template <typename T>
__global__ void tform_gather_kernel(const T* __restrict__ UR, const T* __restrict__ UL, int N, int ns, long ldr,
                                    long sr, long sl, WindowBufs wb0, T* ULI, T* URI) {
    constexpr int NW = WinCap<T>::NW;
    const int z = blockIdx.y, wk = z >> 1;
    const WindowBufs wb = wb_walker<T>(wb0, wk, N);
    const int m = *wb.m;
    const T* ur = UR + (size_t)z * sr;
    const T* ul = UL + (size_t)z * sl;
    T* uli = ULI + (size_t)z * ns * NW;
    T* uri = URI + (size_t)z * NW * ldr;
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < m * ns; e += gridDim.x * blockDim.x) {
        const int k = e / ns, a = e - k * ns;
        const int I = wb.idx[k];
        uri[(size_t)k * ldr + a] = ur[(size_t)I * ldr + a];
        uli[(size_t)a * NW + k] = ul[(size_t)a * N + I];
    }
}

// UR[z][I_k][:] *= exp(c_s (x' - x)) = exp(2 c_s x'_k) for the accepted sites (Eq. UpdateLTRMat: the
// row of the slice's B in the right factor takes the new field), x' the field the window kernel
// left in the slice (xl, batch stride xstride per walker).
template <typename T>
__global__ void tform_scale_rows_kernel(T* UR, int N, int ns, long ldr, long sr, WindowBufs wb0, const int8_t* xl,
                                        long xstride, double c0, double c1) {
    const int z = blockIdx.y, wk = z >> 1, s = z & 1;
    const WindowBufs wb = wb_walker<T>(wb0, wk, N);
    const int m = *wb.m;
    T* ur = UR + (size_t)z * sr;
    const int8_t* x = xl + (size_t)wk * xstride;
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < m * ns; e += gridDim.x * blockDim.x) {
        const int k = e / ns, a = e - k * ns;
        const int I = wb.idx[k];
        const T f = (T)exp(2.0 * (s ? c1 : c0) * (double)x[I]);
        ur[(size_t)I * ldr + a] *= f;
    }
}

template <typename T>
cudaError_t launch_tform_gather(cudaStream_t st, const T* UR, const T* UL, int N, int ns, long ldr, long sr, long sl,
                                WindowBufs wb, T* ULI, T* URI, int nbatch) {
    count_launch();
    tform_gather_kernel<T><<<dim3(64, nbatch), 256, 0, st>>>(UR, UL, N, ns, ldr, sr, sl, wb, ULI, URI);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_tform_scale_rows(cudaStream_t st, T* UR, int N, int ns, long ldr, long sr, WindowBufs wb,
                                    const int8_t* xl, long xstride, const double* c, int nbatch) {
    count_launch();
    tform_scale_rows_kernel<T><<<dim3(64, nbatch), 256, 0, st>>>(UR, N, ns, ldr, sr, wb, xl, xstride, c[0], c[1]);
    return cudaGetLastError();
}

template cudaError_t launch_tform_gather<float>(cudaStream_t, const float*, const float*, int, int, long, long, long,
                                                WindowBufs, float*, float*, int);
template cudaError_t launch_tform_gather<double>(cudaStream_t, const double*, const double*, int, int, long, long,
                                                 long, WindowBufs, double*, double*, int);
template cudaError_t launch_tform_scale_rows<float>(cudaStream_t, float*, int, int, long, long, WindowBufs,
                                                    const int8_t*, long, const double*, int);
template cudaError_t launch_tform_scale_rows<double>(cudaStream_t, double*, int, int, long, long, WindowBufs,
                                                     const int8_t*, long, const double*, int);
template cudaError_t launch_flush_panels<float>(cudaStream_t, float*, float*, const SiteParams&, WindowBufs, int,
                                               Batch);
template cudaError_t launch_flush_panels<double>(cudaStream_t, double*, double*, const SiteParams&, WindowBufs, int,
                                                Batch);
template cudaError_t launch_flush_gemm<float>(cudaStream_t, float*, float*, const SiteParams&, WindowBufs, int, Batch);
template cudaError_t launch_flush_gemm<double>(cudaStream_t, double*, double*, const SiteParams&, WindowBufs, int,
                                              Batch);
template cudaError_t launch_next_block<float>(cudaStream_t, const float*, const float*, const SiteParams&, WindowBufs,
                                              int, int, float*, Batch);
template cudaError_t launch_next_block<double>(cudaStream_t, const double*, const double*, const SiteParams&,
                                               WindowBufs, int, int, double*, Batch);
template cudaError_t launch_flush<float>(cudaStream_t, float*, float*, const SiteParams&, WindowBufs, int);
template cudaError_t launch_flush<double>(cudaStream_t, double*, double*, const SiteParams&, WindowBufs, int);

}  // namespace afq
