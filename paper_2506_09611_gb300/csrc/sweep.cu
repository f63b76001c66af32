// sweep.cu -- the per-slice site loop of the PQMC update sweep in G form.
//
//   local   : persistent cooperative kernel, one grid barrier per site, the
//             rank-1 update G <- G - (d/r) G_{:,i} (e_i^T - G_{i,:}) applied to
//             the whole of G on every accepted flip (Eqs. DetRatiolocal,
//             UpdateLTRlocal restated for G).
//   delayed : a window of consecutive sites is decided by ONE CTA on its diagonal block of G, held in
//   blockfb   registers (FP64 block force bias: in shared memory); the accepted flips I are then applied
//             to the full G as one rank-|I| product G <- G + X Y, the buffered sum of the paper's delayed
//             vectors (Eqs. DelayTMat00, DelayRgenk, FinalDelay) and the block force-bias upgrade
//             (Eq. BlkFrcBsTnew2): the columns of X and rows of Y follow from G[:, I] and G[I, :] by a
//             recursion over the accepts.
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

// The same update with the own rows of G in registers for the whole slice (FP32, N <= 1672 on 152 SMs): thread (g, v)
// holds the 16-byte column vector v of the rows g, g + ng, ... of both spins, RPT rows at most.  An accept
// then moves two rows instead of all of G: the other CTAs need row b only, and its owner cannot know b before
// the grid barrier that fixes it, so with its update every CTA publishes its rows among the next LR_AHEAD
// sites (double-buffered by phase); the rare accept beyond them costs a second barrier.  The arithmetic is
// local_kernel's, element by element.  Bound by the barrier and the round trips to L2 (diagonal, row b):
// 40 x 40, a pass of four slices and two recomputes: 62 ms with G in L2 (9.75 ms of it a slice), 43 ms so.
constexpr int LR_THREADS = 448, LR_AHEAD = 4, LR_RPT_MAX = 11;
inline size_t local_reg_pub(long ld) { return 2 * (size_t)(LR_AHEAD + 1) * 2 * ld; }  // floats of the row buffer

template <int RPT>
__global__ void __launch_bounds__(LR_THREADS, 1) local_reg_kernel(float* Gu, float* Gd, int8_t* xl_g, const double* u,
                                                                  const uint8_t* replay, SiteParams sp, SliceOut so,
                                                                  float* diag, float* pub, GridBar* bar, int* err) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int N = sp.N;
    const long ld = sp.ld;
    const int nblk = gridDim.x, b = blockIdx.x, tid = threadIdx.x, nt = LR_THREADS;
    const int r0 = (int)((long)N * b / nblk), r1 = (int)((long)N * (b + 1) / nblk), nr = r1 - r0;
    const int nv = (N + 3) / 4, ng = nt / nv, g = tid / nv, v = tid - g * nv;
    const bool mine = g < ng;
    double* us = (double*)smem_raw;
    int8_t* xs = (int8_t*)(us + N);
    uint8_t* rp = (uint8_t*)(xs + N);
    __shared__ float colb[2][32];  // G_s[r, b] of the own rows
    __shared__ int s_b, s_nneg;
    __shared__ float s_f[2];
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
    float4 G0[RPT], G1[RPT];
#pragma unroll
    for (int i = 0; i < RPT; ++i) {
        const int r = g + ng * i;
        const bool in = mine && r < nr;
        G0[i] = in ? *(const float4*)(Gu + (long)(r0 + r) * ld + 4 * v) : make_float4(0.f, 0.f, 0.f, 0.f);
        G1[i] = in ? *(const float4*)(Gd + (long)(r0 + r) * ld + 4 * v) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    for (int e = tid; e < 2 * nr; e += nt) {  // diagonals of the own rows into buffer 0
        const int s = e >= nr ? 1 : 0, r = r0 + e - s * nr;
        diag[(0 * 2 + s) * N + r] = (s ? Gd : Gu)[(long)r * ld + r];
    }
    // own rows among the sites [p, p + LR_AHEAD) (slot: site - p) to buffer par; or site p alone to slot
    // LR_AHEAD
    auto publish = [&](int p, int par, bool one) {
        if (!mine) return;
#pragma unroll
        for (int i = 0; i < RPT; ++i) {
            const int r = g + ng * i, w = r0 + r - p;
            if (r < nr && w >= 0 && w < (one ? 1 : LR_AHEAD)) {
                float* o = pub + (size_t)((par * (LR_AHEAD + 1) + (one ? LR_AHEAD : w)) * 2) * ld + 4 * v;
                *(float4*)o = G0[i];
                *(float4*)(o + ld) = G1[i];
            }
        }
    };
    publish(0, 0, false);
    unsigned int* ctr = &bar->count;
    unsigned int nbar = 0;  // grid barriers passed (thread 0)
    const float df00 = (float)sp.dflip[0][0], df01 = (float)sp.dflip[0][1], df10 = (float)sp.dflip[1][0],
                df11 = (float)sp.dflip[1][1], sf0 = (float)sp.sflip[0], sf1 = (float)sp.sflip[1];
    int n_acc = 0, p = 0, base = 0;  // p: next site to test (warp 0); base: first published site
    int cur = 0;                     // diagonal and row buffer of this phase
    __syncthreads();
    for (;;) {
        if (tid < 32) {  // grid barrier (thread 0), then the scan for the next accept, as in local_kernel
            int ok = 1;
            if (tid == 0) ok = grid_arrive_wait(ctr, (++nbar) * (unsigned int)nblk, err) ? 1 : 0;
            __syncwarp();
            ok = __shfl_sync(0xffffffffu, ok, 0);
            int bsel = ok ? N : -1;
            const float* d0 = diag + (cur * 2 + 0) * N;
            const float* d1 = diag + (cur * 2 + 1) * N;
            while (ok && p < N) {
                const int q = p + tid;
                bool acc = false;
                float R = 0.f, rr0 = 1.f, rr1 = 1.f, del0 = df00, del1 = df10;
                if (q < N) {
                    const int xi = xs[q] > 0 ? 0 : 1;
                    del0 = xi ? df01 : df00;
                    del1 = xi ? df11 : df10;
                    rr0 = 1.f + del0 * (1.f - __ldcg(d0 + q));
                    rr1 = 1.f + del1 * (1.f - __ldcg(d1 + q));
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
                        if (R < 0.f) s_nneg += 1;
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
        if (bs >= N) break;
        ++n_acc;
        int slot = bs - base;
        if (slot >= LR_AHEAD) {  // not published (the same in every CTA): its owner does so now
            slot = LR_AHEAD;
            publish(bs, cur, true);
            __syncthreads();
            if (tid == 0 && !grid_arrive_wait(ctr, (++nbar) * (unsigned int)nblk, err)) s_b = -1;
            __syncthreads();
            if (s_b < 0) return;
        }
        const float* row = pub + (size_t)((cur * (LR_AHEAD + 1) + slot) * 2) * ld;  // row b, both spins (past L1)
        float4 rv0 = make_float4(0.f, 0.f, 0.f, 0.f), rv1 = rv0;
        if (mine) {
            rv0 = __ldcg((const float4*)(row + 4 * v));
            rv1 = __ldcg((const float4*)(row + ld + 4 * v));
        }
        float dnew = 0.f, drow = 0.f;  // the own diagonals: one element per thread
        const int ds = tid >= nr ? 1 : 0, dr = tid - ds * nr;
        if (tid < 2 * nr) {
            dnew = __ldcg(diag + (cur * 2 + ds) * N + r0 + dr);
            drow = (r0 + dr == bs ? 1.f : 0.f) - __ldcg(row + ds * ld + r0 + dr);
        }
        if (mine && v == bs >> 2) {  // column b of the own rows
            const int k = bs & 3;
#pragma unroll
            for (int i = 0; i < RPT; ++i) {
                const int r = g + ng * i;
                if (r < nr) {
                    colb[0][r] = k == 0 ? G0[i].x : k == 1 ? G0[i].y : k == 2 ? G0[i].z : G0[i].w;
                    colb[1][r] = k == 0 ? G1[i].x : k == 1 ? G1[i].y : k == 2 ? G1[i].z : G1[i].w;
                }
            }
        }
        __syncthreads();
        // e_b^T - G[b, :], zero beyond N
        const int c0 = 4 * v;
        rv0.x = c0 < N ? (c0 == bs ? 1.f : 0.f) - rv0.x : 0.f;
        rv0.y = c0 + 1 < N ? (c0 + 1 == bs ? 1.f : 0.f) - rv0.y : 0.f;
        rv0.z = c0 + 2 < N ? (c0 + 2 == bs ? 1.f : 0.f) - rv0.z : 0.f;
        rv0.w = c0 + 3 < N ? (c0 + 3 == bs ? 1.f : 0.f) - rv0.w : 0.f;
        rv1.x = c0 < N ? (c0 == bs ? 1.f : 0.f) - rv1.x : 0.f;
        rv1.y = c0 + 1 < N ? (c0 + 1 == bs ? 1.f : 0.f) - rv1.y : 0.f;
        rv1.z = c0 + 2 < N ? (c0 + 2 == bs ? 1.f : 0.f) - rv1.z : 0.f;
        rv1.w = c0 + 3 < N ? (c0 + 3 == bs ? 1.f : 0.f) - rv1.w : 0.f;
        const float nf0 = -s_f[0], nf1 = -s_f[1];
#pragma unroll
        for (int i = 0; i < RPT; ++i) {
            const int r = g + ng * i;
            if (mine && r < nr) {
                vfma_rank1<float>(G0[i], nf0 * colb[0][r], rv0);
                vfma_rank1<float>(G1[i], nf1 * colb[1][r], rv1);
            }
        }
        if (tid < 2 * nr)
            diag[((cur ^ 1) * 2 + ds) * N + r0 + dr] = fma((ds ? nf1 : nf0) * colb[ds][dr], drow, dnew);
        base = bs + 1;
        cur ^= 1;
        publish(base, cur, false);
        __syncthreads();  // every write of the CTA precedes thread 0's arrival at the next barrier
    }
    if (mine) {
#pragma unroll
        for (int i = 0; i < RPT; ++i) {
            const int r = g + ng * i;
            if (r < nr) {
                *(float4*)(Gu + (long)(r0 + r) * ld + 4 * v) = G0[i];
                *(float4*)(Gd + (long)(r0 + r) * ld + 4 * v) = G1[i];
            }
        }
    }
    if (b == 0 && tid == 0) {
        if (so.sign && (s_nneg & 1)) *so.sign = -*so.sign;
        so.stats[0] += N;
        so.stats[1] += n_acc;
        so.stats[2] += n_acc;
        *so.maxr = fmax(*so.maxr, s_maxr);
    }
}

template <int RPT>
static cudaError_t launch_local_reg(cudaStream_t st, float* Gu, float* Gd, int8_t* xl, const double* u,
                                    const uint8_t* replay, const SiteParams& sp, SliceOut so, float* diag, float* pub,
                                    GridBar* bar, int* err, int nblk) {
    const size_t shm = (size_t)sp.N * (sizeof(double) + 2);
    SiteParams spc = sp;
    void* args[] = {&Gu, &Gd, &xl, &u, &replay, &spc, &so, &diag, &pub, &bar, &err};
    count_launch();
    return cudaLaunchCooperativeKernel((void*)local_reg_kernel<RPT>, dim3(nblk), dim3(LR_THREADS), args, shm, st);
}

size_t local_rowbuf_elems(long ld) { return local_reg_pub(ld); }

// Grid size: at most max_blocks CTAs (one per SM) and at least one row each.
template <typename T>
cudaError_t launch_local(cudaStream_t st, T* Gu, T* Gd, int8_t* xl, const double* u, const uint8_t* replay,
                         const SiteParams& sp, SliceOut so, T* colbuf, T* rowbuf, GridBar* bar, int* err,
                         int max_blocks) {
    const int nblk = max_blocks < sp.N ? max_blocks : sp.N;
    if (nblk < 1) return cudaErrorInvalidValue;
    const int nrmax = (sp.N + nblk - 1) / nblk;
    if constexpr (sizeof(T) == 4) {  // the own rows in registers, where they fit
        const int nv = (sp.N + 3) / 4, ng = nv <= LR_THREADS ? LR_THREADS / nv : 0;
        const int rpt = ng > 0 && nrmax <= 32 ? (nrmax + ng - 1) / ng : LR_RPT_MAX + 1;
        if (rpt <= 3) return launch_local_reg<3>(st, Gu, Gd, xl, u, replay, sp, so, colbuf, rowbuf, bar, err, nblk);
        if (rpt <= 6) return launch_local_reg<6>(st, Gu, Gd, xl, u, replay, sp, so, colbuf, rowbuf, bar, err, nblk);
        if (rpt <= LR_RPT_MAX)
            return launch_local_reg<LR_RPT_MAX>(st, Gu, Gd, xl, u, replay, sp, so, colbuf, rowbuf, bar, err, nblk);
    }
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
constexpr int WIN_THREADS = 1024;

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
    wb.Y = (T*)wb.Y + (size_t)j * 2 * NW * N;
    return wb;
}

static size_t window_smem(int n) {
    size_t P = (size_t)n + 1;
    size_t g = 2 * (size_t)n * P * sizeof(double);  // Gs[2][n][n+1]
    size_t s1 = 2 * (size_t)NBMAX * (NBMAX + 1) * sizeof(double);
    size_t vec = 2 * (size_t)n * sizeof(double) + 2 * (size_t)NBMAX * sizeof(double);  // staging vectors
    size_t misc = (size_t)n * (sizeof(int) + 1) + 2 * (size_t)NBMAX * sizeof(double) + 256;
    return g + s1 + vec + misc;
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

// The window's accepts in sequential form, for panel_kernel: accept k at position a_k of the window with
// factor f_k = -Delta_k / r_k leaves the row and column of the block as they were at that moment,
//   Wx[s][k][c] = G[a_k][c] (c > a_k),  Wm[s][k][r] = -f_k G[r][a_k] (r > a_k),  both -f_k at a_k
// (pitch NW; entries before a_k are never read).  Here from the block's frozen rows and columns.
template <typename T>
__device__ __forceinline__ void window_export(const T* Gs, int n, int P, const int* idx,
                                              const T (*fk)[WinCap<T>::NW], int m, T* Wx, T* Wm, int tid) {
    constexpr int NW = WinCap<T>::NW;
    for (int row = tid >> 5; row < 2 * m; row += WIN_THREADS / 32) {
        const int s = row >= m ? 1 : 0, k = row - s * m, a = idx[k];
        const T* Gb = Gs + (size_t)s * n * P;
        const T nf = -fk[s][k];
        const size_t o = ((size_t)s * NW + k) * NW;
        for (int c = a + (tid & 31); c < n; c += 32) {
            Wx[o + c] = c == a ? nf : Gb[a * P + c];
            Wm[o + c] = c == a ? nf : nf * Gb[c * P + a];
        }
    }
}

// Field-change constants in the bulk precision (SiteParams holds them in FP64).
template <typename T>
struct FlipConsts {
    T dflip[2][2], sflip[2];
};

// Warps and register tile of window_reg_kernel for windows of up to NP sites.  Warp 0 decides, TW tile warps
// hold the block (RG row groups x 8 column groups of threads per spin, a thread rows rg + RG i and columns
// cg + 8 j), one warp exports the accepts.  Up to 64 sites warps 4, 8, ... exit at once, so the deciding
// warp has its SM partition to itself (with 128 sites their registers are needed).
template <typename T, int NP>
struct WinTile {
    static constexpr int TW = 8, WPS = TW / 2;
    static constexpr int RG = 4 * WPS, TR = NP / RG, TC = NP / 8, NJ = NP / 32;
    static constexpr bool IDLE = NP <= 64;
    static constexpr int ACTIVE = 32 * (TW + 2);                              // threads at the barriers
    static constexpr int THREADS = ACTIVE + (IDLE ? 32 * ((TW + 1) / 3) : 0);  // with the exiting warps
};

// One window of the delayed update (AFQMC_MODE_DELAYED) or of the constrained-path heat bath
// (WIN_MODE_CP), one block per walker.
//
// The n x n block of both spins (n <= NP) lives in the registers of the tile warps.  Per accept a, two
// barriers: the deciding warp names a; the threads that hold row a and column a put them into shared memory
// (double-buffered by accept parity); every tile thread applies G[r][c] += (-f G[r][a]) G[a][c] to its
// elements while the deciding warp goes on from the same two vectors and the export warp writes them out for
// panel_kernel.  Rows and columns at or before a are never looked at again.
//
// Decisions: lane l keeps 1 - G[q][q] of both spins, the uniform, the field and the ratio of the sites
// q = l + 32 j, and tests 32 sites at a time; a ballot finds the next accept (a rejection leaves G unchanged).
//   Metropolis: R = s(-x)/s(x) r_up r_dn, r_s = 1 + Delta_s (1 - G_s[q][q]), accept iff u < |R|.
//   Constrained-path heat bath (Sec. IV.D, Eq. ptilde): lambda(x) = p(x) s(x) r_up(x) r_dn(x), negative
//   lambda clamped to zero, x = +1 iff u (lambda(+1) + lambda(-1)) < lambda(+1); the walker is removed when
//   both vanish; every site is an accept.
//
// Bound by the latency of the accept chain, one warp's instruction stream: roles are split over warps so
// that each has little to issue per accept.
template <typename T, int MODE, int NP>
__global__ void __launch_bounds__(WinTile<T, NP>::THREADS) window_reg_kernel(
    const T* __restrict__ Gu0, int8_t* xl0, const double* __restrict__ u0, const uint8_t* __restrict__ replay0,
    int N, long ld, FlipConsts<T> fc, SliceOut so0, int s0, int n, WindowBufs wb0, const T* __restrict__ blk0,
    int* err, Batch bt) {
    using W = WinTile<T, NP>;
    constexpr int NW = WinCap<T>::NW, RG = W::RG, TR = W::TR, TC = W::TC, NJ = W::NJ;
    constexpr unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31, hw = __shfl_sync(FULL, threadIdx.x >> 5, 0), wk = blockIdx.x;
    if (W::IDLE && hw > 0 && (hw & 3) == 0) return;
    const int warp = W::IDLE ? hw - 1 - hw / 4 : hw - 1;  // -1: decides, < TW: tile, TW: export
    auto block_sync = [&] {
        __syncwarp();  // the barrier counts whole warps
        named_barrier_sync(1, W::ACTIVE);
    };
    const WindowBufs wb = wb_walker<T>(wb0, wk, N);
    const T* G = Gu0 + (size_t)wk * bt.gstride;
    const T* src0 = blk0 ? blk0 + (size_t)wk * 2 * NW * NW : G + (size_t)s0 * ld + s0;  // the block, spin up
    const T* src1 = blk0 ? src0 + NW * NW : src0 + (size_t)N * ld;
    const long lds = blk0 ? NW : ld;
    __shared__ T srow[2][2][NP], scol[2][2][NP];  // [accept parity][spin]: G[a][:], G[:, a]
    __shared__ T s_f[2][2];                       // [accept parity][spin]: f = -Delta / r
    __shared__ int s_a[2];                        // [accept parity]: the accept, -1 at the end

    if (warp >= 0 && warp < W::TW) {  // ---- tile warps ----
        const int s = warp >= W::WPS ? 1 : 0, rg = (warp - s * W::WPS) * 4 + (lane >> 3), cg = lane & 7;
        const T* sp = s ? src1 : src0;
        T g[TR][TC];
#pragma unroll
        for (int i = 0; i < TR; ++i)
#pragma unroll
            for (int j = 0; j < TC; ++j) {
                const int r = rg + RG * i, c = cg + 8 * j;
                g[i][j] = (r < n && c < n) ? sp[r * lds + c] : T(0);
            }
        for (int par = 0;; par ^= 1) {
            block_sync();
            const int a = s_a[par];
            if (a < 0) return;
            if (rg == (a & (RG - 1))) {
#pragma unroll
                for (int j = 0; j < TC; ++j) {
                    T t[TR];
#pragma unroll
                    for (int i = 0; i < TR; ++i) t[i] = g[i][j];
                    srow[par][s][cg + 8 * j] = reg_pick<T, TR>(t, a / RG);
                }
            }
            if (cg == (a & 7)) {
#pragma unroll
                for (int i = 0; i < TR; ++i) {
                    T t[TC];
#pragma unroll
                    for (int j = 0; j < TC; ++j) t[j] = g[i][j];
                    scol[par][s][rg + RG * i] = reg_pick<T, TC>(t, a >> 3);
                }
            }
            block_sync();
            const T nf = -s_f[par][s];
            T rv[TC];
#pragma unroll
            for (int j = 0; j < TC; ++j) rv[j] = srow[par][s][cg + 8 * j];
#pragma unroll
            for (int i = 0; i < TR; ++i) {
                // an FP64 or 128-site update is bound by its multiply-adds: rows (and columns) at or before
                // a in every thread are left out
                if ((sizeof(T) == 8 || NP > 64) && RG * i + RG - 1 <= a) continue;
                const T wv = nf * scol[par][s][rg + RG * i];
#pragma unroll
                for (int j = 0; j < TC; ++j) {
                    if (sizeof(T) == 8 && 8 * j + 7 <= a) continue;
                    g[i][j] = fma(wv, rv[j], g[i][j]);
                }
            }
        }
    }
    if (warp == W::TW) {  // ---- export warp: row a and -f column a of accept m, -f at position a ----
        for (int m = 0;; ++m) {
            const int par = m & 1;
            block_sync();
            const int a = s_a[par];
            if (a < 0) return;
            block_sync();
            if (lane == 0) wb.idx[m] = s0 + a;
#pragma unroll
            for (int s = 0; s < 2; ++s) {
                const T nf = -s_f[par][s];
                T* wx = (T*)wb.Wx + ((size_t)s * NW + m) * NW;
                T* wm = (T*)wb.Wm + ((size_t)s * NW + m) * NW;
#pragma unroll
                for (int j = 0; j < NJ; ++j) {
                    const int q = lane + 32 * j;
                    wx[q] = q == a ? nf : srow[par][s][q];
                    wm[q] = q == a ? nf : nf * scol[par][s][q];
                }
            }
        }
    }
    // ---- deciding warp ----
    int8_t* xl = xl0 + (size_t)wk * bt.xstride + s0;
    const double* u = u0 + (size_t)wk * 2 * N + s0;
    const uint8_t* rep = replay0 ? replay0 + (size_t)wk * 2 * N + s0 : nullptr;
    const SliceOut so = so_walker(so0, wk, N);
    const bool forced = rep != nullptr;
    T b0[NJ], b1[NJ], ul[NJ], rat[NJ], det[NJ];  // 1 - G[q][q] up and down, uniform, ratio (norm), r_up r_dn
    int xs[NJ];
    unsigned repm[NJ], accm[NJ], upm[NJ], valid[NJ];  // lane masks: forced, accepted, x = +1 drawn, q < n
#pragma unroll
    for (int j = 0; j < NJ; ++j) {
        const int q = lane + 32 * j;
        const bool in = q < n;
        b0[j] = in ? T(1) - src0[q * lds + q] : T(0);
        b1[j] = in ? T(1) - src1[q * lds + q] : T(0);
        ul[j] = in ? (T)u[q] : T(0);
        xs[j] = in ? xl[q] : 1;
        valid[j] = __ballot_sync(FULL, in);
        repm[j] = __ballot_sync(FULL, in && forced && rep[q] != 0);
        accm[j] = upm[j] = 0u;
        rat[j] = det[j] = T(0);
    }
    bool dead = MODE == WIN_MODE_CP && so.cp && so.cp[2] != 0.0;
    int m = 0;
#pragma unroll
    for (int j = 0; j < NJ; ++j) {
        // field-change constants of this chunk's sites (Metropolis)
        const bool xp = xs[j] > 0;
        const T x0 = xp ? fc.dflip[0][0] : fc.dflip[0][1], x1 = xp ? fc.dflip[1][0] : fc.dflip[1][1];
        const T sf = xp ? fc.sflip[0] : fc.sflip[1];
        unsigned open = dead ? 0u : valid[j];  // sites of the chunk not decided yet
        while (open) {
            T e0 = x0, e1 = x1, r0, r1, R;
            unsigned ball;
            if (MODE == WIN_MODE_CP) {
                const T p0 = T(1) + fc.dflip[0][0] * b0[j], p1 = T(1) + fc.dflip[1][0] * b1[j];
                const T m0 = T(1) + fc.dflip[0][1] * b0[j], m1 = T(1) + fc.dflip[1][1] * b1[j];
                const T lp = fmax(fc.sflip[0] * p0 * p1, T(0)), lm = fmax(fc.sflip[1] * m0 * m1, T(0));
                R = lp + lm;
                const bool up = forced ? ((repm[j] >> lane) & 1u) != 0 : ul[j] * R < lp;
                r0 = up ? p0 : m0;
                r1 = up ? p1 : m1;
                e0 = up ? fc.dflip[0][0] : fc.dflip[0][1];
                e1 = up ? fc.dflip[1][0] : fc.dflip[1][1];
                const unsigned site = open & (0u - open);  // one site at a time
                ball = __ballot_sync(FULL, R > T(0) && isfinite(R)) & site;
                upm[j] |= __ballot_sync(FULL, up) & ball;
                if ((site >> lane) & 1u) {
                    rat[j] = R;
                    det[j] = r0 * r1;
                }
                if (!ball) {
                    dead = true;
                    break;
                }
            } else {
                r0 = T(1) + e0 * b0[j];
                r1 = T(1) + e1 * b1[j];
                R = sf * r0 * r1;
                const bool want = forced ? ((repm[j] >> lane) & 1u) != 0 : ul[j] < fabs(R);
                ball = __ballot_sync(FULL, want && isfinite(R)) & open;  // never on a ratio that is not finite
            }
            // sites before the first accept are rejected; it and they are decided now
            const unsigned bit = ball & (0u - ball), done = ball ? open & (bit | (bit - 1u)) : open;
            if (MODE != WIN_MODE_CP && ((done >> lane) & 1u)) rat[j] = R;
            open &= ~done;
            if (!ball) break;
            accm[j] |= bit;
            const int first = __ffs(ball) - 1, par = m & 1;
            T f0, f1;
            if (sizeof(T) == 4) {  // every lane's factors, under the ballot's latency
                const T q0 = -fast_quot(e0, r0), q1 = -fast_quot(e1, r1);
                if (lane == first) {
                    s_a[par] = 32 * j + first;
                    s_f[par][0] = q0;
                    s_f[par][1] = q1;
                }
                block_sync();
                f0 = __shfl_sync(FULL, q0, first);
                f1 = __shfl_sync(FULL, q1, first);
            } else {  // one quotient for both spins while the tile warps store: even lanes up, odd lanes down
                if (lane == 0) s_a[par] = 32 * j + first;
                block_sync();
                const T n0 = __shfl_sync(FULL, e0, first), n1 = __shfl_sync(FULL, e1, first);
                const T d0 = __shfl_sync(FULL, r0, first), d1 = __shfl_sync(FULL, r1, first);
                const T fq = -fast_quot((lane & 1) ? n1 : n0, (lane & 1) ? d1 : d0);
                if (lane < 2) s_f[par][lane] = fq;
                f0 = __shfl_sync(FULL, fq, 0);
                f1 = __shfl_sync(FULL, fq, 1);
            }
            block_sync();
#pragma unroll
            for (int i = j; i < NJ; ++i) {
                const int q = lane + 32 * i;
                b0[i] = fma(f0 * scol[par][0][q], srow[par][0][q], b0[i]);
                b1[i] = fma(f1 * scol[par][1][q], srow[par][1][q], b1[i]);
            }
            ++m;
        }
    }
    if (lane == 0) s_a[m & 1] = -1;
    block_sync();
    // decisions, ratios, fields and the walker's sums
    double c0 = 0.0, c1 = 0.0;
    int nneg = 0;
    T maxr = T(0);
    bool bad = false;
#pragma unroll
    for (int j = 0; j < NJ; ++j) {
        const int q = lane + 32 * j;
        const bool acc = ((accm[j] >> lane) & 1u) != 0, up = ((upm[j] >> lane) & 1u) != 0;
        if (q < n) {
            so.dec[s0 + q] = MODE == WIN_MODE_CP ? up : acc;
            so.ratio[s0 + q] = (double)rat[j];
            bad = bad || !isfinite(rat[j]);
            if (acc) {
                xl[q] = (int8_t)(MODE == WIN_MODE_CP ? (up ? 1 : -1) : -xs[j]);
                if (MODE == WIN_MODE_CP) {
                    c0 += log((double)rat[j]);
                    c1 += log(fabs((double)det[j]));
                } else {
                    if (rat[j] < T(0)) ++nneg;
                    maxr = fmax(maxr, fabs(rat[j]));
                }
            }
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        nneg += __shfl_xor_sync(FULL, nneg, o);
        maxr = fmax(maxr, __shfl_xor_sync(FULL, maxr, o));
        if (MODE == WIN_MODE_CP) {
            c0 += __shfl_xor_sync(FULL, c0, o);
            c1 += __shfl_xor_sync(FULL, c1, o);
        }
    }
    bad = __any_sync(FULL, bad);
    if (lane == 0) {
        *wb.m = m;
        if (bad) set_err(err, DEV_NUMERIC);
        if (so.sign && (nneg & 1)) *so.sign = -*so.sign;
        if (MODE == WIN_MODE_CP && so.cp) {
            so.cp[0] += c0;
            so.cp[1] += c1;
            if (dead) so.cp[2] = 1.0;
        }
        so.stats[0] += n;
        so.stats[1] += m;
        so.stats[2] += m;
        so.stats[3] += (m > 0) ? 1 : 0;
        *so.maxr = fmax(*so.maxr, (double)maxr);
    }
}

// One window of the block force-bias update (Sec. III.B) in FP32, blocks of nb <= NBP sites, one block per
// walker.  Warps 0 and 1 decide (one spin each), eight tile warps hold the window's block in registers as in
// window_reg_kernel.  Per block of sites S:
//   the tile threads put the S x S diagonal block of both spins into shared memory;
//   each deciding warp strips the fields (Eq. BlkFrcBsTnew1) on its spin's block in registers, lane r holding
//   row r: one rank-1 step per site, the registers rotating by one column a step so that the loop is not
//   unrolled; warp 0 proposes from the stripped densities (FP64, as the ratio); each warp takes
//   det(1 + D_F A_FF) as the product of the sequential rank-1 ratios on its block (Eq. BlkFrcBsTnew2);
//   warp 0 accepts or rejects;
//   the accepted flips go through the tile one by one, one block barrier each, the deciding warps writing the
//   rows and columns out for panel_kernel.
// Bound by the latency of that chain: 16 strip steps and about as many ratio steps of one warp per block.
// The FP64 update spreads its multiply-adds over 32 warps instead (window_kernel).
template <int NBP>
__global__ void __launch_bounds__(320) window_fb_kernel(const float* __restrict__ Gu0, int8_t* xl0,
                                                        const double* __restrict__ u0,
                                                        const uint8_t* __restrict__ replay0, SiteParams sp,
                                                        FlipConsts<float> fc, FlipConsts<float> fstrip, SliceOut so0,
                                                        int s0, int n, int nb, WindowBufs wb0,
                                                        const float* __restrict__ blk0, int* err, Batch bt) {
    constexpr int NP = 64, NW = WinCap<float>::NW, RG = 16, TR = 4, TC = 8;
    constexpr unsigned FULL = 0xffffffffu;
    const int tid = threadIdx.x, lane = tid & 31, hw = __shfl_sync(FULL, tid >> 5, 0), wk = blockIdx.x, N = sp.N;
    const WindowBufs wb = wb_walker<float>(wb0, wk, N);
    const float* G = Gu0 + (size_t)wk * bt.gstride;
    const float* src0 = blk0 ? blk0 + (size_t)wk * 2 * NW * NW : G + (size_t)s0 * sp.ld + s0;
    const float* src1 = blk0 ? src0 + NW * NW : src0 + (size_t)N * sp.ld;
    const long lds = blk0 ? NW : sp.ld;
    __shared__ float S1[2][NBP][NBP + 1];           // the current block's S x S of both spins
    __shared__ float srow[2][2][NP], scol[2][2][NP];  // [flip parity][spin]
    __shared__ float s_phi[2][NBP];                 // Delta / r of the flips, in order
    __shared__ float s_diag[2][NBP];                // stripped diagonal
    __shared__ double s_prod[2], s_E[NP];           // ratio products; e^{lm - lp} of every site
    __shared__ unsigned s_flip;                     // proposed flips of the block (lane mask)
    __shared__ int s_acc;

    if (hw >= 2) {  // ---- tile warps ----
        const int w = hw - 2, s = w >> 2, rg = (w & 3) * 4 + (lane >> 3), cg = lane & 7;
        const float* srcp = s ? src1 : src0;
        float g[TR][TC];
#pragma unroll
        for (int i = 0; i < TR; ++i)
#pragma unroll
            for (int j = 0; j < TC; ++j) {
                const int r = rg + RG * i, c = cg + 8 * j;
                g[i][j] = (r < n && c < n) ? srcp[r * lds + c] : 0.f;
            }
        int par = 0;
        for (int p0 = 0; p0 < n; p0 += nb) {
            const int nbk = min(nb, n - p0);
#pragma unroll
            for (int i = 0; i < TR; ++i)
#pragma unroll
                for (int j = 0; j < TC; ++j) {
                    const int r = rg + RG * i - p0, c = cg + 8 * j - p0;
                    if (r >= 0 && r < nbk && c >= 0 && c < nbk) S1[s][r][c] = g[i][j];
                }
            __syncthreads();
            __syncthreads();
            if (!s_acc) continue;
            int q = 0;
            for (unsigned fl = s_flip; fl; fl &= fl - 1, ++q, par ^= 1) {
                const int a = p0 + __ffs(fl) - 1;
                if (rg == (a & (RG - 1))) {
#pragma unroll
                    for (int j = 0; j < TC; ++j) {
                        float t[TR];
#pragma unroll
                        for (int i = 0; i < TR; ++i) t[i] = g[i][j];
                        srow[par][s][cg + 8 * j] = reg_pick<float, TR>(t, a / RG);
                    }
                }
                if (cg == (a & 7)) {
#pragma unroll
                    for (int i = 0; i < TR; ++i) {
                        float t[TC];
#pragma unroll
                        for (int j = 0; j < TC; ++j) t[j] = g[i][j];
                        scol[par][s][rg + RG * i] = reg_pick<float, TC>(t, a >> 3);
                    }
                }
                __syncthreads();
                const float phi = s_phi[s][q];
                float rv[TC];
#pragma unroll
                for (int j = 0; j < TC; ++j) rv[j] = srow[par][s][cg + 8 * j];
#pragma unroll
                for (int i = 0; i < TR; ++i) {
                    const float wv = phi * scol[par][s][rg + RG * i];
#pragma unroll
                    for (int j = 0; j < TC; ++j) g[i][j] = fmaf(wv, rv[j], g[i][j]);
                }
            }
        }
        return;
    }
    // ---- deciding warps: spin hw ----
    const int s = hw;
    int8_t* xl = xl0 + (size_t)wk * bt.xstride + s0;
    const double* u = u0 + (size_t)wk * 2 * N;
    const uint8_t* rep = replay0 ? replay0 + (size_t)wk * 2 * N : nullptr;
    const SliceOut so = so_walker(so0, wk, N);
    auto pair_sync = [&] {
        __syncwarp();
        named_barrier_sync(2, 64);
    };
    float* Wx = (float*)wb.Wx + (size_t)s * NW * NW;
    float* Wm = (float*)wb.Wm + (size_t)s * NW * NW;
    int m = 0, n_prop = 0, n_acc = 0, nneg = 0, par = 0;
    double maxr = 0.0;
    bool bad = false;
    for (int p0 = 0; p0 < n; p0 += nb) {
        const int nbk = min(nb, n - p0), i = s0 + p0 + lane, blk = (s0 + p0) / nb;
        const bool in = lane < nbk;
        const int x = in ? xl[p0 + lane] : 1;
        const double uq = in ? u[i] : 0.0, ua = u[N + blk];
        const bool forced = rep && in && rep[i] != 0, force_acc = rep && rep[N + blk] != 0;
        const unsigned xup = __ballot_sync(FULL, x > 0);
        __syncthreads();  // S1 is there
        float g[NBP];
        // (a) stripped force bias: G <- G - (d/r) G[:, a] (e_a^T - G[a, :]) for every site a of the block,
        //     d = exp(-c x_a) - 1; g[j] is column (a + j) mod NBP before step a.  As many steps as the block
        //     has sites: with all NBP of them one-site blocks at 40 x 40 took 55.3 ms a pass, so 31.7 ms.
#pragma unroll
        for (int j = 0; j < NBP; ++j) g[j] = (in && j < nbk) ? S1[s][lane][j] : 0.f;
#pragma unroll 1
        for (int a = 0; a < nbk; ++a) {
            const float db = (xup >> a) & 1u ? fstrip.dflip[s][0] : fstrip.dflip[s][1];
            const float r0 = __shfl_sync(FULL, g[0], a);
            const float rr = 1.f + db * (1.f - r0);
            const float f = fast_quot(db, rr) * g[0];
            const float first = g[0] - f * (1.f - r0);
#pragma unroll
            for (int j = 1; j < NBP; ++j) g[j - 1] = fmaf(f, __shfl_sync(FULL, g[j], a), g[j]);
            g[NBP - 1] = first;
        }
        {
            float t[NBP];
#pragma unroll
            for (int j = 0; j < NBP; ++j) t[j] = g[j];
            const float dgv = reg_pick<float, NBP>(t, (lane - nbk) & (NBP - 1));
            if (lane < NBP) s_diag[s][lane] = dgv;
        }
        pair_sync();
        // (b) proposals from lambda(x') = bbar(x') / sum bbar, bbar(x) = s(x) e^{x h}: x' = +1 iff
        //     u < 1 / (1 + E), E = e^{lm - lp}; a flip to x' carries e^{(x - x') h}
        double fac = 1.0;
        if (s == 0) {
            bool flip = false;
            if (in) {
                const double h = sp.c[0] * (1.0 - (double)s_diag[0][lane]) + sp.c[1] * (1.0 - (double)s_diag[1][lane]);
                const double E = exp((hs_log_scalar(sp, -1) - h) - (hs_log_scalar(sp, +1) + h));
                const int xp = rep ? (forced ? 1 : -1) : (uq * (1.0 + E) < 1.0 ? 1 : -1);
                s_E[p0 + lane] = E;
                so.dec[i] = xp > 0 ? 1 : 0;
                flip = xp != x;
                if (flip) {
                    fac = E * sp.sflip[1];  // e^{-2h}: sflip[1] = s(+1)/s(-1) takes the scalar back out
                    if (xp < 0) fac = fast_quot(1.0, fac);
                }
            }
            const unsigned fl = __ballot_sync(FULL, flip);
            if (lane == 0) s_flip = fl;
        }
        pair_sync();
        const unsigned flips = s_flip;
        // (c) det(1 + D_F A_FF) as the product of the sequential rank-1 ratios
        double rprod = 1.0;
        if (flips) {
            float rl = 1.f;
            int q = 0;
#pragma unroll
            for (int j = 0; j < NBP; ++j) g[j] = (in && j < nbk) ? S1[s][lane][j] : 0.f;
#pragma unroll 1
            for (int a = 0; a < nbk; ++a) {
                float f = 0.f;
                if ((flips >> a) & 1u) {  // uniform
                    const float dd = (xup >> a) & 1u ? fc.dflip[s][0] : fc.dflip[s][1];
                    const float rr = 1.f + dd * (1.f - __shfl_sync(FULL, g[0], a));
                    const float phi = fast_quot(dd, rr);
                    if (lane == a) {
                        rl = rr;
                        s_phi[s][q] = phi;
                    }
                    f = phi * g[0];
                    ++q;
                    const float first = g[0];
#pragma unroll
                    for (int j = 1; j < NBP; ++j) g[j - 1] = fmaf(f, __shfl_sync(FULL, g[j], a), g[j]);
                    g[NBP - 1] = first;  // decided columns are not read again
                } else {
                    const float first = g[0];
#pragma unroll
                    for (int j = 1; j < NBP; ++j) g[j - 1] = g[j];
                    g[NBP - 1] = first;
                }
            }
            rprod = (double)rl * fac;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) rprod *= __shfl_xor_sync(FULL, rprod, o);
        }
        if (lane == 0) s_prod[s] = rprod;
        pair_sync();
        ++n_prop;
        if (s == 0) {
            const double R = flips ? s_prod[0] * s_prod[1] : 1.0;
            bool acc = true;
            if (flips) {
                acc = rep ? force_acc : ua < fabs(R);
                if (!isfinite(R)) {
                    acc = false;
                    bad = true;
                }
                if (acc) {
                    if (R < 0) ++nneg;
                    maxr = fmax(maxr, fabs(R));
                }
            }
            if (lane == 0) {
                so.dec[N + blk] = acc ? 1 : 0;
                so.ratio[N + blk] = R;
                s_acc = acc && flips ? 1 : 0;
            }
            if (acc) {
                ++n_acc;
                if ((flips >> lane) & 1u) xl[p0 + lane] = (int8_t)(-x);
            }
        }
        __syncthreads();
        if (!s_acc) continue;
        // (d) the accepted flips, in increasing site order
        int q = 0;
        for (unsigned fl = flips; fl; fl &= fl - 1, ++q, ++m, par ^= 1) {
            const int a = p0 + __ffs(fl) - 1;
            __syncthreads();
            const float phi = s_phi[s][q];
            if (hw == 0 && lane == 0) wb.idx[m] = s0 + a;
#pragma unroll
            for (int j = 0; j < NP / 32; ++j) {
                const int c = lane + 32 * j;
                Wx[(size_t)m * NW + c] = c == a ? phi : srow[par][s][c];
                Wm[(size_t)m * NW + c] = c == a ? phi : phi * scol[par][s][c];
            }
        }
    }
    if (hw != 0) return;
    for (int q = lane; q < n; q += 32) so.ratio[s0 + q] = 1.0 / (1.0 + s_E[q]);
    if (lane == 0) {
        *wb.m = m;
        if (bad) set_err(err, DEV_NUMERIC);
        if (so.sign && (nneg & 1)) *so.sign = -*so.sign;
        so.stats[0] += n_prop;
        so.stats[1] += n_acc;
        so.stats[2] += m;
        so.stats[3] += (m > 0) ? 1 : 0;
        *so.maxr = fmax(*so.maxr, maxr);
    }
}

// One window of the block force-bias update in FP64 (AFQMC_MODE_BLOCKFB) or of the constrained path's
// (WIN_MODE_CPB), one block per walker, the window's block of G in shared memory.
template <int MODE>
__global__ void __launch_bounds__(WIN_THREADS) window_kernel(const double* __restrict__ Gu0, int8_t* xl0,
                                                             const double* u0, const uint8_t* replay0, SiteParams sp,
                                                             SliceOut so0, int s0, int n, int nb, WindowBufs wb0,
                                                             const double* blk0, int* err, Batch bt) {
    using T = double;
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
    size_t off = 2 * (size_t)n * P * sizeof(T);
    T* S1 = (T*)(smem_raw + off);  // [2][NBMAX][NBMAX+1]
    off += 2 * (size_t)NBMAX * (NBMAX + 1) * sizeof(T);
    T* strow = (T*)(smem_raw + off);  // staging: rows [2][n]
    off += 2 * (size_t)n * sizeof(T);
    T* stb = (T*)(smem_raw + off);  // columns [2][NBMAX]
    off += 2 * (size_t)NBMAX * sizeof(T);
    double* fb = (double*)(smem_raw + off);  // scalars [2][NBMAX]
    off += 2 * (size_t)NBMAX * sizeof(double);
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
    // the n x n diagonal block of both spins: from G, or as the previous window's panels left it
    // (pitch NW, spin stride NW^2)
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
    __shared__ double c_dflip[2][2], c_dstrip[2][2];
    if (tid < 4) {
        c_dflip[tid >> 1][tid & 1] = sp.dflip[tid >> 1][tid & 1];
        c_dstrip[tid >> 1][tid & 1] = sp.dstrip[tid >> 1][tid & 1];
    }
    if (tid == 0) s_m = 0;
    __syncthreads();

    __shared__ double s_sign, s_maxr;  // walker sign and max |R|, owned by one thread at a time
    if (tid == 0) {
        s_sign = so.sign ? *so.sign : 1.0;
        s_maxr = 0.0;
    }
    __syncthreads();
    int n_prop = 0, n_acc = 0, n_flip = 0;

    __shared__ int8_t s_xch[NWC];                // constrained path: the field chosen at each site
    __shared__ double s_cpl[2];                  // constrained path: sum ln N_i, sum ln |r_up r_dn|
    __shared__ int s_dead;
    if (MODE == WIN_MODE_CPB && tid == 0) {
        s_cpl[0] = 0.0;
        s_cpl[1] = 0.0;
        s_dead = so.cp ? (so.cp[2] != 0.0) : 0;
    }
    __syncthreads();
    if (MODE == WIN_MODE_CPB) {
        // ---- constrained-path block force bias (Sec. IV.D) ----
        // Per block S of nb sites (no field set yet): the force bias F_i of the current block's
        // diagonal (spin channel sum_s c_s A_s[i][i], charge channel lam (A_up + A_dn - 1)[i][i]),
        // each x_i from q(x_i) = e^{x_i F_i} / (2 cosh F_i); the weight factor
        // prod_i s(x_i) cosh F_i e^{-x_i F_i} prod_s det(1 + Delta_s A_s[S][S]) (the determinant as the
        // product of the sequential rank-1 ratios on a copy of the block); a factor <= 0 removes the
        // walker; the fields are then applied as accepts of the delayed update.
        __shared__ T s_phi2[2][NBMAX];
        __shared__ double s_rs2[2];
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
                    const T dd = c_dflip[tid][xi];
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
                    const T db = c_dstrip[tid][xi];
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
                    const T dd = c_dflip[tid][xi];
                    const T rr = T(1) + dd * (T(1) - S1[(tid * NBMAX + a) * (NBMAX + 1) + a]);
                    s_rs[tid] *= (double)rr;
                    s_phi[tid][q] = dd / rr;
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
    if (MODE == WIN_MODE_CPB) {  // the chosen fields, and the walker's weight factors
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
    // The accepts' rows and columns, from which panel_kernel forms the window's update of all of G
    window_export<T>(Gs, n, P, idx, s_fk, m, (T*)wb.Wx, (T*)wb.Wm, tid);
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

template <typename T, int MODE, int NP>
static cudaError_t launch_window_reg(cudaStream_t st, const T* Gu, int8_t* xl, const double* u, const uint8_t* replay,
                                     const SiteParams& sp, SliceOut so, int s0, int n, WindowBufs wb, const T* blk,
                                     int* err, Batch bt) {
    FlipConsts<T> fc;
    for (int xi = 0; xi < 2; ++xi) {
        for (int s = 0; s < 2; ++s) fc.dflip[s][xi] = (T)sp.dflip[s][xi];
        fc.sflip[xi] = (T)sp.sflip[xi];
    }
    count_launch();
    window_reg_kernel<T, MODE, NP><<<bt.nwk, WinTile<T, NP>::THREADS, 0, st>>>(Gu, xl, u, replay, sp.N, sp.ld, fc, so, s0,
                                                                               n, wb, blk, err, bt);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_window_chain(cudaStream_t st, int mode, const T* Gu, const T* Gd, int8_t* xl,
                                const double* u, const uint8_t* replay, const SiteParams& sp, SliceOut so,
                                int s0, int n, int nb, WindowBufs wb, const T* blk, int* err, Batch bt) {
    (void)Gd;  // spin down follows spin up (N x ld) in every walker's G
    if (bt.nwk < 1) bt.nwk = 1;
    // one accept at a time: the register-tile kernel of the smallest tile that holds the window
    if (mode == AFQMC_MODE_DELAYED) {
        if (n <= 32)
            return launch_window_reg<T, AFQMC_MODE_DELAYED, 32>(st, Gu, xl, u, replay, sp, so, s0, n, wb, blk, err, bt);
        if (n <= 64)
            return launch_window_reg<T, AFQMC_MODE_DELAYED, 64>(st, Gu, xl, u, replay, sp, so, s0, n, wb, blk, err, bt);
        if constexpr (WinCap<T>::NW > 64)
            return launch_window_reg<T, AFQMC_MODE_DELAYED, 128>(st, Gu, xl, u, replay, sp, so, s0, n, wb, blk, err,
                                                                 bt);
        return cudaErrorInvalidValue;
    }
    if constexpr (sizeof(T) == 8) {  // the constrained path runs in FP64 only
        if (mode == WIN_MODE_CP) {
            if (n <= 32)
                return launch_window_reg<T, WIN_MODE_CP, 32>(st, Gu, xl, u, replay, sp, so, s0, n, wb, blk, err, bt);
            return launch_window_reg<T, WIN_MODE_CP, 64>(st, Gu, xl, u, replay, sp, so, s0, n, wb, blk, err, bt);
        }
        if (mode == WIN_MODE_CPB) {
            cudaError_t e = ensure_smem_attr((const void*)window_kernel<WIN_MODE_CPB>, window_smem(WinCap<T>::NW));
            if (e != cudaSuccess) return e;
            count_launch();
            window_kernel<WIN_MODE_CPB><<<bt.nwk, WIN_THREADS, window_smem(n), st>>>(
                Gu, xl, u, replay, sp, so, s0, n, nb, wb, blk, err, bt);
            return cudaGetLastError();
        }
    }
    if (mode != AFQMC_MODE_BLOCKFB || n > WIN_FB || nb > NBMAX) return cudaErrorInvalidValue;
    if constexpr (sizeof(T) == 4) {
        FlipConsts<float> fc, fs;
        for (int xi = 0; xi < 2; ++xi) {
            for (int s = 0; s < 2; ++s) {
                fc.dflip[s][xi] = (float)sp.dflip[s][xi];
                fs.dflip[s][xi] = (float)sp.dstrip[s][xi];
            }
            fc.sflip[xi] = fs.sflip[xi] = (float)sp.sflip[xi];
        }
        count_launch();
        if (nb <= 16)
            window_fb_kernel<16><<<bt.nwk, 320, 0, st>>>(Gu, xl, u, replay, sp, fc, fs, so, s0, n, nb, wb, blk, err, bt);
        else
            window_fb_kernel<32><<<bt.nwk, 320, 0, st>>>(Gu, xl, u, replay, sp, fc, fs, so, s0, n, nb, wb, blk, err, bt);
        return cudaGetLastError();
    } else {
        cudaError_t e = ensure_smem_attr((const void*)window_kernel<AFQMC_MODE_BLOCKFB>, window_smem(WinCap<T>::NW));
        if (e != cudaSuccess) return e;
        count_launch();
        window_kernel<AFQMC_MODE_BLOCKFB><<<bt.nwk, WIN_THREADS, window_smem(n), st>>>(
            Gu, xl, u, replay, sp, so, s0, n, nb, wb, blk, err, bt);
        return cudaGetLastError();
    }
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
// A window's accepts a_0, a_1, ... in order are the rank-1 updates G += w_k q_k with
//   w_k[r] = -f_k (G[r][a_k] + sum_{k'<k} w_k'[r] C[k'][k]),
//   q_k[c] = G[a_k][c] - delta_{c a_k} + sum_{k'<k} (-f_k' C[k][k']) q_k'[c],
// G the matrix before the window and C[k][k'] = G[a_k][a_k'] as it was when the earlier of the two was
// accepted (Wx, Wm of the window kernel): every row's w and every column's q is a short recursion of its
// own, so no update matrix has to be formed on the decisions' critical path.
//   * panel_kernel (main stream, right after the window): w -> X (N x NW), q -> Y (NW x N), and the next
//     window's block of G as this window's update will leave it;
//   * launch_flush_gemm (flush stream): the rank-m product G += X Y over all of G, overlapping the next
//     window's decisions.
// In the T form the raw columns and rows are those of V = T U_L[:, I] and -(U_R[I, :] T).
// ---------------------------------------------------------------------------
template <typename T>
struct PanelArgs {
    const T* G = nullptr; long ld = 0, gw = 0, gs = 0;  // G form: matrix, walker and spin strides
    const T* V = nullptr;  // T form: raw columns [N][NW] and rows [NW][ldy] per (walker, spin)
    const T* R = nullptr;
    int N = 0;             // rows (columns) of the panels
    int s0 = 0, n = 0;     // the window
    int sn = 0, nn = 0;    // the next window (nn = 0: none)
    T* snap = nullptr;
    T* X = nullptr;        // [walker][spin][N][NW]
    T* Y = nullptr;        // [walker][spin][NW][ldy]
    long ldy = 0;
    WindowBufs wb;
};

// Threads per block (four per line) and rows of the next window's block per block.
template <typename T> struct PanelCfg { static constexpr int LT = sizeof(T) == 4 ? 512 : 128, RB = sizeof(T) == 4 ? 16 : 8; };
constexpr int PL_B = 16;  // accepts a line takes at a time (four per thread)

// Elements of the packed coefficient triangle of m accepts: the rows of the b-th group of PL_B accepts hold
// the columns from PL_B b on.
__host__ __device__ inline int panel_tri(int m) {
    const int nb = (m + PL_B - 1) / PL_B;
    return PL_B * PL_B * (nb * (nb + 1) / 2);
}

// Pitch of the column lines: whole 16-byte vectors, an odd number of them.
template <typename T>
__host__ __device__ inline int panel_pitch(int n) {
    constexpr int VW = 16 / sizeof(T);
    return ((n + VW - 1) / VW | 1) * VW;
}

template <typename T>
static size_t panel_smem(int n, int nn) {
    constexpr size_t LN = PanelCfg<T>::LT / 4, RB = PanelCfg<T>::RB;
    const size_t lines = (size_t)panel_tri(n) + LN * panel_pitch<T>(n);
    const size_t block = nn > 0 ? 2 * (size_t)panel_tri(n) + RB * panel_pitch<T>(n) + (size_t)n * nn + RB * nn : 0;
    return (lines > block ? lines : block) * sizeof(T) + 3 * WinCap<T>::NW * sizeof(int);
}

// Asynchronous copy of one element from global to shared memory (zero where !in).
template <typename T>
__device__ __forceinline__ void cp_async_elem(T* dst, const T* src, bool in) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    const int sz = in ? (int)sizeof(T) : 0;
    if (sizeof(T) == 4) asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(d), "l"(src), "r"(sz) : "memory");
    else asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(d), "l"(src), "r"(sz) : "memory");
}
// ... and of 16 bytes (both addresses aligned).
__device__ __forceinline__ void cp_async_16(void* dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}
// count elements from src to dst, lanes of a warp; vec: in 16-byte vectors (aligned, padded to whole vectors).
template <typename T>
__device__ __forceinline__ void cp_async_row(T* dst, const T* src, int count, bool vec, int lane) {
    constexpr int VW = 16 / sizeof(T);
    if (vec)
        for (int c = lane * VW; c < count; c += 32 * VW) cp_async_16(dst + c, src + c);
    else
        for (int c = lane; c < count; c += 32) cp_async_elem(dst + c, src + c, true);
}
__device__ __forceinline__ void cp_async_wait_all() {
    asm volatile("cp.async.commit_group;" ::: "memory");
    asm volatile("cp.async.wait_group 0;" ::: "memory");
}

// The packed triangle E[k'][k] = W[k'][pos[k]], k >= k' (zero elsewhere), W = Wx or Wm of one spin.
template <typename T>
__device__ __forceinline__ void panel_load_tri(T* E, const T* W, const int* pos, int m, int tid, int nt) {
    constexpr int NW = WinCap<T>::NW;
    const int ep = (m + PL_B - 1) / PL_B * PL_B, lane = tid & 31;
    for (int kp = tid >> 5; kp < ep; kp += nt >> 5) {
        const int b = kp / PL_B, k0 = b * PL_B;
        T* row = E + PL_B * (b * ep - PL_B * (b * (b - 1) / 2)) + (kp - k0) * (ep - k0);
        for (int k = k0 + lane; k < ep; k += 32) {
            const bool in = k >= kp && k < m;
            cp_async_elem(row + k - k0, in ? W + (size_t)kp * NW + pos[k] : W, in);
        }
    }
}

// One line through the recursion, in place, by four lanes (h = lane & 3): entry k at line[off[k]]; column
// lines (col) scale by the diagonal, row lines subtract the identity at their own column (gi, global index
// of accept k in gidx[k]) first; neg: the raw line enters negated.  All lanes of a warp call this together.
template <typename T>
__device__ __forceinline__ void panel_line(T* line, const int* off, int step, const T* E, int m, bool col, bool neg,
                                           const int* gidx, int gi, bool own, int lane) {
    constexpr int VW = Vec16<T>::W;
    using V = typename Vec16<T>::V;
    constexpr unsigned FULL = 0xffffffffu;
    const int h = lane & 3, ep = (m + PL_B - 1) / PL_B * PL_B;
    const T* Eb = E;  // rows of group b
    for (int kb = 0; kb < m; kb += PL_B) {
        T v[4];
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            const int k = kb + 4 * h + t;
            T x = T(0);
            if (k < m) {
                x = line[off[k] * step];
                if (neg) x = -x;
                if (!col && gidx && gidx[k] == gi) x -= T(1);
            }
            v[t] = x;
        }
        const T* Ep = E + kb + 4 * h;  // columns kb + 4 h .. of the finished accepts' rows
        for (int k0 = 0, w = ep; k0 < kb; k0 += PL_B, w -= PL_B) {
#pragma unroll
            for (int j = 0; j < PL_B; ++j) {
                const T x = line[off[k0 + j] * step];
                T d[4];
#pragma unroll
                for (int t = 0; t < 4; t += VW) *(V*)(d + t) = *(const V*)(Ep + j * w + t);
#pragma unroll
                for (int t = 0; t < 4; ++t) v[t] = fma(x, d[t], v[t]);
            }
            Ep += PL_B * w - PL_B;
        }
        const int w = ep - kb;
        // FP32 straight-line: entries from m on are zero, as are their coefficients (FP64 leaves them out)
#pragma unroll
        for (int j = 0; j < PL_B; ++j) {
            if (sizeof(T) == 8 && kb + j >= m) break;
            T x = __shfl_sync(FULL, v[j & 3], (lane & ~3) | (j >> 2));
            if (col) x *= Eb[j * w + j];
            if (own && h == 0 && kb + j < m) line[off[kb + j] * step] = x;
            T d[4];
#pragma unroll
            for (int t = 0; t < 4; t += VW) *(V*)(d + t) = *(const V*)(Eb + j * w + 4 * h + t);
#pragma unroll
            for (int t = 0; t < 4; ++t) v[t] = fma(x, d[t], v[t]);  // entries up to j are not read again
        }
        __syncwarp();
        Eb += PL_B * w;
    }
}

// Grid (row blocks, then column blocks of N lines, then blocks of the next window; spin; walker).  A block
// stages raw lines and the coefficient triangle in shared memory by asynchronous copies and takes each
// line through the recursion with four lanes.  A block of the next window forms the w of its RB rows and
// the q of all nn columns and writes G[J][J] + w_J q_J.  Bound by the latency of the recursion (m^2 / 2
// multiply-adds per line).
template <typename T, bool TF>
__global__ void __launch_bounds__(PanelCfg<T>::LT) panel_kernel(PanelArgs<T> a) {
    constexpr int NW = WinCap<T>::NW, LT = PanelCfg<T>::LT, LN = LT / 4, RB = PanelCfg<T>::RB;
    const int wk = blockIdx.z, s = blockIdx.y, tid = threadIdx.x, lane = tid & 31;
    const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
    const int N = a.N, n = a.n, nl = (N + LN - 1) / LN, z = 2 * wk + s, bx = blockIdx.x;
    const WindowBufs wb = wb_walker<T>(a.wb, wk, N);
    const T* G = TF ? nullptr : a.G + (size_t)wk * a.gw + (size_t)s * a.gs;
    const int m = __shfl_sync(0xffffffffu, *wb.m, 0), PC = panel_pitch<T>(n);
    extern __shared__ __align__(16) unsigned char pl_smem[];
    T* E = (T*)pl_smem;
    const T* W0 = (const T*)wb.Wx + (size_t)s * NW * NW;
    const T* W1 = (const T*)wb.Wm + (size_t)s * NW * NW;
    const int tri = panel_tri(m);
    if (bx >= 2 * nl) {  // rows r0 .. r0 + RB - 1 of the next window's block
        T* E1 = E + tri;
        T* bw = E1 + tri;                    // w lines [RB][PC], accept k at its position in the window
        T* bq = bw + RB * PC;                // q lines [m][nn]
        T* gb = bq + (size_t)n * a.nn;       // G[J rows][J] [RB][nn]
        int* gidx = (int*)(gb + RB * a.nn);  // accepts: global index, position in the window, own index
        int *pos = gidx + NW, *idn = pos + NW;
        const int r0 = (bx - 2 * nl) * RB, nr = min(RB, a.nn - r0), nn = a.nn;
        for (int k = tid; k < m; k += LT) {
            gidx[k] = wb.idx[k];
            pos[k] = wb.idx[k] - a.s0;
            idn[k] = k;
        }
        __syncthreads();
        const T* rows = G + (long)(a.sn + r0) * a.ld;
        constexpr int VW = 16 / sizeof(T);
        const bool vc = a.s0 % VW == 0, vn = a.sn % VW == 0 && nn % VW == 0;
        for (int r = warp; r < nr; r += LT / 32) {
            cp_async_row<T>(gb + r * nn, rows + r * a.ld + a.sn, nn, vn, lane);
            cp_async_row<T>(bw + r * PC, rows + r * a.ld + a.s0, n, vc, lane);
        }
        for (int k = warp; k < m; k += LT / 32)
            cp_async_row<T>(bq + k * nn, G + (long)gidx[k] * a.ld + a.sn, nn, vn, lane);
        panel_load_tri<T>(E, W0, pos, m, tid, LT);
        panel_load_tri<T>(E1, W1, pos, m, tid, LT);
        cp_async_wait_all();
        __syncthreads();
        // the next window's sites are not among the accepts: no identity term.  Row lines fill whole warps
        // (8 lines each) so that a warp has lines of one kind.
        constexpr int RW = RB / 8;
        for (int wv = warp; wv * 8 < 8 * RW + nn; wv += LT / 32) {
            const bool col = wv < RW;
            const int l0 = (col ? wv : wv - RW) * 8, l = l0 + (lane >> 2), lim = col ? nr : nn, lc = min(l, lim - 1);
            if (l0 < lim)
                panel_line<T>(col ? bw + lc * PC : bq + lc, col ? pos : idn, col ? 1 : nn, col ? E : E1, m, col, false,
                              nullptr, 0, l < lim, lane);
        }
        __syncthreads();
        T* out = a.snap + (size_t)z * NW * NW + (size_t)r0 * NW;
        // sums of their own, then added: one rounding at G's magnitude, not m
        for (int r = warp; r < nr; r += LT / 32)
            for (int c = lane; c < nn; c += 64) {
                const int c1 = c + 32 < nn ? c + 32 : c;
                T acc = T(0), acc1 = T(0);
                const T* wr = bw + r * PC;
#pragma unroll 8
                for (int k = 0; k < m; ++k) {
                    const T w = wr[pos[k]];
                    acc = fma(w, bq[k * nn + c], acc);
                    acc1 = fma(w, bq[k * nn + c1], acc1);
                }
                out[r * NW + c] = gb[r * nn + c] + acc;
                if (c1 != c) out[r * NW + c1] = gb[r * nn + c1] + acc1;
            }
        return;
    }
    if (m == 0) return;
    const bool col = bx < nl;  // column lines: one per row of G
    const int i0 = (col ? bx : bx - nl) * LN, cnt = min(LN, N - i0);
    T* buf = E + tri;  // column lines [LN][PC] (T form: accept k at k, else at its position), row lines [m][LN]
    int* gidx = (int*)(buf + (size_t)LN * PC);
    int *pos = gidx + NW, *idn = pos + NW;
    for (int k = tid; k < m; k += LT) {
        gidx[k] = TF ? -1 : wb.idx[k];
        pos[k] = wb.idx[k] - a.s0;
        idn[k] = k;
    }
    __syncthreads();
    constexpr int VW = 16 / sizeof(T);
    if (col) {
        for (int r = warp; r < cnt; r += LT / 32)
            cp_async_row<T>(buf + r * PC, TF ? a.V + ((size_t)z * N + i0 + r) * NW : G + (long)(i0 + r) * a.ld + a.s0,
                            TF ? m : n, TF || a.s0 % VW == 0, lane);
    } else {
        for (int k = warp; k < m; k += LT / 32)
            cp_async_row<T>(buf + k * LN, TF ? a.R + ((size_t)z * NW + k) * a.ldy + i0 : G + (long)gidx[k] * a.ld + i0,
                            cnt, !TF, lane);
    }
    panel_load_tri<T>(E, col ? W0 : W1, pos, m, tid, LT);
    cp_async_wait_all();
    __syncthreads();
    if (warp * 8 < cnt) {
        const int l = tid >> 2, lc = min(l, cnt - 1);
        panel_line<T>(col ? buf + lc * PC : buf + lc, col && !TF ? pos : idn, col ? 1 : LN, E, m, col, TF && !col, gidx,
                      i0 + lc, l < cnt, lane);
    }
    __syncthreads();
    if (col) {
        T* out = a.X + ((size_t)z * N + i0) * NW;
        for (int r = warp; r < cnt; r += LT / 32)
            for (int k = lane; k < m; k += 32) out[r * NW + k] = buf[r * PC + (TF ? k : pos[k])];
    } else {
        for (int k = warp; k < m; k += LT / 32)
            for (int c = lane; c < cnt; c += 32) a.Y[((size_t)z * NW + k) * a.ldy + i0 + c] = buf[k * LN + c];
    }
}

template <typename T, bool TF>
static cudaError_t launch_panel_kernel(cudaStream_t st, const PanelArgs<T>& a, int nwk) {
    cudaError_t e = ensure_smem_attr((const void*)panel_kernel<T, TF>, panel_smem<T>(WinCap<T>::NW, WinCap<T>::NW));
    if (e != cudaSuccess) return e;
    constexpr int LN = PanelCfg<T>::LT / 4, RB = PanelCfg<T>::RB;
    count_launch();
    panel_kernel<T, TF><<<dim3(2 * ((a.N + LN - 1) / LN) + (a.nn + RB - 1) / RB, 2, nwk), PanelCfg<T>::LT,
                          panel_smem<T>(a.n, a.nn), st>>>(a);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_flush_panels(cudaStream_t st, const T* Gu, const SiteParams& sp, WindowBufs wb, int s0, int n,
                                int sn, int nn, T* snap, Batch bt) {
    PanelArgs<T> a;
    a.G = Gu; a.ld = sp.ld; a.gw = bt.gstride; a.gs = (long)sp.N * sp.ld;
    a.N = sp.N; a.s0 = s0; a.n = n; a.sn = sn; a.nn = nn;
    a.snap = snap;
    a.X = (T*)wb.X; a.Y = (T*)wb.Y; a.ldy = sp.N;
    a.wb = wb;
    return launch_panel_kernel<T, false>(st, a, bt.nwk);
}

template <typename T>
cudaError_t launch_tform_panels(cudaStream_t st, int ns, WindowBufs wb, int s0, int n, T* V, const T* R, T* Y,
                                int nwk) {
    PanelArgs<T> a;
    a.V = V; a.R = R;
    a.N = ns; a.s0 = s0; a.n = n;
    a.X = V; a.Y = Y; a.ldy = ns;
    a.wb = wb;
    return launch_panel_kernel<T, true>(st, a, nwk);
}

// G <- G + X Y (the N x N rank-m product of launch_flush_panels' panels).
template <typename T>
cudaError_t launch_flush_gemm(cudaStream_t sf, T* Gu, T* Gd, const SiteParams& sp, WindowBufs wb, int nw, Batch bt) {
    (void)Gd;
    constexpr int NW = WinCap<T>::NW;
    const int N = sp.N;
    GemmArgs<T> h;
    h.M = N; h.N = N; h.K = nw; h.Kdev = wb.m; h.kdiv = 2;
    h.A = (const T*)wb.X; h.lda = NW; h.sA = (long)N * NW;
    h.B = (const T*)wb.Y; h.ldb = N; h.sB = (long)NW * N;
    h.C = Gu; h.ldc = sp.ld; h.sC = (long)N * sp.ld;
    h.alpha = T(1); h.beta = T(1);
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
template cudaError_t launch_flush_panels<float>(cudaStream_t, const float*, const SiteParams&, WindowBufs, int, int,
                                               int, int, float*, Batch);
template cudaError_t launch_flush_panels<double>(cudaStream_t, const double*, const SiteParams&, WindowBufs, int, int,
                                                int, int, double*, Batch);
template cudaError_t launch_tform_panels<float>(cudaStream_t, int, WindowBufs, int, int, float*, const float*, float*,
                                               int);
template cudaError_t launch_tform_panels<double>(cudaStream_t, int, WindowBufs, int, int, double*, const double*,
                                                double*, int);
template cudaError_t launch_flush_gemm<float>(cudaStream_t, float*, float*, const SiteParams&, WindowBufs, int, Batch);
template cudaError_t launch_flush_gemm<double>(cudaStream_t, double*, double*, const SiteParams&, WindowBufs, int,
                                              Batch);
template cudaError_t launch_flush<float>(cudaStream_t, float*, float*, const SiteParams&, WindowBufs, int);
template cudaError_t launch_flush<double>(cudaStream_t, double*, double*, const SiteParams&, WindowBufs, int);

}  // namespace afq
