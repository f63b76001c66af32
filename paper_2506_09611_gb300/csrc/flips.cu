// flips.cu -- stateless application of accepted field changes to G in one
// rank-m product (the G form of Eqs. FinalDelay and BlkFrcBsTnew2):
//     G_s <- G_s - G_s[:, I] W_s (E_I^T - G_s[I, :]),
//     W_s  = D_s (1 + (1 - G_s[I, I]) D_s)^{-1},   (D_s)_aa = exp(c_s (x'_a - x_a)) - 1.
#include <cooperative_groups.h>
#include <math.h>

#include <mutex>

#include "internal.h"

namespace afq {

// Scratch layout (bytes), pitch NW = window_max<T>() as in the sweep's flush:
//   [0, 256)      int m, int err, ...
//   [256, ...)    idx[NW] (validated copy of the sites)
//   Wm            2 * NW * NW * T
//   X             2 * N * NW * T
//   Y             4 * NW * N * T
template <typename T>
size_t flips_scratch_bytes(int N) {
    const size_t NW = (size_t)window_max<T>();
    auto al = [](size_t b) { return (b + 255) & ~(size_t)255; };
    return 256 + al(NW * sizeof(int)) + al(2 * NW * NW * sizeof(T)) + al(2 * (size_t)N * NW * sizeof(T)) +
           al(4 * NW * (size_t)N * sizeof(T));
}

template <typename T>
static WindowBufs flips_layout(unsigned char* scratch, int N) {
    const size_t NW = (size_t)window_max<T>();
    auto al = [](size_t b) { return (b + 255) & ~(size_t)255; };
    WindowBufs wb;
    wb.m = (int*)scratch;
    size_t off = 256;
    wb.idx = (int*)(scratch + off);
    off += al(NW * sizeof(int));
    wb.Wm = scratch + off;
    wb.Wx = nullptr;
    off += al(2 * NW * NW * sizeof(T));
    wb.X = scratch + off;
    off += al(2 * (size_t)N * NW * sizeof(T));
    wb.Y = scratch + off;
    return wb;
}

// W_s = D_s M_s^{-1}, M_s = 1 + (1 - G_II) D_s, one CTA per spin in a cluster of two, by in-place
// Gauss-Jordan with partial pivoting.  M lives in registers: thread (rg, cg) holds rows rg + 16 i and columns
// cg + FC j (FC = 16 or 32), up to MP x MP elements.  Step k takes two block barriers: the holders of column
// k put it into shared memory; every warp finds the pivot among the rows not used yet (two integer
// reductions per 32 rows) and the holders of the pivot row put it beside; all threads eliminate.  Rows are
// not swapped: row piv[k] ends as row k of the inverse, with column k the multiplier of equation piv[k].
// Bound by the latency of the steps (64 of them took 2 x 130 us in shared memory with five barriers each and
// both spins in turn).
// The status word wb.m[1] is rewritten by every call: 0, DEV_ARG (a site outside [0, N)) or DEV_NUMERIC (a
// zero pivot in either spin); on either error wb.m[0] (the product's inner dimension) is 0, so G is left
// unchanged.
__device__ __forceinline__ unsigned long long flips_key(double x) {
    return (unsigned long long)__double_as_longlong(fabs(x));
}
__device__ __forceinline__ unsigned long long flips_key(float x) {
    return (unsigned long long)__float_as_uint(fabsf(x));
}

template <typename T, int MP>
struct FlipsTile {
    static constexpr int FC = MP > 64 ? 32 : 16, TR = MP / 16, TC = MP / FC, THREADS = 16 * FC;
};

template <typename T, int MP>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(FlipsTile<T, MP>::THREADS)
    flips_W_kernel(const T* __restrict__ Gu, const T* __restrict__ Gd, long ld, int N, const int* sites,
                   const double* delta, int m, WindowBufs wb, int NWC) {
    using F = FlipsTile<T, MP>;
    constexpr int FC = F::FC, TR = F::TR, TC = F::TC;
    namespace cg = cooperative_groups;
    cg::cluster_group cl = cg::this_cluster();
    const int s = (int)cl.block_rank(), tid = threadIdx.x, lane = tid & 31, rg = tid / FC, cgi = tid % FC;
    const T* G = s ? Gd : Gu;
    __shared__ int sidx[MP];
    __shared__ int piv[MP];
    __shared__ T col[2][MP], row[2][MP];  // by step parity
    __shared__ int s_bad, s_num;
    if (tid == 0) {
        s_bad = 0;
        s_num = 0;
    }
    __syncthreads();
    for (int a = tid; a < m; a += F::THREADS) {
        const int v = sites[a];
        if (v < 0 || v >= N) s_bad = 1;
        sidx[a] = (v < 0 || v >= N) ? 0 : v;
        if (s == 0) wb.idx[a] = sidx[a];
    }
    __syncthreads();
    if (!s_bad) {
        T A[TR][TC];
#pragma unroll
        for (int i = 0; i < TR; ++i)
#pragma unroll
            for (int j = 0; j < TC; ++j) {
                const int r = rg + 16 * i, c = cgi + FC * j;
                A[i][j] = T(0);
                if (r < m && c < m) {
                    const double a0 = (r == c ? 1.0 : 0.0) - (double)G[(long)sidx[r] * ld + sidx[c]];
                    A[i][j] = (T)((r == c ? 1.0 : 0.0) + a0 * delta[s * m + c]);
                }
            }
        unsigned used[MP / 32];  // rows taken as pivots (the same in every thread)
#pragma unroll
        for (int w = 0; w < MP / 32; ++w) used[w] = 0u;
        bool singular = false;
        for (int k = 0; k < m; ++k) {
            const int par = k & 1;
            if (cgi == k % FC) {
#pragma unroll
                for (int i = 0; i < TR; ++i) {
                    T t[TC];
#pragma unroll
                    for (int j = 0; j < TC; ++j) t[j] = A[i][j];
                    col[par][rg + 16 * i] = reg_pick<T, TC>(t, k / FC);
                }
            }
            __syncthreads();
            // the largest entry of the unused rows, ties to the lower row
            unsigned long long best = 0;
            int p = MP;
#pragma unroll
            for (int w = 0; w < MP / 32; ++w) {
                const int r = lane + 32 * w;
                if (r < m && !((used[w] >> lane) & 1u)) {
                    const unsigned long long key = flips_key(col[par][r]) + 1;  // above "no row"
                    if (key > best) {
                        best = key;
                        p = r;
                    }
                }
            }
            const unsigned hi = __reduce_max_sync(0xffffffffu, (unsigned)(best >> 32));
            const unsigned lo = __reduce_max_sync(0xffffffffu, (unsigned)(best >> 32) == hi ? (unsigned)best : 0u);
            const bool mine = best == (((unsigned long long)hi << 32) | lo);
            p = (int)__reduce_min_sync(0xffffffffu, mine ? (unsigned)p : 0xffffffffu);
            const T pv = col[par][p];
            if (!(fabs(pv) > T(0))) singular = true;
#pragma unroll
            for (int w = 0; w < MP / 32; ++w)
                if (w == p >> 5) used[w] |= 1u << (p & 31);
            if (tid == 0) piv[k] = p;
            if (rg == (p & 15)) {
#pragma unroll
                for (int j = 0; j < TC; ++j) {
                    T t[TR];
#pragma unroll
                    for (int i = 0; i < TR; ++i) t[i] = A[i][j];
                    row[par][cgi + FC * j] = reg_pick<T, TR>(t, p >> 4);
                }
            }
            const T inv = T(1) / pv;
            __syncthreads();
            // pivot row scaled by 1 / pivot (its column k: 1 / pivot), the others minus their column entry times it
#pragma unroll
            for (int j = 0; j < TC; ++j) {
                const int c = cgi + FC * j;
                const T rv = c == k ? inv : row[par][c] * inv;
#pragma unroll
                for (int i = 0; i < TR; ++i) {
                    const int r = rg + 16 * i;
                    const T f = col[par][r];
                    if (r == p) A[i][j] = rv;
                    else A[i][j] = c == k ? -f * rv : A[i][j] - f * rv;
                }
            }
        }
        __syncthreads();
        // inverse[k][piv[j]] = A[piv[k]][j]: put M^{-1} D in place through the pivot order
        T* Wm = (T*)wb.Wm + (size_t)s * NWC * NWC;
#pragma unroll
        for (int i = 0; i < TR; ++i) {
            const int r = rg + 16 * i;
            int k = -1;
            if (r < m)
                for (int q = 0; q < m; ++q)
                    if (piv[q] == r) k = q;
#pragma unroll
            for (int j = 0; j < TC; ++j) {
                const int c = cgi + FC * j;
                if (k >= 0 && c < m) Wm[k * NWC + piv[c]] = (T)(delta[s * m + k] * (double)A[i][j]);
            }
        }
        if (singular && tid == 0) s_num = 1;
    }
    cl.sync();
    if (s == 0 && tid == 0) {
        const int num = s_num | *cl.map_shared_rank(&s_num, 1);
        wb.m[0] = (s_bad || num) ? 0 : m;
        wb.m[1] = s_bad ? DEV_ARG : num ? DEV_NUMERIC : 0;
    }
    cl.sync();  // spin down's status is read before its CTA leaves
}

template <typename T, int MP>
static cudaError_t launch_flips_W(cudaStream_t st, const T* Gu, const T* Gd, long ld, int N, const int* sites,
                                  const double* delta, int m, WindowBufs wb) {
    count_launch();
    flips_W_kernel<T, MP><<<2, FlipsTile<T, MP>::THREADS, 0, st>>>(Gu, Gd, ld, N, sites, delta, m, wb, window_max<T>());
    return cudaGetLastError();
}

template <typename T>
static cudaError_t apply_flips_impl(cudaStream_t st, int N, long ld, T* Gu, T* Gd, const int* sites,
                                    const double* delta, int m, unsigned char* scratch) {
    WindowBufs wb = flips_layout<T>(scratch, N);
    cudaError_t e;
    if (m <= 32) e = launch_flips_W<T, 32>(st, Gu, Gd, ld, N, sites, delta, m, wb);
    else if (m <= 64) e = launch_flips_W<T, 64>(st, Gu, Gd, ld, N, sites, delta, m, wb);
    else if constexpr (sizeof(T) == 4) e = launch_flips_W<T, 128>(st, Gu, Gd, ld, N, sites, delta, m, wb);
    else e = cudaErrorInvalidValue;
    if (e != cudaSuccess) return e;
    SiteParams sp{};
    sp.N = N;
    sp.ld = ld;
    return launch_flush<T>(st, Gu, Gd, sp, wb, m);
}

// Copy the call's device status word (wb.m[1], at byte 4 of the scratch) to the host on the call's
// stream, wait for the stream, and map it to an ABI code.
static int flips_status(cudaStream_t st, const unsigned char* scratch) {
    int h = 0;
    if (cudaMemcpyAsync(&h, scratch + sizeof(int), sizeof(int), cudaMemcpyDeviceToHost, st) != cudaSuccess)
        return AFQMC_ERR_CUDA;
    if (cudaStreamSynchronize(st) != cudaSuccess) return AFQMC_ERR_CUDA;
    if (h == DEV_ARG) return AFQMC_ERR_ARG;
    if (h == DEV_NUMERIC) return AFQMC_ERR_NUMERIC;
    return h == 0 ? AFQMC_OK : AFQMC_ERR_CUDA;
}

static int flips_check(int precision, int N, long long ld, void* G_up, void* G_dn, const int* sites,
                       const double* delta, int m) {
    if (precision != AFQMC_PREC_FP64 && precision != AFQMC_PREC_FP32) return AFQMC_ERR_ARG;
    const int NW = precision == AFQMC_PREC_FP64 ? window_max<double>() : window_max<float>();
    if (N < 1 || ld < N || m < 0 || m > NW || !G_up || !G_dn) return AFQMC_ERR_ARG;
    if (m > 0 && (!sites || !delta)) return AFQMC_ERR_ARG;
    return AFQMC_OK;
}

// The scratch of afqmc_apply_flips comes from a memory pool of its own per device that keeps up to
// FLIPS_POOL_KEEP bytes between calls: the device's default pool gives everything back at the first
// synchronisation after a call, and mapping the memory again costs about 200 us a call.  A pool grows by blocks
// of 32 MB (cudaMemPoolAttrReservedMemCurrent) and gives back whole ones, so one block is the least bound that keeps
// anything (with 16 MB a call between synchronisations took 258 us, with 32 MB 61 us: 8 x 8, FP64, 4 changes); it
// holds the scratch of any lattice up to 64 x 64.  Allocation stays ordered on the call's stream, so calls on several
// streams and threads never share a buffer; anything above the bound goes back at the next synchronisation.
constexpr uint64_t FLIPS_POOL_KEEP = 32u << 20;

static cudaError_t flips_alloc(void** p, size_t bytes, cudaStream_t st) {
    constexpr int MAXDEV = 64;
    static std::mutex mu;
    static cudaMemPool_t pools[MAXDEV] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= MAXDEV) return cudaMallocAsync(p, bytes, st);
    cudaMemPool_t pool = nullptr;
    {
        std::lock_guard<std::mutex> lk(mu);
        if (!pools[dev]) {
            cudaMemPoolProps props = {};
            props.allocType = cudaMemAllocationTypePinned;
            props.location.type = cudaMemLocationTypeDevice;
            props.location.id = dev;
            uint64_t keep = FLIPS_POOL_KEEP;
            cudaMemPool_t made = nullptr;
            if ((e = cudaMemPoolCreate(&made, &props)) != cudaSuccess) return e;
            if ((e = cudaMemPoolSetAttribute(made, cudaMemPoolAttrReleaseThreshold, &keep)) != cudaSuccess) {
                cudaMemPoolDestroy(made);
                return e;
            }
            pools[dev] = made;
        }
        pool = pools[dev];
    }
    return cudaMallocFromPoolAsync(p, bytes, pool, st);
}

}  // namespace afq

using namespace afq;

extern "C" int afqmc_apply_flips(int precision, int N, long long ld, void* G_up, void* G_dn, const int* sites,
                                 const double* delta, int m, void* stream) {
    int rc = flips_check(precision, N, ld, G_up, G_dn, sites, delta, m);
    if (rc) return rc;
    if (m == 0) return AFQMC_OK;
    cudaStream_t st = (cudaStream_t)stream;
    const size_t bytes = precision == AFQMC_PREC_FP64 ? flips_scratch_bytes<double>(N) : flips_scratch_bytes<float>(N);
    void* scratch = nullptr;
    if (flips_alloc(&scratch, bytes, st) != cudaSuccess) return AFQMC_ERR_OOM;
    cudaError_t e = precision == AFQMC_PREC_FP64
                        ? apply_flips_impl<double>(st, N, (long)ld, (double*)G_up, (double*)G_dn, sites, delta, m,
                                                   (unsigned char*)scratch)
                        : apply_flips_impl<float>(st, N, (long)ld, (float*)G_up, (float*)G_dn, sites, delta, m,
                                                  (unsigned char*)scratch);
    const int rs = (e == cudaSuccess) ? flips_status(st, (const unsigned char*)scratch) : AFQMC_ERR_CUDA;
    cudaError_t e2 = cudaFreeAsync(scratch, st);
    if (rs != AFQMC_OK) return rs;
    return e2 == cudaSuccess ? AFQMC_OK : AFQMC_ERR_CUDA;
}

// ---------------------------------------------------------------------------
// No-allocation variant.
//
// Some callers cannot allocate device memory at the point where they apply an
// update: code that runs under a fixed device-memory budget owned by a host
// framework, code inside a real-time loop where an allocation (and the
// synchronisation cudaMalloc may imply) is not allowed, or a plugin whose host
// process gives it no allocator.  afqmc_apply_flips_noalloc does exactly the
// work of afqmc_apply_flips, with its scratch in the file-scope device array
// below instead of cudaMallocAsync.
//
// The array is sized for lattices up to NOALLOC_MAX_N sites in either
// precision; every GPU that loads this library holds it until the process
// exits.  Host code cannot use the array's name as a device address, so the
// first call on each device looks the address up with cudaGetSymbolAddress
// while that device is current and caches it.
// ---------------------------------------------------------------------------
namespace afq {

constexpr int NOALLOC_MAX_N = 4096;

constexpr size_t noalloc_align(size_t b) { return (b + 255) & ~(size_t)255; }
constexpr size_t noalloc_bytes_for(size_t NW, size_t esz, size_t N) {
    return 256 + noalloc_align(NW * sizeof(int)) + noalloc_align(2 * NW * NW * esz) + noalloc_align(2 * N * NW * esz) +
           noalloc_align(4 * NW * N * esz);
}
constexpr size_t NOALLOC_BYTES_F32 = noalloc_bytes_for(128, 4, NOALLOC_MAX_N);
constexpr size_t NOALLOC_BYTES_F64 = noalloc_bytes_for(64, 8, NOALLOC_MAX_N);
constexpr size_t NOALLOC_BYTES = NOALLOC_BYTES_F32 > NOALLOC_BYTES_F64 ? NOALLOC_BYTES_F32 : NOALLOC_BYTES_F64;

static __device__ __align__(256) unsigned char g_flips_scratch[NOALLOC_BYTES];

}  // namespace afq

namespace {
constexpr int NOALLOC_MAXDEV = 64;
std::mutex g_noalloc_mu;
void* g_noalloc_addr[NOALLOC_MAXDEV] = {};
}  // namespace

extern "C" int afqmc_apply_flips_noalloc(int precision, int N, long long ld, void* G_up, void* G_dn,
                                         const int* sites, const double* delta, int m, void* stream) {
    int rc = afq::flips_check(precision, N, ld, G_up, G_dn, sites, delta, m);
    if (rc) return rc;
    if (N > afq::NOALLOC_MAX_N) return AFQMC_ERR_ARG;
    const size_t need = precision == AFQMC_PREC_FP64 ? afq::flips_scratch_bytes<double>(N)
                                                     : afq::flips_scratch_bytes<float>(N);
    if (need > afq::NOALLOC_BYTES) return AFQMC_ERR_ARG;
    if (m == 0) return AFQMC_OK;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= NOALLOC_MAXDEV) return AFQMC_ERR_CUDA;
    void* scratch = nullptr;
    {
        std::lock_guard<std::mutex> lk(g_noalloc_mu);
        if (!g_noalloc_addr[dev]) {
            void* p = nullptr;
            if (cudaGetSymbolAddress(&p, afq::g_flips_scratch) != cudaSuccess || !p) return AFQMC_ERR_CUDA;
            g_noalloc_addr[dev] = p;
        }
        scratch = g_noalloc_addr[dev];
    }
    cudaStream_t st = (cudaStream_t)stream;
    cudaError_t e = precision == AFQMC_PREC_FP64
                        ? afq::apply_flips_impl<double>(st, N, (long)ld, (double*)G_up, (double*)G_dn, sites, delta,
                                                        m, (unsigned char*)scratch)
                        : afq::apply_flips_impl<float>(st, N, (long)ld, (float*)G_up, (float*)G_dn, sites, delta, m,
                                                       (unsigned char*)scratch);
    if (e != cudaSuccess) return AFQMC_ERR_CUDA;
    return afq::flips_status(st, (const unsigned char*)scratch);
}
