// FP64 building blocks of the CTMRG sweep: GEMM, axis permutation,
// normalisation, counter-based Gaussian numbers.  GB300 (sm_103a).
#include <cuda_runtime.h>
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <mutex>

#include "dgemm_plan.h"
#include "internal.h"

namespace ctm {

std::atomic<long long> g_launches{0};
thread_local bool dep_in_capture = false;

// ---------------------------------------------------------------------------
// FP64 GEMM, row-major: C[M,N] = alpha op(A) op(B) + beta C.
// GB300 issues an FP64 instruction over 64 cycles per SM quarter, so that
// multiply-adds on padding and idle SMs are all that costs: a few loads per
// multiply-add do not.  Tiles are therefore small and fitted to the shape:
// (32 TM) x (8 TN), TM <= 4, TN <= 9, 256 threads of TM x TN outputs each, K
// taken exactly, next K step prefetched in registers; dgemm_plan picks the
// tile and a split of K by the work of the fullest SM.  64 x 64 tiles padded
// N = 36 and 72 to 64 and 128 (the corners of D = 6) and left 144 x 144
// products on 9 SMs: 144^3 156 -> 15 us, an FP64 sweep at d=2, D=6, chi=48 (all
// its products) 293 -> 146 ms, at d=2, D=3, chi=16 51 -> 6.5 ms.
// ---------------------------------------------------------------------------
namespace {
// Split-K: blockIdx.z takes K range [z*kchunk, (z+1)*kchunk) and writes its
// partial product (alpha=1, beta=0) to C + z*zstride; a second kernel sums
// the partials in fixed order, so results do not depend on scheduling.
// A element (m, k) at A[m * sam + k * sak], B element (k, n) at B[k * sbk + n * sbn].
template <int TM, int TN>
__global__ void __launch_bounds__(256) k_dgemm(int M, int N, int K, double alpha, const double* __restrict__ A,
                                               long long sam, long long sak, const double* __restrict__ B,
                                               long long sbk, long long sbn, double beta, double* __restrict__ C,
                                               int ldc, int kchunk, size_t zstride) {
    dep_wait(A, B, C);
    constexpr int BM = 32 * TM, BN = 8 * TN;
    constexpr int NA = BM * GK / 256, NB = (BN * GK + 255) / 256;
    __shared__ double As[GK][BM + 1];
    __shared__ double Bs[GK][BN + 1];
    // unsigned: the ends of the last split and step may lie beyond 2^31
    const unsigned kbeg = blockIdx.z * (unsigned)kchunk;
    const unsigned kend = min((unsigned)K, kbeg + (unsigned)kchunk);
    C += blockIdx.z * zstride;
    const int tid = threadIdx.x, tx = tid & 7, ty = tid >> 3;
    const long long m0 = (long long)blockIdx.x * BM, n0 = (long long)blockIdx.y * BN;
    // neighbouring threads load along the contiguous direction
    const bool a_k = sak == 1, b_k = sbk == 1;
    double acc[TM][TN];
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TN; ++j) acc[i][j] = 0.0;
    double pa[NA], pb[NB];
    auto load = [&](unsigned k0) {
#pragma unroll
        for (int r = 0; r < NA; ++r) {
            const int idx = tid + 256 * r;
            const int mm = a_k ? idx / GK : idx % BM, kk = a_k ? idx % GK : idx / BM;
            pa[r] = (m0 + mm < M && k0 + kk < kend) ? __ldg(A + (m0 + mm) * sam + (long long)(k0 + kk) * sak) : 0.0;
        }
#pragma unroll
        for (int r = 0; r < NB; ++r) {
            const int idx = tid + 256 * r;
            const int nn = b_k ? idx / GK : idx % BN, kk = b_k ? idx % GK : idx / BN;
            pb[r] = (idx < BN * GK && n0 + nn < N && k0 + kk < kend)
                        ? __ldg(B + (long long)(k0 + kk) * sbk + (n0 + nn) * sbn)
                        : 0.0;
        }
    };
    if (kbeg < kend) load(kbeg);
    for (unsigned k0 = kbeg; k0 < kend; k0 += GK) {
        __syncthreads();
#pragma unroll
        for (int r = 0; r < NA; ++r) {
            const int idx = tid + 256 * r;
            const int mm = a_k ? idx / GK : idx % BM, kk = a_k ? idx % GK : idx / BM;
            As[kk][mm] = pa[r];
        }
#pragma unroll
        for (int r = 0; r < NB; ++r) {
            const int idx = tid + 256 * r;
            const int nn = b_k ? idx / GK : idx % BN, kk = b_k ? idx % GK : idx / BN;
            if (idx < BN * GK) Bs[kk][nn] = pb[r];
        }
        __syncthreads();
        if (k0 + GK < kend) load(k0 + GK);
        const int nk = (int)min((unsigned)GK, kend - k0);
        for (int kk = 0; kk < nk; ++kk) {
            double a[TM], b[TN];
#pragma unroll
            for (int i = 0; i < TM; ++i) a[i] = As[kk][ty + 32 * i];
#pragma unroll
            for (int j = 0; j < TN; ++j) b[j] = Bs[kk][tx + 8 * j];
#pragma unroll
            for (int i = 0; i < TM; ++i)
#pragma unroll
                for (int j = 0; j < TN; ++j) acc[i][j] = fma(a[i], b[j], acc[i][j]);
        }
    }
#pragma unroll
    for (int i = 0; i < TM; ++i) {
        const long long gm = m0 + ty + 32 * i;
        if (gm >= M) continue;
#pragma unroll
        for (int j = 0; j < TN; ++j) {
            const long long gn = n0 + tx + 8 * j;
            if (gn >= N) continue;
            double* c = C + (size_t)gm * ldc + gn;
            const double v = alpha * acc[i][j];
            *c = (beta == 0.0) ? v : fma(beta, *c, v);
        }
    }
}
__global__ void k_splitk_reduce(const double* __restrict__ P, int splits, int M, int N, double alpha,
                                double beta, double* __restrict__ C, int ldc) {
    dep_wait(P, C);
    const size_t total = (size_t)M * N;
    for (size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x; t < total; t += (size_t)gridDim.x * blockDim.x) {
        double acc = 0.0;
#pragma unroll 8
        for (int z = 0; z < splits; ++z) acc += P[(size_t)z * total + t];
        const size_t r = t / N, c = t % N;
        double* cp = C + r * ldc + c;
        *cp = (beta == 0.0) ? alpha * acc : fma(beta, *cp, alpha * acc);
    }
}

// A few rows times one vector over a long K (the one-site density matrix: d^2
// rows of chi^2 D^4): bound by reading A once.  Every CTA takes a K range and
// all rows; the partials [CTA][row] are summed by one warp per row in fixed
// order.  At d=3, D=8, chi=128 (9 x 1 x 67M; one 64 x 64 tile split 304 ways
// before) the one-site density matrix went from 463 to 23 ms, and to 11 with its
// permutes by boxes.  Shorter K, and
// calls without a workspace, stay with the tiles.
constexpr int GEMV_ROWS = 16;
constexpr int GEMV_CTAS = 152 * 4;
__global__ void __launch_bounds__(256) k_gemv_long(int M, int K, const double* __restrict__ A, int lda,
                                                   const double* __restrict__ x, int incx, double* __restrict__ P) {
    dep_wait(A, x, P);
    __shared__ double sm[8][GEMV_ROWS];
    double acc[GEMV_ROWS];
#pragma unroll
    for (int m = 0; m < GEMV_ROWS; ++m) acc[m] = 0.0;
    for (long long k = blockIdx.x * 256ll + threadIdx.x; k < K; k += (long long)gridDim.x * 256) {
        const double xv = __ldg(x + k * incx);
#pragma unroll
        for (int m = 0; m < GEMV_ROWS; ++m)
            if (m < M) acc[m] = fma(__ldg(A + (size_t)m * lda + k), xv, acc[m]);
    }
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
    for (int m = 0; m < GEMV_ROWS; ++m) {
        if (m < M) {
            for (int o = 16; o > 0; o >>= 1) acc[m] += __shfl_xor_sync(0xffffffffu, acc[m], o);
            if (lane == 0) sm[w][m] = acc[m];
        }
    }
    __syncthreads();
    if (threadIdx.x < M) {
        double t = 0.0;
        for (int i = 0; i < 8; ++i) t += sm[i][threadIdx.x];
        P[(size_t)blockIdx.x * M + threadIdx.x] = t;
    }
}

__global__ void k_gemv_sum(const double* __restrict__ P, int parts, int M, double alpha, double beta,
                           double* __restrict__ C, int ldc) {
    dep_wait(P, C);
    const int m = threadIdx.x >> 5, lane = threadIdx.x & 31;
    double t = 0.0;
#pragma unroll 4
    for (int z = lane; z < parts; z += 32) t += P[(size_t)z * M + m];
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if (lane == 0) {
        double* cp = C + (size_t)m * ldc;
        *cp = (beta == 0.0) ? alpha * t : fma(beta, *cp, alpha * t);
    }
}

struct GemmArgs64 {
    int M, N, K;
    double alpha;
    const double* A;
    long long sam, sak;
    const double* B;
    long long sbk, sbn;
    double beta;
    double* C;
    int ldc, kchunk;
    size_t zs;
};
template <int TM, int TN>
void launch(dim3 g, cudaStream_t s, const GemmArgs64& a) {
    launch_dep(k_dgemm<TM, TN>, g, 256, 0, s, a.M, a.N, a.K, a.alpha, a.A, a.sam, a.sak, a.B, a.sbk, a.sbn, a.beta, a.C,
               a.ldc, a.kchunk, a.zs);
}
template <int TM>
void launch_tn(int tn, dim3 g, cudaStream_t s, const GemmArgs64& a) {
    switch (tn) {
        case 1: launch<TM, 1>(g, s, a); break;
        case 2: launch<TM, 2>(g, s, a); break;
        case 3: launch<TM, 3>(g, s, a); break;
        case 4: launch<TM, 4>(g, s, a); break;
        case 5: launch<TM, 5>(g, s, a); break;
        case 6: launch<TM, 6>(g, s, a); break;
        case 7: launch<TM, 7>(g, s, a); break;
        case 8: launch<TM, 8>(g, s, a); break;
        default: launch<TM, 9>(g, s, a); break;
    }
}
}  // namespace

cudaError_t dgemm(bool tA, bool tB, int M, int N, int K, double alpha, const double* A, int lda,
                  const double* B, int ldb, double beta, double* C, int ldc, cudaStream_t s, double* ws,
                  size_t ws_doubles) {
    if (M <= 0 || N <= 0) return cudaSuccess;
    if (N > DGEMM_MAX_N) return cudaErrorInvalidValue;
    if (N == 1 && !tA && M <= GEMV_ROWS && K >= (1 << 16) && ws && ws_doubles >= (size_t)GEMV_CTAS * M) {
        launch_dep(k_gemv_long, GEMV_CTAS, 256, 0, s, M, K, A, lda, B, tB ? 1 : ldb, ws);
        launch_dep(k_gemv_sum, 1, 32 * M, 0, s, ws, GEMV_CTAS, M, alpha, beta, C, ldc);
        return cudaGetLastError();
    }
    const GemmPlan p = dgemm_plan(M, N, K, ws ? ws_doubles : 0);
    const dim3 grid((unsigned)((M + 32 * p.tm - 1) / (32 * p.tm)), (unsigned)((N + 8 * p.tn - 1) / (8 * p.tn)),
                    (unsigned)p.splits);
    GemmArgs64 a{M, N, K, alpha, A, tA ? 1 : lda, tA ? lda : 1, B, tB ? 1 : ldb, tB ? ldb : 1, beta, C, ldc,
                 p.splits > 1 ? p.kchunk : std::max(K, 1), (size_t)M * N};
    if (p.splits > 1) {
        a.C = ws;
        a.ldc = N;
        a.alpha = 1.0;
        a.beta = 0.0;
    }
    switch (p.tm) {
        case 1: launch_tn<1>(p.tn, grid, s, a); break;
        case 2: launch_tn<2>(p.tn, grid, s, a); break;
        default: launch_tn<4>(p.tn, grid, s, a); break;
    }
    if (p.splits > 1) {
        size_t blocks = ((size_t)M * N + 255) / 256;
        if (blocks > 152 * 8) blocks = 152 * 8;
        launch_dep(k_splitk_reduce, (unsigned)blocks, 256, 0, s, ws, p.splits, M, N, alpha, beta, C, ldc);
    }
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Axis permutation by boxes: bound by reading and writing each element once.
// A CTA takes boxes of up to 2048 elements that are contiguous for about 32
// elements both along the source's innermost axes and along the
// destination's.  A box is read in source order by asynchronous 8-byte copies
// into one of three buffers of shared memory, two boxes ahead, and written in
// destination order.  The offsets of a thread's eight elements inside a box are
// the same for every box: they are worked out once and kept in registers, and
// only the box's own origin is decoded per box.  8192 x 8192 transposed in 193 us
// (5.6 TB/s), (36864,9,8,8,64) by (1,0,3,2,4) in 3757 us (5.8 TB/s); the gather
// below, one thread per element with a division for each axis, took 353 and
// 6863 us.  Small arrays still go by the gather.
// ---------------------------------------------------------------------------
namespace {
// One thread per destination element: the source offset from its multi-index.
struct GatherArgs {
    int n;
    unsigned dim[8], stride[8];  // in destination order; source strides
};
__global__ void k_permute_gather(const double* __restrict__ src, double* __restrict__ dst, unsigned total,
                                 const GatherArgs p) {
    dep_wait(src, dst);
    const unsigned o = blockIdx.x * 256 + threadIdx.x;
    if (o >= total) return;
    unsigned rem = o, off = 0;
    for (int a = p.n - 1; a >= 0; --a) {
        const unsigned q = rem / p.dim[a];
        off += (rem - q * p.dim[a]) * p.stride[a];
        rem = q;
    }
    dst[o] = __ldg(src + off);
}

// A source that is already in destination order, eight loads of a thread in
// flight: bound by memory, 4e7 elements in 103 us (6.2 TB/s).
constexpr int COPY_CTAS = 8;  // resident on an SM
__global__ void __launch_bounds__(256, COPY_CTAS) k_copy(const double* __restrict__ src, double* __restrict__ dst,
                                                        unsigned total) {
    dep_wait(src, dst);
    constexpr unsigned U = 8;
    const unsigned long long step = gridDim.x * 256ull * U;
    for (unsigned long long b = blockIdx.x * 256ull * U + threadIdx.x; b < total; b += step) {
        double v[U];
#pragma unroll
        for (unsigned u = 0; u < U; ++u)
            if (b + u * 256 < total) v[u] = __ldg(src + b + u * 256);
#pragma unroll
        for (unsigned u = 0; u < U; ++u)
            if (b + u * 256 < total) dst[b + u * 256] = v[u];
    }
}

constexpr int PERM_THREADS = 256;
constexpr int PERM_EPT = 8;
constexpr int PERM_BOX = PERM_THREADS * PERM_EPT;
constexpr int PERM_STAGES = 3;
constexpr int PERM_CTAS = 4;      // resident on an SM
constexpr int PERM_EXTENT = 512;  // of a box along one axis: an index has 9 bits and a guard bit
constexpr unsigned PERM_GUARD = 0x20080200u;

// Position in shared memory: conflict-free for strides of powers of two.
__host__ __device__ constexpr int perm_swz(int p) { return p + (p >> 4) + (p >> 8); }

// An axis of the box; x / ext is the high word of x * mag (x < 2^11).
struct PermIn {
    unsigned mag, ext, stride, pos, shift;  // shift of its index among the cut axes' (31: not cut)
};
struct PermOut {
    unsigned n, ss, ds, ext, dim, shift;  // boxes along the axis, strides from box to box
};
struct PermPlan {
    int n_in, n_out, total;   // total: elements of a box
    int tile;                 // doubles of a buffer
    bool cut;                 // some box reaches over an edge
    PermIn src[8], dst[8];    // axes of more than one element of a box, innermost first
    PermOut out[8];           // axes of more than one box
    unsigned boxes;
};

__device__ __forceinline__ unsigned perm_digits(const PermIn* ax, int n, unsigned q, unsigned& off, unsigned& pos) {
    unsigned idx = 0;
    off = 0;
    pos = 0;
    for (int j = 0; j < n; ++j) {
        const unsigned t = __umulhi(q, ax[j].mag), x = q - t * ax[j].ext;
        q = t;
        off += x * ax[j].stride;
        pos += x * ax[j].pos;
        if (ax[j].shift != 31) idx |= x << ax[j].shift;
    }
    return idx;
}

__global__ void __launch_bounds__(PERM_THREADS, PERM_CTAS)
k_permute(const double* __restrict__ src, double* __restrict__ dst, const __grid_constant__ PermPlan p) {
    extern __shared__ double perm_tile[];
    unsigned soff[PERM_EPT], doff[PERM_EPT], sidx[PERM_EPT], didx[PERM_EPT], spos[PERM_EPT];
#pragma unroll
    for (int i = 0; i < PERM_EPT; ++i) {
        const unsigned e = threadIdx.x + i * PERM_THREADS;
        unsigned pos;
        if (i * PERM_THREADS >= p.total) break;
        didx[i] = perm_digits(p.dst, p.n_in, e, doff[i], pos);
        sidx[i] = perm_digits(p.src, p.n_in, e, soff[i], pos);
        spos[i] = (unsigned)__cvta_generic_to_shared(perm_tile + perm_swz((int)pos));
    }
    dep_wait(src, dst);
    // origin of box o in source and destination, and the last index inside the
    // array along the cut axes
    auto origin = [&](unsigned o, unsigned& sb, unsigned& db, unsigned& lim) {
        sb = db = 0;
        lim = PERM_GUARD | 0x1ff7fdffu;
        for (int j = 0; j < p.n_out; ++j) {
            const unsigned q = o / p.out[j].n, t = o - q * p.out[j].n;
            o = q;
            sb += t * p.out[j].ss;
            db += t * p.out[j].ds;
            if (p.out[j].shift != 31) {
                const unsigned last = min(p.out[j].dim - t * p.out[j].ext, (unsigned)PERM_EXTENT) - 1;
                lim = (lim & ~(0x1ffu << p.out[j].shift)) | last << p.out[j].shift;
            }
        }
    };
    auto load = [&](unsigned o, int stage) {
        if (o < p.boxes) {
            unsigned sb, db, lim;
            origin(o, sb, db, lim);
#pragma unroll
            for (int i = 0; i < PERM_EPT; ++i)
                if (threadIdx.x + i * PERM_THREADS < p.total &&
                    (!p.cut || ((lim - sidx[i]) & PERM_GUARD) == PERM_GUARD))
                    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(
                                     spos[i] + stage * p.tile * (int)sizeof(double)),
                                 "l"(src + (sb + soff[i]))
                                 : "memory");
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    unsigned next = blockIdx.x;
    int ls = 0, cs = 0;
    for (; ls < PERM_STAGES - 1; ++ls, next += gridDim.x) load(next, ls);
    for (unsigned o = blockIdx.x; o < p.boxes; o += gridDim.x) {
        asm volatile("cp.async.wait_group %0;" ::"n"(PERM_STAGES - 2) : "memory");
        __syncthreads();
        load(next, ls);
        next += gridDim.x;
        ls = ls + 1 == PERM_STAGES ? 0 : ls + 1;
        unsigned sb, db, lim;
        origin(o, sb, db, lim);
        const double* t = perm_tile + cs * p.tile;
        cs = cs + 1 == PERM_STAGES ? 0 : cs + 1;
#pragma unroll
        for (int i = 0; i < PERM_EPT; ++i) {
            const int e = threadIdx.x + i * PERM_THREADS;
            if (e < p.total && (!p.cut || ((lim - didx[i]) & PERM_GUARD) == PERM_GUARD))
                dst[db + doff[i]] = t[perm_swz(e)];
        }
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
}

// The limit of k_permute's shared memory, for its largest box: an attribute of
// the function on a device, not of a launch or a host thread, so it is set
// once for each device.  (Set to every call's own size, another thread's call
// could lower it between this one's setting and its launch.)
cudaError_t permute_attributes() {
    static std::mutex mu;
    static unsigned long long done = 0;  // a bit per device
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(mu);
    if (done >> dev & 1ull) return cudaSuccess;
    constexpr int most = PERM_STAGES * (perm_swz(PERM_BOX - 1) + 1) * (int)sizeof(double);
    e = cudaFuncSetAttribute(k_permute, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
    if (e == cudaSuccess) done |= 1ull << dev;
    return e;
}
}  // namespace

cudaError_t permute(const double* src, double* dst, int ndim, const int* dims, const int* perm,
                    cudaStream_t s) {
    if (ndim < 1 || ndim > 8) return cudaErrorInvalidValue;
    unsigned long long sstride[8];
    unsigned long long total = 1;
    for (int a = ndim - 1; a >= 0; --a) {
        sstride[a] = total;
        total *= (unsigned long long)dims[a];
    }
    if (total == 0) return cudaSuccess;
    if (total >= (1ull << 32)) return cudaErrorInvalidValue;
    // destination axes, those of one element dropped and neighbours that are
    // neighbours in the source too merged
    int n = 0, by_src[8];
    unsigned dim[8], ss[8], ds[8], box[8], pos[8];
    for (int b = 0; b < ndim; ++b) {
        const unsigned d = (unsigned)dims[perm[b]], st = (unsigned)sstride[perm[b]];
        if (d == 1) continue;
        if (n && ss[n - 1] == st * d && (unsigned long long)dim[n - 1] * d < (1ull << 31)) {
            dim[n - 1] *= d;
            ss[n - 1] = st;
        } else {
            dim[n] = d;
            ss[n] = st;
            ++n;
        }
    }
    // Below 2^18 elements the gather: 1.5 to 4.0 us there, where the boxes' set-up
    // makes it 2.2 to 5.0; 4.6 us either way at 2^18, 13.7 and 10.7 at 1.4e6,
    // 361 and 193 at 6.7e7.
    if (total < (1ull << 18)) {
        GatherArgs g;
        g.n = n;
        for (int a = 0; a < n; ++a) {
            g.dim[a] = dim[a];
            g.stride[a] = ss[a];
        }
        launch_dep(k_permute_gather, (unsigned)((total + 255) / 256), 256, 0, s, src, dst, (unsigned)total, g);
        return cudaGetLastError();
    }
    // already in destination order: boxes (180 us for 4e7 elements) have nothing to reorder
    if (n <= 1) {
        launch_dep(k_copy, 152 * COPY_CTAS, 256, 0, s, src, dst, (unsigned)total);
        return cudaGetLastError();
    }
    unsigned st = 1;
    for (int a = n - 1; a >= 0; --a) {
        ds[a] = st;
        st *= dim[a];
        box[a] = 1;
        by_src[a] = a;
    }
    std::sort(by_src, by_src + n, [&](int x, int y) { return ss[x] < ss[y]; });
    auto size = [&] {
        unsigned t = 1;
        for (int a = 0; a < n; ++a) t *= box[a];
        return t;
    };
    // the extent of at most e that cuts an axis into even boxes
    auto even = [&](int a, unsigned e) {
        e = std::min({e, dim[a], (unsigned)PERM_EXTENT});
        const unsigned parts = (dim[a] + e - 1) / e;
        return (dim[a] + parts - 1) / parts;
    };
    // about `want` consecutive elements on one side (at most twice as many)
    auto grow = [&](auto axis_at, unsigned want) {
        unsigned long long prod = 1;
        for (int j = 0; j < n && prod < want; ++j) {
            const int a = axis_at(j);
            box[a] = std::max(box[a], even(a, prod * dim[a] <= 2 * want ? dim[a] : (unsigned)((want + prod - 1) / prod)));
            if (box[a] < dim[a]) break;
            prod *= box[a];
        }
    };
    grow([&](int j) { return n - 1 - j; }, 32);
    unsigned keep[8];
    std::copy(box, box + n, keep);
    grow([&](int j) { return by_src[j]; }, 32);
    if (size() > PERM_BOX) {
        std::copy(keep, keep + n, box);
        grow([&](int j) { return by_src[j]; }, 16);
    }
    // then as much of the innermost axes as a box holds, three cut axes at most;
    // smaller boxes where every SM would not have two
    const unsigned most_box =
        (unsigned)std::min<unsigned long long>(PERM_BOX, std::max<unsigned long long>(PERM_BOX / 2, total / (152 * 2)));
    for (int a = n - 1; a >= 0; --a) {
        const unsigned old = box[a], most = even(a, std::max(1u, most_box / (size() / old)));
        box[a] = std::max(old, most);
        int cuts = 0;
        for (int c = 0; c < n; ++c) cuts += dim[c] % box[c] != 0;
        if (cuts > 3) box[a] = old;
    }
    PermPlan p{};
    p.total = (int)size();
    p.tile = perm_swz(p.total - 1) + 1;
    unsigned w = 1, shift[8], bits = 0;
    for (int a = n - 1; a >= 0; --a) {
        pos[a] = w;
        w *= box[a];
        shift[a] = 31;
        if (dim[a] % box[a]) {
            shift[a] = 10 * bits++;
            p.cut = true;
        }
    }
    if (bits > 3 || p.total > PERM_BOX) return cudaErrorInvalidValue;
    unsigned long long boxes = 1;
    for (int j = 0; j < n; ++j) {
        const int a = n - 1 - j, c = by_src[j];
        const unsigned parts = (dim[a] + box[a] - 1) / box[a];
        boxes *= parts;
        if (parts > 1) p.out[p.n_out++] = {parts, box[a] * ss[a], box[a] * ds[a], box[a], dim[a], shift[a]};
        auto in = [&](int x, unsigned stride) {
            return PermIn{(unsigned)(((1ull << 32) + box[x] - 1) / box[x]), box[x], stride, pos[x], shift[x]};
        };
        if (box[a] > 1) p.dst[p.n_in++] = in(a, ds[a]);
        int k = 0;
        for (int i = 0; i < j; ++i) k += box[by_src[i]] > 1;
        if (box[c] > 1) p.src[k] = in(c, ss[c]);
    }
    p.boxes = (unsigned)boxes;
    const int smem = PERM_STAGES * p.tile * (int)sizeof(double);
    const cudaError_t e = permute_attributes();
    if (e != cudaSuccess) return e;
    launch_dep(k_permute, (unsigned)std::min<unsigned long long>(boxes, 152 * PERM_CTAS), PERM_THREADS, smem, s, src, dst, p);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// elementwise helpers
// ---------------------------------------------------------------------------
namespace {
__global__ void k_scale_cols(double* X, int rows, int cols, int ld, const double* __restrict__ w) {
    dep_wait(X, w);
    const size_t total = (size_t)rows * cols;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x) {
        const int r = (int)(i / cols), c = (int)(i % cols);
        X[(size_t)r * ld + c] *= w[c];
    }
}
__global__ void k_inv_sqrt_cut(const double* __restrict__ sv, double* __restrict__ w, int n, double cut) {
    dep_wait(sv, w);
    const double s0 = sv[0];
    for (int j = threadIdx.x; j < n; j += blockDim.x) {
        const double v = sv[j];
        w[j] = (s0 > 0.0 && v > cut * s0) ? 1.0 / sqrt(v) : 0.0;
    }
}
__global__ void k_maxabs(const double* __restrict__ x, size_t n, unsigned long long* maxbits) {
    dep_wait(x, maxbits);
    double m = 0.0;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
        const double a = fabs(x[i]);
        // NaN compares false: force it through as the largest bit pattern
        m = (a > m || a != a) ? a : m;
    }
    unsigned long long b = __double_as_longlong(m);
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long t = __shfl_xor_sync(0xffffffffu, b, o);
        b = t > b ? t : b;
    }
    __shared__ unsigned long long sm[32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (lane == 0) sm[w] = b;
    __syncthreads();
    if (w == 0) {
        b = (lane < (int)(blockDim.x >> 5)) ? sm[lane] : 0ull;
        for (int o = 16; o > 0; o >>= 1) {
            const unsigned long long t = __shfl_xor_sync(0xffffffffu, b, o);
            b = t > b ? t : b;
        }
        if (lane == 0) atomicMax(maxbits, b);
    }
}
__global__ void k_scale_by_max(double* x, size_t n, const unsigned long long* maxbits, int* flag) {
    dep_wait(x, maxbits, flag);
    const unsigned long long b = *maxbits;
    if (b >= 0x7ff0000000000000ull) {  // Inf or NaN
        if (blockIdx.x == 0 && threadIdx.x == 0) atomicExch(flag, 1);
        return;
    }
    const double m = __longlong_as_double((long long)b);
    if (m == 0.0) {  // an all-zero tensor: the projectors have collapsed
        if (blockIdx.x == 0 && threadIdx.x == 0) atomicCAS(flag, 0, 2);
        return;
    }
    const double inv = 1.0 / m;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
        x[i] *= inv;
}

// Philox4x32-10 (Salmon, Moraes, Dror, Shaw, SC'11), written from the
// published definition: 10 rounds of two 32x32->64 multiplies with the
// key bumped by the Weyl constants between rounds.
__device__ __forceinline__ uint4 philox4x32_10(uint4 c, uint2 k) {
    const unsigned M0 = 0xD2511F53u, M1 = 0xCD9E8D57u, W0 = 0x9E3779B9u, W1 = 0xBB67AE85u;
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        if (r) { k.x += W0; k.y += W1; }
        const unsigned hi0 = __umulhi(M0, c.x), lo0 = M0 * c.x;
        const unsigned hi1 = __umulhi(M1, c.z), lo1 = M1 * c.z;
        c = make_uint4(hi1 ^ c.y ^ k.x, lo1, hi0 ^ c.w ^ k.y, lo0);
    }
    return c;
}
__global__ void k_rng_normal(double* __restrict__ out, size_t n, uint64_t seed, uint64_t sid) {
    const size_t pairs = (n + 1) / 2;
    for (size_t p = blockIdx.x * (size_t)blockDim.x + threadIdx.x; p < pairs; p += (size_t)gridDim.x * blockDim.x) {
        const uint4 r = philox4x32_10(make_uint4((unsigned)p, (unsigned)(p >> 32), (unsigned)sid, (unsigned)(sid >> 32)),
                                      make_uint2((unsigned)seed, (unsigned)(seed >> 32)));
        // two 53-bit uniforms; u1 in (0, 1] for the logarithm
        const double u1 = 1.0 - (double)(((unsigned long long)(r.x >> 5) << 26) | (r.y >> 6)) * 0x1.0p-53;
        const double u2 = (double)(((unsigned long long)(r.z >> 5) << 26) | (r.w >> 6)) * 0x1.0p-53;
        const double rad = sqrt(-2.0 * log(u1));
        double sn, cs;
        sincospi(2.0 * u2, &sn, &cs);
        out[2 * p] = rad * cs;
        if (2 * p + 1 < n) out[2 * p + 1] = rad * sn;
    }
}
// Dot product in two passes with a fixed grid, so the summation order (and
// the result) does not depend on scheduling: pass 1 leaves one partial per
// block, pass 2 (one block) adds them in block order.
constexpr int DOT_BLOCKS = 152 * 4;
__global__ void k_dot_partial(const double* __restrict__ x, const double* __restrict__ y, size_t n,
                              double* __restrict__ part) {
    dep_wait(x, y, part);
    double acc = 0.0;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
        acc = fma(x[i], y[i], acc);
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    __shared__ double sm[32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (lane == 0) sm[w] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int i = 0; i < (int)(blockDim.x >> 5); ++i) t += sm[i];
        part[blockIdx.x] = t;
    }
}
__global__ void k_dot_final(const double* __restrict__ part, int np, double* __restrict__ out) {
    dep_wait(part, out);
    __shared__ double sm[256];
    double t = 0.0;
    for (int i = threadIdx.x; i < np; i += blockDim.x) t += part[i];
    sm[threadIdx.x] = t;
    __syncthreads();
    if (threadIdx.x == 0) {
        double s = 0.0;
        for (int i = 0; i < (int)blockDim.x; ++i) s += sm[i];
        *out = s;
    }
}
// T[a,k,k',b] <- (T[a,k,k',b] + T[a,k',k,b]) / 2, one thread per pair k <= k'
__global__ void k_sym_kk(double* __restrict__ T, int chi, int D) {
    dep_wait(T);
    const size_t total = (size_t)chi * D * D * chi;
    for (size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x; t < total; t += (size_t)gridDim.x * blockDim.x) {
        const size_t b = t % chi, kk2 = (t / chi) % D, kk = (t / ((size_t)chi * D)) % D, a = t / ((size_t)chi * D * D);
        if (kk > kk2) continue;
        const size_t i1 = ((a * D + kk) * D + kk2) * chi + b, i2 = ((a * D + kk2) * D + kk) * chi + b;
        const double v = 0.5 * (T[i1] + T[i2]);
        T[i1] = v;
        T[i2] = v;
    }
}
inline unsigned grid_for(size_t n, unsigned threads = 256) {
    size_t b = (n + threads - 1) / threads;
    if (b > 152 * 32) b = 152 * 32;
    if (b == 0) b = 1;
    return (unsigned)b;
}
// dst[i][j] += src[i][j] for a rows x cols block (row strides lds, ldd)
__global__ void k_add_block(const double* __restrict__ src, int rows, int cols, int lds, double* __restrict__ dst,
                            int ldd) {
    dep_wait(src, dst);
    const size_t total = (size_t)rows * cols;
    for (size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x; t < total; t += (size_t)gridDim.x * blockDim.x) {
        const int i = (int)(t / cols), j = (int)(t % cols);
        dst[(size_t)i * ldd + j] += src[(size_t)i * lds + j];
    }
}
}  // namespace

cudaError_t add_block(const double* src, int rows, int cols, int lds, double* dst, int ldd, cudaStream_t s) {
    if (rows <= 0 || cols <= 0) return cudaSuccess;
    launch_dep(k_add_block, grid_for((size_t)rows * cols), 256, 0, s, src, rows, cols, lds, dst, ldd);
    return cudaGetLastError();
}

cudaError_t scale_cols(double* X, int rows, int cols, int ld, const double* w, cudaStream_t s) {
    if (rows <= 0 || cols <= 0) return cudaSuccess;
    launch_dep(k_scale_cols, grid_for((size_t)rows * cols), 256, 0, s, X, rows, cols, ld, w);
    return cudaGetLastError();
}
cudaError_t inv_sqrt_cut(const double* sv, double* w, int n, double cut, cudaStream_t s) {
    launch_dep(k_inv_sqrt_cut, 1, 256, 0, s, sv, w, n, cut);
    return cudaGetLastError();
}
cudaError_t maxabs(const double* x, size_t n, unsigned long long* maxbits, cudaStream_t s) {
    if (!n) return cudaSuccess;
    launch_dep(k_maxabs, grid_for(n), 256, 0, s, x, n, maxbits);
    return cudaGetLastError();
}
cudaError_t scale_by_max(double* x, size_t n, const unsigned long long* maxbits, int* flag, cudaStream_t s) {
    if (!n) return cudaSuccess;
    launch_dep(k_scale_by_max, grid_for(n), 256, 0, s, x, n, maxbits, flag);
    return cudaGetLastError();
}
// FP64 FMA throughput probe: every thread runs 8 independent FMA chains
// (enough in flight to keep the pipe busy); the result is stored so the
// chains are not optimised away.
__global__ void k_dfma_probe(double* __restrict__ out, int iters, double a, double b) {
    double x[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) x[u] = (double)(threadIdx.x + u) * 1e-3;
    for (int it = 0; it < iters; ++it)
#pragma unroll
        for (int u = 0; u < 8; ++u) x[u] = fma(x[u], a, b);
    double s = 0.0;
#pragma unroll
    for (int u = 0; u < 8; ++u) s += x[u];
    out[blockIdx.x * blockDim.x + threadIdx.x] = s;
}

// out[m] = trace of the n x n matrix As + m n^2, m < nm (one warp per matrix)
__global__ void k_traces(const double* __restrict__ As, int n, int nm, double* __restrict__ out) {
    dep_wait(As, out);
    const int m = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (m >= nm) return;
    const double* a = As + (size_t)m * n * n;
    double t = 0.0;
    for (int i = lane; i < n; i += 32) t += a[(size_t)i * (n + 1)];
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if (lane == 0) out[m] = t;
}

size_t dot_ws_doubles() { return DOT_BLOCKS; }
cudaError_t dot(const double* x, const double* y, size_t n, double* out, double* ws, cudaStream_t s) {
    launch_dep(k_dot_partial, DOT_BLOCKS, 256, 0, s, x, y, n, ws);
    launch_dep(k_dot_final, 1, 256, 0, s, ws, DOT_BLOCKS, out);
    return cudaGetLastError();
}
cudaError_t traces(const double* As, int n, int nm, double* out, cudaStream_t s) {
    launch_dep(k_traces, (nm + 7) / 8, 256, 0, s, As, n, nm, out);
    return cudaGetLastError();
}
cudaError_t dfma_probe(double* out, int blocks, int threads, int iters, cudaStream_t s) {
    ++g_launches;
    k_dfma_probe<<<blocks, threads, 0, s>>>(out, iters, 0.999999, 1e-7);
    return cudaGetLastError();
}
cudaError_t sym_kk(double* T, int chi, int D, cudaStream_t s) {
    launch_dep(k_sym_kk, grid_for((size_t)chi * D * D * chi), 256, 0, s, T, chi, D);
    return cudaGetLastError();
}
cudaError_t rng_normal(double* out, size_t n, uint64_t seed, uint64_t sid, cudaStream_t s) {
    if (!n) return cudaSuccess;
    ++g_launches;
    k_rng_normal<<<grid_for((n + 1) / 2), 256, 0, s>>>(out, n, seed, sid);
    return cudaGetLastError();
}

}  // namespace ctm
