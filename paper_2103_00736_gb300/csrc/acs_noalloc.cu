// KKT residuals of a caller-supplied point without any allocation.
//
// Some callers cannot allocate device memory: code that runs inside another
// framework's memory pool or under a fixed memory budget, real-time loops that
// must not enter the allocator, and drivers that hand over only pre-allocated
// buffers.  This entry point serves them: the caller passes every input and the
// output in device memory it already owns, and the temporary data of the
// computation live in one file-scope device array of fixed size that every GPU
// which loads this library holds until the process exits.
//
// Scratch layout (doubles): two for the counter of finished blocks, kMaxN entries
// for A'y, then kMaxBlocks x 8 block partials.  A'y is accumulated by scattering
// the rows of A (atomic adds), so its summation order, and hence the last bits
// of r_d, may differ from call to call.  The accumulator is cleared at the start
// of every call.  Calls that overlap on the GPU (different streams, or another
// thread) share the array and race; callers must order them.
//
// What bounds it, at n = 1e6 and 1e7 nonzeros: each nonzero is 12 bytes of the
// matrix (18 us of HBM), one random read of x, two FP64 operations (32 us of a
// pipe that does two multiply-adds per clock per SM) and one atomic add in L2.
// Eight lanes a row make the matrix reads coalesced and keep short rows from
// idling a warp; the last block of the second kernel combines the partials.
// Measured: n = 1e6 475 -> 155 us, n = 500 30 -> 18 us a call (before: a
// thread a row, and a fourth kernel in which one thread added up the partials).

#include <math.h>
#include <mutex>

#include "../../include/acs.h"

namespace {

constexpr int kMaxN = 1 << 20;                 // largest n accepted (1,048,576): 8 MiB of A'y
constexpr int kMaxBlocks = 1024;               // block partials: half for the rows, half for the columns
constexpr int kVals = 8;                       // partials per block
constexpr int kThreadsNA = 1024;
constexpr int kLanes = 8;                      // lanes a row of A, or a cone, is spread over
constexpr int kHead = 2;                       // doubles before A'y: the counter of finished blocks

__device__ __align__(256) double g_noalloc_scratch[kHead + kMaxN + kMaxBlocks * kVals];

std::mutex g_setup_mutex;

struct Args {
    int m, n, n_orth, n_soc;
    bool soc_short;                                // the mean cone has at most kLanes entries after its first
    const int *rp, *ci;
    const double *av, *b, *c, *x, *y, *z;
    const int* soc_off;
    double *aty, *prow, *pcol, *out;
    unsigned* done;
};

// Block-wide sums of NV <= 8 values; the first NV threads write them to out.
// Inside a warp a lane gives half of its values away at each of the first steps,
// so that eight values take nine additions a lane (the FP64 pipe is slow).
template <int NV>
__device__ __forceinline__ void block_sum_store(const double (&v)[NV], double* out) {
    constexpr int NP = NV <= 4 ? 4 : 8;
    __shared__ double sh[32][NP];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    double a[NP];
#pragma unroll
    for (int k = 0; k < NP; ++k) a[k] = k < NV ? v[k < NV ? k : 0] : 0.0;
    int o = 16;
#pragma unroll
    for (int c = NP; c > 1; c >>= 1, o >>= 1) {
        const bool up = (lane & o) != 0;
#pragma unroll
        for (int i = 0; i < c / 2; ++i) {
            const double give = up ? a[i] : a[i + c / 2], keep = up ? a[i + c / 2] : a[i];
            a[i] = keep + __shfl_xor_sync(0xffffffffu, give, o);
        }
    }
#pragma unroll
    for (; o > 0; o >>= 1) a[0] += __shfl_xor_sync(0xffffffffu, a[0], o);
    if ((lane & (32 / NP - 1)) == 0) sh[warp][lane / (32 / NP)] = a[0];
    __syncthreads();
    if (warp == 0) {
        // lane (k, q): value k, warps q, q + Q, ... (Q lanes a value)
        constexpr int Q = 32 / NP;
        const int k = lane / Q, q = lane % Q;
        double t = 0.0;
        for (int w = q; w < nw; w += Q) t += sh[w][k];
#pragma unroll
        for (int d = Q / 2; d > 0; d >>= 1) t += __shfl_xor_sync(0xffffffffu, t, d);
        if (q == 0 && k < NV) out[k] = t;
    }
}

__device__ __forceinline__ double lanes_sum(double x) {
#pragma unroll
    for (int o = kLanes / 2; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    return x;
}

// Rows of A, kLanes lanes a row: v += {||Ax - b||^2, b'y, ||b||^2}; y_i A_ij into
// aty[j].  t, nt: this thread and the number of threads.
__device__ __forceinline__ void rows_part(const Args& P, int t, int nt, double (&v)[3]) {
    const int l = t % kLanes;
    constexpr int U = 4;
    // every lane of a warp runs the same number of rounds (its rows past m are empty)
    for (unsigned i0 = (t & ~31) / kLanes; i0 < (unsigned)P.m; i0 += nt / kLanes) {
        const unsigned i = i0 + (t & 31) / kLanes;
        unsigned k = 0, e = 0;                           // k may pass e by a round: no overflow at 2^31
        double yi = 0.0;
        if (i < (unsigned)P.m) {
            k = P.rp[i] + l;
            e = P.rp[i + 1];
            yi = P.y[i];
        }
        double s = 0.0;
        for (; k < e; k += U * kLanes) {
            int j[U];
            double a[U], xj[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const bool in = k + u * kLanes < e;
                j[u] = in ? __ldcs(P.ci + k + u * kLanes) : -1;
                a[u] = in ? __ldcs(P.av + k + u * kLanes) : 0.0;
            }
#pragma unroll
            for (int u = 0; u < U; ++u) xj[u] = j[u] >= 0 ? P.x[j[u]] : 0.0;
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (j[u] >= 0) {
                    s = fma(a[u], xj[u], s);
                    atomicAdd(P.aty + j[u], a[u] * yi);
                }
        }
        s = lanes_sum(s);
        if (l == 0 && i < (unsigned)P.m) {
            const double bi = P.b[i], d = s - bi;
            v[0] += d * d;
            v[1] += bi * yi;
            v[2] += bi * bi;
        }
    }
}

__device__ __forceinline__ double soc_dist2_na(double v1, double t) {
    if (t <= v1) return 0.0;
    if (t <= -v1) return v1 * v1 + t * t;
    const double d = 0.5 * (t - v1);
    return 2.0 * d * d;
}

// Coordinates and cones: v += {||A'y + z - c||^2, c'x, ||x||^2, ||z||^2,
// dist(x,K)^2, dist(z,K)^2, ||c||^2}.
__device__ __forceinline__ void cols_part(const Args& P, int t, int nt, double (&v)[7]) {
    for (int j = t; j < P.n; j += nt) {
        const double xj = P.x[j], zj = P.z[j], cj = P.c[j];
        const double d = __ldcg(P.aty + j) + zj - cj;
        v[0] += d * d;
        v[6] += cj * cj;
        v[1] += cj * xj;
        const double xx = xj * xj, zz = zj * zj;
        v[2] += xx;
        v[3] += zz;
        if (j < P.n_orth) {
            if (xj < 0.0) v[4] += xx;
            if (zj < 0.0) v[5] += zz;
        }
    }
    if (P.n_soc == 0) return;
    // kLanes lanes a cone.  A root and a distance take the warp's FP64 instructions
    // whether 2 or 32 lanes need them, so warps are numbered across the blocks
    // first, and short cones (kLanes a group at a time) leave one cone to each lane
    // before the roots.  Measured, cones' share of a call: n = 600, 300 cones
    // of 2, 12 -> 4 us; n = 1e6, 5e5 cones of 2, 304 -> 53 us (before: eight lanes to
    // every cone, warps in order).
    const int lane = t & 31, l = lane % kLanes, g0 = lane - l;
    const unsigned n_soc = (unsigned)P.n_soc, w = (threadIdx.x >> 5) * gridDim.x + blockIdx.x, nw = nt >> 5;
    if (P.soc_short) {
        for (unsigned q0 = w * 32; q0 < n_soc; q0 += nw * 32) {
            const unsigned q = q0 + lane;
            int a = 0, e = 0;
            if (q < n_soc) {
                a = P.soc_off[q];
                e = P.soc_off[q + 1];
            }
            double sx[kLanes], sz[kLanes];
#pragma unroll
            for (int r = 0; r < kLanes; ++r) {           // the cone of lane g0 + r
                const int j = __shfl_sync(0xffffffffu, a, g0 + r) + 1 + l, er = __shfl_sync(0xffffffffu, e, g0 + r);
                const double xj = j < er ? P.x[j] : 0.0, zj = j < er ? P.z[j] : 0.0;
                sx[r] = xj * xj;
                sz[r] = zj * zj;
                for (int i = j + kLanes; i < er; i += kLanes) {
                    sx[r] = fma(P.x[i], P.x[i], sx[r]);
                    sz[r] = fma(P.z[i], P.z[i], sz[r]);
                }
            }
            int o = kLanes / 2;
#pragma unroll
            for (int c = kLanes; c > 1; c >>= 1, o >>= 1) {   // lane l keeps the sum of cone l
                const bool up = (l & o) != 0;
#pragma unroll
                for (int i = 0; i < c / 2; ++i) {
                    const double gx = up ? sx[i] : sx[i + c / 2], kx = up ? sx[i + c / 2] : sx[i];
                    const double gz = up ? sz[i] : sz[i + c / 2], kz = up ? sz[i + c / 2] : sz[i];
                    sx[i] = kx + __shfl_xor_sync(0xffffffffu, gx, o);
                    sz[i] = kz + __shfl_xor_sync(0xffffffffu, gz, o);
                }
            }
            if (q < n_soc) {
                v[4] += soc_dist2_na(P.x[a], sqrt(sx[0]));
                v[5] += soc_dist2_na(P.z[a], sqrt(sz[0]));
            }
        }
        return;
    }
    constexpr unsigned per = 32 / kLanes;
    for (unsigned q0 = w * per; q0 < n_soc; q0 += nw * per) {
        const unsigned q = q0 + lane / kLanes;
        int a = 0, e = 0;
        if (q < n_soc) {
            a = P.soc_off[q];
            e = P.soc_off[q + 1];
        }
        double sx = 0.0, sz = 0.0;
        for (int j = a + 1 + l; j < e; j += kLanes) {
            const double xj = P.x[j], zj = P.z[j];
            sx = fma(xj, xj, sx);
            sz = fma(zj, zj, sz);
        }
        sx = lanes_sum(sx);
        sz = lanes_sum(sz);
        if (q < n_soc && l < 2) {                        // lane 0 takes x, lane 1 z
            const double d = soc_dist2_na(l == 0 ? P.x[a] : P.z[a], sqrt(l == 0 ? sx : sz));
            if (l == 0) v[4] += d;
            else v[5] += d;
        }
    }
}

// One warp: the six residual values from the sums {||Ax - b||^2, b'y, ||b||^2,
// then those of cols_part}, the same in every lane.
__device__ __forceinline__ void write_residuals(const double (&s)[10], double* out) {
    const int lane = threadIdx.x & 31;
    const double by = s[1], cx = s[4];
    // lane 0: r_p, 1: r_d, 2: r_gap, 3: r_cone, as one quotient of each lane's own
    double num = lane == 1 ? s[3] : s[0], den = lane == 1 ? s[9] : s[2];
    if (lane == 3) {
        num = fmax(s[7], s[8]);                          // the root is monotone
        den = fmax(s[5], s[6]);
    }
    num = sqrt(num);
    den = 1.0 + sqrt(den);
    if (lane == 2) {
        num = fabs(cx - by);
        den = 1.0 + fabs(cx) + fabs(by);
    }
    double r = num / den;
    if (lane == 4) r = cx;
    if (lane == 5) r = by;
    if (lane < 6) out[lane] = r;
}

// One warp: add the blocks' partials (lane l those of blocks l, l + 32, ... in
// order, then a fixed shuffle tree) and write the six residual values.
__device__ __forceinline__ void finish_part(int nb_rows, int nb_cols, const double* prow, const double* pcol,
                                            double* out) {
    const int lane = threadIdx.x & 31;
    double s[10];
#pragma unroll
    for (int k = 0; k < 10; ++k) s[k] = 0.0;
    for (int i = lane; i < nb_rows; i += 32)
#pragma unroll
        for (int k = 0; k < 3; ++k) s[k] += __ldcg(prow + i * kVals + k);
    for (int i = lane; i < nb_cols; i += 32)
#pragma unroll
        for (int k = 0; k < 7; ++k) s[3 + k] += __ldcg(pcol + i * kVals + k);
#pragma unroll
    for (int k = 0; k < 10; ++k)
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s[k] += __shfl_xor_sync(0xffffffffu, s[k], o);
    write_residuals(s, out);
}

__global__ void __launch_bounds__(kThreadsNA) rows_kernel(const Args P) {
    double v[3] = {0.0, 0.0, 0.0};
    rows_part(P, blockIdx.x * blockDim.x + threadIdx.x, gridDim.x * blockDim.x, v);
    block_sum_store<3>(v, P.prow + blockIdx.x * kVals);
}

// The block that ends last combines all partials.
__global__ void __launch_bounds__(kThreadsNA) cols_kernel(const Args P, int nb_rows) {
    double v[7] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
    cols_part(P, blockIdx.x * blockDim.x + threadIdx.x, gridDim.x * blockDim.x, v);
    block_sum_store<7>(v, P.pcol + blockIdx.x * kVals);
    if (threadIdx.x >= 32) return;
    __threadfence();
    __syncwarp();
    unsigned last = 0;
    if (threadIdx.x == 0) last = atomicAdd(P.done, 1u) == gridDim.x - 1 ? 1u : 0u;
    if (!__shfl_sync(0xffffffffu, last, 0)) return;
    __threadfence();
    finish_part(nb_rows, (int)gridDim.x, P.prow, P.pcol, P.out);
}

// Device address of the scratch array in the current device's context,
// looked up on every call: a lookup is a host-side table query that
// allocates nothing, and a cached address would outlive the context it
// belongs to (after cudaDeviceReset the module is loaded again elsewhere).
// The first lookup in a context loads the module; the lock keeps concurrent
// first calls from racing in the runtime's lazy loading.
double* scratch_for_current_device(int* err) {
    std::lock_guard<std::mutex> lock(g_setup_mutex);
    double* p = nullptr;
    if (cudaGetSymbolAddress((void**)&p, g_noalloc_scratch) != cudaSuccess || !p) {
        *err = ACS_ERR_CUDA;
        return nullptr;
    }
    return p;
}

}  // namespace

extern "C" int acs_kkt_residuals_noalloc(int32_t m, int32_t n, const int32_t* row_ptr, const int32_t* col,
                                         const double* val, const double* b, const double* c, const double* x,
                                         const double* y, const double* z, int32_t n_orthant, int32_t n_soc,
                                         const int32_t* soc_offsets, double* residuals, void* cuda_stream) {
    if (m <= 0 || n <= 0 || !row_ptr || !col || !val || !b || !c || !x || !y || !z || !residuals ||
        n_orthant < 0 || n_soc < 0 || (n_soc > 0 && !soc_offsets) || n_orthant > n)
        return ACS_ERR_ARG;
    if (n > kMaxN) return ACS_ERR_LIMIT;
    // an error left by an earlier, unrelated launch is not this call's
    cudaGetLastError();
    int err = ACS_SOLVED;
    double* scratch = scratch_for_current_device(&err);
    if (!scratch) return err;
    const bool soc_short = (long long)n - n_orthant <= (long long)n_soc * (kLanes + 1);
    Args P{m, n, n_orthant, n_soc, soc_short, row_ptr, col, val, b, c, x, y, z, soc_offsets, scratch + kHead,
           scratch + kHead + kMaxN, scratch + kHead + kMaxN + (kMaxBlocks / 2) * kVals, residuals,
           reinterpret_cast<unsigned*>(scratch)};
    cudaStream_t st = (cudaStream_t)cuda_stream;
    // Blocks of 1024 threads, at most two on each of 152 SMs and never more than the
    // scratch has partials for; where 304 blocks of 256 hold everything at once, those:
    // the sums at a block's end take the FP64 pipe for each of its warps in turn.
    // Measured, 256 / 1024 threads: m = 1000, n = 600 19 / 26 us, m = 2000, n = 5000
    // 20 / 31.
    const long long most = 304 < kMaxBlocks / 2 ? 304 : kMaxBlocks / 2;
    const long long soc_block = soc_short ? 128 : 128 / kLanes;   // cones of four warps
    const long long soc_need = (n_soc + soc_block - 1) / soc_block;
    const long long lanes_rows = (long long)m * kLanes;
    const int t_rows = lanes_rows <= 256 * most ? 256 : kThreadsNA, t_cols = n <= 256 * most ? 256 : kThreadsNA;
    const long long rows_need = (lanes_rows + t_rows - 1) / t_rows;
    const long long cols_need = ((long long)n + t_cols - 1) / t_cols;
    const long long wide = cols_need > soc_need ? cols_need : soc_need;
    const int nb_rows = (int)(rows_need < most ? rows_need : most);
    const int nb_cols = (int)(wide < most ? wide : most);
    if (cudaMemsetAsync(scratch, 0, sizeof(double) * ((size_t)n + kHead), st) != cudaSuccess) return ACS_ERR_CUDA;
    rows_kernel<<<nb_rows, t_rows, 0, st>>>(P);
    cols_kernel<<<nb_cols, t_cols, 0, st>>>(P, nb_rows);
    if (cudaGetLastError() != cudaSuccess) return ACS_ERR_CUDA;
    return ACS_SOLVED;
}
