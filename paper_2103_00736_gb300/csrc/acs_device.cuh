// Device code of the conic solver shared by the single-problem launch
// (acs_iter.cu: one team = the whole grid) and the batched launch
// (acs_batch.cu: one team of CTAs per problem): grid/team barriers and
// reductions, sliced-ELLPACK products, the phases of Algorithm 2 and the
// solve loop.  See acs_iter.cu for the method and the precision scheme.
#pragma once

#include <math.h>
#include <stdio.h>

#include "acs_internal.cuh"

namespace acs {

// ---------------------------------------------------------------------------
// synchronisation and reductions
// ---------------------------------------------------------------------------

__device__ __forceinline__ unsigned long long gtimer() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}
__device__ __forceinline__ int ld_volatile_int(const int* p) { return *(volatile const int*)p; }

// Grid-wide reduction and barrier.
//
// A phase leaves its contributions to a reduction in shared memory as one
// value per warp (block_partials).  At the barrier that ends the phase warp 0
// combines the warps and publishes this CTA's partials, the first warps read
// every CTA's partials and combine them in a fixed order, and warp 0 alone
// computes the scalars that steer the loop from them (the `post` function of
// grid_sync_post); everyone else waits at the CTA barrier that follows and
// reads the results in shared memory.  Every CTA thus holds bit-identical
// values (deterministic for a given launch shape).  What bounds these steps
// is the FP64 pipe: it takes a warp instruction in 16 cycles per SM, so a
// scalar operation repeated by all 32 warps costs 512 cycles, and a dependent
// addition has a latency of 64, so a chain of square root and quotients takes
// about 1 us even in one warp.  Measured on 152 CTAs: a barrier that reduces
// one value 5.2 -> 3.9 us, the CG vector step of a 2000-row dense problem
// 13.7 -> 8.7 us, a KKT check of a 1000 x 5000 LP 34 -> 21 us (before: every
// CTA read the partials after the counter had arrived, and every thread
// computed the scalars).
// All waits through memory are bounded
// (kBarrierTimeoutNs): on expiry, or when another CTA has recorded an error,
// the wait records ACS_ERR_DEVICE_TIMEOUT and grid_sync returns false in
// every thread; the caller then leaves the kernel.  A team that is one cluster
// waits in the hardware's barrier.cluster, which has no limit and needs none as
// long as all CTAs leave the loop at the same barrier.  They do: the FP64 loop
// without bulk copies ends only on values that every CTA holds alike.
constexpr int kMaxGrid = 256;   // CTAs of a persistent launch (one per SM)
constexpr int kMaxCluster = 16; // CTAs of a launch that is one cluster

// Scalars that steer the solve loop and the CG, computed once per CTA.
struct CondRange {
    double alpha, lmin, lmax;
    bool any;
};
enum Count : int {
    CT_A = 0, CT_AT, CT_A64, CT_AT64, CT_COND, CT_CHECK, CT_A32, CT_AT32, CT_DENSE, CT_FACTOR, CT_CG, CT_COUNT
};
struct LoopScalars {
    long long count[CT_COUNT];   // passes of this loop (thread 0)
    long long win_cg;            // CG iterations since the last rescaling (thread 0)
    double gam, gam_prev, alpha, alpha_prev, beta, thr;   // CG
    double floor_r, target, best, best_ref;               // polish solves
    double ds, snorm, eta, d0, d1;                        // step norms, inexactness factor
    double res[6], best_mx;                               // residuals of the last check
    CondRange range;                                      // exponent range of a rescaling
    int flat_checks;
    int go;          // CG: the residual is above its target
    int far;         // CG: ... by more than a factor 100
    int bad;         // a non-finite value
    int broke;       // CG: p'Mp <= 0
    int over;        // the deadline of a time-sliced solve has passed
    int trouble;     // the FP32 correction cannot keep up
    int solved;      // every residual is <= tol
    int end32;       // the FP32 outer passes end
};

struct SyncShared {
    int cluster;              // the team is one thread-block cluster (barriers in hardware)
    int team_rank;            // this CTA's rank in the team working on one problem
    int team_size;            // CTAs in the team (the whole grid for a single solve)
    unsigned long long* bar;  // the team's monotonic barrier arrival counter
    double* tpart;            // the team's partials, [team_size * kPartStride]
    double* dM;               // the team's dense scratch for the cached projection operator:
    double* dX;               //   M / its Cholesky factor and L^{-1}, [m * m] each
    unsigned long long deadline;  // global-timer time at which a time-sliced solve pauses (0 = none)
    double out[kMaxRed];      // grid-reduced values of the last barrier
    double wsum[kWarps][kMaxRed];   // the warps' contributions to the next one
    double gsum[kWarps][kMaxRed];   // the CTAs' contributions, by the warp that gathered them
    double cslot[2][kMaxCluster][kMaxRed];   // a cluster's partials, written by its CTAs
    unsigned opmask;          // bit k: value k is combined by max (else by sum)
    int nv;                   // number of values reduced at the next barrier
    LoopScalars lp;           // scalars of the solve loop, written by warp 0 at the barriers
    int fail;
    unsigned gen;             // barrier generation (same sequence in every CTA)
    // column-blocked passes: the mbarrier that completes a block's bulk copy
    // into shared memory, and its phase parity (flips once per block staged)
    unsigned long long stage_bar;
    unsigned stage_phase;
    int cb_next;              // next run of the current segment to deal to a warp
    // the combine phases' two tile slots: their mbarriers and phase parities
    unsigned long long comb_bar[2];
    unsigned comb_phase[2];
};

__device__ __forceinline__ SyncShared& sync_smem() {
    __shared__ SyncShared s;
    return s;
}

// A team is the set of CTAs that work on one problem: the whole grid of a
// single-problem launch, or a group of CTAs (often one) of a batched launch.
// Phases index coordinates, rows and cones by the thread's rank in its team.
__device__ __forceinline__ void team_set(int rank, int size, unsigned long long* bar, double* partials,
                                         double* dense_M = nullptr, double* dense_X = nullptr, int cluster = 0) {
    SyncShared& S = sync_smem();
    if (threadIdx.x == 0) {
        S.cluster = cluster;
        S.team_rank = rank;
        S.team_size = size;
        S.bar = bar;
        S.tpart = partials;
        S.dM = dense_M;
        S.dX = dense_X;
        S.deadline = 0ull;
    }
    __syncthreads();
}
__device__ __forceinline__ int team_rank() { return sync_smem().team_rank; }
__device__ __forceinline__ int team_size() { return sync_smem().team_size; }
__device__ __forceinline__ int global_tid() { return team_rank() * (int)blockDim.x + (int)threadIdx.x; }
__device__ __forceinline__ int global_threads() { return team_size() * (int)blockDim.x; }
// Warps are numbered across the CTAs first, so that work of fewer units than the
// team has warps (rows of a dense problem, cones), or of a fraction more than
// a multiple of them, spreads over all SMs instead of filling the first CTAs:
// with 2320 rows on 152 x 32 warps, 73 SMs did everything.
__device__ __forceinline__ int global_warp() {
    return (int)(threadIdx.x >> 5) * team_size() + team_rank();
}
__device__ __forceinline__ int global_warps() { return global_threads() >> 5; }

// The parameter block of a solve, copied to shared memory once per launch or
// member.  The phases take it by reference, so each field they use is a load
// through a generic address; from a kernel's parameters or from global memory
// that load misses L1 after every barrier (the barrier's acquire empties it), an
// L2 round trip before the first useful load of a phase and again for each
// pointer the compiler cannot keep in a register.  Measured: 0.5 to 1.2 us of every
// phase (the CG passes of a 1000 x 5000 LP 3.4 -> 3.0 and 6.6 -> 6.2 us).
template <typename T, int kWhich = 0>
__device__ __forceinline__ const IterParams<T>& stage_params(const IterParams<T>& P) {
    static_assert(sizeof(IterParams<T>) % 8 == 0, "copied by 8-byte words");
    __shared__ __align__(16) unsigned long long buf[sizeof(IterParams<T>) / 8];
    __syncthreads();                                     // no one reads an earlier block any more
    const unsigned long long* src = reinterpret_cast<const unsigned long long*>(&P);
    for (int i = threadIdx.x; i < (int)(sizeof(IterParams<T>) / 8); i += blockDim.x) buf[i] = src[i];
    __syncthreads();
    return *reinterpret_cast<const IterParams<T>*>(buf);
}

__device__ __forceinline__ double warp_sum(double x) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    return x;
}
__device__ __forceinline__ double warp_max(double x) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x = fmax(x, __shfl_xor_sync(0xffffffffu, x, o));
    return x;
}

// Sums over the warp of NV values at once: at each of the first steps a lane
// gives half of its values to its partner and keeps the other half, so that 8
// values take 9 FP64 additions a lane instead of 40.  On return v[0] of lane l
// holds value warp_sums_index<NV>(l), for l a multiple of 32 / NV.
template <int NV>
__device__ __forceinline__ void warp_sums(double (&v)[NV]) {
    const int lane = threadIdx.x & 31;
    int o = 16;
#pragma unroll
    for (int c = NV; c > 1; c >>= 1, o >>= 1) {
        const bool up = (lane & o) != 0;
#pragma unroll
        for (int i = 0; i < c / 2; ++i) {
            const double give = up ? v[i] : v[i + c / 2];
            const double keep = up ? v[i + c / 2] : v[i];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, give, o);
        }
    }
#pragma unroll
    for (; o > 0; o >>= 1) v[0] += __shfl_xor_sync(0xffffffffu, v[0], o);
}
template <int NV>
__device__ __forceinline__ int warp_sums_index(int lane) {
    return NV == 1 ? 0 : NV == 2 ? lane >> 4 : NV == 4 ? lane >> 3 : lane >> 2;
}

__device__ __forceinline__ bool is_nonzero(double x) {   // without the FP64 pipe
    return (__double_as_longlong(x) << 1) != 0ll;
}

// Stage this CTA's contribution to the values reduced at the next grid_sync:
// one value per warp (warps with nothing but zeros skip their sums).  op: 0 =
// sum, 1 = max.
template <int NV>
__device__ __forceinline__ void block_partials(const double (&v)[NV], const int (&op)[NV]) {
    SyncShared& S = sync_smem();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned mask = 0u;
#pragma unroll
    for (int k = 0; k < NV; ++k) mask |= (op[k] ? 1u : 0u) << k;
    if (mask == 0u) {
        constexpr int NP = NV <= 1 ? 1 : NV <= 2 ? 2 : NV <= 4 ? 4 : 8;
        double a[NP];
        bool nz = false;
#pragma unroll
        for (int k = 0; k < NP; ++k) {
            a[k] = k < NV ? v[k < NV ? k : 0] : 0.0;
            nz |= is_nonzero(a[k]);
        }
        if (__any_sync(0xffffffffu, nz)) warp_sums<NP>(a);
        else a[0] = 0.0;
        const int k = warp_sums_index<NP>(lane);
        if ((lane & (32 / NP - 1)) == 0 && k < NV) S.wsum[warp][k] = a[0];
    } else {
#pragma unroll
        for (int k = 0; k < NV; ++k) {
            const double x = op[k] ? warp_max(v[k]) : warp_sum(v[k]);
            if (lane == 0) S.wsum[warp][k] = x;
        }
    }
    if (threadIdx.x == 0) {
        S.opmask = mask;
        S.nv = NV;
    }
}

// Combine over the warp's lanes the nv values each lane holds, into dst[0, nv).
template <int NV>
__device__ __forceinline__ void warp_sums_to(const double (&x)[kMaxRed], int nv, double* dst) {
    const int lane = threadIdx.x & 31;
    double a[NV];
#pragma unroll
    for (int k = 0; k < NV; ++k) a[k] = x[k];
    warp_sums<NV>(a);
    const int k = warp_sums_index<NV>(lane);
    if ((lane & (32 / NV - 1)) == 0 && k < nv) dst[k] = a[0];
}
__device__ __forceinline__ void warp_combine(const double (&x)[kMaxRed], int nv, unsigned opmask, double* dst) {
    if (opmask == 0u) {
        if (nv <= 1) warp_sums_to<1>(x, nv, dst);
        else if (nv <= 2) warp_sums_to<2>(x, nv, dst);
        else if (nv <= 4) warp_sums_to<4>(x, nv, dst);
        else warp_sums_to<8>(x, nv, dst);
    } else {
#pragma unroll
        for (int k = 0; k < kMaxRed; ++k)
            if (k < nv) {
                const double r = (opmask >> k) & 1u ? warp_max(x[k]) : warp_sum(x[k]);
                if ((threadIdx.x & 31) == 0) dst[k] = r;
            }
    }
    __syncwarp();
}

// Start (or resume, with the generation reached so far) the team's barrier
// sequence and clear the failure flag.
static __device__ void sync_init(unsigned gen) {
    SyncShared& S = sync_smem();
    if (threadIdx.x == 0) {
        S.nv = 0;
        S.fail = 0;
        S.gen = gen;
    }
    __syncthreads();
}

__device__ __forceinline__ void red_add_release(unsigned long long* p, unsigned long long v) {
    asm volatile("red.release.gpu.global.add.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
__device__ __forceinline__ unsigned long long ld_acquire64(const unsigned long long* p) {
    unsigned long long v;
    asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}

// A partial and the generation of the barrier it belongs to, written and read
// as one 16-byte access: a reader that sees the generation has the value.
__device__ __forceinline__ void st_slot(double* slot, double v, unsigned long long tag) {
    asm volatile(
        "{\n\t.reg .b128 q;\n\tmov.b128 q, {%1, %2};\n\tst.relaxed.gpu.global.b128 [%0], q;\n\t}" ::"l"(slot),
        "l"(__double_as_longlong(v)), "l"(tag)
        : "memory");
}
__device__ __forceinline__ double ld_slot(const double* slot, unsigned long long& tag) {
    long long v;
    asm volatile("{\n\t.reg .b128 q;\n\tld.relaxed.gpu.global.b128 q, [%2];\n\tmov.b128 {%0, %1}, q;\n\t}"
                 : "=l"(v), "=l"(tag)
                 : "l"(slot)
                 : "memory");
    return __longlong_as_double(v);
}
__device__ __forceinline__ void fence_gpu() { asm volatile("fence.acq_rel.gpu;" ::: "memory"); }

// A bounded wait's bookkeeping: called with the number of unsuccessful tries
// so far; true when the wait must end (another CTA recorded an error, or the
// time is up, which records ACS_ERR_DEVICE_TIMEOUT).
__device__ __forceinline__ bool wait_expired(int tries, unsigned long long& t0, int* err) {
    if ((tries & 63) != 63) return false;
    if (ld_volatile_int(err) != 0) return true;
    const unsigned long long t = gtimer();
    if (t0 == 0ull) t0 = t;
    if (t - t0 <= kBarrierTimeoutNs) return false;
    atomicCAS(err, 0, ACS_ERR_DEVICE_TIMEOUT);
    return true;
}

// This lane's share of a reducing barrier: waits for the partials of CTAs b0,
// b0 + step, ... and combines them in that order.  Returns false if a wait
// expired.
template <int NV>
__device__ __forceinline__ bool gather_slots(const double* part, unsigned long long tag, int b0, int step, int size,
                                             unsigned opmask, int* err, double (&x)[kMaxRed]) {
    unsigned long long t0 = 0ull;
    bool ok = true;
    for (int b = b0; b < size && ok; b += step) {
        const double* slot = part + (size_t)b * kPartStride;
        double v[NV];
        for (int tries = 0;; ++tries) {
            bool all = true;
#pragma unroll
            for (int k = 0; k < NV; ++k) {
                unsigned long long t;
                v[k] = ld_slot(slot + 2 * k, t);
                all = all && t == tag;
            }
            if (all) break;
            if (wait_expired(tries, t0, err)) { ok = false; break; }
        }
#pragma unroll
        for (int k = 0; k < NV; ++k) x[k] = (opmask >> k) & 1u ? fmax(x[k], v[k]) : x[k] + v[k];
    }
    return ok;
}

// Barrier of all threads of the cluster; what any of them wrote before it is
// visible to all after it.  barrier.cluster counts a warp when it arrives, so its lanes
// have to arrive together; warp 0 comes here from code that only some of them run.
__device__ __forceinline__ void cluster_sync() {
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// v to the same variable of CTA `rank` of the cluster.
__device__ __forceinline__ void st_cluster(double* var, int rank, double v) {
    unsigned local = (unsigned)__cvta_generic_to_shared(var), remote;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(local), "r"(rank));
    asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(remote), "d"(v) : "memory");
}

// The barrier up to the reduced values.
//
// Without values, thread 0 adds 1 to the team's monotonic arrival counter
// with release semantics and spins (acquire) until the counter reaches
// (generation) * (CTAs in the team): about two L2 round trips.
//
// With values the arrival is the value itself: warp 0 combines the warps of
// this CTA, and its lane k writes (partial k, generation) to this CTA's slot;
// lane l of warp w then waits for the slot of CTA 32 w + l, whose tag is the
// news that that CTA has arrived, so that one L2 round trip after the last
// arrival every CTA has every partial (counter, then partials: two).  The
// counter is kept in step for the barriers without values.
//
// The error word is read while the wait is under way, so an error recorded
// just before a barrier may be seen one barrier later; the CTA that recorded it
// has left by then, and the others' next wait ends on the error word.
//
// A team that is one cluster uses the hardware's cluster barrier (which counts
// threads that have not exited, so it cannot wait for a CTA that has left) and
// exchanges partials through distributed shared memory; it reads the error word at
// reducing barriers only.  A team of one CTA needs neither.  The caller follows with a CTA barrier.
static __device__ __noinline__ void grid_reduce(int* err) {
    SyncShared& S = sync_smem();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const bool cluster = S.cluster != 0;
    __syncthreads();                                   // the phase's writes and S.wsum are complete
    const unsigned target = S.gen + 1u;
    const int nv = S.nv;
    const int size = S.team_size;
    if (nv == 0 && cluster) {
        cluster_sync();
        if (threadIdx.x == 0) S.gen = target;
        return;
    }
    if (nv == 0) {
        if (threadIdx.x == 0) {
            bool fail = false;
            const int e = ld_volatile_int(err);
            if (size > 1) {
                red_add_release(S.bar, 1ull);
                const unsigned long long want = (unsigned long long)target * size;
                unsigned long long t0 = 0ull;
                for (int tries = 0; ld_acquire64(S.bar) < want; ++tries)
                    if (wait_expired(tries, t0, err)) { fail = true; break; }
            }
            if (fail || e != 0) S.fail = 1;
            S.gen = target;
        }
        return;
    }
    const unsigned opmask = S.opmask;
    int e = 0;
    if (warp == 0) {
        if (lane == 0) e = ld_volatile_int(err);
        const int nw = (int)(blockDim.x >> 5);
        double x[kMaxRed];
#pragma unroll
        for (int k = 0; k < kMaxRed; ++k) {
            x[k] = 0.0;
            if (k < nv) x[k] = lane < nw ? S.wsum[lane][k] : ((opmask >> k) & 1u ? -INFINITY : 0.0);
        }
        warp_combine(x, nv, opmask, S.out);
        if (size == 1) {
            // the error word is still checked so that a failed problem stops
            if (lane == 0) {
                if (e != 0) S.fail = 1;
                S.gen = target;
                S.nv = 0;
            }
            __syncwarp();
            return;
        }
    }
    if (size == 1) return;
    if (cluster) {
        if (warp == 0 && lane < size)
            for (int k = 0; k < nv; ++k) st_cluster(&S.cslot[target & 1u][S.team_rank][k], lane, S.out[k]);
        cluster_sync();
        if (warp == 0) {
            double x[kMaxRed];
#pragma unroll
            for (int k = 0; k < kMaxRed; ++k) {
                x[k] = 0.0;
                if (k < nv)
                    x[k] = lane < size ? S.cslot[target & 1u][lane][k] : ((opmask >> k) & 1u ? -INFINITY : 0.0);
            }
            warp_combine(x, nv, opmask, S.out);
            if (lane == 0) {
                if (e != 0) S.fail = 1;
                S.gen = target;
                S.nv = 0;
            }
            __syncwarp();
        }
        return;
    }
    double* part = S.tpart + (target & 1u) * (2 * kMaxRed);
    if (warp == 0) {
        fence_gpu();                                    // the phase's writes come before the arrival
        if (lane < (nv <= 3 ? nv : kMaxRed)) st_slot(part + (size_t)S.team_rank * kPartStride + 2 * lane, S.out[lane], target);
        if (lane == 0) atomicAdd(S.bar, 1ull);
    }
    const int nwarp = min((size + 31) >> 5, (int)(blockDim.x >> 5));   // warps that gather
    if (warp < nwarp) {
        double x[kMaxRed];
#pragma unroll
        for (int k = 0; k < kMaxRed; ++k) x[k] = (opmask >> k) & 1u ? -INFINITY : 0.0;
        bool ok;
        const int b0 = warp * 32 + lane, step = nwarp * 32;
        if (nv == 1) ok = gather_slots<1>(part, target, b0, step, size, opmask, err, x);
        else if (nv == 2) ok = gather_slots<2>(part, target, b0, step, size, opmask, err, x);
        else if (nv == 3) ok = gather_slots<3>(part, target, b0, step, size, opmask, err, x);
        else ok = gather_slots<8>(part, target, b0, step, size, opmask, err, x);
        ok = __all_sync(0xffffffffu, ok);
        fence_gpu();                                    // and reads of what the others wrote after it
        warp_combine(x, nv, opmask, S.gsum[warp]);
        if (!ok && lane == 0) S.fail = 1;
    }
    __syncthreads();
    if (warp == 0) {
        if (lane < nv) {
            const bool mx = (opmask >> lane) & 1u;
            double x = S.gsum[0][lane];
            for (int w = 1; w < nwarp; ++w) x = mx ? fmax(x, S.gsum[w][lane]) : x + S.gsum[w][lane];
            S.out[lane] = x;
        }
        if (lane == 0) {
            if (e != 0) S.fail = 1;
            S.gen = target;
            S.nv = 0;
        }
        __syncwarp();
    }
}

// Barrier and reduction, then post(S.out) in warp 0 (every lane, the same
// values; post writes what the loop reads to shared memory).
template <typename Post>
__device__ __forceinline__ bool grid_sync_post(int* err, const Post& post) {
    grid_reduce(err);
    SyncShared& S = sync_smem();
    if (threadIdx.x < 32) post(S.out);
    __syncthreads();
    return S.fail == 0;
}
__device__ __forceinline__ bool grid_sync(int* err) {
    return grid_sync_post(err, [](const double*) {});
}

// Values reduced at the last grid_sync.
template <int NV>
__device__ void grid_combine(double (&out)[NV]) {
    SyncShared& S = sync_smem();
#pragma unroll
    for (int k = 0; k < NV; ++k) out[k] = S.out[k];
}

// ---------------------------------------------------------------------------
// row-parallel sparse products (sliced ELLPACK with G lanes per row)
// ---------------------------------------------------------------------------

// Matrix entries are read once per pass: stream them past L1.
__device__ __forceinline__ int ld_stream(const int* p) { return __ldcs(p); }
__device__ __forceinline__ float ld_stream(const float* p) { return __ldcs(p); }
__device__ __forceinline__ double ld_stream(const double* p) { return __ldcs(p); }

template <typename T> __device__ __forceinline__ const T* sell_vals(const SellMat& M);
template <> __device__ __forceinline__ const float* sell_vals<float>(const SellMat& M) { return M.v32; }
template <> __device__ __forceinline__ const double* sell_vals<double>(const SellMat& M) { return M.v64; }

// Stored value -> arithmetic type.  A BF16 value is the upper half of the
// FP32 value with the same bits, so the conversion is exact.
__device__ __forceinline__ unsigned short ld_stream(const unsigned short* p) { return __ldcs(p); }
template <typename T> __device__ __forceinline__ T val_to(T v) { return v; }
template <typename T> __device__ __forceinline__ T val_to(unsigned short b);
template <> __device__ __forceinline__ float val_to<float>(unsigned short b) {
    return __uint_as_float((unsigned)b << 16);
}

// Layout (see SellMat): a slice holds 32/G rows; chunk c of the slice is 32
// consecutive entries, entry k of local row r at chunk k/G, lane r*G + k%G.
// Warp w handles slices w, w + nwarps, ..., in batches of U chunks; each lane
// accumulates its entries in chunk order, and the G partial sums of a row are
// combined by a fixed shuffle tree, so the result does not depend on the
// launch shape.  epi(row, sum) runs once per real row.
//
// Software pipeline: the column/value loads of the next batch (and the slice
// table entries of the next slice) are issued before the gathers of the
// current batch, so a warp keeps one matrix round trip and one gather round
// trip in flight at the same time instead of one after the other.
template <int U, typename T, typename V>
__device__ __forceinline__ void sell_load_batch(const int* __restrict__ col, const V* __restrict__ val,
                                                int base, int k, int len, int (&c)[U], T (&a)[U]) {
#pragma unroll
    for (int u = 0; u < U; ++u) {
        if (k + u < len) {
            c[u] = ld_stream(col + base + 32 * (k + u));
            a[u] = val_to<T>(ld_stream(val + base + 32 * (k + u)));
        } else {
            c[u] = 0;
            a[u] = T(0);
        }
    }
}

// V: the stored value type (T itself, or BF16 bits for T = float).
template <int G, int U, typename T, typename V, typename Gather, typename Epi>
__device__ __forceinline__ void sell_rows_g(const SellMat& M, const V* __restrict__ val, Gather gather, Epi epi) {
    const int* __restrict__ col = M.col;
    const int lane = threadIdx.x & 31;
    const int nw = global_warps();
    int sl = global_warp();
    if (sl >= M.nslices) return;                        // warp-uniform
    int len = __ldg(M.slen + sl);
    int base = __ldg(M.sptr + sl) + lane;
    int k = 0;
    // slice table entries of the following slice, loaded one slice ahead
    int nsl = sl + nw;
    int nlen = 0, nbase = 0;
    if (nsl < M.nslices) {
        nlen = __ldg(M.slen + nsl);
        nbase = __ldg(M.sptr + nsl) + lane;
    }
    int c[U];
    T a[U];
    sell_load_batch<U>(col, val, base, k, len, c, a);
    T acc = T(0);
    while (true) {
        // next batch: more chunks of this slice, or the first of the next slice
        const bool same = k + U < len;
        const bool have_next = same || nsl < M.nslices;
        int c2[U];
        T a2[U];
        if (same) sell_load_batch<U>(col, val, base, k + U, len, c2, a2);
        else if (have_next) sell_load_batch<U>(col, val, nbase, 0, nlen, c2, a2);
        T x[U];
#pragma unroll
        for (int u = 0; u < U; ++u) x[u] = gather(c[u]);
#pragma unroll
        for (int u = 0; u < U; ++u) acc = fma(a[u], x[u], acc);
        if (!same) {                                    // slice finished
#pragma unroll
            for (int o = G / 2; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
            const int row = sl * (32 / G) + lane / G;
            if ((lane & (G - 1)) == 0 && row < M.nrows) epi(row, acc);
            acc = T(0);
            if (!have_next) break;
            sl = nsl;
            len = nlen;
            base = nbase;
            k = 0;
            nsl = sl + nw;
            if (nsl < M.nslices) {
                nlen = __ldg(M.slen + nsl);
                nbase = __ldg(M.sptr + nsl) + lane;
            }
        } else {
            k += U;
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            c[u] = c2[u];
            a[u] = a2[u];
        }
    }
}

// Chunks per software-pipeline batch: each lane keeps U column/value loads
// and U gathers in flight.  Measured on the large LP (1e7 nonzeros): U = 4,
// 8, 12 give 58.9, 57.9, 70.1 us for the CG A pass and 44.8, 46.2, 51.2 us
// for the A' pass -- the passes are bound by the L2 gather rate, not by the
// depth of the chain -- so 4 stays; FP64 passes at 8 would spill registers.
#ifndef ACS_CG_U
#define ACS_CG_U 4
#endif

// Rows that hold every column in order (dense problems): entry k of a row is
// column k, so the vector is read in order and no column index is loaded (4 of
// 8 bytes an entry in FP32, and one of two dependent loads).  Every lane takes
// the same entries in the same order as above, so the sums are the same.  With
// fewer rows than warps one row's latency is the pass: eight entries a lane in
// flight (sixteen in FP32 gave nothing more).  Measured with the numbering of global_warp(), m = 2320, n = 2900: FP32
// pass over A 24.2 -> 14.0 us, over A' 16.6 -> 9.6, FP64 residual pass 35.6 ->
// 22.7 (phase times, barrier included).
template <typename T, typename V, typename Gather, typename Epi>
__device__ __forceinline__ void dense_rows(const SellMat& M, const V* __restrict__ val, Gather gather, Epi epi) {
    constexpr int U = 8;
    const int lane = threadIdx.x & 31;
    const int g = M.g, ncols = M.full, gl = lane & (g - 1);
    const int len = (ncols + g - 1) / g, h = 32 / g, nw = global_warps();
    for (int sl = global_warp(); sl < M.nslices; sl += nw) {
        const V* v = val + (size_t)sl * len * 32 + lane;
        T acc = T(0);
        for (int k = 0; k < len; k += U) {
            T a[U], x[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int j = (k + u) * g + gl;
                const bool in = j < ncols;
                a[u] = in ? val_to<T>(ld_stream(v + 32 * (k + u))) : T(0);
                x[u] = in ? gather(j) : T(0);
            }
#pragma unroll
            for (int u = 0; u < U; ++u) acc = fma(a[u], x[u], acc);
        }
        for (int o = g / 2; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
        const int row = sl * h + lane / g;
        if (gl == 0 && row < M.nrows) epi(row, acc);
    }
}

template <typename T, typename V, typename Gather, typename Epi>
__device__ __forceinline__ void sell_rows_v(const SellMat& M, const V* val, Gather gather, Epi epi) {
    if (M.full > 0) {
        dense_rows<T>(M, val, gather, epi);
        return;
    }
    constexpr int U = (sizeof(T) == 4) ? ACS_CG_U : 4;
    switch (M.g) {
        case 1: sell_rows_g<1, U, T>(M, val, gather, epi); break;
        case 2: sell_rows_g<2, U, T>(M, val, gather, epi); break;
        case 4: sell_rows_g<4, U, T>(M, val, gather, epi); break;
        case 8: sell_rows_g<8, U, T>(M, val, gather, epi); break;
        case 16: sell_rows_g<16, U, T>(M, val, gather, epi); break;
        default: sell_rows_g<32, U, T>(M, val, gather, epi); break;
    }
}

// FP32 products read the BF16 copy of the values when A is stored in BF16.
template <typename T, typename Gather, typename Epi>
__device__ __forceinline__ void sell_rows(const SellMat& M, Gather gather, Epi epi) {
    if (sizeof(T) == 4 && M.v16 != nullptr) sell_rows_v<T>(M, M.v16, gather, epi);
    else sell_rows_v<T>(M, sell_vals<T>(M), gather, epi);
}

// Two sums per row: sum a*g1(j) and sum a*a*g2(j) (FP64 values).
template <int G, typename G1, typename G2, typename Epi>
__device__ __forceinline__ void sell_rows2_g(const SellMat& M, G1 g1, G2 g2, Epi epi) {
    const int lane = threadIdx.x & 31;
    const int nw = global_warps();
    for (int sl = global_warp(); sl < M.nslices; sl += nw) {
        const int len = __ldg(M.slen + sl);
        int idx = __ldg(M.sptr + sl) + lane;
        double acc1 = 0.0, acc2 = 0.0;
        for (int k = 0; k < len; ++k, idx += 32) {
            const int j = ld_stream(M.col + idx);
            const double a = ld_stream(M.v64 + idx);
            acc1 = fma(a, g1(j), acc1);
            acc2 = fma(a * a, g2(j), acc2);
        }
#pragma unroll
        for (int o = G / 2; o > 0; o >>= 1) {
            acc1 += __shfl_xor_sync(0xffffffffu, acc1, o);
            acc2 += __shfl_xor_sync(0xffffffffu, acc2, o);
        }
        const int row = sl * (32 / G) + lane / G;
        if ((lane & (G - 1)) == 0 && row < M.nrows) epi(row, acc1, acc2);
    }
}

template <typename G1, typename G2, typename Epi>
__device__ __forceinline__ void sell_rows2(const SellMat& M, G1 g1, G2 g2, Epi epi) {
    switch (M.g) {
        case 1: sell_rows2_g<1>(M, g1, g2, epi); break;
        case 2: sell_rows2_g<2>(M, g1, g2, epi); break;
        case 4: sell_rows2_g<4>(M, g1, g2, epi); break;
        case 8: sell_rows2_g<8>(M, g1, g2, epi); break;
        case 16: sell_rows2_g<16>(M, g1, g2, epi); break;
        default: sell_rows2_g<32>(M, g1, g2, epi); break;
    }
}

// ---------------------------------------------------------------------------
// column-blocked products (layout in acs_internal.cuh / acs_cbsell.cuh)
// ---------------------------------------------------------------------------

// Dynamic shared memory of the single-problem FP32 launch: the block of the
// multiplied vector that a column-blocked pass gathers from.
extern __shared__ __align__(16) float acs_cb_smem[];

__device__ __forceinline__ unsigned smem_u32(const void* p) {
    return (unsigned)__cvta_generic_to_shared(p);
}

// Set up the staging barrier (once per launch, before the first pass).
__device__ __forceinline__ void cb_init() {
    SyncShared& S = sync_smem();
    if (threadIdx.x == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&S.stage_bar)) : "memory");
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&S.comb_bar[0])) : "memory");
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&S.comb_bar[1])) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        S.stage_phase = 0u;
        S.comb_phase[0] = S.comb_phase[1] = 0u;
    }
    __syncthreads();
}

// Bounded wait for the staging barrier's current phase (2 s, then the error
// word records ACS_ERR_DEVICE_TIMEOUT; the next grid barrier ends the launch).
__device__ __forceinline__ bool cb_wait_bar(unsigned long long* mbar, unsigned parity, int* err) {
    const unsigned bar = smem_u32(mbar);
    unsigned done = 0;
    const unsigned long long t0 = gtimer();
    int spins = 0;
    while (true) {
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(done)
            : "r"(bar), "r"(parity)
            : "memory");
        if (done) return true;
        if (++spins == 64) {
            spins = 0;
            if (gtimer() - t0 > kBarrierTimeoutNs) {
                atomicCAS(err, 0, ACS_ERR_DEVICE_TIMEOUT);
                return false;
            }
        }
    }
}

// Stage x[c0, c0 + w) in shared memory as FP32.  The vector was written by
// other CTAs before the last grid barrier.  An FP32 vector is copied by the
// bulk-copy engine: thread 0 issues 1-D bulk copies (16-byte multiples; c0 is
// a multiple of 4 and the vector 16-byte aligned) that complete on the
// staging mbarrier, the last w mod 4 entries by plain loads; an FP64 vector
// is read and rounded by all threads, eight loads in flight per thread.
template <typename Src>
__device__ __forceinline__ void cb_stage(float* xs, const Src* __restrict__ x, int c0, int w, int* err) {
    SyncShared& S = sync_smem();
    if constexpr (sizeof(Src) == 4) {
        const int w4 = w & ~3;
        const unsigned parity = S.stage_phase;
        if (w4 > 0 && threadIdx.x == 0) {
            const unsigned bar = smem_u32(&S.stage_bar);
            const unsigned bytes = (unsigned)w4 * 4u;
            // generic-proxy writes to x (other CTAs, before the grid barrier)
            // and generic reads of xs (before the CTA barrier) come first
            asm volatile("fence.proxy.async.global;" ::: "memory");
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes)
                         : "memory");
            constexpr unsigned kChunk = 32768u;
            const char* src = reinterpret_cast<const char*>(x + c0);
            char* dst = reinterpret_cast<char*>(xs);
            for (unsigned o = 0; o < bytes; o += kChunk) {
                const unsigned len = bytes - o < kChunk ? bytes - o : kChunk;
                asm volatile(
                    "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                        smem_u32(dst + o)),
                    "l"(src + o), "r"(len), "r"(bar)
                    : "memory");
            }
        }
        for (int k = w4 + (int)threadIdx.x; k < w; k += blockDim.x) xs[k] = __ldcg(x + c0 + k);
        if (w4 > 0) {
            cb_wait_bar(&S.stage_bar, parity, err);
            __syncthreads();                             // every thread has seen the phase
            if (threadIdx.x == 0) S.stage_phase = parity ^ 1u;
        }
    } else {
        constexpr int kIn = 8;
        const int step = (int)blockDim.x * kIn;
        for (int k0 = threadIdx.x; k0 < w; k0 += step) {
            double v[kIn];
#pragma unroll
            for (int u = 0; u < kIn; ++u) {
                const int k = k0 + u * (int)blockDim.x;
                v[u] = k < w ? __ldcg(x + c0 + k) : 0.0;
            }
#pragma unroll
            for (int u = 0; u < kIn; ++u) {
                const int k = k0 + u * (int)blockDim.x;
                if (k < w) xs[k] = (float)v[u];
            }
        }
    }
}

template <int U>
__device__ __forceinline__ void cb_load_batch(const unsigned short* __restrict__ col, const float* __restrict__ val,
                                              int base, int k, int len, unsigned (&c)[U], float (&a)[U]) {
#pragma unroll
    for (int u = 0; u < U; ++u) {
        if (k + u < len) {
            c[u] = __ldcs(col + base + 32 * (k + u));
            a[u] = __ldcs(val + base + 32 * (k + u));
        } else {
            c[u] = 0u;
            a[u] = 0.f;
        }
    }
}

// Items are multiplied in runs of kCbRun consecutive items, whose entries
// are contiguous: a warp streams a run as one sequence of chunks (lane r of
// chunk c at 32 c + r), whatever the items' lengths, so the next batch of
// column/value loads can always be issued before the current gathers --
// across item and run boundaries.  An item ends at the chunk its end mark
// flags (every item has one).  Runs are dealt to the warps as they ask for
// them (a shared counter): the items of a window are sorted by length, so a
// fixed deal would give some warps the long runs every time.  Which warp
// multiplies a run does not change its sums.
constexpr int kCbRun = 4;

// The next run for this warp (lane 0 takes it from the counter).
__device__ __forceinline__ int cb_take_run(int lane) {
    int r = 0;
    if (lane == 0) r = atomicAdd(&sync_smem().cb_next, 1);
    return __shfl_sync(0xffffffffu, r, 0);
}

// Chunks [c0, c1) of run `run` of the segment [s0, s1) (lanes 0 and 1 load
// the two offsets).
__device__ __forceinline__ void cb_run_chunks(const int* __restrict__ sptr, int s0, int s1, int run, int lane,
                                              int& c0, int& c1) {
    const int i0 = s0 + run * kCbRun;
    const int i1 = min(s1, i0 + kCbRun);
    const int v = lane < 2 ? __ldg(sptr + (lane == 0 ? i0 : i1)) : 0;
    c0 = __shfl_sync(0xffffffffu, v, 0) >> 5;
    c1 = __shfl_sync(0xffffffffu, v, 1) >> 5;
}

// End marks of chunks [c, c + U) as the low U bits (U <= 32).
template <int U>
__device__ __forceinline__ unsigned cb_marks(const unsigned* __restrict__ cend, int c) {
    const unsigned w0 = __ldg(cend + (c >> 5)), w1 = __ldg(cend + (c >> 5) + 1);
    const unsigned long long w = ((unsigned long long)w1 << 32) | w0;
    return (unsigned)(w >> (c & 31)) & ((1u << U) - 1u);
}

// U chunks starting at chunk c: lane r's entries of chunks c .. c + U - 1,
// those at or past chunk c1 read as (column 0, value 0).
template <int U>
__device__ __forceinline__ void cb_load_chunks(const unsigned short* __restrict__ col,
                                               const float* __restrict__ val, int c, int c1,
                                               unsigned (&cc)[U], float (&a)[U]) {
    const size_t e = (size_t)c * 32 + (threadIdx.x & 31);
    const unsigned short* cp = col + e;
    const float* vp = val + e;
#pragma unroll
    for (int u = 0; u < U; ++u) {
        const bool in = c + u < c1;
        cc[u] = in ? __ldcs(cp + 32 * u) : 0u;
        a[u] = in ? __ldcs(vp + 32 * u) : 0.f;
    }
}

// The items [s0, s1) of one block (one CTA's segment), in runs dealt to the
// warps as above: lane r accumulates its row's entries of each item in chunk
// order (FP32, gathers from the staged block xs) and writes the sum to
// part[item * 32 + r] (slot order: one coalesced store per item; the combine
// phases put the rows back in order).  MODE (benchmark variants): 0 the
// pass, 1 the matrix stream without the gathers, 2 without staging first.
template <int U, int MODE = 0>
__device__ __forceinline__ void cb_items(const CbMat& M, const float* xs, int s0, int s1, int warp) {
    const int nruns = (s1 - s0 + kCbRun - 1) / kCbRun;
    int run = warp;                                      // the first runs: one per warp
    if (run >= nruns) return;                            // warp-uniform
    const int lane = threadIdx.x & 31;
    int item = s0 + run * kCbRun;                        // item the next chunk belongs to
    int c, c1;                                           // chunks of the current run
    cb_run_chunks(M.sptr, s0, s1, run, lane, c, c1);
    int nrun = cb_take_run(lane), nc = 0, nc1 = 0;       // the following run, one run ahead
    if (nrun < nruns) cb_run_chunks(M.sptr, s0, s1, nrun, lane, nc, nc1);
    unsigned cc[U];
    float a[U];
    cb_load_chunks<U>(M.col, M.val, c, c1, cc, a);
    unsigned marks = cb_marks<U>(M.cend, c);
    float acc = 0.f;
    while (true) {
        const bool same = c + U < c1;
        const bool have_next = same || nrun < nruns;
        const int cn = same ? c + U : nc;                // first chunk of the next batch
        const int cn1 = same ? c1 : nc1;
        unsigned cc2[U];
        float a2[U];
        cb_load_chunks<U>(M.col, M.val, cn, have_next ? cn1 : cn, cc2, a2);
        const unsigned marks2 = have_next ? cb_marks<U>(M.cend, cn) : 0u;
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (c + u < c1) {                            // warp-uniform
                if (MODE == 1) acc += a[u] + (float)cc[u];
                else acc = fmaf(a[u], xs[cc[u]], acc);
                if (marks & (1u << u)) {                 // the item ends at this chunk
                    __stcg(M.part + (size_t)item * 32 + lane, acc);
                    acc = 0.f;
                    ++item;
                }
            }
        }
        if (!have_next) break;
        if (!same) {                                     // the next run
            item = s0 + nrun * kCbRun;
            nrun = cb_take_run(lane);
            if (nrun < nruns) cb_run_chunks(M.sptr, s0, s1, nrun, lane, nc, nc1);
        }
        c = cn;
        c1 = cn1;
        marks = marks2;
#pragma unroll
        for (int u = 0; u < U; ++u) {
            cc[u] = cc2[u];
            a[u] = a2[u];
        }
    }
}

// One column-blocked pass over the items dealt to this CTA: for each block
// its range touches, stage the block of x, then multiply the range's items
// of that block.  Every slot of every item gets its sum written (0 for a row
// with no entry in the block).  Run by all threads of the CTA, after cb_init
// in the launch.
#ifndef ACS_CB_U
#define ACS_CB_U 6
#endif
template <typename Src, int MODE = 0>
__device__ __forceinline__ void cb_pass(const CbMat& M, const Src* __restrict__ x, int* err) {
    float* xs = acs_cb_smem;
    const int rank = team_rank();
    const int end = __ldg(M.cta_beg + rank + 1);
    int it = __ldg(M.cta_beg + rank);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    if (MODE >= 3) {
        // benchmark variants: the CTA's entries as one linear stream, chunk c
        // to warp c mod nw (3: columns and values, 4: values only)
        const int c0 = __ldg(M.sptr + it) >> 5, c1 = __ldg(M.sptr + end) >> 5;
        float acc = 0.f;
        for (int c = c0 + warp; c < c1; c += 4 * nw) {
            float v[4];
            unsigned cc[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int ch = c + u * nw;
                const size_t idx = (size_t)ch * 32 + lane;
                v[u] = ch < c1 ? __ldcs(M.val + idx) : 0.f;
                cc[u] = (MODE == 3 && ch < c1) ? __ldcs(M.col + idx) : 0u;
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) acc += v[u] + (float)cc[u];
        }
        M.part[(size_t)(rank * nw + warp) * 32 + lane] = acc;
        return;
    }
    while (it < end) {                                   // CTA-uniform
        const int b = it / M.nsl;
        const int bend = min(end, (b + 1) * M.nsl);
        const int c0 = b * M.width;
        __syncthreads();                                 // gathers from the previous block are done
        if (threadIdx.x == 0) sync_smem().cb_next = nw;  // runs after the first one per warp
        if (MODE == 0) cb_stage(xs, x, c0, min(M.ncols - c0, M.width), err);
        __syncthreads();
        cb_items<ACS_CB_U, MODE>(M, xs, it, bend, warp);
        it = bend;
    }
}

// Dynamic shared memory of the launch (bytes).
__device__ __forceinline__ unsigned dyn_smem_bytes() {
    unsigned v;
    asm("mov.u32 %0, %%dynamic_smem_size;" : "=r"(v));
    return v;
}

// Blocks of one combine tile that fit two tile slots in `smem` bytes (at
// least 1).
__host__ __device__ __forceinline__ int cb_combine_group(int nblocks, unsigned smem) {
    const unsigned per = (unsigned)kCbWindow * 6u;       // one block's sums and slot indices of a window
    int g = (int)(smem / (2u * per));
    if (g > nblocks) g = nblocks;
    return g < 1 ? 1 : g;
}

// Adds up the partial sums of the last pass row by row, in block order, and
// calls epi(row, sum) once for every row.  A CTA takes windows of kCbWindow
// rows (rank, rank + CTAs, ...); a tile is one window and a group of G
// blocks: for each block of the group, the window's partial sums (slot
// order) and the slot of each of its rows (ipos, row order) are copied into
// one of two tile slots in shared memory by the bulk-copy engine while the
// threads work on the previous tile.  Thread k owns rows k, k + blockDim, ...
// of the window and adds their sums block after block in registers, reading
// each at its slot.  Shared memory: the two slots (needs 24 KB for G = 1).
// Run by all threads of the CTA, after cb_init in the launch.
constexpr int kCbRowsPerThread = kCbWindow / kThreads;
template <typename Epi>
__device__ __forceinline__ void cb_combine(const CbMat& M, int* err, Epi epi) {
    SyncShared& S = sync_smem();
    const int R = M.nrows, nb = M.nblocks;
    const size_t slab = (size_t)M.nsl * 32;              // slots of one block
    const int nwin = (R + kCbWindow - 1) / kCbWindow;
    const int rank = team_rank(), size = team_size();
    if (rank >= nwin) return;                            // CTA-uniform
    const int G = cb_combine_group(nb, dyn_smem_bytes());
    const int ngroups = (nb + G - 1) / G;
    const int T = ((nwin - 1 - rank) / size + 1) * ngroups;
    char* slots = reinterpret_cast<char*>(acs_cb_smem);
    const unsigned slot_bytes = (unsigned)G * kCbWindow * 6u;
    // tile t: window rank + (t / ngroups) * size, blocks of group t % ngroups
    auto issue = [&](int t) {                            // thread 0
        const int w = rank + (t / ngroups) * size, g = t % ngroups;
        const int r0 = w * kCbWindow, nslots = (min(kCbWindow, R - r0) + 31) & ~31;
        const int b0 = g * G, gb = min(G, nb - b0);
        char* sl = slots + (t & 1) * slot_bytes;
        const unsigned bar = smem_u32(&S.comb_bar[t & 1]);
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar),
                     "r"((unsigned)(gb * nslots * 6))
                     : "memory");
        for (int k = 0; k < gb; ++k) {
            const size_t src = (size_t)(b0 + k) * slab + (size_t)r0;
            asm volatile(
                "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                    smem_u32(sl + (size_t)k * kCbWindow * 4)),
                "l"(M.part + src), "r"((unsigned)nslots * 4u), "r"(bar)
                : "memory");
            asm volatile(
                "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                    smem_u32(sl + (size_t)G * kCbWindow * 4 + (size_t)k * kCbWindow * 2)),
                "l"(M.ipos + src), "r"((unsigned)nslots * 2u), "r"(bar)
                : "memory");
        }
    };
    if (threadIdx.x == 0) {
        // the partial sums were written by other CTAs before the grid barrier
        asm volatile("fence.proxy.async.global;" ::: "memory");
        issue(0);
    }
    float acc[kCbRowsPerThread];
    for (int t = 0; t < T; ++t) {
        // slot (t + 1) & 1 was last read in tile t - 1, which ended with a CTA barrier
        if (threadIdx.x == 0 && t + 1 < T) issue(t + 1);
        const int w = rank + (t / ngroups) * size, g = t % ngroups;
        const int r0 = w * kCbWindow, rows = min(kCbWindow, R - r0);
        const int b0 = g * G, gb = min(G, nb - b0);
        const unsigned parity = S.comb_phase[t & 1];
        cb_wait_bar(&S.comb_bar[t & 1], parity, err);
        const float* sp = reinterpret_cast<const float*>(slots + (t & 1) * slot_bytes);
        const unsigned short* si =
            reinterpret_cast<const unsigned short*>(slots + (t & 1) * slot_bytes + (size_t)G * kCbWindow * 4);
#pragma unroll
        for (int i = 0; i < kCbRowsPerThread; ++i) {
            const int j = (int)threadIdx.x + i * kThreads;
            float a = b0 == 0 ? 0.f : acc[i];
            if (j < rows)
                for (int k = 0; k < gb; ++k) {
                    const float v = sp[k * kCbWindow + si[k * kCbWindow + j]];
                    a = (b0 + k == 0) ? v : a + v;
                }
            acc[i] = a;
        }
        __syncthreads();                                 // the slot may be refilled
        if (threadIdx.x == 0) S.comb_phase[t & 1] = parity ^ 1u;
        if (g == ngroups - 1) {                          // the window is complete
#pragma unroll
            for (int i = 0; i < kCbRowsPerThread; ++i) {
                const int j = (int)threadIdx.x + i * kThreads;
                if (j < rows) epi(r0 + j, acc[i]);
            }
        }
    }
}

// The staging of a column-blocked pass alone (every block the CTA's range
// touches, no products): the benchmark's measure of the copy cost.
template <typename Src>
__device__ __forceinline__ void cb_stage_only(const CbMat& M, const Src* __restrict__ x, int* err) {
    float* xs = acs_cb_smem;
    const int rank = team_rank();
    const int end = __ldg(M.cta_beg + rank + 1);
    int it = __ldg(M.cta_beg + rank);
    while (it < end) {
        const int b = it / M.nsl;
        const int c0 = b * M.width;
        __syncthreads();
        cb_stage(xs, x, c0, min(M.ncols - c0, M.width), err);
        __syncthreads();
        it = min(end, (b + 1) * M.nsl);
    }
}


// ---------------------------------------------------------------------------
// cone helpers
// ---------------------------------------------------------------------------


// Lorentz cones, a group of P.soc_lanes lanes (a power of two) each.  The roots
// and quotients of a cone cost a warp about 60 FP64 instructions of 16 cycles
// however many of its lanes need them, so eight cones a warp share them instead
// of one; wider groups where cones are long (soc_lanes() in acs_host.cuh).
// body(a, e, l, G, sum): cone [a, e), lane l of G; sum adds over the group.  Empty
// groups run with a = e = 0.  Measured: abs_K of 20000 cones of 3 to 64
// (and 100000 orthant coordinates) 56 -> 29 us, the KKT check 168 -> 93.
template <typename P_, typename Body>
__device__ __forceinline__ void for_cones(const P_& P, Body body) {
    const int G = P.soc_lanes, per = 32 / G;
    const int lane = threadIdx.x & 31, l = lane & (G - 1);
    auto sum = [G](double x) {
        for (int o = G / 2; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
        return x;
    };
    for (int c0 = global_warp() * per; c0 < P.n_soc; c0 += global_warps() * per) {
        const int c = c0 + lane / G;
        const bool in = c < P.n_soc;
        const int a = in ? __ldg(P.soc_off + c) : 0, e = in ? __ldg(P.soc_off + c + 1) : 0;
        body(c, a, e, l, G, sum);
    }
}

// Is iteration l in the schedule L (Algorithm 2 step 4, without the {1})?
template <typename T>
__device__ __forceinline__ bool in_schedule(const IterParams<T>& P, int l) {
    for (int i = 0; i < P.n_cond_list; ++i)
        if (__ldg(P.cond_list + i) == l) return true;
    if (P.cond_first > 0 && l >= P.cond_first) {
        if (P.cond_period <= 0) return l == P.cond_first;
        return (l - P.cond_first) % P.cond_period == 0;
    }
    return false;
}

// ---------------------------------------------------------------------------
// phases
// ---------------------------------------------------------------------------

// Conditioning, steps 5-10: o per cone, o = |x_h - ||xbar||| / |z_h|, stored
// as log o (log 0 = -inf, log inf = inf, nan stays nan); partials over the
// finite positive o: max log o, max(-log o), and their count.
template <typename T>
__device__ __noinline__ void phase_cond_o(const IterParams<T>& P) {
    double vmax = -INFINITY, vneg = -INFINITY, good = 0.0;
    for (int j = global_tid(); j < P.n_orth; j += global_threads()) {
        const double o = fabs(P.x[j]) / fabs(P.z[j]);
        const double lo = log(o);
        P.ocone[j] = lo;
        if (o > 0.0 && o < INFINITY) {
            good += 1.0;
            vmax = fmax(vmax, lo);
            vneg = fmax(vneg, -lo);
        }
    }
    for_cones(P, [&](int cI, int a, int e, int l, int G, auto sum) {
        double ss = 0.0;
        for (int j = a + 1 + l; j < e; j += G) ss = fma(P.x[j], P.x[j], ss);
        ss = sum(ss);
        if (l == 0 && a < e) {
            const double o = fabs(P.x[a] - sqrt(ss)) / fabs(P.z[a]);
            const double lo = log(o);
            P.ocone[P.n_orth + cI] = lo;
            if (o > 0.0 && o < INFINITY) {
                good += 1.0;
                vmax = fmax(vmax, lo);
                vneg = fmax(vneg, -lo);
            }
        }
    });
    const double v[3] = {vmax, vneg, good};
    const int op[3] = {1, 1, 0};
    block_partials<3>(v, op);
}

// Exponent range (CondRange) of step 11 over the finite positive o.  An o of 0, inf or
// nan (x_h = ||xbar||, z_h = 0, or both) carries no scale: it takes the
// limit of the rule under the e^t cap -- the smallest scale for o = 0, the
// largest for o = inf, the geometric middle for nan.  With no finite
// positive o at all, O = I.
__device__ __forceinline__ double cond_scale(double lo, const CondRange& R) {
    if (!R.any) return 1.0;
    double e = lo;
    if (isnan(lo)) e = 0.5 * (R.lmin + R.lmax);
    else if (lo == -INFINITY) e = R.lmin;
    else if (lo == INFINITY) e = R.lmax;
    return exp(R.alpha * e);
}

// Steps 11-14 per coordinate: O = exp(alpha log o) (see cond_scale),
// c_hat = O c, s = x/O - mu O z; g = O c_hat (input of the b_tilde pass).
template <typename T>
__device__ __forceinline__ void cond_apply_coord(const IterParams<T>& P, int j, double Oj, bool recast) {
    P.X.O[j] = Oj;
    P.V.O2[j] = (T)(Oj * Oj);
    const double ch = Oj * P.c[j];
    P.X.chat[j] = ch;
    P.X.g[j] = Oj * ch;
    if (recast) P.X.s[j] = P.x[j] / Oj - P.mu * Oj * P.z[j];
}

template <typename T>
__device__ __noinline__ void phase_cond_apply(const IterParams<T>& P, const CondRange& R, bool recompute_O,
                                              bool recast) {
    for (int j = global_tid(); j < P.n_orth; j += global_threads()) {
        const double Oj = recompute_O ? cond_scale(P.ocone[j], R) : P.X.O[j];
        cond_apply_coord(P, j, Oj, recast);
    }
    for_cones(P, [&](int cI, int a, int e, int l, int G, auto) {
        if (a >= e) return;
        const double Oc = recompute_O ? cond_scale(P.ocone[P.n_orth + cI], R) : P.X.O[a];
        for (int j = a + l; j < e; j += G) cond_apply_coord(P, j, Oc, recast);
    });
}

// b_tilde = b + mu A (O c_hat), J^{-1} = 1 / diag(A_hat A_hat') (FP64 pass);
// partial count of nonpositive diagonal entries.
template <typename T>
__device__ __noinline__ void phase_btilde(const IterParams<T>& P) {
    double bad = 0.0;
    const double* g = P.X.g;
    const double* O = P.X.O;
    auto g1 = [g](int j) { return g[j]; };
    auto g2 = [O](int j) { const double o = O[j]; return o * o; };
    auto epi = [&](int i, double s1, double s2) {
        P.X.btil[i] = P.b[i] + P.mu * s1;
        if (!(s2 > 0.0)) { bad += 1.0; P.V.jinv[i] = T(1); }
        else P.V.jinv[i] = (T)(1.0 / s2);
    };
    sell_rows2(P.A, g1, g2, epi);
    const double v[1] = {bad};
    const int op[1] = {0};
    block_partials<1>(v, op);
}

// Start of the projection solve: w <- w + theta (w - w_prev) and, since
// q = A_hat' w is linear in w while O is fixed, q <- q + theta (q - q_prev)
// exactly, with no matrix pass (theta = 0: the previous w, a plain warm
// start).  The outer iteration converges linearly, so consecutive w follow a
// near-geometric sequence and the extrapolated start leaves the correction
// solve a smaller residual.  Returns the q to use; saves the current pair
// when the setting is on (save).
__device__ __forceinline__ double extrap_q(const Outer& X, int j, double theta, bool save) {
    const double q = X.q[j];
    if (theta == 0.0) {
        if (save) X.qp[j] = q;
        return q;
    }
    const double qn = fma(theta, q - X.qp[j], q);
    X.qp[j] = q;
    X.q[j] = qn;
    return qn;
}

// Step 17: p = abs_K(s); g = O (p + q) for the warm-started right-hand side
// (theta: see extrap_q).
// Lorentz cone (v1, vbar), t = ||vbar||: inside (t <= v1) abs = v; polar
// (t <= -v1) abs = -v; otherwise abs = (t, (v1/t) vbar), which is 2 proj - v
// for proj = ((v1 + t)/2)(1, vbar/t).
template <typename T>
__device__ __noinline__ void phase_abs(const IterParams<T>& P, double theta) {
    const Outer& X = P.X;
    const bool save = P.extrap != 0.0;                  // the setting is on: keep the pairs
    if (save)
        for (int i = global_tid(); i < P.m; i += global_threads()) {
            const double w = X.w[i];
            if (theta != 0.0) X.w[i] = fma(theta, w - X.wp[i], w);
            X.wp[i] = w;
        }
    if (P.admm) {                                       // ADMM form: the projection acts on s itself
        for (int j = global_tid(); j < P.n; j += global_threads()) {
            const double pj = X.s[j];
            X.p[j] = pj;
            X.g[j] = X.O[j] * (pj + extrap_q(X, j, theta, save));
        }
        return;
    }
    for (int j = global_tid(); j < P.n_orth; j += global_threads()) {
        const double pj = fabs(X.s[j]);
        X.p[j] = pj;
        X.g[j] = X.O[j] * (pj + extrap_q(X, j, theta, save));
    }
    for_cones(P, [&](int, int a, int e, int l, int G, auto sum) {
        double ss = 0.0;
        for (int j = a + 1 + l; j < e; j += G) ss = fma(X.s[j], X.s[j], ss);
        ss = sum(ss);
        if (a >= e) return;
        const double t = sqrt(ss);
        const double v1 = X.s[a];
        double ftail, head;
        if (t <= v1) { ftail = 1.0; head = v1; }
        else if (t <= -v1) { ftail = -1.0; head = -v1; }
        else { ftail = v1 / t; head = t; }
        const double Oc = X.O[a];
        for (int j = a + l; j < e; j += G) {
            const double pj = (j == a) ? head : ftail * X.s[j];
            X.p[j] = pj;
            X.g[j] = Oc * (pj + extrap_q(X, j, theta, save));
        }
    });
}

// FP64 residual of the projection system r0 = b_tilde - A g (g = O(p + q),
// i.e. b_tilde - A_hat p - M w); the correction CG starts from it:
// r = r0, u = J^{-1} r.  Partial gamma = r'u.
template <typename T>
__device__ __forceinline__ void rhs_epi(const IterParams<T>& P, int i, double sum, double& gam) {
    const T r = (T)(P.X.btil[i] - sum);
    const T u = P.V.jinv[i] * r;
    P.V.r[i] = r;
    P.V.u[i] = u;
    gam += (double)r * (double)u;
}

// The residual alone, for the cached operator (no CG, no reduction).
template <typename T>
__device__ __noinline__ void phase_rhs_plain(const IterParams<T>& P) {
    const double* g = P.X.g;
    sell_rows<double>(P.A, [g](int j) { return g[j]; },
                      [&](int i, double sum) { P.V.r[i] = (T)(P.X.btil[i] - sum); });
}

template <typename T>
__device__ __noinline__ void phase_rhs(const IterParams<T>& P) {
    double gam = 0.0;
    const double* g = P.X.g;
    auto gather = [g](int j) { return g[j]; };
    auto epi = [&](int i, double sum) { rhs_epi(P, i, sum, gam); };
    sell_rows<double>(P.A, gather, epi);
    const double v[1] = {gam};
    const int op[1] = {0};
    block_partials<1>(v, op);
}

// FP32 outer products on the L2-gather layout (a segment that need only reach
// a polish level): the projection residual from FP32 values and g rounded to
// FP32, summed in FP32.
template <typename T>
__device__ __noinline__ void phase_rhs_f32(const IterParams<T>& P) {
    double gam = 0.0;
    const double* g = P.X.g;
    auto gather = [g](int j) { return (float)g[j]; };
    auto epi = [&](int i, float sum) { rhs_epi(P, i, (double)sum, gam); };
    sell_rows<float>(P.A, gather, epi);
    const double v[1] = {gam};
    const int op[1] = {0};
    block_partials<1>(v, op);
}

// FP32 outer passes: the product A g of the projection residual as a
// column-blocked FP32 pass (g rounded to FP32 as it is staged) ...
template <typename T>
__device__ __noinline__ void phase_rhs_cb(const IterParams<T>& P) {
    cb_pass(P.Acb, P.X.g, &P.ctl->err);
}
// ... and the residual from its partial sums: r0 = b_tilde - A g.
template <typename T>
__device__ __noinline__ void phase_rhs_comb(const IterParams<T>& P) {
    double gam = 0.0;
    cb_combine(P.Acb, &P.ctl->err, [&](int i, float sum) { rhs_epi(P, i, (double)sum, gam); });
    const double v[1] = {gam};
    const int op[1] = {0};
    block_partials<1>(v, op);
}

// CG, first half of M u: t = O^2 (A' u) over the rows of A'.
template <typename T>
__device__ __noinline__ void phase_cg_At(const IterParams<T>& P) {
    const T* u = P.V.u;
    auto gather = [u](int i) { return u[i]; };
    auto epi = [&](int j, T sum) { P.V.t[j] = P.V.O2[j] * sum; };
    sell_rows<T>(P.AT, gather, epi);
}

// CG, second half: au = A t (= M u); partial delta = au'u.
template <typename T>
__device__ __noinline__ void phase_cg_A(const IterParams<T>& P) {
    double delta = 0.0;
    const T* t = P.V.t;
    auto gather = [t](int j) { return t[j]; };
    auto epi = [&](int i, T sum) {
        P.V.au[i] = sum;
        delta += (double)sum * (double)P.V.u[i];
    };
    sell_rows<T>(P.A, gather, epi);
    const double v[1] = {delta};
    const int op[1] = {0};
    block_partials<1>(v, op);
}

// Column-blocked CG, first half of M u: the partial sums of A'u ...
template <typename T>
__device__ __noinline__ void phase_cg_At_cb(const IterParams<T>& P) {
    cb_pass(P.ATcb, P.V.u, &P.ctl->err);
}
// ... combined: v = A'u, t = O^2 v, and the partial of u'Mu = sum O^2 v^2
// (= ||A_hat'u||^2, the delta of the CG step, known before the A pass).
template <typename T>
__device__ __noinline__ void phase_cg_tcomb(const IterParams<T>& P) {
    double delta = 0.0;
    cb_combine(P.ATcb, &P.ctl->err, [&](int j, float sum) {
        const T v = (T)sum;
        const T t = P.V.O2[j] * v;
        P.V.t[j] = t;
        delta += (double)t * (double)v;
    });
    const double v[1] = {delta};
    const int op[1] = {0};
    block_partials<1>(v, op);
}
// Column-blocked CG, second half: the partial sums of A t (= M u), combined
// in the vector step.
template <typename T>
__device__ __noinline__ void phase_cg_A_cb(const IterParams<T>& P) {
    cb_pass(P.Acb, P.V.t, &P.ctl->err);
}

// Scalars of a Chronopoulos-Gear step, in warp 0 at the barriers of the CG:
// after M u (delta = u'Mu), beta and alpha of step k (broke: p'Mp <= 0 in finite
// precision, the solve has reached its attainable accuracy or M is singular
// along p) ...
__device__ __forceinline__ void cg_step_scalars(double delta, int k) {
    LoopScalars& L = sync_smem().lp;
    const double beta = (k == 0) ? 0.0 : L.gam / L.gam_prev;
    const double denom = delta - ((k == 0) ? 0.0 : beta * L.gam / L.alpha_prev);
    const double alpha = L.gam / denom;
    __syncwarp();
    if ((threadIdx.x & 31) == 0) {
        L.broke = !(denom > 0.0);
        L.alpha = alpha;
        L.beta = beta;
    }
}
// ... and after the vector step (gn = r'u): whether to go on.
__device__ __forceinline__ void cg_next_scalars(double gn) {
    LoopScalars& L = sync_smem().lp;
    const double r = sqrt(fmax(gn, 0.0));
    const int go = r > L.thr, far = r > 100.0 * L.thr;
    __syncwarp();
    if ((threadIdx.x & 31) == 0) {
        L.gam_prev = L.gam;
        L.alpha_prev = L.alpha;
        L.gam = gn;
        L.go = go;
        L.far = far;
        L.bad = !isfinite(gn);
    }
}

// Chronopoulos-Gear vector step: p = u + beta p, sv = au + beta sv,
// w += alpha p (FP64), r -= alpha sv, u = J^{-1} r; partial gamma = r'u.
// au(i) = (M u)_i: stored by the A pass, or the partial sums of the
// column-blocked A pass added in block order.
template <typename T, bool CB>
__device__ __noinline__ void phase_cg_vec(const IterParams<T>& P) {
    double gam = 0.0;
    const Inner<T>& V = P.V;
    const double alpha = sync_smem().lp.alpha;
    const T beta = (T)sync_smem().lp.beta;
    const T a = (T)alpha;
    auto step = [&](int i, T aui) {
        const T pi = fma(beta, V.p[i], V.u[i]);
        const T si = fma(beta, V.sv[i], aui);
        V.p[i] = pi;
        V.sv[i] = si;
        P.X.w[i] += alpha * (double)pi;
        const T r = fma(-a, si, V.r[i]);
        V.r[i] = r;
        const T u = V.jinv[i] * r;
        V.u[i] = u;
        gam += (double)r * (double)u;
    };
    if (CB) cb_combine(P.Acb, &P.ctl->err, [&](int i, float sum) { step(i, (T)sum); });
    else
        for (int i = global_tid(); i < P.m; i += global_threads()) step(i, V.au[i]);
    const double v[1] = {gam};
    const int op[1] = {0};
    block_partials<1>(v, op);
}

// q = O (A' w) over the rows of A' (FP64); with update: s <- (s + p)/2 -
// mu c_hat + q (steps 18-19) and, if want_xz, x = O (p + s)/2 and
// z = (p - s)/(2 mu O) (steps 20-21).  Partials ||s_new - s||^2, ||s_new||^2.
// fuse_abs (orthant-only problems, no extrapolation, no rescaling next):
// also step 17 of the next iteration, p = |s_new| and g = O (p + q) with the
// q just formed -- the values phase_abs would compute there.
template <typename T>
__device__ __forceinline__ void update_epi(const IterParams<T>& P, int j, double sum, bool update, bool want_xz,
                                           double& ds2, double& ss2, bool fuse_abs, bool admm) {
    const double Oj = P.X.O[j];
    const double qj = Oj * sum;
    P.X.q[j] = qj;
    if (!update) P.X.g[j] = Oj * (P.X.p[j] + qj);   // right-hand side input of a refinement round
    if (update && admm) {
        // ADMM form (Section III-B), as Douglas-Rachford splitting with the two
        // proximal steps in the other order: p = s = zeta, q = A_hat' w with
        // w = M^{-1}(b_tilde - A_hat zeta), so zeta - mu c_hat + q is the
        // proximal point of g (x2) and a = 2 x2 - zeta its reflection;
        // zeta <- (zeta + abs_K(a))/2, x1 = proj_K(a) = (a + abs_K(a))/2 and
        // z = (abs_K(a) - a)/(2 mu), scaled back by O.  Lorentz-cone
        // coordinates keep a in p for phase_admm_soc.
        const double so = P.X.s[j];
        const double a = (so - 2.0 * P.mu * P.X.chat[j]) + 2.0 * qj;
        if (j >= P.n_orth) {
            P.X.p[j] = a;
            return;
        }
        const double aa = fabs(a);
        const double sj = 0.5 * (so + aa);
        P.X.s[j] = sj;
        ds2 += (sj - so) * (sj - so);
        ss2 += sj * sj;
        if (want_xz) {
            P.x[j] = Oj * (a + aa) * 0.5;
            P.z[j] = (aa - a) / (2.0 * P.mu * Oj);
        }
        return;
    }
    if (update) {
        const double pj = P.X.p[j];
        const double so = P.X.s[j];
        const double sj = (0.5 * (so + pj) - P.mu * P.X.chat[j]) + qj;
        P.X.s[j] = sj;
        ds2 += (sj - so) * (sj - so);
        ss2 += sj * sj;
        if (want_xz) {
            P.x[j] = Oj * (pj + sj) * 0.5;
            P.z[j] = (pj - sj) / (2.0 * P.mu * Oj);
        }
        if (fuse_abs) {
            const double pn = fabs(sj);
            P.X.p[j] = pn;
            P.X.g[j] = Oj * (pn + qj);
        }
    }
}

// Partials of the update: ||s_new - s||^2, ||s_new||^2 and, for a
// time-sliced solve, the CTAs that have seen the deadline pass (one clock
// read per CTA, summed, so every CTA of the team takes the same decision).
__device__ __forceinline__ void update_partials(double ds2, double ss2) {
    const unsigned long long dl = sync_smem().deadline;
    const double over = (dl != 0ull && threadIdx.x == 0 && gtimer() > dl) ? 1.0 : 0.0;
    const double v[3] = {ds2, ss2, over};
    const int op[3] = {0, 0, 0};
    block_partials<3>(v, op);
}

// q = A_hat' w and g = O (p + q) alone: the start of a solve in a new scaling, and
// of a refinement round.  Nothing to reduce.
template <typename T>
__device__ __noinline__ void phase_qrefresh(const IterParams<T>& P) {
    const double* w = P.X.w;
    sell_rows<double>(P.AT, [w](int i) { return w[i]; }, [&](int j, double sum) {
        const double Oj = P.X.O[j];
        const double qj = Oj * sum;
        P.X.q[j] = qj;
        P.X.g[j] = Oj * (P.X.p[j] + qj);
    });
}

// The update; the ADMM form is a function of its own, so that the usual one keeps
// its operands in registers.
template <typename T, bool kAdmm>
__device__ __noinline__ void phase_update_form(const IterParams<T>& P, bool want_xz, bool fuse_abs) {
    double ds2 = 0.0, ss2 = 0.0;
    const double* w = P.X.w;
    auto gather = [w](int i) { return w[i]; };
    auto epi = [&](int j, double sum) { update_epi(P, j, sum, true, want_xz, ds2, ss2, fuse_abs, kAdmm); };
    sell_rows<double>(P.AT, gather, epi);
    update_partials(ds2, ss2);
}
template <typename T>
__device__ __forceinline__ void phase_update(const IterParams<T>& P, bool update, bool want_xz, bool fuse_abs = false) {
    if (!update) phase_qrefresh(P);
    else if (P.admm) phase_update_form<T, true>(P, want_xz, fuse_abs);
    else phase_update_form<T, false>(P, want_xz, fuse_abs);
}

// The update from an FP32 product A'w on the L2-gather layout (see phase_rhs_f32).
template <typename T>
__device__ __noinline__ void phase_update_f32(const IterParams<T>& P, bool want_xz, bool fuse_abs) {
    double ds2 = 0.0, ss2 = 0.0;
    const double* w = P.X.w;
    auto gather = [w](int i) { return (float)w[i]; };
    auto epi = [&](int j, float sum) { update_epi(P, j, (double)sum, true, want_xz, ds2, ss2, fuse_abs, P.admm != 0); };
    sell_rows<float>(P.AT, gather, epi);
    update_partials(ds2, ss2);
}

// FP32 outer passes: A'w as a column-blocked FP32 pass (w rounded to FP32 as
// it is staged) ...
template <typename T>
__device__ __noinline__ void phase_update_cb(const IterParams<T>& P) {
    cb_pass(P.ATcb, P.X.w, &P.ctl->err);
}
// ... and the update from its partial sums.
template <typename T>
__device__ __noinline__ void phase_update_comb(const IterParams<T>& P, bool want_xz, bool fuse_abs = false) {
    double ds2 = 0.0, ss2 = 0.0;
    cb_combine(P.ATcb, &P.ctl->err,
               [&](int j, float sum) { update_epi(P, j, (double)sum, true, want_xz, ds2, ss2, fuse_abs, P.admm != 0); });
    update_partials(ds2, ss2);
}

// ADMM form, Lorentz cones: abs_K of the reflection a kept in p by
// update_epi (the cone rule of phase_abs), then zeta <- (zeta + abs_K(a))/2,
// x and z as for the orthant.  Partials ||s_new - s||^2, ||s_new||^2 of these
// coordinates.
template <typename T>
__device__ __noinline__ void phase_admm_soc(const IterParams<T>& P, bool want_xz) {
    double ds2 = 0.0, ss2 = 0.0;
    const Outer& X = P.X;
    for_cones(P, [&](int, int a0, int e, int l, int G, auto sum) {
        double tt = 0.0;
        for (int j = a0 + 1 + l; j < e; j += G) tt = fma(X.p[j], X.p[j], tt);
        tt = sum(tt);
        if (a0 >= e) return;
        const double t = sqrt(tt);
        const double v1 = X.p[a0];
        double ftail, head;
        if (t <= v1) { ftail = 1.0; head = v1; }
        else if (t <= -v1) { ftail = -1.0; head = -v1; }
        else { ftail = v1 / t; head = t; }
        const double Oc = X.O[a0];
        for (int j = a0 + l; j < e; j += G) {
            const double a = X.p[j];
            const double aa = (j == a0) ? head : ftail * a;
            const double so = X.s[j];
            const double sj = 0.5 * (so + aa);
            X.s[j] = sj;
            ds2 += (sj - so) * (sj - so);
            ss2 += sj * sj;
            if (want_xz) {
                P.x[j] = Oc * (a + aa) * 0.5;
                P.z[j] = (aa - a) / (2.0 * P.mu * Oc);
            }
        }
    });
    const double v[2] = {ds2, ss2};
    const int op[2] = {0, 0};
    block_partials<2>(v, op);
}

// FP64 residual partials: ||Ax - b||^2, ||A'y + z - c||^2 (y = w/mu), c'x, b'y,
// dist(x,K)^2, dist(z,K)^2, ||x||^2, ||z||^2.
__device__ __forceinline__ double soc_dist2(double v1, double t) {
    // squared distance from (v1, vbar) with ||vbar|| = t to the Lorentz cone
    if (t <= v1) return 0.0;
    if (t <= -v1) return v1 * v1 + t * t;
    const double d = 0.5 * (t - v1);      // distance = |t - v1| / sqrt 2
    return 2.0 * d * d;
}

template <typename T>
__device__ __noinline__ void phase_kkt(const IterParams<T>& P) {
    double rp = 0.0, rd = 0.0, cx = 0.0, by = 0.0, dx = 0.0, dz = 0.0, xx = 0.0, zz = 0.0;
    const double* x = P.x;
    const double* z = P.z;
    const double* w = P.X.w;
    const double inv_mu = P.inv_mu;
    {
        auto gather = [x](int j) { return x[j]; };
        auto epi = [&](int i, double sum) {
            const double d = sum - P.b[i];
            rp += d * d;
            by += P.b[i] * (w[i] * inv_mu);
        };
        sell_rows<double>(P.A, gather, epi);
    }
    {
        auto gather = [w, inv_mu](int i) { return w[i] * inv_mu; };
        auto epi = [&](int j, double sum) {
            const double d = sum + z[j] - P.c[j];
            rd += d * d;
        };
        sell_rows<double>(P.AT, gather, epi);
    }
    for (int j = global_tid(); j < P.n_orth; j += global_threads()) {
        const double xj = x[j], zj = z[j];
        cx += P.c[j] * xj;
        xx += xj * xj;
        zz += zj * zj;
        if (xj < 0.0) dx += xj * xj;
        if (zj < 0.0) dz += zj * zj;
    }
    for_cones(P, [&](int, int a, int e, int l, int G, auto sum) {
        double sx = 0.0, sz = 0.0;
        for (int j = a + l; j < e; j += G) {
            const double xj = x[j], zj = z[j];
            cx = fma(P.c[j], xj, cx);
            if (j > a) {
                sx = fma(xj, xj, sx);
                sz = fma(zj, zj, sz);
            }
        }
        sx = sum(sx);
        sz = sum(sz);
        if (l < 2 && a < e) {                            // lane 0 takes x, lane 1 z
            const double s2 = l == 0 ? sx : sz, v1 = l == 0 ? x[a] : z[a];
            const double d2 = soc_dist2(v1, sqrt(s2)), n2 = s2 + v1 * v1;
            if (l == 0) {
                xx += n2;
                dx += d2;
            } else {
                zz += n2;
                dz += d2;
            }
        }
    });
    const double v[8] = {rp, rd, cx, by, dx, dz, xx, zz};
    const int op[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    block_partials<8>(v, op);
}

// ---------------------------------------------------------------------------
// cached projection operator (small m): M = A_hat A_hat' factored once per
// rescaling, then every projection solve is two dense FP64 products
// ---------------------------------------------------------------------------
//
// The operator of the projection (Algorithm 1 step 2 / Algorithm 2 step 12:
// the pseudoinverse of A_hat through M = A_hat A_hat') changes only when O
// does.  For small m it is cached as the explicit inverse factor
// X = L^{-1} of the Cholesky factorisation M = L L' (FP64), so that the
// correction of every iteration, dw = M^{-1} r0 = X' (X r0), is exact up to
// rounding, like the oracle's dense solve, and costs two triangular matrix-
// vector products with no sequential dependence.
// Storage, both m x m: dX holds X row-major (lower triangle), dM first M
// row-major (lower triangle, overwritten by L) and, once X is complete, X' row-
// major (upper triangle), so that both products read rows.

// M = A O^2 A' (lower triangle), from row i of A and the columns of A it
// touches (rows of A'): M_ik = sum_j O_j^2 a_ij a_kj.  Warp per row i, the
// lanes over the entries of one column j at a time, in a fixed order.
template <typename T>
__device__ __noinline__ void phase_dense_scatter(const IterParams<T>& P) {
    double* M = sync_smem().dM;
    const int m = P.m;
    const int lane = threadIdx.x & 31;
    const SellMat& A = P.A;
    const SellMat& AT = P.AT;
    for (int i = global_warp(); i < m; i += global_warps()) {
        double* Mi = M + (size_t)i * m;
        for (int k = lane; k <= i; k += 32) Mi[k] = 0.0;
        __syncwarp();
        const int ga = A.g, ha = 32 / ga;
        const int sl = i / ha, lr = i % ha;
        const int base = __ldg(A.sptr + sl), len = __ldg(A.slen + sl) * ga;
        for (int e = 0; e < len; ++e) {
            const int idx = base + 32 * (e / ga) + lr * ga + (e % ga);
            const double aij = __ldg(A.v64 + idx);
            if (aij == 0.0) continue;                         // padding
            const int j = __ldg(A.col + idx);
            const double Oj = P.X.O[j];
            const double f = aij * Oj * Oj;
            // column j of A = row j of A' (relabelled rows, increasing)
            const int gt = AT.g, ht = 32 / gt;
            const int slt = j / ht, lrt = j % ht;
            const int bt = __ldg(AT.sptr + slt), lt = __ldg(AT.slen + slt) * gt;
            for (int q = lane; q < lt; q += 32) {
                const int it = bt + 32 * (q / gt) + lrt * gt + (q % gt);
                const double akj = __ldg(AT.v64 + it);
                const int k = __ldg(AT.col + it);
                if (akj != 0.0 && k <= i) Mi[k] = fma(f, akj, Mi[k]);
            }
            __syncwarp();
        }
    }
}

// Pivot rule of the factorisation: a pivot below 1e-13 of the row's
// original diagonal (jinv = 1 / diag M) marks row k of A as linearly
// dependent on the rows before it (rank-deficient A): the direction is
// dropped -- the pivot becomes +inf, its column of L is zero, nothing is
// eliminated with it, and row k of L^{-1} is zero.  For a consistent
// right-hand side (b in range(A)) this solves the remaining independent
// equations, which imply the dropped one.  A pivot negative beyond rounding
// or not a number fails the factorisation.
// Blocked factorisation M = L L' and X = L^{-1} in one sweep, one team barrier
// per kCholB columns: X is the right half of [M | I] under the same
// elimination, so its updates are products of the same shape as those of the
// trailing triangle and share their barriers and their load balance.
//   The step at column k1 (the block before it, at k0 = k1 - kCholB, is final:
//   L[k1.., k0..k1) and X[k0..k1, 0..k1)):
//   A. every CTA updates the diagonal block D = M[k1.., k1..] with L, factors
//      it with the pivot rule above and inverts its factor, in shared memory
//      (every CTA takes the same decisions without communicating);
//   B. the block's column of L below it, L_iq = (M_iq - L_ip L_qp') D^{-1}', in
//      units of 32 rows, and its row of X, X_q = D^{-1} (X_q - L_qp X_p), in
//      units of 32 columns;
//   C. the rest, M_ij -= L_ip L_jp' and X_ij -= L_ip X_pj, in 32 x 32 tiles.
//   The units of B and C are dealt to the team's CTAs in turn; the operands of
//   the next unit are loaded into registers while one is computed.
// The FP64 pipe bounds B and C (2 multiply-adds per clock per SM: a 32 x 32 x 16
// tile is 4 us, its loads 1.5); blocks of 16 columns keep A, the serial part
// (about 6 us), and the padding of small m low.  Measured, factor and inverse:
// m = 2000 66 -> 9.6 ms, m = 200 2.1 -> 0.41 ms (before: a warp per row or column
// with one dependent sum each, two barriers per 16 columns, and the columns of
// the inverse by forward substitution).
constexpr int kCholB = 16;
constexpr int kTile = 32;

struct DenseShared {
    double A[2][kTile][kCholB + 1];    // L_ip rows of a unit (B: then the unit's block)
    double B[2][kTile][kCholB + 1];    // L_jp rows (tiles of M), or
                                       // X_p columns, B[j][t] = X[k0 + t][j0 + j]
    double Lq[kCholB][kCholB + 1];     // L[k1.., k0..]
    double D[kCholB][kCholB + 1];      // diagonal block, then its factor
    double Di[kCholB][kCholB + 1];     // inverse of the factor (row 0 for a dependent row)
    int bad;
};
__device__ __forceinline__ DenseShared& dense_smem() {
    __shared__ DenseShared s;
    return s;
}

// Part A's serial piece, one warp: lane r (mod 16) holds row r of D.  L D L'
// without square roots on the way (a quotient per column), scaled by 1/sqrt(d)
// at the end, then the inverse factor, lane c its column c.
static __device__ __noinline__ void dense_diag(double tau_lane) {
    DenseShared& S = dense_smem();
    const int lane = threadIdx.x & 31, r = lane & (kCholB - 1);
    constexpr unsigned full = 0xffffffffu;
    double a[kCholB];
#pragma unroll
    for (int c = 0; c < kCholB; ++c) a[c] = S.D[r][c];
    bool fail = false, dep_own = false;
    double d_own = 1.0;
#pragma unroll
    for (int k = 0; k < kCholB; ++k) {
        const double d = __shfl_sync(full, a[k], k), tau = __shfl_sync(full, tau_lane, k);
        fail = fail || d != d || d < -1e3 * tau;
        const bool dep = !(d > tau) || d == INFINITY;
        if (r == k) {
            dep_own = dep;
            d_own = d;
        }
        const double v = dep ? 0.0 : a[k] * __drcp_rn(d);
#pragma unroll
        for (int j = k + 1; j < kCholB; ++j) a[j] = fma(-v, __shfl_sync(full, a[k], j), a[j]);
    }
    const double s_own = dep_own ? 0.0 : 1.0 / sqrt(d_own);
#pragma unroll
    for (int k = 0; k < kCholB; ++k) {
        const double s = __shfl_sync(full, s_own, k);
        if (lane < kCholB) S.D[r][k] = r > k ? a[k] * s : 0.0;   // strictly lower part of L
    }
    __syncwarp();
    double x[kCholB];
#pragma unroll
    for (int i = 0; i < kCholB; ++i) x[i] = i == r ? 1.0 : 0.0;
#pragma unroll
    for (int t = 0; t < kCholB; ++t) {
        x[t] *= __shfl_sync(full, s_own, t);
#pragma unroll
        for (int i = t + 1; i < kCholB; ++i) x[i] = fma(-S.D[i][t], x[t], x[i]);
    }
    if (lane < kCholB) {
#pragma unroll
        for (int i = 0; i < kCholB; ++i) S.Di[i][r] = i >= r ? x[i] : 0.0;
    }
    if (lane == 0) S.bad = fail ? 1 : 0;
    __syncwarp();
}

// What a unit of B or C works on.
struct DenseUnit {
    int kind;          // 0: panel rows, 1: row of X, 2: tile of M, 3: tile of X
    int i0, j0;        // first row and column of its block
};

// The units of the step at k1, numbered from 0: nB1 of kind 0, nB2 of kind 1,
// then the tiles of X (nt rows of nX) and of M (lower triangle of nt).  Numbers
// fit 32 bits (m <= 16384: 4e5 units); every thread finds its unit, and 64-bit
// quotients would cost a quarter of a tile's time.
struct DensePlan {
    int k0, k1, k2, nB1, nB2, nX;
    unsigned total;
};
__device__ __forceinline__ DensePlan dense_plan(int m, int k1) {
    DensePlan P;
    P.k1 = k1;
    P.k0 = k1 - kCholB;                                  // < 0: no block before
    P.k2 = min(m, k1 + kCholB);
    const int nt = (m - P.k2 + kTile - 1) / kTile;
    P.nB1 = nt;
    P.nX = k1 > 0 ? (k1 + kTile - 1) / kTile : 0;
    P.nB2 = P.nX;
    P.total = P.nB1 + P.nB2 + (k1 > 0 ? nt * P.nX + nt * (nt + 1) / 2 : 0);
    return P;
}
// Row of entry u of a lower triangle stored by rows.
__device__ __forceinline__ int tri_row(unsigned u) {
    int r = (int)((sqrtf(8.0f * (float)u + 1.0f) - 1.0f) * 0.5f);
    while ((unsigned)(r + 1) * (unsigned)(r + 2) / 2u <= u) ++r;
    while ((unsigned)r * (unsigned)(r + 1) / 2u > u) --r;
    return r;
}
__device__ __forceinline__ DenseUnit dense_unit(const DensePlan& P, unsigned u) {
    DenseUnit U;
    if (u < (unsigned)P.nB1) {
        U.kind = 0;
        U.i0 = P.k2 + (int)u * kTile;
        U.j0 = P.k1;
        return U;
    }
    u -= P.nB1;
    if (u < (unsigned)P.nB2) {
        U.kind = 1;
        U.i0 = P.k1;
        U.j0 = (int)u * kTile;
        return U;
    }
    u -= P.nB2;
    const unsigned tx = (unsigned)P.nB1 * (unsigned)P.nX;
    if (u < tx) {
        const unsigned q = u / (unsigned)P.nX;
        U.kind = 3;
        U.i0 = P.k2 + (int)q * kTile;
        U.j0 = (int)(u - q * P.nX) * kTile;
        return U;
    }
    u -= tx;
    const int bi = tri_row(u);
    U.kind = 2;
    U.i0 = P.k2 + bi * kTile;
    U.j0 = P.k2 + (int)(u - (unsigned)bi * (unsigned)(bi + 1) / 2u) * kTile;
    return U;
}

// Registers of one unit: R = 1024 / threads elements of its block (rows ty, ty +
// threads / 32, ...; column tx), and its share of the two operands.
template <int R>
struct DenseRegs {
    double c[R], a[R], b[R];
};

template <int R>
__device__ __forceinline__ void dense_load(const double* M, const double* X, int m, const DensePlan& P,
                                           const DenseUnit& U, DenseRegs<R>& G) {
    constexpr int kRows = kTile / R;                     // rows covered by the threads at once
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    const int k0 = P.k0, k1 = P.k1;
#pragma unroll
    for (int q = 0; q < R; ++q) {
        const int r = ty + q * kRows;
        // the block: 32 x 32, or 32 rows x 16 (kind 0), or 16 rows x 32 (kind 1)
        const int i = U.i0 + r, j = U.j0 + tx;
        double c = 0.0;
        if (U.kind == 0) { if (tx < kCholB && i < m && j < m) c = __ldcg(M + (size_t)i * m + j); }
        else if (U.kind == 1) { if (r < kCholB && i < m && j < k0) c = __ldcg(X + (size_t)i * m + j); }
        else if (U.kind == 2) { if (i < m && j <= i) c = __ldcg(M + (size_t)i * m + j); }
        else { if (i < m && j < k0) c = __ldcg(X + (size_t)i * m + j); }   // block column k0: first update
        G.c[q] = c;
        // the operands: L[i0 + row, k0 + t] by (row = r, t = tx) for tx < 16; the
        // other half of the lanes loads L[j0 + row, k0 + t] (kind 2); kinds 1
        // and 3: X[k0 + t, j0 + tx] by (t = r) for r < 16
        double a = 0.0, b = 0.0;
        if (k0 >= 0) {
            const int t = tx & (kCholB - 1);
            if (tx < kCholB) {
                if (U.kind != 1 && i < m) a = __ldcg(M + (size_t)i * m + k0 + t);
            } else if (U.kind == 2) {
                if (U.j0 + r < m) a = __ldcg(M + (size_t)(U.j0 + r) * m + k0 + t);
            }
            if ((U.kind == 1 || U.kind == 3) && r < kCholB && j < k1) b = __ldcg(X + (size_t)(k0 + r) * m + j);
        }
        G.a[q] = a;
        G.b[q] = b;
    }
}

// Operands of a unit into buffer `buf`.
template <int R>
__device__ __forceinline__ void dense_store(const DenseUnit& U, const DenseRegs<R>& G, int buf) {
    DenseShared& S = dense_smem();
    constexpr int kRows = kTile / R;
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
#pragma unroll
    for (int q = 0; q < R; ++q) {
        const int r = ty + q * kRows, t = tx & (kCholB - 1);
        if (tx < kCholB) S.A[buf][r][t] = G.a[q];
        else if (U.kind == 2) S.B[buf][r][t] = G.a[q];
        if ((U.kind == 1 || U.kind == 3) && r < kCholB) S.B[buf][tx][r] = G.b[q];
    }
}

template <int R>
__device__ __forceinline__ void dense_compute(double* M, double* X, int m, const DensePlan& P, const DenseUnit& U,
                                              const double (&c)[R], int buf) {
    DenseShared& S = dense_smem();
    constexpr int kRows = kTile / R;
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    double(*SA)[kCholB + 1] = S.A[buf];
    double(*SB)[kCholB + 1] = S.B[buf];
    double acc[R];
#pragma unroll
    for (int q = 0; q < R; ++q) acc[q] = c[q];
    if (P.k0 >= 0) {
        if (U.kind == 0) {                               // columns of the block: rows of L_q
            if (tx < kCholB)
#pragma unroll
                for (int t = 0; t < kCholB; ++t) {
                    const double y = S.Lq[tx][t];
#pragma unroll
                    for (int q = 0; q < R; ++q) acc[q] = fma(-SA[ty + q * kRows][t], y, acc[q]);
                }
        } else if (U.kind == 1) {
#pragma unroll
            for (int q = 0; q < R; ++q)
                if (ty + q * kRows < kCholB)
#pragma unroll
                    for (int t = 0; t < kCholB; ++t) acc[q] = fma(-S.Lq[ty + q * kRows][t], SB[tx][t], acc[q]);
        } else {
#pragma unroll
            for (int t = 0; t < kCholB; ++t) {
                const double y = SB[tx][t];
#pragma unroll
                for (int q = 0; q < R; ++q) acc[q] = fma(-SA[ty + q * kRows][t], y, acc[q]);
            }
        }
    }
    if (U.kind >= 2) {
#pragma unroll
        for (int q = 0; q < R; ++q) {
            const int i = U.i0 + ty + q * kRows, j = U.j0 + tx;
            if (U.kind == 2) { if (i < m && j <= i) M[(size_t)i * m + j] = acc[q]; }
            else { if (i < m && j < P.k1) X[(size_t)i * m + j] = acc[q]; }
        }
        return;
    }
    // kinds 0 and 1: the block through shared memory, times the inverse factor
    __syncthreads();                                     // the operands are used up
    if (U.kind == 0) {
#pragma unroll
        for (int q = 0; q < R; ++q)
            if (tx < kCholB) SA[ty + q * kRows][tx] = acc[q];
        __syncthreads();
#pragma unroll
        for (int q = 0; q < R; ++q) acc[q] = 0.0;
        if (tx < kCholB)
#pragma unroll
            for (int t = 0; t < kCholB; ++t) {
                const double y = S.Di[tx][t];
#pragma unroll
                for (int q = 0; q < R; ++q) acc[q] = fma(SA[ty + q * kRows][t], y, acc[q]);
            }
#pragma unroll
        for (int q = 0; q < R; ++q) {
            const int i = U.i0 + ty + q * kRows, j = U.j0 + tx;
            if (tx < kCholB && i < m && j < m) M[(size_t)i * m + j] = acc[q];
        }
    } else {
#pragma unroll
        for (int q = 0; q < R; ++q)
            if (ty + q * kRows < kCholB) SB[tx][ty + q * kRows] = acc[q];
        __syncthreads();
#pragma unroll
        for (int q = 0; q < R; ++q) {
            const int r = ty + q * kRows;
            if (r < kCholB) {
                double x = 0.0;
#pragma unroll
                for (int t = 0; t < kCholB; ++t) x = fma(S.Di[r][t], SB[tx][t], x);
                const int i = U.i0 + r, j = U.j0 + tx;
                if (i < m && j < P.k1) X[(size_t)i * m + j] = x;
            }
        }
    }
}

// One barrier a unit: its operands go to one of two buffers, and a thread that
// stores those of the next unit knows from the barrier in between that no one
// still reads the unit before.
template <int R>
__device__ __noinline__ void dense_units(double* M, double* X, int m, int k1) {
    const DensePlan P = dense_plan(m, k1);
    const unsigned size = team_size();
    unsigned u = team_rank();
    if (u >= P.total) return;                            // CTA-uniform
    DenseUnit U = dense_unit(P, u);
    DenseRegs<R> G;
    dense_load<R>(M, X, m, P, U, G);
    for (int buf = 0;; buf ^= 1) {
        dense_store<R>(U, G, buf);
        double c[R];
#pragma unroll
        for (int q = 0; q < R; ++q) c[q] = G.c[q];
        __syncthreads();
        const DenseUnit V = U;
        u += size;
        const bool more = u < P.total;
        if (more) {
            U = dense_unit(P, u);
            dense_load<R>(M, X, m, P, U, G);
        }
        dense_compute<R>(M, X, m, P, V, c, buf);
        if (!more) break;
    }
}

// The step at column k1 (0, kCholB, 2 kCholB, ...).  Returns false (in every
// thread of the team) only for a pivot that is negative beyond rounding or not
// a number.
template <typename T>
__device__ __noinline__ bool dense_factor_step(double* M, double* X, int m, int k1, const T* jinv) {
    DenseShared& S = dense_smem();
    const int k0 = k1 - kCholB;
    __syncthreads();                                     // the shared blocks are free
    for (int e = threadIdx.x; e < kCholB * kCholB; e += blockDim.x) {
        const int r = e / kCholB, c = e % kCholB;
        double d = r == c ? 1.0 : 0.0, l = 0.0;          // rows past m: the identity
        if (k1 + r < m) {
            if (c <= r) d = __ldcg(M + (size_t)(k1 + r) * m + k1 + c);
            if (k0 >= 0) l = __ldcg(M + (size_t)(k1 + r) * m + k0 + c);
        }
        S.D[r][c] = d;
        S.Lq[r][c] = l;
    }
    double tau = 0.0;
    if (threadIdx.x < 32) {
        const int r = threadIdx.x & (kCholB - 1);
        tau = k1 + r < m ? 1e-13 / (double)__ldcg(jinv + k1 + r) : 0.0;
    }
    __syncthreads();
    if (k0 >= 0)
        for (int e = threadIdx.x; e < kCholB * kCholB; e += blockDim.x) {
            const int r = e / kCholB, c = e % kCholB;
            double d = S.D[r][c];
            if (c <= r) {
#pragma unroll
                for (int t = 0; t < kCholB; ++t) d = fma(-S.Lq[r][t], S.Lq[c][t], d);
            }
            S.D[r][c] = d;
        }
    __syncthreads();
    if (threadIdx.x < 32) dense_diag(tau);
    __syncthreads();
    if (S.bad) return false;                             // CTA-uniform (and team-uniform: same data)
    if (team_rank() == 0)                                // the diagonal block of X, its zeros too
        for (int e = threadIdx.x; e < kCholB * kCholB; e += blockDim.x) {
            const int r = e / kCholB, c = e % kCholB;
            if (k1 + r < m && k1 + c < m) X[(size_t)(k1 + r) * m + k1 + c] = S.Di[r][c];
        }
    if (blockDim.x == 1024) dense_units<1>(M, X, m, k1);
    else if (blockDim.x == 512) dense_units<2>(M, X, m, k1);
    else dense_units<4>(M, X, m, k1);
    return true;
}

// M = A O^2 A' for full rows (the dense workloads): 32 x 32 tiles of the lower
// triangle dealt to the team's CTAs, each the sum over j in increasing order of
// 32 x 16 slabs of its two row blocks staged in shared memory (the first scaled
// by O_j^2), the next slab's entries loaded while one is multiplied.  FP64
// throughout; the FP64 pipe bounds it (a slab is 4 us), so the tiles are kept
// small: n = 200, m = 160 has 15 of them.  Measured: m = 160, n = 200 on 16 CTAs
// 65 us (233 on the grid before), m = 800, n = 1000 1.14 -> 0.90 ms, m = 8000, n =
// 10000 612 -> 630 ms (before: 64 x 64 tiles, 1024-thread CTAs only, without the
// prefetch; with 200 tiles to a CTA the larger ones load half as much).
template <int R, typename T>
__device__ __forceinline__ void dense_syrk(const IterParams<T>& P) {
    DenseShared& S = dense_smem();
    double* M = sync_smem().dM;
    constexpr int kRows = kTile / R;
    const int m = P.m, n = P.n;
    const int nt = (m + kTile - 1) / kTile;
    const unsigned ntile = (unsigned)nt * (unsigned)(nt + 1) / 2u;
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    const int t = tx & (kCholB - 1);
    int buf = 0;
    const SellMat& A = P.A;
    const int g = A.g, h = 32 / g;
    for (unsigned u = team_rank(); u < ntile; u += team_size()) {
        const int bi = tri_row(u);
        const int i0 = bi * kTile, k0 = (int)(u - (unsigned)bi * (unsigned)(bi + 1) / 2u) * kTile;
        // the lower half of the lanes loads the rows of block i0, the upper half
        // those of k0; entry j of a full row: slice row / h, chunk j / g
        const double* row[R];
#pragma unroll
        for (int q = 0; q < R; ++q) {
            const int i = (tx < kCholB ? i0 : k0) + ty + q * kRows;
            row[q] = i < m ? A.v64 + __ldg(A.sptr + i / h) + (i % h) * g : nullptr;
        }
        double v[R], acc[R];
        auto load = [&](int j) {
            const double o = j < n && tx < kCholB ? P.X.O[j] : 1.0;
#pragma unroll
            for (int q = 0; q < R; ++q)
                v[q] = j < n && row[q] ? __ldg(row[q] + 32 * (j / g) + (j % g)) * (o * o) : 0.0;
        };
#pragma unroll
        for (int q = 0; q < R; ++q) acc[q] = 0.0;
        load(t);
        for (int j0 = 0; j0 < n; j0 += kCholB, buf ^= 1) {
#pragma unroll
            for (int q = 0; q < R; ++q) (tx < kCholB ? S.A[buf] : S.B[buf])[ty + q * kRows][t] = v[q];
            __syncthreads();
            if (j0 + kCholB < n) load(j0 + kCholB + t);
#pragma unroll
            for (int c = 0; c < kCholB; ++c) {
                const double y = S.B[buf][tx][c];
#pragma unroll
                for (int q = 0; q < R; ++q) acc[q] = fma(S.A[buf][ty + q * kRows][c], y, acc[q]);
            }
        }
#pragma unroll
        for (int q = 0; q < R; ++q) {
            const int i = i0 + ty + q * kRows, k = k0 + tx;
            if (i < m && k <= i) M[(size_t)i * m + k] = acc[q];
        }
    }
}

// M = A O^2 A' for the cached operator.
template <typename T>
__device__ __noinline__ void phase_dense_assemble(const IterParams<T>& P) {
    if (!P.full_rows) phase_dense_scatter(P);
    else if (blockDim.x == 1024) dense_syrk<1>(P);
    else if (blockDim.x == 512) dense_syrk<2>(P);
    else dense_syrk<4>(P);
}

// dM <- X' (upper triangle, row-major), 32 x 32 tiles through shared memory.
static __device__ __noinline__ void dense_transpose(const double* X, double* Mt, int m) {
    DenseShared& S = dense_smem();
    double(*tile)[kTile + 1] = reinterpret_cast<double(*)[kTile + 1]>(&S);   // 8.4 KB of its 24
    const int nt = (m + kTile - 1) / kTile;
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5, nw = blockDim.x >> 5;
    for (unsigned u = team_rank(); u < (unsigned)nt * (unsigned)(nt + 1) / 2u; u += team_size()) {
        const int bi = tri_row(u);
        const int i0 = bi * kTile, j0 = (int)(u - (unsigned)bi * (unsigned)(bi + 1) / 2u) * kTile;
        __syncthreads();
        for (int r = ty; r < kTile; r += nw)
            tile[r][tx] = (i0 + r < m && j0 + tx <= i0 + r) ? __ldcg(X + (size_t)(i0 + r) * m + j0 + tx) : 0.0;
        __syncthreads();
        for (int r = ty; r < kTile; r += nw)
            if (j0 + r < m && i0 + tx < m && i0 + tx >= j0 + r) Mt[(size_t)(j0 + r) * m + i0 + tx] = tile[tx][r];
    }
}

// Rows of a triangular m x m matrix times a vector: out(i, sum_j T_ij v_j), j in
// [0, i] (lower) or [i, m) (upper).  A warp takes R consecutive rows at a time,
// so that their sums over the lanes are taken together (9 additions a lane for
// eight rows instead of 40) and R loads of the matrix per element of v are in
// flight; consecutive groups go to different CTAs.  The FP64 pipe bounds the
// small teams, latency the whole grid (R = 1 there).  Measured, both products:
// m = 2000 on 152 CTAs 429 -> 19 us, m = 200 31 -> 6.8 us (before: a thread per
// row of X, a warp per column of it).
template <int R, bool kUpper, typename Tv, typename Out>
__device__ __forceinline__ void tri_rows(const double* T, int m, const Tv* v, const Out& out) {
    const int lane = threadIdx.x & 31;
    const int size = team_size(), nw = (int)(blockDim.x >> 5) * size;
    const int w = (int)(threadIdx.x >> 5) * size + team_rank();
    const int ng = (m + R - 1) / R;
    constexpr int U = R == 1 ? 8 : R == 2 ? 4 : 1;
    for (int g = w; g < ng; g += nw) {
        // the long rows first: they are the last ones (lower) or the first
        const int i0 = (kUpper ? g : ng - 1 - g) * R;
        const int lo = kUpper ? (i0 & ~31) : 0, hi = kUpper ? m : min(m, i0 + R);
        double a[R];
#pragma unroll
        for (int r = 0; r < R; ++r) a[r] = 0.0;
        for (int j0 = lo + lane; j0 < hi; j0 += 32 * U) {
            double x[U], t[U][R];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int j = j0 + 32 * u;
                x[u] = j < hi ? (double)__ldcg(v + j) : 0.0;
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    const int i = i0 + r;
                    const bool in = i < m && j < hi && (kUpper ? j >= i : j <= i);
                    t[u][r] = in ? __ldcg(T + (size_t)i * m + j) : 0.0;
                }
            }
#pragma unroll
            for (int u = 0; u < U; ++u)
#pragma unroll
                for (int r = 0; r < R; ++r) a[r] = fma(t[u][r], x[u], a[r]);
        }
        warp_sums<R>(a);
        const int i = i0 + warp_sums_index<R>(lane);
        if ((lane & (32 / R - 1)) == 0 && i < m) out(i, a[0]);
    }
}
template <bool kUpper, typename Tv, typename Out>
__device__ __forceinline__ void tri_product(const double* T, int m, const Tv* v, const Out& out) {
    const int per_warp = m / (int)(team_size() * (blockDim.x >> 5));   // rows a warp has
    if (per_warp >= 8) tri_rows<8, kUpper>(T, m, v, out);
    else if (per_warp >= 2) tri_rows<2, kUpper>(T, m, v, out);
    else tri_rows<1, kUpper>(T, m, v, out);
}

// y = X r0 (r0 = the FP64 residual of the projection system, in V.r); y is
// kept in V.p (unused by the dense path).
template <typename T>
__device__ __noinline__ void phase_dense_y(const IterParams<T>& P) {
    tri_product<false>(sync_smem().dX, P.m, P.V.r, [&](int i, double y) { P.V.p[i] = (T)y; });
}

// w += X' y.
template <typename T>
__device__ __noinline__ void phase_dense_x(const IterParams<T>& P) {
    tri_product<true>(sync_smem().dM, P.m, P.V.p, [&](int c, double x) { P.X.w[c] += x; });
}

// ---------------------------------------------------------------------------
// LP crossover polish (FP64; the entry point is acs_polish).  Support
// B = {j : x_j > z_j}; O holds the indicator of B, so that the projection-
// solve phases work with M = A O^2 A' = A_B A_B' unchanged:
//   x~ = O (p + q), p = O x, q = O A'w, w solving M w = b - A O p (refinement
//        rounds of phase_rhs / CG / phase_update from w = 0);
//   y~ = y + d, d solving M d = A O (O z_y), z_y = c - A'y (the same rounds
//        with b_tilde = 0 and p = -O z_y), a Jacobi-preconditioned CG from
//        zero: the least change of y in the metric J = diag(M);
//   z~ = c - A'y~.
// ---------------------------------------------------------------------------

constexpr int kPolishWindow = 100;   // CG iterations over which the residual must halve

struct PolishOut {
    double* px;      // [n] polished x
    double* pw;      // [m] on entry the iterate's w = mu y; on exit mu y~
                     //     (the solves accumulate in P.X.w, a scratch vector)
    double* pz;      // [n] polished z
    double* res;     // [6] residuals of the polished point (as ctl->res) ...
    double* info;    // [5] |B|, CG iterations (dense: corrections) of the x and y
                     //     solves, 1 = completed, 1 = the factored M was used
};

// O = indicator of B, p = O x, q = 0, g = O (p + q), w = 0, and the count |B|.
static __device__ __noinline__ void phase_polish_init(const IterParams<double>& P, float* O2_32) {
    double nb = 0.0;
    for (int j = global_tid(); j < P.n; j += global_threads()) {
        const double o = P.x[j] > P.z[j] ? 1.0 : 0.0;
        nb += o;
        P.X.O[j] = o;
        P.V.O2[j] = o;
        if (O2_32) O2_32[j] = (float)o;
        const double pj = o * P.x[j];
        P.X.p[j] = pj;
        P.X.q[j] = 0.0;
        P.X.g[j] = pj;
        P.X.chat[j] = fabs(pj);                       // magnitudes behind the residual's rounding
    }
    for (int i = global_tid(); i < P.m; i += global_threads()) P.X.w[i] = 0.0;
    const double v[1] = {nb};
    const int op[1] = {0};
    block_partials<1>(v, op);
}

// b_tilde = b and J^{-1} = 1 / diag(A_B A_B') (1 on rows without an entry in B).
template <typename T>
__device__ __noinline__ void phase_polish_jacobi(const IterParams<T>& P) {
    const double* O = P.X.O;
    auto g1 = [](int) { return 0.0; };
    auto g2 = [O](int j) { return O[j]; };
    auto epi = [&](int i, double, double s2) {
        P.X.btil[i] = P.b[i];
        P.V.jinv[i] = (T)(s2 > 0.0 ? 1.0 / s2 : 1.0);
    };
    sell_rows2(P.A, g1, g2, epi);
}

// After the x solve: px = g (= x~); z_y = c - A'(w_iter / mu) into pz; the
// y solve's start p = -O z_y, q = 0, g = O p, w = 0, b_tilde = 0.
static __device__ __noinline__ void phase_polish_ystart(const IterParams<double>& P, const PolishOut& out) {
    const double* pw = out.pw;
    const double inv_mu = P.inv_mu;
    auto gather = [pw, inv_mu](int i) { return pw[i] * inv_mu; };
    auto epi = [&](int j, double sum) {
        const double o = P.X.O[j];
        out.px[j] = P.X.g[j];
        const double zj = P.c[j] - sum;
        out.pz[j] = zj;
        const double pj = -o * zj;
        P.X.p[j] = pj;
        P.X.q[j] = 0.0;
        P.X.g[j] = o * pj;
        P.X.chat[j] = o * (fabs(P.c[j]) + fabs(sum));
    };
    sell_rows<double>(P.AT, gather, epi);
    for (int i = global_tid(); i < P.m; i += global_threads()) {
        P.X.w[i] = 0.0;
        P.X.btil[i] = 0.0;
    }
}

// z~ = c - A'(pw / mu).
static __device__ __noinline__ void phase_polish_z(const IterParams<double>& P, const PolishOut& out) {
    const double* pw = out.pw;
    const double inv_mu = P.inv_mu;
    auto gather = [pw, inv_mu](int i) { return pw[i] * inv_mu; };
    auto epi = [&](int j, double sum) { out.pz[j] = P.c[j] - sum; };
    sell_rows<double>(P.AT, gather, epi);
}

// Products over the rows of A' restricted to the support: a lane whose row
// j has O_j = 0 issues no loads (its result is 0), so a pass costs about the
// support's share of the matrix stream and gathers.  Plain loop (one chunk
// at a time); FP64 values.
template <typename T, typename Epi, typename Gather>
__device__ __forceinline__ void sell_rows_active(const SellMat& M, const double* __restrict__ O, Gather gather,
                                                 Epi epi) {
    const int lane = threadIdx.x & 31;
    const int g = M.g, h = 32 / g;
    const T* __restrict__ val = sell_vals<T>(M);
    for (int sl = global_warp(); sl < M.nslices; sl += global_warps()) {
        const int row = sl * h + lane / g;
        const bool act = row < M.nrows && O[row] != 0.0;
        const int len = __ldg(M.slen + sl);
        int idx = __ldg(M.sptr + sl) + lane;
        T acc = T(0);
        if (act)
            for (int k = 0; k < len; ++k, idx += 32) acc = fma(ld_stream(val + idx), gather(ld_stream(M.col + idx)), acc);
        for (int o = g / 2; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
        if ((lane & (g - 1)) == 0 && row < M.nrows) epi(row, act ? acc : T(0));
    }
}

// The polish's CG half-step t = O^2 A'u and its q refresh q = O A'w,
// g = O (p + q), on the support's rows only (O is the support's indicator).
template <typename T>
__device__ __noinline__ void phase_polish_cg_At(const IterParams<T>& P) {
    const T* u = P.V.u;
    sell_rows_active<T>(P.AT, P.X.O, [u](int i) { return u[i]; },
                        [&](int j, T sum) { P.V.t[j] = P.V.O2[j] * sum; });
}
static __device__ __noinline__ void phase_polish_q(const IterParams<double>& P) {
    const double* w = P.X.w;
    sell_rows_active<double>(P.AT, P.X.O, [w](int i) { return w[i]; }, [&](int j, double sum) {
        const double o = P.X.O[j];
        const double q = o * sum;
        P.X.q[j] = q;
        P.X.g[j] = o * (P.X.p[j] + q);
    });
}

// The projection residual r0 = b_tilde - A g with its rounding floor: the
// partials are r0' J^{-1} r0 and sum_i J^{-1}_i (b_tilde_i^2 + sum_j A_ij^2
// h_j^2), h (in c_hat) the magnitudes whose rounding the residual carries
// (|x_B| for the x solve, |c_B| + |A_B'y| for the y solve).
template <typename T>
__device__ __noinline__ void phase_polish_rhs(const IterParams<T>& P) {
    double gam = 0.0, fl = 0.0;
    const double* g = P.X.g;
    const double* h = P.X.chat;
    auto g1 = [g](int j) { return g[j]; };
    auto g2 = [h](int j) { return h[j] * h[j]; };
    auto epi = [&](int i, double sum, double s2) {
        rhs_epi(P, i, sum, gam);
        const double bt = P.X.btil[i];
        fl += P.V.jinv[i] * (bt * bt + s2);
    };
    sell_rows2(P.A, g1, g2, epi);
    const double v[2] = {gam, fl};
    const int op[2] = {0, 0};
    block_partials<2>(v, op);
}

// M w = b_tilde - A g by FP64 refinement rounds (FP64 residual, Jacobi-PCG
// correction to 1e-13 of the round's residual, the residual's rounding
// floor 64 eps (sum J^{-1}(b_tilde^2 + (Ag)^2))^{1/2} with eps = 2^-52, the
// target rel times the first residual, or cg_max iterations), until the
// residual is at that floor or target, stops falling tenfold a round, or
// `rounds` rounds have run; then q = O A'w and g = O (p + q) for the final w.
// (Residuals in the J^{-1}-norm.)
// When |B| < m, M is singular and the rounding of b_tilde - A g leaves a
// part outside range(M) that no correction removes: the floor ends the
// solve there instead of letting CG drift on it.  Returns false on a failed
// barrier or a non-finite residual.
template <typename T>
__device__ bool polish_solve(const IterParams<double>& P, const IterParams<T>& PT, int rounds, double rel,
                             bool dense, long long& cg_total) {
    LoopScalars& L = sync_smem().lp;
    double gam_last = INFINITY;
    for (int round = 0; round < rounds; ++round) {
        if (round > 0) {
            phase_polish_q(P);
            if (!grid_sync(&P.ctl->err)) return false;
        }
        phase_polish_rhs(PT);
        // an FP32 correction goes down to ~1e-5 of its round's residual; the
        // next round's FP64 residual refines it
        if (!grid_sync_post(&P.ctl->err, [&](const double* t2) {
                const double gam = t2[0], gn = sqrt(fmax(gam, 0.0));
                double floor_r = 64.0 * 0x1p-52 * sqrt(fmax(t2[1], 0.0));
                const double target = round == 0 ? rel * gn : L.target;
                const int bad = !isfinite(gam) || !isfinite(floor_r);
                floor_r = fmax(floor_r, target);
                const double thr = fmax((sizeof(T) == 4 ? 1e-5 : 1e-13) * sqrt(gam), floor_r);
                const int broke = !(gn > floor_r) || (round > 0 && gam > 0.01 * gam_last);
                __syncwarp();
                if ((threadIdx.x & 31) == 0) {
                    L.gam = gam;
                    L.target = target;
                    L.thr = thr;
                    L.gam_prev = L.alpha_prev = 1.0;
                    L.best = L.best_ref = gam;
                    L.bad = bad;
                    L.broke = broke;
                    L.go = gn > thr;
                }
            }))
            return false;
        if (L.bad) return false;
        if (L.broke) break;
        gam_last = L.gam;
        if (sizeof(T) == 8 && dense) {                 // one exact correction: dw = X'(X r0)
            phase_dense_y(P);
            if (!grid_sync(&P.ctl->err)) return false;
            phase_dense_x(P);
            if (!grid_sync(&P.ctl->err)) return false;
            ++cg_total;
            continue;
        }
        // should the floor underestimate that part, the round ends when the
        // smallest residual so far has not halved in kPolishWindow iterations
        int k = 0;
        while (L.go && k < P.cg_max) {
            phase_polish_cg_At(PT);
            if (!grid_sync(&P.ctl->err)) return false;
            phase_cg_A(PT);
            if (!grid_sync_post(&P.ctl->err, [&](const double* dl) { cg_step_scalars(dl[0], k); })) return false;
            if (L.broke) break;                         // attainable accuracy reached
            phase_cg_vec<T, false>(PT);
            if (!grid_sync_post(&P.ctl->err, [&](const double* gn) {
                    cg_next_scalars(gn[0]);
                    const double best = fmin(L.best, gn[0]);
                    const bool window = (k + 1) % kPolishWindow == 0;
                    const int stuck = window && best > 0.5 * L.best_ref;
                    __syncwarp();
                    if ((threadIdx.x & 31) == 0) {
                        L.best = best;
                        if (window) L.best_ref = best;
                        L.broke = stuck;
                    }
                }))
                return false;
            ++k;
            if (L.bad) return false;
            if (L.broke) break;
        }
        cg_total += k;
    }
    phase_polish_q(P);
    return grid_sync(&P.ctl->err);
}

// The whole polish; Q is P with x = px, z = pz, w = pw (its KKT residuals).
// fp32: the corrections by FP32 CG on P32 (the same state, FP32 CG vectors
// and values), refined by the FP64 residual of every round.
static __device__ __noinline__ void polish_loop(const IterParams<double>& P, const IterParams<float>& P32,
                                         const IterParams<double>& Q, const PolishOut& out, int rounds,
                                         double rel, bool fp32) {
    const bool owner = blockIdx.x == 0 && threadIdx.x == 0;
    long long cg_x = 0, cg_y = 0;
    double nb[1] = {0.0};
    bool ok = false;
    // with scratch for it, M = A_B A_B' is factored once (the cached
    // operator's phases with O the indicator of B) and both solves apply
    // L^{-1}; a failed factorisation falls back to CG
    bool dense = sync_smem().dM != nullptr;
    double used_dense = 0.0;
    do {
        if (dense) fp32 = false;
        phase_polish_init(P, fp32 ? P32.V.O2 : nullptr);
        if (!grid_sync(&P.ctl->err)) break;
        {
            grid_combine<1>(nb);
        }
        if (fp32) phase_polish_jacobi(P32);
        else phase_polish_jacobi(P);
        if (!grid_sync(&P.ctl->err)) break;
        if (dense) {
            phase_dense_assemble(P);
            if (!grid_sync(&P.ctl->err)) break;
            bool fine = true;
            for (int k1 = 0; k1 < P.m && dense; k1 += kCholB) {
                if (!dense_factor_step(sync_smem().dM, sync_smem().dX, P.m, k1, P.V.jinv)) dense = false;
                if (!(fine = grid_sync(&P.ctl->err))) break;
            }
            if (!fine) break;
            if (dense) {
                dense_transpose(sync_smem().dX, sync_smem().dM, P.m);
                if (!grid_sync(&P.ctl->err)) break;
                used_dense = 1.0;
            }
        }
        if (!(fp32 ? polish_solve(P, P32, rounds, rel, false, cg_x)
                   : polish_solve(P, P, rounds, rel, dense, cg_x))) break;     // x~ = g
        phase_polish_ystart(P, out);
        if (!grid_sync(&P.ctl->err)) break;
        if (!(fp32 ? polish_solve(P, P32, rounds, rel, false, cg_y)
                   : polish_solve(P, P, rounds, rel, dense, cg_y))) break;     // d = w
        for (int i = global_tid(); i < P.m; i += global_threads()) out.pw[i] += P.mu * P.X.w[i];
        if (!grid_sync(&P.ctl->err)) break;
        phase_polish_z(P, out);
        if (!grid_sync(&P.ctl->err)) break;
        phase_kkt(Q);
        if (!grid_sync(&P.ctl->err)) break;
        double r8[8];
        grid_combine<8>(r8);
        if (owner) {
            out.res[0] = sqrt(r8[0]) / (1.0 + P.bnorm);
            out.res[1] = sqrt(r8[1]) / (1.0 + P.cnorm);
            out.res[2] = fabs(r8[2] - r8[3]) / (1.0 + fabs(r8[2]) + fabs(r8[3]));
            out.res[3] = fmax(sqrt(r8[4]), sqrt(r8[5])) / (1.0 + fmax(sqrt(r8[6]), sqrt(r8[7])));
            out.res[4] = r8[2];
            out.res[5] = r8[3];
        }
        ok = true;
    } while (false);
    if (owner) {
        out.info[0] = nb[0];
        out.info[1] = (double)cg_x;
        out.info[2] = (double)cg_y;
        out.info[3] = ok ? 1.0 : 0.0;
        out.info[4] = used_dense;
        P.ctl->bar_gen = sync_smem().gen;
    }
}

// ---------------------------------------------------------------------------
// the solve loop
// ---------------------------------------------------------------------------

// Algorithm 2 from the state in P (fresh, resumed, or handed over by an FP32
// loop when status0 = ST_SWITCH) until the KKT test passes, the iteration
// limit is reached, or the FP32 correction solve hands over.  Run by every
// thread of every CTA of the problem's team (team_set first); the team's
// barrier generation must be current in shared memory (sync_init).  Returns
// the loop's status, the same in every thread of the team; the team's rank-0
// CTA writes it, the residuals and the counters to P.ctl.
template <typename T>
__device__ __noinline__ int solve_loop(const IterParams<T>& P, int status0) {
    Control* ctl = P.ctl;
    // per-phase time record, kept by thread 0 of the team's CTA 0 in shared memory
    __shared__ unsigned long long s_ph_ns[PH_COUNT], s_ph_n[PH_COUNT], s_last;
    const bool clock_owner = team_rank() == 0 && threadIdx.x == 0;
    if (clock_owner) {
        for (int i = 0; i < PH_COUNT; ++i) { s_ph_ns[i] = 0; s_ph_n[i] = 0; }
        s_last = gtimer();
    }

    // state left by the reset or by an earlier loop (written by the team's
    // rank 0 before a barrier): read past L1
    int l = __ldcg(&ctl->l);
    bool refresh = P.refresh != 0 || status0 == ST_SWITCH;
    int status = ST_RUNNING;
    // FP32 loop of the single-problem launch: column-blocked CG passes, and
    // FP32 outer passes while P.outer32 is on (until ctl->outer32_end is set)
    const bool cbcg = sizeof(T) == 4 && P.Acb.nblocks > 0 && P.ATcb.nblocks > 0;
    int outer32_end = __ldcg(&ctl->outer32_end);
    bool outer32 = cbcg && P.outer32 != 0 && outer32_end == 0;
    LoopScalars& L = sync_smem().lp;
    if (threadIdx.x == 0) {
        for (int i = 0; i < 6; ++i) L.res[i] = __ldcg(&ctl->res[i]);
        L.ds = __ldcg(&ctl->ds);
        L.snorm = __ldcg(&ctl->snorm);
        L.eta = __ldcg(&ctl->eta);
        L.best_mx = INFINITY;
        L.flat_checks = 0;
        L.win_cg = __ldcg(&ctl->win_cg);
        for (int i = 0; i < CT_COUNT; ++i) L.count[i] = 0;
    }
    __syncthreads();
    // the pass counters live in shared memory and are kept by thread 0: in
    // registers they would be spilled around every phase by every thread
    auto count = [&](int which) {
        if (threadIdx.x == 0) ++L.count[which];
    };
    bool ok = true;
    // cached projection operator (FP64 loops only); a factorisation that fails
    // (M singular: rank-deficient A) hands this solve to the CG projection
    // P.dense == 2: start with CG and switch to the cached operator once the
    // CG iterations since the last rescaling exceed P.switch_budget, the cost
    // of one factorisation counted in CG iterations (rent until the price of
    // buying is spent): a member that finishes soon after a rescaling never
    // pays for a factorisation, one whose M is too ill-conditioned for
    // Jacobi-CG pays at most twice the better of the two.  An FP32 loop hands
    // over to the FP64 loop for that, marking the switch in ctl->dense_on; a
    // hand-over for FP32 precision alone continues with FP64 CG under the
    // same rule.
    const bool have_scratch = sync_smem().dM != nullptr;
    bool dense = sizeof(T) == 8 && have_scratch &&
                 (P.dense == 1 || (P.dense == 2 && __ldcg(&ctl->dense_on) != 0));
    bool want_dense = false;                            // FP32 loop: hand over for the switch
    const bool may_switch = P.dense == 2 && (sizeof(T) == 4 ? P.switch_ok != 0 : have_scratch);
    bool dense_failed = __ldcg(&ctl->dense_failed) != 0;
    // a factor held in the problem's own scratch stays valid across a pause
    // (O changes only at rescalings, which refactor)
    bool factor_ok = __ldcg(&ctl->factor_ok) != 0;
    bool factor_kept = P.own_scratch != 0 && factor_ok;
    bool over = false;                                  // deadline of a time-sliced solve passed
    bool extrap_ok = __ldcg(&ctl->extrap_ok) != 0;
    int win_it = __ldcg(&ctl->win_it);
    bool abs_fused = false;                             // p, g of the next iteration already formed
    // FP32 outer products on the L2-gather layout (FP32 loop, a segment that
    // ends at a polish level)
    const bool outer32_l2 = sizeof(T) == 4 && P.outer32_l2 != 0 && !cbcg && P.A.v32 && P.AT.v32;

// grid barrier that ends phase `ph`, with the scalars of the next phases in
// its post function; leaves the enclosing loop on error
#define ACS_SYNC(ph) ACS_SYNC_POST(ph, [](const double*) {})
#define ACS_SYNC_POST(ph, ...)                                            \
    {                                                                     \
        if (!(ok = grid_sync_post(&ctl->err, __VA_ARGS__))) break;        \
        if (clock_owner) {                                                \
            const unsigned long long t_ = gtimer();                       \
            s_ph_ns[ph] += t_ - s_last;                                   \
            s_ph_n[ph] += 1;                                              \
            s_last = t_;                                                  \
        }                                                                 \
    }

    while (ok) {
        if (l >= P.max_iter) { status = ACS_MAX_ITER; break; }
        const int lnext = l + 1;
        const bool cond = (lnext == 1) || in_schedule(P, lnext);
        if (may_switch && !dense && !dense_failed && !cond && L.win_cg > P.switch_budget) {
            if (sizeof(T) == 4) {
                want_dense = true;
                status = ST_SWITCH;
                break;
            }
            dense = true;
            refresh = true;                                     // factor at this iteration
        }
        if (cond) {                                             // steps 5-14
            win_it = 0;                                         // a new scaling: a new rental
            if (threadIdx.x == 0) L.win_cg = 0;
            phase_cond_o(P);
            ACS_SYNC_POST(PH_COND_O, [&](const double* mm) {
                CondRange R;
                R.any = mm[2] > 0.0;                           // some o finite and positive
                R.lmax = mm[0];
                R.lmin = -mm[1];
                const double spread = R.lmax - R.lmin;         // log max o - log min o
                if (!R.any) R.alpha = 0.0;
                else if (!(spread > 0.0)) R.alpha = 1.0;
                else R.alpha = fmin(1.0, P.t_cond / spread);
                if (threadIdx.x == 0) L.range = R;
            });
            phase_cond_apply(P, L.range, true, true);
            ACS_SYNC(PH_COND_APPLY);
            count(CT_COND);
        } else if (refresh) {
            phase_cond_apply(P, CondRange{0.0, 0.0, 0.0, false}, false, false);
            ACS_SYNC(PH_COND_APPLY);
        }
        if (cond || refresh) {
            phase_btilde(P);
            count(CT_A64);
            ACS_SYNC_POST(PH_BTILDE, [&](const double* bb) {
                if (threadIdx.x == 0) L.bad = bb[0] > 0.0;
            });
            if (L.bad) { atomicCAS(&ctl->err, 0, ACS_ERR_FACTOR); ok = false; break; }
            if (cond) factor_ok = false;                    // O changed: the factor is stale
            if (dense && factor_kept && !cond) {
                factor_kept = false;                        // resumed: the cached factor is current
            } else if (dense) {
                factor_kept = false;
                factor_ok = false;
                phase_dense_assemble(P);
                ACS_SYNC(PH_DENSE_ASSEMBLE);
                for (int k1 = 0; k1 < P.m && dense; k1 += kCholB) {
                    if (!dense_factor_step(sync_smem().dM, sync_smem().dX, P.m, k1, P.V.jinv)) {
                        dense = false;
                        dense_failed = true;
                    }
                    ACS_SYNC(PH_DENSE_FACTOR);
                }
                if (!ok) break;
                if (dense) {
                    dense_transpose(sync_smem().dX, sync_smem().dM, P.m);
                    ACS_SYNC(PH_DENSE_INVERSE);
                    count(CT_FACTOR);
                    factor_ok = true;
                }
            }
            phase_update(P, false, false);                      // q = A_hat' w for the warm start
            count(CT_AT64);
            ACS_SYNC(PH_QREFRESH);
            refresh = false;
        }

        // extrapolated start, valid once the previous iteration ran in the
        // same scaling (not on an iteration that rescales); skipped when the
        // previous update already formed p and g (and nothing changed O or g since)
        if (!(abs_fused && !cond && !refresh)) {
            phase_abs(P, (extrap_ok && !cond) ? P.extrap : 0.0);   // step 17
            ACS_SYNC(PH_ABS);
        }
        abs_fused = false;
        extrap_ok = true;
        // Projection solve: `refine` rounds of (FP64 residual, correction CG in
        // precision T); a round after the first refreshes q = A_hat' w first.
        bool trouble = false;                                   // FP32 solve cannot keep up
        if (dense) {
            // one exact correction: dw = X'(X r0)
            phase_rhs_plain(P);
            count(CT_A64);
            ACS_SYNC(PH_RHS);
            phase_dense_y(P);
            ACS_SYNC(PH_DENSE_SOLVE);
            phase_dense_x(P);
            ACS_SYNC(PH_DENSE_SOLVE);
            count(CT_DENSE);
        }
        for (int round = 0; round < (dense ? 0 : P.refine); ++round) {
            if (round > 0) {
                phase_update(P, false, false);
                count(CT_AT64);
                ACS_SYNC(PH_QREFRESH);
            }
            // the step-relative rule needs a previous step in the same scaling;
            // on the first iteration and whenever O changes only the floors apply
            auto start_cg = [&](const double* t1) {
                const double gam = t1[0], g = sqrt(fmax(gam, 0.0));
                const double rel = (isfinite(L.ds) && !cond && round == 0) ? L.eta * L.ds : 0.0;
                const double thr = fmax(fmax(rel, P.cg_tol * L.snorm), P.cg_relfloor * g);
                const int go = g > thr, far = g > 100.0 * thr;
                if (threadIdx.x == 0) {
                    L.gam = gam;
                    L.thr = thr;
                    L.gam_prev = L.alpha_prev = 1.0;
                    L.bad = !isfinite(gam);
                    L.go = go;
                    L.far = far;
                }
            };
            if (outer32) {                                      // r0 from an FP32 product
                phase_rhs_cb(P);
                count(CT_A32);
                ACS_SYNC(PH_RHS);
                phase_rhs_comb(P);
                ACS_SYNC_POST(PH_RHS_COMB, start_cg);
            } else if (outer32_l2) {
                phase_rhs_f32(P);                               // r0 from an FP32 product
                count(CT_A32);
                ACS_SYNC_POST(PH_RHS, start_cg);
            } else {
                phase_rhs(P);                                   // r0 in FP64
                count(CT_A64);
                ACS_SYNC_POST(PH_RHS, start_cg);
            }
            if (L.bad) { status = ACS_ERR_NUMERICAL; break; }
            int k = 0;
            bool broke = false;
            while (L.go && k < P.cg_max) {
                auto step_scalars = [&](const double* dl) { cg_step_scalars(dl[0], k); };
                if (cbcg) {
                    // column-blocked passes: u'Mu = ||A_hat'u||^2 is known after
                    // the first half, the second half's sums are combined in the
                    // vector step
                    phase_cg_At_cb(P);                          // partial sums of A'u
                    count(CT_AT);
                    ACS_SYNC(PH_CG_AT);
                    phase_cg_tcomb(P);                          // t = O^2 A'u, u'Mu
                    ACS_SYNC_POST(PH_CG_TCOMB, step_scalars);
                } else {
                    phase_cg_At(P);                             // t = O^2 A' u
                    count(CT_AT);
                    ACS_SYNC(PH_CG_AT);
                    phase_cg_A(P);                              // au = A t = M u
                    count(CT_A);
                    ACS_SYNC_POST(PH_CG_A, step_scalars);
                }
                if (L.broke) {
                    // keep w -- the next FP64 residual carries on from it
                    broke = true;
                    break;
                }
                if (cbcg) {
                    phase_cg_A_cb(P);                           // partial sums of A t = M u
                    count(CT_A);
                    ACS_SYNC(PH_CG_A);
                    phase_cg_vec<T, true>(P);
                } else {
                    phase_cg_vec<T, false>(P);
                }
                ACS_SYNC_POST(PH_CG_VEC, [&](const double* gn) { cg_next_scalars(gn[0]); });
                ++k;
                if (L.bad) { status = ACS_ERR_NUMERICAL; break; }
            }
            if (!ok || status == ACS_ERR_NUMERICAL) break;
            if (threadIdx.x == 0) {
                L.count[CT_CG] += k;
                L.win_cg += k;
            }
            // an FP32 solve that stalls far above its target cannot refine this M
            if ((broke || k >= P.cg_max) && L.far) trouble = true;
        }
        if (!ok || status == ACS_ERR_NUMERICAL) break;

        const bool check = (lnext % P.check_every == 0) || (lnext == P.max_iter);
        const bool want_xz = check || in_schedule(P, lnext + 1);
        // step 17 of the next iteration in this pass's epilogue (orthant-only,
        // no extrapolation, no rescaling at the next iteration)
        const bool fuse_abs = P.n_soc == 0 && !P.admm && P.extrap == 0.0 && !in_schedule(P, lnext + 1);
        // With exact projections the step norm ||s_l - s_{l-1}|| never grows
        // between rescalings (the iteration map is firmly nonexpansive,
        // Lemma 3); growth beyond what the allowed error explains means the
        // CG error estimate (J-norm of the residual) is too optimistic for
        // this M, so the rule is tightened for the rest of the solve.
        // In the FP32 solve a factor below 1e-4 * cg_eta means the FP32
        // correction cannot reach the accuracy this M needs: the solve
        // continues with an FP64 correction solve instead.
        auto end_step = [&](double d0, double d1) {
            const double ds_new = sqrt(d0), sn = sqrt(d1);
            const int bad = !isfinite(ds_new) || !isfinite(sn);
            const double ds = L.ds;
            double eta = L.eta;
            int tr = 0;
            if (!cond && isfinite(ds) && ds_new > (1.0 + 4.0 * eta) * ds && eta > 1e-8) {
                if (sizeof(T) == 4 && eta <= 1e-4 * P.cg_eta * 1.0000001) tr = 1;
                else eta *= 0.1;
            }
            __syncwarp();
            if (threadIdx.x == 0) {
                L.snorm = sn;
                L.bad = bad;
                L.trouble = bad ? 0 : tr;
                if (!bad) {
                    L.eta = eta;
                    L.ds = ds_new;
                }
            }
        };
        const bool two_parts = P.admm && P.n_soc > 0;            // the cones' share of the update follows
        auto after_update = [&](const double* d2) {
            if (threadIdx.x == 0) {
                L.over = d2[2] > 0.0;
                L.d0 = d2[0];
                L.d1 = d2[1];
            }
            if (!two_parts) end_step(d2[0], d2[1]);
        };
        if (outer32) {                                          // steps 18-21, FP32 product
            phase_update_cb(P);
            count(CT_AT32);
            ACS_SYNC(PH_UPDATE);
            phase_update_comb(P, want_xz, fuse_abs);
            ACS_SYNC_POST(PH_UPD_COMB, after_update);
        } else if (outer32_l2) {
            phase_update_f32(P, want_xz, fuse_abs);             // steps 18-21, FP32 product
            count(CT_AT32);
            ACS_SYNC_POST(PH_UPDATE, after_update);
        } else {
            phase_update(P, true, want_xz, fuse_abs);          // steps 18-21
            count(CT_AT64);
            ACS_SYNC_POST(PH_UPDATE, after_update);
        }
        abs_fused = fuse_abs;
        over = L.over != 0;
        if (two_parts) {
            phase_admm_soc(P, want_xz);
            ACS_SYNC_POST(PH_UPDATE, [&](const double* e2) { end_step(L.d0 + e2[0], L.d1 + e2[1]); });
        }
        if (L.bad) { status = ACS_ERR_NUMERICAL; l = lnext; break; }
        if (L.trouble) trouble = true;
        l = lnext;
        ++win_it;
        if (sizeof(T) == 4 && trouble && P.switch_ok) { status = ST_SWITCH; break; }

        if (check) {
            phase_kkt(P);
            count(CT_A64);
            count(CT_AT64);
            count(CT_CHECK);
            // FP32 outer passes end once the residuals reach outer32_tol, or
            // once they stop falling (the FP32 products' rounding floor): the
            // rest of the solve runs the FP64 passes from the same iterate
            ACS_SYNC_POST(PH_KKT, [&](const double* r8) {
                const double rp = sqrt(r8[0]) / (1.0 + P.bnorm);
                const double rd = sqrt(r8[1]) / (1.0 + P.cnorm);
                const double rg = fabs(r8[2] - r8[3]) / (1.0 + fabs(r8[2]) + fabs(r8[3]));
                const double rc = fmax(sqrt(r8[4]), sqrt(r8[5])) / (1.0 + fmax(sqrt(r8[6]), sqrt(r8[7])));
                const double mx = fmax(fmax(rp, rd), fmax(rg, rc));
                if (threadIdx.x == 0) {
                    L.res[0] = rp;
                    L.res[1] = rd;
                    L.res[2] = rg;
                    L.res[3] = rc;
                    L.res[4] = r8[2];
                    L.res[5] = r8[3];
                    L.bad = !isfinite(mx);
                    L.solved = mx <= P.tol;
                    if (mx < 0.9 * L.best_mx) {
                        L.best_mx = mx;
                        L.flat_checks = 0;
                    } else {
                        ++L.flat_checks;
                    }
                    L.end32 = mx <= P.outer32_tol || L.flat_checks >= kOuter32FlatChecks;
                }
            });
            if (L.bad) { status = ACS_ERR_NUMERICAL; break; }
            if (L.solved) { status = ACS_SOLVED; break; }
            if (outer32 && L.end32) {
                outer32 = false;
                outer32_end = l;
            }
        }
        if (over && l < P.max_iter) { status = ST_PAUSED; break; }
    }
#undef ACS_SYNC
#undef ACS_SYNC_POST

    if (clock_owner) {
        const int err = ld_volatile_int(&ctl->err);
        ctl->status = err != 0 ? err : status;
        if (status == ST_SWITCH && err == 0) ctl->switched_at = l;
        ctl->l = l;
        ctl->cg_iters += L.count[CT_CG];
        for (int i = 0; i < 6; ++i) ctl->res[i] = L.res[i];
        ctl->ds = L.ds;
        ctl->snorm = L.snorm;
        ctl->eta = L.eta;
        ctl->n_cg_A += L.count[CT_A];
        ctl->n_cg_AT += L.count[CT_AT];
        ctl->n_64_A += L.count[CT_A64];
        ctl->n_64_AT += L.count[CT_AT64];
        ctl->n_cond += L.count[CT_COND];
        ctl->n_checks += L.count[CT_CHECK];
        ctl->n_dense_solve += L.count[CT_DENSE];
        ctl->n_dense_factor += L.count[CT_FACTOR];
        ctl->n_32_A += L.count[CT_A32];
        ctl->n_32_AT += L.count[CT_AT32];
        ctl->outer32_end = outer32_end;
        ctl->stage = (sizeof(T) == 8 || status == ST_SWITCH) ? 1 : 0;
        ctl->dense_on = (dense || want_dense) ? 1 : 0;
        ctl->factor_ok = factor_ok ? 1 : 0;
        ctl->dense_failed = dense_failed ? 1 : 0;
        ctl->win_cg = L.win_cg;
        ctl->win_it = win_it;
        ctl->extrap_ok = extrap_ok ? 1 : 0;
        ctl->bar_gen = sync_smem().gen;
        for (int i = 0; i < PH_COUNT; ++i) {
            ctl->phase_ns[i] += s_ph_ns[i];
            ctl->phase_n[i] += s_ph_n[i];
        }
    }
    return status;
}

}  // namespace acs
