// Multi-slot solver engine: many CTR-IBIM systems advanced together on one GPU.
//
// Each slot holds one system (a ctr_ibim handle) and its solver state on the
// device.  The solver is right-preconditioned GMRES(m) (CGS2, FP64 Givens) on
// the operator of Eq. (2.30); every cycle ends by recomputing the true
// residual r = g - A x with the residual pair arithmetic and starting the next
// cycle from it.  With FP32 inner pairs and an FP64-accurate residual this is
// GMRES-based iterative refinement; with the same precision inside and out it
// is plain restarted GMRES.
//
// One engine step runs up to two halves, each captured once as a CUDA graph and replayed:
//   inner half   (slots in state INNER)  one Arnoldi iteration, seven kernels: plan; V_j scaled to unit length
//                and z = Lambda^-1 V_j packed; pairs; finish w = A z; CGS2 as dots, subtract + dots,
//                subtract + norm (the last block of each reduction adds the partials, the last of all also
//                does the Givens update and the slot's state);
//   update half  (slots in state UPDATE; launched only when there is one) triangular solve;
//                x += Lambda^-1 V y, pack; pairs; finish r = g - A x; norm and decision (done / next cycle).
// A small system's step is bound by its launches: the vector part of a 19k-node system took about 160 us in
// some 30 kernels (both halves every step); the solve of such a system went from 16.5 to 14.5 ms.
// The dense pair sums of all slots run in persistent kernels (one per pair
// arithmetic and half) whose blocks take work entries (slot, item of that
// slot's pair schedule: target block, source range, one-sided or symmetric)
// from a list sorted by cost through an atomic counter; entries of slots in
// another state return at once.  A slot's items, partial-sum layout,
// reduction chunks and scalar updates are exactly those of the slot alone, so
// a system's result does not depend on what else the engine holds.
#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstring>
#include <map>
#include <mutex>

#include "engine.cuh"
#include "pairkern.cuh"
#include "tree.cuh"

namespace ctr {

using namespace pk;

namespace {

constexpr int kVecThreads = 256;
constexpr double kUpdateGate = 1e-4;   // |r| / |g| below which refinement residuals are updated
// Work entries carry (slot, item | part << kPartShift): items of a schedule <= kMaxItems, parts <= kMaxParts.
constexpr int kItemMask = (int)kMaxItems;
constexpr int kMaxParts = 127;
constexpr int kMinItemsPerPart = 64;

__device__ __forceinline__ bool inner_active(const SlotDev& s) { return s.stat.state == kSlotInner; }
__device__ __forceinline__ bool update_active(const SlotDev& s) { return s.stat.state == kSlotUpdate; }
// Pair arithmetic of a slot's residual in this cycle: the residual arithmetic for g - A x, the inner
// one for an update r - A d of a small correction d.
__device__ __forceinline__ int res_arith(const SlotDev& s) { return s.upd ? s.inner_prec : s.res_prec; }

__device__ __forceinline__ int arith_index(int prec) { return prec == CTR_FP32_REFINE ? 0 : (prec == CTR_DF64 ? 1 : 2); }
// Whether the parts of the slot's operator application run in this half-step are its last ones.
__device__ __forceinline__ bool whole(const SlotDev& s, int half) {
    return s.part + s.span >= s.nparts[arith_index(half == 0 ? s.inner_prec : res_arith(s))];
}

// ---------------------------------------------------------------- packing
__device__ __forceinline__ void pack_weights(const SlotDev& s, int prec, int64_t t, double a, double b) {
    if (prec == CTR_FP32_REFINE) {
        s.src32[4 * t + 1].z = s.src32[4 * t + 1].w = (float)a;   // duplicated pairs: a and -b
        s.src32[4 * t + 3].z = s.src32[4 * t + 3].w = -(float)b;
    } else if (prec == CTR_FP64) {
        s.src64[2 * t].w = a;
        s.src64[2 * t + 1].w = b;
    } else {
        const float ah = (float)a, bh = (float)b;
        s.srcdf[4 * t].w = ah;
        s.srcdf[4 * t + 1].w = (float)(a - (double)ah);
        s.srcdf[4 * t + 2].w = bh;
        s.srcdf[4 * t + 3].w = (float)(b - (double)bh);
    }
}

// inner: V_j to unit length (V_0 = r / beta; V_j is the last iteration's w, of length scal[2]), z = Lambda^-1 V_j
// and the weights of z
__global__ void k_prep_inner(SlotDev* S) {
    const SlotDev& s = S[blockIdx.y];
    if (!inner_active(s) || s.part != 0) return;   // later parts reuse the packed weights
    const int64_t M = s.M;
    double* v = s.V + (size_t)s.j * s.n;
    const double* w = s.j == 0 ? s.r : v;
    const double f = 1.0 / (s.j == 0 ? s.beta : s.scal[2]);
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < M; t += (int64_t)gridDim.x * blockDim.x) {
        const double v1 = w[t] * f, v2 = w[M + t] * f;
        v[t] = v1;
        v[M + t] = v2;
        const double z1 = v1 * s.il1, z2 = v2 * s.il2;
        s.z[t] = z1;
        s.z[M + t] = z2;
        pack_weights(s, s.inner_prec, s.tinv ? (int64_t)s.tinv[t] : t, s.scale * s.W[t] * z1, s.scale * s.W[t] * z2);
    }
}

// update: d = Lambda^-1 V y (k columns), x += d, and the weights of x (residual g - A x) or, for a
// residual update, d kept in z and its weights in the inner arithmetic (residual r - A d)
__global__ void k_update_x(SlotDev* S) {
    const SlotDev& s = S[blockIdx.y];
    if (!update_active(s) || s.part != 0) return;
    const int64_t M = s.M, n = s.n;
    const int k = s.kdone;
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < M; t += (int64_t)gridDim.x * blockDim.x) {
        double v1 = 0.0, v2 = 0.0;
        for (int i = 0; i < k; ++i) {
            v1 += s.V[(size_t)i * n + t] * s.y[i];
            v2 += s.V[(size_t)i * n + M + t] * s.y[i];
        }
        const double d1 = v1 * s.il1, d2 = v2 * s.il2;
        const double x1 = s.x[t] + d1, x2 = s.x[M + t] + d2;
        s.x[t] = x1;
        s.x[M + t] = x2;
        const int64_t pos = s.tinv ? (int64_t)s.tinv[t] : t;
        if (s.upd) {
            s.z[t] = d1;
            s.z[M + t] = d2;
            pack_weights(s, s.inner_prec, pos, s.scale * s.W[t] * d1, s.scale * s.W[t] * d2);
        } else {
            pack_weights(s, s.res_prec, pos, s.scale * s.W[t] * x1, s.scale * s.W[t] * x2);
        }
    }
}

// ---------------------------------------------------------------- persistent pair kernels
// Work entries (slot, item of that slot's schedule), sorted by decreasing cost.  kShared: every slot
// of this arithmetic has the same pair constants, passed as the launch parameter `pkc` (read from the
// constant bank, no registers); otherwise each item takes its slot's constants.
template <typename Policy, int R, int V, int U, bool kShared>
__global__ void __launch_bounds__(kThreads, Policy::kMinBlocks) k_pairs(SlotDev* S, const int2* __restrict__ items,
                                                    const int* __restrict__ n_items, int* __restrict__ counter,
                                                    int half, int prec, int pol, const float2* __restrict__ exp_tab,
                                                    int* __restrict__ err, const PairConsts pkc,
                                                    const int* __restrict__ need) {
    using Src = typename Policy::Src;
    if (need[pol] == 0) return;   // no slot in this half uses this arithmetic: skip the whole list
    extern __shared__ __align__(128) unsigned char smem_raw[];
    PairSmem<Policy> sm(smem_raw);
    __shared__ __align__(8) uint64_t bar[2];
    __shared__ int cur;
    __shared__ PairConsts kc;
    pair_block_init<Policy>(exp_tab, sm.tab, bar);   // one table per device, shared by every slot
    uint32_t gt = 0;
    const int total = *n_items;
    for (int it = blockIdx.x; it < total;) {   // the first entries need no counter
        const int2 w = items[it];   // slot, item | part << kPartShift
        const SlotDev& s = S[w.x];
        const bool want = half == 0 ? (inner_active(s) && s.inner_prec == prec)
                                    : (update_active(s) && res_arith(s) == prec);
        const int pe = w.y >> kPartShift;
        if (want && pe >= s.part && pe < s.part + s.span) {
            const int item = w.y & kItemMask;
            const Src* src = reinterpret_cast<const Src*>(prec == CTR_FP32_REFINE ? (const void*)s.src32
                                                          : prec == CTR_DF64 ? (const void*)s.srcdf
                                                                             : (const void*)s.src64);
            if constexpr (kShared) {
                if (!run_item<Policy, R, V, U>(s.items[pol][item], src, s.M, s.excl, s.acc, pkc, err, sm.ring,
                                               sm.jred, sm.tab, bar, gt))
                    return;
            } else {
                if (threadIdx.x == 0) kc = s.kc;
                __syncthreads();
                const PairConsts k = kc;   // block-uniform register copy: no shared loads in the pair loops
                if (!run_item<Policy, R, V, U>(s.items[pol][item], src, s.M, s.excl, s.acc, k, err, sm.ring,
                                               sm.jred, sm.tab, bar, gt))
                    return;
            }
        }
        if (threadIdx.x == 0) cur = gridDim.x + atomicAdd(counter, 1);
        __syncthreads();
        it = cur;
        __syncthreads();
    }
}

// finish: diag + the node's accumulated dense sum (read and cleared) + correction of the applied vector;
// inner: w = V_{j+1} = A z;   update: r = g - A x, or r = r - A d (residual update, d in z)
__global__ void __launch_bounds__(kFinishThreads) k_finish(SlotDev* S, int half) {
    const SlotDev& s = S[blockIdx.y];
    if ((half == 0 ? !inner_active(s) : !update_active(s)) || !whole(s, half)) return;
    const int64_t M = s.M;
    const bool upd = (half == 1) && s.upd;
    const double* x = (half == 0 || upd) ? s.z : s.x;
    double* out = (half == 0) ? s.V + (size_t)(s.j + 1) * s.n : s.r;
    finish_rows(s.fin, s.acc, s.tinv, x, [&](int64_t i, int c, double v) {
        const int64_t q = (int64_t)c * M + i;
        const double y = (c == 0 ? s.lam1 : s.lam2) * x[q] + v;
        if (half == 0) out[q] = y;
        else if (upd) out[q] -= y;   // out is r: each thread updates its own entry
        else out[q] = s.g[q] - y;
    });
}

// ---------------------------------------------------------------- vector part (same chunks as alone)
// Blocks of a slot take chunks of its vectors (nblk of them) and leave partial sums; the block that finishes
// last (ticket) adds them in chunk order, so a sum does not depend on which block that is.
constexpr int kDotGroup = 8;   // vectors per pass over a chunk: their warp sums are transposed together

// True in every thread of the block that arrives last; its view of the others' partials is then complete.
__device__ __forceinline__ bool last_block(SlotDev& s) {
    __shared__ int last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
        last = atomicAdd(&s.ticket, 1) == s.nblk - 1;
        if (last) s.ticket = 0;
    }
    __syncthreads();
    if (last) __threadfence();
    return last != 0;
}

// Sum over the block of v[k] of every thread, k < kDotGroup; valid in threads k < kDotGroup (v[k] of thread k).
__device__ __forceinline__ double group_sum(double (&v)[kDotGroup]) {
    __shared__ double sh[kVecThreads / 32][kDotGroup];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int cnt = kDotGroup;
#pragma unroll
    for (int m = 16; m >= 1; m >>= 1) {   // halve the values a lane keeps, then a plain butterfly
        if (cnt > 1) {
            const bool upper = (lane & m) != 0;
            const int h = cnt / 2;
#pragma unroll
            for (int i = 0; i < kDotGroup / 2; ++i) {
                if (i < h) {
                    const double send = upper ? v[i] : v[i + h], keep = upper ? v[i + h] : v[i];
                    v[i] = keep + __shfl_xor_sync(0xffffffffu, send, m);
                }
            }
            cnt = h;
        } else {
            v[0] += __shfl_xor_sync(0xffffffffu, v[0], m);
        }
    }
    __syncthreads();   // the last call's readers are done
    if ((lane & (32 / kDotGroup - 1)) == 0) sh[warp][lane / (32 / kDotGroup)] = v[0];
    __syncthreads();
    double t = 0.0;
    if (threadIdx.x < kDotGroup)
        for (int w = 0; w < kVecThreads / 32; ++w) t += sh[w][threadIdx.x];
    return t;
}

struct Chunk {
    int64_t t0, t1;
};
__device__ __forceinline__ Chunk chunk_of(const SlotDev& s) {
    const int64_t c = (s.n + s.nblk - 1) / s.nblk;
    const int64_t t0 = (int64_t)blockIdx.x * c;
    return Chunk{t0, min(s.n, t0 + c)};
}

// Partial dots <V_i, w>, i <= j, of this block's chunk, and by the last block their sums to out.
__device__ __forceinline__ void chunk_dots(SlotDev& s, const Chunk& c, const double* __restrict__ w,
                                           double* __restrict__ out) {
    const int64_t n = s.n;
    const int j = s.j, nblk = s.nblk;
    for (int i0 = 0; i0 <= j; i0 += kDotGroup) {
        double v[kDotGroup];
#pragma unroll
        for (int k = 0; k < kDotGroup; ++k) v[k] = 0.0;
        const double* a = s.V + (size_t)i0 * n;
        for (int64_t t = c.t0 + threadIdx.x; t < c.t1; t += kVecThreads) {
            const double wt = w[t];
#pragma unroll
            for (int k = 0; k < kDotGroup; ++k)
                if (i0 + k <= j) v[k] += a[(size_t)k * n + t] * wt;
        }
        const double sum = group_sum(v);
        if (threadIdx.x < kDotGroup && i0 + (int)threadIdx.x <= j)
            s.dpart[(size_t)(i0 + threadIdx.x) * nblk + blockIdx.x] = sum;
    }
    if (!last_block(s)) return;
    const int lane = threadIdx.x & 31;
    for (int i = threadIdx.x >> 5; i <= j; i += kVecThreads / 32) {
        double v = 0.0;
        for (int b = lane; b < nblk; b += 32) v += s.dpart[(size_t)i * nblk + b];
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (lane == 0) out[i] = v;
    }
}

// One partial sum per block; by the last block (true there) the total, in every thread.
__device__ __forceinline__ bool chunk_total(SlotDev& s, double mine, double& total) {
    double v[kDotGroup];
#pragma unroll
    for (int k = 0; k < kDotGroup; ++k) v[k] = k == 0 ? mine : 0.0;
    const double sum = group_sum(v);
    if (threadIdx.x == 0) s.dpart[blockIdx.x] = sum;
    if (!last_block(s)) return false;
    const int lane = threadIdx.x & 31;
    double t = 0.0;
    for (int b = lane; b < s.nblk; b += 32) t += s.dpart[b];
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    total = t;
    return true;
}

// w -= V[0..j] c on this block's chunk; returns the thread's sum of squares of the result.
__device__ __forceinline__ double chunk_sub(const SlotDev& s, const Chunk& c, double* __restrict__ w,
                                            const double* __restrict__ coef) {
    const int64_t n = s.n;
    const int j = s.j;
    double ss = 0.0;
    for (int64_t t = c.t0 + threadIdx.x; t < c.t1; t += kVecThreads) {
        double v = w[t];
#pragma unroll 8
        for (int i = 0; i <= j; ++i) v -= s.V[(size_t)i * n + t] * coef[i];
        w[t] = v;
        ss += v * v;
    }
    return ss;
}

__device__ __forceinline__ bool arnoldi_active(const SlotDev& s) {
    return inner_active(s) && (int)blockIdx.x < s.nblk && whole(s, 0);
}

// first Gram-Schmidt coefficients
__global__ void __launch_bounds__(kVecThreads) k_dots(SlotDev* S) {
    SlotDev& s = S[blockIdx.y];
    if (!arnoldi_active(s)) return;
    chunk_dots(s, chunk_of(s), s.V + (size_t)(s.j + 1) * s.n, s.cgs);
}

// w -= V c, second coefficients
__global__ void __launch_bounds__(kVecThreads) k_sub_dots(SlotDev* S) {
    SlotDev& s = S[blockIdx.y];
    if (!arnoldi_active(s)) return;
    const Chunk c = chunk_of(s);
    double* w = s.V + (size_t)(s.j + 1) * s.n;
    (void)chunk_sub(s, c, w, s.cgs);
    chunk_dots(s, c, w, s.cgs2);
}

// Givens update of Hessenberg column j, counters, and the slot's next state (one thread)
__device__ void givens_and_advance(SlotDev& s, double norm2) {
    const int j = s.j, ldh = s.m + 1;
    double* col = s.H + (size_t)j * ldh;
    const double hn = sqrt(norm2);
    double h = s.cgs[0] + s.cgs2[0];   // the column's entry being rotated
    for (int i = 0; i < j; ++i) {
        const double next = s.cgs[i + 1] + s.cgs2[i + 1];
        const double c = s.cs[i], sn = s.sn[i];
        col[i] = c * h + sn * next;
        h = -sn * h + c * next;
    }
    const double den = hypot(h, hn);
    s.cs[j] = h / den;
    s.sn[j] = hn / den;
    col[j] = den;
    col[j + 1] = 0.0;
    const double sj = j == 0 ? s.beta : s.sv[j];
    const double nj = -s.sn[j] * sj;
    s.sv[j] = s.cs[j] * sj;
    s.sv[j + 1] = nj;
    s.scal[2] = hn;
    s.stat.iterations++;
    if (s.inner_prec == CTR_FP32_REFINE) s.stat.matvecs_fp32++; else s.stat.matvecs_fp64++;
    s.budget--;
    const double est = fabs(nj);
    if (!isfinite(est)) s.stat.numeric_error = 1;
    s.part = 0;
    s.span = 1;   // a residual started later in this step runs one part
    if (est <= s.tol_cycle || j + 1 == s.m || s.budget <= 0 || hn == 0.0 || !isfinite(est)) {
        s.kdone = j + 1;
        s.stat.state = kSlotUpdate;
    } else {
        s.j = j + 1;
    }
}

// w -= V c2, its norm, Givens; a slot whose application has parts left waits for the next step instead
__global__ void __launch_bounds__(kVecThreads) k_sub_norm(SlotDev* S, SlotStat* __restrict__ out) {
    SlotDev& s = S[blockIdx.y];
    if (!inner_active(s) || (int)blockIdx.x >= s.nblk) return;
    double total = 0.0;
    if (whole(s, 0)) {
        if (!chunk_total(s, chunk_sub(s, chunk_of(s), s.V + (size_t)(s.j + 1) * s.n, s.cgs2), total)) return;
        if (threadIdx.x == 0) givens_and_advance(s, total);
    } else {
        if (!last_block(s)) return;   // every block has read the state
        if (threadIdx.x == 0) {
            s.part += s.span;
            s.stat.state = kSlotInnerWait;
        }
    }
    if (threadIdx.x == 0) out[blockIdx.y] = s.stat;
}

// Before a half's pair launches (one block): the work counters to zero, and which pair arithmetics any slot
// applies in this half (the inner arithmetic of slots in INNER, the residual arithmetic of slots in UPDATE).
// The persistent pair kernels of the others return at once instead of walking their whole work lists.
__device__ __forceinline__ void begin_half(const SlotDev* S, int cap, int half, int* need, int* counters,
                                           int n_counters, int* tree_counters) {
    __shared__ int f[3];
    if (threadIdx.x < 3) f[threadIdx.x] = 0;
    for (int q = threadIdx.x; q < n_counters; q += blockDim.x) counters[q] = 0;
    if (threadIdx.x < 12) tree_counters[threadIdx.x] = 0;
    __syncthreads();
    for (int q = threadIdx.x; q < cap; q += blockDim.x) {
        const SlotDev& s = S[q];
        if (half == 0 ? inner_active(s) : update_active(s))
            f[arith_index(half == 0 ? s.inner_prec : res_arith(s))] = 1;
    }
    __syncthreads();
    if (threadIdx.x < 3) need[threadIdx.x] = f[threadIdx.x];
}

// Start of the update half, a block per slot: back substitution R y = s, column by column; block 0 also clears
// the work counters and finds the pair arithmetics that the half needs.
__global__ void __launch_bounds__(kVecThreads) k_begin_update(SlotDev* S, int cap, int* need, int* counters,
                                                            int n_counters, int* tree_counters) {
    if (blockIdx.x == 0) begin_half(S, cap, 1, need, counters, n_counters, tree_counters);
    const SlotDev& s = S[blockIdx.x];
    if (!update_active(s) || s.part != 0) return;
    const int k = s.kdone, ldh = s.m + 1;
    for (int l = threadIdx.x; l < k; l += kVecThreads) s.y[l] = s.sv[l];
    __syncthreads();
    for (int i = k - 1; i >= 0; --i) {
        const double* col = s.H + (size_t)i * ldh;
        const double yi = s.y[i] / col[i];
        __syncthreads();
        for (int l = threadIdx.x; l < i; l += kVecThreads) s.y[l] -= col[l] * yi;
        if (threadIdx.x == 0) s.y[i] = yi;
        __syncthreads();
    }
}

// after the residual: converged, out of budget, or the next cycle from r (one thread)
__device__ void decide(SlotDev& s, double norm2) {
    if (s.upd) s.stat.matvecs_fp32++; else s.stat.matvecs_fp64++;
    s.stat.refinements++;
    s.part = 0;
    s.span = 1;
    const double rn = sqrt(norm2);
    s.stat.residual = (s.gnorm > 0.0) ? rn / s.gnorm : 0.0;
    if (!isfinite(rn)) {
        s.stat.numeric_error = 1;
        s.stat.state = kSlotDone;
        return;
    }
    const bool conv = rn <= s.tol_out * s.gnorm;
    const bool out = s.budget <= 0 || (s.refine && s.stat.refinements >= s.max_refine);
    if (conv || out) {
        s.stat.converged = conv ? 1 : 0;
        s.stat.state = kSlotDone;
        return;
    }
    s.beta = rn;
    s.tol_cycle = s.refine ? s.inner_tol * rn : s.tol_out * s.gnorm;
    // The next residual may be updated as r - A d in the inner arithmetic once r is small: the inner
    // operator's error on d (about 1e-7 |A| |d|, |d| ~ |A^-1| |r|) then stays orders of magnitude
    // below the tolerance, while g - A x would need the residual arithmetic at full magnitude.
    s.upd = (s.refine && s.res_update && rn <= kUpdateGate * s.gnorm) ? 1 : 0;
    s.j = 0;
    s.stat.state = kSlotInner;
}

__global__ void __launch_bounds__(kVecThreads) k_residual(SlotDev* S, SlotStat* __restrict__ out) {
    SlotDev& s = S[blockIdx.y];
    if (!update_active(s) || (int)blockIdx.x >= s.nblk) return;
    if (whole(s, 1)) {
        const Chunk c = chunk_of(s);
        double ss = 0.0, total = 0.0;
        for (int64_t t = c.t0 + threadIdx.x; t < c.t1; t += kVecThreads) ss += s.r[t] * s.r[t];
        if (!chunk_total(s, ss, total)) return;
        if (threadIdx.x == 0) decide(s, total);
    } else {
        if (!last_block(s)) return;
        if (threadIdx.x == 0) {
            s.part += s.span;
            s.stat.state = kSlotUpdateWait;
        }
    }
    if (threadIdx.x == 0) out[blockIdx.y] = s.stat;
}

// Estimated pair work of a slot in the step ahead (seconds), and its arithmetic.
__device__ __forceinline__ float step_work(const SlotDev& s, int& a) {
    if (s.stat.state == kSlotInner) a = arith_index(s.inner_prec);
    else if (s.stat.state == kSlotUpdate) a = arith_index(res_arith(s));
    else return 0.f;
    return s.part_s[a];
}

// Start of a step (one block): slots between two parts of an application resume; every slot whose
// application is split gets its span of parts for this step: one, or as many as fit in the pair work of
// all other slots in the step.  A large system thus takes about half of a busy step and one part of an
// otherwise idle one, and the other slots' steps grow by at most that much.
__global__ void __launch_bounds__(kVecThreads) k_plan_step(SlotDev* S, int cap, int* need, int* counters, int n_counters,
                                                         int* tree_counters) {
    __shared__ float red[kVecThreads];
    float w = 0.f;
    for (int q = threadIdx.x; q < cap; q += blockDim.x) {
        SlotDev& s = S[q];
        if (s.stat.state == kSlotInnerWait) s.stat.state = kSlotInner;
        else if (s.stat.state == kSlotUpdateWait) s.stat.state = kSlotUpdate;
        int a = 0;
        w += step_work(s, a);
    }
    red[threadIdx.x] = w;
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if ((int)threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
        __syncthreads();
    }
    const float total = red[0];
    for (int q = threadIdx.x; q < cap; q += blockDim.x) {
        SlotDev& s = S[q];
        int a = 0;
        const float mine = step_work(s, a);
        s.span = 1;
        if (mine > 0.f && s.nparts[a] > 1) {
            const float fit = floorf((total - mine) / mine);
            s.span = max(1, min(s.nparts[a] - s.part, (int)fminf(fit, (float)kMaxParts)));
        }
    }
    begin_half(S, cap, 0, need, counters, n_counters, tree_counters);
}

constexpr int kNV = kNumVar32;   // work lists per arithmetic

template <typename Policy, int R, int V, int U, bool kShared>
int launch_persistent_k(Engine* e, int pol, int var, int half, int prec) {
    const size_t smem = pair_smem_bytes<Policy>();
    static int per_dev[64] = {0};   // resident blocks of this instantiation, per device (attribute set there)
    int dev = 0;
    CTR_CUDA_TRY(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 64) return fail(CTR_ERR_INVALID, "device index");
    int& per_sm = per_dev[dev];
    if (per_sm == 0) {
        int b = 0;
        // dynamic shared memory above the default 48 KB per block needs the kernel's opt-in
        CTR_CUDA_TRY(cudaFuncSetAttribute(k_pairs<Policy, R, V, U, kShared>,
                                          cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        CTR_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_pairs<Policy, R, V, U, kShared>, kThreads,
                                                                   smem));
        per_sm = std::max(1, b);
    }
    const int list = pol * kNV + var;
    k_pairs<Policy, R, V, U, kShared><<<per_sm * e->sms, kThreads, smem, e->stream>>>(
        e->slots.as<SlotDev>(), e->items[pol][var].as<int2>(), e->n_items.as<int>() + list,
        e->counters.as<int>() + 2 * list + half, half, prec, pol, e->exp_tab[pol], e->err, e->kc_val[pol],
        e->need.as<int>());
    CTR_LAUNCHED();
    return CTR_OK;
}

template <typename Policy, int R, int V, int U>
int launch_persistent(Engine* e, int pol, int var, int half, int prec) {
    return e->kc_shared[pol] ? launch_persistent_k<Policy, R, V, U, true>(e, pol, var, half, prec)
                             : launch_persistent_k<Policy, R, V, U, false>(e, pol, var, half, prec);
}

struct PersistentRun {
    Engine* e;
    int var, half;
    template <typename P, int R, int V, int U>
    int run() const { return launch_persistent<P, R, V, U>(e, 0, var, half, CTR_FP32_REFINE); }
};

// Treecode entries of a slot in this half's arithmetic (filtered by the slot's state at run time).
struct EngineTreeAcc {
    const SlotDev* S;
    int half, prec;
    __device__ const TreeView* view(int q) const {
        const SlotDev& s = S[q];
        const bool want = half == 0 ? (inner_active(s) && s.inner_prec == prec) : (update_active(s) && res_arith(s) == prec);
        return (want && s.tv.on) ? &s.tv : nullptr;
    }
};

template <typename Real, int R, int NT>
int launch_tree_engine(Engine* e, int pol, int half, int prec) {
    static std::map<std::pair<int, int>, int> cache;
    const EngineTreeAcc acc{e->slots.as<SlotDev>(), half, prec};
    const int* cnt = e->tree_cnt.as<int>() + 3 * pol;
    int* ctr = e->tree_counters.as<int>() + 4 * pol + 2 * half;
    k_tree_mom<Real, EngineTreeAcc><<<2 * e->sms, kThreads, 0, e->stream>>>(acc, e->tree_ent[pol][0].as<int2>(), cnt,
                                                                          ctr, pol);
    CTR_LAUNCHED();
    k_tree_momred<Real, EngineTreeAcc><<<4 * e->sms, kThreads, 0, e->stream>>>(acc, e->tree_ent[pol][1].as<int2>(),
                                                                             cnt + 1, pol);
    CTR_LAUNCHED();
    if constexpr (sizeof(Real) == 8 && R == kTreeR[1] && NT == kTreeNT[1]) {   // float-float far field
        auto kern = k_tree_far_ff<R, NT, EngineTreeAcc>;
        const int smem = (int)tree_farff_smem(std::max(1, e->tree_np[pol]));   // the largest proxy count admitted
        const int per_sm = far_per_sm(kern, NT, smem, (int)tree_farff_smem(), cache);
        if (per_sm < 0) return per_sm;
        kern<<<per_sm * e->sms, NT, smem, e->stream>>>(acc, e->tree_ent[pol][2].as<int2>(), cnt + 2, ctr + 1);
    } else if constexpr (sizeof(Real) == 4) {
        auto kern = k_tree_far2<R / 2, NT, EngineTreeAcc>;
        const int smem = (int)tree_far2_smem(std::max(1, e->tree_np[pol]));   // the largest proxy count admitted
        const int per_sm = far_per_sm(kern, NT, smem, (int)tree_far2_smem(), cache);
        if (per_sm < 0) return per_sm;
        kern<<<per_sm * e->sms, NT, smem, e->stream>>>(acc, e->tree_ent[pol][2].as<int2>(), cnt + 2, ctr + 1, pol);
    } else {
        auto kern = k_tree_far<Real, R, NT, EngineTreeAcc>;
        const int per_sm = far_per_sm(kern, NT, (int)tree_far_smem<Real>(), (int)tree_far_smem<Real>(), cache);
        if (per_sm < 0) return per_sm;
        kern<<<per_sm * e->sms, NT, tree_far_smem<Real>(), e->stream>>>(acc, e->tree_ent[pol][2].as<int2>(),
                                                                       cnt + 2, ctr + 1, pol);
    }
    CTR_LAUNCHED();
    return CTR_OK;
}

int launch_trees(Engine* e, int half) {
    if (!e->any_tree) return CTR_OK;
    if (e->uses[half][0]) CTR_TRY((launch_tree_engine<float, kTreeR[0], kTreeNT[0]>(e, 0, half, CTR_FP32_REFINE)));
    if (e->uses[half][1]) CTR_TRY((launch_tree_engine<double, kTreeR[1], kTreeNT[1]>(e, 1, half, CTR_DF64)));
    if (e->uses[half][2]) CTR_TRY((launch_tree_engine<double, kTreeR[2], kTreeNT[2]>(e, 2, half, CTR_FP64)));
    return CTR_OK;
}

// One persistent FP32 launch per kernel variant among the occupied slots
int launch_fp32(Engine* e, int half) {
    for (int v = 0; v < kNV; ++v)
        if (e->var_used[v]) CTR_TRY(with_var32(v, PersistentRun{e, v, half}));
    return CTR_OK;
}

}  // namespace

// ---------------------------------------------------------------- host side
static int policy_index(int prec) { return prec == CTR_FP32_REFINE ? 0 : (prec == CTR_DF64 ? 1 : 2); }

Engine::~Engine() {
    for (auto& g : graph_exec)
        if (g) cudaGraphExecDestroy(g);
    if (stream) {
        cudaStreamSynchronize(stream);
        cudaStreamDestroy(stream);
    }
}

int engine_create(int device, int cap, Engine** out) {
    Engine* e = new Engine();
    e->device = device;
    e->cap = cap;
    if (cudaStreamCreateWithFlags(&e->stream, cudaStreamNonBlocking) != cudaSuccess) {
        delete e;
        return fail(CTR_ERR_CUDA, "stream create");
    }
    cudaStream_t stream = e->stream;
    e->host.assign(cap, SlotDev{});
    e->owner.assign(cap, nullptr);
    auto bad = [&](int st) {
        delete e;
        return st;
    };
    int st;
    if ((st = e->slots.alloc(sizeof(SlotDev) * cap)) < 0) return bad(st);
    // the error word of the pair kernels is the state of a stat entry behind the slots' (one copy reads both)
    if ((st = e->stats.alloc(sizeof(SlotStat) * (cap + 1))) < 0) return bad(st);
    static_assert(offsetof(SlotStat, state) == 0, "the error word leads its entry");
    e->err = reinterpret_cast<int*>(e->stats.as<SlotStat>() + cap);
    if ((st = e->n_items.alloc(sizeof(int) * 3 * kNV)) < 0) return bad(st);
    if ((st = e->counters.alloc(sizeof(int) * 2 * 3 * kNV)) < 0) return bad(st);
    if ((st = e->tree_cnt.alloc(sizeof(int) * 9)) < 0) return bad(st);
    if ((st = e->tree_counters.alloc(sizeof(int) * 12)) < 0) return bad(st);
    if (cudaMemsetAsync(e->tree_cnt.p, 0, sizeof(int) * 9, stream) != cudaSuccess)
        return bad(fail(CTR_ERR_CUDA, "memset"));
    if ((st = e->need.alloc(sizeof(int) * 3)) < 0) return bad(st);
    if (cudaMemsetAsync(e->stats.p, 0, sizeof(SlotStat) * (cap + 1), stream) != cudaSuccess)
        return bad(fail(CTR_ERR_CUDA, "memset"));
    if (cudaMemsetAsync(e->n_items.p, 0, sizeof(int) * 3 * kNV, stream) != cudaSuccess)
        return bad(fail(CTR_ERR_CUDA, "memset"));
    for (int q = 0; q < cap; ++q) e->host[q].stat.state = kSlotEmpty;
    if (cudaMemcpyAsync(e->slots.p, e->host.data(), sizeof(SlotDev) * cap, cudaMemcpyHostToDevice, stream) !=
        cudaSuccess)
        return bad(fail(CTR_ERR_CUDA, "slot upload"));
    int sms = 0;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device) != cudaSuccess)
        return bad(fail(CTR_ERR_CUDA, "attribute"));
    e->sms = sms;
    for (int p = 0; p < 3; ++p)
        if ((st = exp_table(device, p, &e->exp_tab[p])) < 0) return bad(st);
    if (cudaStreamSynchronize(stream) != cudaSuccess) return bad(fail(CTR_ERR_CUDA, "sync"));
    *out = e;
    return CTR_OK;
}

// Treecode work lists per pair arithmetic (moment chunks, far clusters, far items of every occupied
// treecode slot), sorted by decreasing cost like the pair items.
static int rebuild_tree_items(Engine* e) {
    bool any = false;
    int counts[9] = {0};
    int np_max[3] = {0, 0, 0};
    for (int p = 0; p < 3; ++p) {
        struct It {
            int2 v;
            double cost;
        };
        std::vector<It> lists[3];
        for (int q = 0; q < e->cap; ++q) {
            ctr_ibim* h = e->owner[q];
            if (!h || !h->tree) continue;
            any = true;
            const SlotDev& s = e->host[q];
            if (policy_index(s.inner_prec) != p && policy_index(s.res_prec) != p) continue;
            const TreeData::Pol& P = h->tree->pol[p];
            np_max[p] = std::max(np_max[p], P.np);
            for (size_t k = 0; k < P.chunks.size(); ++k) lists[0].push_back(It{make_int2(q, (int)k), P.chunk_cost[k]});
            for (int k = 0; k < P.nq; ++k) lists[1].push_back(It{make_int2(q, k), 1.0});
            for (size_t k = 0; k < P.far.size(); ++k) lists[2].push_back(It{make_int2(q, (int)k), P.far_cost[k]});
        }
        for (int k = 0; k < 3; ++k) {
            std::stable_sort(lists[k].begin(), lists[k].end(), [](const It& a, const It& b) { return a.cost > b.cost; });
            std::vector<int2> v(lists[k].size());
            for (size_t i = 0; i < v.size(); ++i) v[i] = lists[k][i].v;
            if ((int64_t)v.size() > e->tree_cap[p][k] || !e->tree_ent[p][k].p) {
                const int64_t capn = std::max<int64_t>(256, (int64_t)v.size() * 2);
                CTR_TRY(e->tree_ent[p][k].alloc(sizeof(int2) * capn));
                e->tree_cap[p][k] = capn;
                e->graph_dirty = true;   // the entry buffer moved
            }
            if (!v.empty())
                CTR_CUDA_TRY(cudaMemcpyAsync(e->tree_ent[p][k].p, v.data(), sizeof(int2) * v.size(),
                                             cudaMemcpyHostToDevice, e->stream));
            counts[3 * p + k] = (int)v.size();
        }
    }
    CTR_CUDA_TRY(cudaMemcpyAsync(e->tree_cnt.p, counts, sizeof(counts), cudaMemcpyHostToDevice, e->stream));
    CTR_CUDA_TRY(cudaStreamSynchronize(e->stream));
    if (any != e->any_tree) {
        e->any_tree = any;
        e->graph_dirty = true;   // the step gains or loses the treecode launches
    }
    for (int p = 0; p < 3; ++p)
        if (np_max[p] != e->tree_np[p]) {
            e->tree_np[p] = np_max[p];
            e->graph_dirty = true;   // the far kernels' shared memory changes
        }
    return CTR_OK;
}

// Rebuild the work lists (every item of every occupied slot's schedule, one list per arithmetic and
// kernel variant; each entry is filtered by its slot's state and part at run time), in decreasing cost
// for the atomic-counter scheduler: each slot's items are already in that order, so the lists are a
// merge of the slots' sequences (ties: lower slot, then lower item first).  A slot whose application
// is split gets its items dealt to the parts in that order, back and forth (0, 1, .., n-1, n-1, .., 0),
// which balances the parts' costs.
static int rebuild_items(Engine* e) {
    bool used[kNV] = {};
    for (int p = 0; p < 3; ++p) {
        struct Seq {
            int q, np;
            const std::vector<double>* cost;
        };
        std::vector<Seq> seqs[kNV];
        for (int q = 0; q < e->cap; ++q) {
            if (!e->owner[q]) continue;
            const SlotDev& s = e->host[q];
            const bool uses = (policy_index(s.inner_prec) == p) || (policy_index(s.res_prec) == p);
            if (!uses) continue;
            const PairSchedule& sc = e->owner[q]->sched[p];
            if (sc.items.size() > (size_t)kItemMask) return fail(CTR_ERR_CAPACITY, "engine: schedule too long");
            const int var = (p == 0) ? sc.var : 0;
            if (p == 0) used[var] = true;
            seqs[var].push_back(Seq{q, std::max(1, s.nparts[p]), &sc.cost});
        }
        // one set of pair constants for every slot of this arithmetic: pass it as a launch parameter
        bool shared = true, any = false;
        PairConsts val{};
        for (int q = 0; q < e->cap && shared; ++q) {
            if (!e->owner[q]) continue;
            const SlotDev& s = e->host[q];
            if (policy_index(s.inner_prec) != p && policy_index(s.res_prec) != p) continue;
            PairConsts c = s.kc;
            c.exp_tab = e->exp_tab[p];
            if (!any) {
                val = c;
                any = true;
            } else if (std::memcmp(&val, &c, sizeof(PairConsts)) != 0) {
                shared = false;
            }
        }
        if (!any) val.exp_tab = e->exp_tab[p];
        if (shared != e->kc_shared[p] || std::memcmp(&val, &e->kc_val[p], sizeof(PairConsts)) != 0) {
            e->kc_shared[p] = shared;
            e->kc_val[p] = val;
            e->graph_dirty = true;   // the captured launches carry the constants
        }
        for (int v = 0; v < kNV; ++v) {
            size_t total = 0;
            for (const Seq& a : seqs[v]) total += a.cost->size();
            std::vector<int2> ent;
            ent.reserve(total);
            std::vector<size_t> pos(seqs[v].size(), 0);
            auto later = [&](int a, int b) {   // heap order: the entry to take next on top
                const double ca = (*seqs[v][a].cost)[pos[a]], cb = (*seqs[v][b].cost)[pos[b]];
                return ca != cb ? ca < cb : a > b;
            };
            std::vector<int> heap;
            for (int a = 0; a < (int)seqs[v].size(); ++a)
                if (!seqs[v][a].cost->empty()) heap.push_back(a);
            std::make_heap(heap.begin(), heap.end(), later);
            while (!heap.empty()) {
                std::pop_heap(heap.begin(), heap.end(), later);
                const int a = heap.back();
                const Seq& sq = seqs[v][a];
                const size_t k = pos[a];
                const int round = (int)(k / (size_t)sq.np), at = (int)(k % (size_t)sq.np);
                const int part = (round & 1) ? sq.np - 1 - at : at;
                ent.push_back(make_int2(sq.q, (int)k | (part << kPartShift)));
                if (++pos[a] < sq.cost->size()) std::push_heap(heap.begin(), heap.end(), later);
                else heap.pop_back();
            }
            if ((int64_t)ent.size() > e->item_cap[p][v]) {
                const int64_t capn = std::max<int64_t>(1024, (int64_t)ent.size() * 2);
                CTR_TRY(e->items[p][v].alloc(sizeof(int2) * capn));
                e->item_cap[p][v] = capn;
                e->graph_dirty = true;   // the item buffer moved
            }
            if (!ent.empty())
                CTR_CUDA_TRY(cudaMemcpyAsync(e->items[p][v].p, ent.data(), sizeof(int2) * ent.size(),
                                             cudaMemcpyHostToDevice, e->stream));
            const int cnt = (int)ent.size();
            CTR_CUDA_TRY(cudaMemcpyAsync(e->n_items.as<int>() + p * kNV + v, &cnt, sizeof(int), cudaMemcpyHostToDevice,
                                         e->stream));
        }
        CTR_CUDA_TRY(cudaStreamSynchronize(e->stream));
    }
    bool uses[2][3] = {};   // arithmetics any slot may apply in the inner and the update half
    for (int q = 0; q < e->cap; ++q) {
        if (!e->owner[q]) continue;
        const SlotDev& s = e->host[q];
        uses[0][policy_index(s.inner_prec)] = uses[1][policy_index(s.res_prec)] = true;
        if (s.res_update) uses[1][policy_index(s.inner_prec)] = true;
    }
    if (std::memcmp(uses, e->uses, sizeof(uses)) != 0) {
        std::memcpy(e->uses, uses, sizeof(uses));
        e->graph_dirty = true;   // the halves gain or lose pair launches
    }
    for (int v = 0; v < kNV; ++v)
        if (used[v] != e->var_used[v]) {
            e->var_used[v] = used[v];
            e->graph_dirty = true;   // the step gains or loses a variant's launches
        }
    return rebuild_tree_items(e);
}

// The kernels of one half of an engine step, in stream order (captured into its graph).
static int enqueue_half(Engine* e, int half) {
    cudaStream_t st = e->stream;
    SlotDev* S = e->slots.as<SlotDev>();
    SlotStat* stats = e->stats.as<SlotStat>();
    const int cap = e->cap, n_counters = 2 * 3 * kNV;
    const dim3 vec(e->vec_blocks, cap), rows(2 * e->vec_blocks, cap);   // a finish block takes half as many rows
    const dim3 chunks(e->max_nblk, cap);
    int *need = e->need.as<int>(), *counters = e->counters.as<int>(), *tree_counters = e->tree_counters.as<int>();
    if (half == 0) {
        k_plan_step<<<1, kVecThreads, 0, st>>>(S, cap, need, counters, n_counters, tree_counters);
        CTR_LAUNCHED();
        k_prep_inner<<<vec, kVecThreads, 0, st>>>(S);
    } else {
        k_begin_update<<<cap, kVecThreads, 0, st>>>(S, cap, need, counters, n_counters, tree_counters);
        CTR_LAUNCHED();
        k_update_x<<<vec, kVecThreads, 0, st>>>(S);
    }
    CTR_LAUNCHED();
    if (e->uses[half][0]) CTR_TRY(launch_fp32(e, half));
    if (e->uses[half][1]) CTR_TRY((launch_persistent<Df64Policy, kRdf, kChunkDf, 1>(e, 1, 0, half, CTR_DF64)));
    if (e->uses[half][2]) CTR_TRY((launch_persistent<Fp64Policy, kR64, kChunk64, 1>(e, 2, 0, half, CTR_FP64)));
    CTR_TRY(launch_trees(e, half));
    k_finish<<<rows, kFinishThreads, 0, st>>>(S, half);
    CTR_LAUNCHED();
    if (half == 0) {
        k_dots<<<chunks, kVecThreads, 0, st>>>(S);
        CTR_LAUNCHED();
        k_sub_dots<<<chunks, kVecThreads, 0, st>>>(S);
        CTR_LAUNCHED();
        k_sub_norm<<<chunks, kVecThreads, 0, st>>>(S, stats);
    } else {
        k_residual<<<chunks, kVecThreads, 0, st>>>(S, stats);
    }
    CTR_LAUNCHED();
    return CTR_OK;
}

static int ensure_graph(Engine* e) {
    if (e->graph_exec[1] && !e->graph_dirty) return CTR_OK;
    for (auto& g : e->graph_exec) {
        if (g) cudaGraphExecDestroy(g);
        g = nullptr;
    }
    if (!e->use_graph) return CTR_OK;
    for (int half = 0; half < 2; ++half) {
        cudaGraph_t g = nullptr;
        const int64_t before = ctr_kernel_launches();
        CTR_CUDA_TRY(cudaStreamBeginCapture(e->stream, cudaStreamCaptureModeThreadLocal));
        const int st = enqueue_half(e, half);
        e->kernels_per_half[half] = ctr_kernel_launches() - before;
        cudaError_t ce = cudaStreamEndCapture(e->stream, &g);
        if (st < 0) {
            if (g) cudaGraphDestroy(g);
            return st;
        }
        if (ce != cudaSuccess) return fail(CTR_ERR_CUDA, std::string("graph capture: ") + cudaGetErrorString(ce));
        ce = cudaGraphInstantiate(&e->graph_exec[half], g, 0);
        cudaGraphDestroy(g);
        if (ce != cudaSuccess) return fail(CTR_ERR_CUDA, std::string("graph instantiate: ") + cudaGetErrorString(ce));
    }
    e->graph_dirty = false;
    return CTR_OK;
}

int engine_admit(Engine* e, ctr_ibim* s, int* slot_out) {
    int q = -1;
    for (int i = 0; i < e->cap; ++i)
        if (!e->owner[i]) {
            q = i;
            break;
        }
    if (q < 0) return fail(CTR_ERR_CAPACITY, "no free engine slot");
    CTR_TRY(engine_prepare_handle(s));
    SlotDev d{};
    d.M = (int)s->M;
    d.n = 2 * s->M;
    d.m = s->kr.m;
    d.nblk = s->kr.nblk;
    d.W = s->na.W;
    d.fin = finish_rows_of(s);
    d.excl = exclusions_of(s);
    d.tinv = s->tree ? s->tree->d_tinv.as<int32_t>() : nullptr;
    if (s->tree) d.tv = s->tree->view;
    d.src32 = s->src32.as<float4>();
    d.src64 = s->src64.as<double4>();
    d.srcdf = s->srcdf.as<float4>();
    d.acc = s->acc.as<unsigned long long>();
    d.g = s->rhs.as<double>();
    d.lam1 = 0.5 * (1.0 + s->eps_out / s->eps_in);
    d.lam2 = 0.5 * (1.0 + s->eps_in / s->eps_out);
    d.il1 = 2.0 / (1.0 + s->eps_out / s->eps_in);
    d.il2 = 2.0 / (1.0 + s->eps_in / s->eps_out);
    d.scale = s->h * s->h * s->h / (4.0 * kPi);
    d.refine = (s->opt.precision == CTR_FP32_REFINE) ? 1 : 0;
    d.inner_prec = s->opt.precision;
    d.res_prec = d.refine ? s->opt.residual : s->opt.precision;
    // a treecode handle's FP32 operator carries its own approximation error (degree 6): its refinement
    // residuals are always formed in full with the residual arithmetic
    d.res_update = (d.refine && s->opt.residual_mode == CTR_RESIDUAL_UPDATE && !s->tree) ? 1 : 0;
    // the slot's two arithmetics were planned at setup from the same options: these are guards
    CTR_TRY(ensure_schedule(s, policy_index(d.inner_prec)));
    CTR_TRY(ensure_schedule(s, policy_index(d.res_prec)));
    d.upd = 0;
    d.part = 0;
    for (int p = 0; p < 3; ++p) {   // parts of one application (treecode handles: always whole)
        const PairSchedule& sc = s->sched[p];
        int64_t np = 1;
        if (e->quantum_s > 0.0 && !s->tree) {
            // a part lasts at least as long as its longest item runs on one block (item_seconds): keep
            // every part at twice that or more, and at kMinItemsPerPart items or more
            const double t = sc.total_cost / kUnitRate[p];
            np = (int64_t)std::ceil(t / e->quantum_s);
            np = std::min<int64_t>(np, (int64_t)(t / (2.0 * item_seconds(p))));
            np = std::min<int64_t>(np, (int64_t)sc.items.size() / kMinItemsPerPart);
        }
        d.nparts[p] = (int)std::max<int64_t>(1, std::min<int64_t>(np, kMaxParts));
        d.part_s[p] = (float)(sc.total_cost / kUnitRate[p] / d.nparts[p]);
    }
    d.span = 1;
    CTR_TRY(pair_consts(s, 0, &d.kc));
    for (int p = 0; p < 3; ++p) {
        d.items[p] = s->sched[p].d_items.as<PairItem>();
        d.BS[p] = s->sched[p].BS;
    }
    double* b = s->vecs.as<double>();
    const int64_t n = d.n;
    d.x = b;
    d.r = b + n;
    d.z = b + 2 * n;
    d.V = s->kr.V.as<double>();
    d.H = s->kr.H.as<double>();
    d.cs = s->kr.cs.as<double>();
    d.sn = s->kr.sn.as<double>();
    d.sv = s->kr.s.as<double>();
    d.y = s->kr.y.as<double>();
    d.cgs = s->kr.y.as<double>() + (d.m + 1);
    d.cgs2 = s->kr.y.as<double>() + 2 * (d.m + 1);
    d.dpart = s->kr.part.as<double>();
    d.scal = s->kr.scal.as<double>();
    d.tol_out = s->opt.tol;
    d.inner_tol = s->opt.inner_tol;
    d.max_refine = s->opt.max_refine;
    d.budget = s->opt.max_iter;
    // initial residual r = g (x = 0) and its norm
    CTR_CUDA_TRY(cudaStreamSynchronize(s->stream));   // the handle's setup work is complete
    CTR_CUDA_TRY(cudaMemsetAsync(d.x, 0, sizeof(double) * n, e->stream));
    CTR_CUDA_TRY(cudaMemcpyAsync(d.r, d.g, sizeof(double) * n, cudaMemcpyDeviceToDevice, e->stream));
    double gn2 = 0.0;
    CTR_TRY(device_dot(s, d.g, d.g, n, &gn2));
    d.gnorm = std::sqrt(gn2);
    d.beta = d.gnorm;
    d.tol_cycle = d.refine ? d.inner_tol * d.gnorm : d.tol_out * d.gnorm;
    d.stat = SlotStat{};
    if (d.gnorm == 0.0) {
        d.stat.state = kSlotDone;
        d.stat.converged = 1;
    } else {
        d.stat.state = kSlotInner;   // the first cycle starts from r = g
    }
    e->host[q] = d;
    e->owner[q] = s;
    CTR_CUDA_TRY(cudaMemcpyAsync(e->slots.as<SlotDev>() + q, &d, sizeof(SlotDev), cudaMemcpyHostToDevice, e->stream));
    CTR_CUDA_TRY(cudaMemcpyAsync(e->stats.as<SlotStat>() + q, &d.stat, sizeof(SlotStat), cudaMemcpyHostToDevice,
                                 e->stream));
    if (d.nblk > e->max_nblk) {   // launch shapes of the captured step change
        e->max_nblk = d.nblk;
        e->graph_dirty = true;
    }
    const int vb = (int)std::min<int64_t>(grid_for(s->M, kVecThreads), 1024);
    if (vb > e->vec_blocks) {
        e->vec_blocks = vb;
        e->graph_dirty = true;
    }
    e->lists_dirty = true;   // the work lists gain its items before the next step
    *slot_out = q;
    return CTR_OK;
}

int engine_retire(Engine* e, int q, ctr_solve_info* info) {
    if (q < 0 || q >= e->cap || !e->owner[q]) return fail(CTR_ERR_INVALID, "bad slot");
    SlotStat st;
    CTR_CUDA_TRY(cudaMemcpyAsync(&st, e->stats.as<SlotStat>() + q, sizeof(SlotStat), cudaMemcpyDeviceToHost, e->stream));
    CTR_CUDA_TRY(cudaStreamSynchronize(e->stream));
    if (st.state == kSlotInnerWait || st.state == kSlotUpdateWait) {
        // retired between two parts of an application (cancelled): its node accumulators hold partial
        // sums; clear them so the handle's next application starts from zero
        ctr_ibim* h = e->owner[q];
        CTR_CUDA_TRY(cudaMemsetAsync(h->acc.p, 0, h->acc.bytes, e->stream));
        CTR_CUDA_TRY(cudaStreamSynchronize(e->stream));
    }
    if (info) {
        info->iterations = st.iterations;
        info->refinements = st.refinements;
        info->matvecs_fp32 = st.matvecs_fp32;
        info->matvecs_fp64 = st.matvecs_fp64;
        info->residual = st.residual;
        info->converged = st.converged;
    }
    SlotDev empty{};
    empty.stat.state = kSlotEmpty;
    e->host[q] = empty;
    e->owner[q] = nullptr;
    CTR_CUDA_TRY(cudaMemcpyAsync(e->slots.as<SlotDev>() + q, &empty, sizeof(SlotDev), cudaMemcpyHostToDevice, e->stream));
    CTR_CUDA_TRY(cudaMemcpyAsync(e->stats.as<SlotStat>() + q, &empty.stat, sizeof(SlotStat), cudaMemcpyHostToDevice,
                                 e->stream));
    e->lists_dirty = true;   // its entries are inert (an empty slot matches no state) until the next rebuild
    return st.numeric_error ? fail(CTR_ERR_NUMERIC, "non-finite residual") : CTR_OK;
}

// One half of a step, the slots' states and the error word read back (they lie side by side on the device).
static int run_half(Engine* e, int half, std::vector<SlotStat>* stats) {
    if (e->graph_exec[half]) {
        CTR_CUDA_TRY(cudaGraphLaunch(e->graph_exec[half], e->stream));
        count_launches(e->kernels_per_half[half]);   // kernels run by the replay
    } else {
        CTR_TRY(enqueue_half(e, half));
    }
    stats->resize(e->cap + 1);
    CTR_CUDA_TRY(cudaMemcpyAsync(stats->data(), e->stats.p, sizeof(SlotStat) * (e->cap + 1), cudaMemcpyDeviceToHost,
                                 e->stream));
    CTR_CUDA_TRY(cudaStreamSynchronize(e->stream));
    const int herr = stats->back().state;
    stats->resize(e->cap);
    if (herr) return fail(CTR_ERR_DEVICE_WAIT, "engine: a bounded device wait expired");
    return CTR_OK;
}

int engine_step(Engine* e, std::vector<SlotStat>* stats) {
    if (e->lists_dirty) {   // one rebuild for all admissions and retirements since the last step
        CTR_TRY(rebuild_items(e));
        e->lists_dirty = false;
    }
    CTR_TRY(ensure_graph(e));
    CTR_TRY(run_half(e, 0, stats));
    bool update = false;   // slots that ended a cycle, or wait between the parts of a residual
    for (const SlotStat& q : *stats) update |= q.state == kSlotUpdate || q.state == kSlotUpdateWait;
    if (update) CTR_TRY(run_half(e, 1, stats));
    e->steps++;
    return CTR_OK;
}

// The handle's solver workspace, sized for the engine (Krylov basis, vectors).
int engine_prepare_handle(ctr_ibim* s) {
    CTR_TRY(ensure_krylov_public(s));
    return CTR_OK;
}

// Solve every handle to completion in one engine (all slots admitted at once).
int engine_solve_all(ctr_ibim* const* hs, int64_t n, int use_graph, std::vector<ctr_solve_info>* infos,
                     int64_t* steps) {
    if (n <= 0) return CTR_OK;
    Engine* e = nullptr;
    CTR_TRY(engine_create(hs[0]->device, (int)n, &e));
    std::unique_ptr<Engine> guard(e);
    e->use_graph = use_graph != 0;
    e->vec_blocks = 1;
    for (int64_t i = 0; i < n; ++i)
        e->vec_blocks = std::max<int>(e->vec_blocks, (int)std::min<int64_t>(grid_for(hs[i]->M, kVecThreads), 1024));
    std::vector<int> slot(n);
    for (int64_t i = 0; i < n; ++i) CTR_TRY(engine_admit(e, hs[i], &slot[i]));
    infos->assign(n, ctr_solve_info{});
    std::vector<int> state(n);
    for (int64_t i = 0; i < n; ++i) state[i] = e->host[slot[i]].stat.state == kSlotDone ? kSlotDone : kSlotInner;
    std::vector<char> done(n, 0);
    std::vector<SlotStat> st;
    int first_error = CTR_OK;
    for (;;) {
        for (int64_t i = 0; i < n; ++i) {
            if (!done[i] && state[i] == kSlotDone) {
                const int r = engine_retire(e, slot[i], &(*infos)[i]);
                if (r < 0 && first_error == CTR_OK) first_error = r;
                done[i] = 1;
            }
        }
        bool left = false;
        for (int64_t i = 0; i < n; ++i) left |= !done[i];
        if (!left) break;
        CTR_TRY(engine_step(e, &st));
        for (int64_t i = 0; i < n; ++i)
            if (!done[i]) state[i] = st[slot[i]].state;
    }
    if (steps) *steps = e->steps;
    return first_error;
}

}  // namespace ctr
