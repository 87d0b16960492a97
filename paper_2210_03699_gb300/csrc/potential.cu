// Reaction potential at arbitrary points (Eq. 2.31) as a tiled pair sum: potential maps and the
// polarization energy (Eq. 3.3).
//
//   psi_rxn(z) = h^3 sum_j W_j [ ((eps_E/eps_I) dGk/dn_y - dG0/dn_y)(z, P_j) psi_j + (G0 - Gk)(z, P_j) dpsi_j ]
//
// by the plain trapezoidal rule on the tube (z away from the surface).  With a_j = h^3 W_j psi_j / (4 pi),
// b_j = h^3 W_j dpsi_j / (4 pi), d = z - P_j, s = 1/r^3, E = e^{-kappa r}, E1 = E (1 + kappa r):
//
//   psi_rxn(z) = sum_j [ a_j (d.n_j) s ((eps_E/eps_I) E1 - 1) + b_j (1 - E) / r ]
//              = sum_j 1/r [ a_j (d.n_j) ((eps_E/eps_I) E1 - 1)/r^2 + b_j (1 - E) ].
//
// The points are the targets (registers), the tube nodes the sources: the packed source arrays of the
// operator (their weight slots rewritten with a, b) streamed through the same two-stage shared-memory
// ring (cp.async.bulk + mbarrier) as the operator's pair items.  A grid of (target block, source split)
// blocks writes per-split FP64 partial sums (per-tile sums folded into FP64), added in split order by a
// second kernel: the result does not depend on scheduling.  Float-float and FP64, and FP32 at few points or
// nodes, take a thread per point and short run of sources instead (map_unit_kernel).  Three arithmetics:
//   Fp32x2  two points per f32x2 instruction, 19 FMA-pipe lane operations + 2 SFU per pair;
//   Df64    float-float (the operator's residual arithmetic), one point per thread;
//   Fp64    IEEE FP64 (the energy of ctr_ibim_energy).
// The split partials live in a workspace the handle keeps and grows (no allocation once it is large
// enough).
#include <cmath>

#include "pairkern.cuh"

namespace ctr {

using namespace pk;

namespace {

// ---------------------------------------------------------------- map policies
struct MapFp32x2 {
    using Src = ulonglong2;   // the operator's packed FP32 node {(x,x),(y,y)} {(z,z),(a,a)} {(nx,nx),(ny,ny)} {(nz,nz),(-b,-b)}
    static constexpr int kVec = 4;
    static constexpr int kTile = 256, kUnit = kTile;
    static constexpr int kPack = 2;
    static constexpr int kR = 2;
    static constexpr int kTab = 0;
    struct Tgt {
        u64 x, y, z;
    };
    using Acc = u64;
    __device__ static Tgt load(const double* xyz, int64_t n, const int64_t* p) {
        float v[2][3];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int64_t q = min(p[h], n - 1);
#pragma unroll
            for (int c = 0; c < 3; ++c) v[h][c] = (float)xyz[3 * q + c];
        }
        return Tgt{pk2(v[0][0], v[1][0]), pk2(v[0][1], v[1][1]), pk2(v[0][2], v[1][2])};
    }
    __device__ static void zero(Acc& a) { a = 0ull; }
    __device__ static void fold(const Acc& a, double* s) {
        float x, y;
        up2(a, x, y);
        s[0] += (double)x;
        s[1] += (double)y;
    }
    // acc += 1/r [ a (d.n) (c1 E1 - 1)/r^2 + b (1 - E) ],  c1 E1 = E (c1 + c1 kappa r)
    __device__ static void pair(const Tgt& T, const Src* S, const PairConsts& k, const float2*, Acc& acc) {
        const ulonglong2 v0 = S[0], v1 = S[1], v2 = S[2], v3 = S[3];
        const u64 dx = sub2(T.x, v0.x), dy = sub2(T.y, v0.y), dz = sub2(T.z, v1.x);
        const u64 r2 = fma2(dz, dz, fma2(dy, dy, mul2(dx, dx)));
        const u64 rinv = rsqrt2(r2);
        const u64 r = mul2(r2, rinv);
        const u64 E = ex2_2(mul2(k.kl2x2, r));
        const u64 dny = fma2(dz, v3.x, fma2(dy, v2.y, mul2(dx, v2.x)));
        const u64 t = fma2(E, fma2(k.c1kap2, r, k.c1x2), k.mone2);
        const u64 ad = mul2(mul2(v1.y, dny), mul2(rinv, rinv));
        acc = fma2(rinv, fma2(ad, t, fma2(v3.y, E, neg2(v3.y))), acc);
    }
};

// float-float node {P.hi, a.hi} {P.lo, a.lo} {n.hi, b.hi} {n.lo, b.lo}
struct MapDf64 {
    using Src = float4;
    static constexpr int kVec = 4;
    static constexpr int kUnit = 128;   // 32, 64 take 5% to 16% longer at large maps
    static constexpr int kPack = 1;
    static constexpr int kTab = kExpHi + kExpLo;
    struct Tgt {
        F2 x, y, z;
    };
    using Acc = F2;
    __device__ static Tgt load(const double* xyz, int64_t n, const int64_t* p) {
        const int64_t q = min(p[0], n - 1);
        F2 c[3];
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            const double v = xyz[3 * q + i];
            const float hi = (float)v;
            c[i] = F2{hi, (float)(v - (double)hi)};
        }
        return Tgt{c[0], c[1], c[2]};
    }
    __device__ static void zero(Acc& a) { a = F2{0.f, 0.f}; }
    __device__ static void fold(const Acc& a, double* s) { s[0] += (double)a.hi + (double)a.lo; }
    __device__ static void pair(const Tgt& T, const Src* S, const PairConsts& k, const float2* tab, Acc& acc) {
        const float4 s0 = S[0], s1 = S[1], s2 = S[2], s3 = S[3];
        const F2 dx = sub(T.x, F2{s0.x, s1.x}), dy = sub(T.y, F2{s0.y, s1.y}), dz = sub(T.z, F2{s0.z, s1.z});
        const F2 r2 = sq3l(dx, dy, dz);
        const F2 rinv = rsqrt_ff(r2);
        const F2 kr = mull(f2(k.kappad), mull(r2, rinv));
        const F2 E = exp_neg_ffl(kr, tab);
        const F2 E1 = addl(E, mull(E, kr));
        const F2 dny = dot3l(dx, dy, dz, F2{s2.x, s3.x}, F2{s2.y, s3.y}, F2{s2.z, s3.z});
        const F2 s = mull(mull(rinv, rinv), rinv);
        const F2 nt = one_minus_any(mull(E1, f2(k.c1d)));   // 1 - c1 E1
        acc_mul(acc, neg(mull(F2{s0.w, s1.w}, s)), mull(dny, nt));
        acc_mul(acc, F2{s2.w, s3.w}, mull(rinv, one_minus(E)));
        acc = fast_two_sum(acc.hi, acc.lo);
    }
};

// FP64 node {P, a} {n, b}
struct MapFp64 {
    using Src = double4;
    static constexpr int kVec = 2;
    static constexpr int kUnit = 64;    // 128: 1.6x the time of a few points, 0.7% less at large maps
    static constexpr int kPack = 1;
    static constexpr int kTab = kExp2F2;
    struct Tgt {
        double x, y, z;
    };
    using Acc = double;
    __device__ static Tgt load(const double* xyz, int64_t n, const int64_t* p) {
        const int64_t q = min(p[0], n - 1);
        return Tgt{xyz[3 * q], xyz[3 * q + 1], xyz[3 * q + 2]};
    }
    __device__ static void zero(Acc& a) { a = 0.0; }
    __device__ static void fold(const Acc& a, double* s) { s[0] += a; }
    // as MapFp32x2; 28 FP64 operations per pair
    __device__ static void pair(const Tgt& T, const Src* S, const PairConsts& k, const float2* tab, Acc& acc) {
        const double4 pa = S[0], nb = S[1];
        const double dx = T.x - pa.x, dy = T.y - pa.y, dz = T.z - pa.z;
        const double r2 = fma(dz, dz, fma(dy, dy, dx * dx));
        const double rinv = rsqrt_d(r2);
        const double r = r2 * rinv;
        const double E = exp_neg_d(r, k, tab);
        const double dny = fma(dz, nb.z, fma(dy, nb.y, dx * nb.x));
        const double t = fma(E, fma(k.c1kap, r, k.c1), -1.0);
        const double ad = pa.w * dny * (rinv * rinv);
        acc = fma(rinv, fma(ad, t, fma(-nb.w, E, nb.w)), acc);
    }
};

// One block: points [blockIdx.x * BS, +BS) against sources [j_begin, j_end) of its split; the sums go to
// part[split * n + point].  Pol: an arithmetic without exponential tables (FP32).
template <typename Pol>
__global__ void __launch_bounds__(kThreads) map_kernel(const typename Pol::Src* __restrict__ src, int M,
                                                       const double* __restrict__ xyz, int64_t n, int per_split,
                                                       double* __restrict__ part, PairConsts kc,
                                                       int* __restrict__ err) {
    using Src = typename Pol::Src;
    constexpr int TILE = Pol::kTile, VEC = Pol::kVec, P = Pol::kPack, R = Pol::kR, RP = R * P;
    constexpr int BS = kThreads * RP;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    Src* ring = reinterpret_cast<Src*>(smem_raw);
    __shared__ __align__(8) uint64_t bar[2];
    if (threadIdx.x == 0) {
        mbar_init(&bar[0], 1);
        mbar_init(&bar[1], 1);
        fence_mbar_init();
    }
    __syncthreads();
    const int tid = threadIdx.x;
    const int j_begin = blockIdx.y * per_split;
    const int j_end = min(M, j_begin + per_split);
    const int ntiles = (j_end > j_begin) ? (j_end - j_begin + TILE - 1) / TILE : 0;
    int64_t pi[RP];
    double s[RP];
    typename Pol::Tgt tg[R];
#pragma unroll
    for (int a = 0; a < RP; ++a) {
        pi[a] = (int64_t)blockIdx.x * BS + a * kThreads + tid;
        s[a] = 0.0;
    }
#pragma unroll
    for (int r = 0; r < R; ++r) tg[r] = Pol::load(xyz, n, &pi[r * P]);
    auto issue = [&](int k) {
        const int j0 = j_begin + k * TILE;
        const uint32_t bytes = (uint32_t)(min(TILE, j_end - j0) * VEC * sizeof(Src));
        fence_proxy_async();
        mbar_expect_tx(&bar[k & 1], bytes);
        bulk_load(ring + (k & 1) * TILE * VEC, src + (size_t)VEC * j0, bytes, &bar[k & 1]);
    };
    if (tid == 0 && ntiles > 0) issue(0);
    for (int k = 0; k < ntiles; ++k) {
        if (tid == 0 && k + 1 < ntiles) issue(k + 1);
        const bool ok = mbar_wait(&bar[k & 1], (k >> 1) & 1, kc.wait_limit);
        if (__syncthreads_or(!ok)) {   // give up: flag, let both copies in flight land, return
            if (tid == 0) {
                atomicOr(err, kErrWait);
                (void)mbar_wait(&bar[k & 1], (k >> 1) & 1);
                if (k + 1 < ntiles) (void)mbar_wait(&bar[(k + 1) & 1], ((k + 1) >> 1) & 1);
            }
            return;
        }
        const Src* tile = ring + (k & 1) * TILE * VEC;
        const int cnt = min(TILE, j_end - (j_begin + k * TILE));
        typename Pol::Acc acc[R];
#pragma unroll
        for (int r = 0; r < R; ++r) Pol::zero(acc[r]);
#pragma unroll 2
        for (int q = 0; q < cnt; ++q) {
#pragma unroll
            for (int r = 0; r < R; ++r) Pol::pair(tg[r], tile + q * VEC, kc, nullptr, acc[r]);
        }
#pragma unroll
        for (int r = 0; r < R; ++r) Pol::fold(acc[r], &s[r * P]);
        __syncthreads();   // this buffer is free for the tile after next
    }
#pragma unroll
    for (int a = 0; a < RP; ++a)
        if (pi[a] < n) part[(size_t)blockIdx.y * n + pi[a]] = s[a];
}

// out[p] = sum over splits of part[split * n + p], in split order
__global__ void map_sum_kernel(const double* __restrict__ part, int splits, int64_t n, double* __restrict__ out) {
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= n) return;
    double v = 0.0;
    for (int q = 0; q < splits; ++q) v += part[(size_t)q * n + p];
    out[p] = v;
}

// A thread per kPack points and unit of kUnit sources, read through L1; part[unit * n + p] is the unit's sum.
// map_unit_sum_kernel adds the units of a group, then the groups, in order.
//   float-float, FP64: every map and energy.  Pipe- and latency-bound: blocks of a (target block, split) grid
//     left SMs idle at few points and made a ragged last wave at many.
//     us, grid -> units (FP64): 3 points, 11,203 nodes 1313 -> 136; 3, 178,575: 2582 -> 140; 500, 44,597:
//     1319 -> 1185; 4000, 178,575: 38,941 -> 35,998.  float-float: 252 -> 115, 424 -> 132, 259 -> 221,
//     5239 -> 4860.
//   FP32: few points or small systems only (map_fp32); the units and groups are then map_kernel's tiles and
//     splits, and a point's result has the same bits from either.
constexpr int kUnitThreads = 128;
template <typename Pol>
__global__ void __launch_bounds__(kUnitThreads) map_unit_kernel(const typename Pol::Src* __restrict__ src, int M,
                                                                const double* __restrict__ xyz, int64_t n,
                                                                int64_t slots, int units, double* __restrict__ part,
                                                                PairConsts kc) {
    constexpr int UNIT = Pol::kUnit, VEC = Pol::kVec, P = Pol::kPack;
    __shared__ float2 tab[Pol::kTab > 0 ? Pol::kTab : 1];
    for (int q = threadIdx.x; q < Pol::kTab; q += kUnitThreads) tab[q] = kc.exp_tab[q];
    __syncthreads();
    const int64_t g = (int64_t)blockIdx.x * kUnitThreads + threadIdx.x;
    const int64_t unit = g / slots;
    if (unit >= units) return;
    int64_t pi[P];
    double s[P];
#pragma unroll
    for (int h = 0; h < P; ++h) {
        pi[h] = g - unit * slots + h * slots;
        s[h] = 0.0;
    }
    const typename Pol::Tgt tg = Pol::load(xyz, n, pi);
    const int j0 = (int)unit * UNIT, cnt = min(UNIT, M - j0);
    const typename Pol::Src* S = src + (size_t)VEC * j0;
    typename Pol::Acc acc;
    Pol::zero(acc);
#pragma unroll 4
    for (int q = 0; q < cnt; ++q) Pol::pair(tg, S + q * VEC, kc, tab, acc);
    Pol::fold(acc, s);
#pragma unroll
    for (int h = 0; h < P; ++h)
        if (pi[h] < n) part[unit * n + pi[h]] = s[h];
}

// a warp per point: a lane adds the units of one group, the groups' sums are then added in order
__global__ void map_unit_sum_kernel(const double* __restrict__ part, int units, int per_group, int64_t n,
                                    double* __restrict__ out) {
    const int64_t p = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (p >= n) return;
    const int lane = threadIdx.x & 31;
    double v = 0.0;
    for (int t0 = 0; t0 < units; t0 += 32 * per_group) {
        const int b = t0 + lane * per_group, e = min(units, b + per_group);
        double s = 0.0;
        for (int t = b; t < e; ++t) s += part[(size_t)t * n + p];
        for (int l = 0; l < 32 && t0 + l * per_group < units; ++l) v += __shfl_sync(0xffffffffu, s, l);
    }
    if (lane == 0) out[p] = v;
}

// a = h^3 W psi / (4 pi), b = h^3 W dpsi / (4 pi) into the weight slots of one packed source array
__global__ void map_pack_kernel(const double* __restrict__ psi, const double* __restrict__ dpsi,
                                const double* __restrict__ W, int64_t M, double scale, int prec,
                                float4* __restrict__ s32, double4* __restrict__ s64, float4* __restrict__ sdf,
                                const int32_t* __restrict__ tinv) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= M) return;
    const double a = scale * W[t] * psi[t], b = scale * W[t] * dpsi[t];
    const int64_t j = tinv ? (int64_t)tinv[t] : t;
    if (prec == CTR_FP32_REFINE) {
        s32[4 * j + 1].z = s32[4 * j + 1].w = (float)a;
        s32[4 * j + 3].z = s32[4 * j + 3].w = -(float)b;
    } else if (prec == CTR_FP64) {
        s64[2 * j].w = a;
        s64[2 * j + 1].w = b;
    } else {
        const float ah = (float)a, bh = (float)b;
        sdf[4 * j].w = ah;
        sdf[4 * j + 1].w = (float)(a - (double)ah);
        sdf[4 * j + 2].w = bh;
        sdf[4 * j + 3].w = (float)(b - (double)bh);
    }
}

template <typename Pol>
constexpr size_t map_smem() {
    static_assert(Pol::kTab == 0, "the tiled map kernel carries no exponential tables");
    return 2 * Pol::kTile * Pol::kVec * sizeof(typename Pol::Src);
}

// Unit sums of one launch: 32 MB of workspace (more only for 8.4 million nodes and up), and at a million threads or more its last wave is a small part.
// More points go in chunks.
constexpr int64_t kUnitSums = 4 << 20;
// FP32 maps of at most this many unit sums take map_unit_kernel: its sources come through L1, not by bulk
// copies, and it holds two points a thread, not four, but its threads fill the chip at any shape.  us, units
// against map_kernel: 2000 points, 44,597 nodes (350,000 sums) 148 : 210; 500, 178,575 (349,000) 164 : 223;
// 1000, 178,575 (698,000) 244 : 218; 4000, 44,597 (700,000) 238 : 207.
constexpr int64_t kUnitSums32 = 1 << 19;

// points of one launch
int64_t unit_chunk(int64_t units, int64_t n) {
    return std::min(n, std::max<int64_t>(32, kUnitSums / units / 32 * 32));
}

template <typename Pol>
int map_units(ctr_ibim* s, const void* src, const double* d_xyz, int64_t n, const PairConsts& kc, int per_group,
              double* d_out) {
    const int64_t M = s->M, units = (M + Pol::kUnit - 1) / Pol::kUnit;
    const int64_t chunk = unit_chunk(units, n);
    CTR_TRY(s->map_ws.alloc(sizeof(double) * (size_t)(units * chunk)));
    for (int64_t p = 0; p < n; p += chunk) {
        const int64_t m = std::min(chunk, n - p), slots = (m + Pol::kPack - 1) / Pol::kPack;
        map_unit_kernel<Pol><<<grid_for(units * slots, kUnitThreads), kUnitThreads, 0, s->stream>>>(
            reinterpret_cast<const typename Pol::Src*>(src), (int)M, d_xyz + 3 * p, m, slots, (int)units,
            s->map_ws.as<double>(), kc);
        CTR_LAUNCHED();
        map_unit_sum_kernel<<<grid_for(32 * m, 256), 256, 0, s->stream>>>(s->map_ws.as<double>(), (int)units, per_group,
                                                                         m, d_out + p);
        CTR_LAUNCHED();
    }
    return CTR_OK;
}

int map_fp32(ctr_ibim* s, const double* d_xyz, int64_t n, const PairConsts& kc, double* d_out) {
    using Pol = MapFp32x2;
    constexpr int BS = kThreads * Pol::kR * Pol::kPack;
    static int per_dev[64] = {0};   // resident blocks per SM of map_kernel, per device
    int dev = 0, sms = 0;
    CTR_CUDA_TRY(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 64) return fail(CTR_ERR_INVALID, "device index");
    CTR_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    const size_t smem = map_smem<Pol>();
    if (per_dev[dev] == 0) {
        int b = 0;
        CTR_CUDA_TRY(cudaFuncSetAttribute(map_kernel<Pol>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        CTR_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, map_kernel<Pol>, kThreads, smem));
        per_dev[dev] = std::max(1, b);
    }
    const int64_t M = s->M;
    const int64_t tblocks = (n + BS - 1) / BS;
    // source splits: about two waves of resident blocks, whole tiles, at least four tiles per split
    const int64_t want = std::max<int64_t>(1, 2LL * per_dev[dev] * sms / std::max<int64_t>(1, tblocks));
    const int64_t max_splits = std::max<int64_t>(1, M / (4 * Pol::kTile));
    int64_t splits = std::min<int64_t>({want, max_splits, 4096});
    int64_t per = (M + splits - 1) / splits;
    per = ((per + Pol::kTile - 1) / Pol::kTile) * Pol::kTile;
    splits = (M + per - 1) / per;
    if ((M + Pol::kTile - 1) / Pol::kTile * n <= kUnitSums32)
        return map_units<Pol>(s, s->src32.p, d_xyz, n, kc, (int)(per / Pol::kTile), d_out);
    CTR_TRY(s->map_ws.alloc(sizeof(double) * (size_t)(splits * n)));
    dim3 grid((unsigned)tblocks, (unsigned)splits);
    map_kernel<Pol><<<grid, kThreads, smem, s->stream>>>(reinterpret_cast<const Pol::Src*>(s->src32.p), (int)M, d_xyz,
                                                         n, (int)per, s->map_ws.as<double>(), kc, s->err.as<int>());
    CTR_LAUNCHED();
    map_sum_kernel<<<grid_for(n, 256), 256, 0, s->stream>>>(s->map_ws.as<double>(), (int)splits, n, d_out);
    CTR_LAUNCHED();
    return CTR_OK;
}

}  // namespace

int64_t energy_workspace_bytes(int64_t M, int64_t n) {
    if (M <= 0 || n <= 0) return 0;
    const int64_t units = (M + MapFp64::kUnit - 1) / MapFp64::kUnit;
    return (int64_t)sizeof(double) * units * unit_chunk(units, n);
}

int potential_map(ctr_ibim* s, const double* d_psi, const double* d_dpsi, int64_t n, const double* d_xyz,
                  double* d_out, int precision) {
    if (n <= 0) return CTR_OK;
    const int64_t M = s->M;
    const double scale = s->h * s->h * s->h / (4.0 * kPi);
    const int32_t* tinv = s->tree ? s->tree->d_tinv.as<int32_t>() : nullptr;
    map_pack_kernel<<<grid_for(M, 256), 256, 0, s->stream>>>(d_psi, d_dpsi, s->na.W, M, scale, precision,
                                                            s->src32.as<float4>(), s->src64.as<double4>(),
                                                            s->srcdf.as<float4>(), tinv);
    CTR_LAUNCHED();
    PairConsts kc;
    CTR_TRY(pair_consts(s, precision == CTR_DF64 ? 1 : (precision == CTR_FP64 ? 2 : 0), &kc));
    if (n > (int64_t)INT32_MAX) return fail(CTR_ERR_CAPACITY, "more than 2^31 - 1 points");
    if (precision == CTR_FP32_REFINE) return map_fp32(s, d_xyz, n, kc, d_out);
    // sqrt(units) units per group: short chains of additions, and the same for any number of points, so a
    // point's result does not depend on the others
    const int64_t unit = precision == CTR_DF64 ? MapDf64::kUnit : MapFp64::kUnit;
    const int per_group = (int)std::ceil(std::sqrt((double)((M + unit - 1) / unit)));
    if (precision == CTR_DF64) return map_units<MapDf64>(s, s->srcdf.p, d_xyz, n, kc, per_group, d_out);
    return map_units<MapFp64>(s, s->src64.p, d_xyz, n, kc, per_group, d_out);
}

}  // namespace ctr
