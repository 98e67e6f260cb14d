// tt_modes.cuh -- the projector in detector modes (float handles).
//
// On the detector circle of projection s every even real SH of order <= L is a
// trigonometric polynomial of the azimuth phi with modes 0, 2, .., L (all of
// 0 .. L when two_theta != 0), so the basis matrix factors exactly,
//   B_s = Q F_s,   Q [C][R] the segment means of the modes (the same for all
//   s), F_s [R][K] the modes' Fourier coefficients of Y_i along the circle,
// R = L + 1 (or 2L + 1); with fewer segments than that, Q = 1 and F_s = B_s.
// Every quantity that lives on rays then needs R values instead of K (l_max 4:
// 5 for 15, l_max 8: 8 or 9 for 45): the adjoint gathers R-vectors and maps
// the gathered sum to the K coefficients once per (voxel, projection),
//   g[x] = sum_s F_s^T t_s[x],   t_s[x] = sum_rays w G'_s,   G' = 2 Q^T (W r).
#pragma once

#include "tt_kernels.cuh"

namespace tt {

// ------------------------------------------------------------ mode adjoint
//
// g[x][i] = sum_s sum_m F_s[m][i] t_s[x][m].  A CTA owns 8 x 4 x 8 voxels, two
// tiles of 128; its voxel threads gather t_s for V voxels each, projection by
// projection.  The map to the K coefficients is a contraction over (s, m) and
// runs on the tensor cores: a tile is the M = 128 rows of tcgen05.mma
// kind::tf32, its A operand written by the voxels' own threads into tensor
// memory (row = lane = thread, so nothing is exchanged), B = F_s, D = the
// gradient rows in tensor memory.  FP32 accuracy comes from the split t = t_hi
// + t_lo, F = F_hi + F_lo and three products; t_hi F_lo and t_lo F_hi
// accumulate over all projections in D_lo, t_hi F_hi in D_hi, which every
// kDrain units is added to FP32 registers and restarted: the tensor cores
// truncate their sums (measured: a step that adds less than one unit in the
// last place is lost), so a chain over all projections would drift by 1e-5 of
// the result.
//
// The rays of a block of voxels lie in a small box of the detector, so each
// projection's box of G' rows is staged in shared memory by one tensor copy
// per plane of rows (zeros outside the detector), which leaves the gather
// without bounds tests, 64-bit addresses or cache misses.  Detector
// coordinates are relative to the box, formed in FP64 at the block's corner:
// their FP32 rounding is that of numbers below 32 instead of the detector's
// size.
//
// The kernel that wrote the rows says whether all of them are finite (it
// leaves its number in *nonfinite otherwise); if not, rays of zero weight are
// skipped by a branch, else they are added like the others (0.278 -> 0.257 ms
// at 64^3 against predicated sums).
//
// Units of UP projections pass through three barriers: `stage` (boxes and F
// operand arrived), `full` (a tile's warps have gathered the unit and stored
// its columns: the boxes may be refilled) and `empty` (its products are
// done).  One thread of the last warp issues all copies and products.
//
// Volumes of too few blocks to fill the chip split the projections between
// the CTAs of a cluster (gridDim.y of them), which add their sums through
// distributed shared memory in a fixed order.
//
// Why: gathering K-channel rows moved 75% of what the L1 path can deliver
// (64^3, l_max 4: 0.366 ms; 128^3, l_max 8: 14.4 ms); R = 5 modes are a third
// of those bytes, 8 a sixth.  What bounds it now is instruction issue (70% of
// the slots at l_max 4; the same gather from global memory, with its bounds
// tests and 64-bit addresses, took 0.358) and, at l_max 8, the latency that
// eight resident warps leave: 0.245 and 6.1 ms.

// One G' row of the box.  Rows of two quads (R4 = 2) are 32 bytes apart, so
// that lanes four rows apart read the same banks: lanes 4 .. 7 of every eight
// read (and sum) their second quad first, and mode_store puts the quads back
// (more than half of the wavefronts were conflicts; 128^3, l_max 8: 6.76 ->
// 6.14 ms, 100^3, l_max 6: 2.54 -> 2.39).
template <int R4, int R1>
struct ModeRow {
    float v[4 * R4 + R1];
};

template <int R4, int R1>
__device__ __forceinline__ void mode_load(ModeRow<R4, R1> &x, uint32_t a4, uint32_t a4b, uint32_t a1)
{
#pragma unroll
    for (int i = 0; i < R4; ++i)
        asm("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
            : "=f"(x.v[4 * i]), "=f"(x.v[4 * i + 1]), "=f"(x.v[4 * i + 2]), "=f"(x.v[4 * i + 3])
            : "r"(i ? a4b : a4));
    if constexpr (R1) asm("ld.shared.f32 %0, [%1];" : "=f"(x.v[4 * R4]) : "r"(a1));
}

// t += w * x, as paired FMAs.  GUARD: only where w > 0 -- a ray of zero weight
// must not be touched when it may hold an infinity or NaN.
template <int R4, int R1, bool GUARD>
__device__ __forceinline__ void mode_fma(ModeRow<R4, R1> &t, float w, const ModeRow<R4, R1> &x)
{
    if (GUARD && !(w > 0.f)) return;
#pragma unroll
    for (int i = 0; i < 4 * R4; i += 2) fma2(t.v[i], t.v[i + 1], w, x.v[i], x.v[i + 1]);
    if constexpr (R1) t.v[4 * R4] = fmaf(w, x.v[4 * R4], t.v[4 * R4]);
}

// Integers as floats: for |x| < 2^22, x + kRound has round(x) in its low bits.
constexpr float kRound = 12582912.f;          // 1.5 * 2^23
constexpr int kRoundBits = 0x4b400000;

// One column of candidate rays of a voxel (see k_adjoint for the enumeration):
// outer offset d = o - oc; du, dv the offsets of the column's first ray's taps
// from the voxel, a4 (with a4b, the quad read second) and a1 the addresses of
// its row.  A column that the clamp
// moves holds no ray of positive weight (such rays lie in the box).
struct ModeColumn {
    float du, dv;
    uint32_t a4, a4b, a1;
};
template <int R4>
__device__ __forceinline__ ModeColumn mode_column(const float4 &cu, const float4 &ce, const int4 &ci, float d, float ic,
                                                  int orow, uint32_t b4, uint32_t b4b, uint32_t b1)
{
    const float xr = (ic + fmaxf(fmaf(ce.z, d, ce.x), fmaf(ce.w, d, ce.y))) + kRound;
    const float di = (xr - kRound) - ic;
    ModeColumn r;
    r.du = fmaf(di, cu.z, d * cu.x);
    r.dv = fmaf(di, cu.w, d * cu.y);
    const uint32_t idx = min((uint32_t)(__float_as_int(xr) * ci.y + orow), (uint32_t)ci.w);
    // (opaque, so that the candidates' addresses are these plus uniform steps)
    asm("mad.lo.u32 %0, %1, %2, %3;" : "=r"(r.a4) : "r"(idx), "n"(16 * R4), "r"(b4));
    if constexpr (R4 == 2) asm("mad.lo.u32 %0, %1, %2, %3;" : "=r"(r.a4b) : "r"(idx), "n"(16 * R4), "r"(b4b));
    else r.a4b = 0;
    asm("mad.lo.u32 %0, %1, 4, %2;" : "=r"(r.a1) : "r"(idx), "r"(b1));
    return r;
}

// Weight of candidate b of a column.
__device__ __forceinline__ float mode_weight(const float4 &cu, const ModeColumn &k, int b)
{
    return __saturatef(1.f - fabsf(k.du + (float)b * cu.z)) * __saturatef(1.f - fabsf(k.dv + (float)b * cu.w));
}

template <int R4, int R1, int NO, int NI>
__device__ __forceinline__ void mode_gather(ModeRow<R4, R1> &t, const float4 &cu, const float4 &ce, const int4 &ci,
                                            float d0, float ic, int orow0, uint32_t b4, uint32_t b4b, uint32_t b1)
{
#pragma unroll
    for (int a = 0; a < NO; ++a) {
        const ModeColumn k = mode_column<R4>(cu, ce, ci, d0 + (float)a, ic, orow0 + a * ci.x, b4, b4b, b1);
        ModeRow<R4, R1> x[NI];
#pragma unroll
        for (int b = 0; b < NI; ++b) mode_load<R4, R1>(x[b], k.a4 + b * ci.y * (16 * R4), k.a4b + b * ci.y * (16 * R4), k.a1 + b * ci.y * 4);
#pragma unroll
        for (int b = 0; b < NI; ++b) mode_fma<R4, R1, false>(t, mode_weight(cu, k, b), x[b]);
    }
}

// Windows of any size (unequal voxel and pixel sizes), and guarded.
template <int R4, int R1, bool GUARD>
__device__ __forceinline__ void mode_gather_any(ModeRow<R4, R1> &t, const float4 &cu, const float4 &ce, const int4 &ci,
                                                float d0, float ic, int orow0, uint32_t b4, uint32_t b4b, uint32_t b1, int order)
{
    const int NO = order & 0xff, NI = (order >> 8) & 0xff;
    for (int a = 0; a < NO; ++a) {
        const ModeColumn k = mode_column<R4>(cu, ce, ci, d0 + (float)a, ic, orow0 + a * ci.x, b4, b4b, b1);
        for (int b = 0; b < NI; ++b) {
            ModeRow<R4, R1> x;
            mode_load<R4, R1>(x, k.a4 + b * ci.y * (16 * R4), k.a4b + b * ci.y * (16 * R4), k.a1 + b * ci.y * 4);
            mode_fma<R4, R1, GUARD>(t, mode_weight(cu, k, b), x);
        }
    }
}

// v = hi + lo with hi rounded to tf32 (11 significant bits, to nearest); the
// tensor cores read lo's 11 leading bits, so hi + lo carries v to about 2^-22
// with errors of random sign.
__device__ __forceinline__ void tf32_split(float v, uint32_t &hi, uint32_t &lo)
{
    hi = (__float_as_uint(v) + 0x1000u) & 0xffffe000u;
    lo = __float_as_uint(v - __uint_as_float(hi));
}

// A projection's operand columns of one voxel: R split modes, hi then lo, in
// consecutive columns.
template <int R4, int R1>
__device__ __forceinline__ void mode_store(uint32_t ta, ModeRow<R4, R1> t)
{
    constexpr int M = 4 * R4 + R1;
    uint32_t v[2 * M];
    if constexpr (R4 == 2) {
        const bool swapped = threadIdx.x & 4;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float a = t.v[i], b = t.v[4 + i];
            t.v[i] = swapped ? b : a;
            t.v[4 + i] = swapped ? a : b;
        }
    }
#pragma unroll
    for (int i = 0; i < M; ++i) tf32_split(t.v[i], v[i], v[M + i]);
    if constexpr (2 * M >= 16) {
        umma::tmem_st16(ta, v);
        if constexpr (R1) umma::tmem_st2(ta + 16, v + 16);
    } else {
        umma::tmem_st8(ta, v);
        if constexpr (R1) umma::tmem_st2(ta + 8, v + 8);
    }
}

// The fixed-order sum of sum_fixed_order by the first 128 threads of the block,
// thread t doing the work of threads t and t + 128.
__device__ __forceinline__ double sum_fixed_order_half(const double *__restrict__ p, long long n, double *red)
{
    constexpr int NT = kThreads / 2;
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const double v = warp_sum(threadIdx.x < NT ? strided_sum(p, n, threadIdx.x + k * NT) : 0.0);
        if (l == 0 && threadIdx.x < NT) red[w + k * (NT / 32)] = v;
    }
    __syncthreads();
    return w == 0 ? warp_sum(l < kThreads / 32 ? red[l] : 0.0) : 0.0;
}

// Infinities.  A voxel that an infinite ray reaches gets NaN from the modes
// (inf - inf, in the split and in the sum over modes) where the sum over the
// K channels is an infinity of one sign, or a NaN.  Behind a tt_adjoint whose
// data are not all finite, this puts the channels' values there, from the
// caller's data R.  (A kernel of its own behind the adjoint took 4 us of every
// call.)
__device__ static void adjoint_infinite_at(const ModeData &d, float *gx, int K, int KP, int x, int y, int z)
{
    bool nan = false;
    for (int i = 0; i < K; ++i) nan = nan || isnan(gx[i]);
    if (!nan) return;
    const double at[3] = {(double)x, (double)y, (double)z};
    float acc[kModeKMax];
    for (int i = 0; i < K; ++i) acc[i] = 0.f;
    for (int s = 0; s < d.S; ++s) {
        const ProjGeom &P = d.geo[s];
        const double jc = P.jc0 + P.jU * at[P.u] + P.jV * at[P.v] + P.jP * at[P.m];
        const double kc = P.kc0 + P.kU * at[P.u] + P.kV * at[P.v] + P.kP * at[P.m];
        const int j1 = (int)fmin(floor(jc + P.hj), d.nj - 1.0), k1 = (int)fmin(floor(kc + P.hk), d.nk - 1.0);
        for (int j = (int)fmax(ceil(jc - P.hj), 0.0); j <= j1; ++j)
            for (int k = (int)fmax(ceil(kc - P.hk), 0.0); k <= k1; ++k) {
                const double du = P.u0 + j * P.uj + k * P.uk + at[P.m] * P.up - at[P.u];
                const double dv = P.v0 + j * P.vj + k * P.vk + at[P.m] * P.vp - at[P.v];
                const float w = (float)(P.step * fmax(0.0, 1.0 - fabs(du)) * fmax(0.0, 1.0 - fabs(dv)));
                const float *r = d.R + (((long long)s * d.nj + j) * d.nk + k) * d.C;
                bool finite = true;
                for (int c = 0; c < d.C; ++c) finite = finite && isfinite(r[c]);
                if (finite || !(w > 0.f)) continue;
                for (int i = 0; i < K; ++i) {
                    float b = 0.f;
                    for (int c = 0; c < d.C; ++c) b = fmaf(d.Bp[((size_t)s * d.CP + c) * KP + i], r[c], b);
                    acc[i] = fmaf(w, b, acc[i]);
                }
            }
    }
    for (int i = 0; i < K; ++i)
        if (isnan(gx[i]) && !isfinite(acc[i])) gx[i] = acc[i];
}
// The voxels that this warp wrote (finds its place again, so that the kernel
// keeps no register for it).
__device__ __noinline__ static void adjoint_infinite(const ModeData &d, bool any, float *g, int K, int KP, int nx, int ny,
                                                     int nz, int ty, int tz)
{
    if (!any) return;
    __syncwarp();
    const int b = blockIdx.x, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int X = b / (tz * ty) * 8, y = (b / tz) % ty * 4 + warp, z = b % tz * 8 + lane;
    if (warp >= 4 || y >= ny || lane >= 8 || z >= nz) return;
    for (int x = X + blockIdx.y; x < min(X + 8, nx); x += gridDim.y)
        adjoint_infinite_at(d, g + (((long long)x * ny + y) * nz + z) * K, K, KP, x, y, z);
}

template <int N, int R4, int R1>
__global__ void __launch_bounds__(kModeThreads, mode_ctas(N))
k_adjoint_modes(const __grid_constant__ ModeParams P, const __grid_constant__ TmaDesc tm4,
                const __grid_constant__ TmaDesc tm1, int ns, int s_base, const ModeOrigin *__restrict__ org,
                const float *__restrict__ FB, int bj, int bk, int nx, int ny, int nz, int ty, int tz,
                float *__restrict__ gpad, int KP, int accumulate, float *__restrict__ gout, int K,
                const double *__restrict__ loss_partials, long long n_partials, double *__restrict__ loss_out,
                LossSlot *loss_slot, unsigned long long loss_seq, const unsigned *__restrict__ nonfinite, unsigned rows_id,
                const __grid_constant__ ModeData data)
{
    constexpr int M = 4 * R4 + R1, SW = 2 * M, UP = modes_up(M), KU = modes_ku(M), V = 2, NVW = kModeVox / V / 32;
    constexpr int kDrain = (N == 16 ? 4 : 8) / UP;                // units per D_hi chain
    constexpr int COLS = KU + 2 * N <= 64 ? 64 : 128;             // tensor-memory columns of a tile
    static_assert(KU + 2 * N <= COLS && UP * SW <= KU, "tensor-memory budget");
    constexpr uint32_t UB = 2u * KU * N * 4u;                     // F operands of a unit: for D_lo, for D_hi

    // kModeStages x UP x (box of rows, box of single values), then kModeStages
    // F operands
    extern __shared__ unsigned char smem_modes[];
    __shared__ __align__(8) uint64_t stage[kModeStages], full, empty;
    __shared__ float4 hdr[64];   // box origins of projections, ring: outer, inner coordinate of the corner; j, k
    __shared__ uint32_t tslot;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // CTA 0 first sums the forward's loss partials (see k_adjoint).
    if (loss_out && blockIdx.x == 0 && blockIdx.y == 0) {
        __shared__ double lred[32];
        const double v = sum_fixed_order_half(loss_partials, n_partials, lred);
        if (threadIdx.x == 0) {
            loss_out[0] = v;
            if (loss_slot) {
                *(volatile double *)&loss_slot->value = v;
                __threadfence_system();
                *(volatile unsigned long long *)&loss_slot->seq = loss_seq;
            }
        }
    }
    if (warp == NVW) umma::tmem_alloc(&tslot, 2 * COLS);
    if (threadIdx.x == 0) {
        umma::mbar_init(&full, NVW);
        umma::mbar_init(&empty, 1);
        for (int t = 0; t < kModeStages; ++t) umma::mbar_init(&stage[t], 2);
    }
    const uint32_t nbox = (uint32_t)(bj * bk), box4 = nbox * 16 * R4, box1 = R1 ? nbox * 4 : 0;
    const uint32_t box4a = mode_align(box4), boxes = box4a + mode_align(box1);   // bytes of a projection's boxes
    const uint32_t ring = mode_align(umma::smem_u32(smem_modes));
    const uint32_t fring = ring + kModeStages * UP * boxes;
    umma::fence_before_sync();
    __syncthreads();
    umma::fence_after_sync();
    const uint32_t tbase = tslot;
    // this CTA's share of the units, [u_begin, u_end): the cluster's CTAs split them
    const int units = (ns + UP - 1) / UP, split = gridDim.y;
    const int u_begin = units * (int)blockIdx.y / split, nu = units * ((int)blockIdx.y + 1) / split - u_begin;
    ns = min(ns, (u_begin + nu) * UP);

    const int b = blockIdx.x;
    const int X = b / (tz * ty) * 8, Y = (b / tz) % ty * 4, Z = b % tz * 8;

    if (warp == NVW) {
        constexpr uint32_t idesc = umma::idesc_tf32_f32(128, N);
        // Box origins of 32 projections, one per lane, in FP64 at the block's
        // corner (the ring's previous 32 but one are done with).
        auto origins = [&](int s0) {
            if (s0 + lane < ns) {
                const ModeOrigin &o = org[s0 + lane];
                const double j = o.j[0] + o.j[1] * X + o.j[2] * Y + o.j[3] * Z;
                const double k = o.k[0] + o.k[1] * X + o.k[2] * Y + o.k[3] * Z;
                const int jb = (int)floor(j + o.jlo), kb = (int)floor(k + o.klo) & ~3;
                const float jr = (float)(j - jb), kr = (float)(k - kb);
                hdr[(s0 + lane) & 63] = make_float4(o.outer_j ? jr : kr, o.outer_j ? kr : jr, __int_as_float(jb),
                                                    __int_as_float(kb));
            }
            __syncwarp();
        };
        // boxes, F operand of unit u into its stage
        auto boxes_of = [&](int u) {
            const int st = u % kModeStages, s0 = (u_begin + u) * UP, n = min(UP, ns - s0);
            umma::mbar_arrive_expect_tx(&stage[st], n * (box4 + box1));
            for (int q = 0; q < n; ++q) {
                const uint32_t dst = ring + (st * UP + q) * boxes;
                const int si = s0 + q, s = s_base + si;
                const int jb = __float_as_int(hdr[si & 63].z), kb = __float_as_int(hdr[si & 63].w);
                umma::tma_load_3d_s(dst, &tm4, 4 * R4 * kb, jb, s, &stage[st]);
                if constexpr (R1) umma::tma_load_3d_s(dst + box4a, &tm1, kb, jb, s, &stage[st]);
            }
        };
        auto operand_of = [&](int u) {
            const int st = u % kModeStages;
            umma::mbar_arrive_expect_tx(&stage[st], UB);
            umma::bulk_g2s_s(fring + st * UB, FB + (size_t)(u_begin + u) * (UB / 4), UB, &stage[st]);
        };
        origins(u_begin * UP);
        if (lane == 0)
            for (int u = 0; u < min(kModeStages, nu); ++u) {
                boxes_of(u);
                operand_of(u);
            }
        bool ok = true;
        int u = 0;
        for (; u < nu; ++u) {
            const int st = u % kModeStages, un = u + kModeStages;   // un: the unit fetched in this step
            if (un * UP % 32 == 0) origins((u_begin + un) * UP);
            if (lane == 0) {
                const uint32_t f = fring + st * UB;
                ok = umma::mbar_wait(&stage[st], (u / kModeStages) & 1, kModeWaitTries) &&
                     umma::mbar_wait(&full, u & 1, kModeWaitTries);
                if (ok) {
                    umma::fence_after_sync();
#pragma unroll
                    for (int tile = 0; tile < 2; ++tile) {
                        const uint32_t a = tbase + tile * COLS, dhi = a + KU, dlo = dhi + N;
#pragma unroll
                        for (int ks = 0; ks < KU / 8; ++ks) {
                            umma::mma_tf32_ts(dlo, a + 8 * ks, umma::smem_desc(f + ks * N * 32, N * 16, 128), idesc,
                                              (u > 0 || ks > 0) ? 1 : 0);
                            umma::mma_tf32_ts(dhi, a + 8 * ks, umma::smem_desc(f + UB / 2 + ks * N * 32, N * 16, 128),
                                              idesc, (u % kDrain > 0 || ks > 0) ? 1 : 0);
                        }
                    }
                    umma::mma_commit(&empty);
                    // every warp has gathered unit u (its boxes are free) and had
                    // seen the products of unit u - 1 done (its operand is free)
                    if (un < nu) boxes_of(un);
                    if (u >= 1 && un - 1 < nu) operand_of(un - 1);
                }
            }
            ok = __shfl_sync(0xffffffffu, ok, 0);
            if (!ok) break;
        }
        // no copy may still be writing shared memory when the CTA exits
        if (!ok && lane == 0)
            for (int n = u; n < min(nu, u + kModeStages); ++n)
                umma::mbar_wait(&stage[n % kModeStages], (n / kModeStages) & 1, kModeWaitTries);
        __syncwarp();
    } else {
        // the thread's voxels, v = 0 and 1 in the tiles of that number, x = 4 v +
        // vx: every eight lanes hold a patch of 4 (z) x 2 (x), whose rays meet
        // in fewer banks than those of eight in a row (128^3, l_max 4:
        // 3.469 -> 3.440 ms; 247 projections of 65 x 55: 0.410 -> 0.405)
        const int vz = (lane & 3) | ((lane >> 1) & 4), vx = ((lane >> 2) & 1) | ((lane >> 3) & 2);
        const float lx = (float)vx, ly = (float)warp, lz = (float)vz;
        const uint32_t tw = tbase + ((uint32_t)(warp * 32) << 16);
        float acc[V][N];
#pragma unroll
        for (int v = 0; v < V; ++v)
#pragma unroll
            for (int i = 0; i < N; ++i) acc[v][i] = 0.f;
        if constexpr (UP * SW < KU) {   // unused columns must be zero, not what an earlier kernel left there
#pragma unroll
            for (int v = 0; v < V; ++v)
#pragma unroll
                for (int i = UP * SW; i < KU; i += 2) {
                    const uint32_t zero[2] = {0, 0};
                    umma::tmem_st2(tw + v * COLS + i, zero);
                }
            umma::tmem_wait_st();
        }
        bool ok = true;                                            // false once a wait gave up: the rest is NaN
        const bool guard = *nonfinite == rows_id;                  // some row is not finite
        const uint32_t quad0 = R4 == 2 ? (lane & 4) * 4 : 0;       // offset of the quad read first
        uint32_t stage_phase = 0, empty_phase = 1, box = ring;
        uint64_t *bar = stage;
        int drain = 0, si = u_begin * UP;
        for (int u = 0; u < nu; ++u) {
            ok = umma::mbar_wait(bar, stage_phase, ok ? kModeWaitTries : 1) && ok;
#pragma unroll 1
            for (int q = 0; q < UP; ++q, ++si, box += boxes) {
                ModeRow<R4, R1> t[V];
#pragma unroll
                for (int v = 0; v < V; ++v)
#pragma unroll
                    for (int i = 0; i < M; ++i) t[v].v[i] = 0.f;
                if (si < ns) {
                    const ModeProj &c = P.p[si];
                    const float4 co = *reinterpret_cast<const float4 *>(c.o), cs = *reinterpret_cast<const float4 *>(c.i);
                    const float4 cu = *reinterpret_cast<const float4 *>(&c.uo), ce = *reinterpret_cast<const float4 *>(&c.au);
                    const int4 ci = *reinterpret_cast<const int4 *>(&c.so);
                    const float2 hd = *reinterpret_cast<const float2 *>(&hdr[si & 63]);
                    const uint32_t b4 = box + quad0, b4b = box + (quad0 ^ 16), b1 = box + box4a;
                    float oc[V], ic[V], d0[V];
                    int orow[V];
                    oc[0] = fmaf(co.z, lz, fmaf(co.y, ly, fmaf(co.x, lx, hd.x)));
                    ic[0] = fmaf(cs.z, lz, fmaf(cs.y, ly, fmaf(cs.x, lx, hd.y)));
                    oc[1] = fmaf(4.f, co.x, oc[0]);
                    ic[1] = fmaf(4.f, cs.x, ic[0]);
#pragma unroll
                    for (int v = 0; v < V; ++v) {
                        const float xr = (oc[v] + co.w) + kRound;   // floor(oc - ho) + 1
                        d0[v] = (xr - kRound) - oc[v];
                        orow[v] = __float_as_int(xr) * ci.x + ci.z;
                    }
#define TT_MODE_CASE(NO_, NI_)                                                                              \
    case 16 * NO_ + NI_:                                                                                    \
        _Pragma("unroll") for (int v = 0; v < V; ++v)                                                       \
            mode_gather<R4, R1, NO_, NI_>(t[v], cu, ce, ci, d0[v], ic[v], orow[v], b4, b4b, b1);                 \
        break;
                    switch (guard ? -1 : c.shape) {
                    TT_MODE_CASE(1, 1) TT_MODE_CASE(1, 2) TT_MODE_CASE(1, 3)
                    TT_MODE_CASE(2, 1) TT_MODE_CASE(2, 2) TT_MODE_CASE(2, 3)
                    TT_MODE_CASE(3, 1) TT_MODE_CASE(3, 2) TT_MODE_CASE(3, 3)
                    case 0:
#pragma unroll
                        for (int v = 0; v < V; ++v)
                            mode_gather_any<R4, R1, false>(t[v], cu, ce, ci, d0[v], ic[v], orow[v], b4, b4b, b1, c.order);
                        break;
                    default:
#pragma unroll
                        for (int v = 0; v < V; ++v)
                            mode_gather_any<R4, R1, true>(t[v], cu, ce, ci, d0[v], ic[v], orow[v], b4, b4b, b1, c.order);
                        break;
                    }
#undef TT_MODE_CASE
                }
                if (q == 0 && u > 0) {
                    ok = umma::mbar_wait(&empty, empty_phase, ok ? kModeWaitTries : 1) && ok;
                    __syncwarp();
                    umma::fence_after_sync();
                    if (++drain == kDrain) {
                        drain = 0;
#pragma unroll
                        for (int v = 0; v < V; ++v)
#pragma unroll
                            for (int i = 0; i < N; i += 16) {
                                float d[16];
                                umma::tmem_ld16(tw + v * COLS + KU + i, d);
#pragma unroll
                                for (int k = 0; k < 16; ++k) acc[v][i + k] += d[k];
                            }
                    }
                }
                __syncwarp();
#pragma unroll
                for (int v = 0; v < V; ++v) mode_store<R4, R1>(tw + v * COLS + q * SW, t[v]);
            }
            umma::tmem_wait_st();
            umma::fence_before_sync();
            __syncwarp();
            if (lane == 0) umma::mbar_arrive(&full);
            empty_phase ^= 1;
            if (++bar == stage + kModeStages) {
                bar = stage;
                box = ring;
                stage_phase ^= 1;
            }
        }
        ok = __all_sync(0xffffffffu, umma::mbar_wait(&empty, (nu - 1) & 1, ok ? kModeWaitTries : 1) && ok);
        umma::fence_after_sync();
        // Every warp is past its last box (the products of the last unit are
        // done): the ring's start now takes the voxels' sums, K floats each, so
        // that a run of eight voxels along z is what g holds of them.
        const uint32_t row = ring + (warp * 32 + vx * 8 + vz) * (K * 4);
#pragma unroll
        for (int v = 0; v < V; ++v)
#pragma unroll
            for (int i = 0; i < N; i += 16) {
                float d[16], e[16];
                umma::tmem_ld16(tw + v * COLS + KU + i, d);
                umma::tmem_ld16(tw + v * COLS + KU + N + i, e);
#pragma unroll
                for (int k = 0; k < 16; ++k)
                    if (i + k < K)
                        asm volatile("st.shared.f32 [%0], %1;" ::"r"(row + (v * 128 * K + i + k) * 4),
                                     "f"(ok ? acc[v][i + k] + (d[k] + e[k]) : __int_as_float(0x7fc00000))
                                     : "memory");
            }
    }
    // The columns go back before the CTA waits for its cluster: a peer may still
    // be waiting to allocate its own, and no CTA may hold any while it waits.
    umma::fence_before_sync();
    __syncthreads();
    umma::fence_after_sync();
    if (warp == NVW) umma::tmem_dealloc(tbase, 2 * COLS);
    if (split > 1) umma::cluster_sync();
    // The cluster's CTAs share out the runs and add the CTAs' sums in their order.
    const int nz8 = min(8, nz - Z) * K;
    if (warp < NVW && Y + warp < ny)
        for (int r = blockIdx.y; r < 8; r += split) {      // tile r / 4, its x row r % 4
            const int x = X + r;
            if (x >= nx) break;
            const long long vox = ((long long)x * ny + Y + warp) * nz + Z;
            const uint32_t at = ring + ((r >> 2) * 128 + warp * 32 + (r & 3) * 8) * (K * 4);
            for (int e = lane; e < nz8; e += 32) {
                float sum;
                if (split == 1) {
                    asm volatile("ld.shared.f32 %0, [%1];" : "=f"(sum) : "r"(at + 4 * e) : "memory");
                } else {
                    sum = umma::cluster_load(at + 4 * e, 0);
                    for (int k = 1; k < split; ++k) sum += umma::cluster_load(at + 4 * e, k);
                }
                if (gout && !accumulate) {
                    gout[vox * K + e] = sum;
                } else {
                    const long long o = (vox + e / K) * KP + e % K;
                    if (accumulate) sum += gpad[o];
                    if (gout) gout[vox * K + e] = sum;
                    else gpad[o] = sum;
                }
            }
        }
    if (split > 1) umma::cluster_sync();                   // no CTA leaves while its sums are read
    if (data.R) adjoint_infinite(data, *nonfinite == rows_id, gout, K, KP, nx, ny, nz, ty, tz);
}

// ------------------------------------------------- back-contraction to modes
// G'[pix][m] = sum_c Q[c][m] R[pix][c], one thread per ray.
template <int R4, int R1>
__global__ void __launch_bounds__(kThreads)
k_backcontract_modes(const float *__restrict__ Q /*[C][kModeQ]*/, const float *__restrict__ R, float *__restrict__ G4,
                     float *__restrict__ G1, long long npix, int nk, int nk1, int C, unsigned *__restrict__ nonfinite,
                     unsigned rows_id)
{
    const long long pix = (long long)blockIdx.x * kThreads + threadIdx.x;
    if (pix >= npix) return;
    constexpr int M = 4 * R4 + R1;
    float t[M];
#pragma unroll
    for (int m = 0; m < M; ++m) t[m] = 0.f;
    const float *r = R + pix * C;
    auto one = [&](int c, float v) {
#pragma unroll
        for (int m = 0; m < M; ++m) t[m] = fmaf(__ldg(Q + c * kModeQ + m), v, t[m]);
    };
    if ((C & 3) == 0) {
        for (int c = 0; c < C; c += 4) {
            const float4 v = __ldg(reinterpret_cast<const float4 *>(r + c));
            one(c, v.x);
            one(c + 1, v.y);
            one(c + 2, v.z);
            one(c + 3, v.w);
        }
    } else {
        for (int c = 0; c < C; ++c) one(c, __ldg(r + c));
    }
#pragma unroll
    for (int i = 0; i < R4; ++i)
        reinterpret_cast<float4 *>(G4 + pix * (4 * R4))[i] = make_float4(t[4 * i], t[4 * i + 1], t[4 * i + 2], t[4 * i + 3]);
    if constexpr (R1) G1[pix / nk * nk1 + pix % nk] = t[4 * R4];
    if (!rows_finite(t)) *nonfinite = rows_id;
}

}  // namespace tt
