// tt_modes_fwd.cu -- forward projection in detector modes: per projection the
// volume's K coefficients are mapped to its R modes (a contraction on the
// tensor cores), and the rays march the mapped volume, whose taps are R
// instead of K values.
//
//   map    V_s[x][m] = sum_i F_s[m][i] c[x][i]
//   march  t[ray][m] = step sum_taps w V_s[tap][m],   I_hat = Q t
//
// The mapped volumes of a chunk of projections live in slots that the next
// chunk reuses.
#include "tt_modes.cuh"

namespace tt {

// NC packed coefficients of a voxel, as loaded.
template <typename S, int NC>
struct RowRegs {
    static constexpr int NW = NC * (int)sizeof(S) / 4;
    unsigned w[NW];
    __device__ __forceinline__ void load(const S *p) { ldg_words<NC * (int)sizeof(S), NC * sizeof(S) % 16 == 0 ? 16 : 8>(p, w); }
    __device__ __forceinline__ float get(int i) const { return word_elem<float, S>(w, i); }
};

// ------------------------------------------------------------ map kernel
//
// A tile is 128 voxels (consecutive along the innermost axis of the packed
// copy the projections read): their coefficients, split into tf32 parts, are
// the rows of the A operand in tensor memory; B holds the F rows of a group of
// projections; the accumulator's row of a voxel is its mode vectors of all
// those projections, stored as rows of four floats (and single values) that
// consecutive lanes write contiguously.  The tensor cores truncate each step's
// sum, a bias that all voxels of a ray add up.  So the order-0 coefficient,
// which exceeds the others in any object and has the same factor Y_00 in every
// projection, stays out of the products and is added to the drained rows by one
// rounded FMA; the cross products come first, then hi * hi from the highest
// order down, so that what is truncated is small.  (With order 0 among the
// products and the orders ascending, projections of objects were 4e-7 (l_max 6)
// and 6e-7 (l_max 8) off, all of one sign; now 1e-7, as the direct march.)
// Warps w and w + 4 share tensor-memory lanes 32 w .., split the
// coefficients of their voxels between them and store every other four
// projections.
constexpr int kMapThreads = 256;
constexpr float kY00f = 0.28209479177387814f;             // 1 / (2 sqrt(pi))

template <typename S, int KP, int M>
__global__ void __launch_bounds__(kMapThreads, 2)
k_map_modes(const S *__restrict__ cpad, const float2 *__restrict__ FM, const int *__restrict__ order, int nproj,
            int group, int n_in, int ny, int n_out, float *__restrict__ slots, long long slot_floats,
            long long slot_vox, int n0 /* modes that order 0 contributes to */)
{
    constexpr int R4 = M / 4, R1 = M & 1, NC = KP / 2;
    extern __shared__ __align__(128) unsigned char map_smem[];
    float *Bh = reinterpret_cast<float *>(map_smem);       // hi, then lo: [KP / 4][N / 8][8][4]
    __shared__ __align__(8) uint64_t done;
    __shared__ uint32_t tslot;
    const int p0 = blockIdx.y * group, P = min(group, nproj - p0), N = (P * M + 15) / 16 * 16;
    float *Bl = Bh + KP * N;
    for (int e = threadIdx.x; e < N * KP; e += kMapThreads) {
        const int n = e / KP, k = e - n * KP, p = n / M;
        const float2 f = p < P ? FM[(size_t)order[p0 + p] * M * KP + (n - p * M) * KP + k] : make_float2(0.f, 0.f);
        const int o = ((k >> 2) * (N / 8) + (n >> 3)) * 32 + (n & 7) * 4 + (k & 3);
        Bh[o] = f.x;
        Bl[o] = f.y;
    }
    const int warp = threadIdx.x >> 5, half = warp >> 2, row = threadIdx.x & 127;
    if (warp == 0) umma::tmem_alloc(&tslot, kMapCols);
    if (threadIdx.x == 0) umma::mbar_init(&done, 1);
    umma::fence_async_smem();
    umma::fence_before_sync();
    __syncthreads();
    umma::fence_after_sync();
    const uint32_t tb = tslot, tw = tb + ((uint32_t)((warp & 3) * 32) << 16), dcol = 2 * KP;
    const uint32_t idesc = umma::idesc_tf32_f32(128, N), sh = umma::smem_u32(Bh), sl = umma::smem_u32(Bl);

    // Rows are taken in whole groups of eight voxels; those behind the row's
    // end are zero, like the border they lie in.
    const int n8 = (n_in + 7) & ~7, npos = n8 * ny * n_out, ntiles = (npos + 127) / 128;
    const S *src = cpad + half * NC;
    int rowi = 0, in = 0;
    RowRegs<S, NC> c;
    float next0 = 0.f;                                     // the voxel's order-0 coefficient
    auto fetch = [&](long long t) {
        const int v = (int)min(t * 128 + row, (long long)npos - 1);
        in = v % n8;
        const int r = v / n8, y = r % ny, out = r / ny;
        rowi = (out + kSlotBorder) * (ny + 2 * kSlotBorder) + y + kSlotBorder;
        // (behind a row's end the packed copy has two zeros, then the next row)
        const S *at = src + (((long long)(out + 2) * (ny + 4) + (y + 2)) * (n_in + 4) + min(in, n_in) + 2) * KP;
        c.load(at);
        next0 = half ? float(at[-NC]) : c.get(0);
    };
    fetch(blockIdx.x);
    bool ok = true;                                        // false once a wait gave up: the rest is NaN
    uint32_t phase = 0;
    for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x, phase ^= 1) {
        const bool live = tile * 128 + row < npos;
        const float y0 = next0;
        const int here4 = rowi * slot_pitch4(n_in) + in + kSlotLead, here1 = rowi * slot_pitch1(n_in) + in + kSlotLead;
#pragma unroll
        for (int i = 0; i < NC; i += 8) {
            uint32_t hi[8], lo[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) tf32_split(c.get(i + k), hi[k], lo[k]);
            umma::tmem_st8(tw + half * NC + i, hi);
            umma::tmem_st8(tw + KP + half * NC + i, lo);
        }
        umma::tmem_wait_st();
        umma::fence_before_sync();
        __syncthreads();      // also: every warp has read the previous tile's accumulators
        if (threadIdx.x == 0) {
            umma::fence_after_sync();
#pragma unroll
            for (int ks = 0; ks < KP / 8; ++ks) {
                const uint64_t bh = umma::smem_desc(sh + ks * N * 32, N * 16, 128);
                const uint64_t bl = umma::smem_desc(sl + ks * N * 32, N * 16, 128);
                umma::mma_tf32_ts(tb + dcol, tb + 8 * ks, bl, idesc, ks > 0);
                umma::mma_tf32_ts(tb + dcol, tb + KP + 8 * ks, bh, idesc, 1);
            }
#pragma unroll
            for (int ks = KP / 8 - 1; ks >= 0; --ks)
                umma::mma_tf32_ts(tb + dcol, tb + 8 * ks, umma::smem_desc(sh + ks * N * 32, N * 16, 128), idesc, 1);
            umma::mma_commit(&done);
        }
        fetch((long long)tile + gridDim.x);                // the next tile's rows travel while the products run
        ok = __all_sync(0xffffffffu, umma::mbar_wait(&done, phase, ok ? kModeWaitTries : 1)) && ok;
        umma::fence_after_sync();
        for (int p = 4 * half; p < P; p += 8) {
            float d[4 * M];
            umma::tmem_ldn<4 * M>(tw + dcol + p * M, d);
#pragma unroll
            for (int t = 0; t < 4; ++t) {
                d[t * M] = fmaf(kY00f, y0, d[t * M]);
                if (n0 > 1)
#pragma unroll
                    for (int i = 1; i < M; ++i)
                        if (i < n0) d[t * M + i] = fmaf(kY00f, y0, d[t * M + i]);
            }
            if (!ok)
#pragma unroll
                for (int i = 0; i < 4 * M; ++i) d[i] = __int_as_float(0x7fc00000);
            float *o = slots + (p0 + p) * slot_floats;
            if (live) {
#pragma unroll
                for (int t = 0; t < 4; ++t) {
                    if (p + t >= P) break;
#pragma unroll
                    for (int g = 0; g < R4; ++g)
                        *reinterpret_cast<float4 *>(o + t * slot_floats + (g * slot_vox + here4) * 4) =
                            make_float4(d[t * M + 4 * g], d[t * M + 4 * g + 1], d[t * M + 4 * g + 2], d[t * M + 4 * g + 3]);
                    if constexpr (R1) o[t * slot_floats + R4 * 4 * slot_vox + here1] = d[t * M + 4 * R4];
                }
            }
        }
        umma::fence_before_sync();
    }
    __syncthreads();
    if (warp == 0) umma::tmem_dealloc(tb, kMapCols);
}

// A ray through an infinite coefficient is a NaN in every mode where the sum
// over channels is an infinity of one sign, or a NaN: the channels' values of
// such a ray, from the packed volume.
template <typename S>
__device__ void project_infinite_as(const ModeVolume &V, const ProjGeom &P, int s, int j, int k, int C, int CP, float *out)
{
    float ur, vr, lo = 0.f, hi = (float)(P.Nm - 1);
    ray_base<float>(P, j, k, ur, vr);
    const float up = (float)P.up, vp = (float)P.vp;
    clip_planes<float>(ur, up, P.Nu, lo, hi);
    clip_planes<float>(vr, vp, P.Nv, lo, hi);
    const S *vol = (const S *)(P.copy ? V.cpadx : V.cpad);
    float acc[kModeKMax];
    for (int i = 0; i < V.K; ++i) acc[i] = 0.f;
    const int phi = min(P.Nm - 1, (int)ceilf(hi));
    for (int p = max(0, (int)floorf(lo)); p <= phi; ++p) {
        const float u = fmaf((float)p, up, ur), v = fmaf((float)p, vp, vr), fu = floorf(u), fv = floorf(v);
        const int iu = min(max((int)fu, -2), P.Nu), iv = min(max((int)fv, -2), P.Nv);
        for (int t = 0; t < 4; ++t) {
            const float w = (t & 1 ? u - fu : 1.f - (u - fu)) * (t & 2 ? v - fv : 1.f - (v - fv));
            const S *tap = vol + ((long long)p * P.sm + (long long)(iu + (t & 1)) * P.su + iv + (t >> 1)) * V.KP;
            for (int i = 0; i < V.K; ++i) acc[i] = fmaf(w, float(tap[i]), acc[i]);
        }
    }
    for (int c = 0; c < C; ++c) {
        float v = 0.f;
        for (int i = 0; i < V.K; ++i) v = fmaf(V.Bp[((size_t)s * CP + c) * V.KP + i], acc[i], v);
        if (!isfinite(v)) out[c] = v;
    }
}
__device__ __noinline__ static void project_infinite(const ModeVolume &V, const ProjGeom &P, int s, int j, int k, int C,
                                                     int CP, float *out)
{
    if (V.prec == TT_BF16) project_infinite_as<__nv_bfloat16>(V, P, s, j, k, C, CP, out);
    else if (V.prec == TT_F16) project_infinite_as<__half>(V, P, s, j, k, C, CP, out);
    else project_infinite_as<float>(V, P, s, j, k, C, CP, out);
}

// ------------------------------------------------------------ march kernel
//
// Two lanes per ray, lane h taking the tap column iv + h: the pair of taps of
// a row is 32 contiguous bytes and a quarter-warp's four neighbouring rays
// span little more than one 128-byte line, so the 80 (R = 5) or 128 (R = 8)
// bytes a ray needs per plane take about that many bytes' wavefronts.  A tile
// is 8 x 16 rays.  The epilogue splits the segments between the two lanes.
constexpr int kMarchTJ = 8, kMarchTK = 16, kMarchThreads = 256;

template <int M, int MODE>
__global__ void __launch_bounds__(kMarchThreads)
k_march_modes(const ProjGeom *__restrict__ geo, const int *__restrict__ order, const float *__restrict__ slots,
              long long slot_floats, long long slot_vox, int nx, int ny, int nz, int nj, int nk, int C, int CP,
              int tiles_k, const float *__restrict__ Q, float *__restrict__ Iout, const float *__restrict__ Id,
              const float *__restrict__ Wd, float *__restrict__ G, float *__restrict__ G1, int nk1,
              double *__restrict__ partials, unsigned *__restrict__ nonfinite, unsigned rows_id,
              const __grid_constant__ ModeVolume V)
{
    constexpr int R4 = M / 4, R1 = M & 1;
    constexpr bool GRAD = MODE != kProject;
    extern __shared__ __align__(16) float Qs[];            // [CP][kModeQ]
    __shared__ Dot2 red[kMarchThreads / 32];
    // the slots mapped last are marched first: they are the ones in L2
    const int slot = gridDim.y - 1 - blockIdx.y, s = order[slot];
    const int tj = blockIdx.x / tiles_k, tk = blockIdx.x - tj * tiles_k;
    const int r = threadIdx.x >> 1, h = threadIdx.x & 1;
    for (int t = threadIdx.x; t < CP * kModeQ; t += kMarchThreads) Qs[t] = Q[t];
    const float *vol = slots ? slots + slot * slot_floats : nullptr;
    const ProjGeom &P = geo[s];
    // neighbouring lanes take the rays along the detector axis that moves more
    // along v, the slots' rows
    const bool along_j = fabs(P.vj) > fabs(P.vk);
    const int j = tj * kMarchTJ + (along_j ? r % kMarchTJ : r / kMarchTK);
    const int k = tk * kMarchTK + (along_j ? r / kMarchTJ : r % kMarchTK);
    const bool valid = j < nj && k < nk;
    float ur, vr;
    ray_base<float>(P, j, k, ur, vr);
    const float up = (float)P.up, vp = (float)P.vp;
    const int Nu = P.Nu, Nv = P.Nv;
    float lo = 0.f, hi = (float)(P.Nm - 1);
    clip_planes<float>(ur, up, Nu, lo, hi);
    clip_planes<float>(vr, vp, Nv, lo, hi);
    int plo = valid ? max(0, (int)floorf(lo)) : 1;
    int phi = valid ? min(P.Nm - 1, (int)ceilf(hi)) : 0;
    if (vol == nullptr) phi = plo - 1;                   // a zero volume: nothing to march

    // Planes plo .. phi have taps from -3 to N + 2 (at most one plane on
    // either side of those with a tap inside, the transverse slopes at most
    // one), the extent of a slot with its border: no clamps.
    constexpr int B = kSlotBorder;
    const int n1 = P.copy ? nx : nz, e1 = slot_pitch4(n1), e2 = (ny + 2 * B) * e1;   // strides of y and the outer axis
    const int sm = P.m == 1 ? e1 : e2, su = P.m == 1 ? e2 : e1;
    const int f1 = slot_pitch1(n1), f2 = (ny + 2 * B) * f1, sm1 = P.m == 1 ? f1 : f2, su1 = P.m == 1 ? f2 : f1;
    float acc[M];
#pragma unroll
    for (int i = 0; i < M; ++i) acc[i] = 0.f;
    // index of tap column iv + h at (u, v) = (0, 0), plane 0, less the bits of
    // the rounded coordinates' exponent
    const unsigned base = (unsigned)(B * (e2 + e1) + kSlotLead + h) - (unsigned)kRoundBits * (unsigned)(su + 1);
    const unsigned base1 = (unsigned)(B * (f2 + f1) + kSlotLead + h) - (unsigned)kRoundBits * (unsigned)(su1 + 1);
    // Two batches of NB planes: one's taps travel while the other is summed.
    constexpr int NB = M <= 5 ? 2 : 1;
    struct Batch {
        float w0[NB], w1[NB], x0[NB][M], x1[NB][M];
    };
    auto load = [&](Batch &q, int p) {
#pragma unroll
        for (int t = 0; t < NB; ++t) {
            const int pt = min(p + t, phi);                // (never past the last plane)
            const float pf = (float)pt;
            // (rounded down, the sum with kRound holds the floor exactly: the taps
            // are k_forward's, those of weight zero included, whose voxel may hold
            // a NaN)
            const float u = fmaf(pf, up, ur), v = fmaf(pf, vp, vr);
            const float ub = __fadd_rd(u, kRound), vb = __fadd_rd(v, kRound);
            const float wu = u - (ub - kRound), wv = v - (vb - kRound);
            const int o = (int)((unsigned)(pt * sm) + __float_as_uint(ub) * (unsigned)su + __float_as_uint(vb) + base);
            const float wvh = p + t > phi ? 0.f : (h ? wv : 1.f - wv);
            q.w0[t] = (1.f - wu) * wvh;
            q.w1[t] = wu * wvh;
#pragma unroll
            for (int g = 0; g < R4; ++g) {
                const float4 ta = __ldg(reinterpret_cast<const float4 *>(vol + g * 4 * slot_vox) + o);
                const float4 tb = __ldg(reinterpret_cast<const float4 *>(vol + g * 4 * slot_vox) + o + su);
                q.x0[t][4 * g] = ta.x; q.x0[t][4 * g + 1] = ta.y; q.x0[t][4 * g + 2] = ta.z; q.x0[t][4 * g + 3] = ta.w;
                q.x1[t][4 * g] = tb.x; q.x1[t][4 * g + 1] = tb.y; q.x1[t][4 * g + 2] = tb.z; q.x1[t][4 * g + 3] = tb.w;
            }
            if constexpr (R1) {
                const int o1 = (int)((unsigned)(pt * sm1) + __float_as_uint(ub) * (unsigned)su1 + __float_as_uint(vb) + base1);
                q.x0[t][4 * R4] = __ldg(vol + R4 * 4 * slot_vox + o1);
                q.x1[t][4 * R4] = __ldg(vol + R4 * 4 * slot_vox + o1 + su1);
            }
        }
    };
    auto sum = [&](const Batch &q) {
#pragma unroll
        for (int t = 0; t < NB; ++t) {
#pragma unroll
            for (int i = 0; i + 1 < M; i += 2) fma2(acc[i], acc[i + 1], q.w0[t], q.x0[t][i], q.x0[t][i + 1]);
            if constexpr (R1) acc[M - 1] = fmaf(q.w0[t], q.x0[t][M - 1], acc[M - 1]);
#pragma unroll
            for (int i = 0; i + 1 < M; i += 2) fma2(acc[i], acc[i + 1], q.w1[t], q.x1[t][i], q.x1[t][i + 1]);
            if constexpr (R1) acc[M - 1] = fmaf(q.w1[t], q.x1[t][M - 1], acc[M - 1]);
        }
    };
    if (plo <= phi) {
        Batch qa, qb;
        load(qa, plo);
        for (int p = plo; p <= phi; p += 2 * NB) {
            load(qb, p + NB);
            sum(qa);
            load(qa, p + 2 * NB);
            sum(qb);
        }
    }
    const float step = (float)P.step;
#pragma unroll
    for (int i = 0; i < M; ++i) acc[i] = (acc[i] + __shfl_xor_sync(0xffffffffu, acc[i], 1)) * step;
    __syncthreads();   // Q staged

    // lane h takes the segments 4 h .. 4 h + 3 of every eight
    const long long pix = ((long long)s * nj + j) * nk + k;
    const bool vec4 = (C & 3) == 0;
    float gm[M], loss = 0.f;
#pragma unroll
    for (int i = 0; i < M; ++i) gm[i] = 0.f;
    for (int c0 = 4 * h; c0 < CP; c0 += 8) {
        float ih[4];
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            const float *q = Qs + (c0 + t) * kModeQ;
            ih[t] = 0.f;
#pragma unroll
            for (int i = 0; i < M; ++i) ih[t] = fmaf(q[i], acc[i], ih[t]);
        }
        if (!valid) continue;
        const long long o = pix * C + c0;
        if constexpr (!GRAD) {
            if (vec4) {
                *reinterpret_cast<float4 *>(Iout + o) = make_float4(ih[0], ih[1], ih[2], ih[3]);
            } else {
#pragma unroll
                for (int t = 0; t < 4; ++t)
                    if (c0 + t < C) Iout[o + t] = ih[t];
            }
        } else {
            float dI[4] = {0.f, 0.f, 0.f, 0.f}, dW[4] = {1.f, 1.f, 1.f, 1.f};
            if (vec4) {
                const float4 ti = __ldg(reinterpret_cast<const float4 *>(Id + o));
                dI[0] = ti.x; dI[1] = ti.y; dI[2] = ti.z; dI[3] = ti.w;
                if (Wd) {
                    const float4 b = __ldg(reinterpret_cast<const float4 *>(Wd + o));
                    dW[0] = b.x; dW[1] = b.y; dW[2] = b.z; dW[3] = b.w;
                }
            } else {
#pragma unroll
                for (int t = 0; t < 4; ++t)
                    if (c0 + t < C) {
                        dI[t] = __ldg(Id + o + t);
                        if (Wd) dW[t] = __ldg(Wd + o + t);
                    }
            }
#pragma unroll
            for (int t = 0; t < 4; ++t) {
                const bool live = c0 + t < C;
                const float rr = live ? ih[t] - dI[t] : 0.f, wr = live ? dW[t] * rr : 0.f;
                loss = fmaf(wr, rr, loss);
                const float *q = Qs + (c0 + t) * kModeQ;
#pragma unroll
                for (int i = 0; i < M; ++i) gm[i] = fmaf(q[i], wr, gm[i]);
            }
        }
    }
    if constexpr (!GRAD) {
        const bool again = valid && !rows_finite(acc);
        __syncwarp();
        if (again && h == 0) project_infinite(V, P, s, j, k, C, CP, Iout + pix * C);
    }
    if constexpr (GRAD) {
#pragma unroll
        for (int i = 0; i < M; ++i) gm[i] = 2.f * (gm[i] + __shfl_xor_sync(0xffffffffu, gm[i], 1));
        loss += __shfl_xor_sync(0xffffffffu, loss, 1);
        if (valid) {
            if (R4 == 1 ? h == 0 : true) {
                const int g = R4 == 1 ? 0 : h;
                *reinterpret_cast<float4 *>(G + pix * (4 * R4) + 4 * g) =
                    g ? make_float4(gm[M - R1 - 4], gm[M - R1 - 3], gm[M - R1 - 2], gm[M - R1 - 1])
                      : make_float4(gm[0], gm[1], gm[2], gm[3]);
            }
            if constexpr (R1)
                if (h == 1) G1[((long long)s * nj + j) * nk1 + k] = gm[M - 1];
        }
        if (valid && !rows_finite(gm)) *nonfinite = rows_id;
        const double tot = dot2_block_sum(Dot2{h == 0 && valid ? loss : 0.f, 0.f}, red);
        if (threadIdx.x == 0) partials[(long long)s * gridDim.x + blockIdx.x] = tot;
    }
}

// ------------------------------------------------------------ launchers

// Projections of a map CTA: as many as its tensor memory holds beside the A
// operand (a multiple of four, the projections a warp stores at a time).
static int map_group(int KP, int M) { return ((int)kMapCols - 2 * KP) / M / 4 * 4; }

template <typename S, int KP, int M>
static cudaError_t run_map(tt_handle *h, const int *order, int n, int copy)
{
    const int n_in = h->N[copy ? 0 : 2], n_out = h->N[copy ? 2 : 0];
    const long long ntiles = ((long long)(n_in + 7) / 8 * 8 * h->N[1] * n_out + 127) / 128;
    const int group = map_group(KP, M), groups = (n + group - 1) / group;
    const int N = (std::min(group, n) * M + 15) / 16 * 16;
    const size_t smem = (size_t)2 * KP * N * 4;
    const auto kern = k_map_modes<S, KP, M>;
    cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    const long long gx = std::min<long long>(ntiles, std::max(1, 2 * h->n_sm / groups));
    cudaEvent_t ev;
    prof_begin(h, TT_KSLOT_PACK, &ev);
    kern<<<dim3((unsigned)gx, groups), kMapThreads, smem, h->stream>>>(
        (const S *)h->cpad + (copy ? h->pad_vox * KP : 0), (const float2 *)h->FM, order, n, group, n_in, h->N[1], n_out,
        h->slots + (copy ? h->slots1 : 0), h->slot_floats, h->slot_vox, h->q_identity ? h->R : 1);
    const cudaError_t e = cudaGetLastError();
    prof_end(h, TT_KSLOT_PACK, ev);
    return e;
}

template <int M, int MODE>
static cudaError_t run_march(tt_handle *h, const int *order, int n, const float *slots, float *Iout, const float *I,
                             const float *W)
{
    const int tiles_k = (h->nk + kMarchTK - 1) / kMarchTK, tiles_j = (h->nj + kMarchTJ - 1) / kMarchTJ;
    const ModeOut mo = mode_out(h);
    cudaEvent_t ev;
    prof_begin(h, TT_KSLOT_FORWARD, &ev);
    k_march_modes<M, MODE><<<dim3(tiles_k * tiles_j, n), kMarchThreads, h->CP * kModeQ * 4, h->stream>>>(
        h->geo, order, slots, h->slot_floats, h->slot_vox, h->N[0], h->N[1], h->N[2], h->nj, h->nk, h->C, h->CP, tiles_k,
        mo.Q, Iout, I, W, (float *)h->G, mo.G1, mo.nk1, h->partials, mo.nonfinite, mo.rows_id,
        ModeVolume{(const char *)h->cpad + h->cpad_origin * h->KP * h->ssize(),
                   (const char *)h->cpad + (h->pad_vox + h->cpadx_origin) * h->KP * h->ssize(), (const float *)h->Bp,
                   h->prec, h->K, h->KP});
    const cudaError_t e = cudaGetLastError();
    prof_end(h, TT_KSLOT_FORWARD, ev);
    return e;
}

template <typename S, int KP, int M>
static cudaError_t run_chunk(tt_handle *h, int at, int n, int copy, float *Iout, const float *I, const float *W, bool grad)
{
    const int *order = h->order + at;
    const float *slots = h->zero_volume ? nullptr : h->slots + (copy ? h->slots1 : 0);
    if (slots) {
        const cudaError_t e = run_map<S, KP, M>(h, order, n, copy);
        if (e != cudaSuccess) return e;
    }
    return grad ? run_march<M, kGradModes>(h, order, n, slots, Iout, I, W)
                : run_march<M, kProject>(h, order, n, slots, Iout, I, W);
}

template <typename S, int KP>
static cudaError_t run_m(tt_handle *h, int at, int n, int copy, float *Iout, const float *I, const float *W, bool grad)
{
    switch (modes_m(h->R)) {
    case 4: return run_chunk<S, KP, 4>(h, at, n, copy, Iout, I, W, grad);
    case 5: return run_chunk<S, KP, 5>(h, at, n, copy, Iout, I, W, grad);
    case 8: return run_chunk<S, KP, 8>(h, at, n, copy, Iout, I, W, grad);
    default: return run_chunk<S, KP, 9>(h, at, n, copy, Iout, I, W, grad);
    }
}

long long mode_forward_ctas(const tt_handle *h)
{
    return (long long)((h->nk + kMarchTK - 1) / kMarchTK) * ((h->nj + kMarchTJ - 1) / kMarchTJ) * h->S;
}

// F rows for the map, [S][M][KP] (hi, lo), without order 0 (see k_map_modes).
__global__ void k_map_operand(const double *__restrict__ F, int S, int R, int K, int M, int KP, float2 *__restrict__ FM)
{
    const long long n = (long long)S * M * KP;
    for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < n;
         e += (long long)gridDim.x * blockDim.x) {
        const int k = (int)(e % KP), m = (int)(e / KP % M), s = (int)(e / ((long long)KP * M));
        float2 v = make_float2(0.f, 0.f);
        if (m < R && k > 0 && k < K) {
            const double f = F[((size_t)s * R + m) * K + k];
            uint32_t hi, lo;
            tf32_split((float)f, hi, lo);
            v.x = __uint_as_float(hi);
            v.y = __uint_as_float((__float_as_uint((float)(f - (double)v.x)) + 0x1000u) & 0xffffe000u);
        }
        FM[e] = v;
    }
}

// The projections that read copy 0 of the packed volume, then copy 1's.
static std::vector<int> projection_order(tt_handle *h)
{
    std::vector<int> order;
    for (int c = 0; c < 2; ++c) {
        h->order_begin[c] = (int)order.size();
        for (int s = 0; s < h->S; ++s)
            if (h->geo_host[s].copy == c) order.push_back(s);
    }
    return order;
}

// Detector pixels that the volume's shadow (its bounding box) covers.
static double shadow(const tt_handle *h, const ProjGeom &g)
{
    auto covered = [&](double at0, double u, double v, double p, int n) {
        double lo = at0, hi = at0;
        for (const double d : {u * (g.Nu - 1), v * (g.Nv - 1), p * (g.Nm - 1)}) (d < 0 ? lo : hi) += d;
        return std::max(0.0, std::min(n - 1.0, hi) - std::max(0.0, lo) + 1.0);
    };
    return covered(g.jc0, g.jU, g.jV, g.jP, h->nj) * covered(g.kc0, g.kU, g.kV, g.kP, h->nk);
}

double shadow_share(const tt_handle *h)
{
    double pixels = 0.0;
    for (const ProjGeom &g : h->geo_host) pixels += shadow(h, g);
    return pixels / (double)h->npix();
}

// Steps of rays through the volume: planes times covered pixels, over all
// projections.
static double ray_steps(const tt_handle *h)
{
    double steps = 0.0;
    for (const ProjGeom &g : h->geo_host) steps += shadow(h, g) * g.Nm;
    return steps;
}

// Sizes of the mode forward, and when it pays (l_max 6 and 8; at 4 the mapped
// volume, five values for fifteen, saves too little: 64^3 x 120 about 360 / 310
// us).  The map costs by voxels times projections (8.4e-6 to 1.1e-5 us each,
// whatever the detector), what the march of the mapped volume saves goes by the
// steps of rays (FP32: 1.9e-5 us each at l_max 6, 2.3e-5 at 8; 2-byte storage,
// whose direct march reads half the bytes: 0.7e-5 and 1.35e-5), and there are
// some 15 us of further launches; hence a floor and a share of the voxels for
// the steps.  Measured, whole projection in us, modes / direct march, 120
// projections unless said:
//   l_max 6  28^3 x 140 98 / 115; 64^3 on 64^2 pixels 558 / 840, on 44^2 451 / 481,
//            on 38^2 440 / 373, on 32^2 370 / 286, on 8^2 342 / 45; 128^3 on
//            128^2 3721 / 6183, on 89^2 3043 / 3711, on 76^2 2763 / 2715, on 16^2
//            2120 / 286; 32^3 on 96^2 172 / 271
//   l_max 8  28^3 x 140 108 / 127; 64^3 on 64^2 576 / 960, on 38^2 456 / 419; 128^3
//            on 128^2 3790 / 7400, on 76^2 2827 / 3360, on 64^2 2580 / 2334, on
//            16^2 2177 / 402
//   2 bytes  l_max 6: 64^3 549 / 402, 128^3 3655 / 2958: never; l_max 8: 28^3 x 160
//            125 / 110, 40^3 201 / 185, 64^3 568 / 649, 128^3 3777 / 5130, on 64^2
//            2522 / 1662; 32^3 on 96^2 179 / 241
void plan_mode_forward(tt_handle *h, size_t reserved)
{
    h->slot_floats = 0;
    const bool half = h->ssize() == 2;
    const double work = (double)h->nvox() * h->S;
    if (!h->R || h->KP < 32 || work < 3e6 || (half && h->KP < 48)) return;
    if (ray_steps(h) < (half ? 2e6 + 0.85 * work : 1e6 + (h->KP < 48 ? 0.43 : 0.33) * work)) return;
    h->order_host = projection_order(h);
    long long single = 0;
    for (int c = 0; c < 2; ++c) {
        const int in = h->N[c ? 0 : 2];
        const long long rows = (long long)(h->N[1] + 2 * kSlotBorder) * (h->N[c ? 2 : 0] + 2 * kSlotBorder);
        h->slot_vox = std::max(h->slot_vox, rows * slot_pitch4(in));
        single = std::max(single, rows * slot_pitch1(in) * h->R1);
    }
    h->slot_floats = (h->slot_vox * 4 * h->R4 + single + 63) / 64 * 64;
    // Slots for either copy's projections: two gigabytes, four where those hold
    // fewer than 24, and at most a sixteenth of the free memory, so that what
    // the caller and the solvers allocate later finds room; fewer than five (of
    // as many projections) are slower than the direct march.  Whole projections
    // in ms by gigabytes of slots 0.5 / 1 / 2 / 4, direct: 100^3, l_max 6, 180
    // projections (44 MB a slot) 3.37 / 3.09 / 2.86 / 2.77, 4.47; 128^3, l_max 8,
    // 240 (79 MB) 12.3 / 8.8 / 7.93 / 7.89, 13.9; 200^3, l_max 6, 60 (297 MB) 28.5 /
    // 13.4 / 8.9 / 7.4, 11.9; 256^3, l_max 8, 36 (602 MB) 40.8 / 40.8 / 18.3 / 13.2,
    // 21.6.
    size_t free_bytes = 0, total = 0;
    if (cudaMemGetInfo(&free_bytes, &total) != cudaSuccess) (void)cudaGetLastError();
    free_bytes -= std::min(free_bytes, reserved);
    const long long slot = 4 * h->slot_floats, gb = 1LL << 30;
    const long long bytes = std::min(std::min(4 * gb, std::max(2 * gb, 24 * slot)), (long long)(free_bytes / 16));
    const int most = std::max(h->order_begin[1], h->S - h->order_begin[1]);
    const int fit = (int)std::min<long long>(most, bytes / slot);
    if (fit < std::min(most, 5)) {
        h->slot_floats = 0;
        return;
    }
    const int parts = (most + fit - 1) / fit;
    h->chunk = (most + parts - 1) / parts;                 // (equal chunks need no more)
    // the copies' borders coincide in cubic volumes: one set of slots serves both
    h->slots1 = h->N[0] == h->N[2] || h->order_begin[1] == 0 || h->order_begin[1] == h->S ? 0 : h->chunk * h->slot_floats;
}

// Zeroes the slots' borders, which no map writes: border rows, and of the others
// the lead and what follows the whole groups of eight voxels.  One warp per row.
// (All of 2 GB by a memset: 0.4 ms of a handle's set-up.)
__global__ void __launch_bounds__(kThreads)
k_zero_borders(float *__restrict__ slots, long long nslots, long long slot_floats, long long slot_vox, int n_in, int ny,
               int n_out, int R4, int R1)
{
    constexpr int B = kSlotBorder;
    const int lane = threadIdx.x & 31, rows = (ny + 2 * B) * (n_out + 2 * B);
    const int p4 = slot_pitch4(n_in), p1 = slot_pitch1(n_in), end = kSlotLead + ((n_in + 7) & ~7);
    const long long n = nslots * rows;
    for (long long w = ((long long)blockIdx.x * kThreads + threadIdx.x) >> 5; w < n; w += (long long)gridDim.x * (kThreads / 32)) {
        const int row = (int)(w % rows), y = row % (ny + 2 * B) - B, o = row / (ny + 2 * B) - B;
        const bool inside = y >= 0 && y < ny && o >= 0 && o < n_out;
        float *slot = slots + w / rows * slot_floats;
        for (int g = 0; g < R4; ++g) {
            float4 *p = reinterpret_cast<float4 *>(slot) + g * slot_vox + (long long)row * p4;
            for (int i = lane; i < p4; i += 32)
                if (!inside || i < kSlotLead || i >= end) p[i] = make_float4(0.f, 0.f, 0.f, 0.f);
        }
        if (R1) {
            float *p = slot + R4 * 4 * slot_vox + (long long)row * p1;
            for (int i = lane; i < p1; i += 32)
                if (!inside || i < kSlotLead || i >= end) p[i] = 0.f;
        }
    }
}

cudaError_t setup_mode_forward(tt_handle *h, const double *F)
{
    if (!h->slots) return cudaSuccess;
    for (int copy = 0; copy < (h->slots1 ? 2 : 1); ++copy) {
        // (one set of slots serves both copies where their extents agree)
        const bool x_inner = h->slots1 ? copy : h->order_begin[1] == 0;
        k_zero_borders<<<8 * h->n_sm, kThreads, 0, h->stream>>>(
            h->slots + copy * h->slots1, h->chunk, h->slot_floats, h->slot_vox, h->N[x_inner ? 0 : 2], h->N[1],
            h->N[x_inner ? 2 : 0], h->R4, h->R1);
    }
    const int M = modes_m(h->R);
    k_map_operand<<<(unsigned)std::min<long long>(((long long)h->S * M * h->KP + 255) / 256, 8LL * h->n_sm), 256, 0,
                    h->stream>>>(F, h->S, h->R, h->K, M, h->KP, (float2 *)h->FM);
    return cudaGetLastError();
}

template <typename S>
cudaError_t launch_forward_modes(tt_handle *h, float *Iout, const float *I, const float *W, bool grad, int s0, int s1)
{
    cudaError_t e = cudaSuccess;
    for (int c = 0; c < 2; ++c) {
        const auto b = h->order_host.begin() + h->order_begin[c];
        const auto end = c == 0 ? h->order_host.begin() + h->order_begin[1] : h->order_host.end();
        const int i0 = (int)(std::lower_bound(b, end, s0) - h->order_host.begin());
        const int i1 = (int)(std::lower_bound(b, end, s1) - h->order_host.begin());
        const int parts = (i1 - i0 + h->chunk - 1) / h->chunk;
        for (int i = 0; i < parts && e == cudaSuccess; ++i) {
            const int a = i0 + (int)((long long)(i1 - i0) * i / parts);
            const int n = i0 + (int)((long long)(i1 - i0) * (i + 1) / parts) - a;
            if constexpr (sizeof(S) == 4)                  // (2-byte storage: l_max 8 only, see plan_mode_forward)
                e = h->KP == 32 ? run_m<S, 32>(h, a, n, c, Iout, I, W, grad) : run_m<S, 48>(h, a, n, c, Iout, I, W, grad);
            else
                e = run_m<S, 48>(h, a, n, c, Iout, I, W, grad);
        }
    }
    return e;
}
template cudaError_t launch_forward_modes<float>(tt_handle *, float *, const float *, const float *, bool, int, int);
template cudaError_t launch_forward_modes<__nv_bfloat16>(tt_handle *, float *, const float *, const float *, bool, int, int);
template cudaError_t launch_forward_modes<__half>(tt_handle *, float *, const float *, const float *, bool, int, int);

}  // namespace tt
