// tt_modes.cu -- set-up and launchers of the detector-mode projector
// (tt_modes.cuh).
#include <cmath>
#include <cstring>

#include <cuda.h>
#include <cudaTypedefs.h>

#include "tt_modes.cuh"

namespace tt {

// The two_theta = 0 circle is a great circle: even functions have even modes
// only.
static int mode_step(const tt_handle *h) { return h->two_theta == 0.0 ? 2 : 1; }

// Detector coordinate range of a block of 8 x 4 x 8 voxels relative to its
// corner: the sum of the slopes' negative, positive parts.
static void block_range(const double *c, double &lo, double &hi)
{
    const double ext[3] = {7.0, 3.0, 7.0};
    lo = hi = 0.0;
    for (int t = 0; t < 3; ++t) (c[1 + t] < 0 ? lo : hi) += ext[t] * c[1 + t];
}

// Tensor map of a plane of row values [S][nj][pitch * w floats], box bj x bk
// pixels of w floats each.
static bool encode_rows(const tt_handle *h, const void *base, int w, int pitch, TmaDesc *out)
{
    const auto enc = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(driver_tensor_map_encoder());
    const cuuint64_t dims[3] = {(cuuint64_t)w * h->nk, (cuuint64_t)h->nj, (cuuint64_t)h->S};
    const cuuint64_t strides[2] = {(cuuint64_t)w * pitch * 4, (cuuint64_t)w * pitch * 4 * h->nj};
    const cuuint32_t box[3] = {(cuuint32_t)(w * h->box_k), (cuuint32_t)h->box_j, 1}, elem[3] = {1, 1, 1};
    CUtensorMap m;
    if (enc(&m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, const_cast<void *>(base), dims, strides, box, elem,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
        return false;
    std::memcpy(out, &m, sizeof(m));
    return true;
}

// Blocks of 8 x 4 x 8 voxels.
static long long mode_blocks(const tt_handle *h)
{
    return (long long)((h->N[0] + 7) / 8) * ((h->N[1] + 3) / 4) * ((h->N[2] + 7) / 8);
}

static size_t modes_smem(const tt_handle *h)
{
    const int M = modes_m(h->R), UP = modes_up(M);
    const uint32_t px = (uint32_t)(h->box_j * h->box_k);
    const size_t boxes = mode_align(px * 16 * h->R4) + (h->R1 ? mode_align(px * 4) : 0);
    const size_t ring = kModeStages * (UP * boxes + 2 * (size_t)modes_ku(M) * modes_n(h->K) * 4);
    return std::max(ring, (size_t)kModeVox * h->K * 4) + 128;   // (the sums at the end)
}

// Whether the adjoint in modes is the faster one.  It has a start and an end (box
// origins, tensor memory, sums: 4 us a block at l_max 2, more above) that few
// projections do not pay for, and its blocks come in waves of those resident;
// the channel kernel's blocks are 32 voxels long in z at l_max 2.  Measured,
// channels / modes in us, an adjoint by itself:
//   l_max 8, 4 projections: 64^3 60.0 / 61.9, 100^3 190 / 197; 8: 99 / 81, 334 / 261
//   l_max 6, 8: 64^3 64.6 / 68.4, 100^3 208 / 220; 12: 84.5 / 78.6, 275 / 257; 1
//     projection 56.6 / 127 at 100^3
//   l_max 4, 4: 64^3 25.1 / 27.3, 100^3 64 / 78; 8: 39.9 / 35.5, 118 / 112
//   fewer blocks than SMs, whole evaluations, 18: 16^3 l_max 4 35.0 / 34.3, 6 36.1 /
//     37.1, 8 41.7 / 43.5; 30: 45.6 / 33.9, 47.4 / 34.0, 53.7 / 39.4
//   l_max 2, less than a wave, 12: 16^3 15.7 / 17.0, 40^3 21.0 / 21.1; 20: 40^3 27.2 /
//     25.1, but evaluations, whose forward does more in modes, 48.3 / 49.0, 24 49.0 / 50.3,
//     28 57.7 / 57.0, FP16 36 x 32 x 33 28 46.2 / 47.4, 32 51.1 / 50.1; more than a wave:
//     56^3 28 56.1 / 60.1, 36 67.9 / 66.3; 78 x 66 x 83 36 129.7 / 131.8, 44 157.9 /
//     156.6; 128^3 28 406.7 / 408.4, 44 603 / 593; z padded by 28%: 100^3 12 119 / 116, 20
//     182 / 166 (but 52^3, little more than a wave, 24: 45 / 51); by 22%: 110 x 100 x 105,
//     evaluations, 20 375 / 375, page-locked buffers 647 / 708
//   l_max 2, five modes (two_theta): 64^3 60 121 / 130, 200 378 / 391; 128^3 120 1586 /
//     1680; 48^3 60 75 / 65; 100^3 40 345 / 328
//   l_max 4, nine modes: 24^3 60 58 / 31, 40^3 60 72 / 68, 48^3 60 94 / 99, 64^3 24 86 / 93,
//     100^3 120 1376 / 1384, 128^3 120 2736 / 2628
//   l_max 4, 2-byte storage, whose forward pays more for the modes' epilogue, whole
//     evaluations: 30 x 28 x 31 18 44.6 / 46.0, 28 47.7 / 47.6, 35 56.9 / 52.2; 40 x 44 x 40
//     18 58.1 / 60.2, 24 63.8 / 65.9, 28 69.9 / 67.9; 50 x 52 x 48 20 83.7 / 78.5
static bool modes_pay(const tt_handle *h, int R)
{
    const long long blocks = mode_blocks(h), wave = (long long)h->n_sm * mode_ctas(16);
    const bool z_padded = 4LL * ((h->N[2] + 31) / 32 * 32) > 5LL * h->N[2];
    if (h->L == 2) {
        if (blocks <= wave) return h->S >= 30;
        if (z_padded && blocks > 2 * wave) return h->S >= (R > 4 ? 40 : 16);
        return R <= 4 && h->S >= 40;
    }
    if (h->L == 4 && R > 8 && 2 * blocks > wave) return false;
    if (h->L == 4 && h->ssize() == 2 && blocks <= 2 * h->n_sm) return h->S >= 28;
    if (blocks <= h->n_sm) return h->S >= (h->L == 4 ? 18 : 20);
    return h->S >= (h->L == 4 ? 8 : h->L == 6 ? 9 : 5);
}

// The handle works in modes when there are at most kMaxModes of them, the band
// limit is 2 .. 8, they pay, and every projection's box -- the rays of a block lie
// within (hj, hk) of its voxels' centres, plus the rounding margin and up to
// three pixels from aligning the box to four -- fits the tensor copies (256
// floats wide) and, kModeStages deep, the shared memory of two CTAs per SM.
// (Pixels much finer than voxels put too many rays around a block; the
// channel kernels take those.)  Coordinates stay below 2^22 in magnitude for
// volumes and detectors of at most 2^14, which the rounding by kRound needs.
void plan_modes(tt_handle *h)
{
    h->R = 0;
    if (h->prec == TT_F64 || h->L < 2 || h->L > 8 || !driver_tensor_map_encoder()) return;
    const int limit = 1 << 14;
    if (h->N[0] > limit || h->N[1] > limit || h->N[2] > limit || h->nj > limit || h->nk > limit) return;
    const int R = std::min(h->two_theta == 0.0 ? h->L + 1 : 2 * h->L + 1, h->C);
    if (R > kMaxModes || !modes_pay(h, R)) return;
    int bj = 1, bk = 4;
    std::vector<AdjConst> adj(h->S);
    h->org_host.resize(h->S);
    for (int s = 0; s < h->S; ++s) {
        const ProjGeom &g = h->geo_host[s];
        const AdjConst &c = adj[s] = adj_const(g);
        double jl, jh, kl, kh;
        block_range(c.jc, jl, jh);
        block_range(c.kc, kl, kh);
        const double wj = jh - jl + 2.0 * g.hj + 0.04, wk = kh - kl + 2.0 * g.hk + 0.04;
        if (!(wj < 200.0) || !(wk < 200.0)) return;
        ModeOrigin &o = h->org_host[s];
        for (int t = 0; t < 4; ++t) {
            o.j[t] = c.jc[t];
            o.k[t] = c.kc[t];
        }
        o.jlo = jl - g.hj - 0.02;
        o.klo = kl - g.hk - 0.02;
        o.outer_j = c.outer_j ? 1 : 0;
        // a column whose first ray is in the box is read to its end
        bj = std::max(bj, (int)std::ceil(wj) + 1 + (c.outer_j ? 0 : c.ni - 1));
        bk = std::max(bk, ((int)std::ceil(wk) + 1 + (c.outer_j ? c.ni - 1 : 0) + 3 + 3) / 4 * 4);
    }
    h->R = R;
    h->R4 = modes_r4(R);
    h->R1 = modes_r1(R);
    h->q_identity = R == h->C;
    h->nk1 = (h->nk + 3) / 4 * 4;
    h->box_j = bj;
    h->box_k = bk;
    // Rows of one quad: a pitch of 4 mod 8 pixels puts neighbouring rows of the
    // box half the banks apart (where the wider box fits).
    if (h->R4 == 1 && bk % 8 == 0) {
        h->box_k = bk + 4;
        if ((bk + 4) * 4 <= 256 && (long long)modes_smem(h) <= kModeMaxSmem) bk += 4;
        h->box_k = bk;
    }
    TmaDesc probe;
    if (bk * 4 * h->R4 > 256 || bj > 256 || (long long)modes_smem(h) > kModeMaxSmem ||
        !encode_rows(h, (const void *)4096, 4 * h->R4, h->nk, &probe) ||
        !encode_rows(h, (const void *)4096, 1, h->nk1, &probe)) {
        h->R = 0;
        return;
    }
    h->mode_params.assign((h->S + ModeParams::kMax - 1) / ModeParams::kMax, ModeParams());
    for (int s = 0; s < h->S; ++s) {
        const AdjConst &c = adj[s];
        ModeProj &p = h->mode_params[s / ModeParams::kMax].p[s % ModeParams::kMax];
        for (int t = 0; t < 3; ++t) {
            p.o[t] = (float)c.oc[1 + t];
            p.i[t] = (float)c.ic[1 + t];
        }
        p.uo = (float)c.uo; p.ui = (float)c.ui; p.vo = (float)c.vo; p.vi = (float)c.vi;
        p.oh = (float)(0.5 - c.ho);
        p.au = (float)(c.au + 0.5); p.lu = (float)c.lu;
        p.av = (float)(c.av + 0.5); p.lv = (float)c.lv;
        p.so = c.outer_j ? bk : 1;
        p.si = c.outer_j ? 1 : bk;
        p.k0 = (int)(0u - (unsigned)kRoundBits * (unsigned)(p.so + p.si));
        p.lim = bj * bk - 1 - (c.ni - 1) * p.si;
        p.shape = (c.no <= 3 && c.ni <= 3) ? 16 * c.no + c.ni : 0;
        p.order = c.no | (c.ni << 8);
    }
}

// F[s][m][i]: Fourier coefficients of Y_i along the detector circle, mode m
// (0: constant; 2t - 1, 2t: cos, sin of t * step times phi), by the 32-point
// rule on the whole circle (exact: two modes of at most 8 each).  The 32 points'
// cosines and sines serve every mode (FP64 is slow here: evaluated for each
// term they were most of a handle's set-up, 160 us at l_max 4).
constexpr int kMatrixThreads = 128;
__global__ void __launch_bounds__(kMatrixThreads)
k_mode_matrix(const double *__restrict__ frames, double cth, double sth, int L, int K, int R, int step,
              double *__restrict__ F)
{
    extern __shared__ double ysh[];   // [32][K]
    __shared__ double cs[32], sn[32];
    const int s = blockIdx.x, t = threadIdx.x;
    if (t < 32) {
        const double *fr = frames + 9 * s;
        double sp, cp;
        sincospi(t / 16.0, &sp, &cp);
        cs[t] = cp;
        sn[t] = sp;
        double q[3];
        for (int r = 0; r < 3; ++r) q[r] = cth * (cp * fr[3 + r] + sp * fr[6 + r]) - sth * fr[r];
        sh_even<double>(L, q[0], q[1], q[2], ysh + t * K, 1);
    }
    __syncthreads();
    for (int e = t; e < R * K; e += kMatrixThreads) {
        const int m = e / K, i = e - m * K, f = (m + 1) / 2 * step;
        const double *wave = (m & 1) ? cs : sn;
        double acc = 0.0;
        for (int n = 0; n < 32; ++n) acc = fma(ysh[n * K + i], m == 0 ? 1.0 : wave[(n * f) & 31], acc);
        F[((size_t)s * R + m) * K + i] = acc * (m == 0 ? 1.0 : 2.0) / 32.0;
    }
}

// The adjoint's B operands: per unit of UP projections two KU x N matrices,
// for D_lo and D_hi, in K-major core-matrix tiles (8 rows x 16 bytes).  Column
// k of the unit is slot k % (2 M) of projection k / (2 M): the slots hold the
// M modes' t_hi, then t_lo; D_lo takes F_lo against t_hi and F_hi against
// t_lo, D_hi F_hi against t_hi.  The projection's step length is folded in.
__global__ void k_mode_operand(const double *__restrict__ F, const ProjGeom *__restrict__ geo, int S, int R, int K,
                               int M, int UP, int KU, int N, float *__restrict__ FB, long long n)
{
    for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < n;
         e += (long long)gridDim.x * blockDim.x) {
        const int k4 = (int)(e & 3), nn = (int)((e >> 2) & 7);
        long long r = e >> 5;
        const int nb = (int)(r % (N / 8));
        r /= N / 8;
        const int kc = (int)(r % (KU / 4));
        r /= KU / 4;
        const bool dhi = r & 1;
        const int u = (int)(r >> 1), k = 4 * kc + k4, i = 8 * nb + nn, q = k / (2 * M), slot = k - q * 2 * M;
        const int s = u * UP + q, m = slot % M;
        const bool tlo = slot >= M;
        float v = 0.f;
        if (q < UP && s < S && m < R && i < K && !(dhi && tlo)) {
            const double f = F[((size_t)s * R + m) * K + i] * geo[s].step;
            uint32_t hi, lo;
            tf32_split((float)f, hi, lo);
            const float rest = (float)(f - (double)__uint_as_float(hi));
            v = (dhi || tlo) ? __uint_as_float(hi)
                             : __uint_as_float((__float_as_uint(rest) + 0x1000u) & 0xffffe000u);
        }
        FB[e] = v;
    }
}

// What the host fills comes first and travels in one copy: mode_org, Qm, order,
// nonfinite (0: rows_id starts at 1); then FB, F64, FM.
size_t place_modes(tt_handle *h, char *base)
{
    size_t at = 0;
    auto place = [&](size_t bytes) {
        const size_t p = at;
        at += (bytes + 255) / 256 * 256;
        return p;
    };
    const size_t org = place(sizeof(ModeOrigin) * h->S), q = place(sizeof(float) * h->CP * kModeQ);
    const size_t ord = place(sizeof(int) * h->S), flag = place(sizeof(unsigned)), host = at;
    const size_t fb = place(sizeof(float) * mode_operand_floats(h));
    const size_t f64 = place(h->q_identity ? 0 : sizeof(double) * h->S * h->R * h->K);
    const size_t fm = place(h->slot_floats ? sizeof(float) * 2 * h->S * modes_m(h->R) * h->KP : 0);
    if (base) {
        h->mode_mem = base;
        h->mode_org = (ModeOrigin *)(base + org);
        h->Qm = (float *)(base + q);
        h->order = (int *)(base + ord);
        h->nonfinite = (unsigned *)(base + flag);
        h->FB = (float *)(base + fb);
        h->F64 = (double *)(base + f64);
        h->FM = base + fm;
        h->mode_host_bytes = host;
    }
    return at;
}

static cudaError_t form_modes(tt_handle *h, const double *frames, const double *node, const double *weight)
{
    const int R = h->R, step = mode_step(h);
    const char *base = (const char *)h->mode_mem;
    std::vector<char> host(h->mode_host_bytes, 0);
    std::memcpy(host.data() + ((char *)h->mode_org - base), h->org_host.data(), sizeof(ModeOrigin) * h->S);
    if (h->slot_floats)
        std::memcpy(host.data() + ((char *)h->order - base), h->order_host.data(), sizeof(int) * h->S);
    // Segment means of the modes by the nodes that B is formed with: B = Q F
    // holds for them at any segment width, beyond the few turns the rule is
    // exact on too.
    float *Q = (float *)(host.data() + ((char *)h->Qm - base));
    for (int c = 0; c < h->C; ++c)
        for (int m = 0; m < R; ++m) {
            double v = 0.0;
            if (h->q_identity) {
                v = c == m ? 1.0 : 0.0;
            } else if (m == 0) {
                v = 1.0;
            } else {
                const double f = (m + 1) / 2 * step, half = 0.5 * (h->seg1[c] - h->seg0[c]);
                const double mid = 0.5 * (h->seg1[c] + h->seg0[c]);
                for (int n = 0; n < kQuadNodes; ++n) {
                    const double a = f * (mid + half * node[n]);
                    v += 0.5 * weight[n] * ((m & 1) ? std::cos(a) : std::sin(a));
                }
            }
            Q[(size_t)c * kModeQ + m] = (float)v;
        }
    cudaError_t e = cudaMemcpyAsync(h->mode_mem, host.data(), host.size(), cudaMemcpyHostToDevice, h->stream);
    if (e != cudaSuccess) return e;
    cudaEvent_t ev;
    prof_begin(h, TT_KSLOT_BASIS, &ev);
    const double *F = h->B64;
    if (!h->q_identity) {
        const double th = 0.5 * h->two_theta;
        k_mode_matrix<<<h->S, kMatrixThreads, 32 * h->K * sizeof(double), h->stream>>>(
            frames, std::cos(th), std::sin(th), h->L, h->K, R, step, h->F64);
        F = h->F64;
    }
    const int M = modes_m(R), UP = modes_up(M), N = modes_n(h->K);
    const long long n = mode_operand_floats(h);
    k_mode_operand<<<(unsigned)std::min<long long>((n + 255) / 256, 8LL * h->n_sm), 256, 0, h->stream>>>(
        F, h->geo, h->S, R, h->K, M, UP, modes_ku(M), N, h->FB, n);
    e = cudaGetLastError();
    prof_end(h, TT_KSLOT_BASIS, ev);
    return e == cudaSuccess ? setup_mode_forward(h, F) : e;
}

// CTAs that share a block of voxels (1, 2, 4 or 8, three units each at least):
// the fewest waves of `slots` resident CTAs, a wave of s-fold split blocks
// lasting 1/s, each doubling counted as 20% for its sums and ramps; beyond a wave
// as it is, only while each keeps 20 projections, which their ramps need.  Over
// 156 sizes (12^3 to 72^3, l_max 2 to 8, 30 to 120 projections) the choice is
// within 3% of the best of the four: 20^3, l_max 4, 60: 60 -> 23 us with 8; 28^3,
// l_max 2, 60: 46 -> 30 with 4; 55 x 65 x 55, l_max 4, 247 (833 blocks on 608 slots):
// 482 -> 434 with 2; 64^3, 120 (1024 on 608) stays whole: 280 / 295 / 312; 48^3, l_max
// 8, 30 (432 on 304) too: 80 / 98 / 133.
static int mode_split(int blocks, int units, int projections, int slots)
{
    int best = 1;
    double least = 1e30, cost = 1.0;
    for (int s = 1; s <= 8 && (s == 1 || (units / s >= 3 && (blocks <= slots || projections / s >= 20))); s *= 2, cost *= 1.2) {
        const double t = cost * (((long long)blocks * s + slots - 1) / slots) / s;
        if (t < 0.999 * least) {
            least = t;
            best = s;
        }
    }
    return best;
}

template <int N, int R4, int R1>
static cudaError_t adjoint_modes_run(tt_handle *h, const float *rows, float *g, bool reduce_loss, const float *data)
{
    constexpr int M = 4 * R4 + R1, UP = modes_up(M), KU = modes_ku(M);
    const int tx = (h->N[0] + 7) / 8, ty = (h->N[1] + 3) / 4, tz = (h->N[2] + 7) / 8;
    TmaDesc tm4 = h->rows_map;
    const TmaDesc &tm1 = R1 ? h->single_map : h->rows_map;
    if (rows != (const float *)h->G && !encode_rows(h, rows, 4 * R4, h->nk, &tm4)) return cudaErrorInvalidValue;
    const auto kern = k_adjoint_modes<N, R4, R1>;
    const size_t smem = modes_smem(h);
    cudaError_t e = cudaSuccess;
    const int nchunk = (int)h->mode_params.size();
    for (int ci = 0; ci < nchunk && e == cudaSuccess; ++ci) {
        const int s0 = ci * ModeParams::kMax, ns = std::min(ModeParams::kMax, h->S - s0);
        const bool last = ci == nchunk - 1;
        static_assert(ModeParams::kMax % UP == 0, "launches start on a unit");
        const int blocks = tx * ty * tz, split = mode_split(blocks, (ns + UP - 1) / UP, ns, h->n_sm * mode_ctas(N));
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)blocks, (unsigned)split);
        cfg.blockDim = dim3(kModeThreads);
        cfg.dynamicSmemBytes = smem;
        cfg.stream = h->stream;
        cudaLaunchAttribute cluster;
        cluster.id = cudaLaunchAttributeClusterDimension;
        cluster.val.clusterDim = {1, (unsigned)split, 1};
        cfg.attrs = &cluster;
        cfg.numAttrs = split > 1 ? 1 : 0;
        cudaEvent_t ev;
        prof_begin(h, TT_KSLOT_ADJOINT, &ev);
        e = cudaLaunchKernelEx(
            &cfg, kern, h->mode_params[ci], tm4, tm1, ns, s0, (const ModeOrigin *)h->mode_org + s0, (const float *)h->FB + (size_t)(s0 / UP) * 2 * KU * N, h->box_j,
            h->box_k, h->N[0], h->N[1], h->N[2], ty, tz, (float *)h->gpad, h->KP, ci > 0 ? 1 : 0,
            last ? g : (float *)nullptr, h->K, (const double *)h->partials, h->n_fwd_ctas,
            (reduce_loss && ci == 0) ? h->loss_dev : (double *)nullptr,
            (reduce_loss && ci == 0 && h->loss_publish) ? h->loss_slot_dev : (LossSlot *)nullptr, h->loss_publish,
            (const unsigned *)h->nonfinite, h->rows_id,
            ModeData{last ? data : nullptr, h->geo, (const float *)h->Bp, h->S, h->nj, h->nk, h->C, h->CP});
        (void)cudaGetLastError();
        prof_end(h, TT_KSLOT_ADJOINT, ev);
    }
    return e;
}

// f<N, R4, R1>() of the handle's layout.
template <typename F>
static cudaError_t with_layout(const tt_handle *h, F f)
{
    auto rows = [&]<int N>() {
        if (h->R4 == 1) return h->R1 ? f.template operator()<N, 1, 1>() : f.template operator()<N, 1, 0>();
        return h->R1 ? f.template operator()<N, 2, 1>() : f.template operator()<N, 2, 0>();
    };
    switch (modes_n(h->K)) {
    case 16: return rows.template operator()<16>();
    case 32: return rows.template operator()<32>();
    case 48: return rows.template operator()<48>();
    default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_adjoint_modes(tt_handle *h, const float *rows, float *g, bool reduce_loss, const float *data)
{
    return with_layout(h, [&]<int N, int R4, int R1>() { return adjoint_modes_run<N, R4, R1>(h, rows, g, reduce_loss, data); });
}

// What a launch of the adjoint needs of the driver, once per handle: the maps of
// the handle's own rows, and leave for the kernel's shared memory (the most that
// any handle takes, so that handles do not narrow it for each other).
static cudaError_t ready_adjoint(tt_handle *h)
{
    if (!encode_rows(h, h->G, 4 * h->R4, h->nk, &h->rows_map)) return cudaErrorInvalidValue;
    if (h->R1 && !encode_rows(h, mode_out(h).G1, 1, h->nk1, &h->single_map)) return cudaErrorInvalidValue;
    return with_layout(h, [&]<int N, int R4, int R1>() {
        return cudaFuncSetAttribute(k_adjoint_modes<N, R4, R1>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kModeMaxSmem);
    });
}

cudaError_t setup_modes(tt_handle *h, const double *frames, const double *node, const double *weight)
{
    if (!h->R) return cudaSuccess;
    const cudaError_t e = ready_adjoint(h);
    return e == cudaSuccess ? form_modes(h, frames, node, weight) : e;
}

// Rows that are their caller's own (the modes are the segments): are they finite?
__global__ void __launch_bounds__(kThreads)
k_check_rows(const float4 *__restrict__ rows, long long n, unsigned *__restrict__ nonfinite, unsigned rows_id)
{
    bool ok = true;
    const long long stride = (long long)gridDim.x * kThreads;
    for (long long i = (long long)blockIdx.x * kThreads + threadIdx.x; i < n; i += 4 * stride) {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            if (i + k * stride >= n) break;
            const float4 v = __ldg(rows + i + k * stride);
            const float w[4] = {v.x, v.y, v.z, v.w};
            ok = ok && rows_finite(w);
        }
    }
    if (!ok) *nonfinite = rows_id;
}

cudaError_t launch_check_rows(tt_handle *h, const float *rows)
{
    const long long n = h->npix() * h->R4;
    ++h->rows_id;
    cudaEvent_t ev;
    prof_begin(h, TT_KSLOT_BACKCONTRACT, &ev);
    k_check_rows<<<(unsigned)std::min<long long>((n + 4 * kThreads - 1) / (4 * kThreads), 8LL * h->n_sm), kThreads, 0,
                   h->stream>>>(reinterpret_cast<const float4 *>(rows), n, h->nonfinite, h->rows_id);
    const cudaError_t e = cudaGetLastError();
    prof_end(h, TT_KSLOT_BACKCONTRACT, ev);
    return e;
}

cudaError_t launch_backcontract_modes(tt_handle *h, const float *R)
{
    const long long npix = h->npix();
    const unsigned blocks = (unsigned)((npix + kThreads - 1) / kThreads);
    float *G4 = (float *)h->G, *G1 = mode_out(h).G1;
    ++h->rows_id;
    cudaEvent_t ev;
    prof_begin(h, TT_KSLOT_BACKCONTRACT, &ev);
    if (h->R4 == 1 && !h->R1) k_backcontract_modes<1, 0><<<blocks, kThreads, 0, h->stream>>>(h->Qm, R, G4, G1, npix, h->nk, h->nk1, h->C, h->nonfinite, h->rows_id);
    else if (h->R4 == 1) k_backcontract_modes<1, 1><<<blocks, kThreads, 0, h->stream>>>(h->Qm, R, G4, G1, npix, h->nk, h->nk1, h->C, h->nonfinite, h->rows_id);
    else if (!h->R1) k_backcontract_modes<2, 0><<<blocks, kThreads, 0, h->stream>>>(h->Qm, R, G4, G1, npix, h->nk, h->nk1, h->C, h->nonfinite, h->rows_id);
    else k_backcontract_modes<2, 1><<<blocks, kThreads, 0, h->stream>>>(h->Qm, R, G4, G1, npix, h->nk, h->nk1, h->C, h->nonfinite, h->rows_id);
    cudaError_t e = cudaGetLastError();
    prof_end(h, TT_KSLOT_BACKCONTRACT, ev);
    return e;
}

}  // namespace tt
