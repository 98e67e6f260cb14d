// tt_internal.cuh -- shared declarations of libtt (handle, per-projection
// ray constants, kernel launchers).  Host code is C++17, device code sm_103a.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>
#include <deque>
#include <string>
#include <vector>

#include "../../include/tt.h"

namespace tt {

// Largest band limit with compiled kernels and its coefficient count.
constexpr int kMaxEll = 12;
constexpr int kMaxSeg = 64;
constexpr int kQuadNodes = 32;      // Gauss-Legendre nodes per detector segment
constexpr int kThreads = 256;       // threads per CTA of the adjoint and the other projector kernels
// Threads of a forward CTA and the ray tile it marches: fwd_tk(LG) rays along
// k (fastest) times fwd_tj(LG) along j, lane_group(K) lanes per ray (8 x 8
// rays at K = 15; 512- and 1024-thread tiles of 16 x 8 and 16 x 16 rays were
// measured 5% and 20% slower at 64^3).
constexpr int kFwdThreads = 256;
__host__ __device__ constexpr int fwd_rays(int LG) { return kFwdThreads / LG; }
__host__ __device__ constexpr int fwd_tk(int LG) { return fwd_rays(LG) >= 256 ? 16 : 8; }
__host__ __device__ constexpr int fwd_tj(int LG) { return fwd_rays(LG) / fwd_tk(LG); }

// Staged forward march (FP32 storage, 16 padded channels): a CTA of eight
// consumer warps and one copy warp marches a tile of kStTJ x kStTK rays with
// its taps read from a ring of shared-memory stages, one plane's box of
// padded-volume voxels per stage, moved by one tensor copy.  The ring holds
// kStRing boxes of the largest size over the projections; a projection with
// smaller boxes runs as many stages as fit, up to kStMaxDepth.  kStEps
// (voxels) widens the box against the rounding of the ray coordinates.
constexpr int kStTJ = 8, kStTK = 16, kStRing = 3, kStMaxDepth = 8;
constexpr int kStConsumers = 256, kStThreads = kStConsumers + 32;
constexpr float kStEps = 1.0f / 64;
constexpr long long kStMaxSmem = 200 * 1024;   // dynamic shared memory the ring may take (one CTA per SM)
constexpr int kStMaxRv = 32;                   // box width along v: 8 x 16 B words per voxel, at most 256 words

// An opaque tensor-map object (the driver's 128-byte, 64-byte aligned
// descriptor of a tiled tensor copy), kept in device memory per projection.
struct alignas(64) TmaDesc {
    unsigned char bytes[128];
};
// Forward kernels a handle can run (tt_set_forward_kernel).
enum { kFwdAuto = 0, kFwdL1 = 1, kFwdStaged = 2 };

// Lane-group width (lanes that share one ray or one voxel, each holding
// KP/LG channels) and padded channel count for a band limit.
__host__ __device__ constexpr int lane_group(int K) { return K <= 4 ? 1 : (K <= 8 ? 2 : 4); }
__host__ __device__ constexpr int padded_k(int K) {
    return ((K + 4 * lane_group(K) - 1) / (4 * lane_group(K))) * (4 * lane_group(K));
}
__host__ __device__ constexpr int num_coeffs(int L) { return (L + 1) * (L + 2) / 2; }
// Voxels a lane group of the adjoint owns: all LG while a lane's accumulators
// (V * KP / LG) fit in 16 registers' worth of channels, else as many as keep
// them within 24 (one for the largest K).
// Lane groups of an adjoint warp along z, the rest side by side in x: eight
// (a warp covers 8 z x 32 / (8 LG) x-columns of V voxels each), all 32 for
// one-lane groups (measured 3% faster for those than 8 z x 4 x).
__host__ __device__ constexpr int adjoint_gz(int LG) { return LG == 1 ? 32 : (32 / LG < 8 ? 32 / LG : 8); }
__host__ __device__ constexpr int adjoint_voxels(int KP, int LG)
{
    return KP / LG <= 4 ? LG : ((24 / (KP / LG)) < 1 ? 1 : ((24 / (KP / LG)) > LG ? LG : 24 / (KP / LG)));
}

// Per-projection constants of the Joseph discretisation, in voxel-index
// units (computed on the host in FP64 from Eq. real_space_geom).
//   plane p (index along the main axis m), ray (j,k):
//     u(j,k,p) = u0 + j*uj + k*uk + p*up   (continuous index along axis u)
//     v(j,k,p) = v0 + j*vj + k*vk + p*vp   (continuous index along axis v)
//   adjoint: the detector point whose ray crosses plane p at voxel (U,V) is
//     jc = jc0 + jU*U + jV*V + jP*p,  kc = kc0 + kU*U + kV*V + kP*p,
//   and every ray that has (U,V) as a bilinear tap lies in
//     |j - jc| < hj, |k - kc| < hk   (the bounding box of the parallelogram
//   |du| < 1, |dv| < 1 in detector coordinates).
struct ProjGeom {
    double u0, uj, uk, up;
    double v0, vj, vk, vp;
    double step;              // a / |p_s,m|
    double jc0, jU, jV, jP;
    double kc0, kU, kV, kP;
    double hj, hk;            // half extents in j and k of the rays around a voxel (|du|, |dv| < 1)
    int m, u, v;              // main and transverse axes (0=x, 1=y, 2=z)
    int Nm, Nu, Nv;
    int sm, su, sv;           // strides of the axes in the padded volume copy the projection reads
    int copy;                 // 0: cpad (z innermost), 1: the x-innermost copy; sv == 1 in both
    // Staged forward: the box of one plane is st_ru rows (along u) of st_rv
    // voxels (along v); st_umid: u is the middle axis (y) of the volume copy,
    // else its outer axis.
    int st_ru, st_rv, st_umid;
};

// Per-projection constants of the adjoint gather in the element type.  The
// candidate rays of a voxel are enumerated over an outer detector axis o and
// an inner axis i ((o, i) = (k, j), or (j, k) when bit 16 of order is set):
//   oc = oc[0] + oc[1] x + oc[2] y + oc[3] z   continuous outer coordinate of
//                                              the voxel centre (likewise ic)
//   du(o,i) = bu(x,y,z) + o uo + i ui,  dv(o,i) = bv(x,y,z) + o vo + i vi
//   columns o = o0 ... o0 + NO - 1,  o0 = floor(oc - ho) + 1
//   column o: i = i0 ... i0 + NI - 1,
//             i0 = floor(ic + max(au + lu (o - oc), av + lv (o - oc))) + 1
// shape = 16 * NO + NI when both are <= 3 (unrolled loops), else 0;
// order = NO | NI << 8 | outer_is_j << 16.
template <typename T>
struct AdjProj {
    T oc[4], ic[4], bu[4], bv[4];
    T uo, ui, vo, vi, ho, au, lu, av, lv, step;
    int shape, order;
};

// Kernel-parameter block holding the constants of up to kMax projections
// (kept under the 32 KB kernel-parameter limit).
template <typename T>
struct AdjParams {
    static constexpr int kMax = sizeof(T) == 4 ? 256 : 128;
    AdjProj<T> p[kMax];
};

// Where a gradient-mode forward writes the back-contracted residual when the
// handle works in detector modes (tt_modes.cuh): rows of `row` floats at the
// kernel's G argument and, with G1, one more value per ray; Q [CP][kModeQ],
// zero padded.
constexpr int kModeQ = 12;          // padded mode count of Q (at most 9 modes)
constexpr int kMaxModes = 9;
constexpr int kModeKMax = 45;       // coefficients of the largest band limit that works in modes (8)
struct ModeOut {
    const float *Q = nullptr;
    float *G1 = nullptr;
    int row = 0, nk1 = 0;             // nk1: row pitch of G1 (the detector's nk rounded up to 4)
    unsigned *nonfinite = nullptr;    // set to rows_id when a value written is not finite
    unsigned rows_id = 0;
};

// Layout of the R modes of a ray or voxel: rows of 4 * R4 floats and, with R1,
// one more value in a separate plane behind all rows (R = 5 and 9 would waste
// three floats of padding otherwise).
__host__ __device__ constexpr int modes_r4(int R) { return R <= 5 ? 1 : 2; }
__host__ __device__ constexpr int modes_r1(int R) { return (R == 5 || R == 9) ? 1 : 0; }

// Mode adjoint (k_adjoint_modes): M = 4 * R4 + R1 stored modes; projections of
// a hand-off unit, its tensor-core operand columns (2 M per projection, to a
// multiple of 8) and channels (to a multiple of 16).
__host__ __device__ constexpr int modes_m(int R) { return 4 * modes_r4(R) + modes_r1(R); }
__host__ __device__ constexpr int modes_up(int M) { return M == 9 ? 1 : 2; }
__host__ __device__ constexpr int modes_ku(int M) { return (2 * M * modes_up(M) + 7) / 8 * 8; }
__host__ __device__ constexpr int modes_n(int K) { return (K + 15) / 16 * 16; }
constexpr int kModeVox = 256;                  // voxels of a CTA: 8 (x) x 4 (y) x 8 (z), two tiles of 128
// A mapped volume (slot): innermost axis first, rows of slot_pitch(n) voxels
// -- kSlotLead zeros, the n voxels, zeros up to the pitch -- and kSlotBorder
// zero rows and planes around them.  The taps of a ray's planes reach three
// voxels beyond the volume (behind a row, into the next row's lead).  The rows
// start on whole sectors, and the pitch modulo a 128-byte line (2 of 8 voxels
// of four values, 16 of 32 single values) keeps neighbouring rays that have
// stepped into the next row off each other's banks.
constexpr int kSlotBorder = 3, kSlotLead = 8;
__host__ __device__ constexpr int slot_pitch4(int n) { return (n + kSlotLead + 7) / 8 * 8 + 2; }
__host__ __device__ constexpr int slot_pitch1(int n) { return (n + kSlotLead + 15) / 32 * 32 + 16; }
constexpr uint32_t kMapCols = 256;             // tensor-memory columns of a map CTA
constexpr int kModeStages = 3;                 // units in flight
constexpr uint32_t kModeWaitTries = 1u << 20;
constexpr long long kModeMaxSmem = 110 * 1024; // two CTAs per SM
constexpr int kModeThreads = kModeVox / 2 + 32;   // two voxels per thread, and the warp that feeds the tensor cores
// Resident CTAs per SM: the accumulators (2 N registers) and the tensor memory
// (256 columns for N > 16) allow two, N = 16 four.
__host__ __device__ constexpr int mode_ctas(int N) { return N == 16 ? 4 : 2; }
__host__ __device__ constexpr uint32_t mode_align(uint32_t b) { return (b + 127) & ~127u; }

// Per-projection constants of the mode adjoint, detector coordinates relative
// to the CTA's box (o: outer, i: inner enumeration axis, see AdjProj): slopes
// along the voxel axes, taps' slopes, oh = 1/2 - ho, the lower edge's au, av
// with 1/2 added, index strides in the box, k0 = -kRoundBits (so + si), the
// largest row index a column may start at.
struct alignas(16) ModeProj {
    float o[3], oh;
    float i[3], pad;
    float uo, vo, ui, vi;
    float au, av, lu, lv;
    int so, si, k0, lim;
    int shape, order, pad2[2];
};
struct ModeParams {
    static constexpr int kMax = 256;
    ModeProj p[kMax];
};
// Detector coordinates of the voxel (x, y, z) = j[0] + j[1] x + ..., and the
// lowest one of a block's candidate rays relative to its corner's.
struct ModeOrigin {
    double j[4], k[4], jlo, klo;
    int outer_j;
};
// What tt_adjoint was given, for voxels that infinite data reach (R NULL: the
// rows come from a residual).
struct ModeData {
    const float *R;
    const ProjGeom *geo;
    const float *Bp;
    int S, nj, nk, C, CP;
};
// The packed volume, for rays through infinite coefficients.
struct ModeVolume {
    const void *cpad, *cpadx;            // interior origins of the copies
    const float *Bp;
    int prec, K, KP;
};
// The adjoint's enumeration constants of a projection in FP64 (see AdjProj).
struct AdjConst {
    double oc[4], ic[4], bu[4], bv[4], jc[4], kc[4];
    double uo, ui, vo, vi, ho, au, lu, av, lv;
    int no, ni;
    bool outer_j;
};

struct LossSlot {
    double value;
    unsigned long long seq;
};

struct Profile {
    struct Pending {
        cudaEvent_t begin, end;
        int slot;
        bool free_end;                 // false when `end` is also the next pair's begin
    };
    bool enabled = false;
    // Inside a chain of back-to-back launches on the stream (nothing else
    // enqueued between them), a launch's end event is the next one's begin.
    bool chain = false;
    cudaEvent_t last_end = nullptr;
    std::deque<Pending> pending;       // recorded pairs, oldest first, not yet folded into the totals
    std::vector<cudaEvent_t> free_events;
    double total_ms[TT_KSLOT_COUNT] = {};
    long long launches[TT_KSLOT_COUNT] = {};
};

}  // namespace tt

struct tt_handle {
    tt_precision prec;
    int dev;
    int n_sm = 0;                        // streaming multiprocessors of dev (grid sizing)
    cudaStream_t stream;
    // Recorded on the old stream when tt_set_stream switches streams; the
    // new stream waits on it, so work still in flight on the old stream
    // (an adjoint behind an early-returned loss) finishes with the handle's
    // buffers before the new stream reuses them.
    cudaEvent_t stream_switch = nullptr;
    int N[3];
    int nj, nk, S, L, K, KP, LG, C, CP;
    double a, b, two_theta;
    std::vector<double> inner, outer, joff, koff, seg0, seg1;
    tt_frame frame;
    std::vector<tt::ProjGeom> geo_host;
    tt::ProjGeom *geo = nullptr;        // device [S]
    double *B64 = nullptr;               // device [S][C][K] FP64
    void *Bp = nullptr;                  // device [S][CP][KP], element type, zero padded
    // Padded coefficient volume, two-voxel zero border, channel innermost:
    // [nx+4][ny+4][nz+4][KP] (z innermost) and, when some projection's main
    // axis is z, a second copy [nz+4][ny+4][nx+4][KP] (x innermost) right
    // after it, so that every projection has a transverse axis of stride one
    // and a bilinear tap pair along it is one contiguous 2*KP-element piece.
    void *cpad = nullptr;
    long long cpad_origin = 0;           // voxel offset of (0,0,0) in cpad
    bool zero_volume = false;            // set around a forward launch whose volume is zero (not packed)
    bool xcopy = false;                  // the x-innermost copy exists
    long long pad_vox = 0;               // voxels of one padded copy
    long long cpadx_origin = 0;          // voxel offset of (0,0,0) in the x-innermost copy (from its start)
    void *arena = nullptr;               // device: holds geo, B64, Bp, cpad, gpad, G, partials, red, mode_mem
    void *gpad = nullptr;                // device [nvox][KP]
    void *G = nullptr;                   // device [S][nj][nk][KP]
    // Detector modes (tt_modes.cuh; 0: the handle works in channels): G holds
    // rows of 4 * R4 mode values, then (R1) one more per ray.
    int R = 0, R4 = 0, R1 = 0;
    bool q_identity = false;             // the modes are the segments (Q = 1)
    void *mode_mem = nullptr;            // in the arena: holds what follows, down to `order`
    size_t mode_host_bytes = 0;          // of it, the part that the host fills
    float *Qm = nullptr;                 // device [CP][kModeQ], zero padded
    unsigned *nonfinite = nullptr;       // device: the last rows_id whose rows were not all finite
    unsigned rows_id = 0;                // number of the rows in G (a new one for each that are written)
    double *F64 = nullptr;               // device [S][R][K]: F_s
    float *FB = nullptr;                 // device: F_s as the adjoint's tensor-core operand
    tt::ModeOrigin *mode_org = nullptr;  // device [S]
    int box_j = 0, box_k = 0;            // the adjoint's detector box (pixels)
    int nk1 = 0;                         // row pitch of the single values' plane (R1)
    tt::TmaDesc rows_map, single_map;    // maps of the rows in G, of their single values
    std::vector<tt::ModeParams> mode_params;   // one block per launch
    // Mode forward (tt_modes_fwd.cu): F rows for the map, the projections
    // reading copy 0, then copy 1 of the packed volume, and the slots of
    // mapped volumes: chunk slots for either copy, zero border.
    void *FM = nullptr;
    int *order = nullptr;                // device [S]
    std::vector<tt::ModeOrigin> org_host;
    std::vector<int> order_host;
    int order_begin[2] = {0, 0};
    float *slots = nullptr;
    long long slot_floats = 0, slot_vox = 0;   // floats of a slot, voxels of its four-value planes
    long long slots1 = 0;                // where copy 1's slots start
    int chunk = 0;                       // slots, the projections of a chunk
    bool fwd_modes = false;              // the forward maps and marches modes
    bool wide_detector = false;          // the volume's shadow covers less than 45% of the detector
    double *partials = nullptr;          // device, per-CTA loss partials
    long long n_partials = 0;            // allocated entries
    long long n_fwd_ctas = 0;            // entries the forward kernel writes
    // Staged forward march: voxels of the largest plane box over the
    // projections, rounded up to even (0 when the kernel does not apply),
    // and whether the forward runs it.
    int stage_cap = 0;
    bool fwd_staged = false;
    tt::TmaDesc *tmaps = nullptr;        // device [S]: tensor map of each projection's plane box
    std::vector<tt::TmaDesc> tmaps_host;
    double *red = nullptr;               // device, dot_blocks(h) partials of the regulariser reductions
    double *loss_dev = nullptr;          // device scalars: [0] loss, [1] regulariser value
    double *loss_pinned = nullptr;       // pinned host scalar
    // Page-locked, device-mapped slot where the adjoint's first CTA publishes
    // the loss of a gradient evaluation (value, then sequence number), so
    // that tt_gradient_residual can return it while the adjoint still runs.
    tt::LossSlot *loss_slot_host = nullptr, *loss_slot_dev = nullptr;
    unsigned long long loss_seq = 0;     // last sequence number handed out
    unsigned long long loss_publish = 0; // sequence number the next evaluation publishes (0: none)
    // host-buffer entry point staging (allocated on first use)
    void *hc = nullptr, *hI = nullptr, *hW = nullptr, *hg = nullptr;
    cudaStream_t copy_stream = nullptr;  // host-buffer path: data chunks copied while the forward runs
    cudaStream_t side[2] = {nullptr, nullptr};  // host-buffer path: forward chunks, two at a time
    std::vector<cudaEvent_t> chunk_ready;
    long long launch_count = 0;
    tt::Profile prof;
    std::vector<tt::AdjParams<float>> adj_f32;     // adjoint constants, one block per launch
    std::vector<tt::AdjParams<double>> adj_f64;

    long long nvox() const { return (long long)N[0] * N[1] * N[2]; }
    long long npix() const { return (long long)S * nj * nk; }
    long long ndata() const { return npix() * C; }
    size_t esize() const { return prec == TT_F64 ? 8 : 4; }                 // API element
    size_t ssize() const { return prec == TT_BF16 || prec == TT_F16 ? 2 : esize(); }  // cpad storage
};

namespace tt {

// Compensated FP32 dot-product accumulation (Ogita, Rump & Oishi, "Accurate
// sum and dot product", SIAM J. Sci. Comput. 26, 2005, algorithm Dot2): the
// rounding error of each product comes from an FMA, that of each sum from
// TwoSum, and both are gathered in a second FP32 word.  The result is about
// as accurate as the dot product summed in twice the working precision, at
// FP32 speed (this GPU's FP64 rate is a small fraction of its FP32 rate).
// The _rn intrinsics keep the compiler from contracting the steps.
struct Dot2 {
    float s, c;
};

__device__ __forceinline__ void dot2_add(Dot2 &a, float x, float y)
{
    const float p = __fmul_rn(x, y);
    const float pe = __fmaf_rn(x, y, -p);          // x y - p, exactly
    const float t = __fadd_rn(a.s, p);
    const float z = __fsub_rn(t, a.s);
    const float e = __fadd_rn(__fsub_rn(a.s, __fsub_rn(t, z)), __fsub_rn(p, z));   // a.s + p - t, exactly
    a.s = t;
    a.c = __fadd_rn(a.c, __fadd_rn(e, pe));
}

__device__ __forceinline__ double dot2_value(const Dot2 &a) { return (double)a.s + (double)a.c; }

// a += x, compensated (Dot2's summation step alone).
__device__ __forceinline__ void dot2_add1(Dot2 &a, float x)
{
    const float t = __fadd_rn(a.s, x);
    const float z = __fsub_rn(t, a.s);
    const float e = __fadd_rn(__fsub_rn(a.s, __fsub_rn(t, z)), __fsub_rn(x, z));
    a.s = t;
    a.c = __fadd_rn(a.c, e);
}

// (s, c) + (s', c') with the same compensation: TwoSum of the leading parts,
// the error added to the sum of the trailing parts.
__device__ __forceinline__ Dot2 dot2_merge(Dot2 a, Dot2 b)
{
    Dot2 r = a;
    dot2_add1(r, b.s);
    r.c = __fadd_rn(r.c, b.c);
    return r;
}

// Deterministic (fixed-order) block sum of one compensated pair per thread,
// in FP32 arithmetic: a warp tree of dot2_merge, the warps' results merged
// by warp 0.  The one conversion to FP64 happens at the end; on this GPU an
// FP64 shuffle tree per CTA costs tens of times more issue time in the FP64
// pipe than the same tree in FP32.  red: one Dot2 of shared memory per warp;
// the leading barrier lets a CTA call it several times in a row.  Result
// valid on thread 0.
__device__ __forceinline__ double dot2_block_sum(Dot2 v, Dot2 *red)
{
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        const Dot2 o = {__shfl_down_sync(0xffffffffu, v.s, off), __shfl_down_sync(0xffffffffu, v.c, off)};
        v = dot2_merge(v, o);
    }
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    __syncthreads();
    if (l == 0) red[w] = v;
    __syncthreads();
    if (w != 0) return 0.0;
    Dot2 t = l < (int)(blockDim.x >> 5) ? red[l] : Dot2{0.f, 0.f};
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        const Dot2 o = {__shfl_down_sync(0xffffffffu, t.s, off), __shfl_down_sync(0xffffffffu, t.c, off)};
        t = dot2_merge(t, o);
    }
    return l == 0 ? dot2_value(t) : 0.0;
}

void set_error(const std::string &msg);
tt_status cuda_fail(cudaError_t e, const char *what);
// Problem validation and Gauss-Legendre rule shared by the entry points.
tt_status validate(const tt_problem *P);
void gauss_legendre(int n, double *x, double *w);
// The rows k_basis reads for one projection: R_s^T p, R_s^T q0, R_s^T q90
// (R_s = R_beta(outer angle) R_alpha(inner angle), FP64), 9 doubles.
void basis_frame(const tt_frame &fr, double inner_angle, double outer_angle, double out[9]);

template <typename T>
const std::vector<AdjParams<T>> &adj_params(const tt_handle *h);
template <>
const std::vector<AdjParams<float>> &adj_params<float>(const tt_handle *h);
template <>
const std::vector<AdjParams<double>> &adj_params<double>(const tt_handle *h);

// Bracket a kernel launch with the handle's profiling events.
void prof_begin(tt_handle *h, int slot, cudaEvent_t *ev);
void prof_end(tt_handle *h, int slot, cudaEvent_t ev);
// While alive, the handle's launches share boundary events (the launches it
// covers must be enqueued back to back on the handle's stream).
struct ProfChain {
    tt_handle *h;
    explicit ProfChain(tt_handle *h_);
    ~ProfChain();
    ProfChain(const ProfChain &) = delete;
    ProfChain &operator=(const ProfChain &) = delete;
};

// Kernel launchers (return the launch error, if any).
// Packs c [nvox][K] into the interior of cpad (channels padded to KP).
template <typename T, typename S>
cudaError_t launch_pack(tt_handle *h, const T *c);
template <typename T>
cudaError_t launch_unpack(tt_handle *h, const T *gpad, T *g);
// Projector launchers: arithmetic in T, the coefficient volume cpad stored as
// S (S = T, or a 2-byte type for T = float); the back-contracted residual G
// is T.
// Projections [s0, s1) only (s1 < 0: to the last); the gradient mode writes
// the loss partials of those projections' CTAs.
template <typename T, typename S>
cudaError_t launch_forward(tt_handle *h, T *Iout, const T *I, const T *W, bool grad, int s0 = 0, int s1 = -1);
template <typename T, typename S>
cudaError_t launch_backcontract(tt_handle *h, const T *R);
// g [nvox][K] (unpadded) = exact-transpose gather of G; S above one
// parameter block runs several launches accumulating in h->gpad.
// With reduce_loss the first launch also sums the forward's per-CTA loss
// partials (h->partials, h->n_fwd_ctas) into h->loss_dev[0], in the order of
// launch_reduce, so that the gradient evaluation needs no separate
// reduction launch.
template <typename T, typename S>
cudaError_t launch_adjoint(tt_handle *h, T *g, bool reduce_loss = false);
// cudaMalloc for what is allocated later than the handle: a handle whose mode
// forward holds memory that is wanted gives its slots up and marches the volume.
cudaError_t handle_malloc(tt_handle *h, void **p, size_t bytes);
// Detector modes: set-up (F_s, Q and the operand; enqueued on the handle's
// stream), the adjoint and the back-contraction.
AdjConst adj_const(const ProjGeom &g);
inline long long mode_operand_floats(const tt_handle *h)
{
    const int M = modes_m(h->R), UP = modes_up(M);
    return (long long)((h->S + UP - 1) / UP) * 2 * modes_ku(M) * modes_n(h->K);
}
// Sets R and the boxes of a handle that can work in detector modes, else R = 0.
void plan_modes(tt_handle *h);
// Bytes of what the modes keep beside the slots; with base, where each part lies.
size_t place_modes(tt_handle *h, char *base);
// frames: device; node, weight: the kQuadNodes of the segments' rule, host.
cudaError_t setup_modes(tt_handle *h, const double *frames, const double *node, const double *weight);
// The forward in modes (tt_modes_fwd.cu): ray tiles (loss partials), sizes
// (slot_floats 0: the handle does not use it; `reserved`: bytes still to be
// allocated), set-up and launch.
void plan_mode_forward(tt_handle *h, size_t reserved);
// Share of the detectors' pixels that the volume's shadow covers.
double shadow_share(const tt_handle *h);
long long mode_forward_ctas(const tt_handle *h);
cudaError_t setup_mode_forward(tt_handle *h, const double *F);
template <typename S>
cudaError_t launch_forward_modes(tt_handle *h, float *Iout, const float *I, const float *W, bool grad, int s0, int s1);
// rows: the mode rows [S][nj][nk][4 R4] (h->G, or a caller's array); data: the
// caller's data that they come from (tt_adjoint), or NULL.
cudaError_t launch_adjoint_modes(tt_handle *h, const float *rows, float *g, bool reduce_loss, const float *data = nullptr);
cudaError_t launch_backcontract_modes(tt_handle *h, const float *R);
// Notes whether a caller's rows are all finite, as the kernels that write rows do.
cudaError_t launch_check_rows(tt_handle *h, const float *rows);
inline ModeOut mode_out(const tt_handle *h)
{
    ModeOut m;
    if (h->R) {
        m.Q = h->Qm;
        m.row = 4 * h->R4;
        m.nk1 = h->nk1;
        m.nonfinite = h->nonfinite;
        m.rows_id = h->rows_id;
        m.G1 = h->R1 ? (float *)h->G + h->npix() * m.row : nullptr;
    }
    return m;
}
// While in scope with on = true the handle works in channels throughout: the
// tap-pair march (or the staged one where it was chosen) and k_adjoint.
struct ChannelScope {
    tt_handle *h;
    int R = 0;
    bool fwd_modes = false;
    long long n_fwd_ctas = 0;
    ChannelScope(tt_handle *h, bool on);
    ~ChannelScope();
};
cudaError_t launch_reduce(tt_handle *h, const double *partials, long long n, double *out,
                          const double *add, double mul);
cudaError_t launch_basis(tt_handle *h, const double *nodes, const double *weights);
template <typename T>
cudaError_t launch_cast_basis(tt_handle *h);

// FP64-accumulated vector kernels for the optimizer.
template <typename T>
cudaError_t vec_dot(tt_handle *h, const T *x, const T *y, long long n, double *partials,
                    double *out, const double *add, double mul);
// y = a*x + b*y with a = ha * (da ? *da : 1), b = hb (y is not read when hb == 0)
template <typename T>
cudaError_t vec_axpby(tt_handle *h, T *y, const T *x, long long n, double ha, const double *da, double hb);
template <typename T>
cudaError_t vec_sub(tt_handle *h, T *out, const T *x, const T *y, long long n);
// Streaming-multiprocessor count of the current device (queried once per
// device ordinal and cached); grids of the grid-stride kernels are capped at
// multiples of it.
int current_sm_count();
// CTAs of the dot-product and regulariser reductions: four per SM.
inline int dot_blocks(const tt_handle *h) { return 4 * h->n_sm; }
// Dynamic shared memory of the staged forward: the stage ring, B_s and 128
// bytes of slack to align the ring; the gradient in modes adds Q, 16 floats a
// segment too (at most 4 KB, which the SM has beyond kStMaxSmem).
inline size_t staged_forward_smem(const tt_handle *h, bool modes)
{
    return (size_t)kStRing * h->stage_cap * 16 * sizeof(float) + (size_t)h->CP * (modes ? 32 : 16) * sizeof(float) + 128;
}

}  // namespace tt
