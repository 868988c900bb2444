// Separable gridder on the tensor cores (tcgen05), L = 32, 24 and 16.
//
// The subgrid image of Eq. (ShiftedDirectImaging) is
//   I_q(x, y) = sum_k V_kq exp(i (a_k X + b_k Y + c_k n'(x, y))),
// with X = x - L/2, Y = y - L/2 and c_k = 2 pi (w_k - w_s) (w_s the subgrid's w
// offset, see the epilogue).  Splitting n'(x, y) = s(x) + t(y) + r(x, y), s and t
// a row and a column of n' (the plan's reference row and column j0: s(x) =
// n'(x, j0), t(y) = n'(j0, y) - n'(j0, j0)), the phasor factors into
//   Ex_k(x) = exp(i (a_k X + c_k s(x))),  Ey_k(y) = exp(i (b_k Y + c_k t(y))),
// times exp(i c_k r(x, y)).  The remainder r is fourth order in (l, m); where
// theta = max |c_k| max |r| is small (the plan checks theta <= 1.38e-3, so that
// theta^2 / 2 <= 2^-20) the factor is taken to first order,
// exp(i c r) = 1 + i c r + O(theta^2 / 2), so
//   I_q(x, y) = S0_q(x, y) + i r(x, y) S1_q(x, y),
//   S_mq(x, y) = sum_k [V_kq Ey_k(y)] [c_k^m Ex_k(x)],   m = 0, 1,
// a complex matrix product over the visibilities: rows (q, y), 128 of them,
// columns (m, x), 64.  Per visibility the CUDA cores form 128 + 64 phasor
// products instead of the L^2 = 1024 of the direct sum, and the tensor cores
// do the contraction.
//
// GEMM.  A[(q, y)][2 k + r] = (Re, Im)[r] of V_kq Ey_k(y) (tensor memory);
// B holds the real 2 x 2 embedding of beta = (c_k sigma)^m Ex_k(x): row
// (m, x, re) = (Re beta, -Im beta), row (m, x, im) = (Im beta, Re beta) over
// K = (k, r), so D[(q, y)][(m, x, re/im)] = (Re, Im) S_mq.  sigma is a power of
// two with max |c_k| sigma <= 1.
//
// Precision.  Both operands are split into FP16 hi + lo parts, A after a power-of-two scale per
// subgrid, and hi + lo holds every value of A to 2^-22 of itself or 2^-13 of a quantum Q, whichever
// is larger: hi is the FP16 value rounded to a multiple of Q, 2^-7 of its polarisation's geometric
// mean |Re V| + |Im V| in the subgrid.  Without that rounding the tensor cores, which truncate, lose
// the products' last bits at every step (1.4e-6 instead of 0.8e-6 of a grid); with one Q per
// subgrid, below its largest value, a cross hand of 1 % would keep 11 bits (3e-5 of its grid).  B's
// phasors are split at multiples of 2^-11: hi + lo holds them to 2^-24 of 1.  The m = 0
// block takes A_hi B_hi + A_hi B_lo + A_lo B_hi; the m = 1 block, which
// contributes at most theta relative, takes A_hi B_hi only.  One MMA of N = 192
// computes A_hi [B_hi (128 rows) | B_lo (m = 0, 64 rows)], a second of N = 64 adds
// A_lo B_hi (m = 0) to the correction columns.  The tensor cores accumulate
// without rounding to nearest, so every 512 visibilities the accumulator is folded
// into the FP32 image in shared memory (RN) and restarted; the fold applies
// I = S0 + i r S1 / sigma, so it keeps one complex image, half of S0 and S1.
//
// Schedule.  One CTA per subgrid and two CTAs per SM (half the tensor memory and 106
// of 227 KB shared memory each): one CTA's start, folds, transform and adder run under
// the other's sums.  A CTA has two sets of four producer warps, an MMA warp and a
// loader warp.  The sets take turns: a stage is two groups of 8 visibilities of one
// set.  Per group, warp yq of the set
//   - forms A of the 8 pixel rows y = 8 yq .. + 7 and all four polarisations (its
//     lane quarter of tensor memory).  The 16 x 256-bit store form gives a thread
//     four of the quarter's rows for two visibilities: two pixel rows x two
//     polarisations, so that each Ey and each V is used twice, without shuffles;
//   - forms B of the pixel columns x = 8 yq .. + 7 (at L = 24 and 16 the quarters
//     without A rows take the B blocks).
// A and B of a group are formed side by side (their chains of phase, sine and cosine,
// split and conversion overlap); A's stage buffer is freed by the set's previous
// MMAs, B has two buffers per set.  Visibilities are staged 256 at a time, as pairs:
// the first batch by the producers, the others by the loader warp, which keeps their
// loads out of the producers' registers; staging.h has the rules of the hand-over.
// Tensor memory (256 columns):
//   accumulator: main (m, re/im, x) 0..127, correction (m = 0) 128..191
//   A of set s at 192 + 32 s, group i at + 16 i: 8 columns hi, 8 lo
//
// What bounds it, and what the choices measured (LOFAR-like plan, 73.9 M visibilities in
// 45.9 k subgrids of about 1600; and the same array with A-terms every 16 s, 18.4 M in
// 89.4 k of about 206):
//   one CTA per SM, 16 producer warps, Ey by shuffles        13.42 ms    7.65 ms
//   two CTAs, fragment stores, exact hi/lo split             13.03       5.62
//   one thread per transform line, columns straight to the
//   grid (the pixel passes around the transform cost a
//   third of a short subgrid's instructions)                 12.69       5.09
//   B around the A stores, A and B side by side              12.02       4.88
//   loader warp (short subgrids: no gain)                    11.51       4.98
//   A-terms ahead in registers instead of late bulk copies   11.43       4.82
//   two rows x two polarisations per thread                  11.28       4.73
//   A's hi by its own size, rounded per polarisation (the
//   figures above: one quantum per subgrid)                  11.41       4.84
//   the waits' failure word (the code it generates)          11.15       4.78
// It is bound by latency and issue of the producers together (busy: issue slots 62 %, the
// shared-memory data pipe 52 %, the tensor pipe 35 %); leaving out any one of the
// V loads, the split, the phasors or the MMA width gained 1 to 10 %.  Measured and not
// kept: A's hi rounded in FP32 with float means (11.72 and 4.94 ms: more registers, and the sums'
// shuffles weigh on short subgrids); one group per stage with two buffers (a stage's hand-over costs each warp
// about 670 cycles: 15.7 ms), polling by the producers (13.2), eight columns per fold
// step (1.46 against 1.42 Mcycles on the first 256 timesteps).
// Every wait is bounded.  After one that runs out a thread skips every later wait, the MMA thread
// issues no more MMAs, the error word is set and the subgrid is not written.
#include "batch_jobs.cuh"
#include "device_common.cuh"
#include "fft_impl.cuh"
#include "staging.h"
#include "tc_common.cuh"

namespace idg {

// device error word of the separable gridder (0 = ok); read and cleared by
// idg_device_errors
__device__ int g_sep_error = 0;

namespace {

using namespace dev;
using namespace tc;

constexpr int NPW = 8;                         // producer warps: two sets of four
constexpr int NP = NPW * 32;                   // producer threads
constexpr int MMA_WARP = NPW, LOAD_WARP = NPW + 1;
constexpr int NT = NP + 64;
constexpr int CTAS = 2;                        // per SM
constexpr int VB = NP;                         // visibilities per staged batch (one per producer)
constexpr int SG = 2;                          // groups of 8 visibilities per stage
constexpr int SPB = VB / (8 * SG);             // stages per batch
constexpr int SPP = 2 * SPB;                   // stages per accumulation period (512 visibilities)
constexpr uint32_t TMEM_COLS = 256;            // two CTAs share an SM's 512

// Layout for subgrid size L (32, 24 or 16).  A has 128 rows: lane quarter yq holds the pixel
// rows y = 8 yq .. + 7 of the four polarisations (see the A entries; quarters from L / 8 on are
// not used: their rows of the accumulator are never read).  B has 6 L rows per group: (m = 0, re), (m = 0, im),
// (m = 1, re), (m = 1, im), then the lo parts of m = 0 re and im, L rows each.
template <int L>
struct SepG {
    static constexpr int SL = L, SPIX = L * L, NQ = L / 8;   // NQ: 8-row (and 8-column) blocks
    static constexpr int B_GROUP = 6 * L * 32;   // B of one group: 6 L rows x 16 K FP16
    static constexpr int B_STAGE = SG * B_GROUP;
    // the subgrid image (polarisation planes, row pitch L + 1): the folded sums, then transformed
    static constexpr int FFT_P = PolPlanes<L>::P, FFT_S = PolPlanes<L>::STRIDE;
    static constexpr int B_OFF = (4 * FFT_S * 8 + 127) / 128 * 128;      // [2 sets][2 buffers][SG groups]
    // staged batches, [2] each, visibility pairs: (b0, b1, c0, c1), (a0, a1, c0, c1) and per
    // polarisation (re0, re1, im0, im1)
    static constexpr int CB_OFF = B_OFF + 4 * B_STAGE, CA_OFF = CB_OFF + 2 * VB * 8;
    static constexpr int VIS_OFF = CA_OFF + 2 * VB * 8;
    static constexpr int SMEM = VIS_OFF + 2 * VB * 32;
    // accumulator: main (m, re/im, x) at 0 .. 4 L, correction (m = 0) at 4 L .. 6 L; then the
    // sets' A, 32 columns each (group i at + 16 i: 8 columns hi, 8 lo)
    static constexpr uint32_t A_COL = 6 * L;
    static constexpr uint32_t IDESC_NB = idesc_m128(6 * L), IDESC_NC = idesc_m128(2 * L);
    static constexpr int XS = L / 2, XC = 4;               // x per set in the fold, in chunks
    static constexpr int PIXT = (SPIX + NP - 1) / NP;            // pixels per producer in the epilogue
    static_assert(L == 32 || L == 24 || L == 16, "subgrid sizes of the separable kernels");
    static_assert(CTAS * (SMEM + 2048) <= 227 * 1024, "shared memory of the SM's CTAs");
    static_assert(B_OFF % 128 == 0 && CB_OFF % 16 == 0, "alignment of the B tiles and the batches");
    static_assert(A_COL % 16 == 0 && A_COL + 2 * 16 * SG <= TMEM_COLS, "tensor memory");
};

__device__ __forceinline__ void producers_sync() { asm volatile("bar.sync 1, %0;" :: "n"(NP) : "memory"); }

// What a launch leaves: subgrid images o[L][L][4] (taper and A-terms applied), their transforms
// in the same place, or the transforms added into the grid o[layer][N][N][4]
enum Out { kImage, kTransform, kGrid };

// NEVER: the self-test's form, whose MMA thread gives up at once.
// One subgrid d of geometry g (Algorithm 1: direct sum, image-domain kernel, "FFT", add to the
// master grid)
template <int L, Out OUT, bool NEVER = false>
__device__ __forceinline__ void gridder_sep_body(const Geometry &g, const DevSubgrid d,
                                                 const float4 *__restrict__ vis, const uint8_t *__restrict__ flags,
                                                 const float4 *__restrict__ aterms, const float *__restrict__ taper,
                                                 float4 *__restrict__ o) {
    using C = SepG<L>;
    constexpr bool FUSED = OUT != kImage;       // transformed here
    constexpr int SL = C::SL, SPIX = C::SPIX, NQ = C::NQ, B_GROUP = C::B_GROUP, B_STAGE = C::B_STAGE;
    constexpr int FFT_P = C::FFT_P, FFT_S = C::FFT_S, XS = C::XS, PIXT = C::PIXT;
    constexpr uint32_t A_COL = C::A_COL;
    extern __shared__ __align__(1024) uint8_t smem[];
    float2 *s_img = (float2 *)smem;                 // 4 planes [L][L + 1]
    uint8_t *sB = smem + C::B_OFF;
    float *s_cb = (float *)(smem + C::CB_OFF), *s_ca = (float *)(smem + C::CA_OFF);
    float *s_vis = (float *)(smem + C::VIS_OFF);
    __shared__ uint32_t s_tmem;
    __shared__ __align__(8) uint64_t s_full[2], s_empty[2], s_foldbar, s_folded, s_drain,
        s_staged[kStagingBarriers], s_unstaged[kStagingBarriers];
    __shared__ int s_given_up;
    __shared__ float s_red[NPW];
    __shared__ int s_exp[NPW][5];
    __shared__ __align__(8) uint32_t s_round[4];

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const bool mma_warp = warp == MMA_WARP, producer = warp < NPW;
    const int kp = d.kp;
    const int total_groups = (kp + 7) / 8, n_stages = (total_groups + SG - 1) / SG;
    const int n_batches = (kp + VB - 1) / VB, n_periods = (n_stages + SPP - 1) / SPP;

    // staging: one visibility's inputs in registers, then its phase coefficients and scaled
    // values in shared memory.  The producers stage the first batch (its loads go out before
    // the set-up below, so their latency overlaps it), a loader warp the others
    struct Raw {
        float4 a, b, uv, sc;
        float2 w;
        bool in, flag;
    };
    const float4 *uvw2 = (const float4 *)g.uvw_f2;
    const float4 *sc2 = (const float4 *)g.scale_f2;
    const size_t bt0 = (size_t)d.bl * g.n_t + d.t0;
    auto load = [&](Raw &r, bool in, int t, int c) {
        r.in = in;
        r.flag = false;
        if (in) {
            const size_t bt = bt0 + t;
            const size_t vi = bt * g.n_chan + d.c0 + c;
            r.uv = uvw2[2 * bt];
            r.w = *(const float2 *)(uvw2 + 2 * bt + 1);
            r.sc = sc2[d.c0 + c];
            r.flag = flags && flags[vi];
            r.a = vis[2 * vi];         // loaded whatever the flag: the load does not wait for it
            r.b = vis[2 * vi + 1];
        }
    };
    // slot i of staging buffer bb: phase coefficients u (f/c) k_uv - u0 k_uv and so on (float
    // pairs, error-free products and sums, rounded once to FP32), scaled V (flagged: 0)
    auto stage = [&](const Raw &r, float scale, int bb, int i) {
        float ca = 0.f, cb = 0.f, cc = 0.f;
        float4 a = make_float4(0.f, 0.f, 0.f, 0.f), b = a;
        if (r.in) {
            ca = pair_coef(r.uv.x, r.uv.y, r.sc.x, r.sc.y, d.a0h, d.a0l);
            cb = pair_coef(r.uv.z, r.uv.w, r.sc.x, r.sc.y, d.b0h, d.b0l);
            cc = pair_coef(r.w.x, r.w.y, r.sc.z, r.sc.w, d.csh, d.csl);
            if (!r.flag) {
                a = make_float4(r.a.x * scale, r.a.y * scale, r.a.z * scale, r.a.w * scale);
                b = make_float4(r.b.x * scale, r.b.y * scale, r.b.z * scale, r.b.w * scale);
            }
        }
        const int at = bb * VB * 2 + (i >> 1) * 4 + (i & 1);
        s_cb[at] = cb;
        s_cb[at + 2] = cc;
        s_ca[at] = ca;
        s_ca[at + 2] = cc;
        float *v = s_vis + bb * VB * 8 + (i >> 1) * 4 + (i & 1);     // [q][pair]
        v[0] = a.x;
        v[2] = a.y;
        v[2 * VB] = a.z;
        v[2 * VB + 2] = a.w;
        v[4 * VB] = b.x;
        v[4 * VB + 2] = b.y;
        v[6 * VB] = b.z;
        v[6 * VB + 2] = b.w;
    };
    // the subgrid's power-of-two scale: largest unflagged |component| of V in [2^11, 2^12)
    auto scale_exponent = [&]() {
        float m = 0.0f;
#pragma unroll
        for (int w = 0; w < NPW; ++w) m = fmaxf(m, s_red[w]);
        int e2 = 0;
        if (m > 0.0f) frexpf(m, &e2);
        return min(12 - e2, 126);      // (a finite scale for the smallest inputs)
    };
    // timestep and channel (in the subgrid) of visibility k; advance() goes n visibilities on
    struct Where {
        int t, c, dt, dc, nc;
        __device__ __forceinline__ Where(int k, int nc_) : t(k / nc_), c(k - t * nc_), dt(0), dc(0), nc(nc_) {}
        __device__ __forceinline__ void step(int n) {
            dt = n / nc;
            dc = n - dt * nc;
        }
        __device__ __forceinline__ void advance() {
            t += dt;
            c += dc;
            if (c >= nc) {
                c -= nc;
                ++t;
            }
        }
    };
    Raw raw = {};
    auto max_of = [](const float4 &a, const float4 &b) {
        return fmaxf(fmaxf(fmaxf(fabsf(a.x), fabsf(a.y)), fmaxf(fabsf(a.z), fabsf(a.w))),
                     fmaxf(fmaxf(fabsf(b.x), fabsf(b.y)), fmaxf(fabsf(b.z), fabsf(b.w))));
    };
    if (mma_warp) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     :: "r"(smem_u32(&s_tmem)), "n"(TMEM_COLS));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    } else if (producer) {
        // the subgrid's largest unflagged |component| (the visibilities past the first batch are
        // read here once more, for the scale; they come back from L2 when they are staged)
        Where at(tid, d.nc);
        load(raw, tid < kp, at.t, at.c);
        // and, per polarisation, the sum of the binary exponents of |Re| + |Im|
        float m = 0.0f;
        int ex[4] = {}, n = 0;
        auto add_exponents = [&](const float4 &a, const float4 &b) {
            ex[0] += __float_as_int(fabsf(a.x) + fabsf(a.y)) >> 23;
            ex[1] += __float_as_int(fabsf(a.z) + fabsf(a.w)) >> 23;
            ex[2] += __float_as_int(fabsf(b.x) + fabsf(b.y)) >> 23;
            ex[3] += __float_as_int(fabsf(b.z) + fabsf(b.w)) >> 23;
            ++n;
        };
        if (kp > VB) {
            at.step(VB);
#pragma unroll 4
            for (int k = VB + tid; k < kp; k += VB) {
                at.advance();
                const size_t vi = (bt0 + at.t) * g.n_chan + d.c0 + at.c;
                const float4 va = vis[2 * vi], vb = vis[2 * vi + 1];
                if (!(flags && flags[vi])) {
                    m = fmaxf(m, max_of(va, vb));
                    add_exponents(va, vb);
                }
            }
        }
        if (raw.in && !raw.flag) {
            m = fmaxf(m, max_of(raw.a, raw.b));
            add_exponents(raw.a, raw.b);
        }
        m = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(m)));      // (m >= 0)
#pragma unroll
        for (int q = 0; q < 4; ++q) ex[q] = __reduce_add_sync(0xffffffffu, ex[q]);
        n = __reduce_add_sync(0xffffffffu, n);
        if (lane == 0) {
            s_red[warp] = m;
#pragma unroll
            for (int q = 0; q < 4; ++q) s_exp[warp][q] = ex[q];
            s_exp[warp][4] = n;
        }
    }
    if (tid == 0) {
        s_given_up = 0;
        for (int s = 0; s < 2; ++s) {
            mbar_init(smem_u32(&s_full[s]), NPW / 2);
            mbar_init(smem_u32(&s_empty[s]), 1);
        }
        mbar_init(smem_u32(&s_foldbar), 1);
        mbar_init(smem_u32(&s_folded), NPW);
        mbar_init(smem_u32(&s_drain), 1);
        for (int k = 0; k < kStagingBarriers; ++k) {
            mbar_init(smem_u32(&s_staged[k]), 1);
            mbar_init(smem_u32(&s_unstaged[k]), NPW);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = s_tmem;

    bool failed = false;
    // the epilogue's A-terms of a producer's pixel ip (A_p, A_q), read straight from L2: the first
    // AHEAD pixels' before the last fold, whose wait covers them, each later pixel's when an
    // earlier one has been used
    constexpr int AHEAD = PIXT < 2 ? PIXT : 2;
    M22 Ap[AHEAD], Aq[AHEAD];
    auto load_aterms = [&](int ip) {
        const int pix = tid + ip * NP;
        if (aterms && pix < SPIX) {
            const float4 *base = aterms + 2 * ((size_t)d.slot * g.n_stations) * SPIX + 2 * pix;
            Ap[ip % AHEAD] = load_m22(base + 2 * (size_t)d.st_p * SPIX);
            Aq[ip % AHEAD] = load_m22(base + 2 * (size_t)d.st_q * SPIX);
        }
    };
    const int yq = warp & 3, set = (warp >> 2) & 1;   // lane quarter (rows 32 yq ..) and producer set

    if (mma_warp) {
        if (lane == 0) {
            // descriptors and tensor-memory addresses advance by constants (the descriptor's
            // address field counts 16-byte units)
            const uint64_t db0 = smem_desc(smem_u32(sB));
            for (int st = 0; st < n_stages; ++st) {
                const int s = st & 1, use = st >> 1;        // set, and its how manieth stage
                const bool first = st % SPP == 0, last = st % SPP == SPP - 1 || st == n_stages - 1;
                if (first && st > 0) {         // the producers have read the previous period
                    wait_or_fail(smem_u32(&s_folded), (uint32_t)(((st / SPP) - 1) & 1), failed, &s_given_up);
                }
                poll_or_fail<NEVER>(smem_u32(&s_full[s]), (uint32_t)(use & 1), failed, &s_given_up);
                if (failed) break;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const int ng = min(SG, total_groups - st * SG);
                const uint64_t dbs = db0 + (uint64_t)(((2 * s + (use & 1)) * B_STAGE) >> 4);
                const uint32_t ats = tmem + A_COL + 16u * SG * (uint32_t)s;
#pragma unroll
                for (int i = 0; i < SG; ++i) {
                    if (i < ng) {
                        const uint64_t db = dbs + (uint64_t)((i * B_GROUP) >> 4);
                        mma_ta_i(tmem, ats + 16u * i, db, C::IDESC_NB, (first && i == 0) ? 0u : 1u);
                        mma_ta_i(tmem + 4u * SL, ats + 16u * i + 8u, db, C::IDESC_NC, 1u);
                    }
                }
                commit(smem_u32(&s_empty[s]));
                if (last) commit(smem_u32(&s_foldbar));
            }
            commit(smem_u32(&s_drain));
            if (!mbar_wait(smem_u32(&s_drain), 0u)) failed = true;     // bounded: let own MMAs finish before the free
        }
    } else if (warp == LOAD_WARP) {
        // batches 1 .. : 32 visibilities at a time, the next ones' loads in flight; a buffer is reused
        // once the producers are done with it
        const float scale = ldexpf(1.0f, scale_exponent());
        Where at(VB + lane, d.nc);
        at.step(32);
        if (n_batches > 1) load(raw, VB + lane < kp, at.t, at.c);
        for (int b = 1; b < n_batches; ++b) {
            const int bb = staging_buffer(b), bar = staging_barrier(b);
            if (b >= kStagingBuffers) wait_or_fail(smem_u32(&s_unstaged[bar]), staging_free_parity(b), failed, &s_given_up);
#pragma unroll 1
            for (int i = lane; i < VB; i += 32) {
                const Raw r = raw;
                at.advance();
                load(raw, b * VB + i + 32 < kp, at.t, at.c);
                stage(r, scale, bb, i);
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&s_staged[bar]));
        }
    } else {
        const int ex = scale_exponent();
        const float scale = ldexpf(1.0f, ex), inv_scale = ldexpf(1.0f, -ex);
        const uint32_t lane_base = tmem + ((uint32_t)(32 * yq) << 16);
        const float csig = g.c_scale, rs = 1.0f / csig;
        constexpr float magic_1 = 6144.0f;      // B's hi: multiples of 2^-11

        // one period's accumulator, I = S0 + i r S1 / sigma of this thread's row (polarisation
        // lane / 8, y = 8 yq + lane % 8) and its set's x, added to the image in FP32 (RN); the
        // accumulator is released right after the loads
        auto fold = [&](int P) {
            wait_or_fail(smem_u32(&s_foldbar), (uint32_t)(P & 1), failed, &s_given_up);
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            constexpr int XC = C::XC;
            if (yq < NQ) {
                // row 8 a + b: polarisation 2 (b / 4) + a / 2, y = 4 (a % 2) + b % 4 of the block
                const int y = 8 * yq + 4 * ((lane >> 3) & 1) + (lane & 3), q = 2 * ((lane >> 2) & 1) + (lane >> 4);
                float2 *img = s_img + q * FFT_S + y * FFT_P + set * XS;
                const float *rp = g.sep + 2 * SL + y * SL + set * XS;
#pragma unroll
                for (int x0 = 0; x0 < XS; x0 += XC) {
                    uint32_t re[XC], im[XC], cr[XC], ci[XC], r1[XC], i1[XC];
                    const uint32_t base = lane_base + (uint32_t)(set * XS + x0);
                    tmem_ld_nowait(base, re);
                    tmem_ld_nowait(base + SL, im);
                    tmem_ld_nowait(base + 2 * SL, r1);
                    tmem_ld_nowait(base + 3 * SL, i1);
                    tmem_ld_nowait(base + 4 * SL, cr);
                    tmem_ld_nowait(base + 5 * SL, ci);
                    tmem_wait_ld(re);
                    tmem_wait_ld(im);
                    tmem_wait_ld(r1);
                    tmem_wait_ld(i1);
                    tmem_wait_ld(cr);
                    tmem_wait_ld(ci);
                    if (x0 + XC == XS) {
                        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                        __syncwarp();
                        if (lane == 0) mbar_arrive(smem_u32(&s_folded));
                    }
#pragma unroll
                    for (int i = 0; i < XC; ++i) {
                        const float rr = rp[x0 + i] * rs;
                        const float vr = fmaf(-rr, __uint_as_float(i1[i]), __uint_as_float(re[i]) + __uint_as_float(cr[i]));
                        const float vi = fmaf(rr, __uint_as_float(r1[i]), __uint_as_float(im[i]) + __uint_as_float(ci[i]));
                        float2 f = P ? img[x0 + i] : make_float2(0.f, 0.f);
                        img[x0 + i] = make_float2(fmaf(vr, inv_scale, f.x), fmaf(vi, inv_scale, f.y));
                    }
                }
            } else {
                asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&s_folded));
            }
        };

        // A entries of a group: row 8 a + b of the quarter is polarisation 2 (b / 4) + a / 2, pixel row
        // y = 8 yq + 4 (a % 2) + b % 4; lane 4 b + jp holds rows b, 8 + b, 16 + b and 24 + b of the
        // visibilities 2 jp and 2 jp + 1 (the 16 x 256-bit fragments), so it forms Ey for two y and
        // multiplies two polarisations with each
        const int jp = lane & 3, qh = lane >> 4;
        const int y0 = 8 * yq + ((lane >> 2) & 3);
        const float Yv = (float)(y0 - SL / 2);
        const f2_t Y2[2] = {f2_bcast(Yv), f2_bcast(Yv + 4.0f)};
        const f2_t ty2[2] = {f2_bcast(yq < NQ ? g.sep[SL + y0] : 0.0f), f2_bcast(yq < NQ ? g.sep[SL + y0 + 4] : 0.0f)};
        auto a_unit = [&](const float *cb, const float *vb, int pair, const uint32_t (&round_a)[2], uint32_t (&e)[16]) {
            const ulonglong2 cf = *(const ulonglong2 *)(cb + 4 * (pair + jp));
            f2_t c2[2], s2[2], n2[2];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                float p0, p1, sn0, cs0, sn1, cs1;
                f2_unpack(f2_fma(cf.y, ty2[h], f2_mul(cf.x, Y2[h])), p0, p1);
                __sincosf(p0, &sn0, &cs0);
                __sincosf(p1, &sn1, &cs1);
                c2[h] = f2_pack(cs0, cs1);
                s2[h] = f2_pack(sn0, sn1);
                n2[h] = f2_mul(s2[h], f2_bcast(-1.0f));
            }
#pragma unroll
            for (int ql = 0; ql < 2; ++ql) {
                const ulonglong2 v = *(const ulonglong2 *)(vb + 2 * VB * (2 * qh + ql) + 4 * (pair + jp));
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int k = 8 * ql + 2 * h;
                    split_pairs(f2_fma(v.y, n2[h], f2_mul(v.x, c2[h])), f2_fma(v.y, c2[h], f2_mul(v.x, s2[h])),
                                round_a[ql], e[k], e[k + 1], e[k + 4], e[k + 5]);
                }
            }
        };
        // B entries of 8 pixel columns from 8 xblk for one group: lane = 8 jl + (x % 8), visibilities
        // 2 jl and 2 jl + 1, which sit in adjacent K slots of each row: one 8-byte store per row (a
        // warp's store covers 256 contiguous bytes).  beta = Ex_k(x) (m = 0: hi and lo) and c_k sigma
        // Ex_k(x) (m = 1: hi), rows (m, re, x) = (Re beta, -Im beta) and (m, im, x) = (Im beta, Re beta)
        const int jl = lane >> 3;
        auto b_unit = [&](const float *ca, int pair, int xblk, f2_t X2, f2_t sx2, uint8_t *Bg) {
            const ulonglong2 cf = *(const ulonglong2 *)(ca + 4 * (pair + jl));
            float p0, p1, sn0, cs0, sn1, cs1;
            f2_unpack(f2_fma(cf.y, sx2, f2_mul(cf.x, X2)), p0, p1);
            __sincosf(p0, &sn0, &cs0);
            __sincosf(p1, &sn1, &cs1);
            const f2_t c2 = f2_pack(cs0, cs1), s2 = f2_pack(sn0, sn1);
            const f2_t cz = f2_mul(cf.y, f2_pack(csig, csig)), zc = f2_mul(cz, c2), zs = f2_mul(cz, s2);
            f2_t hc, lc, hs, ls, hn, ln;
            f2_split(c2, magic_1, hc, lc);
            f2_split(s2, magic_1, hs, ls);
            hn = f2_mul(hs, f2_bcast(-1.0f));
            ln = f2_mul(ls, f2_bcast(-1.0f));
            uint32_t w[6][2];
            pack_pairs(hc, hn, w[0][0], w[0][1]);
            pack_pairs(hs, hc, w[1][0], w[1][1]);
            pack_pairs(zc, f2_mul(zs, f2_bcast(-1.0f)), w[2][0], w[2][1]);
            pack_pairs(zs, zc, w[3][0], w[3][1]);
            pack_pairs(lc, ln, w[4][0], w[4][1]);
            pack_pairs(ls, lc, w[5][0], w[5][1]);
            Bg += (uint32_t)xblk * kSBO + (uint32_t)(jl >> 1) * kLBO + (uint32_t)(lane & 7) * 16 + (uint32_t)(jl & 1) * 8;
#pragma unroll
            for (int q = 0; q < 6; ++q) *(uint2 *)(Bg + NQ * q * kSBO) = make_uint2(w[q][0], w[q][1]);
        };
        auto x_pair = [&](int xblk, f2_t &X2, f2_t &sx2) {
            const int x = 8 * xblk + (lane & 7);
            const float X = (float)(x - SL / 2), sx = g.sep[x];
            X2 = f2_pack(X, X);
            sx2 = f2_pack(sx, sx);
        };
        // this warp's x block: its own number at L = 32; at L = 24 and 16 the quarters without A
        // rows take B blocks instead (16: quarters 2, 3 all of B; 24: quarter 3 the first group's)
        const int xown = SL == 16 ? (yq & 1) : (SL == 24 && yq == 3 ? 0 : yq);
        f2_t X2, sx2;
        x_pair(xown, X2, sx2);

        stage(raw, scale, 0, tid);
        // the quantum Q of A's hi per polarisation: 2^-7 of the geometric mean of |Re V| + |Im V|, as
        // 1536 Q in FP16 (a number with that ulp); 0 (no rounding to it) where there is nothing to go by
        if (warp == 0 && lane < 4) {
            int sum = 0, n = 0;
#pragma unroll
            for (int w = 0; w < NPW; ++w) {
                sum += s_exp[w][lane];
                n += s_exp[w][4];
            }
            const int e = n > 0 ? sum / n - 127 + ex - 7 : -127;
            const float r = e >= -24 && e <= 5 ? ldexpf(1536.0f, e) : 0.0f;
            s_round[lane] = pack_f16x2(r, r);
        }
        producers_sync();
        const uint2 r2 = *(const uint2 *)(s_round + 2 * qh);
        const uint32_t round_a[2] = {r2.x, r2.y};
        int next_fold = 0;
        for (int b = 0; b < n_batches; ++b) {
            const int bb = staging_buffer(b), bar = staging_barrier(b);
            if (b > 0) wait_or_fail(smem_u32(&s_staged[bar]), staging_full_parity(b), failed, &s_given_up);
            const float *cb = s_cb + bb * VB * 2, *ca = s_ca + bb * VB * 2, *vb = s_vis + bb * VB * 8;
            const int st_end = min((b + 1) * SPB, n_stages);
            // B of the stage's first (half 0) or second group (half 1); at L = 24 quarter 3 does the first
            // group's three blocks, 0 and 1 in half 0.  (A group past the last is staged zeros, which no
            // MMA reads.)
            auto b_half = [&](int pair, uint8_t *Bs, int half) {
                if constexpr (SL == 24) {
                    if (yq < NQ) {
                        if (half) b_unit(ca, pair + 4, yq, X2, sx2, Bs + B_GROUP);
                    } else {
                        for (int xblk = 2 * half; xblk < 2 + half; ++xblk) {
                            x_pair(xblk, X2, sx2);
                            b_unit(ca, pair, xblk, X2, sx2, Bs);
                        }
                    }
                } else {
                    if (SL == 32 || yq >= NQ) b_unit(ca, pair + 4 * half, xown, X2, sx2, Bs + half * B_GROUP);
                }
            };
            int pair = set * (4 * SG);      // first visibility pair of the stage
            for (int st = b * SPB + set; st < st_end; st += 2, pair += 8 * SG) {
                const int use = st >> 1;
                const uint32_t ta = lane_base + A_COL + 16u * SG * (uint32_t)set;
                uint8_t *Bs = sB + (2 * set + (use & 1)) * B_STAGE;
                // A and B of a group side by side, so that their chains (phase, sine and cosine, split)
                // overlap.  The B buffer's last reader was the stage before the one waited for here
                uint32_t e[16];
                if (yq < NQ) a_unit(cb, vb, pair, round_a, e);
                b_half(pair, Bs, 0);
                if (use > 0) {       // the MMAs of the set's previous stage are done with A
                    wait_or_fail(smem_u32(&s_empty[set]), (uint32_t)((use - 1) & 1), failed, &s_given_up);
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                }
                if (yq < NQ) {
                    tmem_st_16x256b(ta, e);
                    tmem_st_16x256b(ta + (16u << 16), e + 8);
                    a_unit(cb, vb, pair + 4, round_a, e);
                    tmem_st_16x256b(ta + 16u, e);
                    tmem_st_16x256b(ta + 16u + (16u << 16), e + 8);
                }
                b_half(pair, Bs, 1);
                if (yq < NQ) asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&s_full[set]));
                // the set's first stage of a period is on its way: read out the period before
                if (next_fold < st / SPP) {
                    fold(next_fold);
                    ++next_fold;
                }
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&s_unstaged[bar]));
        }
#pragma unroll
        for (int ip = 0; ip < AHEAD; ++ip) load_aterms(ip);
        while (next_fold < n_periods) {
            fold(next_fold);
            ++next_fold;
        }
        if (n_periods == 0)
            for (int i = tid; i < 4 * FFT_S; i += NP) s_img[i] = make_float2(0.f, 0.f);
    }
    // the taper of this thread's epilogue pixels
    float tw_pre[PIXT];
#pragma unroll
    for (int i = 0; i < PIXT; ++i) tw_pre[i] = producer && tid + i * NP < SPIX ? taper[tid + i * NP] : 0.0f;
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    const bool lost = __syncthreads_or(failed);
    if (lost && tid == 0) atomicExch(&g_sep_error, 1);
    if (!lost) {
        // image-domain kernel per pixel: taper * A_p^H I A_q (the transform's lines centre themselves)
        if (producer) {
#pragma unroll
            for (int ip = 0; ip < PIXT; ++ip) {
                const int pix = tid + ip * NP;
                if (pix >= SPIX) break;
                const int y = pix / SL, x = pix % SL;
                M22 P;
#pragma unroll
                for (int c = 0; c < 4; ++c) P.m[c] = s_img[c * FFT_S + y * FFT_P + x];
                if (d.dws != 0.0f) {      // the sums used w_s: the rest of the w offset, exp(i 2 pi (w_s - w0) n')
                    float sn, cs;
                    sincospif(d.dws * g.nprime[pix], &sn, &cs);     // (dws in half turns: exact reduction)
#pragma unroll
                    for (int c = 0; c < 4; ++c)
                        P.m[c] = make_float2(P.m[c].x * cs - P.m[c].y * sn, P.m[c].x * sn + P.m[c].y * cs);
                }
                if (aterms) P = herm_mul_mul(Ap[ip % AHEAD], P, Aq[ip % AHEAD]);
                if (ip + AHEAD < PIXT) load_aterms(ip + AHEAD);
                if (FUSED) {
                    const float tw = tw_pre[ip] * (1.0f / SPIX);      // with the transform's L^-2
#pragma unroll
                    for (int c = 0; c < 4; ++c)
                        s_img[c * FFT_S + y * FFT_P + x] = make_float2(tw * P.m[c].x, tw * P.m[c].y);
                } else {
                    const float tw = tw_pre[ip];
                    o[2 * pix] = make_float4(tw * P.m[0].x, tw * P.m[0].y, tw * P.m[1].x, tw * P.m[1].y);
                    o[2 * pix + 1] = make_float4(tw * P.m[2].x, tw * P.m[2].y, tw * P.m[3].x, tw * P.m[3].y);
                }
            }
        }
        if (FUSED) {
            __syncthreads();
            // one thread per line and polarisation: rows in place, then columns, which leave with
            // 8-byte reductions (the 8 columns x 4 polarisations of a warp are 256 contiguous bytes
            // of a grid row)
            const int pol = tid & 3, ln = tid >> 2;
            float2 *plane = s_img + pol * FFT_S;
            if (tid < 4 * SL) {
                float2 *row = plane + ln * FFT_P;
                fft_line<SL, -1>([&](int n) { return row[n]; }, [&](int k, float2 v) { row[k] = v; });
            }
            __syncthreads();
            if (tid < 4 * SL) {
                const size_t corner = OUT == kGrid ? ((size_t)d.layer * g.N + d.r0) * g.N + d.q0 : 0;
                const size_t pitch = 4 * (OUT == kGrid ? (size_t)g.N : (size_t)SL);
                float2 *dst = (float2 *)o + (corner + ln) * 4 + pol;
                fft_line<SL, -1>([&](int n) { return plane[n * FFT_P + ln]; },
                                 [&](int k, float2 v) {
                                     if (OUT == kGrid) red_add_f2(dst + k * pitch, v);
                                     else dst[k * pitch] = v;
                                 });
            }
        }
    }
    __syncthreads();
    if (mma_warp)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" :: "r"(tmem), "n"(TMEM_COLS));
}

// one CTA per subgrid of one plan (plan index idx[b] or first + b): subgrid images or transforms
template <int L, Out OUT>
__global__ void __launch_bounds__(NT, CTAS)
gridder_sep_kernel(Geometry g, const int32_t *__restrict__ idx, int64_t first, const float4 *__restrict__ vis,
                   const uint8_t *__restrict__ flags, const float4 *__restrict__ aterms,
                   const float *__restrict__ taper, float4 *__restrict__ out) {
    const int sid = idx ? idx[blockIdx.x] : (int)(first + blockIdx.x);
    gridder_sep_body<L, OUT>(g, g.sub[sid], vis, flags, aterms, taper, out + (size_t)blockIdx.x * L * L * 2);
}

// fused: one CTA per subgrid, transformed and added into the grid
template <int L>
__global__ void __launch_bounds__(NT, CTAS)
gridder_sep_fused_kernel(Geometry g, const int32_t *__restrict__ idx, int64_t first, const float4 *__restrict__ vis,
                         const uint8_t *__restrict__ flags, const float4 *__restrict__ aterms,
                         const float *__restrict__ taper, float4 *__restrict__ grid) {
    allow_dependents();
    const int sid = idx ? idx[blockIdx.x] : (int)(first + blockIdx.x);
    gridder_sep_body<L, kGrid>(g, g.sub[sid], vis, flags, aterms, taper, grid);
    complete_after_primary();
}

// the fused kernel's self-test: see idg_selftest_issue_timeout
template <int L>
__global__ void __launch_bounds__(NT, CTAS)
gridder_sep_give_up_kernel(Geometry g, const int32_t *__restrict__ idx, const float4 *__restrict__ vis,
                           const float4 *__restrict__ aterms, const float *__restrict__ taper,
                           float4 *__restrict__ grid) {
    gridder_sep_body<L, kGrid, true>(g, g.sub[idx[blockIdx.x]], vis, nullptr, aterms, taper, grid);
}

template <int L>
idg_status launch_give_up(const Geometry &g, const SubgridSet &set, const void *vis, const void *aterms,
                          const float *taper, void *grid, cudaStream_t s) {
    auto kern = gridder_sep_give_up_kernel<L>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, SepG<L>::SMEM);
    if (e != cudaSuccess) return cuda_fail(e, "separable gridder smem attribute");
    kern<<<(unsigned)set.count, NT, SepG<L>::SMEM, s>>>(g, set.idx, (const float4 *)vis, (const float4 *)aterms, taper,
                                                       (float4 *)grid);
    e = cudaGetLastError();
    return e == cudaSuccess ? IDG_OK : cuda_fail(e, "separable gridder self-test launch");
}

template <int L>
idg_status launch_sep_set(Out out_kind, const Geometry &g, const SubgridSet &set, const void *vis, const uint8_t *flags,
                          const void *aterms, const float *taper, void *out, cudaStream_t s) {
    auto kern = out_kind == kGrid        ? gridder_sep_fused_kernel<L>
                : out_kind == kTransform ? gridder_sep_kernel<L, kTransform>
                                         : gridder_sep_kernel<L, kImage>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, SepG<L>::SMEM);
    if (e != cudaSuccess) return cuda_fail(e, "separable gridder smem attribute");
    kern<<<(unsigned)set.count, NT, SepG<L>::SMEM, s>>>(g, set.idx, set.first, (const float4 *)vis, flags,
                                                       (const float4 *)aterms, taper, (float4 *)out);
    e = cudaGetLastError();
    return e == cudaSuccess ? IDG_OK : cuda_fail(e, out_kind == kGrid ? "separable fused gridder launch" : "separable gridder launch");
}

}  // namespace

bool separable_size(int L) { return L == 32 || L == 24 || L == 16; }

cudaError_t prepare_gridder_sep_batch() {
    cudaError_t e = cudaFuncSetAttribute(gridder_sep_fused_kernel<32>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         SepG<32>::SMEM);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(gridder_sep_fused_kernel<24>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 SepG<24>::SMEM);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(gridder_sep_fused_kernel<16>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 SepG<16>::SMEM);
    return e;
}

// a batch's launch of the fused kernel over one job's items (the shared-memory attribute
// is set by prepare_tcw_batch_kernels, outside graph capture); pdl: see launch_pdl
idg_status launch_gridder_sep_job(const Geometry &g, const SubgridSet &set, const void *vis, const uint8_t *flags,
                                  const void *aterms, const float *taper, void *grid, void *stream, bool pdl) {
    if (set.count <= 0) return IDG_OK;
    cudaStream_t s = (cudaStream_t)stream;
    const unsigned n = (unsigned)set.count;
    const float4 *v = (const float4 *)vis, *at = (const float4 *)aterms;
    float4 *o = (float4 *)grid;
    cudaError_t e;
    switch (g.L) {
    case 32: e = launch_pdl(gridder_sep_fused_kernel<32>, n, NT, SepG<32>::SMEM, s, pdl, g, set.idx, set.first, v, flags, at, taper, o); break;
    case 24: e = launch_pdl(gridder_sep_fused_kernel<24>, n, NT, SepG<24>::SMEM, s, pdl, g, set.idx, set.first, v, flags, at, taper, o); break;
    case 16: e = launch_pdl(gridder_sep_fused_kernel<16>, n, NT, SepG<16>::SMEM, s, pdl, g, set.idx, set.first, v, flags, at, taper, o); break;
    default: return fail(IDG_ERR_UNSUPPORTED, "the separable gridder needs L = 32, 24 or 16");
    }
    return e == cudaSuccess ? IDG_OK : cuda_fail(e, "separable gridder job launch");
}

static idg_status launch_sep_any(Out kind, const Geometry &g, const SubgridSet &set, const void *vis, const uint8_t *flags,
                                 const void *aterms, const float *taper, void *out, void *stream) {
    if (!separable_size(g.L) || !g.separable)
        return fail(IDG_ERR_UNSUPPORTED, "the separable gridder needs L = 32, 24 or 16 and a separable plan");
    if (set.count <= 0) return IDG_OK;
    switch (g.L) {
    case 32: return launch_sep_set<32>(kind, g, set, vis, flags, aterms, taper, out, (cudaStream_t)stream);
    case 24: return launch_sep_set<24>(kind, g, set, vis, flags, aterms, taper, out, (cudaStream_t)stream);
    default: return launch_sep_set<16>(kind, g, set, vis, flags, aterms, taper, out, (cudaStream_t)stream);
    }
}

idg_status launch_gridder_sep(const Geometry &g, const SubgridSet &set, const void *vis, const uint8_t *flags,
                              const void *aterms, const float *taper, void *out, void *stream) {
    return launch_sep_any(kImage, g, set, vis, flags, aterms, taper, out, stream);
}

idg_status launch_gridder_sep_transform(const Geometry &g, const SubgridSet &set, const void *vis, const uint8_t *flags,
                                        const void *aterms, const float *taper, void *out, void *stream) {
    return launch_sep_any(kTransform, g, set, vis, flags, aterms, taper, out, stream);
}

idg_status launch_gridder_sep_fused(const Geometry &g, const SubgridSet &set, const void *vis, const uint8_t *flags,
                                    const void *aterms, const float *taper, void *grid, void *stream) {
    return launch_sep_any(kGrid, g, set, vis, flags, aterms, taper, grid, stream);
}

idg_status launch_gridder_sep_give_up(const Geometry &g, const SubgridSet &set, const void *vis, const void *aterms,
                                      const float *taper, void *grid, void *stream) {
    if (!separable_size(g.L) || !g.separable || !set.idx)
        return fail(IDG_ERR_UNSUPPORTED, "the separable gridder needs L = 32, 24 or 16 and a separable plan");
    if (set.count <= 0) return IDG_OK;
    switch (g.L) {
    case 32: return launch_give_up<32>(g, set, vis, aterms, taper, grid, (cudaStream_t)stream);
    case 24: return launch_give_up<24>(g, set, vis, aterms, taper, grid, (cudaStream_t)stream);
    default: return launch_give_up<16>(g, set, vis, aterms, taper, grid, (cudaStream_t)stream);
    }
}

idg_status read_sep_error(int *code) {
    int zero = 0, v = 0;
    cudaError_t e = cudaMemcpyFromSymbol(&v, g_sep_error, sizeof(int));
    if (e == cudaSuccess) e = cudaMemcpyToSymbol(g_sep_error, &zero, sizeof(int));
    if (e != cudaSuccess) return cuda_fail(e, "reading the separable gridder error word");
    *code = v;
    return IDG_OK;
}

}  // namespace idg
