// Separable degridder on the tensor cores (tcgen05), L = 32, 24 and 16.
//
// The visibilities of Algorithm 2 from the corrected subgrid image P_q(x, y)
// (taper and A_p P A_q^H applied) are
//   y_kq = sum_{x,y} P_q(x, y) exp(-i (a_k X + b_k Y + c_k n'(x, y))).
// With the split n' = s(x) + t(y) + r(x, y) used by the separable gridder and
// exp(-i c r) = 1 - i c r + O(theta^2 / 2) (theta = max |c| max |r|, checked
// by the plan),
//   y_kq = sum_y Ey*_k(y) [T0_kq(y) - i c_k T1_kq(y)],
//   T_mkq(y) = sum_x Ex*_k(x) Q_mq(x, y),  Q0 = P, Q1 = P r,
//   Ex*_k(x) = exp(-i (a_k X + c_k s(x))),  Ey*_k(y) = exp(-i (b_k Y + c_k t(y))).
// Both terms are one complex matrix product on the tensor cores,
//   T_kq(y) = sum_x Ex*_k(x) Q0_q(x, y) + sum_x (-i c_k Ex*_k(x)) Q1_q(x, y),
// with rows the 128 visibilities of a tile, columns (q, y, re/im) and K = (x, cos/sin)
// twice (m = 0, then m = 1).  The sum over y with the visibility's own phasors,
// y_kq = sum_y Ey*_k(y) T_kq(y), runs on the CUDA cores (FP32, round to nearest).
//
// GEMM.  A holds (cos, sin) of Ex_k(x) (m = 0) and c sigma (-sin, cos) (m = 1, sigma a
// power of two with max |c| sigma <= 1), one tensor-memory row per visibility; B holds
// the 2 x 2 real embedding of Q0 = s P and of Q1 = s r P / sigma (s a power of two per
// subgrid): row re of (q, y) is (Re Q, Im Q), row im (Im Q, -Re Q).  The embedding sits
// on the image side, where it is formed once per subgrid, not per visibility.  The
// m = 0 operands are split into FP16 hi + lo (A's hi a multiple of 2^-11) and take
// A_hi B_hi + A_hi B_lo + A_lo B_hi; the m = 1 term (at most theta relative) takes
// A_hi B_hi.  Per K step of 16 (8 x): four MMAs of N = 128 (96 at L = 24) for two of
// the four polarisations, then the same for the other two (all four at L = 16).  The
// accumulation is 16 MMAs long, so no folds are needed.
//
// Schedule.  One CTA per subgrid, two CTAs per SM (256 tensor-memory columns and 105 KB of
// shared memory each): the prologue of one, and the sums of one, run under the other's
// MMAs.  The prologue brings the grid rows by bulk copy, transforms them (one thread per
// line and polarisation), applies A-terms and taper in registers and writes B.  Then per
// tile a visibility belongs to two threads (warps w and w + 4): each forms A for half of
// the x and the y phasors and the sum for half of the y; the two meet through shared
// memory, each finishing two polarisations.  A ninth warp issues the MMAs.  The phase
// coefficients of the next tile are formed while the last part's MMAs run, the outputs
// of a tile and its Ey* while the first part's do.  X, s(x) and t(y) are kernel-parameter
// constants: tables in shared memory cost 430 of 919 wavefronts per tile.
// Tensor memory: accumulator at 0, A at 128 (hi, lo and m = 1, a column per x).
//
// What bounds it, and what the choices measured (LOFAR-like plan of 45.9 k subgrids of about
// 1600 visibilities, 73.9 M; and A-terms every 16 s, 18.4 M in 89.4 k of about 206):
//   one CTA per SM, embedding on the visibility side, Ey
//   table and re/im exchange in shared memory                11.32 ms    7.51 ms
//   this layout                                               8.35       4.69
//   constants instead of tables                               8.04       4.53
//   one thread per transform line, straight from the rows     7.92       4.36
//   A-terms two pixels ahead                                  7.93       4.24
//   failures seen by every store                              7.88       4.27
// The tensor pipe is 49 % busy (16 cycles per visibility at full rate), issue slots 46 %: a
// CTA's chain per tile (A 1250, MMAs 2 x 1024, sums 2 x 500 cycles, measured alone) leaves
// the tensor cores to the other CTA for just over half its length, and tensor memory has no
// room for a second A beside the accumulator.  Short subgrids are bound by the prologue
// (8 k of 12 k cycles).  Measured and not kept: a coefficient warp (8.53 ms: the
// coefficients were already hidden), MMAs issued by a worker (9.2: issuing blocks the
// warp), A's first half formed during the sums (spills: + 25 %).
// Every wait is bounded.  After one that runs out a thread skips every later wait, the MMA thread
// issues no more MMAs, the error word is set and nothing is written any more (the visibilities of
// the tiles before it have been).
#include "batch_jobs.cuh"
#include "device_common.cuh"
#include "fft_impl.cuh"
#include "tc_common.cuh"

namespace idg {

// device error word of the separable degridder (0 = ok); read and cleared by
// idg_device_errors
__device__ int g_sepd_error = 0;

namespace {

using namespace dev;
using namespace tc;

constexpr int NWW = 8;                          // worker warps
constexpr int MMA_WARP = NWW;
constexpr int NT = NWW * 32 + 32;
constexpr int CTAS = 2;                         // per SM
constexpr int TV = 128;                         // visibilities per tile (rows of A and D)
constexpr uint32_t TMEM_COLS = 256;             // two CTAs share an SM's 512

// Layout for subgrid size L (32, 24 or 16)
template <int L>
struct SepD {
    static constexpr int SL = L, SPIX = L * L;
    static constexpr int KT = L / 8;                // K steps of 16 (8 x, re/im) over the L x
    // a tile's products go in PARTS rounds of QH polarisations into one accumulator of PN columns
    static constexpr int QH = L == 16 ? 4 : 2, PARTS = 4 / QH, PN = QH * 2 * L;
    // D column (B row) of (q', y, re/im) in a part: 2 L q' + 2 YB (y / YB) + YB (re/im) + y % YB
    static constexpr int YB = L == 24 ? 4 : 8;
    // B (fixed per subgrid), each [KT][part][PN rows][16 K]: Q0 hi, Q0 lo, Q1 hi
    static constexpr int TB = 8 * L * 32;           // one K step: 8 L rows x 32 bytes
    static constexpr int B0L = KT * TB, B1H = 2 * KT * TB, B_BYTES = 3 * KT * TB;
    // prologue scratch over B: the subgrid's grid rows, then (with 4 float2 of row padding) its image,
    // pixel by pixel; behind them the transform planes
    static constexpr int FFT_P = PolPlanes<L>::P, FFT_S = PolPlanes<L>::STRIDE;
    static constexpr int PIX_P = 4 * L + 4, FFT_OFF = L * PIX_P * 8, FFT_END = FFT_OFF + 4 * FFT_S * 8;
    static constexpr int PART_OFF = B_BYTES > FFT_END ? B_BYTES : FFT_END;
    static constexpr int SMEM = PART_OFF + 2 * 2 * TV * 16;      // [2 tiles][2 pol pairs][TV] float4 (y halves meet)
    // tensor memory: accumulator, then A hi, lo and m = 1, one column per x
    static constexpr uint32_t A_COL = PN;
    static constexpr uint32_t IDESC = idesc_m128(PN);
    // a worker's half of the x (A) and of the y (sum) of its visibility, in chunks
    static constexpr int H = L / 2, XCH = H % 8 == 0 ? 8 : 4;
    // image pixels by worker warp: tiles of 8 y x 4 x, one B core matrix row set per warp store
    static constexpr int NTILE = (L / 8) * (L / 4), TPW = (NTILE + NWW - 1) / NWW;
    static_assert(L == 32 || L == 24 || L == 16, "subgrid sizes of the separable kernels");
    static_assert(A_COL + 3 * L <= TMEM_COLS, "accumulator and A in the CTA's tensor memory");
    static_assert(PN % 16 == 0 && PN <= 256, "MMA N");
    static_assert(H % YB == 0 && H % XCH == 0, "whole chunks per worker");
    static_assert(FFT_OFF % 16 == 0 && PART_OFF % 16 == 0, "16-byte aligned areas");
    static_assert(CTAS * (SMEM + 2048) <= 227 * 1024, "shared memory of the SM's CTAs");
    static_assert(L <= 32, "one grid row per lane of warp 0");
};

// the two warps of a lane quarter (constant barrier numbers: a register would reserve all 16)
__device__ __forceinline__ void pair_sync(int quarter) {
    switch (quarter) {
    case 0: asm volatile("bar.sync 1, 64;" ::: "memory"); break;
    case 1: asm volatile("bar.sync 2, 64;" ::: "memory"); break;
    case 2: asm volatile("bar.sync 3, 64;" ::: "memory"); break;
    default: asm volatile("bar.sync 4, 64;" ::: "memory"); break;
    }
}

// A of a visibility's x from X0: (cs, sn) of Ex, its FP16 hi and lo parts and the m = 1 factor,
// into its tensor-memory row.  X and s(x) are instruction constants (kernel parameters), so
// the loop reads no memory.
template <int L, int X0>
__device__ __forceinline__ void form_a(const Geometry &g, uint32_t lane_base, float csig, float ca, float cc) {
    using C = SepD<L>;
    constexpr int SL = L, H = C::H, XCH = C::XCH;
    constexpr float magic_1 = 6144.0f;      // split at multiples of 2^-11
    const float cz = cc * csig;
    const f2_t cz2 = f2_pack(cz, cz), nz2 = f2_pack(-cz, -cz);
#pragma unroll
    for (int x0 = X0; x0 < X0 + H; x0 += XCH) {
        uint32_t hi[XCH], lo[XCH], m1[XCH];
#pragma unroll
        for (int i = 0; i < XCH; i += 2) {
            float sn0, cs0, sn1, cs1;
            __sincosf(fmaf(cc, g.sep_s[x0 + i], ca * (float)(x0 + i - SL / 2)), &sn0, &cs0);
            __sincosf(fmaf(cc, g.sep_s[x0 + i + 1], ca * (float)(x0 + i + 1 - SL / 2)), &sn1, &cs1);
            const f2_t c2 = f2_pack(cs0, cs1), s2 = f2_pack(sn0, sn1);
            f2_t hc, lc, hs, ls;
            f2_split(c2, magic_1, hc, lc);
            f2_split(s2, magic_1, hs, ls);
            pack_pairs(hc, hs, hi[i], hi[i + 1]);
            pack_pairs(lc, ls, lo[i], lo[i + 1]);
            pack_pairs(f2_mul(nz2, s2), f2_mul(cz2, c2), m1[i], m1[i + 1]);
        }
        const uint32_t ta = lane_base + C::A_COL + (uint32_t)x0;
        tmem_st(ta, hi);
        tmem_st(ta + SL, lo);
        tmem_st(ta + 2 * SL, m1);
    }
    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}

// Ey* of its y from Y0 as pairs (cs_y, cs_y+1), (sn_y, sn_y+1)
template <int L, int Y0>
__device__ __forceinline__ void form_ey(const Geometry &g, float cb, float cc, f2_t (&ec)[L / 4], f2_t (&es)[L / 4]) {
    constexpr int SL = L, H = L / 2;
#pragma unroll
    for (int j = 0; j < H / 2; ++j) {
        float s0, c0, s1, c1;
        __sincosf(fmaf(cc, g.sep_t[Y0 + 2 * j], cb * (float)(Y0 + 2 * j - SL / 2)), &s0, &c0);
        __sincosf(fmaf(cc, g.sep_t[Y0 + 2 * j + 1], cb * (float)(Y0 + 2 * j + 1 - SL / 2)), &s1, &c1);
        ec[j] = f2_pack(c0, c1);
        es[j] = f2_pack(s0, s1);
    }
}

// Visibilities of subgrid d of geometry g from its image src[L][L][4], or with
// FUSED from the grid src[layer][N][N][4]: split and transformed in shared memory
// first (Algorithm 2: split from the master grid, "IFFT", image-domain kernel, sum).
// NEVER: the self-test's form, whose MMA thread gives up at once.
template <int L, bool FUSED, bool NEVER = false>
__device__ __forceinline__ void degridder_sep_body(const Geometry &g, const DevSubgrid d,
                                                   const float4 *__restrict__ src, const uint8_t *__restrict__ flags,
                                                   const float4 *__restrict__ aterms, const float *__restrict__ taper,
                                                   float4 *__restrict__ vis_out) {
    using C = SepD<L>;
    constexpr int SL = C::SL, SPIX = C::SPIX, KT = C::KT, H = C::H, YB = C::YB, QH = C::QH;
    extern __shared__ __align__(1024) uint8_t smem[];
    float4 *s_part = (float4 *)(smem + C::PART_OFF);
    __shared__ uint32_t s_tmem;
    __shared__ __align__(8) uint64_t s_afull, s_dfull, s_dempty, s_drain, s_gbar;
    __shared__ int s_given_up;
    __shared__ float s_red[NWW];

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int kp = d.kp, n_tiles = (kp + TV - 1) / TV;

    if (warp == MMA_WARP) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     :: "r"(smem_u32(&s_tmem)), "n"(TMEM_COLS));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    if (warp == 0) {
        // barriers by lane 0; then one bulk copy per lane: the subgrid's grid rows (32 L bytes
        // each, contiguous in the grid)
        if (lane == 0) {
            s_given_up = 0;
            mbar_init(smem_u32(&s_afull), NWW);
            mbar_init(smem_u32(&s_dfull), 1);
            mbar_init(smem_u32(&s_dempty), NWW);
            mbar_init(smem_u32(&s_drain), 1);
            mbar_init(smem_u32(&s_gbar), 1);
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
            if (FUSED) mbar_expect_tx(smem_u32(&s_gbar), SPIX * 32);
        }
        __syncwarp();
        if (FUSED && lane < SL) {
            const float4 *gsrc = src + (size_t)d.layer * g.N * g.N * 2;
            bulk_g2s(smem_u32(smem + lane * SL * 32), gsrc + 2 * ((size_t)(d.r0 + lane) * g.N + d.q0), SL * 32,
                     smem_u32(&s_gbar));
        }
    }

    // workers: visibility 32 (warp % 4) + lane of the tile, x and y half warp / 4
    const int quarter = warp & 3, half = warp >> 2, row = 32 * quarter + lane;
    // its coordinates, loaded one tile ahead (the first tile's before the prologue)
    const float4 *uvw2 = (const float4 *)g.uvw_f2;
    const float4 *sc2 = (const float4 *)g.scale_f2;
    const int dt = TV / d.nc, dc = TV - dt * d.nc;
    int vt = row / d.nc, vc = row - vt * d.nc;           // timestep and channel in the subgrid
    float4 ruv = make_float4(0.f, 0.f, 0.f, 0.f), rsc = ruv;
    float2 rw = make_float2(0.f, 0.f);
    uint32_t rvi = 0xFFFFFFFFu;                          // output index, bit 31 = flagged; all ones: none
    auto load_raw = [&](int k) {
        rvi = 0xFFFFFFFFu;
        if (k < kp) {
            const size_t bt = (size_t)d.bl * g.n_t + d.t0 + vt;
            const int c = d.c0 + vc;
            ruv = uvw2[2 * bt];
            rw = *(const float2 *)(uvw2 + 2 * bt + 1);
            rsc = sc2[c];
            rvi = (uint32_t)(bt * g.n_chan + c);
            if (flags && flags[rvi]) rvi |= 0x80000000u;
        }
        vt += dt;
        vc += dc;
        if (vc >= d.nc) {
            vc -= d.nc;
            ++vt;
        }
    };
    if (warp < NWW) load_raw(row);
    __syncthreads();      // the copies' barrier is initialised

    // ---- prologue: the corrected image P = taper A_p I A_q^H, this thread's pixels in registers
    if (FUSED) {
        bool late = false;
        wait_or_fail(smem_u32(&s_gbar), 0u, late, &s_given_up);
        // one thread per line and polarisation: columns from the grid rows, then rows into the image
        const int pol = tid & 3, ln = tid >> 2;
        const float2 *src_col = (const float2 *)smem + 4 * ln + pol;
        float2 *plane = (float2 *)(smem + C::FFT_OFF) + pol * C::FFT_S;
        if (tid < 4 * SL)
            fft_line<SL, +1>([&](int n) { return src_col[n * 4 * SL]; },
                             [&](int k, float2 v) { plane[k * C::FFT_P + ln] = v; });
        __syncthreads();
        if (tid < 4 * SL) {
            const float2 *row = plane + ln * C::FFT_P;
            float2 *dst = (float2 *)smem + ln * C::PIX_P + pol;
            fft_line<SL, +1>([&](int n) { return row[n]; }, [&](int k, float2 v) { dst[4 * k] = v; });
        }
    }
    // the A-terms of this thread's pixels, two pixels ahead
    constexpr int AHEAD = C::TPW < 2 ? C::TPW : 2;
    M22 P[C::TPW], Ap[AHEAD], Aq[AHEAD];
    auto load_aterms = [&](int i) {
        const int tile = warp + NWW * i;
        if (aterms && warp < NWW && tile < C::NTILE) {
            const int y = 8 * (tile / (SL / 4)) + (lane >> 2), x = 4 * (tile % (SL / 4)) + (lane & 3);
            const float4 *base = aterms + 2 * ((size_t)d.slot * g.n_stations) * SPIX + 2 * (y * SL + x);
            Ap[i % AHEAD] = load_m22(base + 2 * (size_t)d.st_p * SPIX);
            Aq[i % AHEAD] = load_m22(base + 2 * (size_t)d.st_q * SPIX);
        }
    };
#pragma unroll
    for (int i = 0; i < AHEAD; ++i) load_aterms(i);
    if (FUSED) __syncthreads();
    if (warp < NWW) {
        float m = 0.0f;
#pragma unroll
        for (int i = 0; i < C::TPW; ++i) {
            const int tile = warp + NWW * i;
            if (tile >= C::NTILE) break;
            const int y = 8 * (tile / (SL / 4)) + (lane >> 2), x = 4 * (tile % (SL / 4)) + (lane & 3), pix = y * SL + x;
            P[i] = load_m22(FUSED ? (const float4 *)smem + y * (C::PIX_P / 2) + 2 * x : src + 2 * pix);
            if (d.dws != 0.0f) {      // the sums use w_s: the rest of the w offset, exp(-i 2 pi (w_s - w0) n')
                float sn, cs;
                sincospif(d.dws * g.nprime[pix], &sn, &cs);     // (dws in half turns: exact reduction)
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    P[i].m[q] = make_float2(P[i].m[q].x * cs + P[i].m[q].y * sn, P[i].m[q].y * cs - P[i].m[q].x * sn);
            }
            if (aterms) P[i] = mul_mul_herm(Ap[i % AHEAD], P[i], Aq[i % AHEAD]);
            if (i + AHEAD < C::TPW) load_aterms(i + AHEAD);
            const float tw = FUSED ? taper[pix] * (1.0f / SPIX) : taper[pix];      // with the transform's L^-2
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                P[i].m[q] = make_float2(tw * P[i].m[q].x, tw * P[i].m[q].y);
                m = fmaxf(m, fmaxf(fabsf(P[i].m[q].x), fabsf(P[i].m[q].y)));
            }
        }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, off));
        if (lane == 0) s_red[warp] = m;
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();      // every pixel is in registers: the scratch area may become B
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = s_tmem;
    float inv_scale;
    {
        float m = 0.0f;
#pragma unroll
        for (int w = 0; w < NWW; ++w) m = fmaxf(m, s_red[w]);
        int e2 = 0;
        if (m > 0.0f) frexpf(m, &e2);
        const float scale = ldexpf(1.0f, 10 - e2);
        inv_scale = ldexpf(1.0f, e2 - 10);
        // B: Q0 = scale P (hi and lo), Q1 = scale r P / sigma (hi).  Row re of (q, y) is (Re Q, Im Q)
        // over K = (x, cs/sn), row im (Im Q, -Re Q): the re row's halves swapped, the new high one negated
        if (warp < NWW) {
            const float rs = scale / g.c_scale;
#pragma unroll
            for (int i = 0; i < C::TPW; ++i) {
                const int tile = warp + NWW * i;
                if (tile >= C::NTILE) break;
                const int y = 8 * (tile / (SL / 4)) + (lane >> 2), x = 4 * (tile % (SL / 4)) + (lane & 3);
                const float rr = g.sep[2 * SL + y * SL + x] * rs;
                uint8_t *Bx = smem + (x >> 3) * C::TB + ((x >> 2) & 1) * kLBO + (x & 3) * 4;
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const float2 p = P[i].m[q];
                    uint32_t h0, l0;
                    split_e(p.x * scale, p.y * scale, h0, l0);
                    const uint32_t h1 = pack_f16x2(p.x * rr, p.y * rr);
#pragma unroll
                    for (int r = 0; r < 2; ++r) {
                        const int n = 2 * SL * q + 2 * YB * (y / YB) + YB * r + y % YB;
                        uint8_t *b = Bx + (n >> 3) * kSBO + (n & 7) * 16;
                        *(uint32_t *)b = r ? __byte_perm(h0, 0u, 0x1032u) ^ 0x80000000u : h0;
                        *(uint32_t *)(b + C::B0L) = r ? __byte_perm(l0, 0u, 0x1032u) ^ 0x80000000u : l0;
                        *(uint32_t *)(b + C::B1H) = r ? __byte_perm(h1, 0u, 0x1032u) ^ 0x80000000u : h1;
                    }
                }
            }
        }
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    __syncthreads();      // B complete

    bool failed = false;
    if (warp == MMA_WARP) {
        if (lane == 0) {
            const uint64_t db0 = smem_desc(smem_u32(smem));
            const uint32_t at = tmem + C::A_COL;
            for (int t = 0; t < n_tiles && !failed; ++t) {
                poll_or_fail<NEVER>(smem_u32(&s_afull), (uint32_t)(t & 1), failed, &s_given_up);
                for (int p = 0; p < C::PARTS; ++p) {
                    const int n = t * C::PARTS + p;
                    if (n > 0) poll_or_fail<NEVER>(smem_u32(&s_dempty), (uint32_t)((n - 1) & 1), failed, &s_given_up);
                    if (failed) break;
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    const uint64_t dbp = db0 + (uint64_t)((p * C::PN * 32) >> 4);
#pragma unroll
                    for (int kk = 0; kk < KT; ++kk) {
                        const uint64_t db = dbp + (uint64_t)((kk * C::TB) >> 4);
                        const uint32_t ak = at + 8u * kk;
                        mma_ta_i(tmem, ak, db, C::IDESC, kk > 0 ? 1u : 0u);                                 // hi x Q0 hi
                        mma_ta_i(tmem, ak, db + (uint64_t)(C::B0L >> 4), C::IDESC, 1u);                     // hi x Q0 lo
                        mma_ta_i(tmem, ak + SL, db, C::IDESC, 1u);                                          // lo x Q0 hi
                        mma_ta_i(tmem, ak + 2 * SL, db + (uint64_t)(C::B1H >> 4), C::IDESC, 1u);            // m = 1
                    }
                    commit(smem_u32(&s_dfull));
                }
            }
            commit(smem_u32(&s_drain));
            if (!mbar_wait(smem_u32(&s_drain), 0u)) s_given_up = 1;     // bounded: let own MMAs finish before the free
        }
    } else {
        const uint32_t lane_base = tmem + ((uint32_t)(32 * quarter) << 16);
        const float csig = g.c_scale;
        // phase coefficients of the tile's visibility from float pairs (error-free products and
        // sums, rounded once), and its output index; formed one tile ahead, while MMAs run
        float ca = 0.f, cb = 0.f, cc = 0.f;
        uint32_t vi = 0xFFFFFFFFu;
        auto form_coef = [&](float &a, float &b, float &c, uint32_t &v) {
            a = b = c = 0.f;
            v = rvi;
            if (rvi != 0xFFFFFFFFu) {
                a = pair_coef(ruv.x, ruv.y, rsc.x, rsc.y, d.a0h, d.a0l);
                b = pair_coef(ruv.z, ruv.w, rsc.x, rsc.y, d.b0h, d.b0l);
                c = pair_coef(rw.x, rw.y, rsc.z, rsc.w, d.csh, d.csl);
            }
        };
        // the two y halves of a visibility meet: each half's warp finishes two polarisations, own
        // their sums over its y, the other half's through shared memory (after the next tile's A)
        float4 own = make_float4(0.f, 0.f, 0.f, 0.f);
        uint32_t ovi = 0xFFFFFFFFu;
        auto finish = [&](int t) {
            pair_sync(quarter);
            const float4 o = s_part[((t & 1) * 2 + half) * TV + row];
            // (read after the pair has met: a wait of the other half that ran out counts too)
            if (ovi != 0xFFFFFFFFu && !s_given_up) {
                float4 v = make_float4((own.x + o.x) * inv_scale, (own.y + o.y) * inv_scale, (own.z + o.z) * inv_scale,
                                       (own.w + o.w) * inv_scale);
                if (ovi & 0x80000000u) v = make_float4(0.f, 0.f, 0.f, 0.f);      // flagged
                // as two 8-byte stores: a complex64 output may start at any multiple of 8 bytes (the other
                // degridders choose by the address, store_vis; here one 16-byte store took the same time)
                float2 *out = (float2 *)vis_out + 4 * (size_t)(ovi & 0x7FFFFFFFu) + 2 * half;
                out[0] = make_float2(v.x, v.y);
                out[1] = make_float2(v.z, v.w);
            }
        };
        form_coef(ca, cb, cc, vi);
        load_raw(TV + row);
        for (int t = 0; t < n_tiles; ++t) {
            const bool active = t * TV + 32 * quarter < kp;      // the same for the whole warp
            // A: this half's x of the visibility's row (the last part of the previous tile was waited
            // for below, so the MMAs are done with A)
            if (active) {
                if (half) form_a<L, H>(g, lane_base, csig, ca, cc);
                else form_a<L, 0>(g, lane_base, csig, ca, cc);
            }
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&s_afull));
            if (t > 0) finish(t - 1);      // every warp was active in the tile before
            // Ey* of this half's y, as pairs (cs_y, cs_y+1), (sn_y, sn_y+1), while the MMAs run
            f2_t ec[H / 2], es[H / 2];
            if (active) {
                if (half) form_ey<L, H>(g, cb, cc, ec, es);
                else form_ey<L, 0>(g, cb, cc, ec, es);
            }
            ovi = vi;
            float acc[4][2];
#pragma unroll
            for (int p = 0; p < C::PARTS; ++p) {
                if (p == C::PARTS - 1 && t + 1 < n_tiles) {
                    form_coef(ca, cb, cc, vi);
                    load_raw((t + 2) * TV + row);
                }
                wait_or_fail(smem_u32(&s_dfull), (uint32_t)((t * C::PARTS + p) & 1), failed, &s_given_up);
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                if (active) {
                    // y_q = sum_y (cs - i sn) T_q(y): Re = sum cs Tr + sn Ti, Im = sum cs Ti - sn Tr
#pragma unroll
                    for (int qp = 0; qp < QH; qp += 2) {
                        f2_t re[2], ip[2], im[2];
#pragma unroll
                        for (int e = 0; e < 2; ++e) re[e] = ip[e] = im[e] = 0ull;
#pragma unroll
                        for (int yc = 0; yc < H / YB; ++yc) {
                            uint32_t r[2][2 * YB];
#pragma unroll
                            for (int e = 0; e < 2; ++e)
                                tmem_ld_nowait(lane_base + (uint32_t)(2 * SL * (qp + e) + half * SL + 2 * YB * yc), r[e]);
#pragma unroll
                            for (int e = 0; e < 2; ++e) tmem_wait_ld(r[e]);
#pragma unroll
                            for (int e = 0; e < 2; ++e)
#pragma unroll
                                for (int j = 0; j < YB / 2; ++j) {
                                    const f2_t Tr = f2_pack(__uint_as_float(r[e][2 * j]), __uint_as_float(r[e][2 * j + 1]));
                                    const f2_t Ti = f2_pack(__uint_as_float(r[e][YB + 2 * j]),
                                                            __uint_as_float(r[e][YB + 2 * j + 1]));
                                    const f2_t c2 = ec[YB / 2 * yc + j], s2 = es[YB / 2 * yc + j];
                                    re[e] = f2_fma(c2, Tr, re[e]);
                                    ip[e] = f2_fma(c2, Ti, ip[e]);
                                    im[e] = f2_fma(s2, Tr, im[e]);
                                    re[e] = f2_fma(s2, Ti, re[e]);
                                }
                        }
#pragma unroll
                        for (int e = 0; e < 2; ++e) {
                            float a0, a1, b0, b1, c0, c1;
                            f2_unpack(re[e], a0, a1);
                            f2_unpack(ip[e], b0, b1);
                            f2_unpack(im[e], c0, c1);
                            acc[p * QH + qp + e][0] = a0 + a1;
                            acc[p * QH + qp + e][1] = (b0 + b1) - (c0 + c1);
                        }
                    }
                }
                asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&s_dempty));
            }
            if (active) {
                s_part[((t & 1) * 2 + (half ^ 1)) * TV + row] =
                    half ? make_float4(acc[0][0], acc[0][1], acc[1][0], acc[1][1])
                         : make_float4(acc[2][0], acc[2][1], acc[3][0], acc[3][1]);
                own = half ? make_float4(acc[2][0], acc[2][1], acc[3][0], acc[3][1])
                           : make_float4(acc[0][0], acc[0][1], acc[1][0], acc[1][1]);
            }
        }
        if (n_tiles > 0 && (n_tiles - 1) * TV + 32 * quarter < kp) finish(n_tiles - 1);
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (tid == 0 && s_given_up) atomicExch(&g_sepd_error, 1);
    if (warp == MMA_WARP)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" :: "r"(tmem), "n"(TMEM_COLS));
}

// one CTA per subgrid of one plan (plan index idx[b] or first + b; image b of sub)
template <int L>
__global__ void __launch_bounds__(NT, CTAS)
degridder_sep_kernel(Geometry g, const int32_t *__restrict__ idx, int64_t first, const float4 *__restrict__ sub,
                     const uint8_t *__restrict__ flags, const float4 *__restrict__ aterms,
                     const float *__restrict__ taper, float4 *__restrict__ vis_out) {
    const int sid = idx ? idx[blockIdx.x] : (int)(first + blockIdx.x);
    degridder_sep_body<L, false>(g, g.sub[sid], sub + (size_t)blockIdx.x * L * L * 2, flags, aterms, taper, vis_out);
}

// fused: one CTA per subgrid, read from the grid
template <int L>
__global__ void __launch_bounds__(NT, CTAS)
degridder_sep_fused_kernel(Geometry g, const int32_t *__restrict__ idx, int64_t first, const float4 *__restrict__ grid,
                           const uint8_t *__restrict__ flags, const float4 *__restrict__ aterms,
                           const float *__restrict__ taper, float4 *__restrict__ vis_out) {
    allow_dependents();
    const int sid = idx ? idx[blockIdx.x] : (int)(first + blockIdx.x);
    degridder_sep_body<L, true>(g, g.sub[sid], grid, flags, aterms, taper, vis_out);
    complete_after_primary();
}

// the fused kernel's self-test: see idg_selftest_issue_timeout
template <int L>
__global__ void __launch_bounds__(NT, CTAS)
degridder_sep_give_up_kernel(Geometry g, const int32_t *__restrict__ idx, const float4 *__restrict__ grid,
                             const float4 *__restrict__ aterms, const float *__restrict__ taper,
                             float4 *__restrict__ vis_out) {
    degridder_sep_body<L, true, true>(g, g.sub[idx[blockIdx.x]], grid, nullptr, aterms, taper, vis_out);
}

template <int L>
idg_status launch_give_up(const Geometry &g, const SubgridSet &set, const void *grid, const void *aterms,
                          const float *taper, void *vis_out, cudaStream_t s) {
    auto kern = degridder_sep_give_up_kernel<L>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, SepD<L>::SMEM);
    if (e != cudaSuccess) return cuda_fail(e, "separable degridder smem attribute");
    kern<<<(unsigned)set.count, NT, SepD<L>::SMEM, s>>>(g, set.idx, (const float4 *)grid, (const float4 *)aterms, taper,
                                                       (float4 *)vis_out);
    e = cudaGetLastError();
    return e == cudaSuccess ? IDG_OK : cuda_fail(e, "separable degridder self-test launch");
}

template <int L>
idg_status launch_sepd_set(bool fused, const Geometry &g, const SubgridSet &set, const void *src, const uint8_t *flags,
                           const void *aterms, const float *taper, void *vis_out, cudaStream_t s) {
    auto kern = fused ? degridder_sep_fused_kernel<L> : degridder_sep_kernel<L>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, SepD<L>::SMEM);
    if (e != cudaSuccess) return cuda_fail(e, "separable degridder smem attribute");
    kern<<<(unsigned)set.count, NT, SepD<L>::SMEM, s>>>(g, set.idx, set.first, (const float4 *)src, flags,
                                                       (const float4 *)aterms, taper, (float4 *)vis_out);
    e = cudaGetLastError();
    return e == cudaSuccess ? IDG_OK
                            : cuda_fail(e, fused ? "separable fused degridder launch" : "separable degridder launch");
}

}  // namespace

cudaError_t prepare_sep_batch_kernels() {
    cudaError_t e = prepare_gridder_sep_batch();
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(degridder_sep_fused_kernel<32>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 SepD<32>::SMEM);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(degridder_sep_fused_kernel<24>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 SepD<24>::SMEM);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(degridder_sep_fused_kernel<16>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 SepD<16>::SMEM);
    return e;
}


idg_status launch_degridder_sep(const Geometry &g, const SubgridSet &set, const void *sub, const uint8_t *flags,
                                const void *aterms, const float *taper, void *vis_out, void *stream) {
    if (!separable_size(g.L) || !g.separable)
        return fail(IDG_ERR_UNSUPPORTED, "the separable degridder needs L = 32, 24 or 16 and a separable plan");
    if (set.count <= 0) return IDG_OK;
    switch (g.L) {
    case 32: return launch_sepd_set<32>(false, g, set, sub, flags, aterms, taper, vis_out, (cudaStream_t)stream);
    case 24: return launch_sepd_set<24>(false, g, set, sub, flags, aterms, taper, vis_out, (cudaStream_t)stream);
    default: return launch_sepd_set<16>(false, g, set, sub, flags, aterms, taper, vis_out, (cudaStream_t)stream);
    }
}

// a batch's launch of the fused kernel over one job's items (the shared-memory attribute
// is set by prepare_tcw_batch_kernels, outside graph capture); pdl: see launch_pdl
idg_status launch_degridder_sep_job(const Geometry &g, const SubgridSet &set, const void *grid, const uint8_t *flags,
                                    const void *aterms, const float *taper, void *vis_out, void *stream, bool pdl) {
    if (set.count <= 0) return IDG_OK;
    cudaStream_t s = (cudaStream_t)stream;
    const unsigned n = (unsigned)set.count;
    const float4 *gr = (const float4 *)grid, *at = (const float4 *)aterms;
    float4 *o = (float4 *)vis_out;
    cudaError_t e;
    switch (g.L) {
    case 32: e = launch_pdl(degridder_sep_fused_kernel<32>, n, NT, SepD<32>::SMEM, s, pdl, g, set.idx, set.first, gr, flags, at, taper, o); break;
    case 24: e = launch_pdl(degridder_sep_fused_kernel<24>, n, NT, SepD<24>::SMEM, s, pdl, g, set.idx, set.first, gr, flags, at, taper, o); break;
    case 16: e = launch_pdl(degridder_sep_fused_kernel<16>, n, NT, SepD<16>::SMEM, s, pdl, g, set.idx, set.first, gr, flags, at, taper, o); break;
    default: return fail(IDG_ERR_UNSUPPORTED, "the separable degridder needs L = 32, 24 or 16");
    }
    return e == cudaSuccess ? IDG_OK : cuda_fail(e, "separable degridder job launch");
}

idg_status launch_degridder_sep_fused(const Geometry &g, const SubgridSet &set, const void *grid, const uint8_t *flags,
                                      const void *aterms, const float *taper, void *vis_out, void *stream) {
    if (!separable_size(g.L) || !g.separable)
        return fail(IDG_ERR_UNSUPPORTED, "the separable degridder needs L = 32, 24 or 16 and a separable plan");
    if (set.count <= 0) return IDG_OK;
    switch (g.L) {
    case 32: return launch_sepd_set<32>(true, g, set, grid, flags, aterms, taper, vis_out, (cudaStream_t)stream);
    case 24: return launch_sepd_set<24>(true, g, set, grid, flags, aterms, taper, vis_out, (cudaStream_t)stream);
    default: return launch_sepd_set<16>(true, g, set, grid, flags, aterms, taper, vis_out, (cudaStream_t)stream);
    }
}

idg_status launch_degridder_sep_give_up(const Geometry &g, const SubgridSet &set, const void *grid, const void *aterms,
                                        const float *taper, void *vis_out, void *stream) {
    if (!separable_size(g.L) || !g.separable || !set.idx)
        return fail(IDG_ERR_UNSUPPORTED, "the separable degridder needs L = 32, 24 or 16 and a separable plan");
    if (set.count <= 0) return IDG_OK;
    switch (g.L) {
    case 32: return launch_give_up<32>(g, set, grid, aterms, taper, vis_out, (cudaStream_t)stream);
    case 24: return launch_give_up<24>(g, set, grid, aterms, taper, vis_out, (cudaStream_t)stream);
    default: return launch_give_up<16>(g, set, grid, aterms, taper, vis_out, (cudaStream_t)stream);
    }
}

idg_status read_sepd_error(int *code) {
    int zero = 0, v = 0;
    cudaError_t e = cudaMemcpyFromSymbol(&v, g_sepd_error, sizeof(int));
    if (e == cudaSuccess) e = cudaMemcpyToSymbol(g_sepd_error, &zero, sizeof(int));
    if (e != cudaSuccess) return cuda_fail(e, "reading the separable degridder error word");
    *code = v;
    return IDG_OK;
}

}  // namespace idg
