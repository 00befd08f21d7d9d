// Cluster-resident persistent sampling kernel for many rows: a whole dense bf16 H = 896 model in ONE 16-CTA cluster, as in
// wrnn_rescl.cu, which advances five to fourteen rows of a batch alone.
//
// What bounds the kernel of up to four rows as rows are added is the bytes of its exchanges: a CTA receives 16 bytes per cycle through
// distributed shared memory whatever the pattern, and a row costs it 1,792 bytes for each state half, as many for the hidden layer and
// 1,024 for the logits, twice per step.  Here the second exchange is gone:
//   * The logits product is split over K, not over rows: a CTA multiplies its own 28 values of the hidden layer with the 256 x 28 weights that
//     belong to them (as many as the 16 x 448 before) and sends its part of the 256 logits of a row to one CTA alone, which adds sixteen parts,
//     draws and sends the symbol to everybody.
//   * The products of R, in the background, hold two whole tiles per lane quadrant of tensor memory (and a quarter of K of a third), so that
//     their sums need no adding up over quadrants.  The tensor cores cut running sums off instead of rounding them, so a chain is
//     seven products long and is then added to the sum with a rounded addition.
//   * A CTA's new state values are one run of bytes in every receiver's image and travel as one bulk copy each: stores of 16 bytes fill the
//     load / store pipe until the other SMs have taken them, and the fragment loads of the background wait behind them.
//   * The rows of a cluster are two pipes that share nothing but the weights, so that one computes while the other waits for an exchange.
// Per CTA (rank r of its cluster): state units 28 r .. 28 r + 27 of both halves with their 168 rows of R, rows 28 r .. of O1 and O3, columns
// 28 r .. of O2 and O4; the draw of one row of the cluster.  Warps 0..7 are the chains of the pipes, warps 8..15 multiply R (see wrnn_rescl.cu).
// Every wait is bounded; a warp that gives up records where, skips its remaining waits and sends and keeps meeting its barriers, and all CTAs
// leave through the final cluster barrier.
#include <algorithm>
#include <cmath>

#include "wrnn_rescl.cuh"

namespace wrnn {

namespace {
constexpr int RM = 14;                                       // most rows of a cluster
constexpr int RPH = 40, RPF = 136, RPQ = 40;                 // floats per row of partial sums: hidden layer, whole tiles of R, quarters of K of the others
constexpr size_t RW_HID = 2 * 28 * 512;                      // O1 (O3) rows of a CTA as A fragments: two tiles
constexpr size_t RW_LOG = 16 * 2 * 512;                      // O2 (O4) columns: sixteen tiles of two k-tiles
constexpr int R_SMALL = 2 * 3 * CU * 3 + 2 * 32;              // I of the CTA's units [half][gate][unit][3], b1, b3 (32 each)
constexpr size_t RB_SMEM = 2 * RW_HID + 2 * RW_LOG + CW_R2 + R_SMALL * 4;
static_assert(RB_SMEM % 16 == 0, "the weights are copied in 16-byte pieces");
constexpr int RX_COL = 2 * 28 * 2 * 4;                        // columns of tensor memory: [half][28 k-tiles][tiles q, 4 + q][4], then [half][7][tile 8][4]
static_assert(RX_COL + 2 * 7 * 4 == CTC, "tensor memory of nine tiles");
// sb: most rows of a pipe
__host__ __device__ constexpr size_t rw_slice(int sb) { return (size_t)7 * sb * 16; }                // a CTA's values of one half of the state
__host__ __device__ constexpr size_t rw_img(int sb) { return CCS * rw_slice(sb); }                   // operand image of one half of the state
__host__ __device__ constexpr size_t rw_q(int sb) { return (size_t)8 * sb * 16; }                    // of the CTA's own hidden-layer values
constexpr size_t RW_RX = 16 * 1024;                                                                 // parts of the logits of one row
__host__ __device__ constexpr size_t rw_hid(int sb) { return (size_t)4 * 2 * sb * RPH * 4; }
__host__ __device__ constexpr size_t rw_full(int sb) { return (size_t)2 * sb * RPF * 4; }
__host__ __device__ constexpr size_t rw_quart(int sb) { return (size_t)4 * 2 * sb * RPQ * 4; }
__host__ __device__ constexpr size_t rw_smem(int sb)
{
    return RB_SMEM + 4 * rw_img(sb) + 2 * rw_q(sb) + 2 * rw_slice(sb) + RW_RX + rw_hid(sb) + rw_full(sb) + rw_quart(sb);
}
constexpr int RW_GUARDS = 8;             // of the checked form: behind the weights, the images, q, the new state, logits, hidden sums, R h (2)
static_assert(RW_RX >= (size_t)RM * CPR * 4, "scratch of the plain steps");
__host__ __device__ constexpr int rw_sb(int rows) { return rows <= 8 ? 4 : rows <= 12 ? 6 : 7; }
size_t rw_launch_smem(int rows, bool checked) { return rw_smem(rw_sb(rows)) + (checked ? RW_GUARDS * CL_GUARD : 0); }
}  // namespace

struct ResRowsPack {
    uint8_t *d_blob = nullptr;               // [16 ranks][shared memory | tensor memory]
    long long *d_prof = nullptr;             // [16]
    int max_clusters = 0;
    bool checked = false;                    // every call runs the checked form
    ClScales sc;
};

// SB: most rows of a pipe.  MODE 0: plain sampling; MODE 1: forced symbols, dumps, phase stamps and
// the self-test predicate; MODE 2: these and the checks.
template <int SB, int MODE>
__global__ void __launch_bounds__(512, 1) rows_cluster_kernel(const __grid_constant__ ClParams p)
{
    constexpr bool DBG = MODE != 0, CHK = MODE == 2;
    constexpr int NG = (SB + 3) / 4;                                     // groups of four rows, and the rows whose gates a warp of a chain computes
    constexpr int H = 2 * CK;
    constexpr int NR = 2 * SB;
    static_assert(SB == 4 || SB == 6 || SB == 7, "a CTA draws one row");
    extern __shared__ __align__(128) uint8_t smem[];
    __shared__ __align__(8) unsigned long long xw, xy[2][2], xl, xs[2];  // arrivals: weights, [pipe] state halves, parts of the logits, [pipe] symbols
    __shared__ uint32_t s_tmem;
    __shared__ int s_last[2][16];                                        // cl_wide_steps
    __shared__ uint32_t s_sym[2][16];                                    // [coarse half?][drawing CTA]: the symbol that is fed back
    __shared__ long long s_prof[DBG ? 16 : 1];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int g4 = lane >> 2, t4 = lane & 3;
    const int cl = blockIdx.x / CCS;
    const int row0 = cl * p.nr, nrc = min(p.nr, p.batch - row0);
    unsigned rank_u;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank_u));
    const int rank = (int)rank_u;
    // Two pipes: rows 0 .. of the cluster on warps 0..3 (chain) and 8..11 (background), the others on the other warps.  Row j of a pipe is
    // drawn by CTA 8 * pipe + j.
    const int pipe = (warp >> 2) & 1, w4 = warp & 3;
    const int rows0 = (nrc + 1) >> 1, rows = pipe ? nrc - rows0 : rows0, rb = pipe * SB;

    // ---- shared memory carve-up (must match rw_smem).  [half]: O3, O1; O4, O2
    const uint4 *wH[2] = {reinterpret_cast<const uint4 *>(smem + RW_HID), reinterpret_cast<const uint4 *>(smem)};
    const uint4 *wL[2] = {reinterpret_cast<const uint4 *>(smem + 2 * RW_HID + RW_LOG), reinterpret_cast<const uint4 *>(smem + 2 * RW_HID)};
    const uint32_t r2_addr = smem_u32(smem + 2 * RW_HID + 2 * RW_LOG);
    const float *sI = reinterpret_cast<const float *>(smem + RB_SMEM - R_SMALL * 4);               // [half][gate][unit][3]
    const float *sb1 = sI + 2 * 3 * CU * 3, *sb3 = sb1 + 32;
    constexpr size_t G = CHK ? CL_GUARD : 0;
    constexpr size_t SLICE = rw_slice(SB), XIMG = rw_img(SB), QIMG = rw_q(SB);
    constexpr size_t X0 = RB_SMEM + G, Q0 = X0 + 4 * XIMG + G, Y0 = Q0 + 2 * QIMG + G, L0 = Y0 + 2 * SLICE + G, P0 = L0 + RW_RX + G, F0 = P0 + rw_hid(SB) + G,
                     T0 = F0 + rw_full(SB) + G, END = T0 + rw_quart(SB) + G;
    uint8_t *ximg = smem + X0;                                           // [2: coarse, fine][pipe] state image
    uint8_t *qimg = smem + Q0 + pipe * QIMG;                             // this CTA's hidden-layer values
    uint8_t *ystage = smem + Y0 + pipe * SLICE;                          // its new state values
    float *lpart = reinterpret_cast<float *>(smem + L0);                 // [16 CTAs][even, odd quads of logits][32][4]
    float *hid = reinterpret_cast<float *>(smem + P0);                   // [4 quarters of K][NR][40]: hidden layer
    float *full = reinterpret_cast<float *>(smem + F0);                  // [NR][136]: rows 0 .. 127 of R h
    float *quart = reinterpret_cast<float *>(smem + T0);                 // [4 quarters of K][NR][40]: rows 128 .. 167
    static_assert(END == rw_smem(SB) + (CHK ? RW_GUARDS * CL_GUARD : 0), "the carve-up is what rw_smem says");
    auto guard = [&](int i) { return smem + (i == 0 ? X0 : i == 1 ? Q0 : i == 2 ? Y0 : i == 3 ? L0 : i == 4 ? P0 : i == 5 ? F0 : i == 6 ? T0 : END) - G; };
    // Operand images: [quad of k][SB rows][16 bytes], a producer's four values of a row being high x 4, low x 4; the B fragment of lane (column g = row,
    // part; t = quad of the k-tile) is one 8-byte load.  So that the four quads of half a warp lie on different banks, four rows change places in
    // two of four quads, and of seven rows those in a group of four are 0, 4, 1, 5 or 2, 6, 3 (of six 0 .. 3, 4, 5).
    constexpr uint32_t QSTR = 16 * SB;
    auto img_off = [](int quad, int row) { return (uint32_t)(quad * QSTR) + (SB == 4 ? row ^ (quad & 2) : row) * 16; };
    auto row_of = [](int g, int t) { return SB == 7 ? 4 * (t & 1) + 2 * g + (t >> 1) : 4 * g + t; };              // row t of group g
    constexpr uint32_t GSTR = SB == 7 ? 32 : 64;
    const uint32_t frag = t4 * QSTR + (SB == 4 ? (g4 >> 1) ^ (t4 & 2) : row_of(0, g4 >> 1)) * 16 + (g4 & 1) * 8;  // of k-tile 0, group 0

    // ---- one-time load: weights, zero images, barriers, tensor memory
    long long s0 = 0;                                                    // steps that cl_wide_steps took
    const uint8_t *blob = p.blob + (size_t)rank * (RB_SMEM + CB_TMEM);
    {
        int wide = 0;
        if (p.h_in)
            for (int i = tid; i < nrc * H; i += 512) wide |= fabsf(__ldcg(p.h_in + (size_t)row0 * H + i)) > CL_WIDE;
        if (tid == 0) {
            mbar_init(smem_u32(&xw), 1); mbar_init(smem_u32(&xl), 1);
            for (int i = 0; i < 2; ++i) { mbar_init(smem_u32(&xy[i][0]), 1); mbar_init(smem_u32(&xy[i][1]), 1); mbar_init(smem_u32(&xs[i]), 1); }
            mbar_fence_init();
            fence_proxy_async();
            cl_load_bulk(smem_u32(smem), blob, (uint32_t)RB_SMEM, smem_u32(&xw));
        }
        uint4 *z = reinterpret_cast<uint4 *>(ximg);
        for (int i = tid; i < (int)((L0 - X0) / 16); i += 512) z[i] = make_uint4(0, 0, 0, 0);
        if (warp == 1) {
            asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem)), "r"(512) : "memory");
            asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
        }
        if (DBG && tid < 16) s_prof[tid] = 0;
        tc_fence_before();
        wide = __syncthreads_or(wide);
        tc_fence_after();
        if (wide) {
            if (tid < nrc) { s_last[0][tid] = p.c_in ? p.c_in[row0 + tid] : 128; s_last[1][tid] = p.f_in ? p.f_in[row0 + tid] : 0; }
            __syncthreads();
            s0 = cl_wide_steps<CL_BF16>(p, row0, nrc, rank, lpart, s_last);
            if (rank == 0 && tid < nrc) {
                if (p.c_st_out) p.c_st_out[row0 + tid] = (uint8_t)s_last[0][tid];
                if (p.f_st_out) p.f_st_out[row0 + tid] = (uint8_t)s_last[1][tid];
            }
            if (s0 == p.n_steps) {
                mbar_wait(smem_u32(&xw), 0, p.limit_ns);                  // no copy in flight when the CTA leaves
                if (warp == 1) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(s_tmem), "r"(512) : "memory");
                return;
            }
        }
        cl_load_tmem(s_tmem, blob + RB_SMEM, warp, lane);
        // images of the initial state
        if (p.h_in)
            for (int i = tid; i < nrc * H; i += 512) {
                const int st = i / H, j = i - st * H, half_f = j >= CK, k = j - half_f * CK;
                const float x = __ldcg(p.h_in + (size_t)(row0 + st) * H + j) * CL_STATE;
                __half *im = reinterpret_cast<__half *>(ximg + (2 * half_f + (st >= rows0)) * XIMG + img_off(k >> 2, st < rows0 ? st : st - rows0)) + (k & 3);
                im[0] = __float2half_rn(x);
                im[4] = __float2half_rn(x - __half2float(im[0]));
            }
        fence_proxy_async_cta();                                         // before bulk copies of the peers go over what this CTA wrote
    }
    bool bad = !mbar_wait(smem_u32(&xw), 0, p.limit_ns);                 // this thread gave up: it skips waits and sends from here on
    if (bad && atomicCAS(&p.status->code, DEV_OK, DEV_TIMEOUT) == DEV_OK) { p.status->cta = blockIdx.x; p.status->step = 0; p.status->phase = 9; }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (CHK) {
        if (tid < RW_GUARDS) cl_guard_fill(guard(tid));
        if (tid == 0 && END != p.smem_bytes) cl_record(p.status, -2);
        __syncthreads();
        if (p.poke && blockIdx.x == 3 && tid == 0) full[rw_full(SB) / 4] = 0.f;
    }
    // a store of n bytes at an offset of a region of `size` bytes
    auto store_ok = [&](uint32_t off, uint32_t n, size_t size) {
        if (!CHK || off + n <= size) return true;
        cl_record(p.status, -1);
        return false;
    };
    cluster_sync_all();                                                  // every peer's barriers are initialised before anyone sends
    const uint32_t tmem = s_tmem;

    Waiter wt{p.status, p.limit_ns};
    const bool prof_on = DBG && p.prof != nullptr && blockIdx.x == 0 && warp == 0;
    long long prof_t = clock64();
#define STAMP(i) do { if (DBG && prof_on) { const long long now_ = clock64(); if (lane == 0) s_prof[i] += now_ - prof_t; prof_t = now_; } } while (0)
#define STAMP0() do { if (DBG && prof_on) prof_t = clock64(); } while (0)
    auto wait_bar = [&](unsigned long long *b, unsigned parity, int step, int phase) {
        if (bad) return;
        const unsigned a = smem_u32(b);
        unsigned long long t0 = 0; unsigned cnt = 0;
        while (!mbar_try(a, parity & 1u))
            if ((++cnt & 1023u) == 0 && wt.expired(t0, step, phase)) { bad = true; break; }
    };
    auto part_sum = [&](const float (&c)[4], float &lo, float &hi) { lo = c[0] + c[1]; hi = c[2] + c[3]; };

    // ---- rows of R times one half of the state, accumulated over both halves (warps 8..15).  Lane quadrant q = w & 3 holds tiles q and
    // 4 + q and a quarter of K of tile 8 in its tensor memory; with that quarter go the 24 rows in shared memory.
    auto background = [&]() {
        constexpr int GN = NG;
        const int rq = w4;
        float sum[2][GN][4], ax[3][GN][4];
        auto clear = [&]() {
#pragma unroll
            for (int g = 0; g < GN; ++g)
#pragma unroll
                for (int k = 0; k < 4; ++k) { sum[0][g][k] = sum[1][g][k] = 0.f; ax[0][g][k] = ax[1][g][k] = ax[2][g][k] = 0.f; }
        };
        auto products = [&](int half_f) {
            const uint32_t b0 = smem_u32(ximg + (2 * half_f + pipe) * XIMG) + frag;
            const uint32_t tc = tmem + ((uint32_t)(32 * rq) << 16) + half_f * 28 * 8;
            const uint32_t tx = tmem + ((uint32_t)(32 * rq) << 16) + RX_COL + half_f * 7 * 4;
            const uint32_t a0 = r2_addr + (uint32_t)(((half_f * CK8 + 14 * rq + (lane >> 4)) * CRS + ((lane >> 3) & 1) * 8 + (lane & 7)) * 16);
            const uint32_t a1 = r2_addr + (uint32_t)(((half_f * CK8 + 14 * rq + ((lane >> 3) & 1)) * CRS + 16 + (lane & 7)) * 16);
            uint32_t r0[8], r1[8];
            uint2 c0[GN], c1[GN];
            auto load = [&](int kt, uint32_t (&r)[8], uint2 (&b)[GN]) {
                cl_tmem_ld8(tc + kt * 8, r);
#pragma unroll
                for (int g = 0; g < GN; ++g) b[g] = cl_lds8(b0 + kt * 4 * QSTR + g * GSTR);
            };
            load(0, r0, c0);
#pragma unroll 1
            for (int c = 0; c < 4; ++c) {
                float acc[2][GN][4];
#pragma unroll
                for (int g = 0; g < GN; ++g)
#pragma unroll
                    for (int k = 0; k < 4; ++k) acc[0][g][k] = acc[1][g][k] = 0.f;
                auto mmas = [&](const uint32_t (&r)[8], const uint2 (&b)[GN]) {
#pragma unroll
                    for (int j = 0; j < 2; ++j)
#pragma unroll
                        for (int g = 0; g < GN; ++g) cl_mma(acc[j][g], make_uint4(r[4 * j], r[4 * j + 1], r[4 * j + 2], r[4 * j + 3]), b[g].x, b[g].y);
                };
                auto seven = [&](auto EX_C) {
                    constexpr bool EX = decltype(EX_C)::value;
#pragma unroll
                    for (int i = 0; i < 7; ++i) {
                        uint32_t x[4], t[6];
                        if (EX) {
                            asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];" : "=r"(x[0]), "=r"(x[1]), "=r"(x[2]), "=r"(x[3]) : "r"(tx + 4 * i));
                            cl_ldmatrix4(a0 + i * 2 * CRS * 16, *reinterpret_cast<uint32_t (*)[4]>(&t));
                            asm volatile("ldmatrix.sync.aligned.m8n8.x2.shared.b16 {%0,%1}, [%2];" : "=r"(t[4]), "=r"(t[5]) : "r"(a1 + i * 2 * CRS * 16) : "memory");
                        }
                        auto extra = [&](const uint2 (&b)[GN]) {
                            if (EX)
#pragma unroll
                                for (int g = 0; g < GN; ++g) {
                                    cl_mma(ax[0][g], make_uint4(x[0], x[1], x[2], x[3]), b[g].x, b[g].y);
                                    cl_mma(ax[1][g], make_uint4(t[0], t[1], t[2], t[3]), b[g].x, b[g].y);
                                    cl_mma(ax[2][g], make_uint4(t[4], 0, t[5], 0), b[g].x, b[g].y);
                                }
                        };
                        tmem_wait_ld();
                        if (i & 1) { load(7 * c + i + 1, r0, c0); mmas(r1, c1); extra(c1); }
                        else { if (i < 6) load(7 * c + i + 1, r1, c1); mmas(r0, c0); extra(c0); }
                    }
                    if (c < 3) load(7 * c + 7, r0, c0);
                };
                if (c == rq) seven(std::true_type{});
                else seven(std::false_type{});
#pragma unroll
                for (int g = 0; g < GN; ++g)
#pragma unroll
                    for (int k = 0; k < 4; ++k) { sum[0][g][k] += acc[0][g][k]; sum[1][g][k] += acc[1][g][k]; }
            }
        };
        auto store = [&]() {
#pragma unroll
            for (int g = 0; g < GN; ++g) {
                if (row_of(g, t4) >= SB) continue;
                const int st = rb + row_of(g, t4);
                float *d = full + st * RPF + 16 * rq + g4, *e = quart + (rq * NR + st) * RPQ + g4;
                part_sum(sum[0][g], d[0], d[8]);
                part_sum(sum[1][g], d[64], d[72]);
                part_sum(ax[0][g], e[0], e[8]);
                part_sum(ax[1][g], e[16], e[24]);
                e[32] = ax[2][g][0] + ax[2][g][1];
            }
        };
        // the initial state
        clear();
#pragma unroll 1
        for (int half_f = 0; half_f < 2; ++half_f) products(half_f);
        store();
        __syncthreads();
        cl_cluster_arrive();
        __syncthreads();
        cl_cluster_wait();
        const unsigned T = rows ? (unsigned)(p.n_steps - s0) : 0;
#pragma unroll 1
        for (unsigned s2 = 0; s2 < T; ++s2) {
            clear();
            cl_bar_sync(2 + 8 * pipe, 256);
            products(0);
            cl_bar_sync(2 + 8 * pipe, 256);
            products(1);
            store();
            cl_bar_arrive(4 + 8 * pipe, 256);
        }
    };
    if (warp >= 8) background();
    else {
        // ---- fixed addresses: what to add to an address of mine
        const uint32_t sbase = smem_u32(smem);
        const uint32_t dy = map_to_rank(sbase, (unsigned)(w4 + 4 * (lane & 3))) - sbase;         // state: CTAs w, w + 4, ..
        uint32_t dl[NG];                                                 // parts of the logits: the CTA that draws row t of group g
#pragma unroll
        for (int g = 0; g < NG; ++g) dl[g] = map_to_rank(sbase, (unsigned)(8 * pipe + row_of(g, t4))) - sbase;
        const uint32_t ds = map_to_rank(sbase, (unsigned)(lane & 15)) - sbase;        // symbols
        const int skip_at = (DBG && rank == p.skip_rank) ? (int)(p.skip_step - s0) : -1;
        const unsigned ybytes = (unsigned)XIMG, sbytes = 4u * rows;
        const bool draws = rank >> 3 == pipe && (rank & 7) < rows, drawer = w4 == 3 && draws;        // this CTA draws a row of this pipe; this warp does
        const int grow0 = row0 + pipe * rows0, gd = grow0 + (draws ? rank & 7 : 0);
        unsigned long long *const xyp = xy[pipe], *const xsp = &xs[pipe];
        const int BAR = 8 * pipe;

        // ---- the rows whose gates this warp computes (unit = lane), their last symbols
        const bool unit_on = lane < CU;
        const int gu = unit_on ? lane : 0, gj = CU * rank + gu;
        int row[NG], st[NG], frame[NG], rem[NG], c_prev[NG], f_prev[NG];              // (st: a row that exists)
        bool on[NG];
        float hC[NG], hF[NG];
        const float *g_row[NG];
        const int w_q = p.row_lag > 0 ? 1 : p.row_stride / p.hop, w_r = p.row_lag > 0 ? 0 : p.row_stride - w_q * p.hop;      // staggered rows: a frame per step of the call
#pragma unroll
        for (int i = 0; i < NG; ++i) {
            row[i] = w4 + 4 * i;
            on[i] = row[i] < rows;
            st[i] = on[i] ? row[i] : 0;
            const int gb = min(grow0 + st[i], p.batch - 1);
            c_prev[i] = s0 > 0 ? s_last[0][min(gb - row0, 15)] : p.c_in ? p.c_in[gb] : 128;
            f_prev[i] = s0 > 0 ? s_last[1][min(gb - row0, 15)] : p.f_in ? p.f_in[gb] : 0;
            hC[i] = hF[i] = 0.f;
            if (on[i] && unit_on && p.h_in) { hC[i] = __ldcg(p.h_in + (size_t)gb * H + gj); hF[i] = __ldcg(p.h_in + (size_t)gb * H + CK + gj); }
            g_row[i] = p.g + (size_t)gb * p.n_frames * 3 * H + gj;
            const long long pos = p.row_lag > 0 ? s0 * p.hop : (p.step0 + s0) * p.row_stride + ((long long)p.stream0 + gb) * p.row_offset_mul;
            frame[i] = (int)(pos / p.hop);
            rem[i] = (int)(pos - (long long)frame[i] * p.hop);
        }
        const long long u_pos = p.step0 + s0 - (long long)gd * p.row_lag;             // step of the row that this CTA draws
        int c_drawn = 0;                                                 // its coarse symbol of this step
        int16_t *out_row = p.out ? p.out + (long long)gd * p.out_pitch + s0 : nullptr;

        float dbg_v[DBG ? NG : 1][4];                                    // what the dumps want of this half-step's gates
        auto dump_gates = [&](int half_g, long long s) {
#pragma unroll
            for (int i = 0; i < NG; ++i) {
                if (!on[i] || !unit_on) continue;
                const int jj = half_g * CK + gj, gb = grow0 + row[i], k = DBG ? i : 0;
                if (p.dbg_gates) { float *o = p.dbg_gates + ((size_t)(s0 + s) * p.batch + gb) * 3 * H; o[jj] = dbg_v[k][0]; o[H + jj] = dbg_v[k][1]; o[2 * H + jj] = dbg_v[k][2]; }
                if (p.dbg_h) p.dbg_h[((size_t)(s0 + s) * p.batch + gb) * H + jj] = dbg_v[k][3];
            }
        };
        struct GatePre { float pu, pr, pe, ae; };
        // row i of R h of row b
        auto r_row = [&](int b, int i) {
            if (i < 128) return full[(rb + b) * RPF + i] * p.sc.inv_R;
            const float *q = quart + (rb + b) * RPQ + i - 128;
            return ((q[0] + q[NR * RPQ]) + (q[2 * NR * RPQ] + q[3 * NR * RPQ])) * p.sc.inv_R;
        };
        // everything of the gates of one half that does not depend on the pending draw (fine units: the coarse symbol of this step;
        // coarse units: the last fine one)
        auto gates_prepare = [&](int half_g, const float (&gv)[3], int i) {
            const float *Iu = sI + (half_g * 3 * CU + gu) * 3, *Ir = Iu + CU * 3, *Ie = Ir + CU * 3;
            GatePre q = {gv[0], gv[1], gv[2], 0.f};
            if (half_g) { const float x = scale8(f_prev[i]); q.pu = fmaf(Iu[1], x, q.pu); q.pr = fmaf(Ir[1], x, q.pr); q.pe = fmaf(Ie[1], x, q.pe); }
            const float x = scale8(c_prev[i]);
            q.pu = fmaf(Iu[0], x, q.pu); q.pr = fmaf(Ir[0], x, q.pr); q.pe = fmaf(Ie[0], x, q.pe);
            return q;
        };
        auto gates_add_r = [&](int half_g, GatePre &q, int i) {
            q.pu += r_row(st[i], half_g * 3 * CU + gu);
            q.pr += r_row(st[i], half_g * 3 * CU + CU + gu);
            q.ae = r_row(st[i], half_g * 3 * CU + 2 * CU + gu);
        };
        auto gates = [&](int half_g, int drawn, const GatePre &q, int i) {
            const float *Iu = sI + (half_g * 3 * CU + gu) * 3 + 1 + half_g, *Ir = Iu + CU * 3, *Ie = Ir + CU * 3;
            const float x = scale8(drawn);
            const float u = cl_sigmoid(fmaf(*Iu, x, q.pu)), r = cl_sigmoid(fmaf(*Ir, x, q.pr));
            const float e = cl_tanh(fmaf(r, q.ae, fmaf(*Ie, x, q.pe)));
            const float hn = fmaf(u, half_g ? hF[i] : hC[i], (1.0f - u) * e);
            if (half_g) hF[i] = hn; else hC[i] = hn;
            if (DBG) { const int k = DBG ? i : 0; dbg_v[k][0] = u; dbg_v[k][1] = r; dbg_v[k][2] = e; dbg_v[k][3] = hn; }
        };
        // all rows' values are there before the first is staged, and one fence is for all of them: row by row the second one waits for the
        // first one's stores and fence (64 rows 6.63 -> 6.52, 256 rows 20.33 -> 20.05 us per step)
        auto stage = [&](int half_g) {
#pragma unroll
            for (int i = 0; i < NG; ++i)
                if (unit_on && on[i]) {
                    __half *d = reinterpret_cast<__half *>(ystage + img_off(7 * rank + (lane >> 2), row[i]) - 7 * rank * QSTR) + (lane & 3);
                    const float v = (half_g ? hF[i] : hC[i]) * CL_STATE;
                    const __half hi = __float2half_rn(v);
                    d[0] = hi;
                    d[4] = __float2half_rn(v - __half2float(hi));
                }
            fence_proxy_async_cta();
        };
        // the new state values of this CTA's units -> images in four CTAs of the cluster (the staged values are overwritten when symbols have
        // come that depend on what every CTA made of these copies)
        auto send_y = [&](int half_g, long long s) {
            if (bad || lane >= 4 || (DBG && (int)s == skip_at)) return;
            const uint32_t off = (uint32_t)(rank * SLICE);
            if (!store_ok(off, SLICE, XIMG)) return;
            cl_copy_bulk(sbase + (uint32_t)(X0 + (2 * half_g + pipe) * XIMG) + off + dy, smem_u32(ystage), (uint32_t)SLICE, smem_u32(&xyp[half_g]) + dy);
        };
        // ---- prologue: coarse gates of step 0 (the background warps have multiplied R by the initial state)
        const bool lead = w4 == 0 && lane == 0;
        if (lead && rows) mbar_arrive_expect(smem_u32(&xyp[0]), ybytes);
        __syncthreads();
        // The products read the images of the initial state, over which the peers store their first one: nobody sends before
        // every CTA has arrived here (the loop needs nothing of the kind: whoever sends has received something from everybody)
        cl_cluster_arrive();
#pragma unroll
        for (int i = 0; i < NG; ++i)
            if (on[i]) {
                float gv[3];
                const float *g = g_row[i] + (size_t)frame[i] * 3 * H;
#pragma unroll
                for (int gate = 0; gate < 3; ++gate) gv[gate] = __ldg(g + gate * H);
                GatePre gp = gates_prepare(0, gv, i);
                gates_add_r(0, gp, i);
                gates(0, f_prev[i], gp, i);
            }
        stage(0);
        __syncthreads();
        cl_cluster_wait();
        // a pipe without rows sends nothing: it would not wait for what it is sent, and the cluster barrier at the end does not hold a CTA back
        // until a copy into it has landed
        if (rows) send_y(0, 0);
        if (DBG) dump_gates(0, 0);

        // Half-step n = 2 s + 1 is the coarse half of step s (input y_c(s): coarse head -> c_s, then the fine gates of step s),
        // n = 2 s the fine half (input y_f(s - 1): fine head -> f_{s-1}, R h_{s-1} completed, then the coarse gates of step s).
        // A peer may overwrite an image, the parts of the logits or the symbols only after it has received what this CTA sends after its last use.
        const unsigned T = rows ? (unsigned)(p.n_steps - s0) : 0;        // (a call has fewer than 2^31 steps)
        auto half_step = [&](auto HALF_C, const unsigned n) {
            constexpr int half = decltype(HALF_C)::value;                // 1: coarse half
            constexpr int in = half ? 0 : 1;                             // image of its input
            const long long s = n >> 1;
            const bool last = n == 2 * T;
            const unsigned yuse = (n - 1) >> 1, quse = n - 1;
            if (lead && !bad) {
                if (draws) mbar_arrive_expect(smem_u32(&xl), (unsigned)RW_RX);
                mbar_arrive_expect(smem_u32(xsp), sbytes);
                if (!last) mbar_arrive_expect(smem_u32(&xyp[half]), ybytes);
            }
            float gv[NG][3];
#pragma unroll
            for (int i = 0; i < NG; ++i) {
                if (!half) { frame[i] += w_q; rem[i] += w_r; if (rem[i] >= p.hop) { rem[i] -= p.hop; ++frame[i]; } }
                const float *g = g_row[i] + (size_t)frame[i] * 3 * H + half * CK;
                if (!last && on[i])
#pragma unroll
                    for (int gate = 0; gate < 3; ++gate) gv[i][gate] = __ldg(g + gate * H);
                else gv[i][0] = gv[i][1] = gv[i][2] = 0.f;
            }
            // ---- hidden layer: this CTA's 28 rows (two tiles), K in four quarters; weight fragments before the wait
            {
                uint4 av[2][7];
                const uint4 *A = wH[half] + 7 * w4 * 32 + lane;
#pragma unroll
                for (int i = 0; i < 7; ++i) { av[0][i] = A[i * 32]; av[1][i] = A[(28 + i) * 32]; }
                STAMP0();
                wait_bar(&xyp[in], yuse, (int)s, 1 + 4 * half);
                STAMP(8 * half + 0);
                const uint32_t b0 = sbase + (uint32_t)(X0 + (2 * in + pipe) * XIMG) + 28 * w4 * QSTR + frag;
                float acc[NG][2][2][4];
#pragma unroll
                for (int g = 0; g < NG; ++g)
#pragma unroll
                    for (int k = 0; k < 16; ++k) acc[g][k >> 3][(k >> 2) & 1][k & 3] = 0.f;
#pragma unroll
                for (int i = 0; i < 7; ++i)
#pragma unroll
                    for (int g = 0; g < NG; ++g) {
                        const uint2 b = cl_lds8(b0 + i * 4 * QSTR + g * GSTR);
                        cl_mma(acc[g][0][i & 1], av[0][i], b.x, b.y);
                        cl_mma(acc[g][1][i & 1], av[1][i], b.x, b.y);
                    }
#pragma unroll
                for (int g = 0; g < NG; ++g) {
                    if (row_of(g, t4) >= SB) continue;
#pragma unroll
                    for (int tile = 0; tile < 2; ++tile) {
#pragma unroll
                        for (int k = 0; k < 4; ++k) acc[g][tile][0][k] += acc[g][tile][1][k];
                        float *d = hid + (w4 * NR + rb + row_of(g, t4)) * RPH + tile * 16 + g4;
                        part_sum(acc[g][tile][0], d[0], d[8]);
                    }
                }
            }
            cl_bar_sync(1 + BAR, 128);
            STAMP(8 * half + 1);
            // ---- K-split sums, bias, relu, parts: the operand image of this CTA's own values
            if (lane + 32 * w4 < 7 * rows) {
                const int i = lane + 32 * w4, quad = i % 7, b = i / 7;
                const float4 bias = *reinterpret_cast<const float4 *>((half ? sb1 : sb3) + 4 * quad);
                float4 v = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
                for (int sp = 0; sp < 4; ++sp) {
                    const float4 a = *reinterpret_cast<const float4 *>(hid + (sp * NR + rb + b) * RPH + 4 * quad);
                    v.x += a.x; v.y += a.y; v.z += a.z; v.w += a.w;
                }
                const float inv = p.sc.inv_O1[1 - half], qs = p.sc.q_scale[1 - half];
                v.x = fmaxf(fmaf(v.x, inv, bias.x), 0.f) * qs; v.y = fmaxf(fmaf(v.y, inv, bias.y), 0.f) * qs;
                v.z = fmaxf(fmaf(v.z, inv, bias.z), 0.f) * qs; v.w = fmaxf(fmaf(v.w, inv, bias.w), 0.f) * qs;
                uint2 lo;
                const uint2 hi = cl_split4(v.x, v.y, v.z, v.w, lo);
                *reinterpret_cast<uint4 *>(qimg + img_off(quad, b)) = make_uint4(hi.x, hi.y, lo.x, lo.y);
            }
            uint4 lv[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) lv[i] = wL[half][(8 * w4 + i) * 32 + lane];
            STAMP(8 * half + 2);
            cl_bar_sync(2 + BAR, 256);   // the background warps are done with the last half-step, and go on
            STAMP(8 * half + 3);
            // ---- this CTA's part of the logits: warp w has logits 64 w .. 64 w + 63 of all rows, in two pairs of tiles of which a lane holds four
            // consecutive ones (quad 8 v + 2 g, or 8 v + 2 (g - 4) + 1, of pair v)
            {
                const uint32_t b0 = smem_u32(qimg) + frag;
                const uint32_t a = smem_u32(lpart) + rank * 1024 + ((g4 >> 2) * 128 + 4 * (8 * w4 + (g4 & 3))) * 4, bar = smem_u32(&xl);
#pragma unroll
                for (int g = 0; g < NG; ++g) {
                    const uint2 k0 = cl_lds8(b0 + g * GSTR), k1 = cl_lds8(b0 + 4 * QSTR + g * GSTR);
                    float acc[4][4] = {};
#pragma unroll
                    for (int j = 0; j < 4; ++j) cl_mma(acc[j], lv[2 * j], k0.x, k0.y);
#pragma unroll
                    for (int j = 0; j < 4; ++j) cl_mma(acc[j], lv[2 * j + 1], k1.x, k1.y);
#pragma unroll
                    for (int v = 0; v < 2; ++v) {
                        float l[4];
                        part_sum(acc[2 * v], l[0], l[1]);
                        part_sum(acc[2 * v + 1], l[2], l[3]);
                        if (row_of(g, t4) < rows && !bad && store_ok(a + 64 * v - smem_u32(lpart), 16, RW_RX)) st_async_v4(a + 64 * v + dl[g], l[0], l[1], l[2], l[3], bar + dl[g]);
                    }
                }
            }
            STAMP(8 * half + 4);
            // ---- what does not depend on the draw
            GatePre gp[NG];
#pragma unroll
            for (int i = 0; i < NG; ++i) {
                gp[i] = gates_prepare(half, gv[i], i);
                if (half) gates_add_r(half, gp[i], i);
            }
            STAMP(8 * half + 5);
            // ---- one warp of the CTA that draws a row: the sum of its parts, the draw, the symbol to everybody
            if (drawer) {
                const long long t = half ? s : s - 1;
                const float u01 = uniform24(p.seed, p.stream0 + (unsigned)gd, (unsigned long long)(u_pos + t), half ? 0u : 1u);
                int forced = -1;
                if (DBG) {
                    const uint8_t *fz = half ? p.c_forced : p.f_forced;
                    if (fz) forced = fz[(size_t)gd * p.n_steps + s0 + t];
                }
                const float4 *bias = reinterpret_cast<const float4 *>(p.wb[half ? 2 : 3]) + 2 * lane;
                const float4 ba = __ldg(bias), bb = __ldg(bias + 1);
                wait_bar(&xl, quse, (int)s, 2 + 4 * half);
                float4 va = {0.f, 0.f, 0.f, 0.f}, vb = {0.f, 0.f, 0.f, 0.f}, vc = va, vd = vb;
                const float4 *lp = reinterpret_cast<const float4 *>(lpart) + lane;
#pragma unroll
                for (int c = 0; c < 16; c += 2) {
                    const float4 a0 = lp[64 * c], b0 = lp[64 * c + 32], a1 = lp[64 * c + 64], b1 = lp[64 * c + 96];
                    va.x += a0.x; va.y += a0.y; va.z += a0.z; va.w += a0.w;
                    vb.x += b0.x; vb.y += b0.y; vb.z += b0.z; vb.w += b0.w;
                    vc.x += a1.x; vc.y += a1.y; vc.z += a1.z; vc.w += a1.w;
                    vd.x += b1.x; vd.y += b1.y; vd.z += b1.z; vd.w += b1.w;
                }
                const float inv = p.sc.inv_O2[1 - half];
                const float l[8] = {fmaf(va.x + vc.x, inv, ba.x), fmaf(va.y + vc.y, inv, ba.y), fmaf(va.z + vc.z, inv, ba.z), fmaf(va.w + vc.w, inv, ba.w),
                                    fmaf(vb.x + vd.x, inv, bb.x), fmaf(vb.y + vd.y, inv, bb.y), fmaf(vb.z + vd.z, inv, bb.z), fmaf(vb.w + vd.w, inv, bb.w)};
                const int drawn = cl_draw(l, u01, lane), fed = (DBG && forced >= 0) ? forced : drawn;
                if (lane < 16 && !bad) cl_st_async4(smem_u32(&s_sym[half][rank]) + ds, (uint32_t)fed, smem_u32(xsp) + ds);
                if (DBG && p.dbg_logits && !bad) {
                    float *d = p.dbg_logits + (((size_t)(s0 + t) * p.batch + gd) * 2 + (half ? 0 : 1)) * 256 + 8 * lane;
#pragma unroll
                    for (int k = 0; k < 8; ++k) d[k] = l[k];
                }
                if (lane == 0 && !bad) {
                    if (DBG) {
                        uint8_t *o = half ? p.c_out : p.f_out;
                        if (o) o[(size_t)gd * p.n_steps + s0 + t] = (uint8_t)drawn;
                    }
                    if (!half && out_row) out_row[s - 1] = (int16_t)(256 * c_drawn + fed - 32768);
                }
                if (half) c_drawn = fed;
            }
            wait_bar(xsp, quse, (int)s, 3 + 4 * half);
            STAMP(8 * half + 6);
            if (!half) cl_bar_sync(4 + BAR, 256);                        // R h is complete
#pragma unroll
            for (int i = 0; i < NG; ++i) {
                const int fed = (int)s_sym[half][8 * pipe + st[i]] & 255;
                if (!half) gates_add_r(half, gp[i], i);
                if (half) c_prev[i] = fed; else f_prev[i] = fed;
            }
            if (!last) {
#pragma unroll
                for (int i = 0; i < NG; ++i) gates(half, half ? c_prev[i] : f_prev[i], gp[i], i);
                stage(half);
            }
            STAMP(8 * half + 7);
            if (!last) {
                cl_bar_sync(1 + BAR, 128);
                send_y(half, s);
                if (DBG && !bad) dump_gates(half, s);
            }
        };
#pragma unroll 1
        for (unsigned s2 = 0; s2 < T; ++s2) {
            half_step(std::integral_constant<int, 1>{}, 2 * s2 + 1);
            half_step(std::integral_constant<int, 0>{}, 2 * s2 + 2);
        }
        // ---- results, unless a warp gave up
        const bool any_bad = __syncthreads_or(bad);
        if (!any_bad)
#pragma unroll
            for (int i = 0; i < NG; ++i) {
                if (!on[i]) continue;
                const int gb = grow0 + row[i];
                if (unit_on && p.h_out) { p.h_out[(size_t)gb * H + gj] = hC[i]; p.h_out[(size_t)gb * H + CK + gj] = hF[i]; }
                if (rank == 0 && lane == 0) {
                    if (p.c_st_out) p.c_st_out[gb] = (uint8_t)c_prev[i];
                    if (p.f_st_out) p.f_st_out[gb] = (uint8_t)f_prev[i];
                }
            }
    }
    if (warp >= 8) __syncthreads_or(bad);
#undef STAMP
#undef STAMP0
    // nobody leaves while a peer may still write into its shared memory
    if (DBG && p.prof && blockIdx.x == 0 && tid < 16) p.prof[tid] = s_prof[tid];
    if (CHK && tid < RW_GUARDS && !cl_guard_ok(guard(tid))) cl_record(p.status, tid);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 1) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
    cluster_sync_all();
}

// ---------------------------------------------------------------------------------------------
static const void *rw_kernel_of(int rows, int mode)
{
#define RW_K(N) (mode == 2 ? (const void *)rows_cluster_kernel<N, 2> : mode ? (const void *)rows_cluster_kernel<N, 1> : (const void *)rows_cluster_kernel<N, 0>)
    return rw_sb(rows) == 4 ? RW_K(4) : rw_sb(rows) == 6 ? RW_K(6) : RW_K(7);
#undef RW_K
}

// Rows per cluster and clusters of a batch: waves of clusters of up to eight rows (4.60 to 4.75 us per step, 5 to 8 rows) or of up to fourteen
// (6.52 to 6.74 us, 9 to 14 rows), whichever all waves together take less time with, evenly filled: with seven clusters at a time 6.7 against 9.5 us
// from 64 to 98 rows, 9.6 against 13.6 to 112, 13.7 against 14.3 to 168 and 19.2 to 196, 19.2 against 20.1 to 224, 20.4 against 24 to 280.  (57 to
// 63 rows, nine per cluster, would take 6.5 instead of 9.3; they stay two waves, the launch that wrnn_launch_info has always stated at 57 rows.)
static void rw_geometry(const ResRowsPack &k, int batch, int *nr, int *n_clusters)
{
    const int c = k.max_clusters, few = (batch + 8 * c - 1) / (8 * c), many = (batch + RM * c - 1) / (RM * c);
    const int waves = batch <= 9 * c || 48 * few <= 68 * many ? few : many;
    *nr = (batch + waves * c - 1) / (waves * c);
    *n_clusters = (batch + *nr - 1) / *nr;
}

int resrows_prepare(wrnn_model *m)
{
    if (m->sparse || m->H != 2 * CK || m->dtype != WRNN_BF16 || m->variant != 0) { m->err = "cluster-resident kernel of many rows: dense bf16 H = 896 only"; return WRNN_ERR_UNSUPPORTED; }
    ResRowsPack k;
    { const char *d = getenv("WRNN_DEBUG"); k.checked = d && d[0] == '1'; }
    for (int rows : {8, 12, 14})
        for (int mode = 0; mode < (k.checked ? 3 : 2); ++mode) {
            const void *f = rw_kernel_of(rows, mode);
            if (cudaFuncSetAttribute(f, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess || !allow_smem(f, m->device, rw_launch_smem(rows, mode == 2))) {
                cudaGetLastError(); m->err = "cluster-resident kernel of many rows does not fit this device"; return WRNN_ERR_UNSUPPORTED;
            }
        }
    {
        cudaLaunchConfig_t cfg; cudaLaunchAttribute at[1];
        cl_fill_launch(1, rw_launch_smem(RM, false), &cfg, at, 0);
        if (cudaOccupancyMaxActiveClusters(&k.max_clusters, rw_kernel_of(RM, 0), &cfg) != cudaSuccess || k.max_clusters < 1) {
            cudaGetLastError(); m->err = "cluster-resident kernel of many rows: no 16-CTA cluster of this size fits the device"; return WRNN_ERR_UNSUPPORTED;
        }
    }
    // fp16 weights, every matrix scaled by a power of two (see rescl_prepare)
    if (!m->half) m->half = new ClHalf(m, 1);
    const HalfMatrix &R = m->half->R, *O = m->half->O;
    k.sc = m->half->sc;
    const size_t cta_bytes = RB_SMEM + CB_TMEM;
    std::vector<uint8_t> blob(CCS * cta_bytes, 0);
    parallel_for(CCS, [&](int rank) {
        uint8_t *base = blob.data() + (size_t)rank * cta_bytes;
        for (int h = 0; h < 2; ++h) {
            for (int t = 0; t < 2; ++t)
                pack_448(O[h].part[0], CU * rank + 16 * t, std::min(16, CU - 16 * t), reinterpret_cast<uint16_t *>(base + h * RW_HID + (size_t)t * 28 * 512));
            // columns 28 rank .. of the logits rows, 28 of 32 used: tile j of pair w holds at row g logits 4 quad + 2 j and at row g + 8 the next
            uint16_t *lg = reinterpret_cast<uint16_t *>(base + 2 * RW_HID + h * RW_LOG);
            for (int w = 0; w < 8; ++w)
                for (int j = 0; j < 2; ++j)
                    for (int r = 0; r < 16; ++r) {
                        const int g = r & 7, quad = 8 * w + (g < 4 ? 2 * g : 2 * (g - 4) + 1), logit = 4 * quad + 2 * j + (r >> 3);
                        uint16_t src[32] = {};
                        std::memcpy(src, &O[2 + h].part[0][(size_t)logit * CK + CU * rank], CU * 2);
                        for (int kt = 0; kt < 2; ++kt) frag_row(lg + ((size_t)(4 * w + 2 * j + kt)) * 256, g, r >> 3, src + 16 * kt);
                    }
        }
        pack_r2(R.part[0], rank, reinterpret_cast<uint16_t *>(base + 2 * RW_HID + 2 * RW_LOG));
        float *sm = reinterpret_cast<float *>(base + RB_SMEM - R_SMALL * 4);
        for (int i = 0; i < 6 * CU; ++i)
            for (int c = 0; c < 3; ++c) sm[i * 3 + c] = m->hI[r_row_at(rank, i) / (2 * CK) * 3 + c];
        float *b = sm + 6 * CU * 3;
        for (int r = 0; r < CU; ++r) { b[r] = m->hb1[CU * rank + r]; b[32 + r] = m->hb3[CU * rank + r]; }
        // tensor memory: lane quadrant q has tiles q and 4 + q, all of K, and quarter q of K (in both halves) of tile 8
        for (int i = 0; i < 16 * CRT; ++i) {
            const int tile = i >> 4;
            const uint16_t *src = &R.part[0][r_row_at(rank, i)];
            for (int kt = 0; kt < 56; ++kt) {
                const int half_f = kt / 28, k = kt % 28, q = tile < 8 ? tile & 3 : k / 7;
                const int c0 = tile < 8 ? ((half_f * 28 + k) * 2 + (tile >> 2)) * 4 : RX_COL + (half_f * 7 + k % 7) * 4;
                cl_pack_tmem_row(base + RB_SMEM, q, c0, i & 7, (i >> 3) & 1, src + 16 * kt);
            }
        }
    });
    ResRowsPack *pk = new ResRowsPack(k);
    if (cudaMalloc((void **)&pk->d_blob, blob.size()) != cudaSuccess || cudaMemcpy(pk->d_blob, blob.data(), blob.size(), cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMalloc((void **)&pk->d_prof, 16 * sizeof(long long)) != cudaSuccess || cudaMemset(pk->d_prof, 0, 16 * sizeof(long long)) != cudaSuccess) {
        cudaGetLastError();
        cudaFree(pk->d_blob); cudaFree(pk->d_prof);
        delete pk;
        m->err = "device allocation for the cluster-resident kernel of many rows failed";
        return WRNN_ERR_NOMEM;
    }
    m->resrows = pk;
    return WRNN_OK;
}

void resrows_destroy(wrnn_model *m)
{
    if (!m->resrows) return;
    cudaFree(m->resrows->d_blob); cudaFree(m->resrows->d_prof);
    delete m->resrows;
    m->resrows = nullptr;
}

int resrows_launch_info(const wrnn_model *m, int batch, int *n_ctas, int *n_threads, int *smem, int64_t *weight_bytes)
{
    int nr, n_clusters;
    rw_geometry(*m->resrows, batch, &nr, &n_clusters);
    if (n_ctas) *n_ctas = n_clusters * CCS;
    if (n_threads) *n_threads = 512;
    if (smem) *smem = (int)rw_launch_smem(nr, m->resrows->checked);
    if (weight_bytes) *weight_bytes = (int64_t)CCS * (int64_t)(RB_SMEM + CB_TMEM);
    return WRNN_OK;
}

int resrows_clusters(const wrnn_model *m, int batch)
{
    int nr, n_clusters;
    rw_geometry(*m->resrows, batch, &nr, &n_clusters);
    return std::min(n_clusters, m->resrows->max_clusters);
}

int resrows_run(wrnn_model *m, const StepArgs &a, cudaStream_t s)
{
    const ResRowsPack &k = *m->resrows;
    ClParams p;
    int n_clusters;
    cl_fill_params(m, a, k.sc, &p);
    rw_geometry(k, a.batch, &p.nr, &n_clusters);
    p.blob = k.d_blob;
    p.prof = m->prof_enabled ? k.d_prof : nullptr;
    if (k.checked) { const char *poke = getenv("WRNN_DEBUG_POKE"); p.poke = poke && poke[0] == '1'; }
    cudaLaunchConfig_t cfg; cudaLaunchAttribute at[1];
    p.smem_bytes = (unsigned)rw_launch_smem(p.nr, k.checked);
    cl_fill_launch(n_clusters, p.smem_bytes, &cfg, at, s);
    void *args[] = {&p};
    const cudaError_t e = cudaLaunchKernelExC(&cfg, rw_kernel_of(p.nr, k.checked ? 2 : cl_wants_dumps(m, p)), args);
    if (e != cudaSuccess) {
        m->err = std::string("cluster-resident kernel of many rows: launch failed: ") + cudaGetErrorString(e);
        cudaGetLastError();
        return WRNN_ERR_CUDA;
    }
    ++g_launches;
    m->prof_cl = 2;
    return WRNN_OK;
}

int resrows_phase_cycles(const wrnn_model *m, long long *out16)
{
    return m->resrows && cudaMemcpy(out16, m->resrows->d_prof, 16 * sizeof(long long), cudaMemcpyDeviceToHost) == cudaSuccess ? WRNN_OK : WRNN_ERR_CUDA;
}

}  // namespace wrnn
