// Cluster-resident persistent sampling kernel: a whole dense H = 896 model lives in ONE 16-CTA cluster, most of the recurrent
// matrix in tensor memory and everything else in shared memory, and a cluster advances its own rows alone.  Three kinds of
// model: bf16 weights, fp32 weights, the Fused Subscale WaveRNN 2x.
//
// A step of the sampler (Fig. 1 of the paper) is a chain of exchanges, not of arithmetic: what bounds it is how long it
// takes to hand the state, the hidden layer and the logits from the SM that computed them to the SMs that need them, twice per
// step.  A bf16 model is 6.1 MB; the shared memory of a 16-CTA cluster is 3.6 MB, but its tensor memory is another 4.2 MB.  With
// the model inside one cluster every exchange is an all-gather through distributed shared memory (measured here: 420 cycles +
// 0.87 per byte and receiver, against 1,000 - 1,500 cycles for the same through L2 and across the chip), clusters never meet, and
// seven of them advance seven times as many rows in the same time.  us per step: 1 to 7 rows 3.27, 8 rows 3.69, 28 rows 4.30
// (the kernels before: 4.73 at one row, 5.6 at 8, 9.5 at 16, 25 at 28; more rows of a bf16 model: wrnn_resrows.cu); fp32 5.0 up to 7
// rows and 6.0 up to 14, with several models alive up to 0.9 more, with where the streamed weights lie (7.4 at one row, 55 and more at several); fused 3.5 (4.54).
//
// Per CTA (rank r of its cluster): state units 28 r .. 28 r + 27 of both halves with their 168 rows of R, rows 28 r .. of O1
// and O3, rows 16 r .. of O2 and O4.
//   * Warps 0..7 are the chain: hidden layer (K split over four warps per tile), logits (K over seven), draw and gates (one row of
//     the batch per warp: every CTA draws every row of its cluster, so that the drawn symbol never leaves the warp), sends.
//   * Warps 8..15 multiply the rows of R in the background, from when the hidden layer is on its way; the chain waits for them
//     after the draw of the fine half (before it: 3.63 us per step at one row).
//   * R: 144 of the 168 rows in tensor memory, the other 24 in shared memory.  Both feed mma.sync: a column is one register of an A
//     fragment for the warps of its lane quadrant, so tcgen05.ld brings four fragments per instruction and no shared-memory
//     load is spent on them.  (tcgen05.mma takes 46 cycles per K = 16 whatever N is up to 64; at eight operand columns mma.sync at 8
//     cycles per sub-partition does three times as much per cycle, and needs no read-back of accumulators: 6.4 us per step
//     with tcgen05.mma.)
//   * fp32 values cross the cluster as high and low fp16 parts of the value scaled by a power of two: 23 bits, so that a quarter of
//     all values are off by a unit in the last place of fp32, 2^-23 at most; bf16 weights are fp16 exactly after such a scaling.  Stored
//     by their producers straight into every receiver's operand image.
//   * What limits the precision is not this but the tensor cores, which cut running sums off instead of rounding them: see r_frag and NCH.
//     2-norm of the error against 64 bits over 300 steps, gates / state / logits, in units of 1e-7 (exact three-way split of the kernel
//     before, plain fp32 for fp32 weights; chains of fourteen products; now): bf16, one row 1.03 / 1.92 / 2.04, 1.18 / 2.30 / 2.69,
//     0.72 / 1.21 / 1.68; fp32, one row 1.03 / 1.90 / 2.00, 1.72 / 3.52 / 4.67, 0.75 / 1.26 / 1.83; fp32, eight rows 0.82 / 1.63 / 1.95,
//     1.72 / 3.54 / 4.55, 0.73 / 1.22 / 1.83; fused 1.05 / 1.88 / 2.11, 1.23 / 2.34 / 2.78, 0.76 / 1.22 / 1.82.  Several bf16 rows per
//     cluster: 0.92 / 1.75 / 2.30 (5.6 / 7.5 / 33 before).
//   * What is sent to one receiver should be one run of bytes, and one instruction of a warp: a single row has an image of its
//     own (112 contiguous bytes per CTA; as one row of four, 16-byte pieces 64 bytes apart: 3.84 us per step, 3.63).
//   * fp32 weights: see W2 below.  Fused: 12 inputs per gate row, 64 logits as four softmaxes of 16.
// What bounds it now, at one row: 3 x 2 all-gathers of 430 - 570 cycles, 2 x 390 for a draw, 2 x 200 for the gates, and products and sums of
// 2 x 500, in 6,500 cycles; stalls are on barriers first.  In the form of 3.39 us: without the shared-
// memory loads of the hidden layer's weights it would be 3.12 us; holding them in registers (setmaxnreg) starves the background
// warps (3.51 - 4.4), loading them half a step ahead delays the logits (3.53).
// Every wait is bounded; a warp that gives up records where, skips its remaining waits and sends and keeps meeting its
// barriers, and all CTAs leave through the final cluster barrier.
#include <algorithm>
#include <cmath>

#include "wrnn_rescl.cuh"

namespace wrnn {

namespace {
constexpr int CPH = 40, CPL = 24;              // floats per (K-split, row) of the partial sums: conflict-free for the fragment owners
constexpr size_t CW_HID = 2 * 28 * 512;                      // O1 (O3) rows of a CTA as A fragments: two tiles
constexpr size_t CW_LOG = 28 * 512;                          // O2 (O4) rows: one tile
// I of the CTA's units [half][gate][unit][3 or 12], b1, b3 (32 each), b2, b4
__host__ __device__ constexpr int cl_small(int kind) { return 2 * 3 * CU * cl_nin(kind) + 2 * 32 + 2 * CL; }
__host__ __device__ constexpr size_t cl_blob_smem(int kind)
{
    return (kind == CL_F32 ? 2 : 1) * (2 * CW_HID + 2 * CW_LOG) + (kind == CL_F32 ? 0 : CW_R2) + cl_small(kind) * 4;
}
static_assert(cl_blob_smem(CL_BF16) % 16 == 0 && cl_blob_smem(CL_F32) % 16 == 0 && cl_blob_smem(CL_FUSED) % 16 == 0, "the blob is copied in 16-byte pieces");
// fp32 weights, second part and the rows without room: [CTA][half][warp][k-tile v of 14][fragments of v][32 lanes][16 B] in an array of
// its own, read from L2
__host__ __device__ constexpr int cl_nf(int rj, int v) { return v < 7 ? (rj ? 2 : 4) : 3; }                       // fragments of a k-tile
__host__ __device__ constexpr int cl_fo(int rj, int v) { return v < 7 ? v * (rj ? 2 : 4) : 7 * (rj ? 2 : 4) + (v - 7) * 3; }   // before it
__host__ __device__ constexpr int cl_fw(int w8) { return w8 < 4 ? w8 * cl_fo(0, 14) : 4 * cl_fo(0, 14) + (w8 - 4) * cl_fo(1, 14); }   // before warp w8
constexpr int CF_HALF = cl_fw(8);                            // fragments of a half: 336
constexpr size_t CB_STREAM = (size_t)2 * CF_HALF * 512;
constexpr size_t C_PART = 7 * 4 * CPL * 4;                   // partial sums of the logits rows; of the hidden rows
static_assert(C_PART >= 4 * 4 * CPH * 4, "the partial sums of both products share a buffer");
constexpr size_t C_PART_R = 4 * 4 * CPR * 4;                 // R h
__host__ __device__ constexpr size_t cl_smem(int kind)
{
    return cl_blob_smem(kind) + 3 * CQ * 64 /* operand images: two state halves, hidden layer */ + 4 * 1024 /* logits */ + C_PART + C_PART_R + 4 * 2 * CU * 2 /* staged state */;
}
constexpr int CL_GUARDS = 8;             // of the checked form: behind the weights, the images (3), logits, sums, R h, staged state
// What a launch asks for: never so little that an SM would take a second CTA, which would wait for the first one's tensor memory
size_t cl_launch_smem(int kind) { return std::max(cl_smem(kind), (size_t)200 * 1024 + 16); }
size_t cl_checked_smem(int kind) { return cl_smem(kind) + CL_GUARDS * CL_GUARD; }
}  // namespace

struct ResClPack {
    uint8_t *d_blob = nullptr;               // [16 ranks][shared memory | tensor memory]
    uint4 *d_stream = nullptr;               // fp32 weights: [16 ranks][CB_STREAM]
    int kind = CL_BF16;
    long long *d_prof = nullptr;             // [16]
    int max_clusters = 0;
    bool checked = false;                    // every call runs the checked form
    ClScales sc;
};

// ROWS: rows of a cluster: 1, 3 (two: sent as they are) or 4 (three or four); fp32 weights 1 or 2.  MODE 0: plain sampling; MODE 1: forced symbols, dumps, phase stamps and the self-test predicate; MODE 2:
// these and the checks.
// Warps 0..7 are the chain: hidden layer, logits, then (one row of the batch each) draw and gates, and all sends.  Warps 8..15
// multiply the rows of R in the background, while the chain waits for exchanges.
// W2: fp32 weights, as high and low fp16 parts (error 2^-23 of a weight).  They are twice as much: the heads and the high parts of
// nine tiles of R stay resident, the rest of R (344 KB per CTA and step) comes from L2 every step, in fragment order, straight
// into the registers of the background warps.
// FUSED: two 16-bit samples per step, one per half of the state, each as four 4-bit softmaxes of 16 consecutive logits; one row.
template <int ROWS, int MODE, int KIND>
__global__ void __launch_bounds__(512, 1) resident_cluster_kernel(const __grid_constant__ ClParams p)
{
    constexpr bool W2 = KIND == CL_F32, FUSED = KIND == CL_FUSED;
    constexpr int NP = W2 ? 2 : 1;                                       // parts of a weight
    constexpr int NIN = cl_nin(KIND), NX = NIN / 3;                      // scalars of I per row, per symbol
    constexpr bool ONE = ROWS == 1, TWO = ROWS == 2;
    constexpr size_t CB_SMEM = cl_blob_smem(KIND), CS_IMG = CQ * 64, CS_PART = C_PART, CS_PARTR = C_PART_R;
    constexpr int CMAXR = 4;
    constexpr int NCH = W2 ? 4 : 2;                                      // chains of a sum in the heads; low parts of weights apart
    constexpr int IR = ONE ? 1 : 4;                                      // rows that share a quad of an operand image
    constexpr bool DBG = MODE != 0, CHK = MODE == 2;
    extern __shared__ __align__(128) uint8_t smem[];
    __shared__ __align__(8) unsigned long long xw, xy[2], xq, xl;        // arrivals: weights, state halves, hidden layer, logits
    __shared__ uint32_t s_tmem;
    __shared__ int s_sym[2][16];                                         // cl_wide_steps
    __shared__ float s_u[2][CMAXR];                                      // [coarse half?][row]: uniform, conditioning frame
    __shared__ int s_fr[2][CMAXR];
    __shared__ long long s_prof[MODE != 0 ? 16 : 1];
    constexpr int H = 2 * CK;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int g4 = lane >> 2, t4 = lane & 3;
    const int cl = blockIdx.x / CCS;
    const int row0 = cl * p.nr, nrc = min(p.nr, p.batch - row0);
    unsigned rank_u;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank_u));
    const int rank = (int)rank_u;

    // ---- shared memory carve-up (must match cl_smem)
    // [half]: O3, O1 ([part][tile]); O4, O2 ([part])
    const uint4 *wH[2] = {reinterpret_cast<const uint4 *>(smem + NP * CW_HID), reinterpret_cast<const uint4 *>(smem)};
    const uint4 *wL[2] = {reinterpret_cast<const uint4 *>(smem + NP * (2 * CW_HID + CW_LOG)), reinterpret_cast<const uint4 *>(smem + NP * 2 * CW_HID)};
    const uint32_t r2_addr = smem_u32(smem + NP * (2 * CW_HID + 2 * CW_LOG));
    const float *sI = reinterpret_cast<const float *>(smem + CB_SMEM - cl_small(KIND) * 4);        // [half][gate][unit][NIN]
    const float *sb1 = sI + 2 * 3 * CU * NIN, *sb3 = sb1 + 32, *sb2 = sb3 + 32, *sb4 = sb2 + CL;
    constexpr size_t G = CHK ? CL_GUARD : 0;
    constexpr size_t X0 = CB_SMEM + G, XSTR = CS_IMG + G, Q0 = X0 + 2 * XSTR, L0 = Q0 + XSTR, P0 = L0 + CMAXR * 1024 + G, R0 = P0 + CS_PART + G,
                     Y0 = R0 + CS_PARTR + G, END = Y0 + CMAXR * 2 * CU * 2 + G;
    uint8_t *ximg = smem + X0;                                           // [2: coarse, fine] state image
    float *lbuf = reinterpret_cast<float *>(smem + L0);                  // [rows][256]
    float *part = reinterpret_cast<float *>(smem + P0);                  // K-split sums of the hidden rows, then of the logits rows
    float *partR = reinterpret_cast<float *>(smem + R0);                 // [4 quarters of K][rows][168]: R h
    uint8_t *ystage = smem + Y0;                                         // [row][quad][16 bytes]: new state values of this CTA's units
    static_assert(END == cl_smem(KIND) + (CHK ? CL_GUARDS * CL_GUARD : 0), "the carve-up is what cl_smem says");
    auto guard = [&](int i) { return smem + (i == 0 ? CB_SMEM : i <= 3 ? X0 + i * XSTR - G : i == 4 ? P0 - G : i == 5 ? R0 - G : i == 6 ? Y0 - G : END - G); };

    // Operand image of a vector: [group][quad][IR rows][high x 4, low x 4] -- a producer's four values of a row travel in one 16-byte
    // store, and the B fragment of lane (column g = row, part; t = quad of the k-tile) is one 8-byte load.  The k order of a tile
    // is permuted accordingly in all weights: slot c holds k = 4 ((c & 7) / 2) + 2 (c / 8) + (c & 1).
    constexpr uint32_t QSTR = 16 * IR;
    auto img_off = [](int st, int quad) { return ONE ? (uint32_t)quad * 16 : (uint32_t)(quad * 4 + st) * 16; };
    const uint32_t frag = t4 * QSTR + (ONE ? g4 & 1 : TWO ? g4 & 3 : g4) * 8;                            // of k-tile 0

    // ---- one-time load: weights, zero images, barriers, tensor memory
    long long s0 = 0;                                                    // steps that cl_wide_steps took
    {
        int wide = 0;
        if (p.h_in)
            for (int i = tid; i < nrc * H; i += 512) wide |= fabsf(__ldcg(p.h_in + (size_t)row0 * H + i)) > CL_WIDE;
        const uint8_t *blob = p.blob + (size_t)rank * (CB_SMEM + CB_TMEM);
        if (tid == 0) {
            mbar_init(smem_u32(&xw), 1); mbar_init(smem_u32(&xy[0]), 1); mbar_init(smem_u32(&xy[1]), 1); mbar_init(smem_u32(&xq), 1); mbar_init(smem_u32(&xl), 1);
            mbar_fence_init();
            fence_proxy_async();
            cl_load_bulk(smem_u32(smem), blob, (uint32_t)CB_SMEM, smem_u32(&xw));
        }
        uint4 *z = reinterpret_cast<uint4 *>(ximg);
        for (int i = tid; i < (int)(3 * XSTR / 16); i += 512) z[i] = make_uint4(0, 0, 0, 0);
        if (warp == 1) {
            asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem)), "r"(512) : "memory");
            asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
        }
        if (DBG && tid < 16) s_prof[tid] = 0;
        tc_fence_before();
        wide = __syncthreads_or(wide);
        tc_fence_after();
        if (wide) {
            cl_await_projection();
            if (tid < nrc) {
                if (FUSED) { s_sym[0][tid] = p.a_in ? p.a_in[0] : 0x8000; s_sym[1][tid] = p.b_in ? p.b_in[0] : 0x8000; }
                else { s_sym[0][tid] = p.c_in ? p.c_in[row0 + tid] : 128; s_sym[1][tid] = p.f_in ? p.f_in[row0 + tid] : 0; }
            }
            __syncthreads();
            s0 = cl_wide_steps<KIND>(p, row0, nrc, rank, partR, s_sym);
            if (rank == 0 && tid < nrc) {
                if (FUSED) { if (p.a_st_out) p.a_st_out[0] = (uint16_t)s_sym[0][0]; if (p.b_st_out) p.b_st_out[0] = (uint16_t)s_sym[1][0]; }
                else { if (p.c_st_out) p.c_st_out[row0 + tid] = (uint8_t)s_sym[0][tid]; if (p.f_st_out) p.f_st_out[row0 + tid] = (uint8_t)s_sym[1][tid]; }
            }
            if (s0 == p.n_steps) {
                mbar_wait(smem_u32(&xw), 0, p.limit_ns);                  // no copy in flight when the CTA leaves
                if (warp == 1) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(s_tmem), "r"(512) : "memory");
                return;
            }
        }
        cl_load_tmem(s_tmem, blob + CB_SMEM, warp, lane);
        cl_await_projection();
        // images of the initial state
        if (p.h_in)
            for (int i = tid; i < nrc * H; i += 512) {
                const int st = i / H, j = i - st * H, half_f = j >= CK, k = j - half_f * CK;
                const float x = __ldcg(p.h_in + (size_t)(row0 + st) * H + j) * CL_STATE;
                __half *im = reinterpret_cast<__half *>(ximg + half_f * XSTR + img_off(st, k >> 2)) + (k & 3);
                im[0] = __float2half_rn(x);
                im[4] = __float2half_rn(x - __half2float(im[0]));
            }
        if (ROWS == 4) fence_proxy_async_cta();                          // before bulk copies of the peers go over what this CTA wrote
    }
    bool bad = !mbar_wait(smem_u32(&xw), 0, p.limit_ns);                 // this thread gave up: it skips waits and sends from here on
    if (bad && atomicCAS(&p.status->code, DEV_OK, DEV_TIMEOUT) == DEV_OK) { p.status->cta = blockIdx.x; p.status->step = 0; p.status->phase = 9; }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (CHK) {
        if (tid < CL_GUARDS) cl_guard_fill(guard(tid));
        if (tid == 0 && END != p.smem_bytes) cl_record(p.status, -2);
        __syncthreads();
        if (p.poke && blockIdx.x == 3 && tid == 0) partR[CS_PARTR / 4] = 0.f;
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

    // ---- rows of R times one half of the state, accumulated over both halves (warps 8..15).  Lane quadrant w & 3 holds a quarter
    // of K of all tiles in its tensor memory; of the two warps of a quadrant one takes tiles 0..3 and the rows in shared memory
    // (a tile and a half), the other tiles 4..8, so that a B fragment is loaded once for five or six tiles (these loads and
    // ldmatrix share the load / store pipe with the chain's shuffles).  Columns: [first warp: half][k-tile][4 tiles][4], then
    // [second warp: half][k-tile][5 tiles][4].
    float acc[6][4];
    const int rq = warp & 3, rj = (warp >> 2) & 1;
    const uint32_t r_col = tmem + ((uint32_t)(32 * rq) << 16) + (rj ? 2 * 7 * 16 : 0);
    auto chains = [](const float (&c)[NCH + NP - 1][4], int k) {
        float v = c[0][k] + c[1][k];
        if constexpr (NCH == 4) v += c[2][k] + c[3][k];
        if constexpr (NP == 2) v += c[NCH][k];
        return v;
    };
    auto r_clear = [&]() {
#pragma unroll
        for (int n = 0; n < 6; ++n)
#pragma unroll
            for (int k = 0; k < 4; ++k) acc[n][k] = 0.f;
    };
    auto r_load = [&](int half_f, int kt, uint32_t (&r)[20]) {
        const uint32_t c = r_col + (uint32_t)((half_f * 7 + kt) * (rj ? 20 : 16));
        tmem_ld16(c, *reinterpret_cast<uint32_t (*)[16]>(&r));
        if (rj) asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];" : "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]) : "r"(c + 16));
    };
    // The tensor cores cut the running sum off after every product instead of rounding it: a chain of fourteen is the largest error
    // of the step.  One row needs two of the eight columns; the other six carry the same row, each pair for every fourth k-tile only,
    // which makes four chains of it (two rows: two chains).  State over 300 steps, 2-norm of the error against 64 bits: 1.75e-7 without,
    // 1.21e-7 with.  Adding every product to the sum with rounded additions instead costs registers: 3.7 us per step at one row.
    auto r_frag = [&](int kt, uint32_t addr) {
        if (!ONE && !TWO) return cl_lds8(addr);
        uint2 v;
        asm volatile("{ .reg .pred p; setp.eq.s32 p, %3, %4; mov.b32 %0, 0; mov.b32 %1, 0; @p ld.shared.v2.b32 {%0,%1}, [%2]; }"
                     : "=&r"(v.x), "=&r"(v.y) : "r"(addr), "r"(ONE ? g4 >> 1 : g4 >> 2), "r"(kt & (ONE ? 3 : 1)) : "memory");
        return v;
    };
    auto r_products = [&](int half_f) {
        const uint32_t b0 = smem_u32(ximg + half_f * XSTR) + 7 * rq * 4 * QSTR + frag;
        const uint32_t a0 = r2_addr + (uint32_t)(((half_f * CK8 + 14 * rq + (lane >> 4)) * CRS + ((lane >> 3) & 1) * 8 + (lane & 7)) * 16);
        const uint32_t a1 = r2_addr + (uint32_t)(((half_f * CK8 + 14 * rq + ((lane >> 3) & 1)) * CRS + 16 + (lane & 7)) * 16);
        uint32_t r0[20], r1[20], t0[6], t1[6];
        r_load(half_f, 0, r0);
        uint2 c0, c1;
        auto load = [&](int kt, uint2 &b, uint32_t (&t)[6]) {
            b = r_frag(kt, b0 + kt * 4 * QSTR);
            if (!rj) {
                cl_ldmatrix4(a0 + kt * 2 * CRS * 16, *reinterpret_cast<uint32_t (*)[4]>(&t));
                asm volatile("ldmatrix.sync.aligned.m8n8.x2.shared.b16 {%0,%1}, [%2];" : "=r"(t[4]), "=r"(t[5]) : "r"(a1 + kt * 2 * CRS * 16) : "memory");
            }
        };
        auto mmas = [&](const uint32_t (&r)[20], const uint2 &b, const uint32_t (&t)[6]) {
#pragma unroll
            for (int n = 0; n < 4; ++n)
                cl_mma(acc[n], make_uint4(r[4 * n], r[4 * n + 1], r[4 * n + 2], r[4 * n + 3]), b.x, b.y);
            if (rj) cl_mma(acc[4], make_uint4(r[16], r[17], r[18], r[19]), b.x, b.y);
            else {
                cl_mma(acc[4], make_uint4(t[0], t[1], t[2], t[3]), b.x, b.y);
                cl_mma(acc[5], make_uint4(t[4], 0, t[5], 0), b.x, b.y);
            }
        };
        load(0, c0, t0);
#pragma unroll
        for (int kt = 0; kt < 7; ++kt) {
            tmem_wait_ld();
            if (kt & 1) { if (kt < 6) { r_load(half_f, kt + 1, r0); load(kt + 1, c0, t0); } mmas(r1, c1, t1); }
            else { if (kt < 6) { r_load(half_f, kt + 1, r1); load(kt + 1, c1, t1); } mmas(r0, c0, t0); }
        }
    };
    // the parts of a value are adjacent columns
    auto part_sum = [&](const float (&c)[4], float &lo, float &hi) { lo = c[0] + c[1]; hi = c[2] + c[3]; };
    // Sums over the chains of N values, of which each lane gets its part, from the one that is returned on
    auto chain_sum = [&](auto &v, auto N_C) {
        constexpr int N = decltype(N_C)::value;
        if (TWO) { cl_fold<N>(v, 2, lane); return N / 2 * (t4 >> 1); }
        cl_fold<N>(v, 1, lane); cl_fold<N / 2>(v, 2, lane);
        return N / 4 * (2 * (t4 & 1) + (t4 >> 1));
    };
    auto r_store = [&]() {
        if (ONE) {
            float v[12];
#pragma unroll
            for (int n = 0; n < 5; ++n) part_sum(acc[n], v[2 * n], v[2 * n + 1]);
            v[10] = acc[5][0] + acc[5][1]; v[11] = 0.f;
            const int i0 = chain_sum(v, std::integral_constant<int, 12>{});
            float *d = partR + rq * 4 * CPR + g4;
#pragma unroll
            for (int i = 0; i < 3; ++i)
                if (i0 + i < (rj ? 10 : 11)) d[8 * (i0 + i) + (rj ? 64 : i0 + i < 8 ? 0 : 80)] = v[i];
            return;
        }
        float *d = partR + (rq * 4 + t4) * CPR + g4;
#pragma unroll
        for (int n = 0; n < 4; ++n) part_sum(acc[n], d[(4 * rj + n) * 16], d[(4 * rj + n) * 16 + 8]);
        part_sum(acc[4], d[(rj ? 8 : 9) * 16], d[(rj ? 8 : 9) * 16 + 8]);
        if (!rj) d[160] = acc[5][0] + acc[5][1];
    };

    // fp32 weights: two passes over a half of the state, first the tiles that hold the coarse rows (0..3 and 4, 5), then the others
    // (9 and 10; 6..8).  High parts of tiles 0..8 from tensor memory, the other fragments from L2, requested three k-tiles ahead
    // (some 40 KB in flight per SM) across passes and halves, so that a half-step starts with its first fragments there.  Tile 10
    // has eight rows: its high and low parts share a fragment.
    const uint4 *stream = p.stream + ((size_t)rank * 2 * CF_HALF + cl_fw(warp & 7)) * 32 + lane;
    uint4 sf[W2 ? 3 : 1][4];
    auto w2_request = [&](auto RJ_C, int half_f, auto V_C) {              // k-tile v of the 14 of a half: slot v % 3 (15 are counted)
        constexpr int RJ = decltype(RJ_C)::value, V = decltype(V_C)::value, NF = cl_nf(RJ, V);
        if (!W2) return;
        const uint4 *src = stream + (size_t)(half_f * CF_HALF + cl_fo(RJ, V)) * 32;
#pragma unroll
        for (int i = 0; i < NF; ++i) sf[W2 ? V % 3 : 0][i] = cl_ldg_stream(src + i * 32);
    };
    float keep[2][ONE ? 2 : 4];                                          // sums over the coarse half, per pass
    auto w2_half = [&](auto RJ_C, int half_f, auto start, auto mid) {
        constexpr int RJ = decltype(RJ_C)::value;
        const uint32_t b0 = smem_u32(ximg + half_f * XSTR) + 7 * rq * 4 * QSTR + frag;
        const uint32_t c0 = r_col + (uint32_t)(half_f * 7 * (RJ ? 20 : 16));
        float sum[4][4], low[TWO ? 4 : 1][4];                            // per tile; two rows, with half the chains: low parts of the weights apart
        start();
        cl_for<14>([&](auto V_C) {
            constexpr int V = decltype(V_C)::value, PASS = V / 7, KT = V % 7;
            constexpr int NTM = PASS == 0 ? (RJ ? 2 : 4) : (RJ ? 3 : 0);  // tiles in tensor memory, of which the low parts are streamed
            constexpr int NF = cl_nf(RJ, V);
            if (KT == 0)
#pragma unroll
                for (int n = 0; n < 16; ++n) {
                    sum[n >> 2][n & 3] = 0.f;
                    if (TWO) low[TWO ? n >> 2 : 0][n & 3] = 0.f;
                }
            uint32_t r[16];
            if (NTM == 4) tmem_ld16(c0 + KT * 16, r);
            else if (NTM >= 2) {
                const uint32_t c = c0 + KT * 20 + (PASS ? 8 : 0);
                asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];" : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]),
                             "=r"(r[6]), "=r"(r[7]) : "r"(c));
                if (NTM == 3) asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];" : "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]) : "r"(c + 8));
            }
            const uint2 b = r_frag(KT, b0 + KT * 4 * QSTR);
            tmem_wait_ld();
#pragma unroll
            for (int n = 0; n < NTM; ++n) cl_mma(sum[n], make_uint4(r[4 * n], r[4 * n + 1], r[4 * n + 2], r[4 * n + 3]), b.x, b.y);
#pragma unroll
            for (int i = 0; i < NF; ++i) {
                constexpr int TILES = NTM ? 1 : 2;                       // (tile 9: both parts, tile 10)
                if (TWO && (NTM || i == 1)) cl_mma(low[TWO ? i / TILES : 0], sf[W2 ? V % 3 : 0][i], b.x, b.y);
                else cl_mma(sum[i / TILES], sf[W2 ? V % 3 : 0][i], b.x, b.y);
            }
            if constexpr (V < 11) w2_request(RJ_C, half_f, std::integral_constant<int, V + 3>{});
            if constexpr (V >= 12) w2_request(RJ_C, 1 - half_f, std::integral_constant<int, V - 12>{});
            if constexpr (V == 13) w2_request(RJ_C, 1 - half_f, std::integral_constant<int, 2>{});
            if constexpr (KT == 6) {
                // the rows of this pass, eight apart: 64 and 96 (RJ), 0 and 144
                constexpr int N = PASS == 0 ? (RJ ? 4 : 8) : (RJ ? 6 : 3), NV = N > 4 ? 8 : 4, M = NV / (ONE ? 4 : 2), ROW = RJ ? 64 + 32 * PASS : 144 * PASS;
                float v[NV] = {};
#pragma unroll
                for (int n = 0; n < N / 2; ++n) {
                    part_sum(sum[n], v[2 * n], v[2 * n + 1]);
                    if (TWO) { const int l = TWO ? n : 0; v[2 * n] += low[l][0] + low[l][1]; v[2 * n + 1] += low[l][2] + low[l][3]; }
                }
                if (N == 3) v[2] = (sum[1][0] + sum[1][1]) + (sum[1][2] + sum[1][3]);     // tile 10: its low parts are the lower rows
                const int i0 = chain_sum(v, std::integral_constant<int, NV>{});
                float *d = partR + (rq * 4 + (ONE ? 0 : t4 & 1)) * CPR + ROW + g4;
#pragma unroll
                for (int i = 0; i < M; ++i) {
                    if (!half_f) keep[PASS][i] = v[i];
                    else if (i0 + i < N) d[8 * (i0 + i)] = keep[PASS][i] + v[i];
                }
                if (V == 6) mid();
            }
        });
    };

    // ---- fixed addresses
    const uint32_t sbase = smem_u32(smem);
    // Receivers of what this warp sends, as what to add to an address of mine.  Several rows: a lane stores its piece into each of
    // them in turn.  One row: a lane has a receiver and a piece, so that a warp sends with one instruction.
    uint32_t dy[2], delta4[4];                                           // state: CTAs (warp & 7) + 8 k; hidden layer, logits: (warp & 3) + 4 k
#pragma unroll
    for (int k = 0; k < 2; ++k) dy[k] = map_to_rank(sbase, (unsigned)((warp & 7) + 8 * (ONE ? lane / 7 & 1 : k))) - sbase;
#pragma unroll
    for (int k = 0; k < 4; ++k) delta4[k] = map_to_rank(sbase, (unsigned)((warp & 3) + 4 * (ONE ? lane / 7 & 3 : k))) - sbase;
    const uint32_t delta_l = map_to_rank(sbase, (unsigned)((warp & 3) + 4 * (FUSED ? lane & 3 : lane >> 2 & 3))) - sbase;
    // A lane's piece of this CTA's 28 values: four values of a row, lane = (row of a group of four, quad)
    const int pc_a = lane / 7, pc_quad = lane - 7 * pc_a;
    const bool pc_on = lane < 28;
    const uint32_t pc_off = img_off(pc_a & 3, 7 * rank + pc_quad);
    const int skip_at = (DBG && rank == p.skip_rank) ? (int)(p.skip_step - s0) : -1;

    // ---- the row this warp draws (warps 0..7), its last symbols, and the gates of its unit (lane) in both halves
    const bool drawer = warp < nrc;
    const int st_d = warp & 7, gb = row0 + (drawer ? st_d : 0);          // row of the call
    const bool gater = drawer && lane < CU;
    const int gu = lane < CU ? lane : 0, gj = CU * rank + gu;
    int c_prev = 128, f_prev = 0;
    float hC = 0.f, hF = 0.f;
    if (drawer) {
        if (s0 > 0) { c_prev = s_sym[0][st_d]; f_prev = s_sym[1][st_d]; }
        else if (FUSED) { c_prev = p.a_in ? p.a_in[0] : 0x8000; f_prev = p.b_in ? p.b_in[0] : 0x8000; }
        else { c_prev = p.c_in ? p.c_in[gb] : 128; f_prev = p.f_in ? p.f_in[gb] : 0; }
    }
    auto xin = [](int v, int k) { return FUSED ? scale4((v >> (12 - 4 * k)) & 15) : scale8(v); };    // scalar k of a symbol as the network sees it
    if (gater && p.h_in) { hC = __ldcg(p.h_in + (size_t)gb * H + gj); hF = __ldcg(p.h_in + (size_t)gb * H + CK + gj); }
    const bool writer = drawer && rank == 2 * st_d;                      // the CTA whose drawing warp writes this row's samples
    int drawn_out = 0;
    int16_t *out_row = p.out ? p.out + (long long)(FUSED ? 0 : gb) * p.out_pitch + s0 : nullptr;
    const float *g_row = p.g + (size_t)gb * p.n_frames * 3 * H + gj;

    float dbg_v[4] = {0.f, 0.f, 0.f, 0.f};                               // what the dumps want of this half-step's gates
    auto dump_gates = [&](int half_g, long long s) {
        const int jj = half_g * CK + gj;
        if (p.dbg_gates) { float *o = p.dbg_gates + ((size_t)(s0 + s) * p.batch + gb) * 3 * H; o[jj] = dbg_v[0]; o[H + jj] = dbg_v[1]; o[2 * H + jj] = dbg_v[2]; }
        if (p.dbg_h) p.dbg_h[((size_t)(s0 + s) * p.batch + gb) * H + jj] = dbg_v[3];
    };
    struct GatePre { float pu, pr, pe, ae, ku[NX], kr[NX], ke[NX]; };
    // a row of R h of this row of the batch
    auto r_row = [&](int i) {
        const float *q = partR + st_d * CPR + i;
        const float v = (q[0] + q[4 * CPR]) + (q[8 * CPR] + q[12 * CPR]);
        return v * p.sc.inv_R;
    };
    // everything of the gates of one half that does not depend on the pending draw
    auto gates_prepare = [&](int half_g, const float (&gv)[3]) {
        GatePre q;
        const float *Iu = sI + ((half_g * 3 + 0) * CU + gu) * NIN, *Ir = Iu + CU * NIN, *Ie = Ir + CU * NIN;
        // fine units: the last symbols of both halves are known, the coarse one of this step is pending; coarse units: the coarse
        // symbol is known, the fine one pending
        float su = gv[0], sr = gv[1], se = gv[2];
#pragma unroll
        for (int k = 0; k < NX; ++k) {
            if (half_g) { const float x = xin(f_prev, k); su = fmaf(Iu[NX + k], x, su); sr = fmaf(Ir[NX + k], x, sr); se = fmaf(Ie[NX + k], x, se); }
            const float x = xin(c_prev, k);
            su = fmaf(Iu[k], x, su); sr = fmaf(Ir[k], x, sr); se = fmaf(Ie[k], x, se);
        }
        q.pu = su; q.pr = sr; q.pe = se; q.ae = 0.f;
        const int pend = half_g ? 2 * NX : NX;
#pragma unroll
        for (int k = 0; k < NX; ++k) { q.ku[k] = Iu[pend + k]; q.kr[k] = Ir[pend + k]; q.ke[k] = Ie[pend + k]; }
        return q;
    };
    auto gates_add_r = [&](int half_g, GatePre &q) {
        q.pu += r_row(half_g * 3 * CU + gu);
        q.pr += r_row(half_g * 3 * CU + CU + gu);
        q.ae = r_row(half_g * 3 * CU + 2 * CU + gu);
    };
    auto gates_and_stage = [&](int half_g, long long s, int drawn, const GatePre &q) {
        float pu = q.pu, pr = q.pr, pe = q.pe;
#pragma unroll
        for (int k = 0; k < NX; ++k) {
            const float xk = xin(drawn, k);
            pu = fmaf(q.ku[k], xk, pu); pr = fmaf(q.kr[k], xk, pr); pe = fmaf(q.ke[k], xk, pe);
        }
        const float u = cl_sigmoid(pu), r = cl_sigmoid(pr);
        const float e = cl_tanh(fmaf(r, q.ae, pe));
        const float hn = fmaf(u, half_g ? hF : hC, (1.0f - u) * e);
        if (half_g) hF = hn; else hC = hn;
        if (gater) {
            __half *d = reinterpret_cast<__half *>(ystage + ((lane >> 2) * IR + (ONE ? 0 : st_d)) * 16) + (lane & 3);
            const float x = hn * CL_STATE;
            const __half hi = __float2half_rn(x);
            d[0] = hi;
            d[4] = __float2half_rn(x - __half2float(hi));
            if (DBG) { dbg_v[0] = u; dbg_v[1] = r; dbg_v[2] = e; dbg_v[3] = hn; }
        }
        if (ROWS == 4) fence_proxy_async_cta();
    };
    // three rows of a group travel as four: 48-byte runs in the receivers' images are slower than 64-byte ones (21 rows: 4.74 us
    // per step with three, 4.52 with four)
    const int nsend = (nrc & 3) == 3 ? nrc + 1 : nrc;
    // warps 0..7: the staged state values of this CTA's units -> images in the cluster's CTAs, two each.  Three or four rows: as one copy, which keeps the load /
    // store pipe free for the background warps (16 rows 4.24 -> 4.15, 28 rows 4.39 -> 4.31 us per step; one row 3.32 -> 3.44, two 3.70 -> 3.81: not they).
    // (The staged values are overwritten when logits have come that depend on what every CTA made of these copies.)
    constexpr uint32_t SLICE = 7 * 16 * IR;
    constexpr bool BULK = ROWS == 4;
    const uint32_t dyb = map_to_rank(sbase, (unsigned)((warp & 7) + 8 * (lane & 1))) - sbase;
    auto send_y = [&](int half_g, long long s) {
        if constexpr (BULK) {
            if (bad || lane >= 2 || (DBG && (int)s == skip_at) || !store_ok(rank * SLICE, SLICE, CS_IMG)) return;
            cl_copy_bulk(sbase + (uint32_t)(X0 + half_g * XSTR) + rank * SLICE + dyb, smem_u32(ystage), SLICE, smem_u32(&xy[half_g]) + dyb);
        } else {
            if (bad || (ONE ? lane >= 14 : !pc_on) || (DBG && (int)s == skip_at)) return;
            const uint32_t a = sbase + (uint32_t)(X0 + half_g * XSTR) + pc_off, bar = smem_u32(&xy[half_g]);
            if ((ONE || pc_a < nsend) && store_ok(pc_off, 16, CS_IMG)) {
                const uint4 v = *reinterpret_cast<const uint4 *>(ystage + (pc_quad * IR + (ONE ? 0 : pc_a)) * 16);
#pragma unroll
                for (int k = 0; k < (ONE ? 1 : 2); ++k) cl_st_async16(a + dy[k], v, bar + dy[k]);
            }
        }
    };
    const int n_draw = 32 * nrc;                                         // threads of the drawing warps
    const unsigned qbytes = (unsigned)(nsend * CK * 4), ybytes = BULK ? CCS * SLICE : qbytes, lbytes = FUSED ? 256u : (unsigned)(nrc * 1024);

    // ---- warp 7 prepares, one row per lane, what the draws of a half-step need: the uniform and the conditioning frame (the
    // same for both halves of a step), tracked without a division per step
    long long w_pos = 0;
    int w_frame = 0, w_rem = 0;
    const int w_q = p.row_lag > 0 ? 1 : p.row_stride / p.hop, w_r = p.row_lag > 0 ? 0 : p.row_stride - w_q * p.hop;      // staggered rows: a frame per step of the call
    auto prepare_rows = [&](int half, long long s) {                     // of half-step 2 s + half
        if (lane < (FUSED ? 4 : nrc)) {                                  // FUSED: one lane per nibble
            const long long t = half ? s : s - 1;
            s_u[half][lane] = uniform24(p.seed, p.stream0 + (unsigned)(row0 + (FUSED ? 0 : lane)), (unsigned long long)(w_pos + t),
                                        FUSED ? (half ? 0u : 4u) + (unsigned)lane : (half ? 0u : 1u));
            if (!half) {                                                 // the fine half computes the coarse gates of step s
                w_frame += w_q; w_rem += w_r;
                if (w_rem >= p.hop) { w_rem -= p.hop; ++w_frame; }
            }
            s_fr[half][lane] = w_frame;
        }
    };
    if (warp == 7 && lane < (FUSED ? 4 : nrc)) {
        const long long b = row0 + (FUSED ? 0 : lane), pos = p.row_lag > 0 ? s0 * p.hop : (p.step0 + s0) * p.row_stride + ((long long)p.stream0 + b) * p.row_offset_mul;
        w_pos = p.step0 + s0 - b * p.row_lag;
        w_frame = (int)(pos / p.hop); w_rem = (int)(pos - (long long)w_frame * p.hop);
        prepare_rows(1, 0);
    }

    // ---- prologue: R h of the initial state, coarse gates of step 0
    if (warp >= 8) {
        if (W2) {
            auto pro = [&](auto RJ_C) {
                cl_for<3>([&](auto V_C) { w2_request(RJ_C, 0, V_C); });
#pragma unroll 1
                for (int half_f = 0; half_f < 2; ++half_f) w2_half(RJ_C, half_f, [] {}, [] {});
            };
            if (rj) pro(std::integral_constant<int, 1>{});
            else pro(std::integral_constant<int, 0>{});
        } else {
            r_clear();
#pragma unroll 1
            for (int half_f = 0; half_f < 2; ++half_f) r_products(half_f);
            r_store();
        }
    }
    if (tid == 0) mbar_arrive_expect(smem_u32(&xy[0]), ybytes);
    __syncthreads();
    // The products above read the images of the initial state, over which the peers store their first one: nobody sends before
    // every CTA has arrived here (the loop needs nothing of the kind: whoever sends has received something from everybody)
    cl_cluster_arrive();
    if (drawer) {
        float gv[3];
        const float *g = g_row + (size_t)s_fr[1][st_d] * 3 * H;
#pragma unroll
        for (int gate = 0; gate < 3; ++gate) gv[gate] = __ldg(g + gate * H);
        GatePre gp = gates_prepare(0, gv);
        gates_add_r(0, gp);
        gates_and_stage(0, 0, f_prev, gp);
    }
    __syncthreads();
    cl_cluster_wait();
    if (warp < 8) send_y(0, 0);
    if (DBG && gater) dump_gates(0, 0);

    // Half-step n = 2 s + 1 is the coarse half of step s (input y_c(s): coarse head -> c_s, then the fine gates of step s),
    // n = 2 s the fine half (input y_f(s - 1): fine head -> f_{s-1}, R h_{s-1} completed, then the coarse gates of step s).
    // A peer may overwrite an image, a sum or the logits only after it has received what this CTA sends after its last use.
    const unsigned T = (unsigned)(p.n_steps - s0);                       // (a call has fewer than 2^31 steps)
    auto half_step = [&](auto HALF_C, const unsigned n) {
        constexpr int half = decltype(HALF_C)::value;                    // 1: coarse half
        constexpr int in = half ? 0 : 1;                                 // image of its input
        const long long s = n >> 1;
        const bool last = n == 2 * T;
        const unsigned yuse = (n - 1) >> 1, quse = n - 1;
        const uint32_t xin = sbase + (uint32_t)(X0 + in * XSTR), qin = sbase + (uint32_t)Q0;
        if (tid == 0 && !bad) {
            mbar_arrive_expect(smem_u32(&xq), qbytes);
            mbar_arrive_expect(smem_u32(&xl), lbytes);
            if (!last) mbar_arrive_expect(smem_u32(&xy[half]), ybytes);
        }
        float gv[3] = {0.f, 0.f, 0.f}, u01 = 0.f;
        int forced = -1;
        if (drawer) {
            u01 = s_u[half][FUSED ? lane >> 3 : st_d];
            const float *g = g_row + (size_t)s_fr[half][st_d] * 3 * H + half * CK;
            if (!last)
#pragma unroll
                for (int gate = 0; gate < 3; ++gate) gv[gate] = __ldg(g + gate * H);
            if (DBG) {
                if (FUSED) {
                    const uint16_t *fz = half ? p.a_forced : p.b_forced;
                    if (fz) forced = fz[s0 + (half ? s : s - 1)];
                } else {
                    const uint8_t *fz = half ? p.c_forced : p.f_forced;
                    if (fz) forced = fz[(size_t)gb * p.n_steps + s0 + (half ? s : s - 1)];
                }
            }
        }
        // ---- hidden layer: this CTA's 28 rows (two tiles), K in four quarters; weight fragments before the wait
        {
            uint4 av[NP][7];
            const int tile = warp & 1, split = warp >> 1;
            const uint4 *A = wH[half] + (tile * 28 + 7 * split) * 32 + lane;
#pragma unroll
            for (int w = 0; w < NP; ++w)
#pragma unroll
                for (int i = 0; i < 7; ++i) av[w][i] = A[w * (CW_HID / 16) + i * 32];
            STAMP0();
            wait_bar(&xy[in], yuse, (int)s, 1 + 4 * half);
            if (W2) cl_bar_arrive(half ? 5 : 7, 512);
            STAMP(8 * half + 0);
            const uint32_t b0 = xin + 7 * split * 4 * QSTR + frag;
            uint2 b[7];
            float acc[NCH + NP - 1][4];
#pragma unroll
            for (int i = 0; i < 7; ++i)
                b[i] = cl_lds8(b0 + i * 4 * QSTR);
#pragma unroll
            for (int k = 0; k < 4 * (NCH + NP - 1); ++k) acc[k >> 2][k & 3] = 0.f;
#pragma unroll
            for (int i = 0; i < 7; ++i)
#pragma unroll
                for (int w = 0; w < NP; ++w) cl_mma(acc[w ? NCH : i % NCH], av[w][i], b[i].x, b[i].y);
#pragma unroll
            for (int k = 0; k < 4; ++k) acc[0][k] = chains(acc, k);
            float *d = part + (split * 4 + t4) * CPH + tile * 16 + g4;
            if (!ONE || t4 == 0) part_sum(acc[0], d[0], d[8]);
        }
        cl_bar_sync(1, 256);
        STAMP(8 * half + 1);
        // ---- K-split sums, bias, relu, parts; every sending warp adds up the same sums (cheaper than a hand-over) and serves
        // four CTAs: warps 0..3 the first group of rows, 4..7 the second
        if (warp < 4 && pc_on) {
            const int st = ONE ? 0 : pc_a;
            if (st < nsend && !bad && store_ok(pc_off, 16, CS_IMG)) {
                const float4 bias = *reinterpret_cast<const float4 *>((half ? sb1 : sb3) + 4 * pc_quad);
                float4 v = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
                for (int sp = 0; sp < 4; ++sp) {
                    const float4 a = *reinterpret_cast<const float4 *>(part + (sp * 4 + st) * CPH + 4 * pc_quad);
                    v.x += a.x; v.y += a.y; v.z += a.z; v.w += a.w;
                }
                const float inv = p.sc.inv_O1[1 - half];
                const float qs = p.sc.q_scale[1 - half];
                v.x = fmaxf(fmaf(v.x, inv, bias.x), 0.f) * qs; v.y = fmaxf(fmaf(v.y, inv, bias.y), 0.f) * qs;
                v.z = fmaxf(fmaf(v.z, inv, bias.z), 0.f) * qs; v.w = fmaxf(fmaf(v.w, inv, bias.w), 0.f) * qs;
                uint2 lo;
                const uint2 hi = cl_split4(v.x, v.y, v.z, v.w, lo);
                const uint32_t a = qin + pc_off, bar = smem_u32(&xq);
#pragma unroll
                for (int k = 0; k < (ONE ? 1 : 4); ++k) cl_st_async16(a + delta4[k], make_uint4(hi.x, hi.y, lo.x, lo.y), bar + delta4[k]);
            }
        }
        cl_bar_sync(W2 && !half ? 6 : 2, 512);   // the background warps are done with the last half-step (and, bf16, go on)
        STAMP(8 * half + 2);
        // ---- the cluster's hidden layer -> this CTA's 16 logits rows, K over seven warps
        if (warp < 7) {
            uint4 lv[NP][4];
            const uint4 *A = wL[half] + 4 * warp * 32 + lane;
#pragma unroll
            for (int w = 0; w < NP; ++w)
#pragma unroll
                for (int i = 0; i < 4; ++i) lv[w][i] = A[w * (CW_LOG / 16) + i * 32];
            const float4 lbias = *reinterpret_cast<const float4 *>((half ? sb2 : sb4) + (FUSED ? 0 : 4 * (lane & 3)));
            wait_bar(&xq, quse, (int)s, 2 + 4 * half);
            STAMP(8 * half + 3);
            const uint32_t b0 = qin + 4 * warp * 4 * QSTR + frag;
            uint2 b[4];
            float acc[NCH + NP - 1][4];
#pragma unroll
            for (int i = 0; i < 4; ++i)
                b[i] = cl_lds8(b0 + i * 4 * QSTR);
#pragma unroll
            for (int k = 0; k < 4 * (NCH + NP - 1); ++k) acc[k >> 2][k & 3] = 0.f;
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int w = 0; w < NP; ++w) cl_mma(acc[w ? NCH : i % NCH], lv[w][i], b[i].x, b[i].y);
#pragma unroll
            for (int k = 0; k < 4; ++k) acc[0][k] = chains(acc, k);
            float *d = part + (warp * 4 + t4) * CPL + g4;
            if (!ONE || t4 == 0) part_sum(acc[0], d[0], d[8]);
            if (warp >= 4) cl_bar_arrive(3, 224);
            else {
                cl_bar_sync(3, 224);
                STAMP(8 * half + 4);
                if (lane < (FUSED ? 4 : ONE ? 16 : 4 * nrc) && !bad) {
                    const int st = ONE ? 0 : lane >> 2;
                    float4 v = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
                    for (int sp = 0; sp < 7; ++sp) {
                        const float4 a = *reinterpret_cast<const float4 *>(part + (sp * 4 + st) * CPL + (FUSED ? 0 : 4 * (lane & 3)));
                        v.x += a.x; v.y += a.y; v.z += a.z; v.w += a.w;
                    }
                    const float inv = p.sc.inv_O2[1 - half];
                    const uint32_t a = smem_u32(lbuf + (FUSED ? 4 * rank : st * 256 + CL * rank + 4 * (lane & 3))), bar = smem_u32(&xl);
#pragma unroll
                    for (int k = 0; k < (ONE ? 1 : 4); ++k) {
                        const uint32_t d = ONE ? delta_l : delta4[k];
                        if (CHK && !store_ok(a - smem_u32(lbuf), 16, CMAXR * 1024)) continue;
                        st_async_v4(a + d, fmaf(v.x, inv, lbias.x), fmaf(v.y, inv, lbias.y), fmaf(v.z, inv, lbias.z), fmaf(v.w, inv, lbias.w), bar + d);
                    }
                }
                STAMP(8 * half + 5);
            }
        } else if (!last) prepare_rows(1 - half, half ? s + 1 : s);
        float dbg_l[8] = {};
        // ---- one row per warp: what does not depend on the draw, the draw, the gates
        if (drawer) {
            GatePre gp = gates_prepare(half, gv);
            if (half) gates_add_r(half, gp);
            wait_bar(&xl, quse, (int)s, 3 + 4 * half);
            STAMP0();
            float l[8];
            int drawn;
            if (FUSED) {
                // 64 logits: two per lane; lanes [8 k, 8 k + 8) are the softmax of nibble k (most significant first)
                const float2 a = reinterpret_cast<const float2 *>(lbuf)[lane];
                l[0] = a.x; l[1] = a.y;
                const int nib = group16_softmax_draw(l[0], l[1], u01, lane);
                drawn = (__shfl_sync(FULL, nib, 0) << 12) | (__shfl_sync(FULL, nib, 8) << 8) | (__shfl_sync(FULL, nib, 16) << 4) | __shfl_sync(FULL, nib, 24);
            } else {
                const float4 a = *reinterpret_cast<const float4 *>(lbuf + st_d * 256 + 8 * lane), b = *reinterpret_cast<const float4 *>(lbuf + st_d * 256 + 8 * lane + 4);
                l[0] = a.x; l[1] = a.y; l[2] = a.z; l[3] = a.w; l[4] = b.x; l[5] = b.y; l[6] = b.z; l[7] = b.w;
                drawn = cl_draw(l, u01, lane);
            }
            const int fed = (DBG && forced >= 0) ? forced : drawn;
            STAMP(8 * half + 6);
            if (!half) {
                cl_bar_sync(4, 256 + n_draw);                            // R h is complete: as a rule not before the draw (3.63 us per step with the wait there)
                gates_add_r(half, gp);
            }
            if (!last) gates_and_stage(half, s, fed, gp);
            STAMP(8 * half + 7);
            if (half) c_prev = fed; else f_prev = fed;
            drawn_out = drawn;
            if (DBG)
#pragma unroll
                for (int k = 0; k < (FUSED ? 2 : 8); ++k) dbg_l[k] = l[k];
        }
        if (!last) {
            cl_bar_sync(1, 256);
            send_y(half, s);
        }
        // the samples (and the dumps) leave when the state is on its way
        if (DBG && gater && !last && !bad) dump_gates(half, s);
        if (DBG && p.dbg_logits && writer && !bad) {
            float *d = p.dbg_logits + (((size_t)(s0 + (half ? s : s - 1)) * p.batch + gb) * 2 + (half ? 0 : 1)) * (FUSED ? 64 : 256) + (FUSED ? 2 : 8) * lane;
#pragma unroll
            for (int k = 0; k < (FUSED ? 2 : 8); ++k) d[k] = dbg_l[k];
        }
        if (writer && lane == 0 && !bad) {
            if (DBG) {
                if (FUSED) {
                    uint16_t *o = half ? p.a_out : p.b_out;
                    if (o) o[s0 + (half ? s : s - 1)] = (uint16_t)drawn_out;
                } else {
                    uint8_t *o = half ? p.c_out : p.f_out;
                    if (o) o[(size_t)gb * p.n_steps + s0 + (half ? s : s - 1)] = (uint8_t)drawn_out;
                }
            }
            // (fused: the two streams side by side, a_s and the sample part B emits in step s)
            if (FUSED) { if (out_row) out_row[half ? s : p.n_steps + s - 1] = (int16_t)((half ? c_prev : f_prev) - 32768); }
            else if (!half && out_row) out_row[s - 1] = (int16_t)(256 * c_prev + f_prev - 32768);
        }
    };
    if (warp < 8) {
#pragma unroll 1
        for (unsigned s2 = 0; s2 < T; ++s2) {
            half_step(std::integral_constant<int, 1>{}, 2 * s2 + 1);
            half_step(std::integral_constant<int, 0>{}, 2 * s2 + 2);
        }
    } else {
        // ---- the rows of R, right after the hidden layer is sent (its sums and sends do not share the load / store pipe with them)
        if (W2) {
            // More to do: it starts as soon as the half of the state is there (barriers 5 and 7, at which the chain only arrives), and
            // the coarse rows come first, the others when the gates have theirs.  Barriers 2 and 6, at which these warps only
            // arrive, tell the chain that the products of the last half-step are done.  Both alternate: whoever only arrives may
            // be one half-step ahead of the others, and cannot be two, because the other pair of barriers lies between.
            auto loop = [&](auto RJ_C) {
#pragma unroll 1
                for (unsigned n = 0; n < 2 * T; ++n) {
                    const int half_f = (int)(n & 1);
                    w2_half(RJ_C, half_f, [&] { cl_bar_arrive(half_f ? 6 : 2, 512); cl_bar_sync(half_f ? 7 : 5, 512); },
                            [&] { if (half_f) cl_bar_arrive(4, 256 + n_draw); });
                }
            };
            if (rj) loop(std::integral_constant<int, 1>{});
            else loop(std::integral_constant<int, 0>{});
        } else {
#pragma unroll 1
            for (unsigned s2 = 0; s2 < T; ++s2) {
                r_clear();
                cl_bar_sync(2, 512);
                r_products(0);
                cl_bar_sync(2, 512);
                r_products(1);
                r_store();
                cl_bar_arrive(4, 256 + n_draw);
            }
        }
    }
#undef STAMP
#undef STAMP0

    // ---- results; nobody leaves while a peer may still write into its shared memory
    const int any_bad = __syncthreads_or(bad);
    if (!any_bad) {
        if (gater && p.h_out) { p.h_out[(size_t)gb * H + gj] = hC; p.h_out[(size_t)gb * H + CK + gj] = hF; }
        if (writer && lane == 0) {
            if (FUSED) {
                if (p.a_st_out) p.a_st_out[0] = (uint16_t)c_prev;
                if (p.b_st_out) p.b_st_out[0] = (uint16_t)f_prev;
            } else {
                if (p.c_st_out) p.c_st_out[gb] = (uint8_t)c_prev;
                if (p.f_st_out) p.f_st_out[gb] = (uint8_t)f_prev;
            }
        }
    }
    if (DBG && p.prof && blockIdx.x == 0 && tid < 16) p.prof[tid] = s_prof[tid];
    if (CHK && tid < CL_GUARDS && !cl_guard_ok(guard(tid))) cl_record(p.status, tid);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 1) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
    cluster_sync_all();
}

// ---------------------------------------------------------------------------------------------
static const void *cl_kernel_of(int nr, int mode, int kind)
{
#define CL_K(R, K) (mode == 2 ? (const void *)resident_cluster_kernel<R, 2, K> : mode ? (const void *)resident_cluster_kernel<R, 1, K> : (const void *)resident_cluster_kernel<R, 0, K>)
    if (kind == CL_FUSED) return CL_K(1, CL_FUSED);
    if (kind == CL_F32) return nr == 1 ? CL_K(1, CL_F32) : CL_K(2, CL_F32);
    return nr == 1 ? CL_K(1, CL_BF16) : nr == 2 ? CL_K(3, CL_BF16) : CL_K(4, CL_BF16);
#undef CL_K
}


// Rows per cluster and clusters of a batch.  Clusters never wait for one another, so a batch of more rows than the resident
// clusters take at CMAXR rows each runs as several waves of clusters, evenly filled.
static void cl_geometry(const ResClPack &k, int batch, int clusters, int *nr, int *n_clusters)
{
    const int per = k.kind == CL_BF16 ? 4 : 2, most = k.max_clusters * per, waves = (batch + most - 1) / most;
    const int c = clusters > 0 && waves == 1 ? std::min(k.max_clusters, std::max(clusters, (batch + per - 1) / per)) : k.max_clusters;
    *nr = (batch + waves * c - 1) / (waves * c);
    *n_clusters = (batch + *nr - 1) / *nr;
}

int rescl_prepare(wrnn_model *m)
{
    const int H = m->H;
    if (m->sparse || H != 2 * CK) { m->err = "cluster-resident kernel: dense H = 896 only"; return WRNN_ERR_UNSUPPORTED; }
    ResClPack k;
    { const char *d = getenv("WRNN_DEBUG"); k.checked = d && d[0] == '1'; }
    k.kind = m->variant == 1 ? CL_FUSED : m->dtype == WRNN_F32 ? CL_F32 : CL_BF16;
    for (int nr : {1, 2, 4})
        for (int mode = 0; mode < (k.checked ? 3 : 2); ++mode) {
            const void *f = cl_kernel_of(nr, mode, k.kind);
            if (cudaFuncSetAttribute(f, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess || !allow_smem(f, m->device, mode == 2 ? cl_checked_smem(k.kind) : cl_launch_smem(k.kind))) {
                cudaGetLastError(); m->err = "cluster-resident kernel does not fit this device"; return WRNN_ERR_UNSUPPORTED;
            }
        }
    {
        cudaLaunchConfig_t cfg; cudaLaunchAttribute at[1];
        cl_fill_launch(1, cl_launch_smem(k.kind), &cfg, at, 0);
        if (cudaOccupancyMaxActiveClusters(&k.max_clusters, cl_kernel_of(k.kind == CL_BF16 ? 4 : 1, 0, k.kind), &cfg) != cudaSuccess || k.max_clusters < 1) {
            cudaGetLastError(); m->err = "cluster-resident kernel: no 16-CTA cluster of this size fits the device"; return WRNN_ERR_UNSUPPORTED;
        }
    }
    // fp16 weights, every matrix scaled by a power of two to at most 2^14: the eight bits of a bf16 weight are kept unless it is
    // below 2^-28 of the largest one, where at most 2^-39 of that is lost; fp32 weights as two parts (2^-23 of a weight)
    const bool w2 = k.kind == CL_F32;
    const int NP = w2 ? 2 : 1, NIN = cl_nin(k.kind), LR = cl_rows(k.kind);
    m->half = new ClHalf(m, NP);
    const HalfMatrix &R = m->half->R, *O = m->half->O;
    k.sc = m->half->sc;
    const size_t smem_bytes = cl_blob_smem(k.kind), cta_bytes = smem_bytes + CB_TMEM;
    std::vector<uint8_t> stream(w2 ? CCS * CB_STREAM : 0, 0);
    std::vector<uint8_t> blob(CCS * cta_bytes, 0);
    // part w of row i of a CTA's 168 rows of R: half * 84 + gate * 28 + unit
    auto r_row = [&](int rank, int w, int i) { return &R.part[w][r_row_at(rank, i)]; };
    parallel_for(CCS, [&](int rank) {
        uint8_t *base = blob.data() + (size_t)rank * cta_bytes;
        for (int h = 0; h < 2; ++h)
            for (int w = 0; w < NP; ++w) {
                for (int t = 0; t < 2; ++t)
                    pack_448(O[h].part[w], CU * rank + 16 * t, std::min(16, CU - 16 * t), reinterpret_cast<uint16_t *>(base + (h * NP + w) * CW_HID + (size_t)t * 28 * 512));
                pack_448(O[2 + h].part[w], LR * rank, LR, reinterpret_cast<uint16_t *>(base + NP * 2 * CW_HID + (h * NP + w) * CW_LOG));
            }
        if (!w2) pack_r2(R.part[0], rank, reinterpret_cast<uint16_t *>(base + 2 * CW_HID + 2 * CW_LOG));
        float *sm = reinterpret_cast<float *>(base + smem_bytes - cl_small(k.kind) * 4);
        for (int i = 0; i < 6 * CU; ++i) {
            const size_t row = (size_t)((i / CU) % 3) * H + (size_t)(i / (3 * CU)) * CK + CU * rank + i % CU;
            for (int c = 0; c < NIN; ++c) sm[i * NIN + c] = m->hI[row * NIN + c];
        }
        float *b = sm + 6 * CU * NIN;
        for (int r = 0; r < CU; ++r) { b[r] = m->hb1[CU * rank + r]; b[32 + r] = m->hb3[CU * rank + r]; }
        for (int r = 0; r < LR; ++r) { b[64 + r] = m->hb2[LR * rank + r]; b[64 + CL + r] = m->hb4[LR * rank + r]; }
        // tensor memory: lane quadrant q holds quarter q of the k-tiles of both halves of the state; columns as the kernel states them
        for (int i = 0; i < 16 * CRT; ++i) {
            const int tile = i >> 4, reg0 = (i >> 3) & 1;
            const uint16_t *src = r_row(rank, 0, i);
            for (int kt = 0; kt < 56; ++kt) {
                const int half_f = kt / 28, q = kt % 28 / 7, k7 = kt % 7;
                const int c0 = tile < 4 ? (half_f * 7 + k7) * 16 + 4 * tile : 2 * 7 * 16 + (half_f * 7 + k7) * 20 + 4 * (tile - 4);
                cl_pack_tmem_row(base + smem_bytes, q, c0, i & 7, reg0, src + 16 * kt);
            }
        }
        if (!w2) return;
        // streamed fragments of warp w8 = 4 j + q: pass 0 the low parts of tiles 0..3 (j = 0) or 4, 5; pass 1 tile 9 (both parts) and
        // tile 10 (high parts over low parts), or the low parts of tiles 6..8
        uint16_t *st = reinterpret_cast<uint16_t *>(stream.data() + (size_t)rank * CB_STREAM);
        for (int half_f = 0; half_f < 2; ++half_f)
            for (int w8 = 0; w8 < 8; ++w8)
                for (int v = 0; v < 14; ++v)
                    for (int f = 0; f < cl_nf(w8 >> 2, v); ++f) {
                        const int j = w8 >> 2, kt = 28 * half_f + 7 * (w8 & 3) + v % 7;
                        uint16_t *frag = st + ((size_t)half_f * CF_HALF + cl_fw(w8) + cl_fo(j, v) + f) * 256;
                        for (int r = 0; r < 16; ++r) {
                            int row, w = 1;
                            if (v < 7) row = 16 * (j ? 4 + f : f) + r;
                            else if (j) row = 16 * (6 + f) + r;
                            else if (f < 2) { row = 144 + r; w = f; }
                            else { row = 160 + (r & 7); w = r >> 3; }
                            frag_row(frag, r & 7, r >> 3, r_row(rank, w, row) + 16 * kt);
                        }
                    }
    });
    ResClPack *pk = new ResClPack(k);
    if (cudaMalloc((void **)&pk->d_blob, blob.size()) != cudaSuccess || cudaMemcpy(pk->d_blob, blob.data(), blob.size(), cudaMemcpyHostToDevice) != cudaSuccess ||
        (w2 && (cudaMalloc((void **)&pk->d_stream, stream.size()) != cudaSuccess || cudaMemcpy(pk->d_stream, stream.data(), stream.size(), cudaMemcpyHostToDevice) != cudaSuccess)) ||
        cudaMalloc((void **)&pk->d_prof, 16 * sizeof(long long)) != cudaSuccess || cudaMemset(pk->d_prof, 0, 16 * sizeof(long long)) != cudaSuccess) {
        cudaGetLastError();
        cudaFree(pk->d_blob); cudaFree(pk->d_stream); cudaFree(pk->d_prof);
        delete pk;
        m->err = "device allocation for the cluster-resident kernel failed";
        return WRNN_ERR_NOMEM;
    }
    m->rescl = pk;
    return WRNN_OK;
}

void rescl_packed(wrnn_model *m)
{
    delete m->half;
    m->half = nullptr;
}

void rescl_destroy(wrnn_model *m)
{
    rescl_packed(m);
    if (!m->rescl) return;
    cudaFree(m->rescl->d_blob); cudaFree(m->rescl->d_stream); cudaFree(m->rescl->d_prof);
    delete m->rescl;
    m->rescl = nullptr;
}

int rescl_supported(const wrnn_model *m, int batch)
{
    return m->rescl && batch >= 1 && batch <= m->max_batch ? WRNN_OK : WRNN_ERR_UNSUPPORTED;
}

int rescl_launch_info(const wrnn_model *m, int batch, int *n_ctas, int *n_threads, int *smem, int64_t *weight_bytes)
{
    int nr, n_clusters;
    cl_geometry(*m->rescl, batch, 0, &nr, &n_clusters);
    if (n_ctas) *n_ctas = n_clusters * CCS;
    if (n_threads) *n_threads = 512;
    if (smem) *smem = (int)(m->rescl->checked ? cl_checked_smem(m->rescl->kind) : cl_launch_smem(m->rescl->kind));
    if (weight_bytes) *weight_bytes = (int64_t)CCS * (int64_t)(cl_blob_smem(m->rescl->kind) + CB_TMEM + (m->rescl->kind == CL_F32 ? CB_STREAM : 0));
    return WRNN_OK;
}

int rescl_clusters(const wrnn_model *m, int batch, int clusters)
{
    int nr, n_clusters;
    cl_geometry(*m->rescl, batch, clusters, &nr, &n_clusters);
    return std::min(n_clusters, m->rescl->max_clusters);
}

int rescl_run(wrnn_model *m, const StepArgs &a, cudaStream_t s)
{
    const ResClPack &k = *m->rescl;
    ClParams p;
    int nr, n_clusters;
    cl_geometry(k, a.batch, a.clusters, &nr, &n_clusters);
    cl_fill_params(m, a, k.sc, &p);
    p.nr = nr; p.blob = k.d_blob; p.stream = k.d_stream;
    p.prof = m->prof_enabled ? k.d_prof : nullptr;
    if (k.checked) { const char *poke = getenv("WRNN_DEBUG_POKE"); p.poke = poke && poke[0] == '1'; }
    const bool dbg = cl_wants_dumps(m, p);
    cudaLaunchConfig_t cfg; cudaLaunchAttribute at[2];
    p.smem_bytes = (unsigned)(k.checked ? cl_checked_smem(k.kind) : cl_launch_smem(k.kind));
    // (a lone cluster: several that start while blocks of the projection still run end up on other SMs, and 16 rows take 4.21 instead of 4.15 us per step)
    cl_fill_launch(n_clusters, p.smem_bytes, &cfg, at, s, !a.g && n_clusters == 1);
    void *args[] = {&p};
    const cudaError_t e = cudaLaunchKernelExC(&cfg, cl_kernel_of(nr, k.checked ? 2 : dbg, k.kind), args);
    if (e != cudaSuccess) {
        m->err = std::string("cluster-resident kernel launch failed: ") + cudaGetErrorString(e);
        cudaGetLastError();
        return WRNN_ERR_CUDA;
    }
    ++g_launches;
    m->prof_cl = 1;
    return WRNN_OK;
}

int rescl_phase_cycles(const wrnn_model *m, long long *out16)
{
    return m->rescl && cudaMemcpy(out16, m->rescl->d_prof, 16 * sizeof(long long), cudaMemcpyDeviceToHost) == cudaSuccess ? WRNN_OK : WRNN_ERR_CUDA;
}

}  // namespace wrnn
