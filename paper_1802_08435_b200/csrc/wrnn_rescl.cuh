// What the two kernels that keep a whole dense H = 896 model in one 16-CTA cluster share (wrnn_rescl.cu: up to four rows per cluster;
// wrnn_resrows.cu: five to fourteen): sizes, parameters, fragment layout of the weights, launch, and the plain fp32 steps for states
// that the operand images do not hold.
#pragma once
#include <cuda_fp16.h>

#include <cmath>
#include <cstdlib>
#include <cstring>
#include <type_traits>

#include "wrnn_cl.cuh"
#include "wrnn_cluster.cuh"
#include "wrnn_half.h"
#include "wrnn_internal.h"
#include "wrnn_tc.cuh"

namespace wrnn {

// What the power-of-two scaled operands are divided by again: 2^-14 over the power of two in R, in the hidden layers and logits rows; the
// one of the hidden-layer values ([0] coarse half)
struct ClScales {
    float inv_R = 0.f, inv_O1[2] = {0.f, 0.f}, inv_O2[2] = {0.f, 0.f}, q_scale[2] = {0.f, 0.f};
    ClScales() = default;
    // R, then O1, O3, O2, O4
    ClScales(const wrnn_model *m, const HalfMatrix &R, const HalfMatrix *O)
    {
        // products of operands scaled by 2^(14 - exponent) each
        inv_R = std::ldexp(1.f, R.exp - 28);
        for (int h = 0; h < 2; ++h) {
            const int eq = hidden_exp(h ? m->hO3 : m->hO1, h ? m->hb3 : m->hb1);
            inv_O1[h] = std::ldexp(1.f, O[h].exp - 28);
            q_scale[h] = std::ldexp(1.f, 14 - eq);
            inv_O2[h] = std::ldexp(1.f, O[2 + h].exp - 14 + eq - 14);
        }
    }
};
// A model's matrices as fp16 parts, for the packers of both kernels while it is created
struct ClHalf {
    HalfMatrix R, O[4];                      // O1, O3, O2, O4
    ClScales sc;
    ClHalf(const wrnn_model *m, int np) : R(m->hR, np), O{{m->hO1, np}, {m->hO3, np}, {m->hO2, np}, {m->hO4, np}}, sc(m, R, O) {}
};

namespace {
constexpr int CK = 448;                  // H / 2
constexpr int CU = 28;                   // state units of one half, hidden-layer rows per CTA
constexpr int CL = 16;                   // logits rows per CTA
constexpr int CCS = 16;                  // CTAs per cluster
constexpr int CK8 = CK / 8, CQ = CK / 4; // groups of eight and of four values of a half
constexpr int CRT = 9, CRS = 6 * CU - 16 * CRT;             // of the 168 rows of R: tiles of 16 in tensor memory, the 24 rows left in shared memory
constexpr int CPR = 6 * CU;              // rows of R of a CTA
constexpr size_t CW_R2 = 2 * CK8 * CRS * 16;                 // 24 rows of R as core matrices [k / 8][3][8][16 B]
constexpr int CTC = 2 * 7 * CRT * 4;                         // columns of tensor memory: nine tiles of R as A fragments, four registers each
constexpr size_t CB_TMEM = (size_t)CTC * 128 * 4;
enum { CL_BF16 = 0, CL_F32 = 1, CL_FUSED = 2 };                // kinds of model: bf16 weights, fp32 weights, the Fused Subscale WaveRNN 2x (bf16)
__host__ __device__ constexpr int cl_nin(int kind) { return kind == CL_FUSED ? 12 : 3; }
__host__ __device__ constexpr int cl_rows(int kind) { return kind == CL_FUSED ? 4 : CL; }       // logits rows per CTA in use

struct ClParams {
    int batch, nr;              // rows of the call, rows per cluster
    long long n_steps, step0;
    unsigned stream0;
    unsigned long long seed;
    int n_frames, hop, row_stride, row_offset_mul, row_lag;
    long long out_pitch;
    const uint8_t *blob;
    const uint4 *stream;
    const float *g;                          // [batch][n_frames][3H]
    ClScales sc;
    const float *h_in; float *h_out;
    const uint8_t *c_in, *f_in; uint8_t *c_st_out, *f_st_out;
    const uint8_t *c_forced, *f_forced;
    uint8_t *c_out, *f_out;
    // the fused variant's 16-bit counterparts of the byte arrays (part A = the coarse half, part B = the fine half)
    const uint16_t *a_in, *b_in; uint16_t *a_st_out, *b_st_out;
    const uint16_t *a_forced, *b_forced; uint16_t *a_out, *b_out;
    int16_t *out;
    float *dbg_gates, *dbg_h, *dbg_logits;
    DevStatus *status;
    unsigned long long limit_ns;
    int skip_rank; long long skip_step;      // self-test: CTAs of this rank withhold the state they publish at this step (-1: none)
    long long *prof;
    int poke; unsigned smem_bytes;           // checked form: one deliberate write past the end of region 6, by CTA 3; shared memory of the launch
    // for cl_wide_steps: the model as the any-shape kernel has it, and its scratch rows
    const void *wR, *wO[4];                  // R; O1, O3, O2, O4: 4 x 4 blocks, row by row
    const float *wI, *wb[4];                 // I; b1, b3, b2, b4
    float *q, *logits;                       // [batch][H / 2], [batch][256]
};
__device__ __forceinline__ void cl_ldmatrix4(uint32_t addr, uint32_t (&r)[4])
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];" : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void cl_st_async16(unsigned addr, uint4 v, unsigned mbar)
{
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1, %2, %3, %4}, [%5];" ::"r"(addr), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w), "r"(mbar) : "memory");
}
// f(0), .., f(N - 1) with compile-time arguments
template <int N, int I = 0, typename F>
__device__ __forceinline__ void cl_for(F &&f)
{
    if constexpr (I < N) { f(std::integral_constant<int, I>{}); cl_for<N, I + 1>(f); }
}
__device__ __forceinline__ void cl_st_async4(unsigned addr, uint32_t v, unsigned mbar)
{
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.b32 [%0], %1, [%2];" ::"r"(addr), "r"(v), "r"(mbar) : "memory");
}
__device__ __forceinline__ void cl_tmem_ld8(uint32_t c, uint32_t (&r)[8])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];" : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]) : "r"(c));
}
// before anything that the projection of this call writes (g, the status word) is used
__device__ __forceinline__ void cl_await_projection() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// The weights of a CTA, once per launch: 390 KB, bound by the loads in flight.  Shared memory: bulk copies (one thread), which the caller awaits
// on `bar`; a CTA has them in flight while its warps fill tensor memory.  (One row, 120 steps: 2 us less per call than with a 16-byte piece per
// thread and round trip, 418 -> 416 us; a fresh fp32 model's 1,200 steps 6.13 -> 6.00 ms.)
__device__ __forceinline__ void cl_load_bulk(uint32_t dst, const uint8_t *src, uint32_t bytes, uint32_t bar)
{
    constexpr uint32_t PIECE = 16384;
    mbar_arrive_expect(bar, bytes);
    for (uint32_t o = 0; o < bytes; o += PIECE)
        asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst + o), "l"(src + o), "r"(min(PIECE, bytes - o)), "r"(bar) : "memory");
}
// what the threads of this CTA wrote to shared memory, to the bulk copies that start after the next barrier
__device__ __forceinline__ void fence_proxy_async_cta() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
// bulk copy into a CTA of the cluster, counted on a barrier there
__device__ __forceinline__ void cl_copy_bulk(uint32_t dst, uint32_t src, uint32_t bytes, uint32_t bar)
{
    asm volatile("cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst), "r"(src), "r"(bytes), "r"(bar) : "memory");
}
// Tensor memory: [4 lane quadrants][126 groups of four columns][32 lanes][16 B], a quadrant per warp modulo four, eight groups in flight per lane
__device__ __forceinline__ void cl_load_tmem(uint32_t tmem, const uint8_t *src, int warp, int lane)
{
    constexpr int NGRP = CTC / 4;
    const uint4 *s = reinterpret_cast<const uint4 *>(src) + (size_t)(warp & 3) * NGRP * 32 + lane;
    const uint32_t dst = tmem + ((uint32_t)(32 * (warp & 3)) << 16);
#pragma unroll 1
    for (int c = 8 * (warp >> 2); c < NGRP; c += 32) {
        uint4 v[8];
#pragma unroll
        for (int k = 0; k < 8; ++k)
            if (c + k < NGRP) v[k] = __ldg(s + (size_t)(c + k) * 32);
#pragma unroll
        for (int k = 0; k < 8; ++k)
            if (c + k < NGRP)
                asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1,%2,%3,%4};" ::"r"(dst + 4 * (c + k)), "r"(v[k].x), "r"(v[k].y), "r"(v[k].z), "r"(v[k].w) : "memory");
    }
    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ uint4 cl_ldg_stream(const uint4 *p)
{
    uint4 v;
    asm volatile("ld.global.nc.L1::no_allocate.v4.b32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
    return v;
}
// Steps of a cluster whose rows were given a state beyond what the operand images hold (CL_WIDE): plain fp32, one row of a matrix per
// warp, everything exchanged through global memory, until no state is that large any more (a unit that changes is below one from then
// on; what is not finite stays here).  Rare, so nothing of it is fast.  Returns the number of steps taken; sym [2][16] carries the
// last symbols of the rows.  The state is in p.h_out throughout.
constexpr float CL_WIDE = 2.f, CL_STATE = 16384.f;            // CL_STATE: what the state is multiplied by in the images (fp16 ends at 65504)
template <int KIND>
__device__ __noinline__ long long cl_wide_steps(const ClParams &p, int row0, int nrc, int rank, float *A, int (*sym)[16])
{
    constexpr bool FUSED = KIND == CL_FUSED;
    constexpr int H = 2 * CK, NIN = cl_nin(KIND), NX = NIN / 3, LR = cl_rows(KIND), NL = CCS * LR;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    // row `row` of a matrix of `cols` columns times x, on every lane
    auto dot = [&](const void *M, int row, int cols, const float *x) {
        float acc = 0.f;
        for (int c = lane; c < cols / 4; c += 32) {
            const size_t at = ((size_t)(row >> 2) * (cols / 4) + c) * 16 + 4 * (row & 3);
            const float4 v = make_float4(__ldcg(x + 4 * c), __ldcg(x + 4 * c + 1), __ldcg(x + 4 * c + 2), __ldcg(x + 4 * c + 3));       // (a caller's state: floats at any address)
            float4 w;
            if (KIND == CL_F32) w = __ldg(reinterpret_cast<const float4 *>(static_cast<const float *>(M) + at));
            else {
                const uint2 b = __ldg(reinterpret_cast<const uint2 *>(static_cast<const uint16_t *>(M) + at));
                w = make_float4(bf16lo(b.x), bf16hi(b.x), bf16lo(b.y), bf16hi(b.y));
            }
            acc = fmaf(w.x, v.x, fmaf(w.y, v.y, fmaf(w.z, v.z, fmaf(w.w, v.w, acc))));
        }
        return warp_sum(acc);
    };
    auto x_of = [](int v, int k) { return FUSED ? scale4((v >> (12 - 4 * k)) & 15) : scale8(v); };
    // gates of one half: half 1 with the symbol of this step in sym[0], the last ones in `last`
    auto gates = [&](int half_g, long long s, const int (*last)[16]) {
        for (int i = tid; i < nrc * CU; i += 512) {
            const int st = i / CU, u = i - st * CU, j = half_g * CK + CU * rank + u, gb = row0 + st;
            const long long pos = (p.step0 + s) * p.row_stride + ((long long)p.stream0 + gb) * p.row_offset_mul;
            const float *g = p.g + ((size_t)gb * p.n_frames + (size_t)(p.row_lag > 0 ? s : pos / p.hop)) * 3 * H + j;
            float pre[3];
            for (int gate = 0; gate < 3; ++gate) {
                const float *I = p.wI + ((size_t)gate * H + j) * NIN;
                float v = g[gate * H];
                for (int k = 0; k < NX; ++k) {
                    v = fmaf(I[k], x_of(last[0][st], k), fmaf(I[NX + k], x_of(last[1][st], k), v));
                    if (half_g) v = fmaf(I[2 * NX + k], x_of(sym[0][st], k), v);
                }
                pre[gate] = v;
            }
            const float *a = A + st * CPR + half_g * 3 * CU + u;
            const float uu = sigmoidf_acc(pre[0] + a[0]), r = sigmoidf_acc(pre[1] + a[CU]), e = tanhf(fmaf(r, a[2 * CU], pre[2]));
            float *h = p.h_out + (size_t)gb * H + j;
            const float hn = fmaf(uu, __ldcg(h), (1.0f - uu) * e);
            __stcg(h, hn);
            if (p.dbg_gates) { float *o = p.dbg_gates + ((size_t)s * p.batch + gb) * 3 * H; o[j] = uu; o[H + j] = r; o[2 * H + j] = e; }
            if (p.dbg_h) p.dbg_h[((size_t)s * p.batch + gb) * H + j] = hn;
        }
        cluster_sync_all();
    };
    // head of one half (0: coarse): hidden layer, logits, the draw of row `warp`, the same in every CTA; the symbol fed back
    auto head = [&](int hd, long long s) {
        for (int i = warp; i < nrc * CU; i += 16) {
            const int gb = row0 + i / CU, row = CU * rank + i % CU;
            const float v = dot(p.wO[hd], row, CK, p.h_out + (size_t)gb * H + hd * CK);
            if (lane == 0) __stcg(p.q + (size_t)gb * CK + row, fmaxf(v + p.wb[hd][row], 0.f));
        }
        cluster_sync_all();
        for (int i = warp; i < nrc * LR; i += 16) {
            const int gb = row0 + i / LR, row = LR * rank + i % LR;
            const float v = dot(p.wO[2 + hd], row, CK, p.q + (size_t)gb * CK);
            if (lane == 0) __stcg(p.logits + (size_t)gb * 256 + row, v + p.wb[2 + hd][row]);
        }
        cluster_sync_all();
        if (warp < nrc) {
            const int gb = row0 + warp;
            const unsigned long long t = (unsigned long long)(p.step0 - (long long)gb * p.row_lag + s);
            const float *L = p.logits + (size_t)gb * 256;
            constexpr int PER = NL / 32;
            float l[8];
            for (int k = 0; k < PER; ++k) l[k] = __ldcg(L + PER * lane + k);
            int drawn;
            if (FUSED) {
                const int nib = group16_softmax_draw(l[0], l[1], uniform24(p.seed, p.stream0 + (unsigned)gb, t, 4 * hd + (lane >> 3)), lane);
                drawn = (__shfl_sync(FULL, nib, 0) << 12) | (__shfl_sync(FULL, nib, 8) << 8) | (__shfl_sync(FULL, nib, 16) << 4) | __shfl_sync(FULL, nib, 24);
            } else drawn = warp_softmax_draw(l, uniform24(p.seed, p.stream0 + (unsigned)gb, t, hd), lane);
            int fed = drawn;
            if (FUSED) { const uint16_t *fz = hd ? p.b_forced : p.a_forced; if (fz) fed = fz[s]; }
            else { const uint8_t *fz = hd ? p.f_forced : p.c_forced; if (fz) fed = fz[(size_t)gb * p.n_steps + s]; }
            if (rank == warp) {
                if (p.dbg_logits)
                    for (int k = 0; k < PER; ++k) p.dbg_logits[(((size_t)s * p.batch + gb) * 2 + hd) * NL + PER * lane + k] = l[k];
                if (lane == 0) {
                    if (FUSED) {
                        uint16_t *o = hd ? p.b_out : p.a_out;
                        if (o) o[s] = (uint16_t)drawn;
                        if (p.out) p.out[hd ? p.n_steps + s : s] = (int16_t)(fed - 32768);
                    } else {
                        uint8_t *o = hd ? p.f_out : p.c_out;
                        if (o) o[(size_t)gb * p.n_steps + s] = (uint8_t)drawn;
                        if (hd && p.out) p.out[(long long)gb * p.out_pitch + s] = (int16_t)(256 * sym[0][warp] + fed - 32768);
                    }
                }
            }
            __syncwarp();
            if (lane == 0) sym[hd][warp] = fed;
        }
        __syncthreads();
    };
    long long s = 0;
    for (bool wide = true; wide && s < p.n_steps; ++s) {
        for (int i = warp; i < nrc * CPR; i += 16) {
            const int st = i / CPR, r = i - st * CPR;                        // as in the blob: half * 84 + gate * 28 + unit
            const float v = dot(p.wR, (r / CU) % 3 * H + r / (3 * CU) * CK + CU * rank + r % CU, H, p.h_out + (size_t)(row0 + st) * H);
            if (lane == 0) A[st * CPR + r] = v;
        }
        __shared__ int last[2][16];
        if (tid < 32) last[tid >> 4][tid & 15] = sym[tid >> 4][tid & 15];
        __syncthreads();
        cluster_sync_all();                                                  // everybody has read the old state
        gates(0, s, last);
        head(0, s);
        gates(1, s, last);
        head(1, s);
        int any = 0;
        for (int i = tid; i < nrc * H; i += 512) any |= fabsf(__ldcg(p.h_out + (size_t)row0 * H + i)) > CL_WIDE;
        wide = __syncthreads_or(any);
        cluster_sync_all();
    }
    return s;
}

// one row (g of a fragment's upper or lower eight) of the A fragment of a k-tile: lane (g, t) holds it at k 4t, 4t + 1 and at
// 4t + 2, 4t + 3 (the permuted k order), registers `lower` and 2 + `lower`
void frag_row(uint16_t *frag, int g, int lower, const uint16_t *src)
{
    for (int t = 0; t < 4; ++t) {
        uint16_t *d = frag + (4 * g + t) * 8 + 2 * lower;
        d[0] = src[4 * t]; d[1] = src[4 * t + 1]; d[4] = src[4 * t + 2]; d[5] = src[4 * t + 3];
    }
}
// fragments of rows first .. first + n_rows - 1 (up to 16) of a matrix of 448 columns
void pack_448(const std::vector<uint16_t> &M, int first, int n_rows, uint16_t *dst)
{
    for (int r = 0; r < n_rows; ++r)
        for (int kt = 0; kt < 28; ++kt) frag_row(dst + (size_t)kt * 256, r & 7, r >> 3, &M[(size_t)(first + r) * CK + 16 * kt]);
}
// where row i of a CTA's 168 rows of R starts in R: half * 84 + gate * 28 + unit
size_t r_row_at(int rank, int i) { return ((size_t)((i / CU) % 3) * 2 * CK + (size_t)(i / (3 * CU)) * CK + CU * rank + i % CU) * 2 * CK; }
// the 24 rows of R beyond the tiles in tensor memory, as core matrices in the permuted k order
void pack_r2(const std::vector<uint16_t> &R, int rank, uint16_t *r2)
{
    for (int i = 0; i < CRS; ++i)
        for (int k8 = 0; k8 < 2 * CK8; ++k8) {
            const uint16_t *src = &R[r_row_at(rank, 16 * CRT + i)] + 16 * (k8 >> 1) + 2 * (k8 & 1);
            for (int c = 0; c < 8; ++c) r2[((size_t)k8 * CRS + i) * 8 + c] = src[4 * (c >> 1) + (c & 1)];
        }
}
// row g (of the upper or lower eight) of a fragment whose four registers are columns c0 .. c0 + 3 (a multiple of four) of quadrant q
void cl_pack_tmem_row(uint8_t *tm, int q, int c0, int g, int lower, const uint16_t *src)
{
    frag_row(reinterpret_cast<uint16_t *>(tm) + ((size_t)q * (CTC / 4) + c0 / 4) * 256, g, lower, src);
}

// the parameters that a call and the model give
void cl_fill_params(wrnn_model *m, const StepArgs &a, const ClScales &sc, ClParams *q)
{
    ClParams &p = *q;
    p = ClParams();
    p.batch = a.batch;
    p.n_steps = a.n_steps; p.step0 = a.step0; p.stream0 = a.stream0; p.seed = a.seed;
    p.n_frames = m->cond_dim ? a.n_frames : 1;
    p.hop = m->cond_dim ? a.hop : 1;
    p.row_stride = m->cond_dim ? a.row_stride : 0;
    p.row_offset_mul = m->cond_dim ? a.row_offset_mul : 0;
    p.row_lag = a.row_lag; p.out_pitch = a.out_pitch ? a.out_pitch : a.n_steps;
    p.g = a.g ? a.g : m->g; p.sc = sc;
    p.h_in = a.h_in; p.h_out = a.h_out; p.c_in = a.c_in; p.f_in = a.f_in; p.c_st_out = a.c_st_out; p.f_st_out = a.f_st_out;
    p.c_forced = a.c_forced; p.f_forced = a.f_forced; p.c_out = a.c_out; p.f_out = a.f_out; p.out = a.out;
    p.a_in = a.a_in; p.b_in = a.b_in; p.a_st_out = a.a_st_out; p.b_st_out = a.b_st_out;
    p.a_forced = a.a_forced; p.b_forced = a.b_forced; p.a_out = a.a_out; p.b_out = a.b_out;
    p.dbg_gates = a.dbg_gates; p.dbg_h = a.dbg_h; p.dbg_logits = a.dbg_logits;
    p.status = m->status;
    p.limit_ns = m->wait_limit_ns();
    p.skip_rank = m->dbg_skip_cta >= 0 ? m->dbg_skip_cta % CCS : -1; p.skip_step = m->dbg_skip_step;
    p.wR = m->R.vals; p.wI = m->I; p.q = m->q; p.logits = m->logits;
    p.wO[0] = m->O1.vals; p.wO[1] = m->O3.vals; p.wO[2] = m->O2.vals; p.wO[3] = m->O4.vals;
    p.wb[0] = m->b1; p.wb[1] = m->b3; p.wb[2] = m->b2; p.wb[3] = m->b4;
}
// whether a call wants more than samples and the final state: forced symbols, dumps, stamps or a withheld word
bool cl_wants_dumps(const wrnn_model *m, const ClParams &p)
{
    return m->dbg_skip_cta >= 0 || p.prof || p.c_forced || p.f_forced || p.c_out || p.f_out || p.a_forced || p.b_forced || p.a_out || p.b_out || p.dbg_gates ||
           p.dbg_h || p.dbg_logits;
}
// `early`: behind the projection of this call, which it may overlap (at: two attributes)
void cl_fill_launch(int n_clusters, size_t smem, cudaLaunchConfig_t *cfg, cudaLaunchAttribute *at, cudaStream_t s, bool early = false)
{
    std::memset(cfg, 0, sizeof(*cfg));
    cfg->gridDim = dim3(n_clusters * CCS);
    cfg->blockDim = dim3(512);
    cfg->dynamicSmemBytes = smem;
    cfg->stream = s;
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = CCS; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
    if (early) { at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization; at[1].val.programmaticStreamSerializationAllowed = 1; }
    cfg->attrs = at;
    cfg->numAttrs = early ? 2 : 1;
}
}  // namespace

}  // namespace wrnn
