// The conditioning network of the Subscale WaveRNN (Sections 4.1 and 5.3 of the paper): a masked dilated 1-D CNN with
// relus through which the WaveRNN that generates sub-tensor s sees the FUTURE context of the sub-tensors z < s -- ten
// layers, kernels of size 3, 384 convolution channels, 768 residual channels, five stages of increasing dilation, a
// future horizon of 128 positions.  The paper prints no equations for it; the reading built here:
//     X[i][z]    = u_{B i + z} / 32768 for z < s, 0 otherwise                              (block input, masked to earlier rows)
//     x_0[i]     = W_in X[i] + b_in
//     a_l[i]     = relu(b_conv[l] + sum_{t = 0..taps-1} W_conv[l][t] x_l[i + t d_l])       (connections reach forward only)
//     x_{l+1}[i] = x_l[i] + W_res[l] a_l[i] + b_res[l]
//     v_s[i]     = frame_s[(B i + s) div hop] + W_out relu(x_last[i]) + b_out
// with the zero vector at positions at or beyond the row length in every layer, and bf16-rounded matrices.
//
// A chunk of positions is a chain of matrix products over (positions x channels), so it runs on the fifth-generation
// tensor cores: one CTA per tile of 128 positions x BN output channels; the activations (M side) enter as bf16 high and
// low parts of their fp32 values (two MMAs into the same TMEM accumulator, operand error 2^-17), the weights (N side)
// as bf16; operands come in by TMA (128-byte swizzle) through a ring of mbarriers, a dilated tap being nothing but a
// row offset of the activation box; one thread issues tcgen05.mma, four warps drain the accumulator with tcgen05.ld and
// apply bias / relu / residual.  The residual stream is kept in fp32 beside its bf16 parts.  Every mbarrier wait is bounded.
//
// Two ways through the layers.  A call for any positions of any rows computes, in every layer, all positions that the ones
// it wants depend on (124 beyond the last of them: 1.48 times the work at 128 positions).  A staggered generation from its first to its
// last position keeps the last positions of every layer in rings and computes 64 new ones of each per block: x_l at positions p + reach_l .. + 63
// (reach_l: how far the layers from l on look ahead), from two blocks before the row starts, so that no needed position is left out.
#include <cuda_bf16.h>

#include <algorithm>
#include <cstring>
#include <new>

#include "wrnn_cl.cuh"
#include "wrnn_cluster.cuh"
#include "wrnn_internal.h"
#include "wrnn_tc.cuh"

struct wrnn_subscale_net {
    int B = 0, n_layers = 0, taps = 0, conv_ch = 0, res_ch = 0, cond_dim = 0, reach = 0, device = 0;
    std::vector<int> dilation;
    __nv_bfloat16 *Wc = nullptr;      // [layers][taps][conv_ch][res_ch]
    __nv_bfloat16 *Wr = nullptr;      // [layers][res_ch][conv_ch]
    __nv_bfloat16 *Wo = nullptr;      // [64][res_ch] (rows >= cond_dim zero)
    float *W_in = nullptr /* [B][res_ch] */, *b_in = nullptr, *b_conv = nullptr, *b_res = nullptr, *b_out = nullptr;
    // activations of one call: n_seg row segments of n_alloc positions each
    int n_seg = 0, n_alloc = 0;
    float *xf = nullptr;                              // [n_seg * n_alloc][res_ch] fp32 residual stream
    __nv_bfloat16 *xh = nullptr, *xl = nullptr;       // its bf16 high / low parts (relu'd after the last layer)
    __nv_bfloat16 *ah = nullptr, *al = nullptr;       // [n_seg * n_alloc][conv_ch] convolution outputs
    CUtensorMap tmWc, tmWr, tmWo, tmXh, tmXl, tmAh, tmAl;
    // rings of a staggered generation: x_0 .. x_{n_layers} of every row, the last SN_RING positions (parts: with a copy of the first 64 behind
    // them, so that a box of 64 positions that starts anywhere is one run); convolution outputs of one block
    float *rf = nullptr;                              // [n_layers][B][SN_RING][res_ch]
    __nv_bfloat16 *rh = nullptr, *rl = nullptr;       // [n_layers + 1][B][SN_RING + 64][res_ch]
    __nv_bfloat16 *bh = nullptr, *bl = nullptr;       // [B][64][conv_ch]
    CUtensorMap tmRh, tmRl, tmBh, tmBl;
    cudaStream_t side[2] = {nullptr, nullptr};        // the network's, the stepping calls' while they overlap
    cudaEvent_t ev[5] = {};                           // network of an even, odd block done; stepping of one; fork
    wrnn::DevStatus *status = nullptr;
    std::string err;
};

namespace wrnn {

constexpr int SN_BM = 128;           // positions per tile (the M side: one TMEM lane per position)
constexpr int SN_THREADS = 384;      // warp 0: TMA of the high parts, warp 1: MMA issuer, warps 2, 3: TMA of the low parts, of the weights, warps 4..11: epilogue
enum { SN_CONV = 0, SN_RES = 1, SN_OUT = 2 };
constexpr int SN_RING = 128;         // positions of a ring: a block of 64 and, at most, the 2 x 32 before it that a tap reaches back to

struct SubnetGemmParams {
    int n_kb_tap;                    // 64-wide k-blocks per tap
    int taps, dil;                   // taps of this product and their distance in positions (1 tap for RES / OUT)
    int w_row0, w_tap_rows;          // first row of this layer in the weight tensor, rows between taps
    int n_alloc;                     // positions per row segment of the activation tensors
    int n_pos;                       // positions of a segment this product must write ([0, n_pos))
    int C_out;                       // channels of the output tensor (row pitch)
    const float *bias;               // [C_out] of this layer
    // positions: segment b holds row r_lo + b from position p_lo - b * lag on; positions >= L hold zeros
    int r_lo; long long p_lo; int lag; long long L;
    float *xf; __nv_bfloat16 *oh, *ol;      // RES: fp32 stream (in/out) and its parts; CONV: oh / ol = convolution outputs
    int relu_parts;                          // RES: the parts hold relu(x) (after the last layer: operand of the output product)
    // OUT
    float *v; int n_steps, cond_dim; const float *frames; int n_frames, hop, Bsub;
    const float *b_out;
    // rings: rows r_lo .. r_lo + n_seg - 1, row r at position t0 - r * lag; the product writes positions + reach .. + reach + 63
    int n_seg, reach, a_idx0, a_slot0;       // first row of the activation operand in its array, its slot
    long long t0;
    float *xf_out;
    DevStatus *status;
    unsigned long long limit_ns;
};

// shared memory by its own addresses: through pointers of no known space every store to it would order the global loads around it
__device__ __forceinline__ float4 sn_lds(uint32_t a) { float4 v; asm volatile("ld.shared.v4.f32 {%0,%1,%2,%3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(a)); return v; }
__device__ __forceinline__ float sn_lds1(uint32_t a) { float v; asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(a)); return v; }
__device__ __forceinline__ void sn_sts(uint32_t a, float4 v) { asm volatile("st.shared.v4.f32 [%0], {%1,%2,%3,%4};" ::"r"(a), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w)); }
__device__ __forceinline__ void sn_sts(uint32_t a, uint4 v) { asm volatile("st.shared.v4.b32 [%0], {%1,%2,%3,%4};" ::"r"(a), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w)); }
template <int N>
__device__ __forceinline__ void sn_copy_async(uint32_t dst, const void *src)
{
    if (N == 16) asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src));
    else asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst), "l"(src));
}

template <int N>
__device__ __forceinline__ void sn_tmem_ld(uint32_t a, float (&r)[N])
{
    if constexpr (N == 32) tmem_ld32(a, r);
    else if constexpr (N == 8) tmem_ld8(a, r);
    else tmem_ld16(a, reinterpret_cast<uint32_t (&)[16]>(r));
}

// RING: a tile of 128 is 64 positions of each of two rows.  NS (convolution): a cluster of NS CTAs shares a tile, each with 1 / NS of the k-blocks
// -- of which it has 36 one after the other, each 715 cycles of shared-memory traffic (44 KB in, 56 KB out to the MMAs) -- and adds up 1 / NS of the
// channels.
template <int BN, int MODE, int STAGES, bool RING, int NS = 1>
__global__ void __launch_bounds__(SN_THREADS, 1) subnet_gemm_kernel(const __grid_constant__ CUtensorMap tmAh, const __grid_constant__ CUtensorMap tmAl,
                                                                    const __grid_constant__ CUtensorMap tmW, const SubnetGemmParams p)
{
    extern __shared__ uint8_t smem_raw[];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int me = (int)blockIdx.x % NS, nt = (int)blockIdx.x / NS, mt = blockIdx.y, seg = blockIdx.z;       // (me: rank in the cluster)
    static_assert(NS == 1 || (MODE == SN_CONV && RING && NS <= 3), "only these");
    constexpr int CT = BN / NS, XS = CT * 4 + 16;               // channels that a CTA finishes; bytes of a row of sums that it is sent
    constexpr uint32_t A_BYTES = SN_BM * TC_BK * 2, W_BYTES = BN * TC_BK * 2, STAGE_BYTES = 2 * A_BYTES + W_BYTES;
    constexpr int TMEM_COLS = BN <= 64 ? 64 : BN <= 128 ? 128 : 256;
    __shared__ __align__(8) uint64_t full[STAGES], empty[STAGES], done, part;
    __shared__ uint32_t tmem_slot;
    __shared__ __align__(16) float s_bias[BN];
    uint8_t *ring = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    const uint32_t ring0 = smem_u32(ring);

    if (tid == 0) {
        for (int i = 0; i < STAGES; ++i) { mbar_init(smem_u32(&full[i]), 3); mbar_init(smem_u32(&empty[i]), 1); }
        mbar_init(smem_u32(&done), 1);
        if (NS > 1) { mbar_init(smem_u32(&part), 1); mbar_expect_tx(smem_u32(&part), (NS - 1) * SN_BM * CT * 4); }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)), "r"(TMEM_COLS) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    for (int i = tid; i < BN; i += SN_THREADS) s_bias[i] = MODE != SN_OUT ? __ldg(p.bias + nt * BN + i) : i < p.cond_dim ? __ldg(p.b_out + i) : 0.f;
    tc_fence_before();
    if (NS > 1) cluster_sync_all();                              // every peer's barrier is initialised before anyone sends
    else __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_slot;
    if (tid < 3) tma_prefetch_map(tid == 0 ? &tmAh : tid == 1 ? &tmAl : &tmW);
    // Programmatic dependent launch: the next product of the chain may be scheduled when this one's MMAs are issued (its CTAs set up their barriers
    // and TMEM on SMs that this grid has left or never used, and load their first weights); nothing of the previous product is read before
    // it has completed.  (Not earlier: a waiting CTA takes an SM, and a chain that may run ahead fills the chip with them, which keeps the
    // clusters of a stepping call from starting.)
    if (warp != 3) asm volatile("griddepcontrol.wait;" ::: "memory");

    const int nkb = p.taps * p.n_kb_tap / NS;
    const int arow0 = seg * p.n_alloc + mt * SN_BM;          // first activation row (position) of this tile
    bool ok = true;
    if ((warp == 0 || warp == 2 || warp == 3) && lane == 0) {
        // one producer per operand: a tiled load occupies its issuing thread for some 230 cycles, and with all three in one
        // thread a k-block took 1,200 cycles whatever the rows (a convolution launch 22 us from one row to sixteen)
        const int op = warp == 0 ? 0 : warp - 1;                // high parts, low parts, weights
        const CUtensorMap *tm = op == 0 ? &tmAh : op == 1 ? &tmAl : &tmW;
        const uint32_t off = op * A_BYTES, bytes = op < 2 ? A_BYTES : W_BYTES;
        const int ystep = op < 2 ? p.dil : p.w_tap_rows, tap0 = me * nkb / p.n_kb_tap;
        int st = 0, ph = 1, kc = (me * nkb - tap0 * p.n_kb_tap) * TC_BK, y = (op < 2 ? (RING ? p.a_slot0 : arow0) : p.w_row0 + nt * BN) + tap0 * ystep;
        if (RING && op < 2) y &= SN_RING - 1;
        for (int kb = 0; kb < nkb; ++kb) {
            if (!mbar_wait(smem_u32(&empty[st]), ph, p.limit_ns)) { ok = false; break; }
            const uint32_t fb = smem_u32(&full[st]);
            mbar_expect_tx(fb, bytes);
            if (RING && op < 2) tma_load_3d(ring0 + st * STAGE_BYTES + off, tm, fb, kc, y, p.a_idx0 + 2 * mt);
            else tma_load_2d(ring0 + st * STAGE_BYTES + off, tm, fb, kc, y);
            kc += TC_BK;
            if (kc == p.n_kb_tap * TC_BK) {
                kc = 0; y += ystep;
                if (RING && op < 2) y &= SN_RING - 1;
            }
            if (++st == STAGES) { st = 0; ph ^= 1; }
        }
    } else if (warp == 1 && lane == 0) {
        const uint32_t idesc = umma_idesc_bf16(SN_BM, BN);
        for (int kb = 0; kb < nkb; ++kb) {
            const int st = kb % STAGES, ph = (kb / STAGES) & 1;
            if (!mbar_wait(smem_u32(&full[st]), ph, p.limit_ns)) { ok = false; break; }
            tc_fence_after();
            const uint32_t base = ring0 + st * STAGE_BYTES;
            // (eight MMAs in one sequence; with a descriptor built for each, an MMA took 87 cycles whatever its width)
            umma_bf16_kblock_parts(tmem, umma_desc_lo(base), umma_desc_lo(base + A_BYTES), umma_desc_lo(base + 2 * A_BYTES), idesc, kb ? 1u : 0u);
            umma_commit(smem_u32(&empty[st]));
        }
        if (ok) umma_commit(smem_u32(&done));
        asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    } else if (warp >= 4) {
        // A lane drains a position (a lane of TMEM), but a position's channels are what is contiguous in memory: values go through a slab of shared
        // memory per warp (rows padded by 16 bytes), so that a warp reads and writes whole lines.  The residual stream is in its slab
        // before the product is done; the others use the stages, which are free then.  (A residual product's epilogue with a lane per
        // position took 20,000 cycles, three times its MMAs.)
        const int q = warp & 3, cg = (warp >> 2) - 1;           // TMEM lane quadrant this warp may read; which half of the channels it does
        const int sg = RING ? 2 * mt + q / 2 : seg, j0 = RING ? 32 * (q & 1) : mt * SN_BM + 32 * q;         // its rows are positions j0 .. j0 + 31
        const long long pos0 = (RING ? p.t0 - (long long)(p.r_lo + sg) * p.lag + p.reach : p.p_lo - (long long)seg * p.lag) + j0;
        // rows that a valid output may read; at or beyond the row length every layer holds zeros
        const int n_live = RING ? (sg < p.n_seg ? 32 : 0) : max(0, min(32, p.n_pos - j0));
        const bool inside = pos0 + lane < p.L;
        // where row i's values lie: as fp32, as parts (with a copy behind the ring), from its array's first row of this segment on
        const int r = p.r_lo + sg, s0 = (int)(pos0 & (SN_RING - 1));
        auto slot = [&](int i) { return (s0 + i) & (SN_RING - 1); };
        auto frow = [&](int i) { return RING ? slot(i) : i; };
        auto prow = [&](int i) { return RING && MODE == SN_RES ? slot(i) : i; };
        constexpr int CH = CT / 2, CC = CH % 32 == 0 ? 32 : CH % 16 == 0 ? 16 : 8;                  // channels that this warp finishes, in chunks of so many
        const size_t fbase = (RING ? (size_t)r * SN_RING : (size_t)seg * p.n_alloc + j0) * p.C_out + nt * BN + CT * me + CH * cg;
        const size_t pbase = (!RING ? (size_t)seg * p.n_alloc + j0 : MODE == SN_CONV ? (size_t)r * 64 + j0 : (size_t)r * (SN_RING + 64)) * p.C_out + nt * BN + CT * me + CH * cg;
        constexpr int FS = CH * 4 + 16, PS = CH * 2 + 16;       // bytes of a slab's row: fp32, a part
        // a pass of the warp over N 16-byte pieces per row: f(row, piece)
        auto pieces = [&](auto N_C, auto &&f) {
            constexpr int N = decltype(N_C)::value, ROWS = N % 3 ? 32 : 96 / N, IT = ROWS * N / 32;        // (so many rows in whole iterations)
            int row[IT], c[IT];
#pragma unroll
            for (int k = 0; k < IT; ++k) { row[k] = (lane + 32 * k) / N; c[k] = lane + 32 * k - row[k] * N; }
#pragma unroll 2
            for (int i = 0; i < 32; i += ROWS)
#pragma unroll
                for (int k = 0; k < IT; ++k)
                    if (i + row[k] < n_live) f(i + row[k], c[k]);
        };
        const uint32_t fslab = ring0 + STAGES * STAGE_BYTES + (4 * cg + q) * 32 * FS;                  // residual stream, frames
        const uint32_t hslab = ring0 + (4 * cg + q) * 64 * PS, lslab = hslab + 32 * PS;
        if (MODE == SN_RES)
            pieces(std::integral_constant<int, CH / 4>{}, [&](int i, int c) { sn_copy_async<16>(fslab + i * FS + 16 * c, p.xf + fbase + frow(i) * p.C_out + 4 * c); });
        // rows that are an output, their frames
        const long long first = RING ? -pos0 : 0, end = RING ? p.L - pos0 : p.n_steps - j0;
        auto wanted = [&](int i) { return i < n_live && i >= first && i < end; };
        if (MODE == SN_OUT) {
            const int mine = wanted(lane) ? (int)(((long long)p.Bsub * (pos0 + lane) + r) / p.hop) : 0;
#pragma unroll 8
            for (int i = 0; i < 32; ++i) {
                const float *f = p.frames + ((size_t)r * p.n_frames + __shfl_sync(FULL, mine, i)) * p.cond_dim;
                if (wanted(i)) {
                    if (lane + 32 * cg < p.cond_dim) sn_copy_async<4>(fslab + i * FS + 4 * lane, f + lane + 32 * cg);
                }
            }
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncwarp();
        if (mbar_wait(smem_u32(&done), 0, p.limit_ns)) {
            tc_fence_after();
            const uint32_t xslab = ring0 + STAGES * STAGE_BYTES + (32 * q + lane) * XS + 4 * CH * cg;   // this lane's row of the sums of the others (NS > 1)
#pragma unroll 1
            for (int k = 1; k < NS; ++k) {                                      // their share to each of the others: theirs of CTA (me + 1 + n) mod NS is in slot n
                const int to = (me + k) % NS;
                const uint32_t a = map_to_rank(xslab + (NS - 1 - k) * SN_BM * XS, (unsigned)to), b = map_to_rank(smem_u32(&part), (unsigned)to);
#pragma unroll
                for (int c0 = 0; c0 < CH; c0 += CC) {
                    float acc[CC];
                    sn_tmem_ld<CC>(tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(CT * to + CH * cg + c0), acc);
                    tmem_wait_ld();
#pragma unroll
                    for (int c = 0; c < CC; c += 4) st_async_v4(a + 4 * (c0 + c), acc[c], acc[c + 1], acc[c + 2], acc[c + 3], b);
                }
            }
            const bool here = NS == 1 || mbar_wait(smem_u32(&part), 0, p.limit_ns);
            ok = here;
#pragma unroll 1
            for (int c0 = 0; c0 < CH; c0 += CC) {
                float acc[CC];
                sn_tmem_ld<CC>(tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(CT * me + CH * cg + c0), acc);
                tmem_wait_ld();
                if (NS > 1 && here) {
                    // in the order of the CTAs, whoever adds
#pragma unroll
                    for (int c = 0; c < CC; c += 4) {
                        const float4 a = sn_lds(xslab + 4 * (c0 + c)), b = NS > 2 ? sn_lds(xslab + SN_BM * XS + 4 * (c0 + c)) : make_float4(0.f, 0.f, 0.f, 0.f);
                        auto sum = [&](float own, float n1, float n2) { return NS == 2 ? own + n1 : me == 0 ? (own + n1) + n2 : me == 1 ? (n2 + own) + n1 : (n1 + n2) + own; };
                        acc[c] = sum(acc[c], a.x, b.x); acc[c + 1] = sum(acc[c + 1], a.y, b.y); acc[c + 2] = sum(acc[c + 2], a.z, b.z); acc[c + 3] = sum(acc[c + 3], a.w, b.w);
                    }
                }
                const uint32_t f4 = fslab + lane * FS + 4 * c0;
                if (MODE == SN_OUT) {
#pragma unroll
                    for (int c = 0; c < CC; c += 4) {
                        float4 x = sn_lds(f4 + 4 * c);
                        const float4 b = *reinterpret_cast<const float4 *>(s_bias + CT * me + CH * cg + c0 + c);
                        x.x += acc[c] + b.x; x.y += acc[c + 1] + b.y; x.z += acc[c + 2] + b.z; x.w += acc[c + 3] + b.w;
                        sn_sts(f4 + 4 * c, x);
                    }
                    continue;
                }
#pragma unroll
                for (int c = 0; c < CC; c += 4) {
                    const float4 b = *reinterpret_cast<const float4 *>(s_bias + CT * me + CH * cg + c0 + c);
                    float4 x = {0.f, 0.f, 0.f, 0.f};
                    if (MODE == SN_RES) {
                        x = sn_lds(f4 + 4 * c);
                        x.x = inside ? x.x + (acc[c] + b.x) : 0.f; x.y = inside ? x.y + (acc[c + 1] + b.y) : 0.f;
                        x.z = inside ? x.z + (acc[c + 2] + b.z) : 0.f; x.w = inside ? x.w + (acc[c + 3] + b.w) : 0.f;
                        sn_sts(f4 + 4 * c, x);
                        if (p.relu_parts) x = make_float4(fmaxf(x.x, 0.f), fmaxf(x.y, 0.f), fmaxf(x.z, 0.f), fmaxf(x.w, 0.f));
                    } else if (inside) x = make_float4(fmaxf(acc[c] + b.x, 0.f), fmaxf(acc[c + 1] + b.y, 0.f), fmaxf(acc[c + 2] + b.z, 0.f), fmaxf(acc[c + 3] + b.w, 0.f));
                    acc[c] = x.x; acc[c + 1] = x.y; acc[c + 2] = x.z; acc[c + 3] = x.w;
                }
#pragma unroll
                for (int c = 0; c < CC; c += 8) {
                    uint32_t hi[4], lo[4];
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const float a = acc[c + 2 * k], b = acc[c + 2 * k + 1];
                        const __nv_bfloat16 h0 = __float2bfloat16_rn(a), h1 = __float2bfloat16_rn(b);
                        const __nv_bfloat16 l0 = __float2bfloat16_rn(a - __bfloat162float(h0)), l1 = __float2bfloat16_rn(b - __bfloat162float(h1));
                        hi[k] = (uint32_t)__bfloat16_as_ushort(h0) | ((uint32_t)__bfloat16_as_ushort(h1) << 16);
                        lo[k] = (uint32_t)__bfloat16_as_ushort(l0) | ((uint32_t)__bfloat16_as_ushort(l1) << 16);
                    }
                    sn_sts(hslab + lane * PS + 2 * (c0 + c), make_uint4(hi[0], hi[1], hi[2], hi[3]));
                    sn_sts(lslab + lane * PS + 2 * (c0 + c), make_uint4(lo[0], lo[1], lo[2], lo[3]));
                }
            }
            __syncwarp();
            if (MODE == SN_OUT) {
                float *v = p.v + ((size_t)(RING ? r : seg) * p.n_steps + j0) * p.cond_dim;
#pragma unroll 8
                for (int i = 0; i < 32; ++i)
                    if (wanted(i)) {
                        if (lane + 32 * cg < p.cond_dim) v[i * p.cond_dim + lane + 32 * cg] = sn_lds1(fslab + i * FS + 4 * lane);
                    }
            } else {
                if (MODE == SN_RES && (!RING || !p.relu_parts))                 // (nobody reads the last layer's ring as fp32)
                    pieces(std::integral_constant<int, CH / 4>{}, [&](int i, int c) { *reinterpret_cast<float4 *>(p.xf_out + fbase + frow(i) * p.C_out + 4 * c) = sn_lds(fslab + i * FS + 16 * c); });
                pieces(std::integral_constant<int, CH / 8>{}, [&](int i, int c) {
                    const int o = prow(i) * p.C_out + 8 * c;
                    const float4 h = sn_lds(hslab + i * PS + 16 * c), l = sn_lds(lslab + i * PS + 16 * c);
                    *reinterpret_cast<float4 *>(p.oh + pbase + o) = h; *reinterpret_cast<float4 *>(p.ol + pbase + o) = l;
                    if (RING && MODE == SN_RES && slot(i) < 64) {
                        *reinterpret_cast<float4 *>(p.oh + pbase + o + SN_RING * p.C_out) = h; *reinterpret_cast<float4 *>(p.ol + pbase + o + SN_RING * p.C_out) = l;
                    }
                });
            }
            tc_fence_before();
        } else ok = false;
    }
    if (!ok && atomicCAS(&p.status->code, DEV_OK, DEV_TIMEOUT) == DEV_OK) { p.status->cta = blockIdx.x; p.status->step = blockIdx.y; p.status->phase = 20 + MODE; }
    if (NS > 1) cluster_sync_all();                              // nobody leaves while a peer may still send to it
    else __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS) : "memory");
    }
}

// x_0 = W_in X + b_in for the positions [0, n_pos) of every segment, fp32 and bf16 parts (N1, N2 of the reading above).  A block
// takes SN_IN_POS positions: a weight is read once for all of them.
constexpr int SN_IN_POS = 8;
// RING: 64 positions of every row, from p_lo - row * lag on, into the rings
template <bool RING>
__global__ void subnet_input_kernel(const int16_t *__restrict__ hist, const float *__restrict__ W_in, const float *__restrict__ b_in, int Bsub,
                                    long long L, int C, int r_lo, long long p_lo, int lag, int n_alloc, int n_pos, float *__restrict__ xf,
                                    __nv_bfloat16 *__restrict__ xh, __nv_bfloat16 *__restrict__ xl)
{
    const int seg = blockIdx.y, j0 = blockIdx.x * SN_IN_POS, r = r_lo + seg;
    const long long pos0 = p_lo - (long long)(RING ? r : seg) * lag + j0;
    __shared__ __align__(16) float X[64][SN_IN_POS];
    for (int i = threadIdx.x; i < Bsub * SN_IN_POS; i += blockDim.x) {
        const int z = i / SN_IN_POS, q = i % SN_IN_POS;
        X[z][q] = (z < r && pos0 + q < L && (!RING || pos0 + q >= 0)) ? (float)hist[(size_t)z * L + pos0 + q] * (1.0f / 32768.0f) : 0.f;
    }
    __syncthreads();
    const size_t row = (size_t)seg * n_alloc + j0;
    for (int c = threadIdx.x; c < C; c += blockDim.x) {
        float v[SN_IN_POS];
        const float b = b_in[c];
#pragma unroll
        for (int q = 0; q < SN_IN_POS; ++q) v[q] = b;
        for (int z = 0; z < r; ++z) {
            const float w = W_in[(size_t)z * C + c];
#pragma unroll
            for (int q = 0; q < SN_IN_POS; ++q) v[q] = fmaf(w, X[z][q], v[q]);
        }
#pragma unroll
        for (int q = 0; q < SN_IN_POS; ++q) {
            if (j0 + q >= n_pos) break;
            const float x = pos0 + q < L ? v[q] : 0.f;
            const __nv_bfloat16 h = __float2bfloat16_rn(x), l = __float2bfloat16_rn(x - __bfloat162float(h));
            const int slot = (int)((pos0 + q) & (SN_RING - 1));
            const size_t o = (RING ? (size_t)r * (SN_RING + 64) + slot : row + q) * C + c;
            xf[RING ? ((size_t)r * SN_RING + slot) * C + c : o] = x;
            xh[o] = h;
            xl[o] = l;
            if (RING && slot < 64) { xh[o + (size_t)SN_RING * C] = h; xl[o + (size_t)SN_RING * C] = l; }
        }
    }
}

static float round_bf16_host(float v)
{
    uint32_t b;
    std::memcpy(&b, &v, 4);
    b += 0x7fffu + ((b >> 16) & 1u);
    b &= 0xffff0000u;
    float r;
    std::memcpy(&r, &b, 4);
    return r;
}

static bool upload_bf16(__nv_bfloat16 **dst, const float *src, size_t n, size_t n_alloc)
{
    std::vector<uint16_t> h(n_alloc, 0);
    for (size_t i = 0; i < n; ++i) {
        const float r = round_bf16_host(src[i]);
        uint32_t b;
        std::memcpy(&b, &r, 4);
        h[i] = (uint16_t)(b >> 16);
    }
    return cudaMalloc((void **)dst, n_alloc * 2) == cudaSuccess && cudaMemcpy(*dst, h.data(), n_alloc * 2, cudaMemcpyHostToDevice) == cudaSuccess;
}

static bool upload_f32(float **dst, const float *src, size_t n)
{
    return cudaMalloc((void **)dst, n * 4) == cudaSuccess && cudaMemcpy(*dst, src, n * 4, cudaMemcpyHostToDevice) == cudaSuccess;
}

static void free_acts(wrnn_subscale_net *n)
{
    cudaFree(n->xf); cudaFree(n->xh); cudaFree(n->xl); cudaFree(n->ah); cudaFree(n->al);
    n->xf = nullptr; n->xh = n->xl = n->ah = n->al = nullptr; n->n_seg = n->n_alloc = 0;
}

// activation tensors for n_seg segments of n_pos positions (grown on demand; synchronises when it grows; a schedule of calls reserves
// what its largest one takes, see subnet_reserve).  Zeroed in the order of stream s, on which the call runs: the default stream's order means
// nothing to a stream that does not block with it.
static int ensure_acts(wrnn_subscale_net *n, int n_seg, int n_pos, cudaStream_t s)
{
    const int n_alloc = ((n_pos + SN_BM - 1) / SN_BM) * SN_BM + SN_BM;       // tiles are whole, taps may reach one tile further
    if (n_seg <= n->n_seg && n_alloc <= n->n_alloc) return WRNN_OK;
    cudaDeviceSynchronize();
    free_acts(n);
    const size_t rows = (size_t)n_seg * n_alloc;
    if (cudaMalloc((void **)&n->xf, rows * n->res_ch * 4) != cudaSuccess || cudaMalloc((void **)&n->xh, rows * n->res_ch * 2) != cudaSuccess ||
        cudaMalloc((void **)&n->xl, rows * n->res_ch * 2) != cudaSuccess || cudaMalloc((void **)&n->ah, rows * n->conv_ch * 2) != cudaSuccess ||
        cudaMalloc((void **)&n->al, rows * n->conv_ch * 2) != cudaSuccess) {
        cudaGetLastError(); free_acts(n); n->err = "activation buffers of the conditioning network do not fit"; return WRNN_ERR_NOMEM;
    }
    if (cudaMemsetAsync(n->xh, 0, rows * n->res_ch * 2, s) != cudaSuccess || cudaMemsetAsync(n->xl, 0, rows * n->res_ch * 2, s) != cudaSuccess ||
        cudaMemsetAsync(n->ah, 0, rows * n->conv_ch * 2, s) != cudaSuccess || cudaMemsetAsync(n->al, 0, rows * n->conv_ch * 2, s) != cudaSuccess ||
        cudaMemsetAsync(n->xf, 0, rows * n->res_ch * 4, s) != cudaSuccess) {
        cudaGetLastError(); free_acts(n); n->err = "activation buffers of the conditioning network could not be cleared"; return WRNN_ERR_CUDA;
    }
    if (!make_map(&n->tmXh, n->xh, (long long)rows, n->res_ch, SN_BM) || !make_map(&n->tmXl, n->xl, (long long)rows, n->res_ch, SN_BM) ||
        !make_map(&n->tmAh, n->ah, (long long)rows, n->conv_ch, SN_BM) || !make_map(&n->tmAl, n->al, (long long)rows, n->conv_ch, SN_BM)) {
        free_acts(n); n->err = "tensor map encoding failed"; return WRNN_ERR_CUDA;
    }
    n->n_seg = n_seg; n->n_alloc = n_alloc;
    return WRNN_OK;
}

constexpr int SN_BN_CONV = 96, SN_BN_RES = 96, SN_BN_OUT = 64;
constexpr int SN_ST_CONV = 4, SN_ST_RES = 3, SN_ST_OUT = 4;
// launch with programmatic stream serialization: the kernel may start while its predecessor in the stream drains (it waits for
// the predecessor's completion itself, with griddepcontrol.wait, before it reads anything)
template <typename K>
static void pdl_launch(K kernel, dim3 grid, int smem, cudaStream_t s, const CUtensorMap &a, const CUtensorMap &b, const CUtensorMap &w, const SubnetGemmParams &p, int cluster = 1)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid; cfg.blockDim = dim3(SN_THREADS); cfg.dynamicSmemBytes = (size_t)smem; cfg.stream = s;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    at[1].id = cudaLaunchAttributeClusterDimension;
    at[1].val.clusterDim.x = (unsigned)cluster; at[1].val.clusterDim.y = 1; at[1].val.clusterDim.z = 1;
    cfg.attrs = at; cfg.numAttrs = cluster > 1 ? 2 : 1;
    cudaLaunchKernelEx(&cfg, kernel, a, b, w, p);
}

// stages, and a slab of fp32 values for the epilogue of all but the convolution
template <int BN, int ST> constexpr int sn_smem(bool slab) { return ST * (2 * SN_BM * TC_BK * 2 + BN * TC_BK * 2) + 1024 + (slab ? 2 * SN_BM * (BN * 2 + 16) : 0); }
constexpr int SN_SMEM_CONV = sn_smem<SN_BN_CONV, SN_ST_CONV>(false), SN_SMEM_RES = sn_smem<SN_BN_RES, SN_ST_RES>(true), SN_SMEM_OUT = sn_smem<SN_BN_OUT, SN_ST_OUT>(true);
constexpr int sn_smem_split(int ns) { return SN_SMEM_CONV + (ns - 1) * SN_BM * (SN_BN_CONV / ns * 4 + 16); }

// k-blocks of a product over so many channels: beyond the last channel both operands' boxes are filled with zeros
static int sn_kbs(int channels) { return (channels + TC_BK - 1) / TC_BK; }

// The whole network for the segments of one call: v[seg][n_steps][cond_dim] (the conditioning vectors the stepping call
// of these rows consumes).  Segment b is row r_lo + b from position p_lo - b * lag on.
int subnet_run(wrnn_subscale_net *n, const int16_t *hist, const float *frames, int n_frames, int hop, long long L, int r_lo, int n_rows,
               long long p_lo, int lag, int n_steps, float *v, unsigned long long limit_ns, cudaStream_t s)
{
    if (n_rows <= 0 || n_steps <= 0) return WRNN_OK;
    const int n0 = n_steps + n->reach;                       // positions of x_0 a segment needs
    int rc = ensure_acts(n, n_rows, n0, s);
    if (rc != WRNN_OK) return rc;
    if (cudaMemsetAsync(n->status, 0, sizeof(DevStatus), s) != cudaSuccess) return WRNN_ERR_CUDA;
    subnet_input_kernel<false><<<dim3((n0 + SN_IN_POS - 1) / SN_IN_POS, n_rows), 256, 0, s>>>(hist, n->W_in, n->b_in, n->B, L, n->res_ch, r_lo, p_lo, lag, n->n_alloc, n0, n->xf, n->xh, n->xl);
    ++g_launches;
    SubnetGemmParams p;
    std::memset(&p, 0, sizeof(p));
    p.n_alloc = n->n_alloc; p.r_lo = r_lo; p.p_lo = p_lo; p.lag = lag; p.L = L; p.status = n->status; p.limit_ns = limit_ns;
    int need = n0;                                           // positions of x_l still needed
    for (int l = 0; l < n->n_layers; ++l) {
        const int d = n->dilation[l];
        need -= (n->taps - 1) * d;                           // positions of a_l and x_{l+1}
        const int mtiles = (need + SN_BM - 1) / SN_BM;
        // a_l = relu(conv): K = taps x res_ch, N = conv_ch
        p.n_kb_tap = sn_kbs(n->res_ch); p.taps = n->taps; p.dil = d; p.w_row0 = l * n->taps * n->conv_ch; p.w_tap_rows = n->conv_ch;
        p.n_pos = need; p.C_out = n->conv_ch; p.bias = n->b_conv + (size_t)l * n->conv_ch; p.oh = n->ah; p.ol = n->al; p.xf = nullptr; p.relu_parts = 0;
        pdl_launch(subnet_gemm_kernel<SN_BN_CONV, SN_CONV, SN_ST_CONV, false>, dim3(n->conv_ch / SN_BN_CONV, mtiles, n_rows), SN_SMEM_CONV, s,
                   n->tmXh, n->tmXl, n->tmWc, p);
        // x_{l+1} = x_l + W_res a_l + b_res: K = conv_ch, N = res_ch
        p.n_kb_tap = sn_kbs(n->conv_ch); p.taps = 1; p.dil = 0; p.w_row0 = l * n->res_ch; p.w_tap_rows = 0;
        p.C_out = n->res_ch; p.bias = n->b_res + (size_t)l * n->res_ch; p.oh = n->xh; p.ol = n->xl; p.xf = p.xf_out = n->xf; p.relu_parts = l == n->n_layers - 1;
        pdl_launch(subnet_gemm_kernel<SN_BN_RES, SN_RES, SN_ST_RES, false>, dim3(n->res_ch / SN_BN_RES, mtiles, n_rows), SN_SMEM_RES, s,
                   n->tmAh, n->tmAl, n->tmWr, p);
        g_launches += 2;
    }
    // v = frames + W_out relu(x_last) + b_out
    p.n_kb_tap = sn_kbs(n->res_ch); p.taps = 1; p.dil = 0; p.w_row0 = 0; p.w_tap_rows = 0; p.n_pos = n_steps; p.C_out = 0; p.bias = nullptr;
    p.v = v; p.n_steps = n_steps; p.cond_dim = n->cond_dim; p.frames = frames; p.n_frames = n_frames; p.hop = hop; p.Bsub = n->B; p.b_out = n->b_out;
    pdl_launch(subnet_gemm_kernel<SN_BN_OUT, SN_OUT, SN_ST_OUT, false>, dim3(1, (n_steps + SN_BM - 1) / SN_BM, n_rows), SN_SMEM_OUT, s,
               n->tmXh, n->tmXl, n->tmWo, p);
    ++g_launches;
    if (cudaGetLastError() != cudaSuccess) { n->err = "conditioning network launch failed"; return WRNN_ERR_CUDA; }
    return WRNN_OK;
}

// ---- the rings: 64 positions of a staggered generation at a time
static void free_rings(wrnn_subscale_net *n)
{
    cudaFree(n->rf); cudaFree(n->rh); cudaFree(n->rl); cudaFree(n->bh); cudaFree(n->bl);
    n->rf = nullptr; n->rh = n->rl = n->bh = n->bl = nullptr;
    for (cudaStream_t &s : n->side) { if (s) cudaStreamDestroy(s); s = nullptr; }
    for (cudaEvent_t &e : n->ev) { if (e) cudaEventDestroy(e); e = nullptr; }
}

// (zeroed in the order of stream s, which the streams of the network and of the stepping calls follow)
int subnet_ring_reserve(wrnn_subscale_net *n, cudaStream_t s)
{
    if (n->rf) return WRNN_OK;
    // (a pair of rows beyond an odd last one is read, not used: one row more)
    const size_t rows = (size_t)n->n_layers * n->B, part_rows = (rows + n->B + 1) * (SN_RING + 64), conv_rows = (size_t)(n->B + 1) * 64;
    int least = 0, greatest = 0;
    cudaDeviceGetStreamPriorityRange(&least, &greatest);
    bool ok = cudaMalloc((void **)&n->rf, rows * SN_RING * n->res_ch * 4) == cudaSuccess && cudaMalloc((void **)&n->rh, part_rows * n->res_ch * 2) == cudaSuccess &&
              cudaMalloc((void **)&n->rl, part_rows * n->res_ch * 2) == cudaSuccess && cudaMalloc((void **)&n->bh, conv_rows * n->conv_ch * 2) == cudaSuccess &&
              cudaMalloc((void **)&n->bl, conv_rows * n->conv_ch * 2) == cudaSuccess && cudaMemsetAsync(n->rf, 0, rows * SN_RING * n->res_ch * 4, s) == cudaSuccess &&
              cudaMemsetAsync(n->rh, 0, part_rows * n->res_ch * 2, s) == cudaSuccess && cudaMemsetAsync(n->rl, 0, part_rows * n->res_ch * 2, s) == cudaSuccess &&
              cudaMemsetAsync(n->bh, 0, conv_rows * n->conv_ch * 2, s) == cudaSuccess && cudaMemsetAsync(n->bl, 0, conv_rows * n->conv_ch * 2, s) == cudaSuccess;
    ok = ok && make_map_rows(&n->tmRh, n->rh, (long long)(rows + n->B + 1), SN_RING + 64, n->res_ch) && make_map_rows(&n->tmRl, n->rl, (long long)(rows + n->B + 1), SN_RING + 64, n->res_ch) &&
         make_map_rows(&n->tmBh, n->bh, n->B + 1, 64, n->conv_ch) && make_map_rows(&n->tmBl, n->bl, n->B + 1, 64, n->conv_ch);
    // the stepping calls first: a cluster of theirs needs sixteen free SMs of one part of the chip, a product of the network any
    ok = ok && cudaStreamCreateWithPriority(&n->side[0], cudaStreamNonBlocking, least) == cudaSuccess &&
         cudaStreamCreateWithPriority(&n->side[1], cudaStreamNonBlocking, greatest) == cudaSuccess;
    for (cudaEvent_t &e : n->ev) ok = ok && cudaEventCreateWithFlags(&e, cudaEventDisableTiming) == cudaSuccess;
    if (!ok) { cudaGetLastError(); free_rings(n); n->err = "rings of the conditioning network do not fit"; return WRNN_ERR_NOMEM; }
    return WRNN_OK;
}
cudaStream_t subnet_side(const wrnn_subscale_net *n, int i) { return n->side[i]; }
cudaEvent_t subnet_event(const wrnn_subscale_net *n, int i) { return n->ev[i]; }
// what the rings can follow: rows whose slots agree (a tile has two), and a block of 64 computed while the one before it is stepped
bool subnet_ring_fits(const wrnn_subscale_net *n, int lag)
{
    for (int d : n->dilation)
        if ((n->taps - 1) * d > 64) return false;
    return lag % SN_RING == 0 && lag - n->reach >= 2 * 64;
}

// The next 64 positions: rows r_lo .. r_lo + n_rows - 1, row r from position t0 - r * lag on (t0 a multiple of 64; a row starts at
// -64 ceil(reach / 64)).  v[B][64][cond_dim]; what belongs to positions below 0 or at and beyond L is not written.
int subnet_ring_run(wrnn_subscale_net *n, const int16_t *hist, const float *frames, int n_frames, int hop, long long L, int r_lo, int n_rows, long long t0, int lag,
                    float *v, int free_sms, unsigned long long limit_ns, cudaStream_t s)
{
    const size_t fl = (size_t)n->B * SN_RING * n->res_ch, pl = (size_t)n->B * (SN_RING + 64) * n->res_ch;       // a layer of the rings
    subnet_input_kernel<true><<<dim3(64 / SN_IN_POS, n_rows), 256, 0, s>>>(hist, n->W_in, n->b_in, n->B, L, n->res_ch, r_lo, t0 + n->reach, lag, 0, 64, n->rf, n->rh, n->rl);
    SubnetGemmParams p;
    std::memset(&p, 0, sizeof(p));
    p.r_lo = r_lo; p.n_seg = n_rows; p.t0 = t0; p.lag = lag; p.L = L; p.status = n->status; p.limit_ns = limit_ns;
    p.n_pos = 64;
    const int tiles = (n_rows + 1) / 2;
    int reach = n->reach;
    for (int l = 0; l < n->n_layers; ++l) {
        const int d = n->dilation[l];
        reach -= (n->taps - 1) * d;
        p.reach = reach;
        p.n_kb_tap = sn_kbs(n->res_ch); p.taps = n->taps; p.dil = d; p.w_row0 = l * n->taps * n->conv_ch; p.w_tap_rows = n->conv_ch;
        p.a_idx0 = l * n->B + r_lo; p.a_slot0 = (int)((t0 + reach) & (SN_RING - 1));
        p.C_out = n->conv_ch; p.bias = n->b_conv + (size_t)l * n->conv_ch; p.oh = n->bh; p.ol = n->bl; p.relu_parts = 0;
        // as many CTAs per tile as find an SM beside the stepping call (and share the k-blocks evenly)
        const int n_tiles = n->conv_ch / SN_BN_CONV, kbs = n->taps * p.n_kb_tap;
        const int ns = 3 * n_tiles * tiles <= free_sms && kbs % 3 == 0 ? 3 : 2 * n_tiles * tiles <= free_sms && kbs % 2 == 0 ? 2 : 1;
        auto conv = [&](auto NS_C) {
            constexpr int NS = decltype(NS_C)::value;
            pdl_launch(subnet_gemm_kernel<SN_BN_CONV, SN_CONV, SN_ST_CONV, true, NS>, dim3(NS * n_tiles, tiles, 1), sn_smem_split(NS), s, n->tmRh, n->tmRl, n->tmWc, p, NS);
        };
        if (ns == 3) conv(std::integral_constant<int, 3>{});
        else if (ns == 2) conv(std::integral_constant<int, 2>{});
        else conv(std::integral_constant<int, 1>{});
        p.n_kb_tap = sn_kbs(n->conv_ch); p.taps = 1; p.dil = 0; p.w_row0 = l * n->res_ch; p.w_tap_rows = 0;
        p.a_idx0 = r_lo; p.a_slot0 = 0; p.relu_parts = l == n->n_layers - 1;
        p.C_out = n->res_ch; p.bias = n->b_res + (size_t)l * n->res_ch; p.oh = n->rh + (l + 1) * pl; p.ol = n->rl + (l + 1) * pl;
        p.xf = n->rf + l * fl; p.xf_out = p.relu_parts ? nullptr : n->rf + (l + 1) * fl;
        pdl_launch(subnet_gemm_kernel<SN_BN_RES, SN_RES, SN_ST_RES, true>, dim3(n->res_ch / SN_BN_RES, tiles, 1), SN_SMEM_RES, s, n->tmBh, n->tmBl, n->tmWr, p);
    }
    p.n_kb_tap = sn_kbs(n->res_ch); p.taps = 1; p.dil = 0; p.w_row0 = 0; p.w_tap_rows = 0; p.C_out = 0; p.bias = nullptr;
    p.a_idx0 = n->n_layers * n->B + r_lo; p.a_slot0 = (int)(t0 & (SN_RING - 1)); p.reach = 0;
    p.v = v; p.n_steps = 64; p.cond_dim = n->cond_dim; p.frames = frames; p.n_frames = n_frames; p.hop = hop; p.Bsub = n->B; p.b_out = n->b_out;
    pdl_launch(subnet_gemm_kernel<SN_BN_OUT, SN_OUT, SN_ST_OUT, true>, dim3(1, tiles, 1), SN_SMEM_OUT, s, n->tmRh, n->tmRl, n->tmWo, p);
    g_launches += 2 + 2 * n->n_layers;
    if (cudaGetLastError() != cudaSuccess) { n->err = "conditioning network launch failed"; return WRNN_ERR_CUDA; }
    return WRNN_OK;
}
int subnet_clear_status(wrnn_subscale_net *n, cudaStream_t s) { return cudaMemsetAsync(n->status, 0, sizeof(DevStatus), s) == cudaSuccess ? WRNN_OK : WRNN_ERR_CUDA; }

int subnet_reserve(wrnn_subscale_net *n, int n_rows, int n_steps, cudaStream_t s) { return ensure_acts(n, n_rows, n_steps + n->reach, s); }
int subnet_reach(const wrnn_subscale_net *n) { return n->reach; }
int subnet_B(const wrnn_subscale_net *n) { return n->B; }
int subnet_cond_dim(const wrnn_subscale_net *n) { return n->cond_dim; }
int subnet_status(wrnn_subscale_net *n)
{
    DevStatus st;
    if (cudaMemcpy(&st, n->status, sizeof(st), cudaMemcpyDeviceToHost) != cudaSuccess) return WRNN_ERR_CUDA;
    return st.code == DEV_OK ? WRNN_OK : WRNN_ERR_TIMEOUT;
}

}  // namespace wrnn

using namespace wrnn;

extern "C" int wrnn_subscale_net_create(const wrnn_subscale_net_params *q, wrnn_subscale_net **out)
{
    if (out) *out = nullptr;
    if (!q || !out || !q->dilation || !q->W_in || !q->b_in || !q->W_conv || !q->b_conv || !q->W_res || !q->b_res || !q->W_out || !q->b_out)
        return WRNN_ERR_INVALID_ARG;
    if (q->B < 1 || q->B > 64 || q->n_layers < 1 || q->n_layers > 64 || q->taps < 1 || q->taps > 8 || q->cond_dim < 1 || q->cond_dim > 64)
        return WRNN_ERR_INVALID_ARG;
    // the tensor-core tiling: whole channel tiles
    if (q->conv_ch < SN_BN_CONV || q->conv_ch % SN_BN_CONV || q->res_ch < SN_BN_RES || q->res_ch % SN_BN_RES) return WRNN_ERR_UNSUPPORTED;
    int dev = 0;
    cudaDeviceProp prop;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaGetDeviceProperties(&prop, dev) != cudaSuccess) { cudaGetLastError(); return WRNN_ERR_CUDA; }
    if (prop.major != 10) return WRNN_ERR_UNSUPPORTED;
    wrnn_subscale_net *n = new (std::nothrow) wrnn_subscale_net();
    if (!n) return WRNN_ERR_NOMEM;
    n->B = q->B; n->n_layers = q->n_layers; n->taps = q->taps; n->conv_ch = q->conv_ch; n->res_ch = q->res_ch; n->cond_dim = q->cond_dim; n->device = dev;
    n->dilation.assign(q->dilation, q->dilation + q->n_layers);
    n->reach = 0;
    for (int d : n->dilation) {
        if (d < 1 || d > SN_BM / 2) { delete n; return WRNN_ERR_INVALID_ARG; }
        n->reach += (q->taps - 1) * d;
    }
    const size_t nc = (size_t)q->n_layers * q->taps * q->conv_ch * q->res_ch, nr = (size_t)q->n_layers * q->res_ch * q->conv_ch;
    std::vector<float> win((size_t)q->res_ch * q->B);
    for (int c = 0; c < q->res_ch; ++c)                      // transposed: [B][res_ch]
        for (int z = 0; z < q->B; ++z) win[(size_t)z * q->res_ch + c] = round_bf16_host(q->W_in[(size_t)c * q->B + z]);
    bool ok = upload_bf16(&n->Wc, q->W_conv, nc, nc) && upload_bf16(&n->Wr, q->W_res, nr, nr) &&
              upload_bf16(&n->Wo, q->W_out, (size_t)q->cond_dim * q->res_ch, (size_t)64 * q->res_ch) &&
              upload_f32(&n->W_in, win.data(), win.size()) && upload_f32(&n->b_in, q->b_in, q->res_ch) &&
              upload_f32(&n->b_conv, q->b_conv, (size_t)q->n_layers * q->conv_ch) && upload_f32(&n->b_res, q->b_res, (size_t)q->n_layers * q->res_ch) &&
              upload_f32(&n->b_out, q->b_out, q->cond_dim) && cudaMalloc((void **)&n->status, sizeof(DevStatus)) == cudaSuccess &&
              cudaMemset(n->status, 0, sizeof(DevStatus)) == cudaSuccess;
    ok = ok && make_map(&n->tmWc, n->Wc, (long long)q->n_layers * q->taps * q->conv_ch, q->res_ch, SN_BN_CONV) &&
         make_map(&n->tmWr, n->Wr, (long long)q->n_layers * q->res_ch, q->conv_ch, SN_BN_RES) && make_map(&n->tmWo, n->Wo, 64, q->res_ch, SN_BN_OUT);
    auto allow = [](auto kernel, int smem) { return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) == cudaSuccess; };
    constexpr int sc = SN_SMEM_CONV, sr = SN_SMEM_RES, so = SN_SMEM_OUT;
    ok = ok && allow(subnet_gemm_kernel<SN_BN_CONV, SN_CONV, SN_ST_CONV, false>, sc) && allow(subnet_gemm_kernel<SN_BN_CONV, SN_CONV, SN_ST_CONV, true>, sc) &&
         allow(subnet_gemm_kernel<SN_BN_CONV, SN_CONV, SN_ST_CONV, true, 2>, sn_smem_split(2)) && allow(subnet_gemm_kernel<SN_BN_CONV, SN_CONV, SN_ST_CONV, true, 3>, sn_smem_split(3)) &&
         allow(subnet_gemm_kernel<SN_BN_RES, SN_RES, SN_ST_RES, false>, sr) && allow(subnet_gemm_kernel<SN_BN_RES, SN_RES, SN_ST_RES, true>, sr) &&
         allow(subnet_gemm_kernel<SN_BN_OUT, SN_OUT, SN_ST_OUT, false>, so) && allow(subnet_gemm_kernel<SN_BN_OUT, SN_OUT, SN_ST_OUT, true>, so);
    // (uploads and the cleared status word are in the default stream's order, which not every caller's stream follows)
    ok = ok && cudaStreamSynchronize(0) == cudaSuccess;
    if (!ok) { cudaGetLastError(); wrnn_subscale_net_destroy(n); return WRNN_ERR_NOMEM; }
    *out = n;
    return WRNN_OK;
}

extern "C" void wrnn_subscale_net_destroy(wrnn_subscale_net *n)
{
    if (!n) return;
    cudaSetDevice(n->device);
    cudaDeviceSynchronize();
    free_acts(n);
    free_rings(n);
    cudaFree(n->Wc); cudaFree(n->Wr); cudaFree(n->Wo); cudaFree(n->W_in); cudaFree(n->b_in); cudaFree(n->b_conv); cudaFree(n->b_res);
    cudaFree(n->b_out); cudaFree(n->status);
    cudaGetLastError();
    delete n;
}

extern "C" int wrnn_subscale_net_conditioning(wrnn_subscale_net *n, const int16_t *hist, const float *frames, int32_t n_frames, int32_t hop,
                                              int32_t row, int64_t L, float *v, void *cuda_stream)
{
    if (!n || !hist || !frames || !v || hop < 1 || row < 0 || row >= n->B || L < 1 || L > (1ll << 24)) return WRNN_ERR_INVALID_ARG;
    if (((long long)n->B * (L - 1) + row) / hop >= n_frames) return WRNN_ERR_INVALID_ARG;
    if (cudaSetDevice(n->device) != cudaSuccess) return WRNN_ERR_CUDA;
    return subnet_run(n, hist, frames, n_frames, hop, L, row, 1, 0, 0, (int)L, v, 2000000000ull, (cudaStream_t)cuda_stream);
}

extern "C" int wrnn_subscale_net_status(wrnn_subscale_net *n) { return n ? subnet_status(n) : WRNN_ERR_INVALID_ARG; }
