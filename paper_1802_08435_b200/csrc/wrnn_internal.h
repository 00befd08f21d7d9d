// Host-side structures shared by the translation units of libwrnn.so.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <atomic>
#include <cstdlib>
#include <cstring>
#include <string>
#include <thread>
#include <vector>

#include "../../include/wrnn.h"
#include "wrnn_device.cuh"

namespace wrnn {

// A matrix stored as compressed block rows of 4x4 blocks (Section 3.2).  A dense matrix is
// the same structure with every block present.  vals holds nnz blocks of 16 weights each,
// block-row-major inside a block (vals[i][4 r + c] = W[4 br + r][4 bc + c]), in the model's
// storage type (fp32 or bf16).
struct BsrDev {
    int rows4 = 0, cols4 = 0, nnz = 0;
    int *row_ptr = nullptr;        // [rows4 + 1]
    uint16_t *col = nullptr;       // [nnz] block column
    void *vals = nullptr;          // [nnz][16]
};

// Host image of the same thing (after masking and rounding), kept for the packers of the
// specialised kernels.
struct BsrHost {
    int rows4 = 0, cols4 = 0;
    std::vector<int> row_ptr;
    std::vector<uint16_t> col;
    std::vector<float> vals;       // fp32 values (already rounded to the storage type)
};

// Everything one stepping call needs besides the model (device pointers).
struct StepArgs {
    const float *cond;       // [batch][n_frames][cond_dim] (unused by the step kernels: g is projected)
    int n_frames, hop, row_stride, row_offset_mul;
    long long n_steps;
    int batch;
    unsigned long long seed;
    long long step0;
    unsigned stream0;
    const float *h_in;  float *h_out;            // may be null
    const uint8_t *c_in, *f_in; uint8_t *c_st_out, *f_st_out;
    const uint8_t *c_forced, *f_forced;          // [batch][n_steps] or null
    uint8_t *c_out, *f_out;                      // [batch][n_steps] or null
    int16_t *out;                                // [batch][n_steps] or null
    float *dbg_gates, *dbg_h, *dbg_logits;       // or null
    // staggered subscale rows: row b of the call is row_lag steps behind row b - 1 and takes one conditioning frame per
    // step of the call (0 = rows in lock step); out_pitch = samples between the rows of `out` (0 = n_steps)
    int row_lag;
    long long out_pitch;
    // projected conditioning [batch][n_frames][3H] that is there already (null: projected from cond by this call), with a status word that is cleared
    const float *g;
    int clusters;            // at most so many 16-CTA clusters at a time, where four rows per cluster (two with fp32 weights) allow it; 0, and
                             // always more than four rows per cluster: as many as there are
    // fused subscale variant: 16-bit samples of parts A and B in place of the bytes above (batch 1)
    const uint16_t *a_in, *b_in; uint16_t *a_st_out, *b_st_out;
    const uint16_t *a_forced, *b_forced;         // [n_steps] or null
    uint16_t *a_out, *b_out;                     // [n_steps] or null
};

struct ResidentPack;   // packed weights of the shared-memory-resident kernels (opaque here)
struct BatchedPack;    // fragment-packed weights and activation images of the batched kernel (opaque here)
struct SparsePack;     // compressed block rows of the block-sparse kernel on several clusters (opaque here)
struct Sparse1Pack;    // the same inside one cluster
struct ResF32Pack;     // per-CTA fp32 weight shards of the single-stream fp32 resident kernel (opaque here)
struct ResClPack;      // per-CTA weights of the cluster-resident kernel (opaque here)
struct ResRowsPack;    // the same of its form for many rows
struct ClHalf;         // fp16 matrices that both are packed from
struct BcPack;         // per-CTA weight slices and stacked activation images of the cluster-partitioned multi-row kernel

}  // namespace wrnn

struct wrnn_subscale_net;   // the conditioning network of the Subscale WaveRNN (wrnn_subnet.cu)

struct wrnn_model {
    int H = 0, cond_dim = 0, dtype = 0, kernel = 0, max_batch = 0;
    int variant = 0;                // 0: WaveRNN (Eq. 2); 1: Fused Subscale WaveRNN 2x (I has 12 columns, O2 / O4 64 rows)
    int device = 0, n_sms = 0;
    bool sparse = false;
    int mask_br = 4, mask_bc = 4;   // shape of one block of the sparsity masks (Section 3.2)

    // generic format
    wrnn::BsrDev R, O1, O2, O3, O4;
    float *I = nullptr;            // [3H][3] fp32 (values rounded to storage type; masked column zeroed)
    float *b_gate = nullptr, *b1 = nullptr, *b2 = nullptr, *b3 = nullptr, *b4 = nullptr;
    float *W_condT = nullptr;      // [cond_dim][3H] fp32 (rounded values), transposed for coalescing
    int64_t weight_bytes = 0;      // packed bytes read per step (values + indices + row pointers)

    // per-call scratch owned by the model
    float *g = nullptr;            // projected conditioning [batch][n_frames][3H]
    size_t g_cap = 0;              // floats
    float *hbuf[2] = {nullptr, nullptr};   // [max_batch][H]
    float *a_fine = nullptr;       // [max_batch][3][H/2]  R h of the fine rows, kept across the coarse head
    float *q = nullptr;            // [max_batch][H/2]
    float *logits = nullptr;       // [max_batch][256]
    uint8_t *c_cur = nullptr, *c_prev = nullptr, *f_prev = nullptr;   // [max_batch]
    unsigned long long *bar = nullptr;     // grid barrier counter
    wrnn::DevStatus *status = nullptr;     // device status word
    // host staging for wrnn_sample_host
    float *stage_cond = nullptr; size_t stage_cond_cap = 0;
    int16_t *stage_out = nullptr; size_t stage_out_cap = 0;
    uint8_t *sub_scratch = nullptr; size_t sub_cap = 0;   // history, conditioning and carry state of wrnn_sample_subscale_dependent

    wrnn::ResidentPack *resident = nullptr;
    wrnn::ResF32Pack *resf32 = nullptr;
    wrnn::ResClPack *rescl = nullptr;
    wrnn::ResRowsPack *resrows = nullptr;
    wrnn::ClHalf *half = nullptr;     // while the model is created
    int prof_cl = 0;                  // the last call with phase timing ran on the cluster-resident kernel (2: on its form for many rows)
    // wrnn_selftest_lost_word: bound of every device-side wait (0 = the default of two seconds) and the CTA / step whose
    // publication (or operand load) is withheld (-1 = none)
    unsigned long long dbg_limit_ns = 0;
    int dbg_skip_cta = -1;
    long long dbg_skip_step = -1;
    // At least a millisecond: waits are also for a CTA's own copies in flight (weights, operands), some microseconds, and one that gave up on them
    // could leave before they land in its shared memory.
    unsigned long long wait_limit_ns() const { return dbg_limit_ns ? std::max(dbg_limit_ns, 1000000ull) : 2000000000ull; }
    bool prof_enabled = false;      // wrnn_phase_profile: the resident kernels stamp their phases
    wrnn::BatchedPack *batched = nullptr;
    wrnn::SparsePack *sparse_pack = nullptr;
    wrnn::Sparse1Pack *sparse1 = nullptr;
    wrnn::BcPack *bcluster = nullptr;

    // host images for packers
    wrnn::BsrHost hR, hO1, hO2, hO3, hO4;
    std::vector<float> hI, hb_gate, hb1, hb2, hb3, hb4;

    std::string err;
};

namespace wrnn {

extern std::atomic<long long> g_launches;

// Whether the persistent cluster kernels are launched with the cooperative attribute (the driver then refuses the launch
// unless all clusters can be co-resident).  Co-residency is checked against the occupancy API when a model is created, so
// the attribute is a second line of defence; it is dropped under WRNN_NO_COOP=1 and when a CUDA injection library is
// loaded into the process (a profiler: kernel replay does not accept cooperative cluster launches).
inline bool coop_launch_allowed()
{
    const char *no_coop = getenv("WRNN_NO_COOP");
    if (no_coop && no_coop[0] == '1') return false;
    const char *inj = getenv("CUDA_INJECTION64_PATH");
    return !(inj && inj[0]);
}

// wrnn_api.cu: argument checks shared by the stepping entry points (fills the cond / state part of StepArgs)
int check_step(wrnn_model *m, const wrnn_cond *cond, int64_t n_steps, int32_t batch, const wrnn_state *st, StepArgs *a);

// wrnn_generic.cu
int generic_launch_info(const wrnn_model *m, int batch, int *n_ctas, int *n_threads, int *smem);
int generic_run(wrnn_model *m, const StepArgs &a, cudaStream_t s);   // returns wrnn_status
// `status`, if given, is cleared; a kernel launched behind it with programmatic stream serialization may start at once and waits itself
int cond_project(wrnn_model *m, const float *cond, int batch, int n_frames, float *g, wrnn::DevStatus *status, cudaStream_t s);
void noalloc_warm(int device);   // resolves the device address of the fixed scratch array of wrnn_sample_noalloc (once per device)
int fold_launch(const int16_t *x, long long n_total, int B, int16_t *sub, bool unfold, cudaStream_t s);
int fs2_unfold_launch(const int16_t *ab, long long n, int16_t *u, cudaStream_t s);
int subscale_cond_launch(const int16_t *hist, const float *frames, const float *V, const float *bias, float *v, int B, long long L, int F,
                         int D, int n_frames, int hop, int r_lo, int n_rows, long long p_lo, int lag, int n_steps, cudaStream_t s);

// wrnn_subnet.cu: the masked dilated conditioning network on the tensor cores, for the segments of one stepping call
int subnet_run(wrnn_subscale_net *n, const int16_t *hist, const float *frames, int n_frames, int hop, long long L, int r_lo, int n_rows,
               long long p_lo, int lag, int n_steps, float *v, unsigned long long limit_ns, cudaStream_t s);
int subnet_reserve(wrnn_subscale_net *n, int n_rows, int n_steps, cudaStream_t s);        // activations for calls of up to that many rows and steps
// the same in blocks of 64 positions for a whole staggered generation, on rings (see wrnn_subnet.cu)
bool subnet_ring_fits(const wrnn_subscale_net *n, int lag);
int subnet_ring_reserve(wrnn_subscale_net *n, cudaStream_t s);
int subnet_ring_run(wrnn_subscale_net *n, const int16_t *hist, const float *frames, int n_frames, int hop, long long L, int r_lo, int n_rows, long long t0, int lag,
                    float *v, int free_sms, unsigned long long limit_ns, cudaStream_t s);
int subnet_clear_status(wrnn_subscale_net *n, cudaStream_t s);
cudaStream_t subnet_side(const wrnn_subscale_net *n, int i);              // 0: the network's, 1: the stepping calls'
cudaEvent_t subnet_event(const wrnn_subscale_net *n, int i);
int subnet_reach(const wrnn_subscale_net *n);
int subnet_B(const wrnn_subscale_net *n);
int subnet_cond_dim(const wrnn_subscale_net *n);

// the bits of a value that is a bf16 number already
inline uint16_t bf16_bits(float rounded)
{
    uint32_t b;
    std::memcpy(&b, &rounded, 4);
    return (uint16_t)(b >> 16);
}

// f(0), .., f(n - 1) on a few host threads (or, where none can be had, here); f does not throw
template <typename F>
void parallel_for(int n, F f)
{
    const int nt = std::max(1, std::min({n, 8, (int)std::thread::hardware_concurrency()}));
    auto run = [&f, n, nt](int t) { for (int i = t; i < n; i += nt) f(i); };
    std::vector<std::thread> threads;
    int started = 1;                             // the shares taken: this thread has the first
    try {
        threads.reserve(nt);
        for (; started < nt; ++started) threads.emplace_back(run, started);
    } catch (...) {}
    run(0);
    for (int t = started; t < nt; ++t) run(t);
    for (std::thread &t : threads) t.join();
}

// Lets `fn` be launched with `need` bytes of dynamic shared memory: with as much as a block can have.  The limit belongs to the
// function, not to a model: set to what one model needs, it would refuse the launches of a larger one that is alive.
inline bool allow_smem(const void *fn, int device, size_t need)
{
    int most = 0;
    cudaFuncAttributes fa;
    const bool ok = cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin, device) == cudaSuccess && cudaFuncGetAttributes(&fa, fn) == cudaSuccess &&
                    need + fa.sharedSizeBytes <= (size_t)most && cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, most - (int)fa.sharedSizeBytes) == cudaSuccess;
    if (!ok) cudaGetLastError();
    return ok;
}

// wrnn_resident.cu
int resident_supported(const wrnn_model *m, int batch, std::string *why);
int resident_prepare(wrnn_model *m);                                  // pack + upload at create
void resident_destroy(wrnn_model *m);
int resident_launch_info(const wrnn_model *m, int batch, int *n_ctas, int *n_threads, int *smem,
                         int64_t *weight_bytes);
int resident_run(wrnn_model *m, const StepArgs &a, cudaStream_t s);
int resident_phase_cycles(const wrnn_model *m, long long *out16);
int resident_pair_supported(const wrnn_model *m, int batch);          // two streams per launch on the same weights (batch 2 or 4)
int resident_pair_run(wrnn_model *m, const StepArgs &a, int pair, cudaStream_t s);

// host packers shared by the resident kernels (wrnn_resident.cu)
void dense_row_bf16(const BsrHost &M, int row, int c0, int n, uint16_t *dst);       // dense row of a block-row matrix -> bf16 bits of columns [c0, c0 + n)
void pack_tile(const std::vector<std::vector<uint16_t>> &rows, int K, uint16_t *dst);   // rows[16][K] -> m16n8k16 A fragments [K/16][32 lanes][8]

// wrnn_rescl.cu: rows of a dense H = 896 model (bf16 or fp32), the whole model in one cluster (R in tensor memory)
int rescl_supported(const wrnn_model *m, int batch);
int rescl_prepare(wrnn_model *m);
void rescl_destroy(wrnn_model *m);
void rescl_packed(wrnn_model *m);        // gives up what only the packers of the cluster-resident kernels need
int rescl_launch_info(const wrnn_model *m, int batch, int *n_ctas, int *n_threads, int *smem, int64_t *weight_bytes);
int rescl_run(wrnn_model *m, const StepArgs &a, cudaStream_t s);
int rescl_phase_cycles(const wrnn_model *m, long long *out16);
int rescl_clusters(const wrnn_model *m, int batch, int clusters);        // on the chip at a time, with StepArgs.clusters = clusters

// wrnn_resrows.cu: five to fourteen rows per cluster (bf16)
int resrows_prepare(wrnn_model *m);
void resrows_destroy(wrnn_model *m);
int resrows_launch_info(const wrnn_model *m, int batch, int *n_ctas, int *n_threads, int *smem, int64_t *weight_bytes);
int resrows_run(wrnn_model *m, const StepArgs &a, cudaStream_t s);
int resrows_phase_cycles(const wrnn_model *m, long long *out16);
int resrows_clusters(const wrnn_model *m, int batch);

// wrnn_resf32.cu: the same role for dense fp32 models (every matrix sharded chip-wide, nothing replicated)
int resf32_supported(const wrnn_model *m, int batch, std::string *why);
int resf32_prepare(wrnn_model *m);
void resf32_destroy(wrnn_model *m);
int resf32_launch_info(const wrnn_model *m, int batch, int *n_ctas, int *n_threads, int *smem, int64_t *weight_bytes);
int resf32_run(wrnn_model *m, const StepArgs &a, cudaStream_t s);
int resf32_phase_cycles(const wrnn_model *m, long long *out16);

// wrnn_sparse.cu
// the form inside one cluster; the sparse_* functions choose
int sparse1_prepare(wrnn_model *m);
void sparse1_destroy(wrnn_model *m);
void sparse1_launch_info(const wrnn_model *m, int *n_ctas, int *n_threads, int *smem, int64_t *weight_bytes);
int sparse1_run(wrnn_model *m, const StepArgs &a, cudaStream_t s);
int sparse_supported(const wrnn_model *m, int batch, std::string *why);
int sparse_prepare(wrnn_model *m);
void sparse_destroy(wrnn_model *m);
int sparse_launch_info(const wrnn_model *m, int batch, int *n_ctas, int *n_threads, int *smem, int64_t *weight_bytes);
int sparse_run(wrnn_model *m, const StepArgs &a, cudaStream_t s);

// wrnn_batched.cu
int batched_supported(const wrnn_model *m, int batch, std::string *why);
int batched_prepare(wrnn_model *m);
void batched_destroy(wrnn_model *m);
int batched_launch_info(const wrnn_model *m, int batch, int *n_ctas, int *n_threads, int *smem, int64_t *weight_bytes);
int batched_run(wrnn_model *m, const StepArgs &a, cudaStream_t s);
std::vector<uint16_t> dense_bf16_bits(const BsrHost &M);   // host block rows -> dense row-major bf16 bits

// wrnn_bcluster.cu
int bcluster_supported(const wrnn_model *m, int batch, std::string *why);
int bcluster_prepare(wrnn_model *m);
void bcluster_destroy(wrnn_model *m);
int bcluster_launch_info(const wrnn_model *m, int batch, int *n_ctas, int *n_threads, int *smem, int64_t *weight_bytes);
int bcluster_run(wrnn_model *m, const StepArgs &a, cudaStream_t s);

}  // namespace wrnn
