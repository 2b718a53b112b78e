// extern "C" boundary of the LapH block library (declared in include/laph.h):
// argument validation, plans (phase tables, tile tables, kernel parameters),
// stream-ordered execution and the simple one-shot entry points.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <functional>
#include <new>
#include <string>
#include <vector>

#include "laph.h"
#include "laph_internal.cuh"

using laph::InstDev;
using laph::TileDev;

namespace laph {
int record_cuda_error(cudaError_t e, const char *where);
}

namespace {

thread_local char g_last_cuda[256] = "";

int cuda_fail(cudaError_t e, const char *where)
{
    snprintf(g_last_cuda, sizeof(g_last_cuda), "%s: %s", where, cudaGetErrorString(e));
    return LAPH_ERR_CUDA;
}

}  // namespace

// the same record for the other translation units
int laph::record_cuda_error(cudaError_t e, const char *where) { return cuda_fail(e, where); }

namespace {

#define CK(call)                                         \
    do {                                                 \
        cudaError_t e_ = (call);                         \
        if (e_ != cudaSuccess) return cuda_fail(e_, #call); \
    } while (0)

bool is_tc_mode(int mode) { return mode >= LAPH_MODE_TC_F16X3 && mode <= LAPH_MODE_TC_BF16; }

constexpr int MAX_N = 4096;
constexpr int MAX_P = 4096;
constexpr int MAX_L = 512;
constexpr int32_t MAX_MOM = 1 << 20;
// Sites summed between the reductions of partial sums: FP32 CUDA-core sums
// (round to nearest) on the FP32 path; tensor-core FP32 accumulation, whose
// error grows linearly with the number of additions, on the split path.
constexpr int SIMT_DEFAULT_CHUNK = 1024;
constexpr int TC_DEFAULT_CHUNK = 128;
// Tensor-core path: sites per block of the FP64 site reduction.  A tile
// covers one block; its FP32 running sums become one FP32 partial per
// output, and the partials of all blocks are added in FP64.
constexpr int TC_DEFAULT_SUM = 8192;
// Largest B-operand buffer of the tensor-core path: the timeslices of a batch
// are processed in chunks whose stage images fit in it.
constexpr size_t PSI_CAP_BYTES = 24ull << 30;
// Cutting units into drains (see the plan's `emit`).  Work of a tile beside its
// stages, in stages: a tile of one drain (16 stages) takes as long as 23 stages
// of a long one (113 us for 7 tiles per CTA at L=24, N=32, 7 momenta, one
// timeslice, against 0.7 us a stage).  Bytes moved in the time of a stage (about
// 0.6 us at 4 TB/s).  The gain below which the tiles stay whole, the waves of
// tiles above which a thin last wave no longer matters, and the most bytes of
// extra partials.
constexpr int TILE_STAGES = 8;
constexpr double SPLIT_BYTES_PER_STAGE = 2.4e6;
constexpr double SPLIT_MARGIN = 0.03;
constexpr int SPLIT_MAX_WAVES = 10;
constexpr size_t SPLIT_MAX_BYTES = 1ull << 30;
// Estimates for the choice of the tile shape (see the plan's `shape_us`), fitted
// to the triplets at L=32, N=64, 19 momenta (us per stage of a long tile, 208 /
// 192 / 128 accumulator columns in layout 0: 0.734 / 0.695 / 0.625;
// layout 1, 208 / 176 / 128 columns: 0.747 / 0.698 / 0.636) and to the B-operand
// pass (bytes written and read per us).
constexpr double STAGE_US = 0.45, STAGE_US_COL = 0.00137;
constexpr double PAIR_STAGE_US = 0.46, PAIR_STAGE_US_COL = 0.00137;   // CTA pairs: 0.746 us at 208 columns
constexpr double RING_COST = 1.11;
constexpr double PSI_BYTES_US = 6.3e6, PSI_BYTES_US_ROWS2 = 5.3e6;
constexpr double SHAPE_MARGIN = 0.03;
constexpr int SHAPE_MIN_STAGES = 16;   // per SM
// Jobs of the B-operand pass per SM below which jobs are made shorter.
constexpr int PSI_JOBS_PER_SM = 8;
// Blocks of a scale or blocking launch that may find nothing to do (see
// prep_runs): about 1 ns each, against a few microseconds for another launch.
constexpr long long PREP_IDLE_BLOCKS = 4096;

}  // namespace

namespace laph {
// A schedule of the tensor-core path: tile width (complex columns), sites per
// block of the FP64 site reduction, drain interval of the tensor core's FP32
// accumulation, timeslices per chunk (-1: the wave model, -2: the largest
// chunk within the workspace cap; resolved when applied) and tile order.
struct Sched {
    int tile_cols, sum_sites, chunk_sites;
    long long per_chunk;
    int order;
    int rows2;           // 1: the row-doubled layout of the complex product (64 complex rows per tile); 2: CTA pairs
    int chunk_sites_b;   // drain interval of tiles without meson rows (0: chunk_sites)
};
}  // namespace laph

struct laph_plan {
    int mode = 0;
    unsigned flags = 0;
    int device = 0;
    int n_inst = 0;
    int total_ts = 0;
    std::vector<InstDev> h_inst;               // pointer fields unset
    std::vector<long long> phi_elems;          // complex64 entries of phi per instance
    std::vector<long long> outB_elems, outM_elems;
    std::vector<int32_t> momenta0;             // instance 0's momenta (the autotuner's accuracy probe)
    std::vector<int> h_T, h_ts_base;
    InstDev *d_inst = nullptr;
    float2 *d_phase = nullptr;
    TileDev *d_tiles = nullptr;
    long long n_tiles = 0;
    int *d_status = nullptr;
    int tile_rows = 0, tile_cols = 0, chunk_sites = 0, grid = 0;
    int chunk_sites_b = 0;   // drain interval of tiles without meson rows (0: chunk_sites)
    size_t out_bytes = 16;   // bytes per output entry: complex128, or complex64 with LAPH_PLAN_OUT_C64
    int rows2 = 0;                             // tensor-core path: the row-doubled layout
    int sum_sites = 0;                         // tensor-core path: sites per block of the FP64 reduction
    int max_staged = 0, max_P = 0;
    size_t ws_bytes = 0, off_maxbits = 0, off_counter = 0, ws_zero_bytes = 0;
    // tensor-core path: chunks of (instance, timeslice) units and their B-operand images
    laph::PsiUnit *d_units = nullptr;
    std::vector<laph::PsiUnit> h_units;
    int psi_group = laph::TC_PSI_GROUP;   // stages per job of the B-operand pass
    // laph_plan_execute_host: copy streams and per-chunk events, made on first use
    cudaStream_t h2d = nullptr, d2h = nullptr;
    // tensor-core path: the FP64 site reduction of chunk c runs on `side`
    // while the B-operand pass of chunk c+1 runs on the caller's stream;
    // ev_tc[c]: contraction c done, ev_red[c]: reduction c done
    cudaStream_t side = nullptr;
    std::vector<cudaEvent_t> ev_tc, ev_red;
    std::vector<cudaEvent_t> ev_in, ev_out;
    struct Chunk {
        int unit0, n_units;
        long long n_jobs;
        long long tile0, n_tiles;
        long long n_red;         // blocks of the FP64 reduction
        int n_split;             // trailing units cut into drains
        long long n_red_split;   // blocks of their reduction
    };
    std::vector<Chunk> chunks;
    // launches of the scale and blocking passes over the whole batch: consecutive units of similar size
    struct PrepRun {
        int unit0, n_units, nblk;   // nblk, elems: the most of any unit
        long long elems;
    };
    std::vector<PrepRun> prep;
    // where units are cut into drains: the same schedule with whole site blocks,
    // for laph_plan_set_chunk_sites.  Its tiles and units follow the cut ones in
    // d_tiles, d_units and h_units (tile0 and unit0 count from the start of
    // those), so that the call changes host values only: an execute in flight and
    // a captured graph keep the tables that their launches were made for.
    std::vector<Chunk> whole_chunks;
    long long whole_n_tiles = 0;
    double whole_flops = 0.0;
    // schedule of the tensor-core path: timeslices per chunk (0: chunks filled by
    // bytes) and tile order within a timeslice (0: column tiles outer, 1: row
    // tiles outer); with LAPH_PLAN_AUTOTUNE the candidates' timings
    long long sched_per_chunk = 0;
    int sched_order = 0;
    laph::Sched sched{};
    bool tuned = false;
    // LAPH_PLAN_AUTOTUNE: every candidate, its time (ms) and its probe error (-1: not probed)
    std::vector<laph::Sched> tune_cand;
    std::vector<long long> tune_pc;
    std::vector<float> tune_ms;
    std::vector<double> tune_err;
    size_t off_psi = 0, off_part = 0;
    // tensor-core path: flops the tensor pipe executes per execute (every MMA of
    // every tile: 2 x 128 rows x the tile's real columns x 48 real K entries
    // per stage x the split terms)
    double mma_flops = 0.0;
    // LAPH_PLAN_TIMING: ring of event pairs around the contraction launches
    static constexpr int RING = 256;
    // (contraction launches; pv_* for the B-operand launches of the tensor-core path)
    // (rd_*: the FP64 site reductions, in the slots of their contraction launches)
    std::vector<cudaEvent_t> ev_begin, ev_end, pv_begin, pv_end, rd_begin, rd_end;
    long long n_timed = 0, n_ptimed = 0;
};

extern "C" {

int64_t laph_triple_index(int i, int j, int k)
{
    if (!(0 <= i && i < j && j < k)) return -1;
    return laph::binom3(k) + laph::binom2(j) + i;
}

const char *laph_status_string(int status)
{
    switch (status) {
    case LAPH_OK: return "ok";
    case LAPH_ERR_ARG: return "invalid argument";
    case LAPH_ERR_CUDA: return g_last_cuda[0] ? g_last_cuda : "CUDA runtime error";
    case LAPH_ERR_WORKSPACE: return "workspace missing, too small or misaligned";
    case LAPH_ERR_UNSUPPORTED: return "mode or shape not supported on this device";
    case LAPH_ERR_TIMEOUT: return "a bounded device wait expired";
    case LAPH_ERR_DEVICE: return "a device-side check failed";
    default: return "unknown status";
    }
}

const char *laph_last_cuda_error(void) { return g_last_cuda; }

int laph_version(void) { return 1 * 10000 + 1 * 100 + 0; }

int laph_phase_table(int L, const int32_t *momenta, int n_mom, void *out, void *stream)
{
    if (L < 1 || L > MAX_L || n_mom < 1 || n_mom > MAX_P || !momenta || !out) return LAPH_ERR_ARG;
    if (((uintptr_t)out) % 16) return LAPH_ERR_ARG;
    for (int q = 0; q < 3 * n_mom; q++)
        if (momenta[q] > MAX_MOM || momenta[q] < -MAX_MOM) return LAPH_ERR_ARG;
    cudaStream_t s = (cudaStream_t)stream;
    int32_t *d_mom = nullptr;
    CK(cudaMallocAsync((void **)&d_mom, sizeof(int32_t) * 3 * n_mom, s));
    CK(cudaMemcpyAsync(d_mom, momenta, sizeof(int32_t) * 3 * n_mom, cudaMemcpyHostToDevice, s));
    cudaError_t e = laph::launch_phase_table(L, d_mom, n_mom, (double2 *)out, nullptr, s);
    cudaError_t e2 = cudaFreeAsync(d_mom, s);
    if (e != cudaSuccess) return cuda_fail(e, "phase_table");
    if (e2 != cudaSuccess) return cuda_fail(e2, "cudaFreeAsync");
    CK(cudaStreamSynchronize(s));  // the momenta live in caller memory only until return
    return LAPH_OK;
}

int laph_diquarks(const void *phi, int L, int T, int N, void *out, void *stream)
{
    if (!phi || !out || L < 1 || L > MAX_L || T < 1 || N < 2 || N > MAX_N) return LAPH_ERR_ARG;
    if ((long long)N > 3LL * L * L * L) return LAPH_ERR_ARG;
    if (((uintptr_t)phi) % 8 || ((uintptr_t)out) % 16) return LAPH_ERR_ARG;
    cudaError_t e = laph::launch_diquarks((const float2 *)phi, L, T, N, (float2 *)out, (cudaStream_t)stream);
    if (e == cudaErrorInvalidValue) return LAPH_ERR_UNSUPPORTED;
    if (e != cudaSuccess) return cuda_fail(e, "diquarks");
    return LAPH_OK;
}

int laph_baryon_dense(const void *packed, int T, int N, int n_mom, void *dense, void *stream)
{
    if (!packed || !dense || T < 1 || N < 3 || N > MAX_N || n_mom < 1 || n_mom > MAX_P) return LAPH_ERR_ARG;
    if (((uintptr_t)packed) % 16 || ((uintptr_t)dense) % 16) return LAPH_ERR_ARG;
    cudaError_t e = laph::launch_dense_fill((const double2 *)packed, T, N, n_mom, (double2 *)dense,
                                           (cudaStream_t)stream);
    if (e != cudaSuccess) return cuda_fail(e, "dense_fill");
    return LAPH_OK;
}

// ------------------------------------------------------------------ plans

static void free_plan(laph_plan *p)
{
    if (!p) return;
    cudaFree(p->d_inst);
    cudaFree(p->d_phase);
    cudaFree(p->d_units);
    for (cudaEvent_t e : p->ev_in) cudaEventDestroy(e);
    for (cudaEvent_t e : p->ev_out) cudaEventDestroy(e);
    if (p->h2d) cudaStreamDestroy(p->h2d);
    if (p->d2h) cudaStreamDestroy(p->d2h);
    for (cudaEvent_t e : p->ev_tc) cudaEventDestroy(e);
    for (cudaEvent_t e : p->ev_red) cudaEventDestroy(e);
    if (p->side) cudaStreamDestroy(p->side);
    cudaFree(p->d_tiles);
    cudaFree(p->d_status);
    for (cudaEvent_t e : p->ev_begin) cudaEventDestroy(e);
    for (cudaEvent_t e : p->ev_end) cudaEventDestroy(e);
    for (cudaEvent_t e : p->pv_begin) cudaEventDestroy(e);
    for (cudaEvent_t e : p->pv_end) cudaEventDestroy(e);
    for (cudaEvent_t e : p->rd_begin) cudaEventDestroy(e);
    for (cudaEvent_t e : p->rd_end) cudaEventDestroy(e);
    delete p;
}

static int autotune(laph_plan *p, const laph::Sched &def,
                    const std::function<cudaError_t(const laph::Sched &)> &apply);
static cudaError_t ensure_side(laph_plan *p);
static std::vector<laph_plan::PrepRun> prep_runs(const laph_plan *p, int unit0, int n_units);

static int tc_supported(int device)
{
    int major = 0, minor = 0;
    if (cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, device) != cudaSuccess) return 0;
    if (cudaDeviceGetAttribute(&minor, cudaDevAttrComputeCapabilityMinor, device) != cudaSuccess) return 0;
    return major == 10 && minor == 3;
}

int laph_plan_create(const laph_instance *inst, int n_inst, int mode, unsigned flags, laph_plan **plan_out)
{
    return laph_plan_create_opts(inst, n_inst, mode, flags, nullptr, plan_out);
}

int laph_plan_create_opts(const laph_instance *inst, int n_inst, int mode, unsigned flags, const laph_plan_options *opts,
                          laph_plan **plan_out)
{
    if (!inst || n_inst < 1 || !plan_out) return LAPH_ERR_ARG;
    const int opt_chunk = opts ? opts->chunk_sites : 0, opt_sum = opts ? opts->sum_sites : 0;
    const int opt_chunk_b = opts ? opts->chunk_sites_b : 0;
    if (opt_chunk < 0 || opt_chunk > (1 << 24) || opt_sum < 0 || opt_sum > (1 << 24)) return LAPH_ERR_ARG;
    if (opt_chunk_b < 0 || opt_chunk_b > (1 << 24)) return LAPH_ERR_ARG;
    if (opts && (opts->layout < 0 || opts->layout > 1)) return LAPH_ERR_ARG;
    if (opts && opts->tile_cols != 0 && !laph::tc_shape_supported(opts->tile_cols, opts->layout)) return LAPH_ERR_ARG;
    if (mode < 0 || mode >= LAPH_NUM_MODES) return LAPH_ERR_ARG;
    if ((flags & LAPH_PLAN_OUT_C64) && !is_tc_mode(mode)) return LAPH_ERR_UNSUPPORTED;
    const bool skipB = flags & LAPH_PLAN_SKIP_B, skipM = flags & LAPH_PLAN_SKIP_M;
    if (skipB && skipM) return LAPH_ERR_ARG;
    // several fields: triplets (skip M) or doublets (skip B), tensor-core modes only
    const bool fields = flags & LAPH_PLAN_FIELDS;
    const int kind = !fields ? laph::INST_BLOCKS : (skipM ? laph::INST_TRIPLETS : laph::INST_DOUBLETS);
    if (fields && !(skipB || skipM)) return LAPH_ERR_ARG;
    if (fields && !is_tc_mode(mode)) return LAPH_ERR_UNSUPPORTED;
    for (int n = 0; n < n_inst; n++) {
        const laph_instance &I = inst[n];
        if (I.L < 1 || I.L > MAX_L || I.T < 1 || I.N < 1 || I.N > MAX_N || I.n_mom < 1 || I.n_mom > MAX_P ||
            !I.momenta)
            return LAPH_ERR_ARG;
        if (!skipB && !fields && I.N < 3) return LAPH_ERR_ARG;
        // a second vector count only for doublets
        if (I.n_col < 0 || I.n_col > MAX_N || (I.n_col && I.n_col != I.N && kind != laph::INST_DOUBLETS))
            return LAPH_ERR_ARG;
        if ((long long)I.N > 3LL * I.L * I.L * I.L) return LAPH_ERR_ARG;
        for (int q = 0; q < 3 * I.n_mom; q++)
            if (I.momenta[q] > MAX_MOM || I.momenta[q] < -MAX_MOM) return LAPH_ERR_ARG;
    }
    int device = 0;
    CK(cudaGetDevice(&device));
    if (is_tc_mode(mode) && !tc_supported(device)) return LAPH_ERR_UNSUPPORTED;

    laph_plan *p = new (std::nothrow) laph_plan();
    if (!p) return LAPH_ERR_ARG;
    p->mode = mode;
    p->flags = flags;
    p->device = device;
    p->n_inst = n_inst;
    const bool tc = is_tc_mode(mode);
    p->tile_rows = tc ? laph::TC_TR : laph::SIMT_TR;
    p->tile_cols = tc ? laph::TC_TC : laph::SIMT_TC;
    p->chunk_sites = opt_chunk ? opt_chunk : (tc ? TC_DEFAULT_CHUNK : SIMT_DEFAULT_CHUNK);
    p->chunk_sites_b = opt_chunk_b;
    p->out_bytes = (flags & LAPH_PLAN_OUT_C64) ? sizeof(float2) : sizeof(double2);
    p->momenta0.assign(inst[0].momenta, inst[0].momenta + 3 * inst[0].n_mom);

    // ---- per-instance descriptors and phase tables
    long long phase_total = 0;
    std::vector<long long> phase_off(n_inst);
    int ts = 0;
    for (int n = 0; n < n_inst; n++) {
        const laph_instance &I = inst[n];
        InstDev d;
        memset(&d, 0, sizeof(d));
        d.L = I.L;
        d.T = I.T;
        d.N = I.N;
        d.P = I.n_mom;
        d.V = (long long)I.L * I.L * I.L;
        d.Vs = d.V + (d.V & 1);
        d.blk_off = -1;
        d.nblk = (int)((d.V + laph::TC_BS - 1) / laph::TC_BS);
        d.n_trip = laph::binom3(I.N);
        d.kind = kind;
        d.out_c64 = (flags & LAPH_PLAN_OUT_C64) ? 1 : 0;
        d.n_fields = kind == laph::INST_TRIPLETS ? 3 : (kind == laph::INST_DOUBLETS ? 2 : 1);
        d.blkv_off = -1;
        d.mes_rows = skipM ? 0 : I.N;
        d.pair_rows = skipB ? 0 : (kind == laph::INST_TRIPLETS ? I.N * I.N : (int)laph::binom2(I.N));
        d.rows = d.mes_rows + d.pair_rows;
        d.Nc = (kind == laph::INST_DOUBLETS && I.n_col) ? I.n_col : I.N;
        d.cols = d.Nc * I.n_mom;
        d.n_ct = (d.cols + laph::TC_TC - 1) / laph::TC_TC;
        d.n_st = (int)((3 * d.V + laph::TC_KSTAGE - 1) / laph::TC_KSTAGE);
        d.ts_base = ts;
        p->h_ts_base.push_back(ts);
        p->h_T.push_back(I.T);
        ts += I.T;
        p->h_inst.push_back(d);
        p->phi_elems.push_back((long long)I.T * std::max(I.N, d.Nc) * d.V * 3);   // the larger field
        p->outB_elems.push_back(skipB ? 0
                                      : (long long)I.T * I.n_mom *
                                            (kind == laph::INST_TRIPLETS ? (long long)I.N * I.N * I.N : d.n_trip));
        p->outM_elems.push_back(skipM ? 0 : (long long)I.T * I.n_mom * I.N * d.Nc);
        p->h_inst.back().n_outB = p->outB_elems.back() / I.T;
        p->h_inst.back().n_outM = p->outM_elems.back() / I.T;
        phase_off[n] = phase_total;
        phase_total += (long long)I.n_mom * d.Vs;
    }
    p->total_ts = ts;

    int rc = LAPH_OK;
    cudaError_t e;
#define PCK(call)                                 \
    do {                                          \
        e = (call);                               \
        if (e != cudaSuccess) {                   \
            rc = cuda_fail(e, #call);             \
            free_plan(p);                         \
            return rc;                            \
        }                                         \
    } while (0)

    PCK(cudaMalloc((void **)&p->d_phase, sizeof(float2) * phase_total));
    PCK(cudaMemset(p->d_phase, 0, sizeof(float2) * phase_total));
    {
        int32_t *d_mom = nullptr;
        PCK(cudaMalloc((void **)&d_mom, sizeof(int32_t) * 3 * MAX_P));
        for (int n = 0; n < n_inst && rc == LAPH_OK; n++) {
            const laph_instance &I = inst[n];
            e = cudaMemcpy(d_mom, I.momenta, sizeof(int32_t) * 3 * I.n_mom, cudaMemcpyHostToDevice);
            if (e == cudaSuccess) e = laph::launch_phase_table(I.L, d_mom, I.n_mom, nullptr, p->d_phase + phase_off[n], 0);
            if (e == cudaSuccess) e = cudaDeviceSynchronize();
            if (e != cudaSuccess) rc = cuda_fail(e, "phase table");
            p->h_inst[n].phase = p->d_phase + phase_off[n];
        }
        cudaFree(d_mom);
        if (rc != LAPH_OK) {
            free_plan(p);
            return rc;
        }
    }
    PCK(cudaMalloc((void **)&p->d_inst, sizeof(InstDev) * n_inst));
    PCK(cudaMemcpy(p->d_inst, p->h_inst.data(), sizeof(InstDev) * n_inst, cudaMemcpyHostToDevice));
    PCK(cudaMalloc((void **)&p->d_status, sizeof(int)));
    PCK(cudaMemset(p->d_status, 0, sizeof(int)));

    // ---- tile table: (instance, t, column tile, row tile), skipping column
    // tiles whose every k is <= the smallest j of a diquark-only row tile;
    // in the remaining tiles of such a row tile the leading columns with
    // k <= that j are skipped in steps of 8 (cskip).  The tensor-core path
    // processes the (instance, t) units in chunks whose B-operand images fit
    // the Psi buffer; the tiles of one column tile are consecutive, so the
    // CTAs that share a stage image run side by side.
    std::vector<TileDev> tiles;
    std::vector<laph::PsiUnit> units;
    std::vector<std::vector<TileDev>> ones(n_inst);
    std::vector<size_t> unit_bytes(n_inst);
    size_t psi_total = 0;
    // the (row tile, column tile) pairs of one timeslice of every instance for
    // tiles of TC complex columns
    auto build_tiles = [&](int TC, int rows2) {
        p->tile_cols = TC;
        p->rows2 = tc ? rows2 : 0;
        p->tile_rows = !tc ? laph::SIMT_TR : (rows2 == 1 ? laph::TC_TR_ROWS2 : laph::TC_TR);
        const int TR = p->tile_rows;
        const int skip_step = rows2 ? 16 : 8;   // column skips keep the UMMA N a multiple of 16
        p->max_staged = 0;
        for (int n = 0; n < n_inst; n++) {
            InstDev &d = p->h_inst[n];
            d.n_ct = (d.cols + TC - 1) / TC;
            std::vector<TileDev> &one = ones[n];
            one.clear();
            const bool trip = d.kind == laph::INST_TRIPLETS;
            // per row tile: the smallest j of a baryon row tile (rows of pairs i < j need only columns k > j; -1:
            // every column) and the contiguous range of vectors its rows use (for triplets: of phi_u, and
            // [w_lo, w_hi] of phi_v)
            struct RowTile {
                int jmin, v_lo, v_hi, w_lo, w_hi;
            };
            std::vector<RowTile> rts;
            for (int row0 = 0; row0 < d.rows; row0 += TR) {
                RowTile r{-1, d.N, -1, d.N, -1};
                for (int g = row0; g < std::min(row0 + TR, d.rows); g++) {
                    int i = g, j = g;
                    if (g >= d.mes_rows && trip) {
                        const int q = g - d.mes_rows;
                        i = q / d.N;
                        j = q - i * d.N;
                        r.w_lo = std::min(r.w_lo, j);
                        r.w_hi = std::max(r.w_hi, j);
                        j = i;
                    } else if (g >= d.mes_rows) {
                        laph::pair_of(g - d.mes_rows, i, j);
                        if (g == row0) r.jmin = j;
                    }
                    r.v_lo = std::min(r.v_lo, i);
                    r.v_hi = std::max(r.v_hi, j);
                }
                rts.push_back(r);
            }
            for (int col0 = 0; col0 < d.cols; col0 += TC) {
                const int nc = std::min(TC, d.cols - col0);
                const int kmin = col0 / d.P, kmax = (col0 + nc - 1) / d.P;
                for (int row0 = 0; row0 < d.rows; row0 += TR) {
                    const RowTile &rt = rts[row0 / TR];
                    const int jmin = rt.jmin, v_lo = rt.v_lo, v_hi = rt.v_hi, w_hi = rt.w_hi;
                    int w_lo = rt.w_lo;
                    if (jmin >= 0 && kmax <= jmin) continue;
                    const int nv = v_hi - v_lo + 1;
                    const int nw = trip ? w_hi - w_lo + 1 : 0;
                    if (!trip) w_lo = 0;
                    p->max_staged = std::max(p->max_staged, tc ? nv + nw : nv + (kmax - kmin + 1));
                    const long long psi_ct =
                        tc ? (long long)(col0 / TC) * d.n_st * laph::tc_stage_bytes(TC, rows2) : 0;
                    int cskip = 0;
                    if (tc && jmin >= 0) {
                        const int lead = std::max(0, std::min(nc, (jmin + 1) * d.P - col0));
                        cskip = (lead / skip_step) * skip_step;
                    }
                    one.push_back(TileDev{n, 0, row0, col0, v_lo, nv, w_lo, nw, kmin, kmax - kmin + 1, nc, cskip,
                                          psi_ct, 0, d.n_st, 0});
                }
            }
            p->max_P = std::max(p->max_P, d.P);
        }
    };
    // site blocks of the FP64 reduction (tensor-core path) and the workspace
    // bytes of one (instance, timeslice): its B-operand stage images and the
    // FP32 partials of all its site blocks
    auto set_sum = [&](int sum_sites) {
        p->sum_sites = tc ? sum_sites : 0;
        psi_total = 0;
        for (int n = 0; n < n_inst; n++) {
            InstDev &d = p->h_inst[n];
            d.sc_stages = tc ? std::max(1, std::min(d.n_st, sum_sites / laph::TC_BS)) : d.n_st;
            d.n_sc = (d.n_st + d.sc_stages - 1) / d.sc_stages;
            unit_bytes[n] = tc ? (size_t)d.n_ct * d.n_st * laph::tc_stage_bytes(p->tile_cols, p->rows2) +
                                     (size_t)d.n_sc * (size_t)(d.n_outB + d.n_outM) * sizeof(float2)
                               : 0;
            psi_total += (size_t)d.T * unit_bytes[n];
        }
    };
    int sms = 0;
    PCK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device));
    // persistent workers that claim tiles: CTAs, or pairs of CTAs
    auto workers = [&]() { return std::max(1, p->rows2 == 2 ? sms / 2 : sms); };
    // units per chunk: one instance -> the count (within the cap) that
    // leaves the fewest partly filled waves of persistent CTAs (want_largest:
    // the largest count within the cap); several instances -> chunks filled
    // in order up to an even share of the total (per_chunk 0)
    size_t psi_target = 0;
    auto chunking = [&](bool want_largest) -> long long {
        psi_target = 0;
        if (!tc) return 0;
        if (flags & LAPH_PLAN_CHUNK_PER_TIMESLICE) return 1;
        if (n_inst == 1) {
            const long long U = p->h_inst[0].T, tpu = (long long)ones[0].size() * p->h_inst[0].n_sc;
            const long long n_max =
                std::max(1LL, std::min(U, (long long)(PSI_CAP_BYTES / std::max<size_t>(unit_bytes[0], 1))));
            if (want_largest) return n_max;
            long long best = -1, best_rounds = 0;
            for (long long n = 1; n <= n_max; n++) {
                const long long full = U / n, rest = U % n;
                const long long w = workers(), rounds = full * ((n * tpu + w - 1) / w) + (rest * tpu + w - 1) / w;
                if (best < 0 || rounds <= best_rounds) {
                    best = n;
                    best_rounds = rounds;
                }
            }
            return best;
        }
        const long long n_chunks = (long long)((psi_total + PSI_CAP_BYTES - 1) / PSI_CAP_BYTES);
        psi_target = (psi_total + n_chunks - 1) / (size_t)std::max(1LL, n_chunks);
        return 0;
    };
    // instances in decreasing order of work per timeslice (stages x tiles),
    // so that the dynamically scheduled tiles of a chunk start with the longest
    std::vector<int> order(n_inst);
    auto make_order = [&]() {
        for (int n = 0; n < n_inst; n++) order[n] = n;
        if (tc)
            std::stable_sort(order.begin(), order.end(), [&](int a, int b) {
                return (long long)p->h_inst[a].n_st * (long long)ones[a].size() >
                       (long long)p->h_inst[b].n_st * (long long)ones[b].size();
            });
    };
    size_t psi_max = 0, part_max = 0;
    // tile, unit and chunk tables for a schedule (pc timeslices per chunk, or
    // chunks filled up to psi_target bytes when pc is 0).  On the tensor-core
    // path every (row tile, column tile) of a timeslice becomes one tile per
    // site block; order 0 runs them as (column tile, site block, row tile), so
    // that the tiles sharing one range of B stage images run side by side,
    // order 1 as (row tile, site block, column tile).
    // The last n_split units are cut into tiles of one drain interval (see
    // PsiUnit::split).
    auto drain_stages = [&]() { return std::max(1, p->chunk_sites * 3 / laph::TC_KSTAGE); };
    auto emit_tables = [&](long long pc, int tile_order, int n_split) {
        const int cs = drain_stages(), first_split = p->total_ts - n_split;
        tiles.clear();
        units.clear();
        p->chunks.clear();
        psi_max = part_max = 0;
        laph_plan::Chunk cur{};
        size_t cur_bytes = 0, cur_psi = 0;
        long long cur_part = 0;   // float2 entries of the chunk's partial buffer
        for (int n : order) {
            const InstDev &d = p->h_inst[n];
            const long long n_out = d.n_outB + d.n_outM;
            // the tiles of one timeslice: one per site block, or one per drain interval
            auto tiles_of = [&](bool split) {
                if (!tc) return ones[n];
                std::vector<TileDev> one;
                for (const TileDev &u : ones[n])
                    for (int sc = 0; sc < d.n_sc; sc++) {
                        const int b0 = sc * d.sc_stages, b1 = std::min(b0 + d.sc_stages, d.n_st);
                        const int step = split ? cs : b1 - b0, dps = split ? (d.sc_stages + cs - 1) / cs : 1;
                        for (int s0 = b0; s0 < b1; s0 += step) {
                            TileDev v = u;
                            v.s0 = s0;
                            v.nst = std::min(step, b1 - s0);
                            v.part_off = ((long long)sc * dps + (s0 - b0) / step) * n_out;
                            one.push_back(v);
                        }
                    }
                std::stable_sort(one.begin(), one.end(), [tile_order](const TileDev &x, const TileDev &y) {
                    const int xa = tile_order ? x.row0 : x.col0, ya = tile_order ? y.row0 : y.col0;
                    const int xb = tile_order ? x.col0 : x.row0, yb = tile_order ? y.col0 : y.row0;
                    if (xa != ya) return xa < ya;
                    if (x.s0 != y.s0) return x.s0 < y.s0;
                    return xb < yb;
                });
                return one;
            };
            std::vector<TileDev> one;
            int one_split = -1;
            for (int t = 0; t < d.T; t++) {
                const bool split = tc && (int)units.size() >= first_split;
                if (one_split != (split ? 1 : 0)) {
                    one = tiles_of(split);
                    one_split = split ? 1 : 0;
                }
                if (tc) {
                    const bool full = pc > 0 ? cur.n_units >= pc : cur_bytes + unit_bytes[n] > psi_target;
                    if (cur.n_units > 0 && full) {
                        p->chunks.push_back(cur);
                        psi_max = std::max(psi_max, cur_psi);
                        part_max = std::max(part_max, (size_t)cur_part * sizeof(float2));
                        cur = laph_plan::Chunk{};
                        cur.unit0 = (int)units.size();
                        cur.tile0 = (long long)tiles.size();
                        cur_bytes = cur_psi = 0;
                        cur_part = 0;
                    }
                    units.push_back(laph::PsiUnit{n, t, split ? cs : 0, 0, (long long)cur_psi, cur.n_jobs, cur_part,
                                                  split ? cur.n_red_split : cur.n_red});
                    cur.n_units++;
                    cur.n_jobs += (long long)d.n_ct * ((d.n_st + p->psi_group - 1) / p->psi_group);
                    if (split) {
                        cur.n_split++;
                        cur.n_red_split += (n_out + laph::TC_RED_BLOCK_SPLIT - 1) / laph::TC_RED_BLOCK_SPLIT;
                    } else {
                        cur.n_red += (n_out + laph::TC_RED_BLOCK - 1) / laph::TC_RED_BLOCK;
                    }
                }
                for (TileDev u : one) {
                    u.t = t;
                    if (tc) {
                        u.psi_off += (long long)cur_psi;
                        u.part_off += cur_part;
                    }
                    tiles.push_back(u);
                }
                if (tc) {
                    cur.n_tiles += (long long)one.size();
                    cur_bytes += unit_bytes[n];
                    cur_psi += (size_t)d.n_ct * d.n_st * laph::tc_stage_bytes(p->tile_cols, p->rows2);
                    cur_part += (long long)d.n_sc * (split ? (d.sc_stages + cs - 1) / cs : 1) * n_out;
                }
            }
        }
        if (tc && cur.n_units > 0) {
            p->chunks.push_back(cur);
            psi_max = std::max(psi_max, cur_psi);
            part_max = std::max(part_max, (size_t)cur_part * sizeof(float2));
        }
        p->n_tiles = (long long)tiles.size();
        p->mma_flops = 0.0;
        if (tc) {
            const int terms = (mode == LAPH_MODE_TC_F16X3 || mode == LAPH_MODE_TC_BF16X3) ? 3 : 1;
            for (const TileDev &u : tiles) {
                const int n_real = p->rows2 ? ((u.ncols + 15) & ~15) - u.cskip : 2 * ((u.ncols + 7) & ~7) - 2 * u.cskip;
                p->mma_flops += 2.0 * laph::TC_TR * (p->rows2 == 2 ? 2 : 1) * n_real * (2 * laph::TC_KSTAGE) * terms * u.nst;
            }
        }
        p->h_units = units;
        p->whole_chunks.clear();
        p->sched_per_chunk = pc;
        p->sched_order = tile_order;
    };
    // Time of the last chunk's contraction, in K stages, when its last n_split
    // units are cut into drains: whole tiles start in table order on the first
    // CTA that is free, the short tiles of the cut units then fill the chip
    // evenly.  A cut unit costs the traffic of its extra partials too (written and
    // read once each, SPLIT_BYTES_PER_STAGE bytes in the time of a stage).
    auto last_chunk_time = [&](int n_split, size_t *extra_bytes) -> double {
        const int cs = drain_stages();
        const laph_plan::Chunk &c = p->chunks.back();
        std::vector<long long> free_at(workers(), 0);   // a heap, earliest first
        const auto later = std::greater<long long>();
        long long end = 0, total = 0, longest = 0;
        *extra_bytes = 0;
        for (int u = 0; u < c.n_units; u++) {
            const InstDev &d = p->h_inst[units[c.unit0 + u].inst];
            const bool split = u >= c.n_units - n_split;
            const long long pairs = (long long)ones[units[c.unit0 + u].inst].size();
            for (int b0 = 0; b0 < d.n_st; b0 += d.sc_stages) {
                const int st = std::min(d.sc_stages, d.n_st - b0), nd = split ? (st + cs - 1) / cs : 1;
                total += pairs * (st + nd * TILE_STAGES);
                if (split) {
                    longest = std::max<long long>(longest, std::min(st, cs) + TILE_STAGES);
                    *extra_bytes += (size_t)(nd - 1) * (size_t)(d.n_outB + d.n_outM) * sizeof(float2);
                    continue;
                }
                for (long long q = 0; q < pairs; q++) {
                    std::pop_heap(free_at.begin(), free_at.end(), later);
                    free_at.back() += st + TILE_STAGES;
                    end = std::max(end, free_at.back());
                    std::push_heap(free_at.begin(), free_at.end(), later);
                }
            }
        }
        if (n_split) end = std::max(end, total / workers() + longest);
        return (double)end + 2.0 * (double)*extra_bytes / SPLIT_BYTES_PER_STAGE;
    };
    // The tables of a schedule, with as many trailing units of the last chunk
    // cut into drains as pays: none of a batch that fills the chip anyway, all
    // of a small one (one timeslice at L=24, N=32 is 18 tiles of up to 1024
    // stages on 152 SMs), a few where the last wave of tiles is thin.  Units
    // are cut only where both kinds of tile share one drain interval, within
    // SPLIT_MAX_BYTES of extra partials.
    std::function<void(long long, int)> emit = [&](long long pc, int tile_order) {
        p->psi_group = laph::TC_PSI_GROUP;
        emit_tables(pc, tile_order, 0);
        if (!tc || p->chunks.empty()) return;
        long long jobs = 0;
        for (const laph_plan::Chunk &c : p->chunks) jobs = std::max(jobs, c.n_jobs);
        // the B-operand pass walks a job's stages one after the other: shorter jobs until every SM has PSI_JOBS_PER_SM
        while (p->psi_group > 1 && jobs < (long long)PSI_JOBS_PER_SM * sms) {
            p->psi_group /= 2;
            jobs *= 2;
        }
        const laph_plan::Chunk last = p->chunks.back();
        int best = 0;
        if ((p->chunk_sites_b == 0 || p->chunk_sites_b == p->chunk_sites) && last.n_tiles <= (long long)SPLIT_MAX_WAVES * workers()) {
            size_t extra = 0;
            double best_t = last_chunk_time(0, &extra) * (1.0 - SPLIT_MARGIN);
            for (int u = 1; u <= last.n_units; u = u < 4 || u == last.n_units ? u + 1 : std::min(2 * u, last.n_units)) {
                const double t = last_chunk_time(u, &extra);
                if (extra > SPLIT_MAX_BYTES) break;
                if (t < best_t) {
                    best = u;
                    best_t = t;
                }
            }
        }
        if (p->psi_group != laph::TC_PSI_GROUP) emit_tables(pc, tile_order, 0);
        if (best == 0) return;
        const std::vector<TileDev> whole_tiles = tiles;
        const std::vector<laph::PsiUnit> whole_units = units;
        std::vector<laph_plan::Chunk> whole = p->chunks;
        const long long n_whole = p->n_tiles;
        const double flops = p->mma_flops;
        emit_tables(pc, tile_order, best);
        for (laph_plan::Chunk &c : whole) {
            c.unit0 += (int)units.size();
            c.tile0 += (long long)tiles.size();
        }
        tiles.insert(tiles.end(), whole_tiles.begin(), whole_tiles.end());
        units.insert(units.end(), whole_units.begin(), whole_units.end());
        p->h_units = units;
        p->whole_chunks = whole;
        p->whole_n_tiles = n_whole;
        p->whole_flops = flops;
    };
    // device copies of the tables and the workspace layout (tensor-core modes:
    // per-timeslice max |phi| bits and one tile counter per chunk, both cleared
    // by every execute, the site-blocked copies of phi, then the B-operand
    // images of one chunk)
    std::function<cudaError_t()> upload = [&]() -> cudaError_t {
        cudaError_t er = cudaSuccess;
        cudaFree(p->d_tiles);
        cudaFree(p->d_units);
        p->d_tiles = nullptr;
        p->d_units = nullptr;
        if (!tiles.empty()) {
            if ((er = cudaMalloc((void **)&p->d_tiles, sizeof(TileDev) * tiles.size())) != cudaSuccess) return er;
            er = cudaMemcpy(p->d_tiles, tiles.data(), sizeof(TileDev) * tiles.size(), cudaMemcpyHostToDevice);
            if (er != cudaSuccess) return er;
        }
        if (!units.empty()) {
            if ((er = cudaMalloc((void **)&p->d_units, sizeof(laph::PsiUnit) * units.size())) != cudaSuccess) return er;
            er = cudaMemcpy(p->d_units, units.data(), sizeof(laph::PsiUnit) * units.size(), cudaMemcpyHostToDevice);
            if (er != cudaSuccess) return er;
        }
        if (tc) {
            p->grid = sms;
            p->off_maxbits = 0;
            p->off_counter = ((sizeof(unsigned) * p->total_ts + 255) / 256) * 256;
            size_t off = p->off_counter + ((sizeof(unsigned) * p->chunks.size() + 255) / 256) * 256;
            p->ws_zero_bytes = off;
            for (int n = 0; n < n_inst; n++) {
                InstDev &d = p->h_inst[n];
                const size_t blk_bytes = (((size_t)d.T * d.nblk * d.N * laph::TC_SLOT * sizeof(float2) + 255) / 256) * 256;
                d.blk_off = (long long)off;
                off += blk_bytes;
                if (d.kind == laph::INST_TRIPLETS) {
                    d.blkv_off = (long long)off;
                    off += blk_bytes;
                }
            }
            p->off_psi = off;
            off += ((psi_max + 255) / 256) * 256;
            p->off_part = off;
            off += ((part_max + 255) / 256) * 256;
            p->ws_bytes = off;
            er = cudaMemcpy(p->d_inst, p->h_inst.data(), sizeof(InstDev) * n_inst, cudaMemcpyHostToDevice);
        } else {
            p->grid = 0;
            p->ws_bytes = 0;
        }
        return er;
    };
    // a whole schedule: tile width, site block, drain interval, chunking
    // (-1: the wave model, -2: the largest chunk within the cap) and tile order
    std::function<cudaError_t(const laph::Sched &)> apply = [&](const laph::Sched &c) -> cudaError_t {
        build_tiles(tc ? c.tile_cols : laph::SIMT_TC, c.rows2);
        set_sum(c.sum_sites);
        make_order();
        p->chunk_sites = c.chunk_sites;
        p->chunk_sites_b = c.chunk_sites_b;
        const long long model = chunking(c.per_chunk == -2);   // also sets psi_target for several instances
        const long long pc = c.per_chunk >= 0 ? c.per_chunk : model;
        emit(pc, c.order);
        if (tc) p->prep = prep_runs(p, 0, p->total_ts);
        p->sched = c;
        return upload();
    };
    const int opt_cols = opts ? opts->tile_cols : 0, opt_layout = opts ? opts->layout : 0;
    laph::Sched def{opt_cols ? opt_cols : (opt_layout ? 176 : laph::TC_TC),
                    opt_sum ? opt_sum : TC_DEFAULT_SUM, p->chunk_sites, -1, 0, opt_layout, opt_chunk_b};
    // Estimated time (us) of an execute's B-operand pass and contraction with
    // tiles of nc columns in layout r2.  A stage of a tile costs STAGE_US +
    // STAGE_US_COL per accumulator column (both layouts); whole tiles on the
    // first free CTA where there are few waves of them, else (or where the last
    // wave can be cut into drains) spread evenly.  A stage ring of fewer than
    // four buffers costs RING_COST.  `cut`: as if a thin last wave could always be
    // cut; `real`: as this plan is, whose tiles stay whole where it has two drain
    // intervals, one timeslice per chunk or too many extra partials.
    struct ShapeUs {
        double cut, real;
    };
    const bool per_ts = (flags & LAPH_PLAN_CHUNK_PER_TIMESLICE) && p->total_ts > 1;
    auto shape_us = [&](int nc, int r2) -> ShapeUs {
        build_tiles(nc, r2);
        set_sum(def.sum_sites);
        const int ring = laph::tc_ring_depth(p->max_staged, nc, r2);
        if (p->max_staged > laph::TC_MAX_STAGED || !ring) return {1e300, 1e300};
        auto stage_us = [&](const TileDev &u) {
            const int n_real = r2 ? ((u.ncols + 15) & ~15) - u.cskip : 2 * ((u.ncols + 7) & ~7) - 2 * u.cskip;
            return r2 == 2 ? PAIR_STAGE_US + PAIR_STAGE_US_COL * n_real : STAGE_US + STAGE_US_COL * n_real;
        };
        const int cs = drain_stages(), w = workers();
        // the contraction of instances [n0, n1), all their timeslices or one of each
        auto contraction = [&](int n0, int n1, bool one_t) -> ShapeUs {
            double total = 0.0, extra = 0.0;   // extra: bytes of the partials when every unit is cut
            long long n_tiles = 0, n_units = 0;
            int st_max = 1;
            for (int n = n0; n < n1; n++) {
                const InstDev &d = p->h_inst[n];
                const int T = one_t ? 1 : d.T;
                for (const TileDev &u : ones[n]) total += stage_us(u) * d.n_st * T;
                n_tiles += (long long)ones[n].size() * d.n_sc * T;
                n_units += T;
                for (int b0 = 0; b0 < d.n_st; b0 += d.sc_stages)
                    extra += (double)T * ((std::min(d.sc_stages, d.n_st - b0) + cs - 1) / cs - 1) *
                             (double)(d.n_outB + d.n_outM) * sizeof(float2);
                st_max = std::max(st_max, d.sc_stages);
            }
            const double even = total / w;
            if (n_tiles > (long long)SPLIT_MAX_WAVES * w) return {even, even};
            std::vector<double> free_at(w, 0.0);
            const auto later = std::greater<double>();
            double end = 0.0;
            for (int n = n0; n < n1; n++) {
                const InstDev &d = p->h_inst[n];
                for (int t = 0; t < (one_t ? 1 : d.T); t++)
                    for (const TileDev &u : ones[n])
                        for (int b0 = 0; b0 < d.n_st; b0 += d.sc_stages) {
                            std::pop_heap(free_at.begin(), free_at.end(), later);
                            free_at.back() += stage_us(u) * (std::min(d.sc_stages, d.n_st - b0) + TILE_STAGES);
                            end = std::max(end, free_at.back());
                            std::push_heap(free_at.begin(), free_at.end(), later);
                        }
            }
            // two waves or more: one wave of tiles is cut; fewer: every unit
            const bool many = n_tiles >= 2 * w;
            const double us = std::min(end, (many ? 1.04 : 1.0 + (double)TILE_STAGES / std::min(cs, st_max)) * even);
            if (many) extra *= std::min(1.0, (double)((w * n_units + n_tiles - 1) / n_tiles) / (double)n_units);
            const bool whole = per_ts || (def.chunk_sites_b && def.chunk_sites_b != def.chunk_sites) ||
                               extra > (double)SPLIT_MAX_BYTES;
            return {us, whole ? end : us};
        };
        ShapeUs us = contraction(0, n_inst, false);
        double bytes = 0.0;
        if (per_ts) us.real = 0.0;
        for (int n = 0; n < n_inst; n++) {
            const InstDev &d = p->h_inst[n];
            if (per_ts) us.real += d.T * contraction(n, n + 1, true).real;
            bytes += (double)d.T * ((double)d.n_ct * d.n_st * laph::tc_stage_bytes(nc, r2) + 24.0 * d.Nc * d.V);
        }
        const double f = ring < 4 ? RING_COST : 1.0, psi = bytes / (r2 ? PSI_BYTES_US_ROWS2 : PSI_BYTES_US);
        return {us.cut * f + psi, us.real * f + psi};
    };
    // The default shape is 104 columns of layout 0, or 96 where the row vectors
    // a tile stages would leave its ring shallower than four buffers.  A plan
    // with enough work takes another shape where the estimate is better by
    // SHAPE_MARGIN: layout 1 has half the B-operand bytes and 64-row tiles
    // (meson rows alone fill half of a 128-row tile), a narrower tile of layout 0
    // may cover the columns in as many tiles, CTA pairs keep a stage ring of four
    // buffers with many row vectors.  Every shape adds the same products over the
    // same drains; within a k-step the layouts hand the products of imaginary parts
    // over in exchanged slots, which changes no bit of the tensor core's sum (tested
    // for all shapes).  Only with chunk_sites_b does a shape matter: it decides which
    // rows share a tile with meson rows.
    if (tc && !opt_cols && !opt_layout) {
        const ShapeUs us104 = shape_us(def.tile_cols, 0);
        if (laph::tc_ring_depth(p->max_staged, def.tile_cols, 0) < 4 &&
            laph::tc_ring_depth(p->max_staged, 96, 0) > laph::tc_ring_depth(p->max_staged, def.tile_cols, 0))
            def.tile_cols = 96;
        long long stages = 0;
        for (int n = 0; n < n_inst; n++)
            stages += (long long)ones[n].size() * p->h_inst[n].n_st * p->h_inst[n].T;
        // (a plan whose default tiles cannot stage their row vectors stays refused)
        if (us104.cut < 1e300 && stages >= (long long)SHAPE_MIN_STAGES * sms) {
            const std::pair<int, int> shapes[] = {{def.tile_cols, 0}, {96, 0},  {80, 0},  {64, 0},
                                                  {208, 1},           {176, 1}, {128, 1}, {laph::TC_PAIR_COLS, 2}};
            constexpr int NSH = sizeof(shapes) / sizeof(shapes[0]);
            ShapeUs us[NSH];
            for (int k = 0; k < NSH; k++)
                us[k] = k == 0 && def.tile_cols != 96 ? us104 : shape_us(shapes[k].first, shapes[k].second);
            // the lowest estimate, if better than that of shape `best` by the margin
            auto lowest = [&](int best, double ShapeUs::*e) {
                double limit = us[best].*e * (1.0 - SHAPE_MARGIN);
                for (int k = 0; k < NSH; k++)
                    if (us[k].*e < limit) {
                        best = k;
                        limit = us[k].*e;
                    }
                return best;
            };
            // where the tiles stay whole, another shape than that of a plan whose last wave can be cut only if it is
            // better by the margin again (L=18, N=40, 27 momenta, one timeslice, chunk_sites_b 192: 626 us with 35 tiles
            // of 104 columns, 560 with 56 of 128 columns in layout 1; L=24, T=8, one timeslice per chunk 6850, 6320)
            const std::pair<int, int> sh = shapes[lowest(lowest(0, &ShapeUs::cut), &ShapeUs::real)];
            def.tile_cols = sh.first;
            def.rows2 = sh.second;
        }
    }
    PCK(apply(def));
    if (tc && p->max_staged > laph::TC_MAX_STAGED) {
        free_plan(p);
        return LAPH_ERR_UNSUPPORTED;
    }
    if (tc && (flags & LAPH_PLAN_AUTOTUNE)) {
        // candidates, each timed on seeded synthetic inputs of the plan's
        // shapes (autotune_time); a coordinate search over tile width x tile
        // order x chunking, then the site-block size, then the drain interval
        // (kept only within the accuracy limit of the probe)
        const int rc_t = autotune(p, def, apply);
        if (rc_t != LAPH_OK) {
            free_plan(p);
            return rc_t;
        }
        p->tuned = true;
    }
    if (tc) PCK(ensure_side(p));
    if (flags & LAPH_PLAN_TIMING) {
        p->ev_begin.resize(laph_plan::RING, nullptr);
        p->ev_end.resize(laph_plan::RING, nullptr);
        p->pv_begin.resize(laph_plan::RING, nullptr);
        p->pv_end.resize(laph_plan::RING, nullptr);
        p->rd_begin.resize(laph_plan::RING, nullptr);
        p->rd_end.resize(laph_plan::RING, nullptr);
        for (int r = 0; r < laph_plan::RING; r++) {
            PCK(cudaEventCreate(&p->ev_begin[r]));
            PCK(cudaEventCreate(&p->ev_end[r]));
            PCK(cudaEventCreate(&p->pv_begin[r]));
            PCK(cudaEventCreate(&p->pv_end[r]));
            PCK(cudaEventCreate(&p->rd_begin[r]));
            PCK(cudaEventCreate(&p->rd_end[r]));
        }
    }
#undef PCK
    *plan_out = p;
    return LAPH_OK;
}

int laph_plan_workspace_size(const laph_plan *plan, size_t *bytes)
{
    if (!plan || !bytes) return LAPH_ERR_ARG;
    *bytes = plan->ws_bytes;
    return LAPH_OK;
}

int laph_plan_describe(const laph_plan *plan, int *mode, int *tile_rows, int *tile_cols, int *chunk_sites, int *grid,
                       int64_t *n_tiles)
{
    if (!plan) return LAPH_ERR_ARG;
    if (mode) *mode = plan->mode;
    if (tile_rows) *tile_rows = plan->tile_rows;
    if (tile_cols) *tile_cols = plan->tile_cols;
    if (chunk_sites) *chunk_sites = plan->chunk_sites;
    if (grid) *grid = plan->grid;
    if (n_tiles) *n_tiles = plan->n_tiles;
    return LAPH_OK;
}

int laph_plan_sum_sites(const laph_plan *plan, int *sum_sites, int *max_site_blocks)
{
    if (!plan) return LAPH_ERR_ARG;
    int mx = 0;
    for (const InstDev &d : plan->h_inst) mx = std::max(mx, is_tc_mode(plan->mode) ? d.n_sc : 0);
    if (sum_sites) *sum_sites = plan->sum_sites;
    if (max_site_blocks) *max_site_blocks = mx;
    return LAPH_OK;
}

// Where units are cut into drains of one interval, another interval takes the
// cut back: the tables of whole site blocks, made with the plan, take over.  The
// workspace layout stays; whole site blocks need a part of it.
int laph_plan_set_chunk_sites(laph_plan *plan, int chunk_sites)
{
    if (!plan || chunk_sites < 0 || chunk_sites > (1 << 24)) return LAPH_ERR_ARG;
    const bool tc = is_tc_mode(plan->mode);
    if (chunk_sites == 0) chunk_sites = tc ? TC_DEFAULT_CHUNK : SIMT_DEFAULT_CHUNK;
    if (chunk_sites != plan->chunk_sites && !plan->whole_chunks.empty()) {
        plan->chunks.swap(plan->whole_chunks);
        plan->n_tiles = plan->whole_n_tiles;
        plan->mma_flops = plan->whole_flops;
        plan->whole_chunks.clear();
    }
    plan->chunk_sites = chunk_sites;
    return LAPH_OK;
}

static laph::TcConfig tc_config(const laph_plan *p)
{
    laph::TcConfig cfg;
    cfg.elem = (p->mode == LAPH_MODE_TC_BF16X3 || p->mode == LAPH_MODE_TC_BF16) ? 1 : 0;
    cfg.terms = (p->mode == LAPH_MODE_TC_F16X3 || p->mode == LAPH_MODE_TC_BF16X3) ? 3 : 1;
    cfg.chunk_sites = p->chunk_sites;
    cfg.chunk_sites_b = p->chunk_sites_b;
    cfg.psi_bytes = p->off_part - p->off_psi;
    cfg.ncols = p->tile_cols;
    cfg.rows2 = p->rows2;
    cfg.grid = p->grid;
    cfg.max_staged = p->max_staged;
    cfg.debug_stall = (p->flags & LAPH_PLAN_DEBUG_STALL) ? 1 : 0;
    return cfg;
}

// The side stream (of a plan of several chunks) and one pair of events per chunk (made outside any stream
// capture: at plan creation and before each autotuning candidate).
static cudaError_t ensure_side(laph_plan *p)
{
    cudaError_t e;
    if (p->chunks.size() > 1 && !p->side &&
        (e = cudaStreamCreateWithFlags(&p->side, cudaStreamNonBlocking)) != cudaSuccess)
        return e;
    while (p->ev_tc.size() < p->chunks.size()) {
        cudaEvent_t a = nullptr, b = nullptr;
        if ((e = cudaEventCreateWithFlags(&a, cudaEventDisableTiming)) != cudaSuccess) return e;
        if ((e = cudaEventCreateWithFlags(&b, cudaEventDisableTiming)) != cudaSuccess) {
            cudaEventDestroy(a);
            return e;
        }
        p->ev_tc.push_back(a);
        p->ev_red.push_back(b);
    }
    return cudaSuccess;
}

// B-operand pass, contraction and FP64 site reduction of chunk ci (tensor-core
// path), with the timing events of LAPH_PLAN_TIMING around each launch.  The
// reduction runs on the plan's side stream after the contraction (event
// ev_tc[ci]), the last chunk's on `s`; the contraction of chunk ci waits for
// the reduction of chunk ci - 1, which reads the same partial buffer (event
// ev_red[ci - 1]), so that everything is back in `s` at the end.
static int launch_tc_chunk(laph_plan *p, char *ws, size_t ci, const laph::TcConfig &cfg, cudaStream_t s)
{
    if ((p->chunks.size() > 1 && !p->side) || p->ev_tc.size() < p->chunks.size()) return LAPH_ERR_ARG;
    cudaError_t e;
    const bool timing = !p->ev_begin.empty();
    unsigned *maxbits = (unsigned *)(ws + p->off_maxbits);
    uint8_t *psi = (uint8_t *)(ws + p->off_psi);
    unsigned *counters = (unsigned *)(ws + p->off_counter);
    float2 *part = (float2 *)(ws + p->off_part);
    const laph_plan::Chunk &c = p->chunks[ci];
    const int ps = (int)(p->n_ptimed % laph_plan::RING), cs = (int)(p->n_timed % laph_plan::RING);
    if (timing) CK(cudaEventRecord(p->pv_begin[ps], s));
    e = laph::launch_psi(p->d_inst, p->d_units + c.unit0, c.n_units, c.n_jobs, p->psi_group, maxbits, cfg.elem, cfg.ncols, cfg.rows2,
                         psi, s);
    if (e != cudaSuccess) return cuda_fail(e, "psi");
    if (timing) {
        CK(cudaEventRecord(p->pv_end[ps], s));
        p->n_ptimed++;
    }
    if (ci > 0) CK(cudaStreamWaitEvent(s, p->ev_red[ci - 1], 0));
    if (timing) CK(cudaEventRecord(p->ev_begin[cs], s));
    e = laph::launch_tc(p->d_inst, p->d_tiles + c.tile0, c.n_tiles, maxbits, psi, part, counters + ci, cfg,
                        p->d_status, s);
    if (e == cudaErrorNotSupported) return LAPH_ERR_UNSUPPORTED;
    if (e != cudaSuccess) return cuda_fail(e, "tc contraction");
    if (timing) {
        CK(cudaEventRecord(p->ev_end[cs], s));
        p->n_timed++;
    }
    // the last chunk has nothing left to run beside its reduction
    const cudaStream_t rs = ci + 1 < p->chunks.size() ? p->side : s;
    if (rs != s) {
        CK(cudaEventRecord(p->ev_tc[ci], s));
        CK(cudaStreamWaitEvent(rs, p->ev_tc[ci], 0));
    }
    if (timing) CK(cudaEventRecord(p->rd_begin[cs], rs));
    e = laph::launch_reduce(p->d_inst, p->d_units + c.unit0, c.n_units, c.n_split, c.n_red, c.n_red_split, maxbits, part,
                            rs);
    if (e != cudaSuccess) return cuda_fail(e, "site reduction");
    if (timing) CK(cudaEventRecord(p->rd_end[cs], rs));
    CK(cudaEventRecord(p->ev_red[ci], rs));
    return LAPH_OK;
}

// The units [unit0, unit0 + n_units) in runs that share a scale and a blocking
// launch.  A launch has as many blocks per unit as the largest of its units
// needs, so a run ends where the blocks without work would outnumber the others
// (and PREP_IDLE_BLOCKS): units come in decreasing order of work, so these are few
// runs.  One launch for L=4 timeslices beside a single L=48 one is 13,824 blocks
// for each of them, 8 of which have work (5000 of them, N=8: 36.5 -> 1.0 ms an execute; one L=24 and
// 300 L=8 timeslices, N=16: 578 -> 302 us).
static std::vector<laph_plan::PrepRun> prep_runs(const laph_plan *p, int unit0, int n_units)
{
    std::vector<laph_plan::PrepRun> runs;
    long long need = 0;
    for (int u = unit0; u < unit0 + n_units; u++) {
        const int n = p->h_units[u].inst, nb = p->h_inst[n].nblk;
        const long long elems = p->phi_elems[n] / p->h_T[n];
        if (!runs.empty()) {
            laph_plan::PrepRun &r = runs.back();
            const int most = std::max(r.nblk, nb);
            const long long all = (long long)most * (r.n_units + 1);
            if (all - (need + nb) <= std::max(need + nb, PREP_IDLE_BLOCKS)) {
                need += nb;
                r.n_units++;
                r.nblk = most;
                r.elems = std::max(r.elems, elems);
                continue;
            }
        }
        need = nb;
        runs.push_back({u, 1, nb, elems});
    }
    return runs;
}

// Scale and site-blocked copy of the units of these runs.
static int launch_prep(laph_plan *p, char *ws, const std::vector<laph_plan::PrepRun> &runs, cudaStream_t s)
{
    unsigned *maxbits = (unsigned *)(ws + p->off_maxbits);
    const InstDev &d = p->h_inst[0];   // the kind of instance is the plan's
    for (const laph_plan::PrepRun &r : runs) {
        const laph::PsiUnit *units = p->d_units + r.unit0;
        cudaError_t e = laph::launch_scale_max(p->d_inst, units, r.n_units, d.n_fields, r.elems, maxbits, s);
        if (e != cudaSuccess) return cuda_fail(e, "scale_max");
        e = laph::launch_blockify(p->d_inst, units, r.n_units, r.nblk, d.kind == laph::INST_TRIPLETS, maxbits, s);
        if (e != cudaSuccess) return cuda_fail(e, "blockify");
    }
    return LAPH_OK;
}

// cleared: the pointer upload has cleared the counters and scales already
static int launch_batch(laph_plan *p, void *workspace, cudaStream_t s, bool cleared = false)
{
    cudaError_t e;
    const bool timing = !p->ev_begin.empty();
    if (is_tc_mode(p->mode)) {
        if (!workspace || ((uintptr_t)workspace) % 256) return LAPH_ERR_WORKSPACE;
        char *ws = (char *)workspace;
        if (!cleared) CK(cudaMemsetAsync(ws, 0, p->ws_zero_bytes, s));
        const int rc = launch_prep(p, ws, p->prep, s);
        if (rc != LAPH_OK) return rc;
        const laph::TcConfig cfg = tc_config(p);
        for (size_t ci = 0; ci < p->chunks.size(); ci++) {
            const int rc = launch_tc_chunk(p, ws, ci, cfg, s);
            if (rc != LAPH_OK) return rc;
        }
    } else {
        laph::SimtConfig cfg;
        cfg.chunk_sites = p->chunk_sites;
        const int cs = (int)(p->n_timed % laph_plan::RING);
        if (timing) CK(cudaEventRecord(p->ev_begin[cs], s));
        e = laph::launch_simt(p->d_inst, p->d_tiles, p->n_tiles, cfg, p->d_status, s);
        if (e != cudaSuccess) return cuda_fail(e, "simt contraction");
        if (timing) {
            CK(cudaEventRecord(p->ev_end[cs], s));
            p->n_timed++;
        }
    }
    return LAPH_OK;
}

static int ring_times(const std::vector<cudaEvent_t> &b, const std::vector<cudaEvent_t> &e, long long count, int n,
                      float *ms)
{
    if (!ms || n < 1 || b.empty()) return LAPH_ERR_ARG;
    if (n > laph_plan::RING || n > count) return LAPH_ERR_ARG;
    for (int q = 0; q < n; q++) {
        const int slot = (int)((count - n + q) % laph_plan::RING);
        CK(cudaEventSynchronize(e[slot]));
        CK(cudaEventElapsedTime(&ms[q], b[slot], e[slot]));
    }
    return LAPH_OK;
}

// The autotuner.  Every candidate schedule is applied to the plan and timed
// on seeded synthetic inputs of the plan's shapes (pseudo-random entries in
// [-1, 1), outputs and a workspace allocated for the duration): one warm-up
// execute and one timed execute on an internal stream.  The search is by
// coordinates: tile shape (layout 0 at 104, 96, 80 and 64 columns, layout 1 at
// 176, 192, 208 and 128 columns) x tile order x chunking (the wave model, the
// largest chunk within the cap), then the site-block size of the
// FP64 reduction (half and twice the default), then the drain interval of the
// tensor core's accumulation (half and one and a half times the default; the
// separate interval of tiles without meson rows is left to the caller: at the
// 64-timeslice L=32 workload 1.5 times the default gained under 1% and raised
// the baryon error from 2.8e-6 to 4.1e-6).  A drain interval is kept only if
// the error of (instance 0, timeslice 0) against the FP32 CUDA-core path (its
// accuracy probe) stays within TUNE_ERR_LIMIT or within the default's own
// probe error; plans of several fields have no FP32 path and keep the default
// interval.  Finally the three fastest accepted schedules and the default one
// are timed twice more, each keeps its lowest time, and the fastest is applied
// if it beats the default by more than TUNE_MARGIN (else the default is).
constexpr double TUNE_ERR_LIMIT = 5e-6;   // half the 1e-5 bound of the split-precision modes
// A tuned schedule replaces the default one only if it is faster by more than
// this fraction.  Near-ties are timing noise (at the 64-timeslice L=32
// workload layout 1 with 208 columns and layout 0 with 104 came within 0.3% of
// each other, and the choice flipped from box to box), and the default's
// smaller chunks overlap the copies of laph_plan_execute_host better (there
// layout 1's chunks of 25 timeslices left 4-5 ms more of copying exposed per
// execute than the default's 10).
constexpr double TUNE_MARGIN = 0.01;

struct TuneState {
    std::vector<void *> phi, ob, om;
    cudaStream_t st = nullptr;
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    laph_plan *ref = nullptr;                // FP32 plan of instance 0, timeslice 0
    void *refB = nullptr, *refM = nullptr;
    double *acc = nullptr;                   // device: difference and reference norms
};

static int tune_time(laph_plan *p, TuneState &ts, float *ms)
{
    const bool needB = !(p->flags & LAPH_PLAN_SKIP_B), needM = !(p->flags & LAPH_PLAN_SKIP_M);
    const bool fields = p->flags & LAPH_PLAN_FIELDS;
    void *ws = nullptr;
    cudaError_t e;
    int rc = LAPH_OK;
    if ((e = ensure_side(p)) != cudaSuccess) return cuda_fail(e, "ensure_side");
    if ((e = cudaMalloc(&ws, std::max<size_t>(p->ws_bytes, 256))) != cudaSuccess) return cuda_fail(e, "cudaMalloc");
    if (fields) {
        // one field buffer serves every field of an instance (timing and accuracy probe only)
        const int nf = (p->flags & LAPH_PLAN_SKIP_M) ? 3 : 2;
        std::vector<const void *> f;
        std::vector<void *> o;
        for (int n = 0; n < p->n_inst; n++) {
            for (int k = 0; k < nf; k++) f.push_back(ts.phi[n]);
            o.push_back(nf == 3 ? ts.ob[n] : ts.om[n]);
        }
        e = laph::launch_set_pointers(p->d_inst, 0, p->n_inst, nullptr, nf == 3 ? o.data() : nullptr,
                                      nf == 3 ? nullptr : o.data(), ws, ts.st, f.data(), nf);
    } else {
        e = laph::launch_set_pointers(p->d_inst, 0, p->n_inst, ts.phi.data(), needB ? ts.ob.data() : nullptr,
                                      needM ? ts.om.data() : nullptr, ws, ts.st);
    }
    if (e != cudaSuccess) rc = cuda_fail(e, "set_pointers");
    if (rc == LAPH_OK) rc = launch_batch(p, ws, ts.st);
    if (rc == LAPH_OK && (e = cudaEventRecord(ts.e0, ts.st)) != cudaSuccess) rc = cuda_fail(e, "event");
    if (rc == LAPH_OK) rc = launch_batch(p, ws, ts.st);
    if (rc == LAPH_OK && (e = cudaEventRecord(ts.e1, ts.st)) != cudaSuccess) rc = cuda_fail(e, "event");
    if (rc == LAPH_OK && (e = cudaEventSynchronize(ts.e1)) != cudaSuccess) rc = cuda_fail(e, "event");
    if (rc == LAPH_OK && (e = cudaEventElapsedTime(ms, ts.e0, ts.e1)) != cudaSuccess) rc = cuda_fail(e, "event");
    cudaStreamSynchronize(ts.st);
    cudaFree(ws);
    return rc;
}

// Relative Frobenius error of (instance 0, timeslice 0) of the last timed
// execute against the FP32 path (the larger of the B and M errors).
static int tune_probe(laph_plan *p, TuneState &ts, double *err)
{
    cudaError_t e;
    const bool needB = !(p->flags & LAPH_PLAN_SKIP_B), needM = !(p->flags & LAPH_PLAN_SKIP_M);
    const InstDev &d = p->h_inst[0];
    if (!ts.ref) {
        laph_instance one{d.L, 1, d.N, d.P, p->momenta0.data(), 0};
        laph_plan_options o{};
        int rc = laph_plan_create_opts(&one, 1, LAPH_MODE_FP32_SIMT, p->flags & (LAPH_PLAN_SKIP_B | LAPH_PLAN_SKIP_M),
                                       &o, &ts.ref);
        if (rc != LAPH_OK) return rc;
        if (needB && (e = cudaMalloc(&ts.refB, std::max<long long>(d.n_outB, 1) * sizeof(double2))) != cudaSuccess)
            return cuda_fail(e, "cudaMalloc");
        if (needM && (e = cudaMalloc(&ts.refM, std::max<long long>(d.n_outM, 1) * sizeof(double2))) != cudaSuccess)
            return cuda_fail(e, "cudaMalloc");
        if ((e = cudaMalloc((void **)&ts.acc, 4 * sizeof(double))) != cudaSuccess) return cuda_fail(e, "cudaMalloc");
        const void *ph[1] = {ts.phi[0]};
        void *rb[1] = {ts.refB}, *rm[1] = {ts.refM};
        rc = laph_plan_execute(ts.ref, ph, needB ? rb : nullptr, needM ? rm : nullptr, nullptr, ts.st);
        if (rc != LAPH_OK) return rc;
    }
    if ((e = cudaMemsetAsync(ts.acc, 0, 4 * sizeof(double), ts.st)) != cudaSuccess) return cuda_fail(e, "memset");
    const bool c64 = p->out_bytes == sizeof(float2);
    if (needB && (e = laph::launch_diff_norms(ts.ob[0], c64, (const double2 *)ts.refB, d.n_outB, ts.acc, ts.st)) !=
                     cudaSuccess)
        return cuda_fail(e, "diff_norms");
    if (needM && (e = laph::launch_diff_norms(ts.om[0], c64, (const double2 *)ts.refM, d.n_outM, ts.acc + 2, ts.st)) !=
                     cudaSuccess)
        return cuda_fail(e, "diff_norms");
    double h[4] = {0, 0, 0, 0};
    if ((e = cudaMemcpyAsync(h, ts.acc, sizeof(h), cudaMemcpyDeviceToHost, ts.st)) != cudaSuccess)
        return cuda_fail(e, "memcpy");
    if ((e = cudaStreamSynchronize(ts.st)) != cudaSuccess) return cuda_fail(e, "sync");
    const double eb = h[1] > 0 ? std::sqrt(h[0] / h[1]) : 0.0, em = h[3] > 0 ? std::sqrt(h[2] / h[3]) : 0.0;
    *err = std::max(eb, em);
    return LAPH_OK;
}

static int autotune(laph_plan *p, const laph::Sched &def, const std::function<cudaError_t(const laph::Sched &)> &apply)
{
    const bool needB = !(p->flags & LAPH_PLAN_SKIP_B), needM = !(p->flags & LAPH_PLAN_SKIP_M);
    const bool fields = p->flags & LAPH_PLAN_FIELDS;
    TuneState ts;
    int rc = LAPH_OK;
    cudaError_t e = cudaSuccess;
    size_t best = 0;
    std::vector<char> accepted;   // candidates within the accuracy limit (all but rejected drain intervals)
    p->tune_cand.clear();
    p->tune_pc.clear();
    p->tune_ms.clear();
    p->tune_err.clear();
    auto run = [&](const laph::Sched &c, bool probe) -> int {
        cudaError_t er = apply(c);
        if (er != cudaSuccess) return cuda_fail(er, "autotune apply");
        if (p->max_staged > laph::TC_MAX_STAGED) return LAPH_ERR_UNSUPPORTED;
        float ms = 0.f;
        int r = tune_time(p, ts, &ms);
        if (r != LAPH_OK) return r;
        double err = -1.0;
        if (probe && (r = tune_probe(p, ts, &err)) != LAPH_OK) return r;
        p->tune_cand.push_back(c);
        p->tune_pc.push_back(p->sched_per_chunk);
        p->tune_ms.push_back(ms);
        p->tune_err.push_back(err);
        accepted.push_back(1);
        return LAPH_OK;
    };
#define TCK(call)                            \
    do {                                     \
        if ((e = (call)) != cudaSuccess) {   \
            rc = cuda_fail(e, #call);        \
            goto done;                       \
        }                                    \
    } while (0)
#define TRC(call)                            \
    do {                                     \
        if ((rc = (call)) != LAPH_OK) goto done; \
    } while (0)
    TCK(cudaStreamCreateWithFlags(&ts.st, cudaStreamNonBlocking));
    TCK(cudaEventCreate(&ts.e0));
    TCK(cudaEventCreate(&ts.e1));
    ts.phi.assign(p->n_inst, nullptr);
    ts.ob.assign(p->n_inst, nullptr);
    ts.om.assign(p->n_inst, nullptr);
    for (int n = 0; n < p->n_inst; n++) {
        TCK(cudaMalloc(&ts.phi[n], p->phi_elems[n] * sizeof(float2)));
        TCK(laph::launch_fill_pattern((float2 *)ts.phi[n], p->phi_elems[n], 1000u + (unsigned)n, ts.st));
        if (needB) TCK(cudaMalloc(&ts.ob[n], std::max<long long>(p->outB_elems[n], 1) * p->out_bytes));
        if (needM) TCK(cudaMalloc(&ts.om[n], std::max<long long>(p->outM_elems[n], 1) * p->out_bytes));
    }
    {
        // 1: tile width x tile order x chunking (the largest chunk only for one instance)
        const bool one_inst = p->n_inst == 1 && !(p->flags & LAPH_PLAN_CHUNK_PER_TIMESLICE);
        const std::pair<int, int> shapes[] = {{def.tile_cols, def.rows2}, {104, 0}, {96, 0},  {80, 0}, {64, 0},
                                              {176, 1},           {192, 1}, {208, 1}, {128, 1}, {laph::TC_PAIR_COLS, 2}};
        for (size_t k = 0; k < sizeof(shapes) / sizeof(shapes[0]); k++) {
            const int nc = shapes[k].first, r2 = shapes[k].second;
            if (k > 0 && nc == def.tile_cols && r2 == def.rows2) continue;
            for (long long pc : {-1LL, -2LL})
                for (int o = 0; o < 2; o++) {
                    if (pc == -2 && !one_inst) continue;
                    TRC(run(laph::Sched{nc, def.sum_sites, def.chunk_sites, pc, o, r2, def.chunk_sites_b}, false));
                }
        }
        for (size_t k = 1; k < p->tune_ms.size(); k++)
            if (p->tune_ms[k] < p->tune_ms[best]) best = k;
        // 2: site-block size of the FP64 reduction
        const laph::Sched b1 = p->tune_cand[best];
        for (int sum : {def.sum_sites / 2, def.sum_sites * 2}) {
            if (sum < 1024 || sum > (1 << 20)) continue;
            laph::Sched c = b1;
            c.sum_sites = sum;
            TRC(run(c, false));
            if (p->tune_ms.back() < p->tune_ms[best]) best = p->tune_ms.size() - 1;
        }
        // 3: drain interval, within the accuracy limit of the probe
        if (!fields) {
            const laph::Sched b2 = p->tune_cand[best];
            TRC(run(b2, true));   // the accuracy of the default interval
            const double err_def = p->tune_err.back();
            const size_t def_k = p->tune_ms.size() - 1;
            if (p->tune_ms[def_k] < p->tune_ms[best]) best = def_k;
            for (int cs : {def.chunk_sites / 2, (def.chunk_sites * 3) / 2}) {
                if (cs < 8) continue;
                laph::Sched c = b2;
                c.chunk_sites = cs;
                c.chunk_sites_b = 0;
                TRC(run(c, true));
                const double err = p->tune_err.back();
                accepted.back() = err <= TUNE_ERR_LIMIT || err <= err_def;
                if (accepted.back() && p->tune_ms.back() < p->tune_ms[best]) best = p->tune_ms.size() - 1;
            }
        }
        // 4: the three fastest accepted schedules are timed twice more, and
        // each keeps the lowest of its times, so that one noisy timing does
        // not decide between close candidates; the default schedule (candidate
        // 0) is timed again with them and keeps its place unless the fastest
        // beats it by more than TUNE_MARGIN
        auto same = [&](size_t qa, size_t qb) {
            const laph::Sched &a = p->tune_cand[qa], &b = p->tune_cand[qb];
            return a.tile_cols == b.tile_cols && a.sum_sites == b.sum_sites && a.chunk_sites == b.chunk_sites &&
                   a.per_chunk == b.per_chunk && a.order == b.order && a.rows2 == b.rows2 &&
                   a.chunk_sites_b == b.chunk_sites_b;
        };
        std::vector<size_t> top;
        for (size_t k = 0; k < p->tune_ms.size(); k++) {
            if (!accepted[k]) continue;
            bool dup = false;
            for (size_t q : top)
                if (same(q, k)) {
                    p->tune_ms[q] = std::min(p->tune_ms[q], p->tune_ms[k]);   // the same schedule timed again
                    dup = true;
                }
            if (!dup) top.push_back(k);
            std::sort(top.begin(), top.end(), [&](size_t a, size_t b) { return p->tune_ms[a] < p->tune_ms[b]; });
            if (top.size() > 3) top.pop_back();
        }
        size_t def_k = 0;
        bool def_in_top = false;
        for (size_t q : top)
            if (same(q, 0)) {
                def_k = q;
                def_in_top = true;
            }
        if (!def_in_top) top.push_back(0);
        for (int rep = 0; rep < 2 && top.size() > 1; rep++)
            for (size_t k : top) {
                TCK(apply(p->tune_cand[k]));
                float ms = 0.f;
                TRC(tune_time(p, ts, &ms));
                p->tune_ms[k] = std::min(p->tune_ms[k], ms);
            }
        best = top[0];
        for (size_t k : top)
            if (p->tune_ms[k] < p->tune_ms[best]) best = k;
        if (!same(best, def_k) && p->tune_ms[best] > (1.0 - TUNE_MARGIN) * p->tune_ms[def_k]) best = def_k;
    }
    TCK(apply(p->tune_cand[best]));
    TCK(cudaMemsetAsync(p->d_status, 0, sizeof(int), ts.st));
    TCK(cudaStreamSynchronize(ts.st));
done:
#undef TCK
#undef TRC
    if (ts.st) cudaStreamSynchronize(ts.st);
    if (ts.ref) laph_plan_destroy(ts.ref);
    cudaFree(ts.refB);
    cudaFree(ts.refM);
    cudaFree(ts.acc);
    for (int n = 0; n < (int)ts.phi.size(); n++) {
        cudaFree(ts.phi[n]);
        cudaFree(ts.ob[n]);
        cudaFree(ts.om[n]);
    }
    if (ts.e0) cudaEventDestroy(ts.e0);
    if (ts.e1) cudaEventDestroy(ts.e1);
    if (ts.st) cudaStreamDestroy(ts.st);
    return rc;
}

int laph_plan_schedule(const laph_plan *plan, int64_t *timeslices_per_chunk, int *tile_order, int *n_chunks,
                       int *n_candidates, float *candidate_ms)
{
    if (!plan) return LAPH_ERR_ARG;
    if (timeslices_per_chunk) *timeslices_per_chunk = plan->sched_per_chunk;
    if (tile_order) *tile_order = plan->sched_order;
    if (n_chunks) *n_chunks = (int)plan->chunks.size();
    if (n_candidates) *n_candidates = (int)plan->tune_ms.size();
    if (candidate_ms)
        for (size_t k = 0; k < plan->tune_ms.size() && k < 8; k++) candidate_ms[k] = plan->tune_ms[k];
    return LAPH_OK;
}

int laph_plan_drain_sites(const laph_plan *plan, int *chunk_sites, int *chunk_sites_b)
{
    if (!plan) return LAPH_ERR_ARG;
    if (chunk_sites) *chunk_sites = plan->chunk_sites;
    if (chunk_sites_b) *chunk_sites_b = plan->chunk_sites_b ? plan->chunk_sites_b : plan->chunk_sites;
    return LAPH_OK;
}

int laph_plan_tuning(const laph_plan *plan, int cap, laph_tune_record *rec, int *n_candidates)
{
    if (!plan || cap < 0 || (cap > 0 && !rec)) return LAPH_ERR_ARG;
    const int n = (int)plan->tune_ms.size();
    if (n_candidates) *n_candidates = n;
    for (int k = 0; k < n && k < cap; k++) {
        const laph::Sched &c = plan->tune_cand[k];
        rec[k].tile_cols = c.tile_cols;
        rec[k].layout = c.rows2;
        rec[k].sum_sites = c.sum_sites;
        rec[k].chunk_sites = c.chunk_sites;
        rec[k].chunk_sites_b = c.chunk_sites_b ? c.chunk_sites_b : c.chunk_sites;
        rec[k].tile_order = c.order;
        rec[k].timeslices_per_chunk = plan->tune_pc[k];
        rec[k].ms = plan->tune_ms[k];
        rec[k].probe_err = plan->tune_err[k];
    }
    return LAPH_OK;
}

int laph_plan_kernel_times(laph_plan *plan, int n, float *ms)
{
    if (!plan) return LAPH_ERR_ARG;
    return ring_times(plan->ev_begin, plan->ev_end, plan->n_timed, n, ms);
}

int laph_plan_operand_times(laph_plan *plan, int n, float *ms)
{
    if (!plan) return LAPH_ERR_ARG;
    return ring_times(plan->pv_begin, plan->pv_end, plan->n_ptimed, n, ms);
}

int laph_plan_reduce_times(laph_plan *plan, int n, float *ms)
{
    if (!plan || !is_tc_mode(plan->mode)) return LAPH_ERR_ARG;
    return ring_times(plan->rd_begin, plan->rd_end, plan->n_timed, n, ms);
}

int laph_plan_contraction_launches(const laph_plan *plan, int *n)
{
    if (!plan || !n) return LAPH_ERR_ARG;
    *n = is_tc_mode(plan->mode) ? (int)plan->chunks.size()
                                : (int)((plan->n_tiles + 0x7ffffffeLL) / 0x7fffffffLL);
    return LAPH_OK;
}

int laph_plan_tensor_flops(const laph_plan *plan, double *flops)
{
    if (!plan || !flops) return LAPH_ERR_ARG;
    *flops = plan->mma_flops;
    return LAPH_OK;
}

int laph_plan_launches_per_execute(const laph_plan *plan, int *n)
{
    if (!plan || !n) return LAPH_ERR_ARG;
    const int ptr_launches = (plan->n_inst + 63) / 64;
    int prep = 0;   // scale, blockify
    for (const laph_plan::PrepRun &r : plan->prep) prep += 2 * ((r.n_units + 65534) / 65535);
    if (is_tc_mode(plan->mode))
        *n = ptr_launches + prep + 3 * (int)plan->chunks.size() /* psi, contraction, FP64 site reduction */ +
             (!plan->chunks.empty() && plan->chunks.back().n_split > 0 &&
              plan->chunks.back().n_split < plan->chunks.back().n_units) /* a reduction for either kind of unit */;
    else
        *n = ptr_launches + (int)((plan->n_tiles + 0x7ffffffeLL) / 0x7fffffffLL);
    return LAPH_OK;
}

int laph_plan_execute(laph_plan *plan, const void *const *phi, void *const *out_B, void *const *out_M,
                      void *workspace, void *stream)
{
    if (!plan || !phi || (plan->flags & LAPH_PLAN_FIELDS)) return LAPH_ERR_ARG;
    const bool needB = !(plan->flags & LAPH_PLAN_SKIP_B), needM = !(plan->flags & LAPH_PLAN_SKIP_M);
    if ((needB && !out_B) || (needM && !out_M)) return LAPH_ERR_ARG;
    for (int n = 0; n < plan->n_inst; n++) {
        if (!phi[n] || ((uintptr_t)phi[n]) % 8) return LAPH_ERR_ARG;
        if (needB && (!out_B[n] || ((uintptr_t)out_B[n]) % 16)) return LAPH_ERR_ARG;
        if (needM && (!out_M[n] || ((uintptr_t)out_M[n]) % 16)) return LAPH_ERR_ARG;
    }
    int cur = 0;
    CK(cudaGetDevice(&cur));
    if (cur != plan->device) return LAPH_ERR_ARG;
    cudaStream_t s = (cudaStream_t)stream;
    const bool tc = is_tc_mode(plan->mode);
    if (tc && (!workspace || ((uintptr_t)workspace) % 256)) return LAPH_ERR_WORKSPACE;
    cudaError_t e = laph::launch_set_pointers(plan->d_inst, 0, plan->n_inst, phi, needB ? out_B : nullptr,
                                              needM ? out_M : nullptr, workspace, s, nullptr, 1, workspace,
                                              tc ? plan->ws_zero_bytes : 0);
    if (e != cudaSuccess) return cuda_fail(e, "set_pointers");
    return launch_batch(plan, workspace, s, true);
}

int laph_plan_execute_fields(laph_plan *plan, const void *const *fields, void *const *out, void *workspace,
                             void *stream)
{
    if (!plan || !fields || !out || !(plan->flags & LAPH_PLAN_FIELDS)) return LAPH_ERR_ARG;
    const bool trip = plan->flags & LAPH_PLAN_SKIP_M;
    const int nf = trip ? 3 : 2;
    for (int n = 0; n < plan->n_inst; n++) {
        for (int f = 0; f < nf; f++)
            if (!fields[nf * n + f] || ((uintptr_t)fields[nf * n + f]) % 8) return LAPH_ERR_ARG;
        if (!out[n] || ((uintptr_t)out[n]) % 16) return LAPH_ERR_ARG;
    }
    int cur = 0;
    CK(cudaGetDevice(&cur));
    if (cur != plan->device) return LAPH_ERR_ARG;
    cudaStream_t s = (cudaStream_t)stream;
    if (!workspace || ((uintptr_t)workspace) % 256) return LAPH_ERR_WORKSPACE;
    cudaError_t e = laph::launch_set_pointers(plan->d_inst, 0, plan->n_inst, nullptr, trip ? out : nullptr,
                                              trip ? nullptr : out, workspace, s, fields, nf, workspace,
                                              plan->ws_zero_bytes);
    if (e != cudaSuccess) return cuda_fail(e, "set_pointers");
    return launch_batch(plan, workspace, s, true);
}

int laph_plan_host_workspace_size(const laph_plan *plan, size_t *bytes)
{
    if (!plan || !bytes) return LAPH_ERR_ARG;
    size_t total = ((plan->ws_bytes + 255) / 256) * 256;
    for (int n = 0; n < plan->n_inst; n++) {
        total += ((plan->phi_elems[n] * sizeof(float2) + 255) / 256) * 256;
        total += ((plan->outB_elems[n] * plan->out_bytes + 255) / 256) * 256;
        total += ((plan->outM_elems[n] * plan->out_bytes + 255) / 256) * 256;
    }
    *bytes = total;
    return LAPH_OK;
}

// laph_plan_execute_host without the clean-up after a failure
static int execute_host_body(laph_plan *plan, const void *const *phi_host, void *const *out_B_host, void *const *out_M_host,
                      void *workspace, cudaStream_t s)
{
    if (!phi_host || !workspace || ((uintptr_t)workspace) % 256) return LAPH_ERR_ARG;
    if (plan->flags & LAPH_PLAN_FIELDS) return LAPH_ERR_UNSUPPORTED;
    const bool needB = !(plan->flags & LAPH_PLAN_SKIP_B), needM = !(plan->flags & LAPH_PLAN_SKIP_M);
    if ((needB && !out_B_host) || (needM && !out_M_host)) return LAPH_ERR_ARG;
    int cur = 0;
    CK(cudaGetDevice(&cur));
    if (cur != plan->device) return LAPH_ERR_ARG;
    char *ws = (char *)workspace;
    size_t off = ((plan->ws_bytes + 255) / 256) * 256;
    std::vector<const void *> dphi(plan->n_inst);
    std::vector<void *> dB(plan->n_inst), dM(plan->n_inst);
    for (int n = 0; n < plan->n_inst; n++) {
        if (!phi_host[n] || (needB && !out_B_host[n]) || (needM && !out_M_host[n])) return LAPH_ERR_ARG;
        dphi[n] = ws + off;
        off += ((plan->phi_elems[n] * sizeof(float2) + 255) / 256) * 256;
        dB[n] = ws + off;
        off += ((plan->outB_elems[n] * plan->out_bytes + 255) / 256) * 256;
        dM[n] = ws + off;
        off += ((plan->outM_elems[n] * plan->out_bytes + 255) / 256) * 256;
    }
    cudaError_t e = laph::launch_set_pointers(plan->d_inst, 0, plan->n_inst, dphi.data(), needB ? dB.data() : nullptr,
                                              needM ? dM.data() : nullptr, ws, s);
    if (e != cudaSuccess) return cuda_fail(e, "set_pointers");

    if (!is_tc_mode(plan->mode)) {
        for (int n = 0; n < plan->n_inst; n++)
            CK(cudaMemcpyAsync((void *)dphi[n], phi_host[n], plan->phi_elems[n] * sizeof(float2), cudaMemcpyHostToDevice,
                               s));
        int rc = launch_batch(plan, ws, s);
        if (rc != LAPH_OK) return rc;
        for (int n = 0; n < plan->n_inst; n++) {
            if (needB)
                CK(cudaMemcpyAsync(out_B_host[n], dB[n], plan->outB_elems[n] * plan->out_bytes, cudaMemcpyDeviceToHost,
                                   s));
            if (needM)
                CK(cudaMemcpyAsync(out_M_host[n], dM[n], plan->outM_elems[n] * plan->out_bytes, cudaMemcpyDeviceToHost,
                                   s));
        }
        CK(cudaStreamSynchronize(s));
        return LAPH_OK;
    }

    // tensor-core path, chunk by chunk: the inputs of every chunk are queued
    // on one copy stream up front (chunk c lands while chunk c-1 computes), and
    // the outputs of chunk c are copied out on a second stream while chunk c+1
    // computes.  The inputs go first so that no copy in of a later chunk is
    // queued behind a copy out that waits for an earlier chunk's results.
    const size_t nc = plan->chunks.size();
    if (!plan->h2d) {
        CK(cudaStreamCreateWithFlags(&plan->h2d, cudaStreamNonBlocking));
        CK(cudaStreamCreateWithFlags(&plan->d2h, cudaStreamNonBlocking));
    }
    while (plan->ev_in.size() < nc) {
        cudaEvent_t a = nullptr, b = nullptr;
        CK(cudaEventCreateWithFlags(&a, cudaEventDisableTiming));
        CK(cudaEventCreateWithFlags(&b, cudaEventDisableTiming));
        plan->ev_in.push_back(a);
        plan->ev_out.push_back(b);
    }
    CK(cudaMemsetAsync(ws, 0, plan->ws_zero_bytes, s));
    // the copy streams start after everything already queued on `stream`
    CK(cudaEventRecord(plan->ev_out[0], s));
    CK(cudaStreamWaitEvent(plan->h2d, plan->ev_out[0], 0));
    CK(cudaStreamWaitEvent(plan->d2h, plan->ev_out[0], 0));
    const laph::TcConfig cfg = tc_config(plan);
    for (size_t ci = 0; ci < nc; ci++) {
        const laph_plan::Chunk &c = plan->chunks[ci];
        for (int u = c.unit0; u < c.unit0 + c.n_units; u++) {
            const int n = plan->h_units[u].inst, t = plan->h_units[u].t;
            const size_t bytes = plan->phi_elems[n] / plan->h_T[n] * sizeof(float2);
            CK(cudaMemcpyAsync((char *)dphi[n] + t * bytes, (const char *)phi_host[n] + t * bytes, bytes,
                               cudaMemcpyHostToDevice, plan->h2d));
        }
        CK(cudaEventRecord(plan->ev_in[ci], plan->h2d));
    }
    for (size_t ci = 0; ci < nc; ci++) {
        const laph_plan::Chunk &c = plan->chunks[ci];
        CK(cudaStreamWaitEvent(s, plan->ev_in[ci], 0));
        int rc = launch_prep(plan, ws, prep_runs(plan, c.unit0, c.n_units), s);
        if (rc == LAPH_OK) rc = launch_tc_chunk(plan, ws, ci, cfg, s);
        if (rc != LAPH_OK) return rc;
        // the outputs of chunk ci are final once its site reduction (side stream) is done
        CK(cudaStreamWaitEvent(plan->d2h, plan->ev_red[ci], 0));
        for (int u = c.unit0; u < c.unit0 + c.n_units; u++) {
            const int n = plan->h_units[u].inst, t = plan->h_units[u].t;
            if (needB) {
                const size_t bytes = plan->outB_elems[n] / plan->h_T[n] * plan->out_bytes;
                CK(cudaMemcpyAsync((char *)out_B_host[n] + t * bytes, (char *)dB[n] + t * bytes, bytes,
                                   cudaMemcpyDeviceToHost, plan->d2h));
            }
            if (needM) {
                const size_t bytes = plan->outM_elems[n] / plan->h_T[n] * plan->out_bytes;
                CK(cudaMemcpyAsync((char *)out_M_host[n] + t * bytes, (char *)dM[n] + t * bytes, bytes,
                                   cudaMemcpyDeviceToHost, plan->d2h));
            }
        }
    }
    CK(cudaStreamSynchronize(plan->d2h));
    CK(cudaStreamSynchronize(s));
    return LAPH_OK;
}

int laph_plan_execute_host(laph_plan *plan, const void *const *phi_host, void *const *out_B_host,
                           void *const *out_M_host, void *workspace, void *stream)
{
    if (!plan) return LAPH_ERR_ARG;
    cudaStream_t s = (cudaStream_t)stream;
    const int rc = execute_host_body(plan, phi_host, out_B_host, out_M_host, workspace, s);
    if (rc != LAPH_OK) {
        // copies queued before the failure still read or write the caller's
        // host buffers: they finish before the caller gets the buffers back
        if (plan->h2d) cudaStreamSynchronize(plan->h2d);
        if (plan->d2h) cudaStreamSynchronize(plan->d2h);
        cudaStreamSynchronize(s);
    }
    return rc;
}

int laph_get_device_status(laph_plan *plan, void *stream, int *status)
{
    if (!plan || !status) return LAPH_ERR_ARG;
    cudaStream_t s = (cudaStream_t)stream;
    int h = 0;
    CK(cudaMemcpyAsync(&h, plan->d_status, sizeof(int), cudaMemcpyDeviceToHost, s));
    CK(cudaStreamSynchronize(s));
    CK(cudaMemsetAsync(plan->d_status, 0, sizeof(int), s));
    *status = (h & laph::STATUS_TIMEOUT) ? LAPH_ERR_TIMEOUT : (h & laph::STATUS_CHECK) ? LAPH_ERR_DEVICE : LAPH_OK;
    return LAPH_OK;
}

int laph_plan_destroy(laph_plan *plan)
{
    if (!plan) return LAPH_ERR_ARG;
    free_plan(plan);
    return LAPH_OK;
}

// ------------------------------------------------------- simple entry points

static int one_shot(const void *phi, int L, int T, int N, const int32_t *momenta, int n_mom, void *out, int mode,
                    void *stream, bool baryon)
{
    if (!phi || !out) return LAPH_ERR_ARG;
    laph_instance inst = {L, T, N, n_mom, momenta};
    laph_plan *plan = nullptr;
    int rc = laph_plan_create(&inst, 1, mode, baryon ? LAPH_PLAN_SKIP_M : LAPH_PLAN_SKIP_B, &plan);
    if (rc != LAPH_OK) return rc;
    cudaStream_t s = (cudaStream_t)stream;
    void *ws = nullptr;
    if (plan->ws_bytes) {
        cudaError_t e = cudaMallocAsync(&ws, plan->ws_bytes, s);
        if (e != cudaSuccess) {
            laph_plan_destroy(plan);
            return cuda_fail(e, "cudaMallocAsync");
        }
    }
    void *o = out;
    rc = laph_plan_execute(plan, &phi, baryon ? &o : nullptr, baryon ? nullptr : &o, ws, stream);
    if (ws) cudaFreeAsync(ws, s);
    int dev = LAPH_OK;
    int rc2 = laph_get_device_status(plan, stream, &dev);  // synchronises the stream
    laph_plan_destroy(plan);
    if (rc != LAPH_OK) return rc;
    if (rc2 != LAPH_OK) return rc2;
    return dev;
}

int laph_baryon_blocks(const void *phi, int L, int T, int N, const int32_t *momenta, int n_mom, void *out, int mode,
                       void *stream)
{
    return one_shot(phi, L, T, N, momenta, n_mom, out, mode, stream, true);
}

int laph_meson_blocks(const void *phi, int L, int T, int N, const int32_t *momenta, int n_mom, void *out, int mode,
                      void *stream)
{
    return one_shot(phi, L, T, N, momenta, n_mom, out, mode, stream, false);
}

// Triplets (three fields) or doublets (two fields) of one instance.
static int one_shot_fields(const void *const *fields, int L, int T, int N, const int32_t *momenta, int n_mom,
                           void *out, int mode, void *stream, bool triplets)
{
    if (!out) return LAPH_ERR_ARG;
    laph_instance inst = {L, T, N, n_mom, momenta};
    laph_plan *plan = nullptr;
    int rc = laph_plan_create(&inst, 1, mode, LAPH_PLAN_FIELDS | (triplets ? LAPH_PLAN_SKIP_M : LAPH_PLAN_SKIP_B),
                              &plan);
    if (rc != LAPH_OK) return rc;
    cudaStream_t s = (cudaStream_t)stream;
    void *ws = nullptr;
    if (plan->ws_bytes) {
        cudaError_t e = cudaMallocAsync(&ws, plan->ws_bytes, s);
        if (e != cudaSuccess) {
            laph_plan_destroy(plan);
            return cuda_fail(e, "cudaMallocAsync");
        }
    }
    void *o = out;
    rc = laph_plan_execute_fields(plan, fields, &o, ws, stream);
    if (ws) cudaFreeAsync(ws, s);
    int dev = LAPH_OK;
    int rc2 = laph_get_device_status(plan, stream, &dev);  // synchronises the stream
    laph_plan_destroy(plan);
    if (rc != LAPH_OK) return rc;
    if (rc2 != LAPH_OK) return rc2;
    return dev;
}

int laph_projection(const void *v, const void *s, int L, int T, int Nv, int Ns, const int32_t *momenta, int n_mom,
                    void *out, int mode, void *stream)
{
    if (!out || Ns < 1) return LAPH_ERR_ARG;
    laph_instance inst = {L, T, Nv, n_mom, momenta, Ns};
    laph_plan *plan = nullptr;
    int rc = laph_plan_create(&inst, 1, mode, LAPH_PLAN_FIELDS | LAPH_PLAN_SKIP_B, &plan);
    if (rc != LAPH_OK) return rc;
    cudaStream_t st = (cudaStream_t)stream;
    void *ws = nullptr;
    if (plan->ws_bytes) {
        cudaError_t e = cudaMallocAsync(&ws, plan->ws_bytes, st);
        if (e != cudaSuccess) {
            laph_plan_destroy(plan);
            return cuda_fail(e, "cudaMallocAsync");
        }
    }
    const void *f[2] = {v, s};
    void *o = out;
    rc = laph_plan_execute_fields(plan, f, &o, ws, stream);
    if (ws) cudaFreeAsync(ws, st);
    int dev = LAPH_OK;
    int rc2 = laph_get_device_status(plan, stream, &dev);  // synchronises the stream
    laph_plan_destroy(plan);
    if (rc != LAPH_OK) return rc;
    if (rc2 != LAPH_OK) return rc2;
    return dev;
}

int laph_triplet_blocks(const void *phi, const void *psi, const void *chi, int L, int T, int N,
                        const int32_t *momenta, int n_mom, void *out, int mode, void *stream)
{
    const void *f[3] = {phi, psi, chi};
    return one_shot_fields(f, L, T, N, momenta, n_mom, out, mode, stream, true);
}

int laph_doublet_blocks(const void *phi, const void *psi, int L, int T, int N, const int32_t *momenta, int n_mom,
                        void *out, int mode, void *stream)
{
    const void *f[2] = {phi, psi};
    return one_shot_fields(f, L, T, N, momenta, n_mom, out, mode, stream, false);
}

}  // extern "C"
