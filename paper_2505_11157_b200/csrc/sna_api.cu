// C ABI of the library (declared in include/sna.h): plan life cycle, introspection and the compute entry
// points.  Host-side validation happens here; kernels live in the other translation units.
#include "../../include/sna.h"

#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <mutex>
#include <new>
#include <numeric>
#include <string>
#include <vector>

#include "sna_kernels.cuh"
#include "sna_plan.hpp"

namespace {

thread_local char g_last_error[512] = "";

void set_error(const char* fmt, ...) __attribute__((format(printf, 1, 2)));
void set_error(const char* fmt, ...) {
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(g_last_error, sizeof(g_last_error), fmt, ap);
    va_end(ap);
}

sna_status_t cuda_fail(cudaError_t e, const char* what) {
    set_error("%s: %s", what, cudaGetErrorString(e));
    return SNA_ERR_CUDA;
}

bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

}  // namespace

struct sna_plan {
    sna::HostPlan host;
    sna::DevPlan dev{};
    std::vector<int32_t> band_lengths[4];      // of the four band streams (DevBand::lengths)
    int device = 0;
    std::vector<int> unvisited;        // input rings that the dense dk/dv kernel does not write (weight zero, or in no window)
    bool is_global = false;            // created by sna_plan_create_global: every window is a whole ring
    void* dev_blob = nullptr;          // one allocation holding every device table
    mutable std::mutex ws_mutex;
    mutable void* ws = nullptr;        // workspace grown on demand by sna_backward
    mutable size_t ws_bytes = 0;
};

namespace {

bool supported_C(int C) { return C >= 4 && C <= 128 && C % 4 == 0; }

sna_status_t check_problem(const sna_plan_t* plan, int B, int H, int C) {
    if (plan == nullptr) { set_error("plan is NULL"); return SNA_ERR_INVALID_ARG; }
    if (plan->dev_blob == nullptr) { set_error("plan was created host-only; it cannot compute"); return SNA_ERR_INVALID_ARG; }
    if (B <= 0 || H <= 0 || C <= 0) { set_error("B, H and C must be positive"); return SNA_ERR_INVALID_ARG; }
    if (!supported_C(C)) { set_error("C=%d unsupported (a multiple of 4 between 4 and 128)", C); return SNA_ERR_UNSUPPORTED; }
    // The plan's tables, and by contract the caller's tensors, live on the device the plan was created on; launching
    // with another device current would hand that device foreign addresses.
    int current = -1;
    if (cudaGetDevice(&current) != cudaSuccess || current != plan->device) {
        set_error("the current CUDA device (%d) is not the plan's device (%d)", current, plan->device);
        return SNA_ERR_INVALID_ARG;
    }
    const long long N = (long long)B * H;
    const long long big = std::max((long long)plan->host.nlat_in * plan->host.nlon_in,
                                   (long long)plan->host.nlat_out * plan->host.nlon_out);
    if (N > 0x7fffffffLL || N * big > 0x7fffffffLL) { set_error("problem too large: B*H*nlat*nlon must fit in 31 bits"); return SNA_ERR_UNSUPPORTED; }
    return SNA_OK;
}

template <typename... P>
bool all_aligned(P... ptrs) { return (aligned16(ptrs) && ...); }

long long points_in(const sna_plan_t* plan) { return (long long)plan->host.nlat_in * plan->host.nlon_in; }
long long points_out(const sna_plan_t* plan) { return (long long)plan->host.nlat_out * plan->host.nlon_out; }
size_t stats_elems(const sna_plan_t* plan, int B, int H) {
    return (size_t)B * H * plan->host.nlat_out * plan->host.nlon_out;
}
bool tf32_supported(const sna_plan_t* plan, int C) {
    return (C == 16 || C == 32 || C == 64) && plan->host.nlon_out >= 32 && !plan->is_global && sna::band_path_supported(plan->dev, C);
}
size_t round256(size_t x) { return (x + 255) / 256 * 256; }

}  // namespace

extern "C" {

const char* sna_status_string(sna_status_t s) {
    switch (s) {
        case SNA_OK: return "SNA_OK";
        case SNA_ERR_INVALID_ARG: return "SNA_ERR_INVALID_ARG";
        case SNA_ERR_UNSUPPORTED: return "SNA_ERR_UNSUPPORTED";
        case SNA_ERR_EMPTY_NEIGHBORHOOD: return "SNA_ERR_EMPTY_NEIGHBORHOOD";
        case SNA_ERR_ALLOC: return "SNA_ERR_ALLOC";
        case SNA_ERR_CUDA: return "SNA_ERR_CUDA";
        case SNA_ERR_AMBIGUOUS_TIE: return "SNA_ERR_AMBIGUOUS_TIE";
        case SNA_ERR_WORKSPACE: return "SNA_ERR_WORKSPACE";
    }
    return "SNA_ERR_UNKNOWN";
}

const char* sna_last_error_message(void) { return g_last_error; }

// Measured on the benchmark configurations (fwd+bwd, against whole rings only): 128 gives -4 % at 361x720, -1.5 % at
// 128x256 and -0.7 % on the 2:1 down-sampling case; 96 and below lose, because a masked 128-row block uses at most
// W / (ps * 127 + W) of its entries.
constexpr int DENSE_MIN_WIDTH = 128;

static sna_status_t plan_create(int nlat_in, int nlon_in, int nlat_out, int nlon_out, sna_grid_t grid_in,
                                sna_grid_t grid_out, double theta_cutoff, bool upload, sna_plan_t** plan_out,
                                bool global = false) {
    if (plan_out == nullptr) { set_error("plan_out is NULL"); return SNA_ERR_INVALID_ARG; }
    sna_plan* plan = new (std::nothrow) sna_plan();
    if (plan == nullptr) { set_error("out of host memory"); return SNA_ERR_ALLOC; }
    std::string why;
    sna::PlanStatus ps;
    try {
        ps = sna::build_plan(nlat_in, nlon_in, nlat_out, nlon_out, (int)grid_in, (int)grid_out, theta_cutoff, plan->host, why);
    } catch (const std::bad_alloc&) {
        delete plan;
        set_error("out of host memory while building the table");
        return SNA_ERR_ALLOC;
    }
    if (ps != sna::PLAN_OK) {
        delete plan;
        set_error("%s", why.c_str());
        return ps == sna::PLAN_INVALID ? SNA_ERR_INVALID_ARG : ps == sna::PLAN_UNSUPPORTED ? SNA_ERR_UNSUPPORTED
             : ps == sna::PLAN_EMPTY ? SNA_ERR_EMPTY_NEIGHBORHOOD : SNA_ERR_AMBIGUOUS_TIE;
    }
    if (!upload) { *plan_out = plan; return SNA_OK; }
    // the kernels walk the table without rings of weight zero; plan->host keeps every member for the table queries
    sna::HostPlan weighted;
    const bool dropped = sna::drop_zero_weight_rings(plan->host, weighted);
    const sna::HostPlan& hp = dropped ? weighted : plan->host;
    // heavy-first orders
    std::vector<int32_t> row_order(hp.nlat_out), t_row_order(hp.nlat_in);
    std::iota(row_order.begin(), row_order.end(), 0);
    std::iota(t_row_order.begin(), t_row_order.end(), 0);
    std::stable_sort(row_order.begin(), row_order.end(), [&](int a, int b) { return hp.row_nnz[a] > hp.row_nnz[b]; });
    std::stable_sort(t_row_order.begin(), t_row_order.end(), [&](int a, int b) { return hp.t_row_nnz[a] > hp.t_row_nnz[b]; });
    std::vector<int32_t> win_lat(hp.windows.size()), win_m(hp.windows.size()), t_lat(hp.t_windows.size()), t_m(hp.t_windows.size());
    for (size_t i = 0; i < hp.windows.size(); ++i) { win_lat[i] = hp.windows[i].lat; win_m[i] = hp.windows[i].m; }
    for (size_t i = 0; i < hp.t_windows.size(); ++i) { t_lat[i] = hp.t_windows[i].lat; t_m[i] = hp.t_windows[i].m; }
    std::vector<float> log2_omega(hp.nlat_in);
    for (int h = 0; h < hp.nlat_in; ++h) log2_omega[h] = (float)std::log2(hp.omega[h]);

    sna::BandStream bands[4];          // forward and transposed, each with all windows and without the dense kernels' ones
    sna::DenseLists dense, t_dense;
#ifdef SNA_PROF
    const int32_t zero_status[512] = {};   // room for the per-role profile of a -DSNA_PROF build
#else
    const int32_t zero_status[64] = {};
#endif
    bool t_consecutive = false;
    plan->is_global = global;
    // Windows at least this many input columns wide (and whole rings) run on the dense tcgen05 kernels, as masked blocks;
    // narrower ones stay on the band kernels, whose 8-column tiles waste less on a slanted band.
    const int dense_min_width = DENSE_MIN_WIDTH;
    try {
        sna::build_dense_lists(hp, dense, dense_min_width);
        sna::build_transposed_dense_lists(hp, t_dense, dense_min_width);
        // rows with the longest lists first: the dense kernels run one block per SM, so the long tiles must not start last
        std::stable_sort(dense.rows.begin(), dense.rows.end(), [&](int a, int b) { return dense.ptr[a + 1] - dense.ptr[a] > dense.ptr[b + 1] - dense.ptr[b]; });
        std::stable_sort(t_dense.rows.begin(), t_dense.rows.end(), [&](int a, int b) { return t_dense.ptr[a + 1] - t_dense.ptr[a] > t_dense.ptr[b + 1] - t_dense.ptr[b]; });
        if (global) {
            sna::build_global_bands(hp, bands[0], bands[2]);
            t_consecutive = true;
        } else {
            sna::build_forward_band(hp, bands[0]);
            sna::build_forward_band(hp, bands[1], dense_min_width);
            t_consecutive = sna::build_transposed_band(hp, bands[2]);
            sna::build_transposed_band(hp, bands[3], dense_min_width);
        }
    } catch (const std::bad_alloc&) {
        delete plan;
        set_error("out of host memory while building the band streams");
        return SNA_ERR_ALLOC;
    }
    static_assert(sizeof(sna::BandColumn) == 16, "read as int4");

    // pack everything into one device allocation (each array 256-byte aligned)
    struct Piece { const void* src; size_t bytes; size_t offset; };
    std::vector<Piece> pieces = {
        {hp.row_ptr.data(), hp.row_ptr.size() * 4, 0}, {win_lat.data(), win_lat.size() * 4, 0}, {win_m.data(), win_m.size() * 4, 0},
        {row_order.data(), row_order.size() * 4, 0}, {hp.t_row_ptr.data(), hp.t_row_ptr.size() * 4, 0}, {t_lat.data(), t_lat.size() * 4, 0},
        {t_m.data(), t_m.size() * 4, 0}, {t_row_order.data(), t_row_order.size() * 4, 0}, {log2_omega.data(), log2_omega.size() * 4, 0},
        {dense.ptr.data(), dense.ptr.size() * 4, 0}, {dense.lat.data(), dense.lat.size() * 4, 0}, {dense.m.data(), dense.m.size() * 4, 0},
        {dense.rows.data(), dense.rows.size() * 4, 0}, {t_dense.ptr.data(), t_dense.ptr.size() * 4, 0}, {t_dense.lat.data(), t_dense.lat.size() * 4, 0},
        {t_dense.m.data(), t_dense.m.size() * 4, 0}, {t_dense.rows.data(), t_dense.rows.size() * 4, 0}, {zero_status, sizeof(zero_status), 0}};
    const size_t first_band_piece = pieces.size();
    constexpr size_t BAND_PIECES = 4;
    for (const sna::BandStream& b : bands) {
        pieces.push_back({b.chunk_ptr.data(), b.chunk_ptr.size() * 4, 0});
        pieces.push_back({b.columns.data(), b.columns.size() * sizeof(sna::BandColumn), 0});
        pieces.push_back({b.masks.data(), b.masks.size() * 4, 0});
        pieces.push_back({b.order.data(), b.order.size() * 4, 0});
    }
    size_t total = 0;
    for (Piece& p : pieces) { p.offset = total; total += round256(p.bytes); }
    cudaError_t e = cudaGetDevice(&plan->device);
    if (e != cudaSuccess) { delete plan; return cuda_fail(e, "cudaGetDevice"); }
    e = cudaMalloc(&plan->dev_blob, total);
    if (e != cudaSuccess) { delete plan; set_error("cudaMalloc of %zu bytes: %s", total, cudaGetErrorString(e)); return SNA_ERR_ALLOC; }
    try {
        std::vector<char> blob(total);       // one copy instead of one per piece
        for (const Piece& p : pieces)
            if (p.bytes != 0) std::memcpy(blob.data() + p.offset, p.src, p.bytes);
        e = cudaMemcpy(plan->dev_blob, blob.data(), total, cudaMemcpyHostToDevice);
    } catch (const std::bad_alloc&) {
        cudaFree(plan->dev_blob);
        delete plan;
        set_error("out of host memory while uploading the plan");
        return SNA_ERR_ALLOC;
    }
    if (e != cudaSuccess) { cudaFree(plan->dev_blob); delete plan; return cuda_fail(e, "cudaMemcpy of plan tables"); }
    auto at = [&](size_t i) { return (const int32_t*)((char*)plan->dev_blob + pieces[i].offset); };
    sna::DevPlan& d = plan->dev;
    d.nlat_in = hp.nlat_in; d.nlon_in = hp.nlon_in; d.nlat_out = hp.nlat_out; d.nlon_out = hp.nlon_out; d.ps = hp.ps;
    d.row_ptr = at(0); d.win_lat = at(1); d.win_m = at(2); d.row_order = at(3);
    d.t_row_ptr = at(4); d.t_win_lat = at(5); d.t_win_m = at(6); d.t_row_order = at(7);
    d.log2_omega = (const float*)at(8);
    d.dense_ptr = at(9); d.dense_lat = at(10); d.dense_m = at(11); d.dense_rows = at(12);
    d.t_dense_ptr = at(13); d.t_dense_lat = at(14); d.t_dense_m = at(15); d.t_dense_rows = at(16);
    d.dev_status = (int*)((char*)plan->dev_blob + pieces[17].offset);
    for (int h = 0; h < hp.nlat_in; ++h) if (t_dense.ptr[h + 1] == t_dense.ptr[h]) plan->unvisited.push_back(h);
    d.n_dense_rows = (int)dense.rows.size();
    d.n_t_dense_rows = (int)t_dense.rows.size();
    d.dense_blocks = dense.blocks;
    d.dense_longest = dense.longest;
    d.dense_fraction = hp.nnz > 0 ? (float)((double)dense.pairs / (double)hp.nnz) : 0.f;
    d.dense_all = dense.pairs == hp.nnz ? 1 : 0;
    d.pairs = hp.nnz * hp.nlon_out;
    d.longest_row = *std::max_element(hp.row_nnz.begin(), hp.row_nnz.end());
    d.longest_t_row = *std::max_element(hp.t_row_nnz.begin(), hp.t_row_nnz.end()) / hp.ps;
    d.is_global = global ? 1 : 0;
    d.t_consecutive = t_consecutive ? 1 : 0;
    sna::DevBand* dev_bands[4] = {&d.fwd, &d.fwdb, &d.t, &d.tb};
    for (size_t i = 0; i < 4; ++i) {
        const size_t f = first_band_piece + BAND_PIECES * i;
        plan->band_lengths[i] = std::move(bands[i].lengths);
        const sna::BandStream& b = bands[i];
        if (b.chunk_ptr.empty()) continue;
        const int groups = (int)b.order.size();
        *dev_bands[i] = sna::DevBand{at(f), (const int4*)at(f + 1), (const uint32_t*)at(f + 2), at(f + 3), plan->band_lengths[i].data(),
                                     groups, b.one_row, (long long)b.chunk_ptr.back() * (b.one_row ? groups : 1)};
    }
    e = cudaDeviceGetAttribute(&d.num_sms, cudaDevAttrMultiProcessorCount, plan->device);
    if (e != cudaSuccess) { sna_plan_destroy(plan); return cuda_fail(e, "cudaDeviceGetAttribute"); }
    // opt in to the kernels' dynamic shared-memory sizes on this device (once here instead of on every launch)
    e = sna::dense2_prepare_device();
    if (e == cudaSuccess) e = sna::band_prepare_device();
    if (e != cudaSuccess) { sna_plan_destroy(plan); return cuda_fail(e, "cudaFuncSetAttribute"); }
    *plan_out = plan;
    return SNA_OK;
}

sna_status_t sna_plan_create(int nlat_in, int nlon_in, int nlat_out, int nlon_out, sna_grid_t grid_in,
                             sna_grid_t grid_out, double theta_cutoff, sna_plan_t** plan_out) {
    return plan_create(nlat_in, nlon_in, nlat_out, nlon_out, grid_in, grid_out, theta_cutoff, true, plan_out);
}

sna_status_t sna_plan_create_global(int nlat_in, int nlon_in, int nlat_out, int nlon_out, sna_grid_t grid_in,
                                    sna_grid_t grid_out, sna_plan_t** plan_out) {
    // theta_cutoff = pi selects every input point for every output point; no distance is evaluated
    return plan_create(nlat_in, nlon_in, nlat_out, nlon_out, grid_in, grid_out, 3.14159265358979323846, true, plan_out, true);
}

sna_status_t sna_plan_create_host_only(int nlat_in, int nlon_in, int nlat_out, int nlon_out, sna_grid_t grid_in,
                                       sna_grid_t grid_out, double theta_cutoff, sna_plan_t** plan_out) {
    return plan_create(nlat_in, nlon_in, nlat_out, nlon_out, grid_in, grid_out, theta_cutoff, false, plan_out);
}

sna_status_t sna_plan_destroy(sna_plan_t* plan) {
    if (plan == nullptr) return SNA_OK;
    cudaError_t e1 = plan->dev_blob ? cudaFree(plan->dev_blob) : cudaSuccess;
    cudaError_t e2 = plan->ws ? cudaFree(plan->ws) : cudaSuccess;
    delete plan;
    if (e1 != cudaSuccess) return cuda_fail(e1, "cudaFree");
    if (e2 != cudaSuccess) return cuda_fail(e2, "cudaFree");
    return SNA_OK;
}

sna_status_t sna_plan_check(const sna_plan_t* plan) {
    if (!plan) { set_error("plan is NULL"); return SNA_ERR_INVALID_ARG; }
    if (plan->dev_blob == nullptr) return SNA_OK;
    cudaError_t e = cudaDeviceSynchronize();
    if (e != cudaSuccess) return cuda_fail(e, "cudaDeviceSynchronize");
    int status = 0;
    e = cudaMemcpy(&status, plan->dev.dev_status, sizeof(int), cudaMemcpyDeviceToHost);
    if (e != cudaSuccess) return cuda_fail(e, "cudaMemcpy of the device status word");
    if (status != 0) {
        // reported once: the word is cleared so that the plan can be used (and checked) again
        e = cudaMemset(plan->dev.dev_status, 0, sizeof(int));
        if (e != cudaSuccess) return cuda_fail(e, "cudaMemset of the device status word");
        set_error("a kernel gave up on a bounded wait; its outputs are incomplete");
        return SNA_ERR_CUDA;
    }
    return SNA_OK;
}

sna_status_t sna_debug_exercise_bounded_wait(const sna_plan_t* plan, int polls, void* cuda_stream) {
    if (!plan || plan->dev_blob == nullptr) { set_error("needs a plan that lives on a GPU"); return SNA_ERR_INVALID_ARG; }
    if (polls < 1 || polls > 100000) { set_error("polls must be between 1 and 100000"); return SNA_ERR_INVALID_ARG; }
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev != plan->device) { set_error("the plan's device is not current"); return SNA_ERR_INVALID_ARG; }
    cudaError_t e = sna::launch_bounded_wait_probe(plan->dev, polls, (cudaStream_t)cuda_stream);
    if (e != cudaSuccess) return cuda_fail(e, "probe launch");
    return SNA_OK;
}

sna_status_t sna_plan_get_nnz(const sna_plan_t* plan, int64_t* nnz) {
    if (!plan || !nnz) { set_error("NULL argument"); return SNA_ERR_INVALID_ARG; }
    *nnz = plan->host.nnz;
    return SNA_OK;
}

sna_status_t sna_plan_get_colatitudes(const sna_plan_t* plan, double* theta_in, double* theta_out) {
    if (!plan) { set_error("plan is NULL"); return SNA_ERR_INVALID_ARG; }
    if (theta_in) std::memcpy(theta_in, plan->host.theta_in.data(), sizeof(double) * plan->host.nlat_in);
    if (theta_out) std::memcpy(theta_out, plan->host.theta_out.data(), sizeof(double) * plan->host.nlat_out);
    return SNA_OK;
}

sna_status_t sna_plan_get_quad_weights(const sna_plan_t* plan, double* omega_in) {
    if (!plan || !omega_in) { set_error("NULL argument"); return SNA_ERR_INVALID_ARG; }
    std::memcpy(omega_in, plan->host.omega.data(), sizeof(double) * plan->host.nlat_in);
    return SNA_OK;
}

sna_status_t sna_plan_get_table(const sna_plan_t* plan, int64_t* row_ptr, int32_t* lat_in, int32_t* lon_off) {
    if (!plan || !row_ptr || !lat_in || !lon_off) { set_error("NULL argument"); return SNA_ERR_INVALID_ARG; }
    const sna::HostPlan& hp = plan->host;
    int64_t n = 0;
    for (int h = 0; h < hp.nlat_out; ++h) {
        row_ptr[h] = n;
        for (int e = hp.row_ptr[h]; e < hp.row_ptr[h + 1]; ++e) {
            const sna::RingWindow& w = hp.windows[e];
            // canonical order: offsets ascending in [0, nlon_in): 0..m first, then nlon_in-m..nlon_in-1
            if (w.m < 0) {
                for (int o = 0; o < hp.nlon_in; ++o) { lat_in[n] = w.lat; lon_off[n++] = o; }
            } else {
                for (int o = 0; o <= w.m; ++o) { lat_in[n] = w.lat; lon_off[n++] = o; }
                for (int o = hp.nlon_in - w.m; o < hp.nlon_in; ++o) { lat_in[n] = w.lat; lon_off[n++] = o; }
            }
        }
    }
    row_ptr[hp.nlat_out] = n;
    return SNA_OK;
}

sna_status_t sna_plan_get_table_transposed(const sna_plan_t* plan, int64_t* row_ptr, int32_t* lat_out, int32_t* lon_off) {
    if (!plan || !row_ptr || !lat_out || !lon_off) { set_error("NULL argument"); return SNA_ERR_INVALID_ARG; }
    const sna::HostPlan& hp = plan->host;
    int64_t n = 0;
    for (int hin = 0; hin < hp.nlat_in; ++hin) {
        for (int r = 0; r < hp.ps; ++r) {
            row_ptr[(int64_t)hin * hp.ps + r] = n;
            for (int e = hp.t_row_ptr[hin]; e < hp.t_row_ptr[hin + 1]; ++e) {
                const sna::RingWindow& w = hp.t_windows[e];
                auto emit = [&](int lo, int hi) {
                    for (int o = lo; o <= hi; ++o)
                        if (o % hp.ps == r) { lat_out[n] = w.lat; lon_off[n++] = o; }
                };
                if (w.m < 0) emit(0, hp.nlon_in - 1);
                else { emit(0, w.m); emit(hp.nlon_in - w.m, hp.nlon_in - 1); }
            }
        }
    }
    row_ptr[(int64_t)hp.nlat_in * hp.ps] = n;
    return SNA_OK;
}

size_t sna_workspace_bytes(const sna_plan_t* plan, int B, int H, int C) {
    if (plan == nullptr || B <= 0 || H <= 0 || C <= 0) return 0;
    return round256(2 * stats_elems(plan, B, H) * sizeof(float));
}

int sna_forward_kernel_count(const sna_plan_t* plan, int C, int with_lse) {
    if (plan == nullptr || plan->dev_blob == nullptr || !supported_C(C)) return 0;
    if (plan->is_global || sna::dense2_global_supported(plan->dev, C)) return 1;
    return (with_lse && sna::dense2_path_chosen(plan->dev, C, 1 << 20)) ? 2 : 1;
}

// The passes that run on the dense and the band kernels, one after the other (where the dense ones do not run alone).
static bool forward_on_both(const sna_plan_t* plan, int N, int C, bool with_lse) { return with_lse && sna::dense2_path_chosen(plan->dev, C, N); }
// The dense backward kernels take the whole-ring and wide windows when they are at least a tenth of the work (measured on the
// benchmark configurations: -8 % on the dq stage at a 22 % share, -6 % at 13 %).
static bool dq_on_both(const sna_plan_t* plan, int N, int C) { return plan->dev.dense_fraction >= 0.10f && sna::dense2_path_chosen(plan->dev, C, N); }
static bool dkdv_on_both(const sna_plan_t* plan, int N, int C) { return plan->dev.n_t_dense_rows > 0 && dq_on_both(plan, N, C); }

int sna_forward_kernel_count_for(const sna_plan_t* plan, int B, int H, int C, int with_lse) {
    if (check_problem(plan, B, H, C) != SNA_OK) return 0;
    return !sna::dense2_global_chosen(plan->dev, C, B * H, sna::Pass::FORWARD) && forward_on_both(plan, B * H, C, with_lse != 0) ? 2 : 1;
}

int sna_backward_kernel_count_for(const sna_plan_t* plan, int B, int H, int C) {
    if (check_problem(plan, B, H, C) != SNA_OK) return 0;
    const int N = B * H;
    return (!sna::dense2_global_chosen(plan->dev, C, N, sna::Pass::DQ) && dq_on_both(plan, N, C) ? 2 : 1) +
           (!sna::dense2_global_chosen(plan->dev, C, N, sna::Pass::DKDV) && dkdv_on_both(plan, N, C) ? 2 : 1);
}

// out_cf: if not null, the output is wanted there too, channels first (the band kernels write it themselves)
static sna_status_t forward_into(const sna_plan_t* plan, const float* q, const float* k, const float* v, float* out,
                            float* lse, int B, int H, int C, void* cuda_stream, float* out_cf) {
    sna_status_t st = check_problem(plan, B, H, C);
    if (st != SNA_OK) return st;
    if (!q || !k || !v || !out) { set_error("q, k, v and out must not be NULL"); return SNA_ERR_INVALID_ARG; }
    if (!all_aligned(q, k, v, out) || (reinterpret_cast<uintptr_t>(lse) & 3u)) { set_error("device pointers must be 16-byte aligned"); return SNA_ERR_INVALID_ARG; }
    cudaError_t e;
    if (sna::dense2_global_chosen(plan->dev, C, B * H, sna::Pass::FORWARD)) {
        // every window is a whole ring (a global plan, or a cutoff that reaches every point): the dense kernel alone
        // produces the final out and, if asked for, lse (64x128, N = 4, without lse: 5.44 ms on the generic kernel, 0.25 ms here)
        e = sna::launch_forward_dense2(plan->dev, q, k, v, out, lse, B * H, C, (cudaStream_t)cuda_stream);
    } else if (forward_on_both(plan, B * H, C, lse != nullptr)) {
        // whole-ring and wide windows on the tcgen05 kernel (its partial result travels in out / lse), the rest on the band kernel
        e = sna::launch_forward_dense2(plan->dev, q, k, v, out, lse, B * H, C, (cudaStream_t)cuda_stream);
        if (e == cudaSuccess) e = sna::launch_forward_band(plan->dev, q, k, v, out, lse, B * H, C, true, false, (cudaStream_t)cuda_stream, out_cf);
        out_cf = nullptr;
    } else if (sna::band_path_supported(plan->dev, C) && !sna::generic_chosen(plan->dev, C, B * H, sna::Pass::FORWARD)) {
        e = sna::launch_forward_band(plan->dev, q, k, v, out, lse, B * H, C, false, false, (cudaStream_t)cuda_stream, out_cf);
        out_cf = nullptr;
    } else {
        e = sna::launch_forward_generic(plan->dev, q, k, v, out, lse, B * H, C, (cudaStream_t)cuda_stream);
    }
    if (e != cudaSuccess) return cuda_fail(e, "forward launch");
    if (out_cf != nullptr) e = sna::launch_cl_to_cf(out, out_cf, B * H, C, points_out(plan), (cudaStream_t)cuda_stream);
    if (e != cudaSuccess) return cuda_fail(e, "layout launch");
    return SNA_OK;
}

sna_status_t sna_forward_ex(const sna_plan_t* plan, const float* q, const float* k, const float* v, float* out,
                            float* lse, int B, int H, int C, void* cuda_stream) {
    return forward_into(plan, q, k, v, out, lse, B, H, C, cuda_stream, nullptr);
}

sna_status_t sna_forward(const sna_plan_t* plan, const float* q, const float* k, const float* v, float* out,
                         int B, int H, int C, void* cuda_stream) {
    return sna_forward_ex(plan, q, k, v, out, nullptr, B, H, C, cuda_stream);
}

// *_cf: if not null, the gradients are wanted there, channels first, and the channels-last buffers are scratch
static sna_status_t backward_dq_into(const sna_plan_t* plan, const float* q, const float* k, const float* v,
                             const float* dout, const float* out, const float* lse, float* dq, float* D,
                             int B, int H, int C, void* cuda_stream, float* dq_cf) {
    sna_status_t st = check_problem(plan, B, H, C);
    if (st != SNA_OK) return st;
    if (!q || !k || !v || !dout || !lse || !dq || !D) { set_error("q, k, v, dout, lse, dq and D must not be NULL"); return SNA_ERR_INVALID_ARG; }
    if (!all_aligned(q, k, v, dout, dq, out) || ((reinterpret_cast<uintptr_t>(lse) | reinterpret_cast<uintptr_t>(D)) & 3u)) { set_error("device pointers must be 16-byte aligned"); return SNA_ERR_INVALID_ARG; }
    cudaError_t e;
    if (out != nullptr && out != dq && sna::dense2_global_chosen(plan->dev, C, B * H, sna::Pass::DQ)) {
        e = sna::launch_backward_dq_dense2(plan->dev, q, k, v, dout, out, lse, dq, D, B * H, C, (cudaStream_t)cuda_stream);
    } else if (out != nullptr && out != dq && dq_on_both(plan, B * H, C)) {
        // whole-ring and wide windows on the tcgen05 kernel (its part of dq is written first), the rest is added by the band kernel
        e = sna::launch_backward_dq_dense2(plan->dev, q, k, v, dout, out, lse, dq, nullptr, B * H, C, (cudaStream_t)cuda_stream);
        if (e == cudaSuccess) e = sna::launch_backward_dq_band(plan->dev, q, k, v, dout, out, lse, dq, D, B * H, C, true, false, (cudaStream_t)cuda_stream, dq_cf);
        dq_cf = nullptr;
    } else if (out != nullptr && sna::band_path_supported(plan->dev, C) && (out == dq || !sna::generic_chosen(plan->dev, C, B * H, sna::Pass::DQ))) {
        e = sna::launch_backward_dq_band(plan->dev, q, k, v, dout, out, lse, dq, D, B * H, C, false, false, (cudaStream_t)cuda_stream, dq_cf);
        dq_cf = nullptr;
    } else {
        e = sna::launch_backward_dq_generic(plan->dev, q, k, v, dout, out, lse, dq, D, B * H, C, (cudaStream_t)cuda_stream);
    }
    if (e != cudaSuccess) return cuda_fail(e, "backward dq launch");
    if (dq_cf != nullptr) e = sna::launch_cl_to_cf(dq, dq_cf, B * H, C, points_out(plan), (cudaStream_t)cuda_stream);
    if (e != cudaSuccess) return cuda_fail(e, "layout launch");
    return SNA_OK;
}

sna_status_t sna_backward_dq(const sna_plan_t* plan, const float* q, const float* k, const float* v,
                             const float* dout, const float* out, const float* lse, float* dq, float* D,
                             int B, int H, int C, void* cuda_stream) {
    return backward_dq_into(plan, q, k, v, dout, out, lse, dq, D, B, H, C, cuda_stream, nullptr);
}

static sna_status_t backward_dkdv_into(const sna_plan_t* plan, const float* q, const float* k, const float* v,
                               const float* dout, const float* lse, const float* D, float* dk, float* dv,
                               int B, int H, int C, void* cuda_stream, float* dk_cf, float* dv_cf) {
    sna_status_t st = check_problem(plan, B, H, C);
    if (st != SNA_OK) return st;
    if (!q || !k || !v || !dout || !lse || !D || !dk || !dv) { set_error("q, k, v, dout, lse, D, dk and dv must not be NULL"); return SNA_ERR_INVALID_ARG; }
    if (!all_aligned(q, k, v, dout, dk, dv) || ((reinterpret_cast<uintptr_t>(lse) | reinterpret_cast<uintptr_t>(D)) & 3u)) { set_error("device pointers must be 16-byte aligned"); return SNA_ERR_INVALID_ARG; }
    cudaError_t e;
    if (sna::dense2_global_chosen(plan->dev, C, B * H, sna::Pass::DKDV)) {
        // the dense kernel writes only the rings some window refers to; the others get their (zero) gradient here
        const size_t ring_bytes = (size_t)plan->host.nlon_in * C * sizeof(float), pitch = ring_bytes * plan->host.nlat_in;
        for (size_t i = 0; i < plan->unvisited.size(); ++i) {
            const size_t off = ring_bytes * plan->unvisited[i];
            e = cudaMemset2DAsync((char*)dk + off, pitch, 0, ring_bytes, (size_t)B * H, (cudaStream_t)cuda_stream);
            if (e == cudaSuccess) e = cudaMemset2DAsync((char*)dv + off, pitch, 0, ring_bytes, (size_t)B * H, (cudaStream_t)cuda_stream);
            if (e != cudaSuccess) return cuda_fail(e, "clearing the gradients of input rings without windows");
        }
        e = sna::launch_backward_dkdv_dense2(plan->dev, q, k, v, dout, lse, D, dk, dv, B * H, C, (cudaStream_t)cuda_stream);
    } else if (dkdv_on_both(plan, B * H, C)) {
        // whole-ring and wide windows on the tcgen05 kernel (its part of dk, dv is written first), the band kernel adds the rest
        e = sna::launch_backward_dkdv_dense2(plan->dev, q, k, v, dout, lse, D, dk, dv, B * H, C, (cudaStream_t)cuda_stream);
        if (e == cudaSuccess) e = sna::launch_backward_dkdv_band(plan->dev, q, k, v, dout, lse, D, dk, dv, B * H, C, true, false, (cudaStream_t)cuda_stream, dk_cf, dv_cf);
        dk_cf = nullptr;
    } else if (sna::band_path_supported(plan->dev, C) && !sna::generic_chosen(plan->dev, C, B * H, sna::Pass::DKDV)) {
        e = sna::launch_backward_dkdv_band(plan->dev, q, k, v, dout, lse, D, dk, dv, B * H, C, false, false, (cudaStream_t)cuda_stream, dk_cf, dv_cf);
        dk_cf = nullptr;
    } else {
        e = sna::launch_backward_dkdv_generic(plan->dev, q, k, v, dout, lse, D, dk, dv, B * H, C, (cudaStream_t)cuda_stream);
    }
    if (e != cudaSuccess) return cuda_fail(e, "backward dk/dv launch");
    if (dk_cf != nullptr) {
        e = sna::launch_cl_to_cf(dk, dk_cf, B * H, C, points_in(plan), (cudaStream_t)cuda_stream);
        if (e == cudaSuccess) e = sna::launch_cl_to_cf(dv, dv_cf, B * H, C, points_in(plan), (cudaStream_t)cuda_stream);
        if (e != cudaSuccess) return cuda_fail(e, "layout launch");
    }
    return SNA_OK;
}

sna_status_t sna_backward_dkdv(const sna_plan_t* plan, const float* q, const float* k, const float* v,
                               const float* dout, const float* lse, const float* D, float* dk, float* dv,
                               int B, int H, int C, void* cuda_stream) {
    return backward_dkdv_into(plan, q, k, v, dout, lse, D, dk, dv, B, H, C, cuda_stream, nullptr, nullptr);
}

sna_status_t sna_backward_ex(const sna_plan_t* plan, const float* q, const float* k, const float* v,
                             const float* dout, const float* out, const float* lse, float* dq, float* dk, float* dv,
                             void* workspace, size_t workspace_bytes, int B, int H, int C, void* cuda_stream) {
    sna_status_t st = check_problem(plan, B, H, C);
    if (st != SNA_OK) return st;
    if (!q || !k || !v || !dout || !dq || !dk || !dv) { set_error("q, k, v, dout, dq, dk and dv must not be NULL"); return SNA_ERR_INVALID_ARG; }
    if (!all_aligned(q, k, v, dout, dq, dk, dv, out) || (reinterpret_cast<uintptr_t>(lse) & 3u)) { set_error("device pointers must be 16-byte aligned"); return SNA_ERR_INVALID_ARG; }
    if (workspace == nullptr || (reinterpret_cast<uintptr_t>(workspace) & 255u)) { set_error("workspace must be non-NULL and 256-byte aligned"); return SNA_ERR_INVALID_ARG; }
    if (workspace_bytes < sna_workspace_bytes(plan, B, H, C)) { set_error("workspace too small: %zu < %zu bytes", workspace_bytes, sna_workspace_bytes(plan, B, H, C)); return SNA_ERR_WORKSPACE; }
    cudaStream_t stream = (cudaStream_t)cuda_stream;
    const int N = B * H;
    float* ws_lse = (float*)workspace;
    float* ws_D = ws_lse + stats_elems(plan, B, H);
    cudaError_t e;
    const bool dense_alone = sna::dense2_global_chosen(plan->dev, C, N, sna::Pass::FORWARD);
    if (plan->is_global && (dense_alone || !sna::band_path_supported(plan->dev, C))) {
        if (lse == nullptr || out == nullptr) {
            // recompute the forward pass.  The dense dq kernel may not read out from the dq buffer, so out goes into
            // the dk buffer (written only after the dq stage) when that is large enough; otherwise only the
            // statistics are recomputed and the generic dq kernel runs.
            const bool fits = (long long)plan->host.nlat_in * plan->host.nlon_in >= (long long)plan->host.nlat_out * plan->host.nlon_out;
            if (fits && dense_alone) {
                e = sna::launch_forward_dense2(plan->dev, q, k, v, dk, ws_lse, N, C, stream);
                out = dk;
            } else {
                e = sna::launch_forward_generic(plan->dev, q, k, v, nullptr, ws_lse, N, C, stream);
                out = nullptr;
            }
            if (e != cudaSuccess) return cuda_fail(e, "statistics launch");
            lse = ws_lse;
        }
    } else if (sna::band_path_supported(plan->dev, C)) {
        if (lse == nullptr || out == nullptr) {
            // recompute the forward pass: lse into the workspace, out into the dq buffer, which the dq stage
            // reads row by row before it overwrites the same rows with dq
            // (into the dk buffer, which is written only after that stage, if the dense kernels help: they may not read out from
            // the buffer that they write dq to.  256x512 -> 128x256, N = 4: 733 -> 677 us)
            const bool fits = (long long)plan->host.nlat_in * plan->host.nlon_in >= (long long)plan->host.nlat_out * plan->host.nlon_out;
            if (fits && sna::dense2_path_chosen(plan->dev, C, N)) {
                e = sna::launch_forward_dense2(plan->dev, q, k, v, dk, ws_lse, N, C, stream);
                if (e == cudaSuccess) e = sna::launch_forward_band(plan->dev, q, k, v, dk, ws_lse, N, C, true, false, stream);
                out = dk;
            } else {
                e = sna::launch_forward_band(plan->dev, q, k, v, dq, ws_lse, N, C, false, false, stream);
                out = dq;
            }
            if (e != cudaSuccess) return cuda_fail(e, "statistics launch");
            lse = ws_lse;
        }
    } else if (lse == nullptr) {   // recompute the softmax statistics
        e = sna::launch_forward_generic(plan->dev, q, k, v, nullptr, ws_lse, N, C, stream);
        if (e != cudaSuccess) return cuda_fail(e, "statistics launch");
        lse = ws_lse;
    }
    st = sna_backward_dq(plan, q, k, v, dout, out, lse, dq, ws_D, B, H, C, cuda_stream);
    if (st != SNA_OK) return st;
    return sna_backward_dkdv(plan, q, k, v, dout, lse, ws_D, dk, dv, B, H, C, cuda_stream);
}

sna_status_t sna_backward(const sna_plan_t* plan, const float* q, const float* k, const float* v, const float* dout,
                          float* dq, float* dk, float* dv, int B, int H, int C, void* cuda_stream) {
    sna_status_t st = check_problem(plan, B, H, C);
    if (st != SNA_OK) return st;
    const size_t need = sna_workspace_bytes(plan, B, H, C);
    void* ws;
    {
        std::lock_guard<std::mutex> lock(plan->ws_mutex);
        if (plan->ws_bytes < need) {
            // a larger workspace than ever before: wait for work that may still use the old one, then replace it
            cudaError_t e = cudaDeviceSynchronize();
            if (e != cudaSuccess) return cuda_fail(e, "cudaDeviceSynchronize");
            if (plan->ws) cudaFree(plan->ws);
            plan->ws = nullptr;
            plan->ws_bytes = 0;
            e = cudaMalloc(&plan->ws, need);
            if (e != cudaSuccess) { set_error("cudaMalloc of %zu workspace bytes: %s", need, cudaGetErrorString(e)); return SNA_ERR_ALLOC; }
            plan->ws_bytes = need;
        }
        ws = plan->ws;
    }
    return sna_backward_ex(plan, q, k, v, dout, nullptr, nullptr, dq, dk, dv, ws, need, B, H, C, cuda_stream);
}

// ---- channels-first entry points --------------------------------------------------------------------------
namespace {
struct CfState { float *q, *k, *v, *out, *lse; };
size_t in_elems(const sna_plan_t* plan, int B, int H, int C) { return (size_t)B * H * plan->host.nlat_in * plan->host.nlon_in * C; }
size_t out_elems(const sna_plan_t* plan, int B, int H, int C) { return stats_elems(plan, B, H) * C; }
CfState carve_state(const sna_plan_t* plan, void* state, int B, int H, int C) {
    char* p = (char*)state;
    CfState s;
    s.q = (float*)p;   p += round256(out_elems(plan, B, H, C) * sizeof(float));
    s.k = (float*)p;   p += round256(in_elems(plan, B, H, C) * sizeof(float));
    s.v = (float*)p;   p += round256(in_elems(plan, B, H, C) * sizeof(float));
    s.out = (float*)p; p += round256(out_elems(plan, B, H, C) * sizeof(float));
    s.lse = (float*)p;
    return s;
}
}  // namespace

size_t sna_cf_state_bytes(const sna_plan_t* plan, int B, int H, int C) {
    if (!plan || B <= 0 || H <= 0 || !supported_C(C)) return 0;
    return 2 * round256(out_elems(plan, B, H, C) * sizeof(float)) + 2 * round256(in_elems(plan, B, H, C) * sizeof(float)) +
           round256(stats_elems(plan, B, H) * sizeof(float));
}

size_t sna_cf_scratch_bytes(const sna_plan_t* plan, int B, int H, int C) {
    if (!plan || B <= 0 || H <= 0 || !supported_C(C)) return 0;
    return 2 * round256(out_elems(plan, B, H, C) * sizeof(float)) + 2 * round256(in_elems(plan, B, H, C) * sizeof(float)) +
           sna_workspace_bytes(plan, B, H, C);
}

sna_status_t sna_forward_cf(const sna_plan_t* plan, const float* q_cf, const float* k_cf, const float* v_cf, float* out_cf,
                            void* state, size_t state_bytes, int B, int H, int C, void* cuda_stream) {
    sna_status_t st = check_problem(plan, B, H, C);
    if (st != SNA_OK) return st;
    if (!q_cf || !k_cf || !v_cf || !out_cf) { set_error("q, k, v and out must not be NULL"); return SNA_ERR_INVALID_ARG; }
    if (!all_aligned(q_cf, k_cf, v_cf, out_cf)) { set_error("device pointers must be 16-byte aligned"); return SNA_ERR_INVALID_ARG; }
    if (state == nullptr || (reinterpret_cast<uintptr_t>(state) & 255u)) { set_error("state must be non-NULL and 256-byte aligned"); return SNA_ERR_INVALID_ARG; }
    if (state_bytes < sna_cf_state_bytes(plan, B, H, C)) { set_error("state too small: %zu < %zu bytes", state_bytes, sna_cf_state_bytes(plan, B, H, C)); return SNA_ERR_WORKSPACE; }
    if ((long long)B * H > 65535) { set_error("the channels-first entry points take at most 65535 batch*head slices"); return SNA_ERR_UNSUPPORTED; }
    cudaStream_t stream = (cudaStream_t)cuda_stream;
    const CfState s = carve_state(plan, state, B, H, C);
    const long long p_in = (long long)plan->host.nlat_in * plan->host.nlon_in, p_out = (long long)plan->host.nlat_out * plan->host.nlon_out;
    cudaError_t e = sna::launch_cf_to_cl(q_cf, s.q, B * H, C, p_out, stream);
    if (e == cudaSuccess) e = sna::launch_cf_to_cl(k_cf, s.k, B * H, C, p_in, stream);
    if (e == cudaSuccess) e = sna::launch_cf_to_cl(v_cf, s.v, B * H, C, p_in, stream);
    if (e != cudaSuccess) return cuda_fail(e, "layout launch");
    return forward_into(plan, s.q, s.k, s.v, s.out, s.lse, B, H, C, cuda_stream, out_cf);
}

sna_status_t sna_backward_cf(const sna_plan_t* plan, const float* dout_cf, const void* state, size_t state_bytes,
                             void* scratch, size_t scratch_bytes, float* dq_cf, float* dk_cf, float* dv_cf,
                             int B, int H, int C, void* cuda_stream) {
    sna_status_t st = check_problem(plan, B, H, C);
    if (st != SNA_OK) return st;
    if (!dout_cf || !dq_cf || !dk_cf || !dv_cf) { set_error("dout, dq, dk and dv must not be NULL"); return SNA_ERR_INVALID_ARG; }
    if (!all_aligned(dout_cf, dq_cf, dk_cf, dv_cf)) { set_error("device pointers must be 16-byte aligned"); return SNA_ERR_INVALID_ARG; }
    if (state == nullptr || (reinterpret_cast<uintptr_t>(state) & 255u) || scratch == nullptr || (reinterpret_cast<uintptr_t>(scratch) & 255u)) {
        set_error("state and scratch must be non-NULL and 256-byte aligned");
        return SNA_ERR_INVALID_ARG;
    }
    if (state_bytes < sna_cf_state_bytes(plan, B, H, C) || scratch_bytes < sna_cf_scratch_bytes(plan, B, H, C)) {
        set_error("state or scratch too small: %zu / %zu bytes given, %zu / %zu needed", state_bytes, scratch_bytes,
                  sna_cf_state_bytes(plan, B, H, C), sna_cf_scratch_bytes(plan, B, H, C));
        return SNA_ERR_WORKSPACE;
    }
    if ((long long)B * H > 65535) { set_error("the channels-first entry points take at most 65535 batch*head slices"); return SNA_ERR_UNSUPPORTED; }
    cudaStream_t stream = (cudaStream_t)cuda_stream;
    const CfState s = carve_state(plan, const_cast<void*>(state), B, H, C);
    char* p = (char*)scratch;
    float* dout = (float*)p; p += round256(out_elems(plan, B, H, C) * sizeof(float));
    float* dq = (float*)p;   p += round256(out_elems(plan, B, H, C) * sizeof(float));
    float* dk = (float*)p;   p += round256(in_elems(plan, B, H, C) * sizeof(float));
    float* dv = (float*)p;   p += round256(in_elems(plan, B, H, C) * sizeof(float));
    cudaError_t e = sna::launch_cf_to_cl(dout_cf, dout, B * H, C, points_out(plan), stream);
    if (e != cudaSuccess) return cuda_fail(e, "layout launch");
    float* D = (float*)p;
    st = backward_dq_into(plan, s.q, s.k, s.v, dout, s.out, s.lse, dq, D, B, H, C, cuda_stream, dq_cf);
    if (st != SNA_OK) return st;
    return backward_dkdv_into(plan, s.q, s.k, s.v, dout, s.lse, D, dk, dv, B, H, C, cuda_stream, dk_cf, dv_cf);
}

sna_status_t sna_forward_tf32(const sna_plan_t* plan, const float* q, const float* k, const float* v, float* out,
                              float* lse, int B, int H, int C, void* cuda_stream) {
    sna_status_t st = check_problem(plan, B, H, C);
    if (st != SNA_OK) return st;
    if (!q || !k || !v || !out) { set_error("q, k, v and out must not be NULL"); return SNA_ERR_INVALID_ARG; }
    if (!all_aligned(q, k, v, out) || (reinterpret_cast<uintptr_t>(lse) & 3u)) { set_error("device pointers must be 16-byte aligned"); return SNA_ERR_INVALID_ARG; }
    if (!tf32_supported(plan, C)) { set_error("the reduced-precision variant needs C in {16, 32, 64} and nlon_out >= 32"); return SNA_ERR_UNSUPPORTED; }
    cudaError_t e = sna::launch_forward_band(plan->dev, q, k, v, out, lse, B * H, C, false, true, (cudaStream_t)cuda_stream);
    if (e != cudaSuccess) return cuda_fail(e, "forward launch");
    return SNA_OK;
}

sna_status_t sna_backward_tf32(const sna_plan_t* plan, const float* q, const float* k, const float* v,
                               const float* dout, const float* out, const float* lse, float* dq, float* dk, float* dv,
                               void* workspace, size_t workspace_bytes, int B, int H, int C, void* cuda_stream) {
    sna_status_t st = check_problem(plan, B, H, C);
    if (st != SNA_OK) return st;
    if (!q || !k || !v || !dout || !dq || !dk || !dv) { set_error("q, k, v, dout, dq, dk and dv must not be NULL"); return SNA_ERR_INVALID_ARG; }
    if (!all_aligned(q, k, v, dout, dq, dk, dv, out) || (reinterpret_cast<uintptr_t>(lse) & 3u)) { set_error("device pointers must be 16-byte aligned"); return SNA_ERR_INVALID_ARG; }
    if (workspace == nullptr || (reinterpret_cast<uintptr_t>(workspace) & 255u)) { set_error("workspace must be non-NULL and 256-byte aligned"); return SNA_ERR_INVALID_ARG; }
    if (workspace_bytes < sna_workspace_bytes(plan, B, H, C)) { set_error("workspace too small: %zu < %zu bytes", workspace_bytes, sna_workspace_bytes(plan, B, H, C)); return SNA_ERR_WORKSPACE; }
    if (!tf32_supported(plan, C)) { set_error("the reduced-precision variant needs C in {16, 32, 64} and nlon_out >= 32"); return SNA_ERR_UNSUPPORTED; }
    cudaStream_t stream = (cudaStream_t)cuda_stream;
    const int N = B * H;
    float* ws_lse = (float*)workspace;
    float* ws_D = ws_lse + stats_elems(plan, B, H);
    cudaError_t e;
    if (lse == nullptr || out == nullptr) {   // recompute the forward pass: lse into the workspace, out into the dq buffer
        e = sna::launch_forward_band(plan->dev, q, k, v, dq, ws_lse, N, C, false, true, stream);
        if (e != cudaSuccess) return cuda_fail(e, "statistics launch");
        lse = ws_lse;
        out = dq;
    }
    e = sna::launch_backward_dq_band(plan->dev, q, k, v, dout, out, lse, dq, ws_D, N, C, false, true, stream);
    if (e == cudaSuccess) e = sna::launch_backward_dkdv_band(plan->dev, q, k, v, dout, lse, ws_D, dk, dv, N, C, false, true, stream);
    if (e != cudaSuccess) return cuda_fail(e, "backward launch");
    return SNA_OK;
}

}  // extern "C"

// ---------------------------------------------------------------------------------------------------------
// Allocation-free backward pass: the scratch for the softmax statistics lives in the library image.
// ---------------------------------------------------------------------------------------------------------

// lse and D of up to SNA_STATIC_SCRATCH_MAX_POINTS output points.  In host code this name is only a handle for
// the runtime, not a device address: the address is looked up per device below and passed to the kernels.
static __device__ __align__(256) float g_static_scratch[2 * SNA_STATIC_SCRATCH_MAX_POINTS];

namespace {
constexpr int MAX_DEVICES = 64;
std::mutex g_static_scratch_mutex;
float* g_static_scratch_ptr[MAX_DEVICES] = {};

// Device address of g_static_scratch on the current device; resolved on the first call per device.
sna_status_t static_scratch_for_current_device(float** ptr_out) {
    int dev = -1;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return cuda_fail(e, "cudaGetDevice");
    if (dev < 0 || dev >= MAX_DEVICES) { set_error("device ordinal %d out of range", dev); return SNA_ERR_UNSUPPORTED; }
    std::lock_guard<std::mutex> lock(g_static_scratch_mutex);
    if (g_static_scratch_ptr[dev] == nullptr) {
        void* p = nullptr;
        e = cudaGetSymbolAddress(&p, g_static_scratch);
        if (e != cudaSuccess) return cuda_fail(e, "cudaGetSymbolAddress(static scratch)");
        if (p == nullptr) { set_error("cudaGetSymbolAddress returned a null address"); return SNA_ERR_CUDA; }
        g_static_scratch_ptr[dev] = static_cast<float*>(p);
    }
    *ptr_out = g_static_scratch_ptr[dev];
    return SNA_OK;
}
}  // namespace

extern "C" sna_status_t sna_backward_static(const sna_plan_t* plan, const float* q, const float* k, const float* v,
                                            const float* dout, float* dq, float* dk, float* dv,
                                            int B, int H, int C, void* cuda_stream) {
    sna_status_t st = check_problem(plan, B, H, C);
    if (st != SNA_OK) return st;
    const size_t points = stats_elems(plan, B, H);
    if (points > (size_t)SNA_STATIC_SCRATCH_MAX_POINTS) {
        set_error("problem has %zu output points; the static scratch of sna_backward_static holds at most %d "
                  "(use sna_backward or sna_backward_ex)", points, SNA_STATIC_SCRATCH_MAX_POINTS);
        return SNA_ERR_WORKSPACE;
    }
    float* scratch = nullptr;
    st = static_scratch_for_current_device(&scratch);
    if (st != SNA_OK) return st;
    // statistics are recomputed into the scratch (lse half, then D half); nothing needs clearing
    return sna_backward_ex(plan, q, k, v, dout, nullptr, nullptr, dq, dk, dv, scratch,
                           sizeof(float) * 2 * (size_t)SNA_STATIC_SCRATCH_MAX_POINTS, B, H, C, cuda_stream);
}


#ifdef SNA_PROF
// Profiling builds only: copies the per-role cycle counters that a -DSNA_PROF kernel left in the plan's status area.
extern "C" int sna_debug_read(const sna_plan_t* plan, long long* out, int count) {
    cudaDeviceSynchronize();
    return (int)cudaMemcpy(out, plan->dev.dev_status + 2, (size_t)count * 8, cudaMemcpyDeviceToHost);
}
#endif
