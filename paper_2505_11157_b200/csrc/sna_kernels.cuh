// Device-side view of a plan and the launchers of the CUDA kernels.
#pragma once
#include <cuda_runtime.h>
#include <cstdint>

namespace sna {

// A band stream on the device (the host's BandStream, sna_plan.hpp).
struct DevBand {
    const int32_t* chunk_ptr;       // [stream rows + 1]
    const int4* columns;            // BAND_CHUNK per chunk
    const uint32_t* masks;          // 32 per chunk
    const int32_t* order;           // ring groups, longest stream first
    const int32_t* lengths;         // in host memory: chunks per stream row of order[i]
    int groups;
    int one_row;                    // 1: every group walks row 0 (global attention)
    long long chunks;               // of all stream rows
};

// All pointers are device memory owned by the plan.
struct DevPlan {
    int nlat_in, nlon_in, nlat_out, nlon_out, ps;
    int num_sms;                // of the plan's device
    // forward table, run-length form: windows [row_ptr[h], row_ptr[h+1]) of output latitude h
    const int32_t* row_ptr;
    const int32_t* win_lat;     // input ring
    const int32_t* win_m;       // half width in input columns, -1 = whole ring
    const int32_t* row_order;   // output latitudes, most table entries first
    // transposed table: windows [t_row_ptr[h'], t_row_ptr[h'+1]) of input latitude h'
    const int32_t* t_row_ptr;
    const int32_t* t_win_lat;   // output ring
    const int32_t* t_win_m;
    const int32_t* t_row_order; // input latitudes, most work first
    const float* log2_omega;    // [nlat_in] log2 of the per-point quadrature weight
    // band streams of the mma.sync kernels (see sna_plan.hpp): forward and transposed, each with all windows and with the ones
    // the dense kernels serve left out (null for a global plan)
    DevBand fwd, fwdb, t, tb;
    // the dense kernels' lists
    const int32_t* dense_ptr;       // [nlat_out+1] the dense kernels' windows per output latitude
    const int32_t* dense_lat;       // their input rings
    const int32_t* dense_m;         // their half widths in input columns, -1 = whole ring
    const int32_t* dense_rows;      // output latitudes with at least one such window
    int n_dense_rows;
    // the same for the transposed side (dk/dv): per input latitude, the output rings that attend to it through such a window
    const int32_t* t_dense_ptr;     // [nlat_in+1]
    const int32_t* t_dense_lat;     // output rings
    const int32_t* t_dense_m;       // half widths in input columns, -1 = whole ring
    const int32_t* t_dense_rows;    // input latitudes with at least one such output ring
    int n_t_dense_rows;
    long long dense_blocks, dense_longest;      // 128-column blocks that the tiles of one longitude range walk: all of them, the longest
    float dense_fraction;           // share of the table's entries that the dense kernels' windows cover
    int dense_all;                  // 1: they cover every one (a share that rounds to 1 may still leave narrow windows out)
    long long pairs, longest_row, longest_t_row;      // table entries of a slice; of the output point and of the input point with most
    int* dev_status;                // set to non-zero by a kernel whose bounded wait ran out
    int t_consecutive;              // 1: transposed tiles are 8 consecutive input columns; 0: split by residue mod ps
    int is_global;                  // 1: every window is a whole ring; the band streams have one row
};

// Band kernels (sna_kernels_band.cu: mma.sync; C <= 64); same contracts as the generic launchers.
// after_dense: the dense kernels have served their windows (see below) and left partial results in the output buffers; the
// band kernels walk the remaining windows and continue from those.  lp: reduced-precision variant (C = 16, 32, 64), every
// product is one FP16 MMA (operands rounded to 11 significant bits).  *_cf: if not null, the results go there in channels-first
// planes ([slices][C][points]; forward: there too); the channels-last buffers still carry the dense kernels' partial results.
cudaError_t band_prepare_device();   // once per device: opt in to the kernels' shared-memory sizes
bool band_path_supported(const DevPlan& p, int C);
cudaError_t launch_forward_band(const DevPlan& p, const float* q, const float* k, const float* v, float* out, float* lse,
                                int N, int C, bool after_dense, bool lp, cudaStream_t stream, float* out_cf = nullptr);
// out is required (D_i = dout_i . out_i); out and dq may be the same buffer unless after_dense.
cudaError_t launch_backward_dq_band(const DevPlan& p, const float* q, const float* k, const float* v, const float* dout,
                                    const float* out, const float* lse, float* dq, float* Dws, int N, int C, bool after_dense, bool lp,
                                    cudaStream_t stream, float* dq_cf = nullptr);
cudaError_t launch_backward_dkdv_band(const DevPlan& p, const float* q, const float* k, const float* v, const float* dout,
                                      const float* lse, const float* Dws, float* dk, float* dv, int N, int C, bool after_dense, bool lp,
                                      cudaStream_t stream, float* dk_cf = nullptr, float* dv_cf = nullptr);
// Dense (tcgen05) kernels (sna_kernels_dense2.cu: TMA loads, warp-specialised, operands and accumulators in TMEM) for
// the windows in the plan's dense lists: whole input rings, and wide banded windows as masked blocks.  The forward kernel
// writes the partial result (normalised out, lse) of the output latitudes in p.dense_rows and the band kernel
// continues from it with the narrower windows; both need lse != null then (alone, for a problem of whole rings only, the
// dense kernel does not).  dense2_path_chosen tells whether the pair is used for a problem of N slices.
cudaError_t dense2_prepare_device();   // once per device: opt in to the kernels' shared-memory sizes
bool dense2_path_chosen(const DevPlan& p, int C, int N);
cudaError_t launch_bounded_wait_probe(const DevPlan& p, int polls, cudaStream_t stream);
bool dense2_global_supported(const DevPlan& p, int C);   // the dense kernels can do all the work: no window is left to the band kernels
enum class Pass { FORWARD, DQ, DKDV };
bool dense2_global_chosen(const DevPlan& p, int C, int N, Pass pass);   // ... and are faster than the band kernels
cudaError_t launch_forward_dense2(const DevPlan& p, const float* q, const float* k, const float* v, float* out, float* lse,
                                  int N, int C, cudaStream_t stream);
// The same split for the dq stage: the dense kernel writes its part of dq (out and dq must be different buffers) and,
// if Dws != null, D; the band kernel adds the narrower windows' part.
cudaError_t launch_backward_dq_dense2(const DevPlan& p, const float* q, const float* k, const float* v, const float* dout,
                                      const float* out, const float* lse, float* dq, float* Dws, int N, int C, cudaStream_t stream);
// And for dk/dv: the dense kernel writes its part for the input latitudes in p.t_dense_rows, the band kernel adds the rest.
cudaError_t launch_backward_dkdv_dense2(const DevPlan& p, const float* q, const float* k, const float* v, const float* dout,
                                        const float* lse, const float* Dws, float* dk, float* dv, int N, int C, cudaStream_t stream);

// Layout changes (sna_kernels_layout.cu): [slices][C][P] channels first <-> [slices][P][C] channels last, slices <= 65535.
cudaError_t launch_cf_to_cl(const float* src, float* dst, int slices, int C, long long P, cudaStream_t stream);
cudaError_t launch_cl_to_cf(const float* src, float* dst, int slices, int C, long long P, cudaStream_t stream);

// Generic kernels (any supported C): C/4 lanes cooperate on one grid point.
bool generic_chosen(const DevPlan& p, int C, int N, Pass pass);      // they are faster than the band kernels
// forward: out and/or lse may be null (lse-only pass = softmax statistics).
cudaError_t launch_forward_generic(const DevPlan& p, const float* q, const float* k, const float* v, float* out,
                                   float* lse, int N, int C, cudaStream_t stream);
// dq pass.  lse is required.  If out != null, D_i = dout_i . out_i is used; otherwise D_i is accumulated.
// Writes dq and Dws[i] = D_i.
cudaError_t launch_backward_dq_generic(const DevPlan& p, const float* q, const float* k, const float* v,
                                       const float* dout, const float* out, const float* lse, float* dq, float* Dws,
                                       int N, int C, cudaStream_t stream);
// dk, dv gather pass over the transposed table; needs lse and D of every output point.
cudaError_t launch_backward_dkdv_generic(const DevPlan& p, const float* q, const float* k, const float* v,
                                         const float* dout, const float* lse, const float* Dws, float* dk, float* dv,
                                         int N, int C, cudaStream_t stream);

}  // namespace sna
