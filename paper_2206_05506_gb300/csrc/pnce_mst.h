// The fast m-sequence transform (pnce_mst.cu) as the other translation units see it.
#pragma once

#include "pnce_internal.h"

namespace pnce {

constexpr int kMstMinR = 7, kMstMaxR = 14;

// A serving batch of up to kMstBatchMax requests, passed with the launch: request i has the
// rows row0[i] .. row0[i + 1) of the batch (row0[0] = 0, ascending; the last up to the launch's
// A), N samples each from Y[i] on, and cols[i] = K*L lags per row from H[i] on.
constexpr int kMstBatchMax = 64;                 // a power of two
struct MstBatch {
    int n;
    int row0[kMstBatchMax], cols[kMstBatchMax];
    const float2* Y[kMstBatchMax];
    float2* H[kMstBatchMax];
};

// One launch: rows of y_stride elements at Y (p.lags says which lags go where in H), or,
// with dd, the rows of a serving batch, read from and written to the requests' buffers
// (contiguous lags, K*L of each request).  What follows `factors` is filled in.
struct MstLaunch {
    const float2* Y = nullptr;
    long long y_stride = 0;
    long long A = 0;
    LagMap lags{};
    float2* H = nullptr;
    const pnce_req_desc* dd = nullptr;
    const int* row_req = nullptr;
    const MstBatch* batch = nullptr;   // in host memory; in the place of Y, H, dd and row_req
    bool pdl = false;            // a programmatic dependent of the kernel before it
    long long in_flight = 0;     // rows in flight, in bytes, but a team per SM (0: all that fit)
    // a tensor-core dtype: the samples are rounded to it first, as the quantiser does, or,
    // with operand and factors, taken as the quantiser left them
    int dtype = PNCE_FP32_SIMT;
    const void* operand = nullptr;
    const float* factors = nullptr;
    const uint16_t* tab = nullptr;
    const uint16_t* lagvec = nullptr;
    int lg_parts = 0;
    int late_from = 0;           // teams of a block that start later: from this one on
    int N = 0;
    float invN = 0.f;
    unsigned magic_L = 0;
    int target = 0;              // scale target of dtype
    long long op_pitch = 0;      // bytes of an operand row
};

// Bytes of the tables for a pilot of N bits; 0 where the transform does not apply by length.
size_t mst_table_bytes(int N);
// Fills mst_table_bytes(N) bytes; false if the bits are no m-sequence.  May throw bad_alloc.
bool mst_build_tables(const uint32_t* bits_host, int N, uint16_t* out);
// The same, and the vectors u_j of the lags (N entries).
bool mst_build_tables(const uint32_t* bits_host, int N, uint16_t* out, uint16_t* lagvec);
// Describes tables that lie at tab_dev and sets the kernels' limits on the current device.
cudaError_t mst_setup(MstTables& m, const uint16_t* tab_dev, int N, int num_sms,
                      int max_smem_optin);
// Whether the tensor-core dtypes take the transform with this pilot: where it has tables,
// unless one of the switches that pick a tensor-core kernel (PNCE_TC_*) is set.
bool mst_replaces_tc(const pnce_pilot* pilot);
cudaError_t launch_mst(const MstTables& m, MstLaunch p, cudaStream_t s);
// The first of a block's teams that starts late (teams: none does); two_rounds: every team has two
// rows or more.
int mst_late_from(int r, int teams, bool two_rounds);

// Whether an estimate in a tensor-core dtype is one launch that rounds in registers.  Traced
// calls keep the quantiser as a launch of its own, so that each step is timed; the results
// are the same bits.
inline bool mst_fuses(const pnce_handle* h, const pnce_pilot* pilot) {
    return !h->trace_on && mst_replaces_tc(pilot);
}
// One estimate of A rows, y_stride elements apart, in one launch: FP32, or with dtype rounded.
inline cudaError_t launch_mst_rows(const pnce_pilot* pilot, const float2* Y, long long y_stride,
                                   long long A, const LagMap& lags, int dtype, float2* H,
                                   cudaStream_t s, long long in_flight = 0) {
    MstLaunch l;
    l.in_flight = in_flight;
    l.Y = Y;
    l.y_stride = y_stride;
    l.A = A;
    l.lags = lags;
    l.H = H;
    l.dtype = dtype;
    return launch_mst(pilot->mst, l, s);
}

}  // namespace pnce
