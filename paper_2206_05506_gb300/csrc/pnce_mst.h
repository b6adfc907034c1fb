// The fast m-sequence transform (pnce_mst.cu) as the other translation units see it.
#pragma once

#include "pnce_internal.h"

namespace pnce {

constexpr int kMstMinR = 7, kMstMaxR = 14;

// One launch: rows of y_stride elements at Y (p.lags says which lags go where in H), or,
// with dd, the rows of a serving batch, read from and written to the requests' buffers
// (contiguous lags, K*L of each request).  tab, N, invN and magic_L are filled in.
struct MstLaunch {
    const float2* Y = nullptr;
    long long y_stride = 0;
    long long A = 0;
    LagMap lags{};
    float2* H = nullptr;
    const pnce_req_desc* dd = nullptr;
    const int* row_req = nullptr;
    bool pdl = false;            // a programmatic dependent of the kernel before it
    const uint16_t* tab = nullptr;
    int N = 0;
    float invN = 0.f;
    unsigned magic_L = 0;
};

// Bytes of the tables for a pilot of N bits; 0 where the transform does not apply by length.
size_t mst_table_bytes(int N);
// Fills mst_table_bytes(N) bytes; false if the bits are no m-sequence.  May throw bad_alloc.
bool mst_build_tables(const uint32_t* bits_host, int N, uint16_t* out);
// Describes tables that lie at tab_dev and sets the kernels' limits on the current device.
cudaError_t mst_setup(MstTables& m, const uint16_t* tab_dev, int N, int num_sms,
                      int max_smem_optin);
cudaError_t launch_mst(const MstTables& m, MstLaunch p, cudaStream_t s);

}  // namespace pnce
