// Size-specialised FP32 operator passes for the transform length M = 2187
// (the reduced operator's N-size transforms at N = 2187; see fft_ct.cuh and
// passes_impl.cuh).
#include "passes_impl.cuh"

namespace ghb {

template ghb_status launch_col_ct_m<2187>(int, int, const ColArgs&, const CtTables&, cudaStream_t);
template ghb_status launch_row_ct_m<2187>(int, const RowArgs&, const CtTables&, int, cudaStream_t);

}  // namespace ghb
