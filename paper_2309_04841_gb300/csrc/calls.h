// calls.h -- qaoa_simulate and qaoa_grad with the choice whether the passes over
// small vectors (n <= 20) may overlap their neighbours on the stream.  A lone call
// is faster with it (n = 18 p = 20 gradient, alone: 398 -> 306 us).  The server runs
// requests on their own streams, which fill each other's gaps instead: two such
// chains of overlapping launches gain little from running beside each other (n = 17
// and 18 through the server: together 0.77 to 0.82 of one after the other with
// overlap, 0.68 to 0.71 without).
#pragma once

#include "../../include/qaoa.h"

namespace qaoa {

qaoa_status simulate_call(int n, const void *d_costs, qaoa_cost_type ct, const qaoa_cost_stats *stats,
                          const double *gammas, const double *betas, int p, void *d_state, qaoa_state_type st,
                          int init_plus, void *d_work, size_t work_bytes, double *d_out, bool overlap,
                          qaoa_stream_t stream);
qaoa_status grad_call(int n, const void *d_costs, qaoa_cost_type ct, const qaoa_cost_stats *stats,
                      const double *gammas, const double *betas, int p, void *d_state, void *d_lambda,
                      qaoa_state_type st, void *d_work, size_t work_bytes, double *d_out, bool overlap,
                      qaoa_stream_t stream);

}  // namespace qaoa
