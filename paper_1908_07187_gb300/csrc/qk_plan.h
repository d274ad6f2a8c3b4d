// Fused-mode queue entries and the planner interface (host only).
#pragma once

#include <complex>
#include <cstdint>
#include <functional>
#include <vector>

#include <cuda_runtime.h>

#include "qk.h"
#include "qk_kernels.cuh"

namespace qk {

// A queued unitary op in physical qubits.  U2: 2x2 matrix m on bit q where all
// cmask bits are 1.  PHASE: multiply amplitudes with (i & mask) == val by f.
struct FusedOp {
    enum Kind { U2 = 0, PHASE = 1 } kind = U2;
    int q = 0;
    uint64_t cmask = 0;
    std::complex<double> m[4];
    uint64_t mask = 0, val = 0;
    std::complex<double> f = 1.0;
    Cond cond{};
};

// A queued dense k-qubit gate in physical qubits: 2^k x 2^k device matrix on targets
// tpos[0..k-1] (tpos[0] = register MSB) where all cmask bits are 1.
struct DenseItem {
    int k = 0;
    int tpos[kDenseMaxK];
    uint64_t tmask = 0, cmask = 0;
    const void *mat = nullptr;
    Cond cond{};
};
// Group an ordered list of dense gates into passes (DenseParams); with one gate per
// call (plain mode) the pass holds that gate.
using DenseSink = std::function<qk_status(DenseParams &)>;
qk_status plan_dense(int n, int prec, const std::vector<DenseItem> &ops, const DenseSink &sink);

struct TilePlanner;
TilePlanner *make_planner();
void free_planner(TilePlanner *p);
// Plan an n-qubit (n >= 13) complex64 op list into tile passes; each pass's
// program goes to sink in order (the sink may adjust it before launching it).
// On a planner error *err names it.
using PassSink = std::function<qk_status(TileParams &)>;
qk_status plan_passes(TilePlanner *p, int n, const std::vector<FusedOp> &ops, const PassSink &sink, const char **err);
// the same as programs for tiles in shared memory (SmemTileParams), any n >= 1
using SmemPassSink = std::function<qk_status(SmemTileParams &)>;
qk_status plan_smem_passes(TilePlanner *p, int n, int prec, const std::vector<FusedOp> &ops, const SmemPassSink &sink,
                           const char **err);
// one of them with each pass launched on the context's stream: register tiles for
// complex64 from 13 qubits on, tiles in shared memory otherwise, or one launch per op
// where so few amplitudes are concerned that this is cheaper
qk_status run_fused(TilePlanner *p, qk_ctx *c, const std::vector<FusedOp> &ops);

// context hooks implemented in qk_api.cu
void *ctx_state(qk_ctx *c);
int ctx_n(qk_ctx *c);
int ctx_prec(qk_ctx *c);
int ctx_sms(qk_ctx *c);
cudaStream_t ctx_stream(qk_ctx *c);
const uint8_t *ctx_cbits(qk_ctx *c);
qk_status ctx_run_plain(qk_ctx *c, const FusedOp &op);
qk_status ctx_fail(qk_ctx *c, qk_status s, const char *msg);
void ctx_launch_begin(qk_ctx *c, int cls, double bytes, void **token);
void ctx_launch_end(void *token);

}  // namespace qk
