// FP64 forward on the tensor cores (lr_fx64.cu): eligibility, tables and launch.
#pragma once
#include "lr_internal.h"

namespace lr {
// largest tile (outputs per block) that the tensor-core kernels take for this plan's halos, bounds and
// order; 0 when they do not apply
int fx_max_tile(const FwdParams &P, int order);
// expansion nodes and transforms; max_delay bounds the projection's light times (s); precision: the plan's
void fx_tables(const FwdParams &P, int order, int precision, double max_delay, FxTab &X);
// the plan's table of merged TDI stencils over the orbit's spline pieces: its size (0: none) and its
// computation into F->mem, asynchronous (F->ready); a cudaError_t value
size_t fx_table_bytes(const FwdParams &P, int order);
int fx_table_build(const FwdParams &P, int order, FxPlan *F);
void fx_plan_free(FxPlan *F);
// the launch constants with the table, ready for kernels on `stream`; a cudaError_t value
int fx_table_for(FxPlan *F, void *stream, FxTab *X);
// returns a cudaError_t value; P.tile + P.HL + P.HR (P.tile for KIND_PROJECT) is at most FX_ROWS
int launch_fx64(int kind, int order, const FwdParams &P, int sms, void *stream);

// adjoint kernels (lr_fxbwd.cu) for plans with the table: kind 0 TDI transpose, 1 projection transpose, 2 sky
// partials, as launch_bwd; tiles of link and of strain samples hold at most fx_max_tile samples
struct BwdParams;
int launch_fx_bwd(int kind, int order, const FwdParams &P, const BwdParams &B, FxPlan *F, int sms, void *stream);
}  // namespace lr
