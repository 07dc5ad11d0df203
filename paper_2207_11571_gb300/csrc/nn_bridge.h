// Interface between the solver and the forcing network (nn_*.cu).
#pragma once

#include "dg_common.h"

namespace dgnn {

// Runs the network on every element of state q (context c) and writes the forcing
// s[e][slot * n^3 + node] (float) for variables first_var .. first_var + n_vars - 1.
// flags: kFeaturesReady, the launch that formed the stage state wrote the network's features
// (nn_phase_a_features); kPhaseAFollows, the next launch of the stream is a phase A that runs
// beside the network (dg_ctx::beside_forcing) and may start as soon as the network has.
enum { kFeaturesReady = 1, kPhaseAFollows = 2 };
int nn_forcing_on_state(const nn_model* net, const dg_ctx* c, const double* q, float* s, int* first_var,
                        int* n_vars, cudaStream_t st, int flags = 0);

// Whether the network's input features of context c can be written by the launch that forms
// the stage state (the one-launch network path, every element in one tile batch, no padding
// columns); if so fills *out (the network's feature buffer, means and spreads).  The forcing
// is then evaluated with kFeaturesReady after that launch.
bool nn_phase_a_features(const nn_model* net, const dg_ctx* c, FeatureOut* out);

}  // namespace dgnn
