// What slim_sba_search hands to the kernels of slim_sba_search.cu.
#pragma once

#include "slim_common.cuh"

namespace slim {

struct SbaParams {
    const __half* W;
    const uint16_t* order;       // groups by salience, the most salient first
    unsigned int* status;
    float* ref_m;                // [tiles][M]: m, the largest reference output y of the tile
    double* ref_s;               // [tiles][M]: sum e with e = exp(y - m)
    double2* can;                // [candidates][tiles][M]: with d = y_q - y, sum e (exp(d) - 1 - d) or a lowered log sum exp(y_q), and sum e d
    int M, N, K, G;
    int gt;                      // chunks of CW columns in a group
    int avg_bits, tiles;
    int first, candidates;       // the candidates p = first, first + 1, ... that this walk evaluates (it begins at p = 0 all the same)
    int half_weights;            // the candidates' weights are rounded to fp16
};

// Weight rows per CTA for M tokens and N rows; tiles = 2 ceil(N / rows).
int sba_rows(int M, int N);
// Enqueues a walk over the candidates: kl [candidates][M], fp64.
int sba_search_launch(const void* x, const SbaParams& p, int rows, int g, double* kl, cudaStream_t s);
// errors [candidates]: the means of kl over the tokens.
int sba_mean_launch(const double* kl, double* errors, int candidates, int M, cudaStream_t s);

}  // namespace slim
