// What slim_sba_search hands to the kernels of slim_sba_search.cu.
#pragma once

#include "slim_common.cuh"

namespace slim {

struct SbaParams {
    const __half* W;
    const uint16_t* order;       // groups by salience, the most salient first
    unsigned int* status;
    float* ref_m;                // [tiles][M]: largest reference output of the tile
    double2* ref_s;              // [tiles][M]: sum e, sum e (y - m) with e = exp(y - m)
    float* can_m;                // [candidates][tiles][M]: largest candidate output
    double2* can_s;              // [candidates][tiles][M]: sum exp(y_q - m_q), sum e (y_q - m)
    int M, N, K, G;
    int gt;                      // chunks of CW columns in a group
    int avg_bits, first, candidates, tiles;
    int half_weights;            // the candidates' weights are rounded to fp16
};

// Weight rows per CTA for M tokens and N rows; tiles = 2 ceil(N / rows).
int sba_rows(int M, int N);
// Enqueues all candidates: kl [candidates][M] and errors [candidates], fp64.
int sba_search_launch(const void* x, const SbaParams& p, int rows, int g, double* kl, double* errors, cudaStream_t s);

}  // namespace slim
