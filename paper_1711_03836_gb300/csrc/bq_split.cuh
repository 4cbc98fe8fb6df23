// bq_split.cuh -- launches of the hopping kernels that spread a site over eight or
// two threads (bq_split.cu), and the rules for when they are used.
#pragma once

#include "bq_internal.cuh"

// Eight threads per site. One launch: mode 0 with epilogue epi, or a CG-fused step
// (CNT_CG_MHAT, CNT_CG_MHATDAG; f.partials then takes bq_split_grid(Vh) values per sum
// and f.ticket is zero before and after). FP64 storage means the FP64 units, links of 18 reals.
void bq_split_launch(int prec, int recon, const DslashArgs &a, const CgFuse &f, bool dag, int epi, int mode,
                     cudaStream_t s);
unsigned bq_split_grid(int Vh);  // blocks of 16 sites
// Two threads per site, FP64 on the FP64 units.
void bq_pair64_launch(const DslashArgs &a, bool dag, int epi, cudaStream_t s);

// Where eight threads per site win: lattices of a few thousand sites, up to two blocks of 16
// sites per SM in FP32 / FP16 storage and three in FP64. One iteration of CG, eight threads per
// site against one (FP32, FP16) or two (FP64): V/2 = 2048 23 / 30 us FP32, 25 / 31 us FP16,
// 45 / 108 us FP64; 4096 27 / 30, 27 / 31, 66 / 109; 10368 35 / 31, 35 / 32, 143 / 133 (beyond,
// the shared-memory exchange and the half-width loads cost more than the idle SMs). Mhat^dag Mhat on either
// side of the limits: FP32 15.8 us at V/2 = 4864, 16.6 at 7000; FP64 79 us at 7296, 110 at 9800.
static inline bool bq_use_split(const bq_ctx *c, int prec) {
    if (prec == BQ_PREC_DOUBLE) return c->fp64_arith == BQ_FP64_NATIVE && c->Vh <= 16 * BQ_SMS * 3;
    return c->Vh <= 16 * BQ_SMS * 2;
}
