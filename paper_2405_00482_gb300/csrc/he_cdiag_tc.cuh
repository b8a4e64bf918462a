// he_cdiag_tc.cuh -- the tensor-core form of the ciphertext-diagonal product (he_cdiag_tc.cu).
#pragma once
#include <stdint.h>

#include "he_cdiag_tc_plan.h"
#include "he_internal.cuh"

// the weights of a he_cdmat as residues for the tensor cores
struct CdiagTc {
    unsigned char *wt = nullptr;   // blocks of 128 columns by 64 indices (cdiag_tc_weights_kernel)
    int64_t block[HE_MAX_Q] = {};  // first block of each limb
    int lg_n = 0;
};

int cdiag_tc_tables(he_ctx *ctx);  // at context creation
bool cdiag_tc_supported(const he_ctx *ctx, int level);
// tc, for weights of n >= 8 rows, from the encoded columns (device, [K][level+1][N], NTT and Montgomery
// form); false without memory for it
bool cdiag_tc_prepare(he_ctx *ctx, CdiagTc *tc, int64_t n, int64_t K, int level, const uint64_t *cols);
void cdiag_tc_free(CdiagTc *tc);
// pre [K][2][level+1][N] = the products' sums over the n_ct ciphertexts; scratch: cdiag_tc_words
void cdiag_tc_mac(he_ctx *ctx, const CdiagTc *tc, const he_ct *cts, int n_ct, int level, int64_t K, uint64_t *pre, uint64_t *scratch);
size_t cdiag_tc_words(const he_ctx *ctx, int n_ct, int level);
