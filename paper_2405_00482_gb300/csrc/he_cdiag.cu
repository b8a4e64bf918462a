// he_cdiag.cu -- VFL-NN forward pass with the encrypted operand diagonally encoded (Alg. 3).
//
// The activation matrix A (m x n) is encrypted as its min(m, n) diagonals e_i (Eq. 2), and
// each weight column w_k is one plaintext p_k (w_k repeated with period n).  Column k of the
// product is  sum_i RotL(w_k, i) (x) [[e_i]]  (Sec. 5.3: no O4 at all), where the plaintext
// rotation RotL(., i) is the automorphism X -> X^(5^i) of p_k; in the NTT domain that is the
// index gather p_k[src_i(t)], so the kernel reads p_k through the gather and never key-switches.
//
// Layout: weight plaintexts transposed to [limb][coefficient][K] (Montgomery form) so that the
// K gathered values of one (coefficient, diagonal) are one contiguous row.
#include <algorithm>
#include <new>
#include <utility>
#include <vector>

#include "he_cdiag_tc.cuh"
#include "he_internal.cuh"
#include "he_ntt.cuh"

#define CD_COLS 8      // columns per lane (16 lanes cover 128 columns of one coefficient)
#define CD_WARPS 8     // warps per block (two coefficients each)
#define CD_MAX_IN 1024 // ciphertexts per launch (kernel-parameter table)
#define CD_MAX_OUT 512 // outputs per rescale launch
// The tensor cores (rings of 2^12 to 2^14, primes below 2^60: cdiag_tc_supported) take products of at
// least 8 columns and tc_min_diags diagonals (8 to 25 on the rings in use).  The whole call, tensor cores /
// integer form, in us for 2, 8, 16, 20, 24, 32 and 64 diagonals:
//   N = 2^12,    8 columns, n =   64:    60/41   62/52   63/67   63/74   64/82   65/97   68/154
//   N = 2^13,   16 columns, n =  256:   152/63  157/94 157/135 161/154 162/175 164/217  178/394
//   N = 2^13,    8 columns, n = 4096:  186/82 189/112 194/155 199/173 204/194 214/235  268/400
//   N = 2^14,    8 columns, n =   64: 476/162 488/302 497/505 506/601 515/695 525/890 558/1660
//   N = 2^14,  128 columns, n =  256: 844/587 863/748 877/970 881/1078 882/1186 891/1406 928/2279
#define CD_TC_MIN_COLS 8

struct he_cdmat {
    he_ctx *ctx;
    int64_t n, K;  // rows of W (= columns of A), columns of W
    int level;
    double scale;
    uint64_t *pt;  // [level+1][N][K], NTT + Montgomery form
    CdiagTc tc;    // the tensor-core form besides (he_cdiag_tc.cu), where products may take it
    int tc_min;    // diagonals from which they do
};

namespace {

struct CtTable {
    const uint64_t *p[CD_MAX_IN];
};
struct OutTable {
    uint64_t *p[CD_MAX_OUT];
};

// pre[k][c][u][t] = sum_i ct_i[c][u][t] * pt_k[u][src_i(t)].  Each half-warp takes one
// coefficient t (two per warp, 2 CD_WARPS per block) and its 16 lanes the CD_COLS columns
// k_base + CD_COLS l + (0..7) each, so a half-warp's gather of weight row (u, src_i(t)) is one
// contiguous run of 128 words, and each diagonal's fixed work (automorphism index, ciphertext
// loads, gather address) is shared by 16 multiply-adds per lane.  Ciphertext words are used once
// and loaded with an evict-first hint, so the weight table (read once per diagonal) stays in L2.
// Products of residues below q are summed lazy_terms(q) at a time in 128 bits (8 for 61-bit primes).
__global__ void __launch_bounds__(CD_WARPS * 32, 2) cdiag_mac_kernel(CtTable cts, int n_ct, int nl, const uint64_t *__restrict__ pt, int K,
                                                                    int k_base, uint64_t *pre, const ModConst *__restrict__ mc, int logn) {
    HE_GRID_DEP();
    const int N = 1 << logn;
    const int u = blockIdx.y;
    const uint64_t q = mc[u].q, qinv = mc[u].qinv;
    const int t = blockIdx.x * (2 * CD_WARPS) + (threadIdx.x >> 4);
    const int k0 = k_base + (threadIdx.x & 15) * CD_COLS;
    if (k0 >= K) return;  // no block-wide synchronisation below
    const int kn = K - k0 < CD_COLS ? K - k0 : CD_COLS;
    const bool vec = kn == CD_COLS && (K & 1) == 0;  // rows start 16-byte aligned when K is even
    const uint32_t two_n_mask = (2u << logn) - 1;
    u128 a0[CD_COLS], a1[CD_COLS];
    uint64_t r0[CD_COLS], r1[CD_COLS];
#pragma unroll
    for (int kk = 0; kk < CD_COLS; ++kk) a0[kk] = a1[kk] = 0, r0[kk] = r1[kk] = 0;
    // operands of diagonal i: c0, c1 at t; weights at row src_i(t)
    uint64_t c0n, c1n, pvn[CD_COLS];
    auto fetch = [&](int i, uint32_t g) {
        const uint32_t src = automorph_src(t, g, logn);
        c0n = __ldcs(cts.p[i] + (int64_t)u * N + t);
        c1n = __ldcs(cts.p[i] + ((int64_t)nl + u) * N + t);
        const uint64_t *row = pt + ((int64_t)u * N + src) * K + k0;
        if (vec) {
#pragma unroll
            for (int kk = 0; kk < CD_COLS; kk += 2) {
                const ulonglong2 v = __ldg(reinterpret_cast<const ulonglong2 *>(row + kk));
                pvn[kk] = v.x;
                pvn[kk + 1] = v.y;
            }
        } else {
#pragma unroll
            for (int kk = 0; kk < CD_COLS; ++kk) pvn[kk] = kk < kn ? __ldg(row + kk) : 0;
        }
    };
    uint32_t g = 1;
    int pending = 0;
    const int period = lazy_terms(q);  // diagonals per reduction
    for (int i = 0; i < n_ct; ++i) {
        fetch(i, g);
        g = (uint32_t)(((uint64_t)g * 5u) & two_n_mask);
#pragma unroll
        for (int kk = 0; kk < CD_COLS; ++kk) {
            a0[kk] += (u128)c0n * pvn[kk];
            a1[kk] += (u128)c1n * pvn[kk];
        }
        if (++pending == period) {
#pragma unroll
            for (int kk = 0; kk < CD_COLS; ++kk) {
                r0[kk] = add_mod(r0[kk], redc128(a0[kk], q, qinv), q);
                r1[kk] = add_mod(r1[kk], redc128(a1[kk], q, qinv), q);
                a0[kk] = a1[kk] = 0;
            }
            pending = 0;
        }
    }
    for (int kk = 0; kk < kn; ++kk) {
        r0[kk] = add_mod(r0[kk], redc128(a0[kk], q, qinv), q);
        r1[kk] = add_mod(r1[kk], redc128(a1[kk], q, qinv), q);
        uint64_t *o = pre + (int64_t)(k0 + kk) * 2 * nl * N;
        o[(int64_t)u * N + t] = r0[kk];
        o[((int64_t)nl + u) * N + t] = r1[kk];
    }
}

// encoded columns [K][nl][N] -> transposed [nl][N][K]
__global__ void transpose_cols_kernel(const uint64_t *__restrict__ in, uint64_t *out, int K, int nl, int logn) {
    HE_GRID_DEP();
    const int64_t N = 1 << logn;
    const int64_t total = (int64_t)K * nl * N;
    for (int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; idx < total; idx += (int64_t)gridDim.x * blockDim.x) {
        const int64_t k = idx % K, rest = idx / K;  // rest = u * N + t
        out[idx] = in[k * nl * N + rest];
    }
}

struct CdRescale {
    uint64_t ql, half;
    uint64_t inv[HE_MAX_Q], inv_shoup[HE_MAX_Q];
};

// CTA (k, c, j): v = centred(last limb of output k) mod q_j -> NTT -> out_k = (pre_j - v) q_l^-1
__global__ void cdiag_rescale_kernel(const uint64_t *__restrict__ pre, const uint64_t *__restrict__ last, int level, CdRescale rc, OutTable outs,
                                     int k_first, const uint64_t *__restrict__ d_tw, const ModConst *__restrict__ mc, int logn) {
    HE_GRID_DEP();
    extern __shared__ uint64_t s[];
    const int N = 1 << logn, nl = level + 1;
    const int per = 2 * level;
    const int kl = blockIdx.x / per, c = (blockIdx.x % per) / level, j = blockIdx.x % level;
    const int k = k_first + kl;
    const uint64_t q = mc[j].q;
    const uint64_t *lc = last + ((int64_t)k * 2 + c) * N;
    for (int x = threadIdx.x; x < N; x += blockDim.x) {
        uint64_t r = lc[x] + rc.half;
        if (r >= rc.ql) r -= rc.ql;
        s[SIDX(x)] = reduce_signed((int64_t)r - (int64_t)rc.half, q, mc[j].mu);
    }
    __syncthreads();
    ntt_fwd_smem(s, twiddles(d_tw, j, 0, logn), q, logn);
    const uint64_t *cj = pre + (((int64_t)k * 2 + c) * nl + j) * N;
    uint64_t *o = outs.p[kl] + ((int64_t)c * level + j) * N;
    for (int x = threadIdx.x; x < N; x += blockDim.x) o[x] = mul_shoup(sub_mod(cj[x], s[SIDX(x)], q), rc.inv[j], rc.inv_shoup[j], q);
}

// The same in two phases of small CTAs (he_ntt.cuh, NTT form 2; log N = 12..14): the columns on the
// centred last limb into the output, then the rows with the combination as their store.
template <int LOGN>
__global__ void __launch_bounds__(NTT2_THREADS, 8) cdiag_rescale_cols_kernel(const uint64_t *__restrict__ last, int level, uint64_t ql,
                                                                           const __grid_constant__ OutTable outs, int k_first,
                                                                           const uint64_t *__restrict__ d_tw, const ModConst *__restrict__ mc) {
    HE_GRID_DEP();
    constexpr int N = 1 << LOGN, TILES = (N >> 6) / NTT2_TC;
    __shared__ uint64_t sm[ntt2_cols_smem_words()];
    const int item = blockIdx.x / TILES, c0 = (blockIdx.x % TILES) * NTT2_TC;
    const int kl = item / (2 * level), c = (item / level) % 2, j = item % level;
    const uint64_t q = mc[j].q, mu = mc[j].mu, lift = mc[j].lift, half = ql / 2;
    const uint64_t *lc = last + ((int64_t)(k_first + kl) * 2 + c) * N;
    ntt2_fwd_cols<LOGN>(
        sm, [=](int64_t x) { return lc[x]; },
        [=](uint64_t v) {
            uint64_t r = v + half;
            if (r >= ql) r -= ql;
            return lift_signed((int64_t)r - (int64_t)half, q, lift, mu);
        },
        outs.p[kl] + ((int64_t)c * level + j) * N, c0, TwGlobal{twiddles(d_tw, j, 0, LOGN)}, q);
}
template <int LOGN>
__global__ void __launch_bounds__(NTT2_THREADS, 8) cdiag_rescale_rows_kernel(const uint64_t *__restrict__ pre, int level, const __grid_constant__ CdRescale rc,
                                                                           const __grid_constant__ OutTable outs, int k_first,
                                                                           const uint64_t *__restrict__ d_tw, const ModConst *__restrict__ mc) {
    HE_GRID_DEP();
    constexpr int N = 1 << LOGN, TILES = 64 / NTT2_TR;
    __shared__ uint64_t sm[ntt2_frows_smem_words(LOGN - 6)];
    const int item = blockIdx.x / TILES, b0 = (blockIdx.x % TILES) * NTT2_TR;
    const int kl = item / (2 * level), c = (item / level) % 2, j = item % level;
    const uint64_t q = mc[j].q, inv = rc.inv[j], invs = rc.inv_shoup[j];
    const uint64_t *cj = pre + (((int64_t)(k_first + kl) * 2 + c) * (level + 1) + j) * N;
    uint64_t *o = outs.p[kl] + ((int64_t)c * level + j) * N;
    ntt2_fwd_rows<LOGN>(sm, o, b0, TwGlobal{twiddles(d_tw, j, 0, LOGN)}, mc[j],
                        [=](int x, uint64_t v) { o[x] = mul_shoup(sub_mod(cj[x], v, q), inv, invs, q); });
}

// slots of the diagonals e_i[j] = A[j mod m, (i + j) mod n], repeated over the N/2 slots
__global__ void cdiag_layout_kernel(const double *__restrict__ A, int64_t m, int64_t n, int64_t slots, double *out) {
    HE_GRID_DEP();
    const int64_t lo = m < n ? m : n, hi = m < n ? n : m;
    const int64_t total = lo * slots;
    for (int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; idx < total; idx += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = idx / slots, j = (idx % slots) % hi;
        out[idx] = A[(j % m) * n + (i + j) % n];
    }
}

// weight column k repeated with period n: slots[k][s] = W[s mod n][k]
__global__ void cdiag_weights_kernel(const double *__restrict__ W, int64_t n, int64_t K, int64_t slots, double *out) {
    HE_GRID_DEP();
    const int64_t total = K * slots;
    for (int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; idx < total; idx += (int64_t)gridDim.x * blockDim.x) {
        const int64_t k = idx / slots, s = idx % slots;
        out[idx] = W[(s % n) * K + k];
    }
}

// Z[r][k] from the decrypted slots of output k: slot r (m >= n) or the sum of the n/m groups (m < n)
__global__ void cdiag_decode_kernel(const double *__restrict__ slots, int64_t m, int64_t n, int64_t K, int64_t n_slots, double *Z) {
    HE_GRID_DEP();
    const int64_t total = m * K;
    for (int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; idx < total; idx += (int64_t)gridDim.x * blockDim.x) {
        const int64_t r = idx / K, k = idx % K;
        const double *sl = slots + k * n_slots;
        double v = 0.0;
        const int64_t groups = m >= n ? 1 : n / m;
        for (int64_t g = 0; g < groups; ++g) v += sl[r + g * m];
        Z[idx] = v;
    }
}

int blocks_for(int64_t total) { return (int)std::min<int64_t>((total + 255) / 256, 65535 * 16); }

bool pow2(int64_t v) { return v > 0 && (v & (v - 1)) == 0; }

}  // namespace

extern "C" {

int he_cdiag_encode_weights(he_ctx *ctx, const double *W, int64_t n, int64_t K, int level, he_cdmat **out) {
    if (!ctx || !W || !out || !pow2(n) || n > ctx->n / 2 || K < 1 || K > (1 << 20)) return HE_EINVAL;
    if (level < 1 || level >= ctx->L) return HE_ELEVEL;
    *out = nullptr;
    he_cdmat *cm = new (std::nothrow) he_cdmat();
    if (!cm) return HE_ENOMEM;
    const int64_t N = ctx->n, nl = level + 1;
    cm->ctx = ctx;
    cm->n = n;
    cm->K = K;
    cm->level = level;
    cm->scale = (double)ctx->primes[level];
    if (cudaMalloc(&cm->pt, (size_t)nl * N * K * 8) != cudaSuccess) {
        delete cm;
        return HE_ENOMEM;
    }
    uint64_t *s = ctx_scratch(ctx, (size_t)K * (N / 2) + (size_t)K * N + (size_t)K * nl * N);
    if (!s) {
        he_cdmat_free(cm);
        return HE_ENOMEM;
    }
    double *slots = reinterpret_cast<double *>(s);
    int64_t *coef = reinterpret_cast<int64_t *>(s + K * (N / 2));
    uint64_t *cols = s + K * (N / 2) + K * N;
    LimbMap m{};
    m.n = (int)nl;
    for (int l = 0; l < nl; ++l) m.prime[l] = l;
    ctx->launches += 3;
    launch_k(cdiag_weights_kernel, blocks_for(K * (N / 2)), 256, 0, ctx->stream, W, n, K, N / 2, slots);
    launch_encode(ctx, slots, N / 2, N / 2, (int)K, cm->scale, coef);
    launch_ntt_from_int64(ctx, coef, cols, (int)K, m, 1);
    launch_k(transpose_cols_kernel, blocks_for(K * nl * N), 256, 0, ctx->stream, cols, cm->pt, (int)K, (int)nl, ctx->log_n);
    bool ok = cudaGetLastError() == cudaSuccess;
    // the weights' residues pad the columns to 128: without memory for them the integer form serves
    cm->tc_min = tc_min_diags(ctx->primes.data(), (int)nl, n, K);
    if (K >= CD_TC_MIN_COLS && n >= cm->tc_min && cdiag_tc_supported(ctx, level)) {
        const bool prepared = cdiag_tc_prepare(ctx, &cm->tc, n, K, level, cols);
        ok = ok && (cudaGetLastError() == cudaSuccess || !prepared);
    }
    if (!ok) {
        he_cdmat_free(cm);
        return HE_ECUDA;
    }
    *out = cm;
    return HE_OK;
}

void he_cdmat_free(he_cdmat *cm) {
    if (!cm) return;
    cudaStreamSynchronize(cm->ctx->stream);
    cudaFree(cm->pt);
    cdiag_tc_free(&cm->tc);
    delete cm;
}

int he_cdiag_encode_matrix(he_ctx *ctx, const double *A, int64_t m, int64_t n, double scale, int level, he_pt *outs) {
    if (!ctx || !A || !outs || !pow2(m) || !pow2(n) || std::max(m, n) > ctx->n / 2) return HE_EINVAL;
    if (level < 0 || level >= ctx->L) return HE_ELEVEL;
    const int64_t lo = std::min(m, n), N = ctx->n;
    for (int64_t i = 0; i < lo; ++i)
        if (!outs[i].data) return HE_EINVAL;
    uint64_t *s = ctx_scratch(ctx, (size_t)lo * (N / 2) + (size_t)lo * N);
    if (!s) return HE_ENOMEM;
    double *slots = reinterpret_cast<double *>(s);
    int64_t *coef = reinterpret_cast<int64_t *>(s + lo * (N / 2));
    LimbMap map{};
    map.n = level + 1;
    for (int l = 0; l <= level; ++l) map.prime[l] = l;
    ctx->launches++;
    launch_k(cdiag_layout_kernel, blocks_for(lo * (N / 2)), 256, 0, ctx->stream, A, m, n, N / 2, slots);
    launch_encode(ctx, slots, N / 2, N / 2, (int)lo, scale, coef);
    // every diagonal's transforms in one pair of launches: one launch per diagonal (7 limb-polys on 8-CTA
    // clusters at N = 2^14) took 10.9 us each, 2.8 ms for 256, with most SMs idle
    std::vector<uint64_t *> ptrs((size_t)lo);
    for (int64_t i = 0; i < lo; ++i) {
        ptrs[(size_t)i] = outs[i].data;
        outs[i].level = level;
        outs[i].scale = scale;
    }
    launch_ntt_from_int64_tab(ctx, coef, ptrs.data(), (int)lo, map);
    return cudaGetLastError() == cudaSuccess ? HE_OK : HE_ECUDA;
}

int he_cdiag_matmult(he_ctx *ctx, const he_cdmat *W, const he_ct *cts, int n_ct, he_ct *outs) {
    if (!ctx || !W || !cts || !outs || !same_family(W->ctx, ctx) || n_ct < 1 || n_ct > CD_MAX_IN || n_ct > W->n) return HE_EINVAL;
    const int level = W->level, nl = level + 1;
    for (int i = 0; i < n_ct; ++i) {
        if (!cts[i].data) return HE_EINVAL;
        if (cts[i].level != level) return HE_ELEVEL;
    }
    const int64_t K = W->K, N = ctx->n;
    for (int64_t k = 0; k < K; ++k)
        if (!outs[k].data) return HE_EINVAL;
    bool tc = W->tc.wt && n_ct >= W->tc_min;
    if (tc && wait_gave_up(ctx)) return HE_ETIMEOUT;
    const size_t w_pre = (size_t)K * 2 * nl * N, w_last = (size_t)K * 2 * N;
    // the integer form where the operands' scratch cannot be had: no memory, or a stream under capture
    const size_t w_tc = tc ? cdiag_tc_words(ctx, n_ct, level) : 0;
    if (w_pre + w_last + w_tc > ctx->scratch_words && capturing(ctx->stream)) tc = false;
    uint64_t *pre = tc ? ctx_scratch(ctx, w_pre + w_last + w_tc) : nullptr;
    if (!pre) {
        cudaGetLastError();
        tc = false;
        pre = ctx_scratch(ctx, w_pre + w_last);
    }
    if (!pre) return HE_ENOMEM;
    uint64_t *last = pre + w_pre;
    if (tc) cdiag_tc_mac(ctx, &W->tc, cts, n_ct, level, K, pre, last + w_last);
    CtTable tab;
    for (int i = 0; i < n_ct; ++i) tab.p[i] = cts[i].data;
    const int kmax = 16 * CD_COLS;  // columns per launch (16 lanes)
    for (int64_t kb = 0; kb < K && !tc; kb += kmax) {
        const dim3 grid((unsigned)(N / (2 * CD_WARPS)), (unsigned)nl);
        ctx->launches++;
        launch_k(cdiag_mac_kernel, grid, CD_WARPS * 32, 0, ctx->stream, tab, n_ct, nl, W->pt, (int)K, (int)kb, pre, ctx->d_mc, ctx->log_n);
    }
    // rescale every output: inverse NTT of the last limb of both components, then per (k, c, j)
    LimbMap lm{};
    lm.n = 1;
    lm.prime[0] = level;
    launch_ntt_inv_strided(ctx, pre + (int64_t)level * N, (int64_t)nl * N, last, N, (int)(2 * K), lm);
    CdRescale rc{};
    rc.ql = ctx->primes[level];
    rc.half = rc.ql / 2;
    for (int j = 0; j < level; ++j) {
        const uint64_t q = ctx->primes[j];
        uint64_t base = rc.ql % q, e = q - 2, r = 1;
        while (e) {
            if (e & 1) r = (uint64_t)((u128)r * base % q);
            base = (uint64_t)((u128)base * base % q);
            e >>= 1;
        }
        rc.inv[j] = r;
        rc.inv_shoup[j] = (uint64_t)(((u128)r << 64) / q);
    }
    for (int64_t kf = 0; kf < K; kf += CD_MAX_OUT) {
        const int kn = (int)std::min<int64_t>(CD_MAX_OUT, K - kf);
        OutTable ot;
        for (int k = 0; k < kn; ++k) ot.p[k] = outs[kf + k].data;
        if (use_two_phase(ctx, kn * 2 * level)) {
            const unsigned cols = (unsigned)(kn * 2 * level * ((N >> 6) / NTT2_TC)), rows = (unsigned)(kn * 2 * level * (64 / NTT2_TR));
            auto go = [&](auto L) {
                launch_k(cdiag_rescale_cols_kernel<decltype(L)::value>, cols, NTT2_THREADS, 0, ctx->stream, last, level, rc.ql, ot, (int)kf, ctx->d_tw,
                         ctx->d_mc);
                launch_k(cdiag_rescale_rows_kernel<decltype(L)::value>, rows, NTT2_THREADS, 0, ctx->stream, pre, level, rc, ot, (int)kf, ctx->d_tw, ctx->d_mc);
            };
            if (ctx->log_n == 12) go(std::integral_constant<int, 12>{});
            else if (ctx->log_n == 13) go(std::integral_constant<int, 13>{});
            else go(std::integral_constant<int, 14>{});
            ctx->launches += 2;
            continue;
        }
        ctx->launches++;
        launch_k(cdiag_rescale_kernel, kn * 2 * level, ntt_threads(ctx->log_n), ntt_smem_bytes(ctx->log_n), ctx->stream, pre, last, level, rc, ot, (int)kf, ctx->d_tw, ctx->d_mc, ctx->log_n);
    }
    const double scale = cts[0].scale * W->scale / (double)ctx->primes[level];
    for (int64_t k = 0; k < K; ++k) {
        outs[k].level = level - 1;
        outs[k].scale = scale;
    }
    return cudaGetLastError() == cudaSuccess ? HE_OK : HE_ECUDA;
}

}  // extern "C"

// Eq. 5 as read: A^T's diagonal i is RotL(e_k, r) with k = (-i) mod min(m, n) and r = i when
// m >= n, r = (-k) mod n when m < n
static void transpose_source(int64_t m, int64_t n, int64_t i, int64_t *k, int64_t *r) {
    const int64_t lo = std::min(m, n);
    *k = (lo - i) % lo;
    *r = m >= n ? i : (n - *k) % n;
}

extern "C" {

int he_cdiag_transpose_steps(int64_t m, int64_t n, int32_t *steps, int *n_steps) {
    if (!n_steps || !pow2(m) || !pow2(n) || std::max(m, n) > ((int64_t)1 << 30)) return HE_EINVAL;
    const int64_t lo = std::min(m, n);
    std::vector<int32_t> out;
    for (int64_t i = 0; i < lo; ++i) {
        int64_t k, r;
        transpose_source(m, n, i, &k, &r);
        if (r) out.push_back((int32_t)r);
    }
    std::sort(out.begin(), out.end());
    out.erase(std::unique(out.begin(), out.end()), out.end());
    if (steps)
        for (size_t t = 0; t < out.size(); ++t) steps[t] = out[t];
    *n_steps = (int)out.size();
    return HE_OK;
}

int he_cdiag_transpose(he_ctx *ctx, const he_ct *cts, int64_t m, int64_t n, he_ct *outs) {
    if (!ctx || !cts || !outs || !pow2(m) || !pow2(n) || std::max(m, n) > ctx->n / 2) return HE_EINVAL;
    const int64_t lo = std::min(m, n);
    std::vector<std::pair<int64_t, int32_t>> kr((size_t)lo);
    for (int64_t i = 0; i < lo; ++i) {
        int64_t k, r;
        transpose_source(m, n, i, &k, &r);
        kr[(size_t)i] = {k, (int32_t)r};
        if (!cts[k].data || !outs[i].data || outs[i].data == cts[k].data) return HE_EINVAL;
        if (cts[k].level != cts[0].level) return HE_ELEVEL;
    }
    // all rotations in one batch (steps that are multiples of N/2, here r = 0, are copies)
    std::vector<he_ct> ins((size_t)lo);
    std::vector<int32_t> steps((size_t)lo);
    for (int64_t i = 0; i < lo; ++i) {
        ins[(size_t)i] = cts[kr[(size_t)i].first];
        steps[(size_t)i] = kr[(size_t)i].second;
    }
    return he_rotate_many(ctx, ins.data(), steps.data(), (int)lo, outs);
}

int he_cdiag_decode(he_ctx *ctx, int64_t m, int64_t n, int64_t K, const double *slots, double *Z) {
    if (!ctx || !slots || !Z || !pow2(m) || !pow2(n) || K < 1) return HE_EINVAL;
    if (wait_gave_up(ctx)) return HE_ETIMEOUT;
    ctx->launches++;
    launch_k(cdiag_decode_kernel, blocks_for(m * K), 256, 0, ctx->stream, slots, m, n, K, ctx->n / 2, Z);
    return cudaGetLastError() == cudaSuccess ? HE_OK : HE_ECUDA;
}

}  // extern "C"

void cdiag_set_smem_limits(int max_bytes) { cudaFuncSetAttribute(cdiag_rescale_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, max_bytes); }
