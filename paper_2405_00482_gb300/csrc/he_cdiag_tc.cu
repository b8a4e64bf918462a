// he_cdiag_tc.cu -- the ciphertext-diagonal product of Alg. 3 (he_cdiag.cu) on the tensor cores.
//
//   pre[k][c][u][t] = sum_i ct_i[c][u][t] W_k[u][src_i(t)]  mod q_u
//
// The weight slots repeat with period n, so the weight polynomial is one in X^(N/2n): in
// bit-reversed NTT order its values are constant over aligned blocks of P = N/(2n) coefficients
// (the FFT keeps the other coefficients exactly zero: its first stages add and subtract equal
// values).  Numbering the blocks by the exponent +-5^j of their first point, src_i takes block j of
// an orbit to block j + i mod n.  Per (limb, orbit) the product is then a matrix product with a
// band structure: rows (c, t) of T consecutive blocks, columns k, and the shared index s = j + i,
//   pre[k][(c, t in block j)] = sum_s ct_{s-j}[c][t] W[s][k],
// with ct_i = 0 outside 0 <= i < n_ct.
//
// Residues of 40 to 61 bits meet 16-bit tensor operands through the Chinese remainder theorem (the
// moduli scheme of Ozaki, Uchino and Imamura, "Ozaki scheme II", 2025): with coprime odd moduli
// p_0, .. < 512 every operand's residue is at most 255 in magnitude, exact in bfloat16, and a sum
// of up to TC_DIAGS = 256 products stays at most 255^2 256 < 2^24, exact in the float accumulator.
// With P = prod p_i > 2.01 max|V| the integer V = sum x w follows exactly from its residues:
//   y_i = V (P/p_i)^-1 mod p_i (the factor is multiplied into the weights' residues),
//   V = sum_i y_i (P/p_i) - round(sum_i y_i / p_i) P,
// taken mod q_u term by term.  So the output is the canonical residue of the sum, the same bits as
// exact 64-bit arithmetic: 10 moduli for 40-bit primes, 15 for 60-bit ones, where limb-split
// operands would need 25 and 64 products.
//
// Two kernels per slice of tiles (a tile: 64 rows, two components by 32 coefficients):
// cdiag_tc_residues_kernel writes every modulus' operand of the slice's tiles as the swizzled
// shared-memory blocks that the tensor instruction reads, and cdiag_tc_mma_kernel multiplies them by
// the weights' residues (128 columns: the instruction's M).  A slice holds whole tiles per SM up to
// TC_SLICE_BYTES of operands (61 MB for one tile per SM at 256 diagonals and 10 moduli), so that they
// are still in L2 when the product kernel reads them.  (Converting inside the product kernel instead,
// one CTA doing both in turn, took 1.55 ms where the two kernels take 1.07: the registers of the
// reconstruction left none for the conversion, whose instructions it then waited for.)
//
// The product kernel is specialised by warp: one thread copies the weights' and the tile's blocks (bulk
// copies) through a ring of stages, one warp issues the tcgen05.mma (M 128, N 64, K 16), and 16 warps
// fold each modulus' sums from tensor memory (8 slots of 64 columns) into the reconstruction's
// registers, all three running ahead of each other by their rings.  Every CTA copies all of the weights'
// blocks for itself: the copies are not what it waits for (halves shared within a pair of CTAs took the
// same time, 1.50 against 1.49 ms for the whole call).  The results go through shared memory so that half a
// warp stores 16 rows of one column (stored from the registers, one column per lane, they took 8.5 of a
// slice's 40 us).
//
// 4096 x 256 activations (256 diagonals) by 128 columns at N = 2^14, 7 limbs: 7.5 G modular
// multiply-adds in 0.43 ms (residues: float and integer issue, 68% active) and 0.63 ms (products: short
// tensor instructions about 100 cycles apart, tensor pipe 12% active, and the start and end of each slice),
// against 6.26 ms for the 64-bit integer form (cdiag_mac_kernel), whose multiply-adds take 22 integer
// instructions each.

#include <algorithm>
#include <vector>

#include "he_cdiag_tc.cuh"
#include "he_internal.cuh"

namespace {

constexpr int TC_STAGE_BYTES = TC_A_BYTES + TC_B_BYTES;
constexpr int TC_STAGES = 6, TC_SLOTS = 8;  // ring of operand stages; accumulators in tensor memory, TC_ROWS columns each
constexpr int TC_FOLD_WARPS = 16, TC_THREADS = 32 * (2 + TC_FOLD_WARPS);
constexpr int TC_TR_WORDS = 32 * 17;        // a fold warp's transposition: 32 columns by 16 rows, one pad word
constexpr int TC_SMEM = TC_STAGES * TC_STAGE_BYTES + TC_FOLD_WARPS * TC_TR_WORDS * 8 + 8 * (2 * TC_STAGES + 2 * TC_SLOTS) + 16;
constexpr int TC_TMEM_COLS = TC_SLOTS * TC_ROWS;
constexpr int TC_RES_THREADS = 512;         // residues kernel: thread (row, octet of a chunk)

// per limb: the moduli count and the reconstruction constants
struct TcLimb {
    int32_t n_mod;
    int32_t nd;                 // signed 20-bit digits of a residue mod q: 2 below 2^40, else 3
    int32_t h[TC_MAX_MOD][3];   // (P/p_i) mod q, centred, as three signed 20-bit digits
    int32_t hk[3];              // P mod q likewise
    uint32_t init[3];           // of the digits' sums (tc_digit_init)
    int32_t inv[TC_MAX_MOD];    // (P/p_i)^-1 mod p_i
    uint64_t d40, d40_shoup;    // 2^40 mod q with its Shoup quotient
};
struct TcParams {
    TcLimb limb[HE_MAX_Q];
};
struct TcTables {
    float p[TC_MAX_MOD], pinv[TC_MAX_MOD], sh[TC_MAX_MOD][5];  // p, 1/p, 2^(14 j) mod p centred
};
constexpr TcTables tc_tables() {
    TcTables t{};
    for (int m = 0; m < TC_MAX_MOD; ++m) {
        t.p[m] = (float)TC_MODULI[m];
        t.pinv[m] = (float)(1.0 / TC_MODULI[m]);
        long v = 1;
        for (int j = 0; j < 5; ++j) {
            t.sh[m][j] = (float)(v > TC_MODULI[m] / 2 ? v - TC_MODULI[m] : v);
            v = (v << 14) % TC_MODULI[m];
        }
    }
    return t;
}
__constant__ TcTables c_tc = tc_tables();

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void mbar_init(uint32_t bar, int count) { asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory"); }
// waits for the phase's completion, at most `limit` polls (each suspended for a while by the hardware);
// once a wait gave up (ok false) none waits
__device__ __forceinline__ bool mbar_wait(uint32_t bar, int parity, bool ok, unsigned limit) {
    for (unsigned n = 0; ok && n < limit; ++n) {
        uint32_t done;
        asm volatile(
            "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(done)
            : "r"(bar), "r"(parity)
            : "memory");
        if (done) return true;
    }
    return false;
}
// shared-memory operand descriptor: K-major rows of 128 bytes, 128-byte swizzle, 8-row groups
// 1024 bytes apart
__device__ __forceinline__ uint64_t umma_desc(uint32_t addr) {
    return (uint64_t)((addr & 0x3FFFFu) >> 4) | ((uint64_t)1 << 16) | ((uint64_t)(1024 >> 4) << 32) | ((uint64_t)1 << 46) | ((uint64_t)2 << 61);
}
// float accumulator (bit 4), bfloat16 operands (bits 7, 10), both K-major, N = 64, M = 128
constexpr uint32_t TC_IDESC = (1u << 4) | (1u << 7) | (1u << 10) | ((TC_ROWS / 8) << 17) | ((TC_COLS / 16) << 24);

__device__ __forceinline__ void umma(uint32_t d, uint64_t a, uint64_t b, int accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\ttcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d), "l"(a), "l"(b),
        "r"(TC_IDESC), "r"(accumulate)
        : "memory");
}
// one lane of the calling (converged) warp
__device__ __forceinline__ bool elect_one() {
    uint32_t p;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(p));
    return p != 0;
}
// arrives on bar once the products issued so far are complete
__device__ __forceinline__ void umma_commit(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void tmem_ld16(float (&v)[16], uint32_t addr) {
    uint32_t *r = reinterpret_cast<uint32_t *>(v);
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n\t"
        "tcgen05.wait::ld.sync.aligned;"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]),
          "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(addr)
        : "memory");
}

// the first coefficient (bit-reversed position) of block j of an orbit: exponent +-5^j mod 2N
__device__ __forceinline__ int block_first(int j, int orbit, int logn, int lg_p) {
    const uint32_t mask = (2u << logn) - 1;
    uint32_t e = 1, b = 5;
    for (int x = j; x; x >>= 1) {
        if (x & 1) e = (e * b) & mask;
        b = (b * b) & mask;
    }
    if (orbit) e = (0u - e) & mask;
    return (int)((__brev((e - 1u) >> 1) >> (32 - logn)) >> lg_p) << lg_p;
}

constexpr float TC_MAGIC = 12582912.0f;  // 1.5 2^23: adding it rounds to an integer
// t - p round(t / p) for an integer |t| < 2^24, in [-p/2 - 1, p/2 + 1] (exact: p round(t/p) < 2^24 too)
__device__ __forceinline__ float mod_centred(float t, float p, float pinv) {
    const float m = __fadd_rn(__fmaf_rn(t, pinv, TC_MAGIC), -TC_MAGIC);
    return __fmaf_rn(-p, m, t);
}
// PC 14-bit pieces of x as floats
template <int PC>
__device__ __forceinline__ void split14(float (&a)[PC], uint64_t x) {
    const uint32_t lo = (uint32_t)x, hi = (uint32_t)(x >> 32);
#pragma unroll
    for (int j = 0; j < PC; ++j) {
        const int s = 14 * j;
        const uint32_t w = s < 32 ? __funnelshift_r(lo, hi, s) : hi >> (s - 32);
        a[j] = __fadd_rn(__uint_as_float((w & 0x3FFFu) | 0x4B000000u), -8388608.0f);
    }
}
// x mod p_m centred from its pieces: |t| <= 2^14 (1 + 255 (PC - 1)) < 2^24 before the reduction
template <int PC>
struct TcMod {
    float p, pinv, sh[PC];
    __device__ __forceinline__ explicit TcMod(int m) : p(c_tc.p[m]), pinv(c_tc.pinv[m]) {
#pragma unroll
        for (int j = 1; j < PC; ++j) sh[j] = c_tc.sh[m][j];
    }
    __device__ __forceinline__ float operator()(const float (&a)[PC]) const {
        float t = a[0];
#pragma unroll
        for (int j = 1; j < PC; ++j) t = __fmaf_rn(a[j], sh[j], t);
        return mod_centred(t, p, pinv);
    }
};
// two small integers as bfloat16 (exact: at most 8 significant bits, so the upper halves hold them)
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) { return __byte_perm(__float_as_uint(lo), __float_as_uint(hi), 0x7632); }

struct TcGeom {
    const uint64_t *ct[TC_DIAGS];  // this pass's ciphertexts i0 .. i0 + cnt
    int32_t cnt, i0, nl, K, logn, lg_n, accumulate;
    int32_t first, tiles;          // this slice's tiles, numbered over (limb, row tile)
    int32_t chunks;                // 64-wide chunks of the longest window
    uint32_t wait_limit;           // of the product kernel's waits (mbar_wait)
    int64_t tile_bytes;            // operand blocks of a tile: [modulus][chunk][64 rows x 128 bytes]
};

// a row tile of a limb: T = 32 / P consecutive blocks of P coefficients, or 32 of a block's P
struct TcTile {
    int u, orbit, j0, p0, lg_p, lg_pt, s0;  // s0: the window's first index
    int step0, step1;                       // the window's 16-wide steps that hold diagonals
};
__device__ __forceinline__ TcTile tc_tile_of(const TcGeom &g, int tile) {
    TcTile t;
    const int rt = tile & ((1 << (g.logn - 5)) - 1);
    t.u = tile >> (g.logn - 5);
    t.lg_p = g.logn - 1 - g.lg_n;
    t.lg_pt = t.lg_p < 5 ? t.lg_p : 5;
    const int lg_t = 5 - t.lg_pt, lg_sub = t.lg_p - t.lg_pt, lg_orbit = g.lg_n - lg_t + lg_sub;
    t.orbit = rt >> lg_orbit;
    const int in_orbit = rt & ((1 << lg_orbit) - 1);
    t.j0 = (in_orbit >> lg_sub) << lg_t;
    t.p0 = (in_orbit & ((1 << lg_sub) - 1)) << t.lg_pt;
    // the window starts at a whole chunk of the weights, at or before the tile's first block, and holds
    // the diagonals of its last block
    const int j_first = t.j0 + g.i0, j_last = j_first + (1 << lg_t) - 1;
    t.s0 = j_first & ~(TC_KC - 1);
    t.step0 = (j_first - t.s0) >> 4;
    t.step1 = (j_last - t.s0 + g.cnt + 15) >> 4;
    return t;
}
__device__ __forceinline__ int tc_block(const TcGeom &g, const TcTile &t, int tau) {
    return block_first((t.j0 + tau) & ((1 << g.lg_n) - 1), t.orbit, g.logn, t.lg_p) + t.p0;
}

// One CTA per (tile, chunk).  Four lanes by eight octets of a warp share four rows of a chunk: a load reads
// whole 32-byte sectors of eight ciphertexts, a store whole 128-byte operand rows.
template <int PC>
__device__ __forceinline__ void tc_residues(const TcGeom &g, const TcTile &t, int n_mod, const uint64_t *const *ct, unsigned char *out) {
    const int lane = threadIdx.x & 31, row = (threadIdx.x >> 5) * 4 + (lane & 3), oct = lane >> 2;
    const int tau = (row & 31) >> t.lg_pt;
    const int64_t src = ((int64_t)(row >> 5) * g.nl + t.u) * ((int64_t)1 << g.logn) + tc_block(g, t, tau) + (row & ((1 << t.lg_pt) - 1));
    const int shift = t.s0 - (t.j0 + tau) - g.i0;  // diagonal of the window's index kappa: kappa + shift
    out += row * 128 + ((oct ^ (row & 7)) << 4);
    const int c = blockIdx.y;
    if ((c * 4 + oct / 2) < t.step0 || (c * 4 + oct / 2) >= t.step1) return;  // octets of other steps are never read
    const int i = c * TC_KC + oct * 8 + shift;
    uint64_t x[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) {
        const bool in = (unsigned)(i + e) < (unsigned)g.cnt;
        x[e] = in ? __ldcs(ct[i + e] + src) : 0;
    }
    float a[8][PC];
#pragma unroll
    for (int e = 0; e < 8; ++e) split14<PC>(a[e], x[e]);
    out += (int64_t)c * TC_B_BYTES;
#pragma unroll 1
    for (int m = 0; m < n_mod; ++m, out += (int64_t)g.chunks * TC_B_BYTES) {
        const TcMod<PC> mod(m);
        uint32_t o[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) o[e] = pack_bf16(mod(a[2 * e]), mod(a[2 * e + 1]));
        *reinterpret_cast<uint4 *>(out) = make_uint4(o[0], o[1], o[2], o[3]);
    }
}
__global__ void __launch_bounds__(TC_RES_THREADS, 2) cdiag_tc_residues_kernel(const __grid_constant__ TcGeom g, const TcLimb *__restrict__ limbs, unsigned char *X) {
    HE_GRID_DEP();
    __shared__ const uint64_t *ct[TC_DIAGS];
    for (int i = threadIdx.x; i < g.cnt; i += TC_RES_THREADS) ct[i] = g.ct[i];
    __syncthreads();
    const TcTile t = tc_tile_of(g, g.first + blockIdx.x);
    const TcLimb &lb = limbs[t.u];
    unsigned char *out = X + blockIdx.x * g.tile_bytes;
    if (lb.nd == 2) tc_residues<3>(g, t, lb.n_mod, ct, out);
    else tc_residues<5>(g, t, lb.n_mod, ct, out);
}

// the limit of the product kernel's waits: a constant unless he_set_wait_limit shortened them.  (Read at
// run time by every wait, it cost 20 us of 1480 at 256 diagonals by 128 columns, N = 2^14.)
template <bool SHORT>
__device__ __forceinline__ unsigned tc_wait_limit(const TcGeom &g) {
    return SHORT ? g.wait_limit : HE_WAIT_LIMIT;
}

// folds a unit's sums: the thread's 16 outputs are column 32 (warp % 4) + lane, rows 16 (fw / 4) + r
template <int ND, bool SHORT>
__device__ __forceinline__ bool tc_fold(const TcGeom &g, const TcTile &t, int kb, const TcLimb &lb, const ModConst &mc, uint64_t *pre, uint32_t tmem,
                                        uint32_t acc_full, uint32_t acc_empty, uint64_t *tr, uint32_t &slot_it) {
    const unsigned limit = tc_wait_limit<SHORT>(g);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, part = (warp - 2) >> 2;
    const uint32_t lanes = (uint32_t)(warp & 3) << 21;  // the warp's quarter of the tensor-memory lanes
    uint32_t dig[ND][16];
    float frac[16];
#pragma unroll
    for (int r = 0; r < 16; ++r) {
        frac[r] = 0.0f;
#pragma unroll
        for (int d = 0; d < ND; ++d) dig[d][r] = lb.init[d];
    }
    bool ok = true;
    for (int m = 0; m < lb.n_mod && ok; ++m, ++slot_it) {
        const uint32_t slot = slot_it % TC_SLOTS;
        ok = mbar_wait(acc_full + 8 * slot, (int)((slot_it / TC_SLOTS) & 1), ok, limit);
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        float v[16];
        tmem_ld16(v, tmem + slot * TC_ROWS + (uint32_t)part * 16 + lanes);
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncwarp();
        if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(acc_empty + 8 * slot) : "memory");
        const float p = c_tc.p[m], pinv = c_tc.pinv[m];
        int32_t h[ND];
#pragma unroll
        for (int d = 0; d < ND; ++d) h[d] = lb.h[m][d];
#pragma unroll
        for (int r = 0; r < 16; ++r) {
            const float y = mod_centred(v[r], p, pinv);
            frac[r] = __fmaf_rn(y, pinv, frac[r]);
            const uint32_t yb = __float_as_uint(__fadd_rn(y, TC_MAGIC));
#pragma unroll
            for (int d = 0; d < ND; ++d) dig[d][r] = tc_digit_add(dig[d][r], yb, h[d]);
        }
    }
    // V mod q = dig0 + dig1 2^20 + dig2 2^40 - round(frac) (P mod q)
    const uint64_t q = mc.q, mu = mc.mu;
#pragma unroll
    for (int r = 0; r < 16; ++r) {
        const int k = __float2int_rn(frac[r]);
        const int64_t lo = (int64_t)(int32_t)dig[0][r] - (int64_t)k * lb.hk[0] + (((int64_t)(int32_t)dig[1][r] - (int64_t)k * lb.hk[1]) << 20);
        uint64_t v = reduce_signed(lo, q, mu);
        if constexpr (ND == 3) {
            const int64_t h = (int64_t)(int32_t)dig[2][r] - (int64_t)k * lb.hk[2];
            const uint64_t hv = mul_shoup((uint64_t)(h < 0 ? -h : h), lb.d40, lb.d40_shoup, q);
            v = h < 0 ? sub_mod(v, hv, q) : add_mod(v, hv, q);
        }
        tr[lane * 17 + r] = v;
    }
    // through shared memory, so that half a warp stores the 16 rows of a column: whole sectors
    __syncwarp();
    if (ok) {
        const int64_t N = (int64_t)1 << g.logn;
        const int row = 16 * part + (lane & 15), rr = row & 31;
        uint64_t *o = pre + (int64_t)(row >> 5) * g.nl * N + (int64_t)t.u * N + tc_block(g, t, rr >> t.lg_pt) + (rr & ((1 << t.lg_pt) - 1));
#pragma unroll 4
        for (int i = 0; i < 16; ++i) {
            const int c = 2 * i + (lane >> 4), col = kb * TC_COLS + 32 * (warp & 3) + c;
            if (col < g.K) {
                const uint64_t v = tr[c * 17 + (lane & 15)];
                uint64_t *d = o + (int64_t)col * 2 * g.nl * N;
                *d = g.accumulate ? add_mod(*d, v, q) : v;
            }
        }
    }
    __syncwarp();
    return ok;
}

// Units: the slice's tiles by blocks of 128 columns; neighbouring CTAs take consecutive tiles (same limb,
// orbit and nearly the same window), so the weights' blocks that each copies for itself come from L2.
template <bool SHORT>
__global__ void __launch_bounds__(TC_THREADS, 1) cdiag_tc_mma_kernel(const __grid_constant__ TcGeom g, const __grid_constant__ CdiagTc tc,
                                                                     const TcLimb *__restrict__ limbs, const unsigned char *__restrict__ X, uint64_t *pre,
                                                                     const ModConst *__restrict__ mc, unsigned int *gave_up) {
    HE_GRID_LAUNCH();
    extern __shared__ __align__(1024) unsigned char smem_tc[];  // the swizzle repeats every 1024 bytes
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem_tc + TC_STAGES * TC_STAGE_BYTES) + TC_FOLD_WARPS * TC_TR_WORDS;
    const uint32_t full = smem_u32(bars), empty = full + 8 * TC_STAGES, acc_full = empty + 8 * TC_STAGES, acc_empty = acc_full + 8 * TC_SLOTS,
                   tmem_slot = acc_empty + 8 * TC_SLOTS, drained = tmem_slot + 8;
    const uint32_t full_stage = smem_u32(smem_tc);
    const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;  // warp-uniform
    if (threadIdx.x == 0) {
        for (int i = 0; i < TC_STAGES; ++i) {
            mbar_init(full + 8 * i, 1);
            mbar_init(empty + 8 * i, 1);
        }
        for (int i = 0; i < TC_SLOTS; ++i) {
            mbar_init(acc_full + 8 * i, 1);
            mbar_init(acc_empty + 8 * i, TC_FOLD_WARPS);
        }
        mbar_init(drained, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");  // for the copies' and products' arrivals
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(tmem_slot), "n"(TC_TMEM_COLS) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = *reinterpret_cast<volatile uint32_t *>(bars + 2 * TC_STAGES + 2 * TC_SLOTS);
    HE_GRID_WAIT();
    const int col_blocks = (g.K + TC_COLS - 1) / TC_COLS, units = g.tiles * col_blocks;
    const unsigned limit = tc_wait_limit<SHORT>(g);
    bool ok = true;
    if (warp == 0) {
        if (lane == 0) {  // copies
            asm volatile("fence.proxy.async;" ::: "memory");  // the residues were written through the generic proxy
            uint32_t it = 0;
            for (int unit = blockIdx.x; unit < units && ok; unit += gridDim.x) {
                const int lt = unit % g.tiles, kb = unit / g.tiles;
                const TcTile t = tc_tile_of(g, g.first + lt);
                const int n_mod = limbs[t.u].n_mod, wchunks = max(1, (1 << g.lg_n) / TC_KC);
                const unsigned char *w = tc.wt + tc.block[t.u] * TC_A_BYTES;
                const unsigned char *x = X + lt * g.tile_bytes;
                for (int m = 0; m < n_mod && ok; ++m)
                    for (int c = t.step0 / 4; c * 4 < t.step1 && ok; ++c, ++it) {
                        const uint32_t st = it % TC_STAGES;
                        if (it >= TC_STAGES) ok = mbar_wait(empty + 8 * st, (int)((it / TC_STAGES - 1) & 1), ok, limit);
                        if (!ok) break;
                        const uint32_t bar = full + 8 * st, A = full_stage + st * TC_STAGE_BYTES;
                        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(TC_STAGE_BYTES) : "memory");
                        const int64_t b = ((int64_t)(2 * m + t.orbit) * col_blocks + kb) * wchunks + ((t.s0 / TC_KC + c) & (wchunks - 1));
                        asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(A),
                                     "l"(w + b * TC_A_BYTES), "r"(TC_A_BYTES), "r"(bar)
                                     : "memory");
                        asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(A + TC_A_BYTES),
                                     "l"(x + ((int64_t)m * g.chunks + c) * TC_B_BYTES), "r"(TC_B_BYTES), "r"(bar)
                                     : "memory");
                    }
            }
            // no copy may land after this CTA: where a wait gave up, here or in the other warps, nobody else
            // waits for the last ones (otherwise they are long complete)
            for (uint32_t i = it < TC_STAGES ? 0 : it - TC_STAGES; i < it; ++i)
                if (!mbar_wait(full + 8 * (i % TC_STAGES), (int)((i / TC_STAGES) & 1), true, HE_WAIT_LIMIT)) ok = false;
        }
    } else if (warp == 1) {
        // products: the whole warp walks the rings, one elected lane issues, so that descriptors and
        // addresses stay warp-uniform
        uint32_t it = 0, slot_it = 0;
        for (int unit = blockIdx.x; unit < units && ok; unit += gridDim.x) {
            const TcTile t = tc_tile_of(g, g.first + unit % g.tiles);
            const int n_mod = limbs[t.u].n_mod;
            for (int m = 0; m < n_mod && ok; ++m, ++slot_it) {
                const uint32_t slot = slot_it % TC_SLOTS, d = tmem + slot * TC_ROWS;
                if (slot_it >= TC_SLOTS) ok = mbar_wait(acc_empty + 8 * slot, (int)((slot_it / TC_SLOTS - 1) & 1), ok, limit);
                for (int c = t.step0 / 4; c * 4 < t.step1 && ok; ++c, ++it) {
                    const uint32_t st = it % TC_STAGES;
                    ok = mbar_wait(full + 8 * st, (int)((it / TC_STAGES) & 1), ok, limit);
                    if (!ok) break;
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    const uint32_t A = full_stage + st * TC_STAGE_BYTES;
                    const uint64_t da = umma_desc(A), db = umma_desc(A + TC_A_BYTES);
                    if (elect_one()) {
#pragma unroll
                        for (int k = 0; k < 4; ++k)
                            if (c * 4 + k >= t.step0 && c * 4 + k < t.step1) umma(d, da + 2 * k, db + 2 * k, c * 4 + k > t.step0);
                        umma_commit(empty + 8 * st);
                        if ((c + 1) * 4 >= t.step1) umma_commit(acc_full + 8 * slot);
                    }
                    __syncwarp();
                }
            }
        }
        // likewise the products: none may write tensor memory that has been given back
        if (elect_one()) umma_commit(drained);
        __syncwarp();
        if (!mbar_wait(drained, 0, true, HE_WAIT_LIMIT)) ok = false;
    } else {
        uint32_t slot_it = 0;
        uint64_t *tr = bars - (TC_FOLD_WARPS - (warp - 2)) * TC_TR_WORDS;
        for (int unit = blockIdx.x; unit < units && ok; unit += gridDim.x) {
            const TcTile t = tc_tile_of(g, g.first + unit % g.tiles);
            const TcLimb &lb = limbs[t.u];
            if (lb.nd == 2) ok = tc_fold<2, SHORT>(g, t, unit / g.tiles, lb, mc[t.u], pre, tmem, acc_full, acc_empty, tr, slot_it);
            else ok = tc_fold<3, SHORT>(g, t, unit / g.tiles, lb, mc[t.u], pre, tmem, acc_full, acc_empty, tr, slot_it);
        }
    }
    // every copy and product is complete: the tensor memory is free
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncwarp();
    if (__syncthreads_or(!ok) && threadIdx.x == 0) atomicAdd_system(gave_up, 1u);
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "n"(TC_TMEM_COLS) : "memory");
}

// The weights' residues (W_k(block s) centred) (P/p_i)^-1 mod p_i, centred, as bfloat16, in blocks
// [limb][modulus][orbit][128 columns][64 indices s] laid out as the tensor instruction reads them
// (rows of 128 bytes, swizzled); s runs over a period n (at least 64: shorter periods repeat),
// columns past K are zero.  cols: the encoded columns [K][nl][N], NTT and Montgomery form.
__global__ void __launch_bounds__(256) cdiag_tc_weights_kernel(const uint64_t *__restrict__ cols, int K, int nl, int logn, const TcLimb *__restrict__ limbs,
                                                               const __grid_constant__ CdiagTc tc, const ModConst *__restrict__ mc) {
    HE_GRID_DEP();
    const int N = 1 << logn, n = 1 << tc.lg_n, lg_p = logn - 1 - tc.lg_n, wchunks = gridDim.x;
    const int orbit = blockIdx.y & 1, u = blockIdx.y >> 1, kb = blockIdx.z;
    const TcLimb &lb = limbs[u];
    const uint64_t q = mc[u].q, qinv = mc[u].qinv;
    const int s = threadIdx.x & 63;
    const int at = block_first((blockIdx.x * TC_KC + s) & (n - 1), orbit, logn, lg_p);
    unsigned char *o = tc.wt + (tc.block[u] + ((int64_t)orbit * gridDim.z + kb) * wchunks + blockIdx.x) * TC_A_BYTES + 2 * (s & 7);
    for (int c = threadIdx.x >> 6; c < TC_COLS; c += 4) {
        const int k = kb * TC_COLS + c;
        const uint64_t x = k < K ? redc(0, cols[((int64_t)k * nl + u) * N + at], q, qinv) : 0;
        const bool neg = x > q / 2;
        float a[5];
        split14<5>(a, neg ? q - x : x);
        unsigned char *d = o + c * 128 + (((s >> 3) ^ (c & 7)) << 4);
        for (int m = 0; m < lb.n_mod; ++m) {
            const TcMod<5> mod(m);
            float r = mod_centred(mod(a) * (float)lb.inv[m], mod.p, mod.pinv);
            if (neg) r = -r;
            *reinterpret_cast<uint16_t *>(d + (int64_t)m * 2 * gridDim.z * wchunks * TC_A_BYTES) = (uint16_t)(__float_as_uint(r) >> 16);
        }
    }
}

// ---- host side ----
uint64_t hinv_mod(uint64_t a, uint64_t p) {  // p small, a coprime to p
    for (uint64_t x = 1; x < p; ++x)
        if (a * x % p == 1) return x;
    return 0;
}
// nd signed 20-bit digits of a residue centred mod q < 2^(20 nd)
void digits20(int32_t (&d)[3], uint64_t v, uint64_t q, int nd) {
    int64_t c = v > q / 2 ? (int64_t)(v - q) : (int64_t)v;
    d[0] = d[1] = d[2] = 0;
    for (int j = 0; j < nd; ++j) {
        int64_t r = c & 0xFFFFF;
        if (r >= 0x80000) r -= 0x100000;
        if (j == nd - 1) r = c;  // the last digit keeps what is left, at most 2^19 in magnitude
        d[j] = (int32_t)r;
        c = (c - r) >> 20;
    }
}

}  // namespace

bool cdiag_tc_supported(const he_ctx *ctx, int level) {
    if (ctx->log_n < 12 || ctx->log_n > 14) return false;
    for (int u = 0; u <= level; ++u)
        if (!tc_moduli(ctx->primes[u])) return false;
    return true;
}

// the reconstruction constants of every prime of Q, shared by the context's family
int cdiag_tc_tables(he_ctx *ctx) {
    if (ctx->log_n < 12 || ctx->log_n > 14) return HE_OK;
    std::vector<TcLimb> limbs(ctx->L);
    for (int u = 0; u < ctx->L; ++u) {
        const uint64_t q = ctx->primes[u];
        TcLimb &lb = limbs[u];
        lb = TcLimb{};
        lb.n_mod = tc_moduli(q);
        lb.nd = q < (1ull << 40) ? 2 : 3;
        uint64_t pq = 1;
        for (int m = 0; m < lb.n_mod; ++m) pq = (uint64_t)((u128)pq * TC_MODULI[m] % q);
        digits20(lb.hk, pq, q, lb.nd);
        for (int m = 0; m < lb.n_mod; ++m) {
            uint64_t h = 1, hp = 1;
            for (int j = 0; j < lb.n_mod; ++j)
                if (j != m) {
                    h = (uint64_t)((u128)h * TC_MODULI[j] % q);
                    hp = hp * TC_MODULI[j] % TC_MODULI[m];
                }
            digits20(lb.h[m], h, q, lb.nd);
            lb.inv[m] = (int32_t)hinv_mod(hp, TC_MODULI[m]);
            for (int d = 0; d < 3; ++d) lb.init[d] = tc_digit_init(lb.init[d], lb.h[m][d]);
        }
        lb.d40 = (uint64_t)(((u128)1 << 40) % q);
        lb.d40_shoup = (uint64_t)(((u128)lb.d40 << 64) / q);
    }
    void *d = nullptr;
    if (cudaMalloc(&d, sizeof(TcLimb) * ctx->L) != cudaSuccess) return HE_ENOMEM;
    ctx->sh->owned[6] = ctx->d_tc = d;
    return he_check(cudaMemcpy(d, limbs.data(), sizeof(TcLimb) * ctx->L, cudaMemcpyHostToDevice));
}

bool cdiag_tc_prepare(he_ctx *ctx, CdiagTc *tc, int64_t n, int64_t K, int level, const uint64_t *cols) {
    const int nl = level + 1;
    tc->lg_n = 0;
    while (((int64_t)1 << tc->lg_n) < n) ++tc->lg_n;
    const int col_blocks = (int)((K + TC_COLS - 1) / TC_COLS), wchunks = (int)std::max<int64_t>(1, n / TC_KC);
    int64_t blocks = 0;
    for (int u = 0; u < nl; ++u) {
        tc->block[u] = blocks;
        blocks += (int64_t)tc_moduli(ctx->primes[u]) * 2 * col_blocks * wchunks;
    }
    if (cudaMalloc(&tc->wt, (size_t)blocks * TC_A_BYTES) != cudaSuccess) {
        tc->wt = nullptr;
        return false;
    }
    ctx->launches++;
    launch_k(cdiag_tc_weights_kernel, dim3((unsigned)wchunks, (unsigned)(2 * nl), (unsigned)col_blocks), 256, 0, ctx->stream, cols, (int)K, nl, ctx->log_n,
             (const TcLimb *)ctx->d_tc, *tc, (const ModConst *)ctx->d_mc);
    return true;
}

void cdiag_tc_free(CdiagTc *tc) {
    cudaFree(tc->wt);
    tc->wt = nullptr;
}

static int tc_max_moduli(const he_ctx *ctx, int level) {
    int mods = 0;
    for (int u = 0; u <= level; ++u) mods = std::max(mods, tc_moduli(ctx->primes[u]));
    return mods;
}
size_t cdiag_tc_words(const he_ctx *ctx, int n_ct, int level) {
    return (size_t)tc_scratch_bytes(ctx->sms, (level + 1) * (ctx->n / 32), tc_max_moduli(ctx, level), n_ct) / 8;
}

void cdiag_tc_mac(he_ctx *ctx, const CdiagTc *tc, const he_ct *cts, int n_ct, int level, int64_t K, uint64_t *pre, uint64_t *scratch) {
    const int nl = level + 1, col_blocks = (int)((K + TC_COLS - 1) / TC_COLS), all = nl * (ctx->n / 32), mods = tc_max_moduli(ctx, level);
    unsigned char *X = reinterpret_cast<unsigned char *>(scratch);
    const TcLimb *limbs = static_cast<const TcLimb *>(ctx->d_tc);
    for (int i0 = 0; i0 < n_ct; i0 += TC_DIAGS) {
        TcGeom g{};
        const TcPass pass = tc_pass(ctx->sms, mods, n_ct, i0);
        g.cnt = pass.cnt;
        g.i0 = i0;
        g.nl = nl;
        g.K = (int)K;
        g.logn = ctx->log_n;
        g.lg_n = tc->lg_n;
        g.accumulate = i0 > 0;
        g.wait_limit = ctx->wait_limit;
        g.chunks = pass.chunks;
        g.tile_bytes = pass.tile_bytes;
        for (int i = 0; i < g.cnt; ++i) g.ct[i] = cts[i0 + i].data;
        for (g.first = 0; g.first < all; g.first += pass.slice) {
            g.tiles = std::min(pass.slice, all - g.first);
            ctx->launches += 2;
            launch_k(cdiag_tc_residues_kernel, dim3((unsigned)g.tiles, (unsigned)g.chunks), TC_RES_THREADS, 0, ctx->stream, g, limbs, X);
            launch_k(ctx->wait_limit < HE_WAIT_LIMIT ? cdiag_tc_mma_kernel<true> : cdiag_tc_mma_kernel<false>, std::min(ctx->sms, g.tiles * col_blocks),
                     TC_THREADS, TC_SMEM, ctx->stream, g, *tc, limbs, (const unsigned char *)X, pre, (const ModConst *)ctx->d_mc, ctx->sh->gave_up);
        }
    }
}

void cdiag_tc_set_smem_limits() {
    cudaFuncSetAttribute(cdiag_tc_mma_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, TC_SMEM);
    cudaFuncSetAttribute(cdiag_tc_mma_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, TC_SMEM);
}
