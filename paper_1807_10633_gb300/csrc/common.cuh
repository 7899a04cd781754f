// Internal definitions shared by the library's translation units.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <string>
#include <vector>

#include "vmc.h"

typedef unsigned __int128 u128;

#define VMC_MAX_M 256
#define VMC_WARPS 8
#define VMC_THREADS (VMC_WARPS * 32)

// Device status word bits (latched, cleared by vmc_sync).
#define VMC_DEV_SINGULAR 1u
#define VMC_DEV_OVERFLOW 2u
#define VMC_DEV_NOMOVE 4u
#define VMC_DEV_INCONSISTENT 8u
#define VMC_DEV_TIMEOUT 16u

// What one system's part of the rate store was computed from.  Rates and free-entry rows are laid out by the
// lists, so the moves may read them with the same lists alone (by content) and with no more walkers.
struct StoredRates {
    const void *G = nullptr;     // of the walkers
    int W = 0, n_groups = 0, words = 0;
    uint64_t lists = 0;          // vmc_lists::digest
    double eps = 0.0;            // eps_run
};

// One item of a batched local energy: its rates, and where they and its rows stand in the store.
struct BatchPart : StoredRates {
    size_t rates_at = 0, bits_at = 0;    // 16-byte units; bytes
    int share = 0;                       // walkers per round
};

struct vmc_ctx {
    int device = 0;
    cudaStream_t stream = nullptr;
    unsigned int *d_status = nullptr;
    std::string err;
    void *ws = nullptr;          // scratch for gradient partial sums
    size_t ws_bytes = 0;
    // CTMC rate store (per walker, per group, 128-bit sums), then free-entry rows: its own allocation, which
    // survives the gradient's use of ws
    void *rates = nullptr;
    size_t rates_bytes = 0;
    size_t rates_refused = SIZE_MAX;   // the smallest store that could not be allocated
    void *bits = nullptr;        // in rates: the free-entry rows of the last vmc_local_energy's walkers
    int bits_whole = 0;          // they hold every walker of the last vmc_local_energy
    // rate store bookkeeping (vmc_local_energy -> vmc_ctmc_step)
    StoredRates rates_of;
    int rates_valid = 0;
    uint64_t launches = 0;
    // batched launches: device descriptor table (re-uploaded only when the batch changes)
    void *batch_desc = nullptr;
    size_t batch_desc_bytes = 0;
    std::string batch_host;
    int *d_queue = nullptr;
    std::vector<BatchPart> batch_parts;   // vmc_local_energy_batch -> vmc_ctmc_step_batch, by item (none: not valid)
    int batch_rounds = 1;
    int eloc_threads = 256;        // threads per local-energy CTA (set by the autotuner)
    int g_tensor_cores = 1;        // refresh: G on tcgen05 (1) or CUDA cores (0)
    int refresh_smem = 0;          // refresh: register Gauss-Jordan (0) or shared-memory LU/GJ (1)
    int mixed_gj32 = 0;            // mixed refresh: FP64 LU of C_occ (0) or FP32 register Gauss-Jordan (1)
    int grad_j_tc = 1;             // Jastrow walker sums: tcgen05 digit products (1) or integer pipe (0)
};

// Plain-pointer view of the device lists, passed to kernels by value.
struct ListsView {
    int M;
    int band;      // largest |p - q| with a non-empty double list (pair candidates of a row)
    int cpr;       // warp chunks (32 candidates) per alpha row
    int rpg;       // beta rows per group (their candidates are the band's same-spin q only)
    int cpr_b;     // warp chunks per beta row when rpg == 1
    int n_groups;  // singles blocks of 32 spin orbitals + M * cpr alpha-row chunks + beta groups
    int64_t ns, nds, ndo;
    int64_t ns_pad;          // ns rounded up to a multiple of 4: row stride of the Fock tables and of F
    // singles: owner i and target a of entry e (the Fock tables and F are indexed by it)
    const uint32_t *s_owner;
    const uint16_t *s_a;
    // every move of the walk in canonical order ("flat" entries): the lists of a group's units one
    // after the other; each group starts on an even word of 32 entries, its opposite-spin part and a
    // change of spin among singles on a word (unused places: key 0, never alive).  Same-spin lists
    // and singles stand there once per spin.
    //   key   a | b << 8 | i << 16 | j << 24, spatial orbitals (singles: b = a, j = i)
    //   wcls  per word: bit 0 = spin of a and i, bit 1 = spin of b and j
    //   alive per word: the entries above the current eps_run
    //   rec   {key, v, w, aux}: integral, Jastrow constant; aux = index into a walker's F (singles)
    //   group {first word, first opposite-spin word, end word, units}: units bit 0 = spin of the same-spin
    //         part; the unit of an entry stands in lane (modulo 32) j + i ui + u0 (same spin; ui = bits
    //         1-5, u0 = bits 6-10), j + u2 (opposite spin; u2 = bits 11-15), spin orbital i (singles)
    int words;               // flat words, a multiple of 8
    int scaled;              // FP64 local energy: G scaled by E_a / E_i once per walker (else per entry)
    const uint32_t *key, *alive;
    const uint8_t *wcls;
    const float4 *rec32;
    const double4_32a *rec64;
    const uint4 *group;
    // Fock-sum update tables: Tj[k][e] = (ai|kk), Tjk[k][e] = (ai|kk) - (ak|ki), rows of ns_pad
    // (zero padded); FP64 and FP32 copies
    const double *Tj, *Tjk;
    const float *Tjf, *Tjkf;
    // diagonal tables: Jd[p][q] = (pp|qq), Kd[p][q] = (pq|qp); hd[p] = h_pp; h1 full
    const double *Jd, *Kd, *hd, *h1;
    double e_core;
    // work units of the local energy, [n_groups][32] in canonical order: {key naming the unit's own
    // orbitals (a | b << 16, spatial for kinds 0-1, alpha | beta << 16 for kind 2), flat base,
    // list length at the current eps_run (0: no unit), kind | spin << 2}
    const uint4 *unit_tab;
};

// Correlator product (Sec. III.A): device view of the structure plus the coefficient table.
#define VMC_CPS_MAX_SITES 8        // sites per correlator: 4^8 coefficients, a 16-bit index
#define VMC_CPS_MAX_PER_SITE 16    // correlators covering one site
struct CpsView {
    int n_corr;                    // 0: no correlator product
    int M, nnz;                    // orbitals; total sites over the correlators (= site_ent entries)
    const int32_t *corr_off;       // [n_corr + 1]: sites of correlator l are corr_sites[corr_off[l] ..)
    const int32_t *corr_sites;
    const int32_t *val_off;        // [n_corr + 1]: coefficients of l at values[val_off[l] ..], 4^k of them
    const int32_t *site_off;       // [M + 1]: correlators covering site k are site_ent[site_off[k] ..)
    const uint32_t *site_ent;      // (l << 16) | 4^t, t = the site's digit position in l; l ascending
    // excitations from site r to site t: the correlators that cover one of the two, ascending, with the
    // change of their index by an alpha electron: pair_ent[pair_off[r M + t] ..) = l << 16 | change + 32768
    const int32_t *pair_off;       // [M * M + 1]
    const uint32_t *pair_ent;
    const double *values;          // the coefficients (parameters), FP64, device
    const float *values32;         // FP32 copy made by the last walker (re)initialisation (mixed form)
};

struct vmc_cps {
    int M = 0, n_corr = 0, nnz = 0;
    int64_t n_values = 0;
    void *dev = nullptr;           // one device allocation: offsets, sites, site table, FP32 copy
    CpsView view{};                // values == nullptr (passed with the parameters)
};

struct vmc_lists {
    int M = 0;
    double eps_build = 0.0;
    double eps_run = -1.0;   // eps the effective lengths were computed for
    uint64_t digest = 0;     // of the moves and their magnitudes, in canonical order
    int64_t near_ties_build = 0;   // near ties of the build eps over every candidate (Sec. II.A)
    int64_t ns = 0, nds = 0, ndo = 0;
    // host copies of the sorted magnitudes (for effective lengths at a given eps_run)
    double *h_s_key = nullptr, *h_ds_key = nullptr, *h_do_key = nullptr;
    uint32_t *h_s_off = nullptr, *h_ds_off = nullptr, *h_do_off = nullptr;
    uint32_t *h_base = nullptr;   // flat base of every unit, [n_groups][32]
    void *dev = nullptr;     // one device allocation holding every array
    size_t dev_bytes = 0;
    ListsView view{};
    void *cf = nullptr;      // FP32 copy of C_alpha | C_beta (M x 2M floats at most)
    void *cdig = nullptr;    // FP64-form G: BF16 digit table of C and its row exponents
    void *jsym = nullptr;    // symmetric copies of J: FP64 (2M)^2 then FP32 (2M)^2
    const double *jastrow_for = nullptr;   // J pointer the constants were refreshed for
    uint64_t jastrow_epoch = 0;
};

// The rate store is about to change, or the tables that its rates belong to.
inline void drop_rates(vmc_ctx *ctx) {
    ctx->rates_valid = 0;
    ctx->batch_parts.clear();
}

inline bool same_lists(const StoredRates &r, const vmc_lists *L) {
    return r.lists == L->digest && r.n_groups == L->view.n_groups && r.words == L->view.words;
}

// ------------------------------------------------------------------ small helpers
__host__ __device__ inline int tri_index(int p, int q, int M) {  // p < q
    return p * (2 * M - p - 1) / 2 + (q - p - 1);
}

// Rate store of one system, in 16-byte units: W x n_groups exact rate sums (u128) followed by the
// W x n_groups per-group energy partials (FP64) that the local energy adds in a fixed order.
inline size_t rate_store_units(size_t W, int n_groups) {
    const size_t n = W * (size_t)n_groups;
    return n + (n + 1) / 2;
}

// J read from the upper triangle only
__device__ __forceinline__ double jget(const double *J, int N2, int p, int q) {
    return p <= q ? J[(size_t)p * N2 + q] : J[(size_t)q * N2 + p];
}

// floor(r * 2^64) as an exact 128-bit integer for r >= 0 (r < 2^43 is the caller's job)
__device__ __forceinline__ u128 rate_fixed(double r) {
    const uint64_t bits = (uint64_t)__double_as_longlong(r);
    const int ex = (int)((bits >> 52) & 0x7FF);
    if (ex == 0) return 0;                       // zero and subnormals (< 2^-1022)
    const uint64_t mant = (bits & ((1ull << 52) - 1)) | (1ull << 52);
    const int sh = ex - 1011;                    // r * 2^64 = mant * 2^sh
    if (sh >= 0) return ((u128)mant) << sh;
    if (sh <= -64) return 0;
    return (u128)(mant >> (-sh));
}
__device__ __forceinline__ u128 rate_fixed(float r) {
    const uint32_t bits = __float_as_uint(r);
    const int ex = (int)((bits >> 23) & 0xFF);
    if (ex == 0) return 0;
    const uint64_t mant = (bits & ((1u << 23) - 1)) | (1u << 23);
    const int sh = ex - 86;                      // r = mant 2^(ex-150); r 2^64 = mant 2^(ex-86)
    if (sh >= 0) return ((u128)mant) << sh;
    if (sh <= -64) return 0;
    return (u128)(mant >> (-sh));
}

__device__ __forceinline__ u128 shfl_xor_u128(u128 v, int m) {
    uint64_t lo = (uint64_t)v, hi = (uint64_t)(v >> 64);
    lo = __shfl_xor_sync(0xffffffffu, lo, m);
    hi = __shfl_xor_sync(0xffffffffu, hi, m);
    return ((u128)hi << 64) | lo;
}
__device__ __forceinline__ u128 shfl_up_u128(u128 v, int d) {
    uint64_t lo = (uint64_t)v, hi = (uint64_t)(v >> 64);
    lo = __shfl_up_sync(0xffffffffu, lo, d);
    hi = __shfl_up_sync(0xffffffffu, hi, d);
    return ((u128)hi << 64) | lo;
}
__device__ __forceinline__ u128 shfl_u128(u128 v, int src) {
    uint64_t lo = (uint64_t)v, hi = (uint64_t)(v >> 64);
    lo = __shfl_sync(0xffffffffu, lo, src);
    hi = __shfl_sync(0xffffffffu, hi, src);
    return ((u128)hi << 64) | lo;
}
__device__ __forceinline__ u128 warp_sum_u128(u128 v) {
#pragma unroll
    for (int m = 16; m >= 1; m >>= 1) v += shfl_xor_u128(v, m);
    return v;
}
__device__ __forceinline__ u128 warp_incl_scan_u128(u128 v, int lane) {
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        u128 o = shfl_up_u128(v, d);
        if (lane >= d) v += o;
    }
    return v;
}
__device__ __forceinline__ double warp_sum_f64(double v) {
#pragma unroll
    for (int m = 16; m >= 1; m >>= 1) v += __shfl_xor_sync(0xffffffffu, v, m);
    return v;
}

// Philox4x64-10 (Salmon et al., SC'11): ten rounds, two 64x64->128 products per round.
__device__ __forceinline__ uint64_t philox4x64_word0(uint64_t c0, uint64_t c1, uint64_t c2,
                                                     uint64_t c3, uint64_t k0, uint64_t k1) {
    const uint64_t M0 = 0xD2E7470EE14C6C93ull, M1 = 0xCA5A826395121157ull;
    const uint64_t W0 = 0x9E3779B97F4A7C15ull, W1 = 0xBB67AE8584CAA73Bull;
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        const uint64_t hi0 = __umul64hi(M0, c0), lo0 = M0 * c0;
        const uint64_t hi1 = __umul64hi(M1, c2), lo1 = M1 * c2;
        const uint64_t y0 = hi1 ^ c1 ^ k0, y2 = hi0 ^ c3 ^ k1;
        c0 = y0; c1 = lo1; c2 = y2; c3 = lo0;
        k0 += W0; k1 += W1;
    }
    return c0;
}

// Dependent launches: a kernel launched by launch_dependent may start while the kernel before it on the
// stream still runs, once all CTAs of that one have called launch_dependents (or ended); what the earlier
// kernel writes may be read only after wait_dependency (which returns at once in an ordinary launch).  So
// `dependent` is set only where the kernel before is one of this library's, itself launched ordinarily, and
// the kernel waits before it touches that one's output.
__device__ __forceinline__ void launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void wait_dependency() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

template <typename... KArgs, typename... Args>
cudaError_t launch_dependent(bool dependent, void (*kernel)(KArgs...), dim3 grid, int threads, size_t smem, cudaStream_t stream, Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute a = {};
    a.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    a.val.programmaticStreamSerializationAllowed = dependent ? 1 : 0;
    cfg.attrs = &a;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}

// ------------------------------------------------------------------ host-side helpers
vmc_status set_err(vmc_ctx *ctx, vmc_status st, const std::string &msg);
vmc_status cuda_check(vmc_ctx *ctx, cudaError_t e, const char *what);
vmc_status ensure_workspace(vmc_ctx *ctx, size_t bytes);
vmc_status lists_set_eps(vmc_ctx *ctx, vmc_lists *L, double eps_run);
size_t walker_stride_G(int M, int na, int nb);
size_t walker_stride_A(int na, int nb);

// launchers (defined in the .cu files)
vmc_status launch_refresh_jastrow(vmc_ctx *ctx, vmc_lists *L, const double *J);
vmc_status launch_init_walkers(vmc_ctx *ctx, vmc_lists *L, const vmc_params *P,
                               vmc_walkers *Wk, int full);
struct CpsView;
vmc_status launch_local_energy(vmc_ctx *ctx, const vmc_lists *L, vmc_walkers *Wk, const CpsView &C,
                               double *e_loc, double *t_res);
vmc_status launch_ctmc_step(vmc_ctx *ctx, const vmc_lists *L, const vmc_params *P,
                            vmc_walkers *Wk, uint64_t seed, uint64_t *move_code);
vmc_status launch_screened_moves(vmc_ctx *ctx, const vmc_lists *L, const vmc_walkers *Wk, const CpsView &C,
                                 int w_begin, int n_w, int64_t cap, uint64_t *code, double *ratio, double *contrib,
                                 int64_t *count, int64_t *walked);
vmc_status launch_local_energy_batch(vmc_ctx *ctx, int n, const vmc_batch_item *items);
vmc_status launch_ctmc_step_batch(vmc_ctx *ctx, int n, const vmc_batch_item *items, uint64_t seed);
vmc_status launch_g_umma(vmc_ctx *ctx, const vmc_walkers *Wk, const float *Cf);
size_t g_umma_smem(int M, int na, int nb);
bool g_ozaki_ok(int M, int na, int nb);
size_t g_ozaki_table_bytes(int M);
vmc_status launch_g_ozaki(vmc_ctx *ctx, const vmc_walkers *Wk, const double *Ca, const double *Cb, void *table);
vmc_status launch_grad_J_umma(vmc_ctx *ctx, int W, int M, const uint32_t *bits, const long long *cq, int mode,
                              long long *part, int chunk, int n_chunks);
void grad_j_umma_chunks(int W, int M, int nsm, int *chunk, int *n_chunks);
vmc_status launch_grad(vmc_ctx *ctx, const vmc_walkers *Wk, const double *w, double *dJ,
                       double *dCa, double *dCb);
vmc_status launch_accumulate(vmc_ctx *ctx, const vmc_walkers *Wk, const double *t, const double *e,
                             double *const aO[3], double *const aEO[3], double *sums);
vmc_status launch_amsgrad(vmc_ctx *ctx, double *p, const double *g, double *m, double *n,
                          size_t np, double alpha, double b1, double b2);
vmc_status launch_energy_gradient(vmc_ctx *ctx, size_t n, const double *sums, const double *aO,
                                  const double *aEO, double *g);
vmc_status launch_walker_reduce(vmc_ctx *ctx, int W, const double *t, const double *e,
                                double *out);
vmc_status launch_log_psi(vmc_ctx *ctx, const vmc_walkers *Wk, const vmc_params *P,
                          double *out);
// correlator product (cps.cu)
CpsView cps_view(const vmc_params *P);
vmc_status check_cps(vmc_ctx *ctx, const vmc_params *P, const vmc_walkers *Wk);
vmc_status launch_cps_state(vmc_ctx *ctx, const vmc_params *P, vmc_walkers *Wk);
vmc_status launch_cps_log_psi(vmc_ctx *ctx, const vmc_params *P, const vmc_walkers *Wk, double *out);
