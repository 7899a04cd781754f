// Screened local energy (Sec. II.A, Eq. eloc:hci) and the rejection-free CTMC move (Sec. II.B).
//
// One CTA per walker.  The walker's G (virtual rows only), exp(S) and the orbital -> column /
// slot map are staged in shared memory; the screened lists (shared by all walkers, L2-resident)
// are one flat array of entries in canonical move order, each with its orbitals (i, j, a, b).
// Which entries are moves is a row of bits per walker (i, j occupied, a, b empty, above eps_run),
// made for 64 walkers at once by k_free_bits, or by the walker's own CTA when the row is short.
// Entries belong to "groups":
//   singles : blocks of 32 consecutive spin orbitals i
//   doubles : one group per alpha spin-orbital row i (parts of it if needed); beta rows, which have
//             only the same-spin candidates, share groups.
// A warp takes a group, compacts the set bits of its part of the row and evaluates 32 moves at a
// time.  Each group's CTMC rates are summed as exact 128-bit fixed-point integers (order
// independent) and stored; the CTMC kernel re-walks only the chosen group, from the same bits.
// Every product that enters a rate uses explicitly rounded intrinsics so the two kernels compute
// bit-identical rates.  k_screened_moves walks the lists unit by unit (setup_unit), without the bits.
#include <math.h>

#include <algorithm>
#include <string>
#include <type_traits>
#include <vector>

#include "common.cuh"

namespace {

__device__ __forceinline__ double rmul(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float rmul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float rsub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ double rexp(double x) { return exp(x); }
__device__ __forceinline__ float rexp(float x) { return expf(x); }
__device__ __forceinline__ double rrcp(double x) { return __ddiv_rn(1.0, x); }
__device__ __forceinline__ float rrcp(float x) { return __fdiv_rn(1.0f, x); }

__device__ __forceinline__ unsigned long long abs_bits(double v) {
    return (unsigned long long)__double_as_longlong(v) & 0x7FFFFFFFFFFFFFFFull;
}
// 2 x 2 minor of G; accumulation of a contribution (FP64 form: fused, the FP64 pipe is its bound)
__device__ __forceinline__ float minor2(float a, float d, float b, float c) { return rsub(rmul(a, d), rmul(b, c)); }
__device__ __forceinline__ double minor2(double a, double d, double b, double c) { return __fma_rn(a, d, -__dmul_rn(b, c)); }

// 16-byte vectors of the table precision, and f += sgn * x on them
template <typename real> struct Vec16;
template <> struct Vec16<float> { typedef float4 type; static constexpr int n = 4; };
template <> struct Vec16<double> { typedef double2 type; static constexpr int n = 2; };
__device__ __forceinline__ void vadd(float4 &f, float s, const float4 &x) {
    f.x += s * x.x; f.y += s * x.y; f.z += s * x.z; f.w += s * x.w;
}
__device__ __forceinline__ void vadd(double2 &f, double s, const double2 &x) { f.x += s * x.x; f.y += s * x.y; }
__device__ __forceinline__ float4 vfma2(float4 o, float x, float4 u, float y, float4 v) {   // o - x u - y v
    o.x = o.x - x * u.x - y * v.x; o.y = o.y - x * u.y - y * v.y;
    o.z = o.z - x * u.z - y * v.z; o.w = o.w - x * u.w - y * v.w;
    return o;
}
__device__ __forceinline__ double2 vfma2(double2 o, double x, double2 u, double y, double2 v) {
    o.x = o.x - x * u.x - y * v.x; o.y = o.y - x * u.y - y * v.y;
    return o;
}
// Fock-sum table (same-spin Tjk: 1, other-spin Tj: 0) in the table precision
template <typename real> __device__ __forceinline__ const real *fock_table(const ListsView &L, int same);
template <> __device__ __forceinline__ const float *fock_table<float>(const ListsView &L, int same) {
    return same ? L.Tjkf : L.Tjf;
}
template <> __device__ __forceinline__ const double *fock_table<double>(const ListsView &L, int same) {
    return same ? L.Tjk : L.Tj;
}

// Record of a flat entry: {key, integral, Jastrow constant, index into F}.
__device__ __forceinline__ float4 flat_rec(const ListsView &L, uint32_t e, float) { return __ldg(&L.rec32[e]); }
__device__ __forceinline__ double4_32a flat_rec(const ListsView &L, uint32_t e, double) { return L.rec64[e]; }
__device__ __forceinline__ uint32_t low_bits(float x) { return __float_as_uint(x); }
__device__ __forceinline__ uint32_t low_bits(double x) { return (uint32_t)__double_as_longlong(x); }

// Walker arrays (global) and geometry.
struct WalkerArgs {
    int W, M, na, nb;
    const uint32_t *occ_bits;
    uint16_t *occ_list, *virt_list, *pos;
    uint32_t *occ_bits_w;
    void *G, *AinvT, *S, *F;
    double *e_diag;
    uint64_t *rng;
    uint16_t *cps;       // [W][n_corr] correlator indices (correlator product only)
};

struct SysDesc {
    ListsView L;
    WalkerArgs A;
    const double *J;
    double *e_loc, *t_res;
    u128 *rates;
    uint64_t *move_code;
    uint32_t *bits;          // free-entry rows of walkers w_first .. w_first + w_count - 1
    int w_first, w_count;    // the walkers of this launch (a batch may take several rounds)
    int w_begin, t_begin;    // first position of the system in the launch: walkers, walker tiles
};

struct Geo {
    int M, na, nb, ne, nw, nv_a, nv_b;
    size_t g_stride, a_stride;   // per-walker element strides of G and AinvT
    __device__ int n(int s) const { return s ? nb : na; }
    __device__ size_t g_off(int s) const { return s ? (size_t)nv_a * na : 0; }
    __device__ size_t a_off(int s) const { return s ? (size_t)na * na : 0; }
};

__device__ __forceinline__ Geo make_geo(int M, int na, int nb) {
    Geo g;
    g.M = M; g.na = na; g.nb = nb; g.ne = na + nb; g.nw = (M + 31) / 32;
    g.nv_a = M - na; g.nv_b = M - nb;
    g.g_stride = (size_t)(M - na) * na + (size_t)(M - nb) * nb;
    g.a_stride = (size_t)na * na + (size_t)nb * nb;
    return g;
}

// A work unit: one occupied spin orbital (single) or one occupied pair (double).
template <typename real>
struct Unit {
    uint32_t base, len;   // flat entries
    int kind;      // 0 single, 1 same-spin double, 2 opposite-spin double
    int cls;       // spin for kinds 0 and 1
    int ci, cj;    // columns of i and j
    int i, j;      // spin orbitals
    uint32_t sent; // key naming the unit's own (occupied) orbitals
    real ei, ej;   // 1/E_i, 1/E_j
};

// Shared-memory view of one walker used by the entry evaluation.
template <typename real>
struct View {
    const uint16_t *pos;   // [2M]: occupied -> column, virtual -> 0x8000 | slot
    const real *Ga, *Gb;   // virtual rows of G per spin (shared and padded, or global)
    int lda, ldb;          // their row strides
    __device__ const real *Grow(int s, int slot) const {
        return s ? Gb + (size_t)slot * ldb : Ga + (size_t)slot * lda;
    }
    const real *S;         // walker S in global
    const real *F;         // walker F [2][ns_pad]
    CpsView C;             // correlator product (C.n_corr == 0: none)
    // its tables, staged in shared memory by the local energy (global otherwise): coefficient offsets,
    // and per correlator the position of the walker's current coefficient (cur == nullptr:
    // val_off[l] + cidx[l] from the global indices) and 1/c
    const int32_t *voff, *cur;
    const uint16_t *cidx;  // [n_corr] the walker's correlator indices (global)
    const real *cinv;      // [n_corr] 1 / c_l[n_l] (shared), or nullptr: from the coefficients
    Geo geo;
    __device__ int cur_of(int l) const { return cur ? cur[l] : voff[l] + (int)cidx[l]; }
    __device__ real coef(int k) const;
    __device__ real cinv_of(int l) const { return cinv ? cinv[l] : rrcp(coef(cur_of(l))); }
    __device__ real Ev(int p) const { return rexp(S[p]); }              // p virtual
    __device__ real Eiv(int p) const { return rrcp(rexp(S[p])); }       // p occupied
};

// Correlator coefficient k in the table precision (the mixed form reads the FP32 copy).
template <> __device__ __forceinline__ float View<float>::coef(int k) const { return __ldg(&C.values32[k]); }
template <> __device__ __forceinline__ double View<double>::coef(int k) const { return __ldg(&C.values[k]); }

template <typename real> __device__ __forceinline__ real V0coef(const CpsView &C, int k);
template <> __device__ __forceinline__ float V0coef<float>(const CpsView &C, int k) { return C.values32[k]; }
template <> __device__ __forceinline__ double V0coef<double>(const CpsView &C, int k) { return C.values[k]; }

// Point a view's correlator tables at the global copies (the CTMC choice, the move set).
template <typename real>
__device__ __forceinline__ void cps_global(View<real> &V, const CpsView &C, const uint16_t *cidx) {
    V.C = C; V.voff = C.val_off; V.cur = nullptr;
    V.cidx = cidx; V.cinv = nullptr;
}

// Correlator-product ratio prod_l c_l[n_l + delta_l] / c_l[n_l] of the move that empties spin
// orbitals r0 (and r1) and fills a0 (and a1) (Sec. III.B), over the correlators that cover a changed
// site, ascending, each once.  An excitation's correlators and digit changes depend on its two sites
// alone, so they are listed per ordered site pair (CpsView::pair_ent); a double merges two such lists.
// (Merging the four sites' own lists instead, one step per correlator over four heads, took
// most of the local energy with correlators: 10.9 ms against 9.0 ms here at 8,192 H160 walkers.)
// nx = 2 (single) or 4.  A state index outside the correlator's table (an inconsistent state) gives
// NaN, which the rate check reports.
template <typename real>
__device__ __forceinline__ real cps_ratio(const View<real> &V, int r0, int a0, int r1, int a1, int nx) {
    const int M = V.geo.M;
    const int s0 = r0 >= M, s1 = r1 >= M;                    // spins: a beta digit counts twice
    const int p0 = (r0 - s0 * M) * M + (a0 - s0 * M), p1 = (r1 - s1 * M) * M + (a1 - s1 * M);
    int h0 = __ldg(&V.C.pair_off[p0]), h1 = nx == 4 ? __ldg(&V.C.pair_off[p1]) : 0;
    const int e0 = __ldg(&V.C.pair_off[p0 + 1]), e1 = nx == 4 ? __ldg(&V.C.pair_off[p1 + 1]) : 0;
    uint32_t c0 = h0 < e0 ? __ldg(&V.C.pair_ent[h0]) : 0xFFFFFFFFu, c1 = h1 < e1 ? __ldg(&V.C.pair_ent[h1]) : 0xFFFFFFFFu;
    real r = real(1);
    while (true) {
        const uint32_t l = min(c0, c1) >> 16;                // next correlator, ascending
        if (l == 0xFFFFu) break;
        int delta = 0;
        if (c0 >> 16 == l) {
            delta = ((int)(c0 & 0xFFFFu) - 32768) * (1 + s0);
            c0 = ++h0 < e0 ? __ldg(&V.C.pair_ent[h0]) : 0xFFFFFFFFu;
        }
        if (c1 >> 16 == l) {
            delta += ((int)(c1 & 0xFFFFu) - 32768) * (1 + s1);
            c1 = ++h1 < e1 ? __ldg(&V.C.pair_ent[h1]) : 0xFFFFFFFFu;
        }
        const int k = V.cur_of((int)l) + delta;
        if (k < V.voff[l] || k >= V.voff[l + 1]) return real(NAN);
        r = rmul(r, rmul(V.coef(k), V.cinv_of((int)l)));
    }
    return r;
}

// Unit of lane `lane` in group g, from the lists' unit table (the static (group, lane) -> (i, j,
// list) map, with the list lengths of the current eps_run): active if the list is non-empty and i
// (and j) are occupied in this walker.  Returns false if the lane has no active unit.
template <typename real>
__device__ __forceinline__ bool setup_unit(const ListsView &L, const View<real> &V, int g, int lane,
                                           Unit<real> &u) {
    const int M = L.M;
    const uint4 t = __ldg(&L.unit_tab[(size_t)g * 32 + lane]);
    u.base = t.y; u.len = t.z; u.kind = (int)(t.w & 3); u.cls = (int)(t.w >> 2); u.sent = t.x;
    u.ci = 0; u.cj = 0; u.ei = u.ej = real(0);
    const int lo = (int)(t.x & 0xFFFFu), hi = (int)(t.x >> 16);
    u.i = u.kind == 2 ? lo : u.cls * M + lo;
    u.j = u.kind == 0 ? -1 : (u.kind == 2 ? M + hi : u.cls * M + hi);
    if (u.len == 0) return false;
    u.ci = V.pos[u.i];
    if (u.ci & 0x8000) return false;
    if (u.kind != 0) {
        u.cj = V.pos[u.j];
        if (u.cj & 0x8000) return false;
        u.ej = V.Eiv(u.j);
    }
    u.ei = V.Eiv(u.i);
    return true;
}

template <typename real>
__device__ __forceinline__ Unit<real> shfl_unit(const Unit<real> &u, int src) {
    Unit<real> v;
    v.base = __shfl_sync(0xffffffffu, u.base, src);
    v.len = __shfl_sync(0xffffffffu, u.len, src);
    v.kind = __shfl_sync(0xffffffffu, u.kind, src);
    v.cls = __shfl_sync(0xffffffffu, u.cls, src);
    v.ci = __shfl_sync(0xffffffffu, u.ci, src);
    v.cj = __shfl_sync(0xffffffffu, u.cj, src);
    v.i = __shfl_sync(0xffffffffu, u.i, src);
    v.j = __shfl_sync(0xffffffffu, u.j, src);
    v.ei = __shfl_sync(0xffffffffu, u.ei, src);
    v.ej = __shfl_sync(0xffffffffu, u.ej, src);
    return v;
}

// Are the target orbital(s) of flat entry e unoccupied?
template <typename real>
__device__ __forceinline__ bool entry_free(const ListsView &L, const View<real> &V, int kind, int cls, uint32_t e) {
    const int M = V.geo.M, sa = kind == 2 ? 0 : cls * M, sb = kind == 2 ? M : sa;
    const uint32_t key = __ldg(&L.key[e]);
    return V.pos[sa + (key & 0xFFu)] & V.pos[sb + (key >> 8 & 0xFFu)] & 0x8000;
}

// ratio = psi(m)/psi(n) of a free entry (in-place replacement convention: the fermionic phases
// of H and of the ratio cancel) and contrib = H_nm * ratio.  Every kernel evaluates rates with
// this one sequence of explicitly rounded operations, so they agree bit for bit.
template <typename real, bool kC>
__device__ __forceinline__ void entry_value(const ListsView &L, const View<real> &V, int kind, int cls, int ci,
                                            int cj, real ei, real ej, uint32_t e, real &ratio, real &contrib, int &A,
                                            int &B, int I = -1, int Jo = -1) {
    const int M = V.geo.M;
    const auto r = flat_rec(L, e, real(0));
    const uint32_t key = low_bits(r.x);
    const int s = cls, a = (int)(key & 0xFFu), b = (int)(key >> 8 & 0xFFu);
    // FP64 form with long lists: G elements scaled by E_a / E_i first; otherwise the factors one after the other
    const bool scaled = sizeof(real) == 8 && L.scaled;
    auto elem = [&](int sp, int k, int c, real eic) {
        const real g = V.Grow(sp, V.pos[sp * M + k] & 0x7FFF)[c];
        return scaled ? rmul(rmul(g, V.Ev(sp * M + k)), eic) : g;
    };
    if (kind == 0) {
        const real g = elem(s, a, ci, ei);
        real rt = scaled ? rmul(g, r.z) : rmul(rmul(rmul(g, r.z), V.Ev(s * M + a)), ei);
        if (kC) rt = rmul(rt, cps_ratio<real>(V, I, s * M + a, I, s * M + a, 2));
        ratio = rt;
        contrib = rmul(V.F[low_bits(r.w)], rt);
        A = s * M + a; B = -1;
        return;
    }
    real x;
    if (kind == 1) {
        x = minor2(elem(s, a, ci, ei), elem(s, b, cj, ej), elem(s, a, cj, ej), elem(s, b, ci, ei));
        A = s * M + a; B = s * M + b;
    } else {
        x = rmul(elem(0, a, ci, ei), elem(1, b, cj, ej));
        A = a; B = M + b;
    }
    real rt = rmul(x, r.z);
    if (!scaled) rt = rmul(rmul(rmul(rt, V.Ev(A)), V.Ev(B)), rmul(ei, ej));
    if (kC) rt = rmul(rt, cps_ratio<real>(V, I, A, Jo, B, 4));
    ratio = rt;
    contrib = rmul(r.y, rt);
}

// The same for flat entry e of any unit (its orbitals from the key): ratio, contribution and move code.
// False if it is no move of this walker (bits of other walkers or occupations: nothing is read then).
template <typename real, bool kC>
__device__ __forceinline__ bool flat_entry_value(const ListsView &L, const View<real> &V, bool single, uint32_t e,
                                                 real &ratio, real &contrib, uint64_t &code) {
    const int M = V.geo.M, cls = __ldg(&L.wcls[e >> 5]), sa = cls & 1, sb = cls >> 1;
    const uint32_t key = __ldg(&L.key[e]);
    const int I = sa * M + (int)(key >> 16 & 0xFFu), J = sb * M + (int)(key >> 24);
    int A = sa * M + (int)(key & 0xFFu), B = sb * M + (int)(key >> 8 & 0xFFu);
    if ((V.pos[I] | V.pos[J] | ~(V.pos[A] & V.pos[B])) & 0x8000) return false;
    entry_value<real, kC>(L, V, single ? 0 : (sa == sb ? 1 : 2), sa, V.pos[I], V.pos[J], V.Eiv(I),
                          single ? real(0) : V.Eiv(J), e, ratio, contrib, A, B, I, J);
    code = single ? 1ull | (uint64_t)I << 2 | 1023ull << 12 | (uint64_t)A << 22 | 1023ull << 32
                  : 2ull | (uint64_t)I << 2 | (uint64_t)J << 12 | (uint64_t)A << 22 | (uint64_t)B << 32;
    return true;
}

// Evaluate list entry `idx` of unit u.  Returns false if the target orbital(s) are occupied.
template <typename real, bool kC>
__device__ __forceinline__ bool eval_entry(const ListsView &L, const View<real> &V, const Unit<real> &u,
                                           uint32_t idx, real &ratio, real &contrib, int &A, int &B) {
    if (!entry_free<real>(L, V, u.kind, u.cls, idx)) return false;
    entry_value<real, kC>(L, V, u.kind, u.cls, u.ci, u.cj, u.ei, u.ej, idx, ratio, contrib, A, B, u.i, u.j);
    return true;
}

template <typename real>
__device__ __forceinline__ u128 rate_of(real ratio, unsigned *flag) {
    real r = fabs(ratio);
    if (!(r < (real)8796093022208.0)) {   // 2^43: fixed-point range limit (also catches NaN)
        *flag |= VMC_DEV_OVERFLOW;
        r = (r == r) ? (real)8796093022207.0 : (real)0;
    }
    return rate_fixed(r);
}

template <typename real> struct AccT { typedef double type; };
template <> struct AccT<float> { typedef float type; };

__device__ __forceinline__ double warp_sum_acc(double v) { return warp_sum_f64(v); }
__device__ __forceinline__ double warp_sum_acc(float v) {
#pragma unroll
    for (int m = 16; m >= 1; m >>= 1) v += __shfl_xor_sync(0xffffffffu, v, m);
    return (double)v;
}

// ---------------------------------------------------------------------------------- free entries
// 32 x 32 bit transpose across a warp: lane l holds row l; afterwards lane l holds column l.
__device__ __forceinline__ uint32_t transpose_bits(uint32_t x, int lane) {
#pragma unroll
    for (int k = 16; k >= 1; k >>= 1) {
        const uint32_t m = k == 16 ? 0x0000FFFFu : k == 8 ? 0x00FF00FFu : k == 4 ? 0x0F0F0F0Fu : k == 2 ? 0x33333333u : 0x55555555u;
        const uint32_t y = __shfl_xor_sync(0xffffffffu, x, k);
        const uint32_t keep = (lane & k) ? ~m : m;
        const uint32_t r = __funnelshift_l(y, y, (lane & k) ? 32 - k : k);
        x = (x & keep) | (r & ~keep);
    }
    return x;
}

// Which flat entries are moves, for tiles of 64 walkers: one bit per entry and walker, set if i and j
// are occupied, a and b empty and the entry is above eps_run.  A warp takes 256 consecutive entries:
// lane = entry, the 64 walkers' occupations of an orbital are two words (bit = walker) in shared
// memory, so a few logic operations answer 64 walkers; bit transposes turn lane = entry into
// lane = walker, and every walker's 32 bytes are stored as one sector.
// Grid: (tiles of 64 walkers, splits of the row).  The local energy is launched as its dependent: it stages its
// tables meanwhile and waits before it reads the first bits.
constexpr int kTile = 64;

// Rows of at most this many words are made by the local energy's own CTA (a warp per word, lane = entry):
// at 10 orbitals that is one launch less; from a few hundred words on the tiles of walkers win.
constexpr int kOwnWords = 64;
// While all CTAs are resident at once (four per SM) the launch counts for more: 300 walkers of H14 at
// eps = 1e-4 (about 100 words) 12.5 -> 12.0 us.
constexpr int kOwnWordsSmall = 256, kOwnWalkers = 608;
inline bool own_rows(int words, int W) { return words <= kOwnWords || (words <= kOwnWordsSmall && W <= kOwnWalkers); }

__device__ __forceinline__ void free_bits_tile(const ListsView &L, const uint32_t *__restrict__ occ_bits, int w_first,
                                               int w_end, int tile, int part, int parts, uint32_t *__restrict__ bits,
                                               uint2 *s_occ) {
    const int M = L.M, nw = (M + 31) / 32;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarp = blockDim.x >> 5;
    const int w = w_first + tile * kTile + lane;     // this lane's walkers: w and w + 32
    // s_occ[p]: bit l set if spin orbital p is occupied in walker l of the tile
    for (int t = warp; t < 2 * nw; t += nwarp) {
        const int s = t / nw, k0 = (t - s * nw) * 32;
        const uint32_t x = transpose_bits(w < w_end ? occ_bits[(size_t)w * 2 * nw + t] : 0u, lane);
        const uint32_t y = transpose_bits(w + 32 < w_end ? occ_bits[(size_t)(w + 32) * 2 * nw + t] : 0u, lane);
        if (k0 + lane < M) s_occ[s * M + k0 + lane] = make_uint2(x, y);
    }
    __syncthreads();
    uint32_t *row = bits + (size_t)(tile * kTile + lane) * L.words;
    for (int c = part * nwarp + warp; c * 8 < L.words; c += parts * nwarp) {
        uint32_t key[8], x[8], y[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) key[j] = __ldg(&L.key[c * 256 + 32 * j + lane]);
        const uint2 cl = __ldg((const uint2 *)(L.wcls + c * 8));
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const uint32_t cls = (j < 4 ? cl.x : cl.y) >> (8 * (j & 3));
            const uint2 *oa = s_occ + ((cls & 1u) ? M : 0), *ob = s_occ + ((cls & 2u) ? M : 0);
            const uint32_t k = key[j];
            const uint2 a = oa[k & 0xFFu], b = ob[k >> 8 & 0xFFu], i = oa[k >> 16 & 0xFFu], q = ob[k >> 24];
            x[j] = transpose_bits(i.x & q.x & ~(a.x | b.x), lane);
            y[j] = transpose_bits(i.y & q.y & ~(a.y | b.y), lane);
        }
        const uint4 l0 = __ldg((const uint4 *)(L.alive + c * 8)), l1 = __ldg((const uint4 *)(L.alive + c * 8 + 4));
        if (w < w_end) {
            uint4 *o = (uint4 *)(row + c * 8);
            o[0] = make_uint4(x[0] & l0.x, x[1] & l0.y, x[2] & l0.z, x[3] & l0.w);
            o[1] = make_uint4(x[4] & l1.x, x[5] & l1.y, x[6] & l1.z, x[7] & l1.w);
        }
        if (w + 32 < w_end) {
            uint4 *o = (uint4 *)(row + (size_t)32 * L.words + c * 8);
            o[0] = make_uint4(y[0] & l0.x, y[1] & l0.y, y[2] & l0.z, y[3] & l0.w);
            o[1] = make_uint4(y[4] & l1.x, y[5] & l1.y, y[6] & l1.z, y[7] & l1.w);
        }
    }
}

__global__ void __launch_bounds__(256, 5)
k_free_bits(ListsView L, const uint32_t *__restrict__ occ_bits, int w_first, int w_end, uint32_t *__restrict__ bits) {
    __shared__ uint2 s_occ[2 * VMC_MAX_M];
    launch_dependents();
    free_bits_tile(L, occ_bits, w_first, w_end, blockIdx.x, blockIdx.y, gridDim.y, bits, s_occ);
}

// The same for a batch: blockIdx.x runs over the tiles of all systems (t_begin: first tile of each).
__global__ void __launch_bounds__(256)
k_free_bits_batched(const SysDesc *__restrict__ sys, int n_sys) {
    __shared__ uint2 s_occ[2 * VMC_MAX_M];
    launch_dependents();
    int k = 0;
    while (k + 1 < n_sys && sys[k + 1].t_begin <= (int)blockIdx.x) ++k;
    const SysDesc &d = sys[k];
    free_bits_tile(d.L, d.A.occ_bits, d.w_first, d.w_first + d.w_count, blockIdx.x - d.t_begin, blockIdx.y, gridDim.y,
                   d.bits, s_occ);
}

// One word of one walker's row, by a warp (lane = entry); ow: the walker's occupation words.
__device__ __forceinline__ uint32_t free_word(const ListsView &L, const uint32_t *__restrict__ ow, int nw, int k, int lane) {
    const uint32_t key = __ldg(&L.key[k * 32 + lane]);
    const int cls = __ldg(&L.wcls[k]);
    auto occ = [&](uint32_t p, int s) { return ow[s * nw + (p >> 5)] >> (p & 31u) & 1u; };
    const uint32_t m = occ(key >> 16 & 0xFFu, cls & 1) & occ(key >> 24, cls >> 1) &
                       ~(occ(key & 0xFFu, cls & 1) | occ(key >> 8 & 0xFFu, cls >> 1));
    return __ballot_sync(0xffffffffu, m & 1u) & __ldg(&L.alive[k]);
}

// ---------------------------------------------------------------------------------- local energy
// Exact 128-bit rate sums in two 64-bit halves (units of 2^-64).
struct Sum128 {
    unsigned long long lo, hi;
    __device__ void add(unsigned long long l, unsigned long long h) {
        lo += l;
        hi += h + (lo < l ? 1ull : 0ull);
    }
};
// Any rate, as rate_of: the general path for rates the fast ones below do not take; bit 127 tells of an
// overflow (rates stay below 2^107).
template <typename real> __device__ __noinline__ u128 large_rate(real ratio) {
    unsigned flag = 0;
    const u128 v = rate_of<real>(ratio, &flag);
    return flag ? v | (u128)1 << 127 : v;
}
template <typename real> __device__ __forceinline__ void add_large_rate(Sum128 &q, real ratio, unsigned &flag) {
    const u128 v = large_rate<real>(ratio);
    const unsigned long long hi = (unsigned long long)(v >> 64);
    if (hi >> 63) flag |= VMC_DEV_OVERFLOW;
    q.add((unsigned long long)v, hi & 0x7FFFFFFFFFFFFFFFull);
}
// floor(|ratio| 2^64) added to q, exactly.  FP32: the integer part (below 2^32) and 2^64 times the fraction
// are exact conversions.  FP64, below 1: the mantissa, shifted to the top of 64 bits, goes right by what the
// exponent is below 1/2 (integer pipe: the FP64 pipe is that form's bound).
__device__ __forceinline__ void add_rate(Sum128 &q, float ratio, unsigned &flag) {
    const float r = fabsf(ratio);
    if (r < 4294967296.0f) {
        const float t = truncf(r);
        q.add(__float2ull_rz((r - t) * 18446744073709551616.0f), (unsigned long long)__float2uint_rz(t));
    } else {
        add_large_rate(q, ratio, flag);
    }
}
__device__ __forceinline__ void add_rate(Sum128 &q, double ratio, unsigned &flag) {
    const unsigned long long b = abs_bits(ratio);
    const uint32_t sh = 1022u - (uint32_t)(b >> 52);
    if ((int)sh >= 0) {                                    // below 1
        const unsigned long long m = (b << 11) | 0x8000000000000000ull;
        q.add(sh < 64u ? m >> sh : 0ull, 0ull);
    } else {
        add_large_rate(q, ratio, flag);
    }
}
// Sum over the warp: limbs of 27 bits, whose sums over 32 lanes fit 32 bits.
__device__ __forceinline__ u128 warp_sum(const Sum128 &q) {
    const uint32_t m = 0x7FFFFFFu;
    const uint32_t s0 = __reduce_add_sync(0xffffffffu, (uint32_t)q.lo & m);
    const uint32_t s1 = __reduce_add_sync(0xffffffffu, (uint32_t)(q.lo >> 27) & m);
    const uint32_t s2 = __reduce_add_sync(0xffffffffu, (uint32_t)(q.lo >> 54 | q.hi << 10) & m);
    const uint32_t s3 = __reduce_add_sync(0xffffffffu, (uint32_t)(q.hi >> 17) & m);
    const uint32_t s4 = __reduce_add_sync(0xffffffffu, (uint32_t)(q.hi >> 44));
    return (u128)s0 + ((u128)s1 << 27) + ((u128)s2 << 54) + ((u128)s3 << 81) + ((u128)s4 << 108);
}

// Per spin orbital, in shared memory: exp(S) of an empty one with the element offset of its G row from
// the first alpha row; 1/exp(S) of a filled one with its column.
template <typename real> struct OrbTable;
template <> struct OrbTable<float> {
    float2 *t;
    static constexpr size_t bytes = 8;
    __device__ OrbTable(void *p, int) : t((float2 *)p) {}
    __device__ void set(int p, float e, int off) { t[p] = make_float2(e, __int_as_float(off)); }
    __device__ float e(int p) const { return t[p].x; }
    __device__ int off(int p) const { return __float_as_int(t[p].y); }
    __device__ void get(int p, float &e, int &off) const {
        const float2 v = t[p];
        e = v.x;
        off = __float_as_int(v.y);
    }
};
// (with scaled G rows the entries read the offsets alone)
template <> struct OrbTable<double> {
    double *e_;
    int *off_;
    static constexpr size_t bytes = 12;
    __device__ OrbTable(void *p, int n) : e_((double *)p), off_((int *)((double *)p + n)) {}
    __device__ void set(int p, double e, int off) { e_[p] = e; off_[p] = off; }
    __device__ double e(int p) const { return e_[p]; }
    __device__ void get(int p, double &e, int &off) const { e = e_[p]; off = off_[p]; }
    __device__ int off(int p) const { return off_[p]; }
};

// Value of flat entry e (a move of this walker): returns H_nm and the ratio, adds the rate to q.
// K: 0 single, 1 same-spin double, 2 opposite-spin double, 3 either double (second: a same-spin one,
// whose minor has a second product); sa, sb: M if the spin of (a, i), (b, j) is beta; valid: the lane has
// an entry of its own (the others repeat one and count nothing); key_out: the key (singles: spin orbital i);
// scaled: G[a][i] holds G_ai E_a / E_i.
// The rounding is entry_value's.  The FP64 form multiplies E_a / E_i into G once per walker and element
// (two products each, 12.8 K elements at H160) instead of four products per entry: GB300 has 2 FP64
// multiply-adds per clock and SM, so a batch of 32 spends 16 clocks on every one.  It pays with long lists (rule in
// lists.cu): without doubles the two products per element are what costs.
template <int K, typename real, bool kC, bool scaled>
__device__ __forceinline__ real flat_value(const ListsView &L, const View<real> &V, const OrbTable<real> &orb, uint32_t e,
                                           int sa, int sb, bool second, bool valid, Sum128 &q, unsigned &flag, real &ratio, uint32_t &key_out) {
    const auto r = flat_rec(L, e, real(0));
    const uint32_t key = low_bits(r.x);
    key_out = key;
    const real *G = V.Ga;
    real ea, ei, rt, h;
    int ra, ci;
    if (K == 0) {
        const uint32_t aux = low_bits(r.w);
        const int s = aux >= (uint32_t)L.ns_pad ? V.geo.M : 0, A = s + (int)(key & 0xFFu), I = s + (int)(key >> 24);
        key_out = (uint32_t)I;
        if (scaled) { ra = orb.off(A); ci = orb.off(I); }
        else { orb.get(A, ea, ra); orb.get(I, ei, ci); }
        rt = rmul(G[ra + ci], r.z);
        if (!scaled) rt = rmul(rmul(rt, ea), ei);
        if (kC) rt = rmul(rt, cps_ratio<real>(V, I, A, I, A, 2));
        h = V.F[aux];
    } else {
        const int A = sa + (int)(key & 0xFFu), B = sb + (int)(key >> 8 & 0xFFu);
        const int I = sa + (int)(key >> 16 & 0xFFu), J = sb + (int)(key >> 24);
        real eb, ej;
        int rb, cj;
        if (scaled) {
            ra = orb.off(A); rb = orb.off(B); ci = orb.off(I); cj = orb.off(J);
        } else {
            orb.get(A, ea, ra); orb.get(B, eb, rb); orb.get(I, ei, ci); orb.get(J, ej, cj);
        }
        real x;
        if (K == 1 || (K == 3 && second)) x = minor2(G[ra + ci], G[rb + cj], G[ra + cj], G[rb + ci]);
        else x = rmul(G[ra + ci], G[rb + cj]);
        rt = rmul(x, r.z);
        if (!scaled) rt = rmul(rmul(rmul(rt, ea), eb), rmul(ei, ej));
        if (kC) rt = rmul(rt, cps_ratio<real>(V, I, A, J, B, 4));
        h = r.y;
    }
    if (!valid) rt = real(0);
    add_rate(q, rt, flag);
    ratio = rt;
    return h;
}

// Shared memory of one warp: codes (entry position in the block) of free entries.  32 places before and
// behind the codes may be read: batches are full reads.
constexpr int kFreeMax = 160;
struct WarpBuf {
    uint16_t pad[32], code[kFreeMax + 32];
};

// Running sum of the mixed form's FP32 energy contributions of one group and kind, in a fixed order:
// the entries of the occupied units form windows of 32 places (free or not); after each window its free
// entries go on a stack, and as soon as the stack holds 32 or more the top 32 are added, lane l the
// l-th from below; what is left at the end is added by lanes 0 .. q-1.  Free entries arrive in batches of 32,
// one per lane, with their places.  With a batch the previous full one can be added: the window that
// filled the stack is that of the previous batch's last entry, and q of the new entries lie in
// it too and are what the addition leaves on the stack.  So lanes >= q take the stack (below) and the
// previous batch, lanes < q the new one, rotated by q.
struct StackSum {
    float below = 0.f, last = 0.f;   // the stack's contributions; the previous batch
    int q = 0, n_last = 0;           // entries on the stack; entries of the previous batch (0: none yet)
    uint32_t place = 0;              // places of the previous batch's entries
    __device__ void drain(int qn, float c, int lane, float &acc) {
        const float m = lane < q ? below : last;
        acc += __shfl_sync(0xffffffffu, lane >= qn ? m : c, (lane + qn) & 31);
        below = m;
        q = qn;
    }
    // a batch of n <= 32 entries (lanes < n; only the last one has n < 32): contributions c, places p
    __device__ void batch(float c, uint32_t p, int n, int lane, float &acc) {
        if (n_last) {
            const uint32_t end = __shfl_sync(0xffffffffu, place, 31) | 31u;      // the window's last place
            const unsigned after = __ballot_sync(0xffffffffu, lane >= n || p > end);
            drain(after ? __ffs(after) - 1 : 32, c, lane, acc);
        }
        place = p;
        last = c;
        n_last = n;
    }
    // after the last batch: its own addition if it was full, else what this lane has still to add
    __device__ float finish(int lane, float &acc) {
        if (n_last == 32) {
            drain(0, 0.f, lane, acc);
            return 0.f;
        }
        return lane < n_last ? (lane < q ? below : last) : 0.f;
    }
};

// Local energy of walker w by the whole CTA (any number of warps).  row: the walker's free-entry bits
// (null: made here); smraw: dynamic shared memory.
//
// Warps take the groups dynamically; each group's sums are stored by index, so the result does not depend on
// which warp took it.  A group's free entries are the set bits of a contiguous range of the row: a lane
// reads two words, a popcount prefix ranks its bits, and it writes their positions to the warp's code
// buffer; 32 at a time, one per lane, they are evaluated (flat_value).  Nothing is done for entries that
// are not free: the first version of this walk loaded and tested each of the ~62 K entries of an H160
// walker's occupied pairs to find its 13 K moves, and more than half of its instructions were that test.
// FP64 form: batches run over both kinds of a group.  Mixed form: the kinds are kept apart and the FP32
// sums keep the fixed order of StackSum; an entry's place counts the entries of occupied units only, from the
// unit table.
template <typename real, bool kC, bool scaled>
__device__ __forceinline__ void eloc_walker(const ListsView &L, const WalkerArgs &A, const int w,
                                            const uint32_t *__restrict__ row, double *__restrict__ e_loc,
                                            double *__restrict__ t_res, u128 *__restrict__ rates, unsigned *status,
                                            unsigned char *smraw, const CpsView &C = CpsView{}) {
    constexpr bool kOrder = sizeof(real) == 4;
    const Geo geo = make_geo(A.M, A.na, A.nb);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nt = blockDim.x, nwarp = nt >> 5;
    const int M = geo.M, nw = geo.nw, n_groups = L.n_groups, n_sgl_groups = (2 * M + 31) / 32;
    const int lda = geo.na + 1, ldb = geo.nb + 1;    // padded rows: no bank conflicts on columns
    real *sG = (real *)smraw;
    const size_t g_el = (size_t)geo.nv_a * lda + (size_t)geo.nv_b * ldb;
    // (offsets from smraw, so that every access stays a shared-memory instruction)
    const size_t o_orb = (g_el * sizeof(real) + 7) & ~(size_t)7, o_occ = o_orb + OrbTable<real>::bytes * (size_t)(2 * M);
    const size_t o_row = (o_occ + sizeof(uint32_t) * 2 * nw + 15) & ~(size_t)15;
    const size_t o_buf = o_row + (row ? 0 : sizeof(uint32_t) * (size_t)L.words);   // (words: a multiple of 8)
    OrbTable<real> orb(smraw + o_orb, 2 * M);
    typedef WarpBuf Buf;
    uint32_t *s_occ = (uint32_t *)(smraw + o_occ);   // [2 nw] the walker's occupation words
    uint32_t *s_row = (uint32_t *)(smraw + o_row);   // the walker's free-entry bits if row is null
    Buf *bufs = (Buf *)(smraw + o_buf);
    Buf &wb = bufs[warp];
    // correlator product, after the warp buffers: 1 / c_l[n_l], the current coefficient positions and
    // the coefficient offsets
    real *sCinv = (real *)(bufs + nwarp);
    int32_t *sCur = (int32_t *)(sCinv + ((C.n_corr + 3) & ~3));
    int32_t *sVoff = sCur + C.n_corr;
    // per-group energy partials: global, after the system's rate sums (written and read by this CTA)
    double *eg = (double *)(rates + (size_t)A.W * n_groups) + (size_t)w * n_groups;
    __shared__ int next_group;

    // ---- prologue: stage G into padded rows, exp(S), orbital map
    {
        // the walker's bits are read group by group: bring them to L2 while the tables are staged
        if (tid == 0 && row && L.words > 0)
            asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(row), "r"(4u * (uint32_t)L.words) : "memory");
        const real *Gw = (const real *)A.G + (size_t)w * geo.g_stride;
        const size_t na_el = (size_t)geo.nv_a * geo.na;
        real *sGb = sG + (size_t)geo.nv_a * lda;
        if constexpr (!scaled) {
            // one row per warp, asynchronous copies (all of a thread's in flight; the odd row stride
            // leaves pieces of one element)
            for (int r = warp; r < geo.nv_a + geo.nv_b; r += nwarp) {
                const bool bs = r >= geo.nv_a;
                const int rr = bs ? r - geo.nv_a : r, n = bs ? geo.nb : geo.na;
                const real *src = Gw + (bs ? na_el + (size_t)rr * geo.nb : (size_t)rr * geo.na);
                const uint32_t dst = (uint32_t)__cvta_generic_to_shared(bs ? sGb + (size_t)rr * ldb : sG + (size_t)rr * lda);
                for (int c = lane; c < n; c += 32)
                    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(dst + (uint32_t)(c * sizeof(real))), "l"(src + c),
                                 "n"(sizeof(real)) : "memory");
            }
        }
        if (!row) {
            const uint32_t *ow = A.occ_bits + (size_t)w * 2 * nw;
            for (int k = warp; k < L.words; k += nwarp) {
                const uint32_t x = free_word(L, ow, nw, k, lane);
                if (lane == 0) s_row[k] = x;
            }
        }
        const real *Sw = (const real *)A.S + (size_t)w * 2 * M;
        const uint16_t *pw = A.pos + (size_t)w * 2 * M;
        for (int p = tid; p < 2 * M; p += nt) {
            const int ps = pw[p];
            const real e = rexp(Sw[p]);
            if (ps & 0x8000) orb.set(p, e, (ps & 0x7FFF) * (p < M ? lda : ldb) + (p < M ? 0 : geo.nv_a * lda));
            else orb.set(p, rrcp(e), ps);
        }
        if constexpr (scaled) {
            // rows scaled by E of their orbital and 1/E of their columns'; four rows per warp at a time
            __syncthreads();
            const uint16_t *occ = A.occ_list + (size_t)w * geo.ne, *virt = A.virt_list + (size_t)w * (2 * M - geo.ne);
            for (int s = 0; s < 2; ++s) {
                const int n = geo.n(s), nv = M - n, ld = s ? ldb : lda;
                const real *src = Gw + (s ? na_el : 0);
                real *dst = s ? sGb : sG;
                for (int c = lane; c < n; c += 32) {
                    const real ec = orb.e(s * M + occ[(s ? geo.na : 0) + c]);
                    for (int r0 = warp; r0 < nv; r0 += 4 * nwarp) {
                        real g[4];
#pragma unroll
                        for (int k = 0; k < 4; ++k) g[k] = r0 + k * nwarp < nv ? src[(size_t)(r0 + k * nwarp) * n + c] : real(0);
#pragma unroll
                        for (int k = 0; k < 4; ++k) {
                            const int r = r0 + k * nwarp;
                            if (r < nv) dst[(size_t)r * ld + c] = rmul(rmul(g[k], orb.e(s * M + virt[(s ? geo.nv_a : 0) + r])), ec);
                        }
                    }
                }
            }
        }
        for (int t = tid; t < 2 * nw; t += nt) s_occ[t] = A.occ_bits[(size_t)w * 2 * nw + t];
        if (kC) {
            for (int l = tid; l <= C.n_corr; l += nt) sVoff[l] = C.val_off[l];
            for (int l = tid; l < C.n_corr; l += nt) {
                const int k = C.val_off[l] + (int)A.cps[(size_t)w * C.n_corr + l];
                sCur[l] = k;
                sCinv[l] = rrcp(V0coef<real>(C, k));
            }
        }
        if (tid == 0) next_group = nwarp;
        if (!scaled) asm volatile("cp.async.wait_all;" ::: "memory");
        if (row) wait_dependency();      // the rows (a kernel may still be writing them)
    }
    __syncthreads();

    View<real> V;
    V.Ga = sG; V.F = (const real *)A.F + (size_t)w * 2 * L.ns_pad; V.geo = geo;
    V.C = C; V.voff = sVoff; V.cur = sCur; V.cidx = nullptr; V.cinv = sCinv;
    typedef typename AccT<real>::type acc_t;
    unsigned flag = 0;

    for (int g = warp; g < n_groups;) {
        const uint4 gi = __ldg(&L.group[g]);             // first word, first opposite-spin word, end, spin
        const bool pairs = g >= n_sgl_groups;
        acc_t e_grp = 0;
        Sum128 q{0, 0};
        bool any = false;
        uint32_t to_place = 0;                           // mixed form: place - flat entry of unit `lane`
        StackSum sum;
        float restA = 0.f;                               // what the same-spin part left to add
        bool in_a = true;
        uint32_t carry_e = 0;                            // entries waiting for a full batch (lanes < n_carry)
        int n_carry = 0;
        for (uint32_t w0 = gi.x; w0 < gi.z;) {
            const uint32_t wi = w0 + 2 * lane;
            uint2 x = make_uint2(0u, 0u);
            if (wi < gi.z) {
                x = row ? *(const uint2 *)(row + wi) : *(const uint2 *)(s_row + wi);
                if (wi + 1 >= gi.z) x.y = 0;
            }
            if (!__any_sync(0xffffffffu, x.x | x.y) && n_carry == 0) {
                w0 += 64;
                continue;
            }
            const uint32_t blk = w0 * 32;
            const uint32_t f0 = __popc(x.x), own = f0 + __popc(x.y);
            if constexpr (kOrder) {
                // first block with free entries: the units, for the places of a kind's entries, which its second
                // batch needs.  A long group will have one; a short one (one block) is counted first.
                bool need = !any;
                if (need && gi.z - gi.x <= 20u) {
                    const uint32_t fA = (wi < gi.y ? f0 : 0u) + (wi + 1 < gi.y ? own - f0 : 0u);
                    const uint32_t c = __reduce_add_sync(0xffffffffu, fA << 16 | (own - fA));
                    need = max(c >> 16, c & 0xFFFFu) > 32u;
                }
                if (need) {
                    const uint4 t = __ldg(&L.unit_tab[(size_t)g * 32 + lane]);
                    const int kind = (int)(t.w & 3u), sp = (int)(t.w >> 2);
                    const uint32_t i = t.x & 0xFFFFu, j = kind == 0 ? i : t.x >> 16;
                    const uint32_t bi = s_occ[(kind == 2 ? 0 : sp * nw) + (i >> 5)] >> (i & 31u);
                    const uint32_t bj = s_occ[(kind == 2 ? nw : sp * nw) + (j >> 5)] >> (j & 31u);
                    const uint32_t len = (bi & bj & 1u) ? t.z : 0u;
                    uint32_t us = len;
#pragma unroll
                    for (int d = 1; d < 32; d <<= 1) {
                        const uint32_t o = __shfl_up_sync(0xffffffffu, us, d);
                        if (lane >= d) us += o;
                    }
                    // (same-spin units stand before the opposite-spin ones)
                    const uint32_t uA = __reduce_max_sync(0xffffffffu, kind != 2 && t.z ? us : 0u);
                    to_place = us - len - (kind == 2 ? uA : 0u) - t.y;
                }
            }
            any = true;
            uint32_t sc = own;                           // free entries up to and with the lane's words
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const uint32_t o = __shfl_up_sync(0xffffffffu, sc, d);
                if (lane >= d) sc += o;
            }
            // lanes of this block whose codes fit the buffer
            const int nl = __popc(__ballot_sync(0xffffffffu, sc <= (uint32_t)kFreeMax));
            const uint32_t at0 = sc - own;
            if (lane < nl) {
                uint16_t *at = wb.code + at0;
#pragma unroll 1
                for (uint32_t y = x.x; y; y &= y - 1u) *at++ = (uint16_t)(lane << 6 | (__ffs(y) - 1));
#pragma unroll 1
                for (uint32_t y = x.y; y; y &= y - 1u) *at++ = (uint16_t)(lane << 6 | 32 | (__ffs(y) - 1));
            }
            __syncwarp();
            const int n = (int)__reduce_max_sync(0xffffffffu, lane < nl ? sc : 0u);
            const uint32_t w1 = w0 + 2 * (uint32_t)nl;
            const bool done = w1 >= gi.z;
            // the carried entries and the codes s0 .. s1-1, 32 at a time; end: the last, partly filled
            // batch too (otherwise it is carried)
            auto batches = [&](auto kind, int s0, int s1, bool end) {
                constexpr int K = decltype(kind)::value;
                const int total = n_carry + s1 - s0;
                int t0 = 0;
                for (; t0 < total; t0 += 32) {
                    const int t = t0 + lane, cnt = min(32, total - t0);
                    // (lanes outside the codes read a neighbouring place of the warp's buffer)
                    const uint32_t c = wb.code[s0 - n_carry + t] & 2047u;
                    uint32_t e = blk + c;
                    if (t < n_carry) e = carry_e;
                    if (cnt < 32) {
                        if (!end) {
                            carry_e = e;
                            break;
                        }
                        const uint32_t e0 = __shfl_sync(0xffffffffu, e, 0);
                        if (lane >= cnt) e = e0;
                    }
                    real rt;
                    uint32_t key;
                    const bool opp = K == 2 || (K == 3 && (e >> 5) >= gi.y), beta = (K == 1 || K == 3) && (gi.w & 1u);
                    const real h = flat_value<K, real, kC, scaled>(L, V, orb, e, beta ? M : 0, (opp || beta) ? M : 0, !opp,
                                                           lane < cnt, q, flag, rt, key);
                    if constexpr (kOrder) {
                        // the lane of the entry's unit, modulo 32 (ListsView::group)
                        const uint32_t j = key >> 24, i = key >> 16 & 0xFFu;
                        const uint32_t un = K == 0 ? key : (K == 1 ? j + i * (gi.w >> 1 & 31u) + (gi.w >> 6) : j + (gi.w >> 11));
                        const uint32_t place = e + __shfl_sync(0xffffffffu, to_place, (int)(un & 31u));
                        sum.batch(rmul(h, rt), place, cnt, lane, e_grp);
                    } else {
                        e_grp = __fma_rn(lane < cnt ? h : real(0), rt, e_grp);
                    }
                }
                n_carry = max(0, total - t0);
            };
            if (!pairs) {
                batches(std::integral_constant<int, 0>{}, 0, n, done);
            } else if constexpr (!kOrder) {
                batches(std::integral_constant<int, 3>{}, 0, n, done);
            } else {
                int nA = 0;                              // codes of the block's same-spin part
                if (gi.y > w0) {
                    const uint32_t ws = gi.y - w0, l2 = 2 * (uint32_t)lane;      // words before the opposite-spin part
                    nA = (int)__reduce_max_sync(0xffffffffu, lane >= nl || l2 >= ws ? 0u : (l2 + 1 < ws ? sc : at0 + f0));
                    batches(std::integral_constant<int, 1>{}, 0, nA, w1 >= gi.y);
                }
                if (w1 > gi.y) {
                    if (in_a) {
                        restA = sum.finish(lane, e_grp);
                        sum = StackSum{};
                        in_a = false;
                    }
                    batches(std::integral_constant<int, 2>{}, nA, n, done);
                }
            }
            __syncwarp();
            w0 = w1;
        }
        if constexpr (kOrder) {
            const float rest = sum.finish(lane, e_grp);
            e_grp += restA;
            e_grp += rest;
        }
        u128 q_grp = 0;
        double eg_sum = 0.0;
        if (any) {
            eg_sum = warp_sum_acc(e_grp);   // FP32 lanes in the mixed form: one conversion
            q_grp = warp_sum(q);
        }
        int nxt = 0;
        if (lane == 0) {
            rates[(size_t)w * n_groups + g] = q_grp;
            eg[g] = eg_sum;
            nxt = atomicAdd(&next_group, 1);
        }
        g = __shfl_sync(0xffffffffu, nxt, 0);
    }
    if (flag) atomicOr(status, flag);
    __syncthreads();
    if (warp == 0) {
        // sums over the groups: the energies in a fixed order (lane l takes groups l, l+32, ...), the
        // rates exactly
        double s = 0.0;
        u128 Q = 0;
        for (int g = lane; g < n_groups; g += 32) {
            s += eg[g];
            Q += rates[(size_t)w * n_groups + g];
        }
        s = warp_sum_f64(s);
        Q = warp_sum_u128(Q);
        if (lane == 0) {
            e_loc[w] = A.e_diag[w] + s;
            if (Q == 0) {
                t_res[w] = 0.0;
                atomicOr(status, VMC_DEV_NOMOVE);
            } else {
                const double qh = (double)(uint64_t)(Q >> 64), ql = (double)(uint64_t)Q;
                t_res[w] = __ddiv_rn(1.0, __dadd_rn(qh, __dmul_rn(ql, 0x1p-64)));
            }
        }
    }
    __syncthreads();   // shared memory may be reused for the next walker
}

// CTA widths the local-energy kernels are built for (128, 256, 384, 512 threads), each with the
// minimum of resident CTAs per SM that keeps it at <= 64 registers per thread, so that shared
// memory (the walker's G rows) rather than registers bounds the CTAs per SM.
template <int kT> struct EmB { static constexpr int v = kT >= 512 ? 2 : (kT >= 384 ? 3 : (kT >= 256 ? 4 : 8)); };

template <typename real, int kT, bool kS>
__global__ void __launch_bounds__(kT, EmB<kT>::v)
k_local_energy(ListsView L, WalkerArgs A, int w_first, const uint32_t *__restrict__ bits, double *__restrict__ e_loc,
               double *__restrict__ t_res, u128 *__restrict__ rates, unsigned *status) {
    extern __shared__ __align__(16) unsigned char smraw[];
    eloc_walker<real, false, kS>(L, A, w_first + blockIdx.x, bits ? bits + (size_t)blockIdx.x * L.words : nullptr, e_loc,
                             t_res, rates, status, smraw);
}

// The same with the correlator product (a separate instantiation, so the pair-Jastrow kernel above
// is not touched by it).
template <typename real, int kT, bool kS>
__global__ void __launch_bounds__(kT, EmB<kT>::v)
k_local_energy_cps(ListsView L, WalkerArgs A, CpsView C, int w_first, const uint32_t *__restrict__ bits,
                   double *__restrict__ e_loc, double *__restrict__ t_res, u128 *__restrict__ rates, unsigned *status) {
    extern __shared__ __align__(16) unsigned char smraw[];
    eloc_walker<real, true, kS>(L, A, w_first + blockIdx.x, bits ? bits + (size_t)blockIdx.x * L.words : nullptr, e_loc,
                            t_res, rates, status, smraw, C);
}

// Batched launch over several systems (uneven sizes).  CTAs stay resident and take walkers from
// a global queue; the descriptors are ordered by decreasing cost so the long walkers start first.
template <typename real, int kT>
__global__ void __launch_bounds__(kT, EmB<kT>::v)
k_local_energy_batched(const SysDesc *__restrict__ sys, int n_sys, int total, int *queue, unsigned *status) {
    extern __shared__ __align__(16) unsigned char smraw[];
    __shared__ int s_item;
    for (;;) {
        if (threadIdx.x == 0) s_item = atomicAdd(queue, 1);
        __syncthreads();
        const int t = s_item;
        __syncthreads();
        if (t >= total) break;
        int k = 0;
        while (k + 1 < n_sys && sys[k + 1].w_begin <= t) ++k;
        const SysDesc &d = sys[k];
        const int l = t - d.w_begin;
        const uint32_t *row = d.bits + (size_t)l * d.L.words;
        if (sizeof(real) == 8 && d.L.scaled)
            eloc_walker<real, false, sizeof(real) == 8>(d.L, d.A, d.w_first + l, row, d.e_loc, d.t_res, d.rates, status, smraw);
        else
            eloc_walker<real, false, false>(d.L, d.A, d.w_first + l, row, d.e_loc, d.t_res, d.rates, status, smraw);
    }
}

// ---------------------------------------------------------------------------------- CTMC
// Selection: one warp per walker.  Scans the walker's group sums (u128), draws Philox, finds the
// group whose prefix crosses T and evaluates only that group's free entries, 32 at a time in canonical
// order, with the values of the local-energy kernel.  Writes the move code (0 = no move) and advances the
// walker's counter.  The free entries come from the rows of bits that the local energy left (row), or
// are found here, a word of 32 entries per step (null).  A warp per walker has nothing to hide its
// latency behind in a small call, so what counts is the number of dependent steps: one per 32 free
// entries instead of one per occupied unit (256 walkers of the 10-site ring: 36 -> 26 us for choice and
// update).
template <typename real, bool kC>
__device__ __forceinline__ void select_walker(const ListsView &L, const WalkerArgs &A, const int w,
                                              const u128 *__restrict__ rates, const uint32_t *__restrict__ row,
                                              uint64_t seed, uint64_t *__restrict__ move_code, unsigned *status,
                                              WarpBuf &wb, const CpsView &C = CpsView{}) {
    const Geo geo = make_geo(A.M, A.na, A.nb);
    const int lane = threadIdx.x & 31;
    const int M = geo.M, N2 = 2 * M, n_groups = L.n_groups;
    const real *Gw = (const real *)A.G + (size_t)w * geo.g_stride;
    const real *Sw = (const real *)A.S + (size_t)w * N2;
    const u128 *R = rates + (size_t)w * n_groups;
    const int per = (n_groups + 31) / 32;
    const int g0 = lane * per, g1 = min(n_groups, g0 + per);
    u128 seg = 0;
    for (int g = g0; g < g1; ++g) seg += R[g];
    const u128 incl = warp_incl_scan_u128(seg, lane);
    const u128 Q = shfl_u128(incl, 31);
    const uint64_t U = philox4x64_word0(A.rng[w], 0, 0, 0, seed, (uint64_t)w);
    const uint64_t qh = (uint64_t)(Q >> 64), ql = (uint64_t)Q;
    const u128 T = (u128)U * qh + (u128)__umul64hi(U, ql);
    const unsigned ball = __ballot_sync(0xffffffffu, incl > T);
    int gsel = -1;
    u128 before = 0;
    if (Q != 0 && ball) {
        const int src = __ffs(ball) - 1;
        u128 pre = shfl_u128(incl - seg, src);
        if (lane == src) {
            for (int g = g0; g < g1; ++g) {
                if (pre + R[g] > T) { gsel = g; break; }
                pre += R[g];
            }
        }
        gsel = __shfl_sync(0xffffffffu, gsel, src);
        before = shfl_u128(pre, src);
    }
    uint64_t code = 0;
    if (gsel >= 0) {
        const u128 Tl = T - before;   // threshold inside the group
        View<real> V;
        V.pos = A.pos + (size_t)w * N2; V.Ga = Gw; V.Gb = Gw + geo.g_off(1); V.lda = geo.na; V.ldb = geo.nb;
        V.S = Sw; V.F = (const real *)A.F + (size_t)w * 2 * L.ns_pad; V.geo = geo;
        if (kC) cps_global(V, C, A.cps + (size_t)w * C.n_corr);
        const uint4 gi = __ldg(&L.group[gsel]);
        const bool single = gsel < (N2 + 31) / 32;
        const uint32_t *ow = A.occ_bits + (size_t)w * 2 * geo.nw;
        u128 carry = 0;
        unsigned flag = 0;
        bool found = false;
        for (uint32_t w0 = gi.x; w0 < gi.z && !found;) {
            // 32 words of the group, one per lane; their free entries' codes
            const uint32_t nw = min(32u, gi.z - w0);
            uint32_t x = 0;
            if (row) {
                if ((uint32_t)lane < nw) x = row[w0 + lane];
            } else {
                for (uint32_t k = 0; k < nw; ++k) {
                    const uint32_t y = free_word(L, ow, geo.nw, (int)(w0 + k), lane);
                    if ((uint32_t)lane == k) x = y;
                }
            }
            uint32_t sc = __popc(x);
            const uint32_t own = sc;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const uint32_t o = __shfl_up_sync(0xffffffffu, sc, d);
                if (lane >= d) sc += o;
            }
            const int nl = min((int)nw, __popc(__ballot_sync(0xffffffffu, sc <= (uint32_t)kFreeMax)));
            if (lane < nl) {
                uint16_t *at = wb.code + (sc - own);
                for (; x; x &= x - 1u) *at++ = (uint16_t)(lane << 5 | (__ffs(x) - 1));
            }
            __syncwarp();
            const int n = (int)__shfl_sync(0xffffffffu, sc, nl - 1);
            for (int t0 = 0; t0 < n && !found; t0 += 32) {
                u128 q = 0;
                uint64_t mc = 0;
                if (t0 + lane < n) {
                    real ratio, contrib;
                    if (flat_entry_value<real, kC>(L, V, single, w0 * 32u + wb.code[t0 + lane], ratio, contrib, mc))
                        q = rate_of<real>(ratio, &flag);
                }
                const u128 incl2 = warp_incl_scan_u128(q, lane) + carry;
                const unsigned hit = __ballot_sync(0xffffffffu, q != 0 && incl2 > Tl);
                if (hit) {
                    code = __shfl_sync(0xffffffffu, mc, __ffs(hit) - 1);
                    found = true;
                }
                carry = shfl_u128(incl2, 31);
            }
            __syncwarp();
            w0 += (uint32_t)nl;
        }
        if (!found && lane == 0) atomicOr(status, VMC_DEV_INCONSISTENT);
    } else if (lane == 0) {
        atomicOr(status, VMC_DEV_NOMOVE);
    }
    if (lane == 0) {
        move_code[w] = code;
        A.rng[w] += 1;
    }
}

// bits: the rows of all walkers, or null
template <typename real, bool kC>
__global__ void __launch_bounds__(VMC_THREADS)
k_ctmc_select(ListsView L, WalkerArgs A, CpsView C, const u128 *__restrict__ rates, const uint32_t *__restrict__ bits,
              uint64_t seed, uint64_t *__restrict__ move_code, unsigned *status) {
    __shared__ WarpBuf bufs[VMC_WARPS];
    const int w = blockIdx.x * VMC_WARPS + (threadIdx.x >> 5);
    if (w >= A.W) return;
    select_walker<real, kC>(L, A, w, rates, bits ? bits + (size_t)w * L.words : nullptr, seed, move_code, status,
                            bufs[threadIdx.x >> 5], C);
}

// use_bits: the descriptors' rows hold all walkers (one round)
template <typename real>
__global__ void __launch_bounds__(VMC_THREADS)
k_ctmc_select_batched(const SysDesc *__restrict__ sys, int n_sys, int total, int use_bits, uint64_t seed, unsigned *status) {
    __shared__ WarpBuf bufs[VMC_WARPS];
    const int t = blockIdx.x * VMC_WARPS + (threadIdx.x >> 5);
    if (t >= total) return;
    int k = 0;
    while (k + 1 < n_sys && sys[k + 1].w_begin <= t) ++k;
    const SysDesc &d = sys[k];
    const int w = t - d.w_begin;
    select_walker<real, false>(d.L, d.A, w, d.rates, use_bits ? d.bits + (size_t)w * d.L.words : nullptr, seed, d.move_code,
                               status, bufs[threadIdx.x >> 5]);
}

// Screened move set of one walker, written out in canonical order (Sec. II.A, II.B): one warp per
// walker walks the same groups, units and list entries as the local energy (groups in index order,
// units in lane order, entries in list order) and writes every entry whose targets are free with
// the ratio and contribution the local energy and the CTMC choice use.  Diagnostic path: it also
// counts the list entries the walk reads (singles, doubles), free or not.
template <typename real, bool kC>
__global__ void __launch_bounds__(256)
k_screened_moves(ListsView L, WalkerArgs A, CpsView C, int w_begin, int n_w, int64_t cap, uint64_t *__restrict__ code_out,
                 double *__restrict__ ratio_out, double *__restrict__ contrib_out, int64_t *__restrict__ count_out,
                 int64_t *__restrict__ walked_out, unsigned *status) {
    const int t = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (t >= n_w) return;
    const int w = w_begin + t;
    const int lane = threadIdx.x & 31;
    const Geo geo = make_geo(A.M, A.na, A.nb);
    const int M = geo.M, N2 = 2 * M;
    const real *Gw = (const real *)A.G + (size_t)w * geo.g_stride;
    View<real> V;
    V.pos = A.pos + (size_t)w * N2; V.Ga = Gw; V.Gb = Gw + geo.g_off(1); V.lda = geo.na; V.ldb = geo.nb;
    V.S = (const real *)A.S + (size_t)w * N2; V.F = (const real *)A.F + (size_t)w * 2 * L.ns_pad;
    V.geo = geo;
    if (kC) cps_global(V, C, A.cps + (size_t)w * C.n_corr);
    const unsigned lt_mask = (1u << lane) - 1u;
    int64_t cnt = 0, walked_s = 0, walked_d = 0;
    unsigned flag = 0;
    for (int g = 0; g < L.n_groups; ++g) {
        Unit<real> u;
        const bool act = setup_unit<real>(L, V, g, lane, u);
        unsigned mask = __ballot_sync(0xffffffffu, act);
        while (mask) {
            const int src = __ffs(mask) - 1;
            mask &= mask - 1;
            const Unit<real> v = shfl_unit(u, src);
            if (v.base + v.len > 32u * (uint32_t)L.words) {   // cannot happen: guard, never read
                flag |= VMC_DEV_INCONSISTENT;
                continue;
            }
            if (v.kind == 0) walked_s += v.len; else walked_d += v.len;
            for (uint32_t k0 = 0; k0 < v.len; k0 += 32) {
                const uint32_t k = k0 + lane;
                real ratio = 0, contrib = 0;
                int a = -1, b = -1;
                const bool fr = k < v.len && eval_entry<real, kC>(L, V, v, v.base + k, ratio, contrib, a, b);
                const unsigned bal = __ballot_sync(0xffffffffu, fr);
                if (fr) {
                    const int64_t p = cnt + __popc(bal & lt_mask);
                    if (p < cap) {
                        const uint64_t kind = v.kind == 0 ? 1 : 2;
                        const uint64_t j10 = kind == 2 ? (uint64_t)v.j : 1023ull, b10 = kind == 2 ? (uint64_t)b : 1023ull;
                        const size_t o = (size_t)t * (size_t)cap + (size_t)p;
                        code_out[o] = kind | ((uint64_t)v.i << 2) | (j10 << 12) | ((uint64_t)a << 22) | (b10 << 32);
                        ratio_out[o] = (double)ratio;
                        contrib_out[o] = (double)contrib;
                    }
                }
                cnt += __popc(bal);
            }
        }
    }
    if (lane == 0) {
        count_out[t] = cnt;
        if (walked_out) {
            walked_out[2 * (size_t)t] = walked_s;
            walked_out[2 * (size_t)t + 1] = walked_d;
        }
        if (flag) atomicOr(status, flag);
    }
}

// Asks for [p, p + bytes) in L2 (whole 16-byte pieces inside it).
__device__ __forceinline__ void prefetch_l2(const void *p, size_t bytes) {
    const uintptr_t a = ((uintptr_t)p + 15) & ~(uintptr_t)15, b = ((uintptr_t)p + bytes) & ~(uintptr_t)15;
    if (b > a) asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(a), "r"((uint32_t)(b - a)) : "memory");
}

// Move update: one CTA per walker (Sec. III.B): diagonal energy, Jastrow sums, Fock sums, then the
// rank-1 (singles, opposite-spin doubles) or rank-2 Woodbury (same-spin doubles) update of G and
// AinvT, and the occupation lists, bits and orbital map.
template <typename real, bool kC>
__device__ __forceinline__ void apply_walker(const ListsView &L, const WalkerArgs &A, const double *__restrict__ J,
                                             const int w, const uint64_t *__restrict__ move_code,
                                             unsigned char *smraw, const CpsView &C = CpsView{}) {
    const Geo geo = make_geo(A.M, A.na, A.nb);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nt = blockDim.x, nwarp = nt >> 5;
    const uint64_t code = move_code[w];
    if (code == 0) return;
    const int M = geo.M, ne = geo.ne, N2 = 2 * M;
    uint16_t *pos = (uint16_t *)smraw;
    real *vec = (real *)(smraw + ((2 * sizeof(uint16_t) * (size_t)M + 15) & ~(size_t)15));
    // vec holds: ua[nmax], ub[nmax], gci[M], gcj[M], arow_i[nmax], arow_j[nmax]
    __shared__ double red[32];
    real *Gw = (real *)A.G + (size_t)w * geo.g_stride;
    real *Aw = (real *)A.AinvT + (size_t)w * geo.a_stride;
    real *Sw = (real *)A.S + (size_t)w * N2;
    uint16_t *occ = A.occ_list + (size_t)w * ne;
    uint16_t *virt = A.virt_list + (size_t)w * (2 * M - ne);
    uint32_t *bits = A.occ_bits_w + (size_t)w * 2 * geo.nw;
    uint16_t *posw = A.pos + (size_t)w * N2;
    if (tid == 0 && (geo.g_stride + geo.a_stride) * sizeof(real) <= 48 * 1024) {
        // the rank updates come last and stream G and C_occ^-1: bring them to L2 while the sums are updated, as long
        // as the walkers of all resident CTAs (six per SM) take less than half of it (choice and update of 4,096
        // walkers of H100, mixed: 205 -> 181 us; at H160, 102 KB a walker, 1.52 -> 1.63 ms for 32,768)
        prefetch_l2(Gw, geo.g_stride * sizeof(real));
        prefetch_l2(Aw, geo.a_stride * sizeof(real));
    }
    for (int p = tid; p < N2; p += nt) pos[p] = posw[p];
    __syncthreads();
    const int kind = (int)(code & 3), I = (int)((code >> 2) & 1023), Jo = (int)((code >> 12) & 1023);
    const int Ao = (int)((code >> 22) & 1023), Bo = (int)((code >> 32) & 1023);
    // ---- correlator indices: every (changed orbital, covering correlator) adds its digit change
    if (kC && tid == 0) {
        uint16_t *ci = A.cps + (size_t)w * C.n_corr;
        const int chg[4] = {I, Ao, Jo, Bo};
        for (int x = 0; x < (kind == 2 ? 4 : 2); ++x) {
            const int sp = chg[x] >= M ? 1 : 0, site = chg[x] - sp * M, dg = ((x & 1) ? 1 : -1) * (1 + sp);
            for (int h = C.site_off[site]; h < C.site_off[site + 1]; ++h) {
                const uint32_t ent = C.site_ent[h];
                ci[ent >> 16] = (uint16_t)((int)ci[ent >> 16] + dg * (int)(ent & 0xFFFFu));
            }
        }
    }

    // ---- diagonal energy change (old occupation), FP64
    {
        auto D = [&](int p, int q) -> double {
            const int kp = p % M, kq = q % M;
            double d = L.Jd[(size_t)kp * M + kq];
            if ((p >= M) == (q >= M)) d -= L.Kd[(size_t)kp * M + kq];
            return d;
        };
        double part = 0.0;
        for (int t = tid; t < ne; t += nt) {
            const int K = (t < geo.na ? 0 : M) + occ[t];
            if (K != I) part += D(Ao, K) - D(I, K);
            if (kind == 2 && K != I && K != Jo) part += D(Bo, K) - D(Jo, K);
        }
        part = warp_sum_f64(part);
        if (lane == 0) red[warp] = part;
        __syncthreads();
        if (tid == 0) {
            double dE = L.hd[Ao % M] - L.hd[I % M];
            if (kind == 2) dE += L.hd[Bo % M] - L.hd[Jo % M] + D(Bo, Ao) - D(Jo, Ao);
            for (int k = 0; k < nwarp; ++k) dE += red[k];
            A.e_diag[w] += dE;
        }
    }
    // ---- Jastrow sums: S_p += J_pa [p != a] - J_pi [p != i]  (twice for doubles)
    for (int p = tid; p < N2; p += nt) {
        double d = 0.0;
        if (p != Ao) d += jget(J, N2, p, Ao);
        if (p != I) d -= jget(J, N2, p, I);
        if (kind == 2) {
            if (p != Bo) d += jget(J, N2, p, Bo);
            if (p != Jo) d -= jget(J, N2, p, Jo);
        }
        Sw[p] = (real)((double)Sw[p] + d);
    }
    // ---- Fock sums: each changed spin orbital k of spin t adds +-Tjk[k] to spin t, +-Tj[k] to the other
    {
        typedef typename Vec16<real>::type vec_t;
        constexpr int VE = Vec16<real>::n;
        const int64_t np = L.ns_pad, nvec = np / VE;
        vec_t *F0 = (vec_t *)((real *)A.F + (size_t)w * 2 * np), *F1 = F0 + nvec;
        const real *Tk = fock_table<real>(L, 1), *Tx = fock_table<real>(L, 0);
        const int nch = kind == 2 ? 4 : 2;
        const int chg[4] = {I, Ao, Jo, Bo};
        for (int64_t v = tid; v < nvec; v += nt) {
            vec_t f0 = F0[v], f1 = F1[v];
            for (int c = 0; c < nch; ++c) {
                const int p = chg[c];
                const real sgn = (c & 1) ? real(1) : real(-1);
                const int t = p >= M, k = p - t * M;
                const vec_t jk = __ldg((const vec_t *)(Tk + (size_t)k * np) + v);
                const vec_t jj = __ldg((const vec_t *)(Tx + (size_t)k * np) + v);
                if (t == 0) { vadd(f0, sgn, jk); vadd(f1, sgn, jj); }
                else { vadd(f1, sgn, jk); vadd(f0, sgn, jj); }
            }
            F0[v] = f0; F1[v] = f1;
        }
    }
    // ---- determinant tables: rank-1 per spin (singles, opposite-spin doubles) or rank-2
    //      Woodbury (same-spin doubles) on G and AinvT (Sherman-Morrison, Sec. III.B)
    const int nmax = geo.na > geo.nb ? geo.na : geo.nb, np4 = (nmax + 3) & ~3, mp4 = (M + 3) & ~3;
    real *ua = vec, *ub = ua + np4, *gci = ub + np4, *gcj = gci + mp4, *ari = gcj + mp4, *arj = ari + np4;
    int nsteps = 1;
    int sp[2], fr[2][2], to[2][2], rk[2];
    const int si = I >= M;
    if (kind == 1) { sp[0] = si; fr[0][0] = I - si * M; to[0][0] = Ao - si * M; rk[0] = 1; }
    else if (Jo / M == si) {   // same-spin double
        sp[0] = si; rk[0] = 2;
        fr[0][0] = I - si * M; to[0][0] = Ao - si * M; fr[0][1] = Jo - si * M; to[0][1] = Bo - si * M;
    } else {                   // opposite spin: alpha i->a, beta j->b
        nsteps = 2;
        sp[0] = 0; rk[0] = 1; fr[0][0] = I; to[0][0] = Ao;
        sp[1] = 1; rk[1] = 1; fr[1][0] = Jo - M; to[1][0] = Bo - M;
    }
    // The vectors of step st: ua/ub = R^-1 (G[(a,b),:] - E) with R = G[(a,b), (ci,cj)], the old
    // columns ci (cj) of G and rows ci (cj) of C_occ^-1.  u2, g2, a2 may be null for a rank-1 step
    // (then the second term of the update is zero).
    auto prep = [&](int st, real *u1, real *u2, real *g1, real *g2, real *a1, real *a2) {
        const int s = sp[st], n = geo.n(s), nv = M - n;
        const real *Gs = Gw + geo.g_off(s);
        const real *As = Aw + geo.a_off(s);
        const int ci = pos[s * M + fr[st][0]], sa = pos[s * M + to[st][0]] & 0x7FFF;
        int cj = 0, sb = 0;
        if (rk[st] == 2) { cj = pos[s * M + fr[st][1]]; sb = pos[s * M + to[st][1]] & 0x7FFF; }
        real r00 = Gs[(size_t)sa * n + ci], r01 = 0, r10 = 0, r11 = 1;
        if (rk[st] == 2) { r01 = Gs[(size_t)sa * n + cj]; r10 = Gs[(size_t)sb * n + ci]; r11 = Gs[(size_t)sb * n + cj]; }
        const real det = r00 * r11 - r01 * r10;
        const real i00 = r11 / det, i01 = -r01 / det, i10 = -r10 / det, i11 = r00 / det;
        for (int c = tid; c < n; c += nt) {
            const real va = Gs[(size_t)sa * n + c] - (c == ci ? (real)1 : (real)0);
            const real vb = rk[st] == 2 ? Gs[(size_t)sb * n + c] - (c == cj ? (real)1 : (real)0) : (real)0;
            u1[c] = i00 * va + i01 * vb;
            a1[c] = As[(size_t)ci * n + c];
            if (u2) {
                u2[c] = i10 * va + i11 * vb;
                a2[c] = rk[st] == 2 ? As[(size_t)cj * n + c] : (real)0;
            }
        }
        for (int r = tid; r < nv; r += nt) {
            real x = Gs[(size_t)r * n + ci], y = rk[st] == 2 ? Gs[(size_t)r * n + cj] : (real)0;
            if (r == sa) { x = 1; y = 0; }
            if (rk[st] == 2 && r == sb) { x = 0; y = 1; }
            g1[r] = x;
            if (g2) g2[r] = y;
        }
    };
    // G <- G - g1 u1^T - g2 u2^T (replaced rows taken as unit vectors), C_occ^-1 likewise
    auto update = [&](int st, const real *u1, const real *u2, const real *g1, const real *g2, const real *a1,
                      const real *a2) {
        const int s = sp[st], n = geo.n(s), nv = M - n;
        real *Gs = Gw + geo.g_off(s);
        real *As = Aw + geo.a_off(s);
        const int ci = pos[s * M + fr[st][0]], sa = pos[s * M + to[st][0]] & 0x7FFF;
        int cj = 0, sb = 0;
        if (rk[st] == 2) { cj = pos[s * M + fr[st][1]]; sb = pos[s * M + to[st][1]] & 0x7FFF; }
        typedef typename Vec16<real>::type vec_t;
        constexpr int VE = Vec16<real>::n;
        const bool rk2 = rk[st] == 2;
        if (n % VE == 0 && n > 0 && ((((uintptr_t)Gs) | ((uintptr_t)As)) & 15) == 0) {
            // 16-byte vectors: thread -> fixed column chunk cv, rows r0, r0 + rs, ...
            const int nvc = n / VE, cv = tid % nvc, r0 = tid / nvc, rs = nt / nvc, c0 = cv * VE;
            if (r0 < rs) {
                vec_t zero;
                real *ze = (real *)&zero;
#pragma unroll
                for (int q = 0; q < VE; ++q) ze[q] = real(0);
                const vec_t u = *(const vec_t *)(u1 + c0), v = u2 ? *(const vec_t *)(u2 + c0) : zero;
                vec_t *Gv = (vec_t *)Gs;
#pragma unroll 4
                for (int r = r0; r < nv; r += rs) {
                    vec_t o = Gv[(size_t)r * nvc + cv];
                    if (r == sa || (rk2 && r == sb)) {   // replaced row: old value is a unit vector
                        const int cu = r == sa ? ci : cj;
                        real *oe = (real *)&o;
#pragma unroll
                        for (int q = 0; q < VE; ++q) oe[q] = (c0 + q == cu) ? real(1) : real(0);
                    }
                    Gv[(size_t)r * nvc + cv] = vfma2(o, g1[r], u, g2 ? g2[r] : real(0), v);
                }
                const vec_t b1 = *(const vec_t *)(a1 + c0), b2 = a2 ? *(const vec_t *)(a2 + c0) : zero;
                vec_t *Av = (vec_t *)As;
#pragma unroll 4
                for (int c = r0; c < n; c += rs)
                    Av[(size_t)c * nvc + cv] = vfma2(Av[(size_t)c * nvc + cv], u1[c], b1, u2 ? u2[c] : real(0), b2);
            }
        } else {
            for (size_t t = tid; t < (size_t)nv * n; t += nt) {
                const int r = (int)(t / n), c = (int)(t % n);
                real old = Gs[t];
                if (r == sa) old = (c == ci) ? (real)1 : (real)0;
                if (rk2 && r == sb) old = (c == cj) ? (real)1 : (real)0;
                Gs[t] = old - g1[r] * u1[c] - (g2 ? g2[r] : real(0)) * (u2 ? u2[c] : real(0));
            }
            for (size_t t = tid; t < (size_t)n * n; t += nt) {
                const int c = (int)(t / n), x = (int)(t % n);
                As[t] = As[t] - u1[c] * a1[x] - (u2 ? u2[c] : real(0)) * (a2 ? a2[x] : real(0));
            }
        }
    };
    // occupation list, virtual list, orbital map and bit string of step st (one thread)
    auto relist = [&](int st) {
        const int s = sp[st];
        uint16_t *occs = occ + (s ? geo.na : 0);
        uint16_t *virts = virt + (s ? geo.nv_a : 0);
        const int ci = pos[s * M + fr[st][0]], sa = pos[s * M + to[st][0]] & 0x7FFF;
        int cj = 0, sb = 0;
        if (rk[st] == 2) { cj = pos[s * M + fr[st][1]]; sb = pos[s * M + to[st][1]] & 0x7FFF; }
        occs[ci] = (uint16_t)to[st][0];
        virts[sa] = (uint16_t)fr[st][0];
        posw[s * M + to[st][0]] = (uint16_t)ci;
        posw[s * M + fr[st][0]] = (uint16_t)(0x8000 | sa);
        if (rk[st] == 2) {
            occs[cj] = (uint16_t)to[st][1];
            virts[sb] = (uint16_t)fr[st][1];
            posw[s * M + to[st][1]] = (uint16_t)cj;
            posw[s * M + fr[st][1]] = (uint16_t)(0x8000 | sb);
        }
        uint32_t *bw = bits + s * geo.nw;
        for (int k = 0; k < rk[st]; ++k) {
            const int f = fr[st][k], tt = to[st][k];
            bw[f >> 5] &= ~(1u << (f & 31));
            bw[tt >> 5] |= 1u << (tt & 31);
        }
    };
    __syncthreads();
    if (nsteps == 2) {   // opposite-spin double: the two spins' rank-1 updates share the phases
        prep(0, ua, nullptr, gci, nullptr, ari, nullptr);
        prep(1, ub, nullptr, gcj, nullptr, arj, nullptr);
        __syncthreads();
        update(0, ua, nullptr, gci, nullptr, ari, nullptr);
        update(1, ub, nullptr, gcj, nullptr, arj, nullptr);
        __syncthreads();
        if (tid == 0) { relist(0); relist(1); }
    } else {
        prep(0, ua, ub, gci, gcj, ari, arj);
        __syncthreads();
        update(0, ua, ub, gci, gcj, ari, arj);
        __syncthreads();
        if (tid == 0) relist(0);
    }
}


// 256 threads per walker; six resident CTAs per SM (<= 40 registers): the update is bound by HBM
// latency between its barrier-separated phases, so more walkers in flight per SM pay (12 % faster
// than four per SM at H160, with a few spilled registers)
template <typename real, bool kC>
__global__ void __launch_bounds__(256, 6)
k_ctmc_apply(ListsView L, WalkerArgs A, CpsView C, const double *__restrict__ J, const uint64_t *__restrict__ move_code) {
    extern __shared__ __align__(16) unsigned char smraw[];
    apply_walker<real, kC>(L, A, J, blockIdx.x, move_code, smraw, C);
}

// (The same bounds: left to itself the compiler took 114 registers, two CTAs per SM; the uneven batch of seven systems
// of 2,048 walkers: 725 -> 286 us.)
template <typename real>
__global__ void __launch_bounds__(256, 6)
k_ctmc_apply_batched(const SysDesc *__restrict__ sys, int n_sys) {
    extern __shared__ __align__(16) unsigned char smraw[];
    const int t = blockIdx.x;
    int k = 0;
    while (k + 1 < n_sys && sys[k + 1].w_begin <= t) ++k;
    const SysDesc &d = sys[k];
    apply_walker<real, false>(d.L, d.A, d.J, t - d.w_begin, d.move_code, smraw);
}

}  // namespace

// Shared memory of a local-energy CTA: G rows, orbital table, occupation words, warp buffers and the
// correlator tables.
static size_t eloc_smem_bytes(const ListsView &L, const vmc_walkers *Wk, const CpsView &C, int threads) {
    const bool d = Wk->precision == VMC_FP64;
    const size_t esz = d ? 8 : 4, M = (size_t)Wk->M, na = (size_t)Wk->n_alpha, nb = (size_t)Wk->n_beta;
    const size_t g = esz * ((M - na) * (na + 1) + (M - nb) * (nb + 1)) + 8;
    const size_t orb = (d ? OrbTable<double>::bytes : OrbTable<float>::bytes) * 2 * M + 4 * 2 * ((M + 31) / 32) + 16;
    const size_t warps = (size_t)(threads / 32) * sizeof(WarpBuf);
    // correlator product: 1/c per correlator (padded to 4), coefficient positions and offsets
    const size_t cps = C.n_corr ? esz * (size_t)((C.n_corr + 3) & ~3) + 4 * (2 * (size_t)C.n_corr + 1) : 0;
    const size_t own = own_rows(L.words, Wk->W) ? 4 * (size_t)L.words : 0;      // its bits
    return g + orb + own + warps + cps;
}

// Which walkers the local energy takes: G rows, exp(S), orbital map, 512 bytes per warp and the correlator tables
// within 200 KB.  The line counts the per-site correlator lists, which are no longer staged: what is refused stays
// the same, and the CTA's own sum (eloc_smem_bytes) stays within the 227 KB that it can have.
static bool eloc_fits(const vmc_walkers *Wk, const CpsView &C, int threads) {
    const size_t esz = Wk->precision == VMC_FP64 ? 8 : 4, M = (size_t)Wk->M, na = (size_t)Wk->n_alpha, nb = (size_t)Wk->n_beta;
    const size_t cps = C.n_corr ? esz * (size_t)((C.n_corr + 3) & ~3) + 4 * (2 * (size_t)C.n_corr + 1) + 4 * (M + 1) + 4 * (size_t)C.nnz : 0;
    return esz * ((M - na) * (na + 1) + (M - nb) * (nb + 1) + 2 * M) + 4 * M + 16 + 512 * (size_t)(threads / 32) + cps <= 200 * 1024;
}

static WalkerArgs make_args(vmc_walkers *Wk) {
    WalkerArgs A;
    A.W = Wk->W; A.M = Wk->M; A.na = Wk->n_alpha; A.nb = Wk->n_beta;
    A.occ_bits = Wk->occ_bits; A.occ_bits_w = Wk->occ_bits;
    A.occ_list = Wk->occ_list; A.virt_list = Wk->virt_list; A.pos = Wk->pos;
    A.G = Wk->G; A.AinvT = Wk->AinvT; A.S = Wk->S; A.F = Wk->F; A.e_diag = Wk->e_diag;
    A.rng = Wk->rng_counter;
    A.cps = Wk->cps_state;
    return A;
}

template <typename real, int kT, bool kS>
static cudaError_t eloc_launch_t(const vmc_ctx *ctx, int w0, int W, size_t smem, const ListsView &L, const WalkerArgs &A,
                                 const CpsView &C, double *e_loc, double *t_res, u128 *rates) {
    const uint32_t *bits = own_rows(L.words, A.W) ? nullptr : (const uint32_t *)ctx->bits;
    cudaError_t e;
    if (C.n_corr) {
        e = cudaFuncSetAttribute(k_local_energy_cps<real, kT, kS>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e == cudaSuccess)
            e = launch_dependent(bits != nullptr, k_local_energy_cps<real, kT, kS>, dim3(W), kT, smem, ctx->stream, L, A, C,
                                 w0, bits, e_loc, t_res, rates, ctx->d_status);
        return e;
    }
    e = cudaFuncSetAttribute(k_local_energy<real, kT, kS>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e == cudaSuccess)
        e = launch_dependent(bits != nullptr, k_local_energy<real, kT, kS>, dim3(W), kT, smem, ctx->stream, L, A, w0, bits,
                             e_loc, t_res, rates, ctx->d_status);
    return e;
}
template <typename real, bool kS>
static cudaError_t eloc_launch(const vmc_ctx *ctx, int w0, int W, size_t smem, const ListsView &L, const WalkerArgs &A,
                               const CpsView &C, double *e_loc, double *t_res, u128 *rates) {
    switch (ctx->eloc_threads) {
    case 128: return eloc_launch_t<real, 128, kS>(ctx, w0, W, smem, L, A, C, e_loc, t_res, rates);
    case 256: return eloc_launch_t<real, 256, kS>(ctx, w0, W, smem, L, A, C, e_loc, t_res, rates);
    case 384: return eloc_launch_t<real, 384, kS>(ctx, w0, W, smem, L, A, C, e_loc, t_res, rates);
    default: return eloc_launch_t<real, 512, kS>(ctx, w0, W, smem, L, A, C, e_loc, t_res, rates);
    }
}
template <typename real, int kT>
static cudaError_t eloc_batched_launch_t(const vmc_ctx *ctx, int nsm, size_t se, const SysDesc *tab, int n, int total) {
    int per_sm = 0;
    cudaError_t e = cudaFuncSetAttribute(k_local_energy_batched<real, kT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)se);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_local_energy_batched<real, kT>, kT, se);
    if (e == cudaSuccess)
        e = launch_dependent(true, k_local_energy_batched<real, kT>, dim3(std::max(1, per_sm) * nsm), kT, se, ctx->stream, tab, n,
                             total, ctx->d_queue, ctx->d_status);
    return e;
}
template <typename real>
static cudaError_t eloc_batched_launch(const vmc_ctx *ctx, int nsm, size_t se, const SysDesc *tab, int n, int total) {
    switch (ctx->eloc_threads) {
    case 128: return eloc_batched_launch_t<real, 128>(ctx, nsm, se, tab, n, total);
    case 256: return eloc_batched_launch_t<real, 256>(ctx, nsm, se, tab, n, total);
    case 384: return eloc_batched_launch_t<real, 384>(ctx, nsm, se, tab, n, total);
    default: return eloc_batched_launch_t<real, 512>(ctx, nsm, se, tab, n, total);
    }
}

// Rate store and, behind it in the same allocation, the free-entry rows of one launch's walkers: at most
// kBitsCap bytes of rows (but those of 32 walkers at least); a larger call runs in several launches of *chunk
// walkers.  row = 0: no rows.  When the memory cannot be had the chunk is halved, down to 32 walkers.  A size that
// could not be had is not asked for again where fewer rows will do: the calls after the first find the store as it
// is, allocate nothing and wait for nothing (they may be captured).
constexpr size_t kBitsCap = (size_t)1 << 30;

static size_t row_bytes(const ListsView &L) { return std::max<size_t>(32, sizeof(uint32_t) * (size_t)L.words); }
static size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

// Frees the store and allocates `bytes`; a failed allocation leaves none.
static cudaError_t grow_store(vmc_ctx *ctx, size_t bytes) {
    drop_rates(ctx);
    if (ctx->rates) {
        const cudaError_t e = cudaStreamSynchronize(ctx->stream);
        if (e != cudaSuccess) return e;
        cudaFree(ctx->rates);
        ctx->rates = nullptr;
        ctx->rates_bytes = 0;
    }
    const cudaError_t e = cudaMalloc(&ctx->rates, bytes);
    if (e == cudaSuccess) {
        ctx->rates_bytes = bytes;
        if (bytes >= ctx->rates_refused) ctx->rates_refused = SIZE_MAX;
    } else {
        ctx->rates = nullptr;
    }
    if (e == cudaErrorMemoryAllocation) {
        cudaGetLastError();
        ctx->rates_refused = std::min(ctx->rates_refused, bytes);
    }
    return e;
}

static vmc_status ensure_store(vmc_ctx *ctx, size_t rates_bytes, size_t row, int W, int *chunk) {
    const size_t r = align256(rates_bytes);
    int n = row ? (W + 31) & ~31 : W;
    if (row) {
        const size_t fit = kBitsCap / row & ~(size_t)31;
        if ((size_t)n > fit) n = std::max(32, (int)fit);
    }
    for (;; n = std::max(32, (n / 2 + 31) & ~31)) {
        const size_t bytes = r + row * (size_t)n + 32;     // a read of two words may run past the last row
        if (bytes <= ctx->rates_bytes) break;
        if (row && n > 32 && bytes >= ctx->rates_refused) continue;
        const cudaError_t e = grow_store(ctx, bytes);
        if (e == cudaSuccess) break;
        if (e != cudaErrorMemoryAllocation || !row || n <= 32) return cuda_check(ctx, e, "rate store");
    }
    *chunk = n;
    ctx->bits = (char *)ctx->rates + r;
    return VMC_OK;
}

// Splits of a walker tile's row over CTAs: about 32 CTAs per SM (several short waves), each warp with at
// least two pieces of 256 entries so that the tile's transposed occupations pay, or one while all
// CTAs are resident at once (five per SM) and latency counts.
static int free_bits_parts(int tiles, int words) {
    const int pieces = words / 8, one = std::max(1, (pieces + 7) / 8);
    if ((int64_t)one * tiles <= 152 * 5) return one;
    const int want = (152 * 32 + tiles - 1) / tiles, most = std::max(1, (pieces + 15) / 16);
    return std::max(1, std::min(want, most));
}

vmc_status launch_local_energy(vmc_ctx *ctx, const vmc_lists *L, vmc_walkers *Wk, const CpsView &C, double *e_loc,
                               double *t_res) {
    const size_t smem = eloc_smem_bytes(L->view, Wk, C, ctx->eloc_threads);
    if (!eloc_fits(Wk, C, ctx->eloc_threads)) return set_err(ctx, VMC_ERR_ARG, "walker G table does not fit in shared memory");
    WalkerArgs A = make_args(Wk);
    const bool own = own_rows(L->view.words, Wk->W);
    drop_rates(ctx);
    ctx->bits_whole = 0;
    int chunk = Wk->W;
    const size_t rates_bytes = sizeof(u128) * rate_store_units(Wk->W, L->view.n_groups);
    vmc_status st = ensure_store(ctx, rates_bytes, own ? 0 : row_bytes(L->view), Wk->W, &chunk);
    if (st) return st;
    u128 *rates = (u128 *)ctx->rates;
    cudaError_t e = cudaSuccess;
    for (int w0 = 0; w0 < Wk->W && e == cudaSuccess; w0 += chunk) {
        const int n = std::min(chunk, Wk->W - w0), tiles = (n + kTile - 1) / kTile;
        if (!own) {
            k_free_bits<<<dim3(tiles, free_bits_parts(tiles, L->view.words)), 256, 0, ctx->stream>>>(
                L->view, A.occ_bits, w0, w0 + n, (uint32_t *)ctx->bits);
            ctx->launches += 1;
        }
        if (Wk->precision != VMC_FP64) e = eloc_launch<float, false>(ctx, w0, n, smem, L->view, A, C, e_loc, t_res, rates);
        else if (L->view.scaled) e = eloc_launch<double, true>(ctx, w0, n, smem, L->view, A, C, e_loc, t_res, rates);
        else e = eloc_launch<double, false>(ctx, w0, n, smem, L->view, A, C, e_loc, t_res, rates);
        ctx->launches += 1;
        if (e == cudaSuccess) e = cudaGetLastError();
    }
    ctx->bits_whole = e == cudaSuccess && !own && chunk >= Wk->W;      // for the choice of the next move
    return cuda_check(ctx, e, "k_local_energy");
}

template <typename real, bool kC>
static cudaError_t ctmc_launch(vmc_ctx *ctx, const vmc_lists *L, const vmc_params *P, const WalkerArgs &A,
                               const CpsView &C, int W, size_t smem, uint64_t seed, const u128 *rates,
                               uint64_t *move_code) {
    const int sel_blocks = (W + VMC_WARPS - 1) / VMC_WARPS;
    const uint32_t *bits = ctx->bits_whole ? (const uint32_t *)ctx->bits : nullptr;
    k_ctmc_select<real, kC><<<sel_blocks, VMC_THREADS, 0, ctx->stream>>>(L->view, A, C, rates, bits, seed, move_code,
                                                                         ctx->d_status);
    cudaError_t e = cudaFuncSetAttribute(k_ctmc_apply<real, kC>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e == cudaSuccess) k_ctmc_apply<real, kC><<<W, VMC_THREADS, smem, ctx->stream>>>(L->view, A, C, P->J, move_code);
    return e;
}

vmc_status launch_ctmc_step(vmc_ctx *ctx, const vmc_lists *L, const vmc_params *P, vmc_walkers *Wk,
                            uint64_t seed, uint64_t *move_code) {
    const int M = Wk->M;
    const u128 *rates = (const u128 *)ctx->rates;
    const int nmax = Wk->n_alpha > Wk->n_beta ? Wk->n_alpha : Wk->n_beta;
    const size_t esz = Wk->precision == VMC_FP64 ? 8 : 4;
    const size_t smem = 2 * (2 * (size_t)M) + 32 + esz * (4 * (size_t)((nmax + 3) & ~3) + 2 * (size_t)((M + 3) & ~3));
    WalkerArgs A = make_args(Wk);
    const CpsView C = cps_view(P);
    cudaError_t e;
    if (Wk->precision == VMC_FP64)
        e = C.n_corr ? ctmc_launch<double, true>(ctx, L, P, A, C, Wk->W, smem, seed, rates, move_code)
                     : ctmc_launch<double, false>(ctx, L, P, A, C, Wk->W, smem, seed, rates, move_code);
    else
        e = C.n_corr ? ctmc_launch<float, true>(ctx, L, P, A, C, Wk->W, smem, seed, rates, move_code)
                     : ctmc_launch<float, false>(ctx, L, P, A, C, Wk->W, smem, seed, rates, move_code);
    ctx->launches += 2;
    if (e == cudaSuccess) e = cudaGetLastError();
    return cuda_check(ctx, e, "k_ctmc_select/k_ctmc_apply");
}

// ---------------------------------------------------------------------------------- batches
static size_t apply_smem_bytes(const vmc_walkers *Wk) {
    const int M = Wk->M, nmax = Wk->n_alpha > Wk->n_beta ? Wk->n_alpha : Wk->n_beta;
    const size_t esz = Wk->precision == VMC_FP64 ? 8 : 4;
    return 2 * (2 * (size_t)M) + 32 + esz * (4 * (size_t)((nmax + 3) & ~3) + 2 * (size_t)((M + 3) & ~3));
}

// A batch as launched: walkers, shared memory, rounds of the local energy and, per round, the walkers
// and walker tiles.
struct BatchPlan {
    int total = 0, precision = 0, rounds = 1;
    bool fits = true;                  // every system's walkers fit the local energy's shared memory
    size_t smem_eloc = 0, smem_apply = 0;
    std::vector<int> walkers, tiles;   // per round
    int words = 0;                     // the longest free-entry row
    std::vector<BatchPart> parts;      // the store's layout, by item
};

// The layout of a batch's rate store: every system's rates, then, for as many walkers as a round takes, its
// free-entry rows.  The rounds are doubled until they fit.
static vmc_status place_batch(vmc_ctx *ctx, int n, const vmc_batch_item *items, const std::vector<int> &order, BatchPlan &plan) {
    plan.parts.assign(n, BatchPart());
    size_t units = 0;
    for (int k : order) {
        const vmc_batch_item &it = items[k];
        const ListsView &v = it.lists->view;
        static_cast<StoredRates &>(plan.parts[k]) =
            StoredRates{it.walkers->G, it.walkers->W, v.n_groups, v.words, it.lists->digest, it.eps_run};
        plan.parts[k].rates_at = units;
        units += rate_store_units(it.walkers->W, v.n_groups);
    }
    const size_t bits_at = align256(units * sizeof(u128));
    for (plan.rounds = 1;; plan.rounds *= 2) {
        size_t at = bits_at;
        bool more = false;
        for (int k : order) {
            BatchPart &p = plan.parts[k];
            p.share = ((p.W + plan.rounds - 1) / plan.rounds + 31) & ~31;
            more = more || p.share > 32;
            p.bits_at = at;
            at += row_bytes(items[k].lists->view) * (size_t)p.share;
        }
        const size_t bytes = at + 32;
        if (bytes <= ctx->rates_bytes) return VMC_OK;
        if (more && (bytes - bits_at > kBitsCap || bytes >= ctx->rates_refused)) continue;
        const cudaError_t e = grow_store(ctx, bytes);
        if (e == cudaSuccess) return VMC_OK;
        if (e != cudaErrorMemoryAllocation || !more) return cuda_check(ctx, e, "batched rate store");
    }
}

// Builds (and uploads when changed) the descriptor tables of a batch, most expensive systems first:
// one table over all walkers (used by the CTMC step, and by the local energy when one round is enough),
// then one per round of the local energy.  For the local energy (step = false) it also sizes the shared
// rate store and the free-entry rows: every system's walkers are split over as few rounds as keep the rows within
// kBitsCap.  The CTMC step reads the store as the local energy laid it out, and never resizes it.
static vmc_status prepare_batch(vmc_ctx *ctx, int n, const vmc_batch_item *items, bool step, BatchPlan &plan) {
    if (n < 1 || n > 64 || !items) return set_err(ctx, VMC_ERR_ARG, "1 to 64 batch items");
    std::vector<int> order(n);
    std::vector<double> cost(n);
    for (int k = 0; k < n; ++k) {
        const vmc_batch_item &it = items[k];
        if (!it.lists || !it.params || !it.walkers || !it.d_e_loc || !it.d_t_res || !it.d_move_code)
            return set_err(ctx, VMC_ERR_ARG, "null batch item field");
        if (it.walkers->precision != items[0].walkers->precision)
            return set_err(ctx, VMC_ERR_ARG, "batch items must share the precision");
        if (it.walkers->M != it.lists->M) return set_err(ctx, VMC_ERR_ARG, "lists and walkers disagree on M");
        if (!(it.eps_run >= it.lists->eps_build)) return set_err(ctx, VMC_ERR_ARG, "eps_run below the build eps");
        vmc_status st = lists_set_eps(ctx, const_cast<vmc_lists *>(it.lists), step ? ctx->batch_parts[k].eps : it.eps_run);
        if (st) return st;
        order[k] = k;
        const vmc_lists *L = it.lists;
        cost[k] = (double)(L->ns + 2 * L->nds + L->ndo) * (it.walkers->n_alpha + it.walkers->n_beta) / (2.0 * L->M) +
                  (double)walker_stride_G(it.walkers->M, it.walkers->n_alpha, it.walkers->n_beta);
    }
    std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return cost[a] > cost[b]; });
    int tot = 0;
    size_t se = 0, sa = 0;
    for (int k = 0; k < n; ++k) {
        const vmc_batch_item &it = items[order[k]];
        tot += it.walkers->W;
        se = std::max(se, eloc_smem_bytes(it.lists->view, it.walkers, CpsView{}, ctx->eloc_threads));
        plan.fits = plan.fits && eloc_fits(it.walkers, CpsView{}, ctx->eloc_threads);
        sa = std::max(sa, apply_smem_bytes(it.walkers));
    }
    if (step) {
        plan.parts = ctx->batch_parts;
        plan.rounds = ctx->batch_rounds;
    } else {
        vmc_status st = place_batch(ctx, n, items, order, plan);
        if (st) return st;
    }
    const int rounds = plan.rounds;
    const int n_tabs = rounds == 1 ? 1 : rounds + 1;
    std::string tab(sizeof(SysDesc) * n * n_tabs, '\0');
    SysDesc *d = (SysDesc *)&tab[0];
    int wb = 0, tb = 0;
    for (int k = 0; k < n; ++k) {
        const vmc_batch_item &it = items[order[k]];
        const BatchPart &part = plan.parts[order[k]];
        plan.words = std::max(plan.words, it.lists->view.words);
        d[k].bits = (uint32_t *)((char *)ctx->rates + part.bits_at);
        d[k].w_first = 0;
        d[k].w_count = it.walkers->W;
        d[k].t_begin = tb;
        tb += (it.walkers->W + kTile - 1) / kTile;
        d[k].L = it.lists->view;
        d[k].A = make_args(it.walkers);
        d[k].J = it.params->J;
        d[k].e_loc = it.d_e_loc;
        d[k].t_res = it.d_t_res;
        d[k].rates = (u128 *)ctx->rates + part.rates_at;
        d[k].move_code = it.d_move_code;
        d[k].w_begin = wb;
        wb += it.walkers->W;
    }
    if (rounds == 1) { plan.walkers.push_back(wb); plan.tiles.push_back(tb); }
    for (int r = 0; rounds > 1 && r < rounds; ++r) {
        int w = 0, t = 0;
        for (int k = 0; k < n; ++k) {
            SysDesc &x = d[(size_t)(r + 1) * n + k];
            const int share = plan.parts[order[k]].share;
            x = d[k];
            x.w_first = std::min(r * share, d[k].w_count);
            x.w_count = std::min(share, d[k].w_count - x.w_first);
            x.w_begin = w;
            x.t_begin = t;
            w += x.w_count;
            t += (x.w_count + kTile - 1) / kTile;
        }
        plan.walkers.push_back(w);
        plan.tiles.push_back(t);
    }
    if (tab != ctx->batch_host) {
        ctx->batch_host.clear();               // (until the new table is there)
        if (tab.size() > ctx->batch_desc_bytes) {
            if (ctx->batch_desc) { cudaStreamSynchronize(ctx->stream); cudaFree(ctx->batch_desc); }
            cudaError_t e = cudaMalloc(&ctx->batch_desc, tab.size());
            if (e != cudaSuccess) { ctx->batch_desc = nullptr; ctx->batch_desc_bytes = 0; return cuda_check(ctx, e, "batch table"); }
            ctx->batch_desc_bytes = tab.size();
        }
        if (!ctx->d_queue) {
            cudaError_t e = cudaMalloc(&ctx->d_queue, sizeof(int));
            if (e != cudaSuccess) { ctx->d_queue = nullptr; return cuda_check(ctx, e, "batch queue"); }
        }
        cudaError_t e = cudaMemcpyAsync(ctx->batch_desc, tab.data(), tab.size(), cudaMemcpyHostToDevice, ctx->stream);
        if (e == cudaSuccess) e = cudaStreamSynchronize(ctx->stream);
        if (e != cudaSuccess) return cuda_check(ctx, e, "batch table upload");
        ctx->batch_host = tab;
    }
    plan.total = tot;
    plan.smem_eloc = se;
    plan.smem_apply = sa;
    plan.precision = items[0].walkers->precision;
    return VMC_OK;
}

// Are these the items whose rates the store holds (or fewer walkers of them)?
static bool batch_stored(const vmc_ctx *ctx, int n, const vmc_batch_item *items) {
    if (!items || ctx->batch_parts.empty() || (size_t)n != ctx->batch_parts.size()) return false;
    for (int k = 0; k < n; ++k) {
        const BatchPart &p = ctx->batch_parts[k];
        if (!items[k].lists || p.G != items[k].walkers->G || items[k].walkers->W > p.W || !same_lists(p, items[k].lists)) return false;
    }
    return true;
}

vmc_status launch_local_energy_batch(vmc_ctx *ctx, int n, const vmc_batch_item *items) {
    BatchPlan plan;
    vmc_status st = prepare_batch(ctx, n, items, false, plan);
    if (st) return st;
    const size_t se = plan.smem_eloc;
    if (!plan.fits) return set_err(ctx, VMC_ERR_ARG, "walker G table does not fit in shared memory");
    int dev = 0, nsm = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    drop_rates(ctx);
    for (int r = 0; r < plan.rounds && e == cudaSuccess; ++r) {
        const SysDesc *tab = (const SysDesc *)ctx->batch_desc + (plan.rounds > 1 ? (size_t)(r + 1) * n : 0);
        const int total = plan.walkers[r], tiles = plan.tiles[r];
        if (!total) continue;
        e = cudaMemsetAsync(ctx->d_queue, 0, sizeof(int), ctx->stream);
        if (e != cudaSuccess) break;
        k_free_bits_batched<<<dim3(tiles, free_bits_parts(tiles, plan.words)), 256, 0, ctx->stream>>>(tab, n);
        e = plan.precision == VMC_FP64 ? eloc_batched_launch<double>(ctx, nsm, se, tab, n, total)
                                       : eloc_batched_launch<float>(ctx, nsm, se, tab, n, total);
        ctx->launches += 2;
        if (e == cudaSuccess) e = cudaGetLastError();
    }
    if (e != cudaSuccess) return cuda_check(ctx, e, "k_local_energy_batched");
    ctx->batch_parts = plan.parts;
    ctx->batch_rounds = plan.rounds;
    return VMC_OK;
}

vmc_status launch_ctmc_step_batch(vmc_ctx *ctx, int n, const vmc_batch_item *items, uint64_t seed) {
    if (!batch_stored(ctx, n, items))
        return set_err(ctx, VMC_ERR_ARG, "vmc_local_energy_batch must precede vmc_ctmc_step_batch on the same items");
    BatchPlan plan;
    vmc_status st = prepare_batch(ctx, n, items, true, plan);
    if (st) return st;
    const int total = plan.total, prec = plan.precision;
    const size_t sa = plan.smem_apply;
    const SysDesc *tab = (const SysDesc *)ctx->batch_desc;
    const int sel_blocks = (total + VMC_WARPS - 1) / VMC_WARPS, use_bits = plan.rounds == 1 ? 1 : 0;
    cudaError_t e;
    if (prec == VMC_FP64) {
        k_ctmc_select_batched<double><<<sel_blocks, VMC_THREADS, 0, ctx->stream>>>(tab, n, total, use_bits, seed,
                                                                                ctx->d_status);
        e = cudaFuncSetAttribute(k_ctmc_apply_batched<double>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sa);
        if (e == cudaSuccess) k_ctmc_apply_batched<double><<<total, 256, sa, ctx->stream>>>(tab, n);
    } else {
        k_ctmc_select_batched<float><<<sel_blocks, VMC_THREADS, 0, ctx->stream>>>(tab, n, total, use_bits, seed,
                                                                                ctx->d_status);
        e = cudaFuncSetAttribute(k_ctmc_apply_batched<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sa);
        if (e == cudaSuccess) k_ctmc_apply_batched<float><<<total, 256, sa, ctx->stream>>>(tab, n);
    }
    ctx->launches += 2;
    if (e == cudaSuccess) e = cudaGetLastError();
    ctx->batch_parts.clear();
    return cuda_check(ctx, e, "k_ctmc_*_batched");
}

vmc_status launch_screened_moves(vmc_ctx *ctx, const vmc_lists *L, const vmc_walkers *Wk, const CpsView &C,
                                 int w_begin, int n_w, int64_t cap, uint64_t *code, double *ratio, double *contrib,
                                 int64_t *count, int64_t *walked) {
    WalkerArgs A = make_args(const_cast<vmc_walkers *>(Wk));
    const int blocks = (n_w + VMC_WARPS - 1) / VMC_WARPS;
#define VMC_MOVES(real, kc)                                                                                      \
    k_screened_moves<real, kc><<<blocks, VMC_THREADS, 0, ctx->stream>>>(L->view, A, C, w_begin, n_w, cap, code, \
                                                                       ratio, contrib, count, walked, ctx->d_status)
    if (Wk->precision == VMC_FP64) {
        if (C.n_corr) VMC_MOVES(double, true); else VMC_MOVES(double, false);
    } else {
        if (C.n_corr) VMC_MOVES(float, true); else VMC_MOVES(float, false);
    }
#undef VMC_MOVES
    ctx->launches += 1;
    return cuda_check(ctx, cudaGetLastError(), "k_screened_moves");
}
