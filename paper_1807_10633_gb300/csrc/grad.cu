// Gradient ratios (Sec. III.B) summed over walkers with per-walker weights (a vector-Jacobian
// product of ln psi), AMSGrad (Sec. II.C, Eqs. m1-m2) and the walker sums of Eq. (vmc).
//
// The walker sums are deterministic: the Jastrow block is an exact 64-bit fixed-point sum, and
// for the orbital block each CTA reduces a fixed chunk of walkers into a partial buffer that a
// second kernel adds in chunk order.
#include <math.h>

#include <algorithm>

#include "common.cuh"

namespace {

constexpr int kChunkJ = 256;    // walkers per CTA for dJ
constexpr int kChunkC = 64;     // walkers per dC partial of the mixed form (the length of its FP32 sums)
constexpr int kRowsC = 16;      // orbital rows per CTA (registers per thread) of k_grad_C_reg
constexpr int kWalkC = 64;      // walkers whose orbitals and weights a dC CTA holds at a time

// 32 consecutive spin-orbital occupation bits starting at spin orbital p0 (lane l -> bit l)
__device__ __forceinline__ uint32_t window_bits(const uint32_t *bits_w, int M, int nw, int p0, int lane) {
    const int p = p0 + lane;
    int bit = 0;
    if (p < 2 * M) {
        const int s = p >= M, k = p - s * M;
        bit = (bits_w[s * nw + (k >> 5)] >> (k & 31)) & 1;
    }
    return __ballot_sync(0xffffffffu, bit);
}

// Weights of walker w: mode 0 -> (t[w]); mode 1 -> (t[w], t[w] e[w]).
__device__ __forceinline__ void weights(int mode, const double *t, const double *e, int w, double &c0, double &c1) {
    c0 = t[w];
    c1 = mode ? c0 * e[w] : 0.0;
}

// Fixed-point weights for the Jastrow gradient: cq = round(c 2^s) with s chosen from sum |c| so that
// no partial sum can overflow 63 bits; integer sums are then exact and order independent.
// Also adds sum c0 and sum c1 to sums[0..1] (mode 1).  Two launches, each sum in a fixed order:
// per-CTA partial sums over consecutive walker chunks, then the quantisation over the whole grid.
constexpr int kWeightChunk = 256;   // walkers per partial-sum CTA
constexpr int kWeightParts = 256;   // most partial sums (chunks grow beyond 65,536 walkers)

__global__ void __launch_bounds__(256)
k_weight_partial(int W, int chunk, const double *__restrict__ t, const double *__restrict__ e, int mode,
                 double *__restrict__ part) {
    __shared__ double r[4][8];
    double a0 = 0.0, a1 = 0.0, s0 = 0.0, s1 = 0.0;
    const int w0 = blockIdx.x * chunk, w1 = min(W, w0 + chunk);
    for (int w = w0 + threadIdx.x; w < w1; w += blockDim.x) {
        double c0, c1;
        weights(mode, t, e, w, c0, c1);
        a0 += fabs(c0); a1 += fabs(c1); s0 += c0; s1 += c1;
    }
    a0 = warp_sum_f64(a0); a1 = warp_sum_f64(a1); s0 = warp_sum_f64(s0); s1 = warp_sum_f64(s1);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (lane == 0) { r[0][warp] = a0; r[1][warp] = a1; r[2][warp] = s0; r[3][warp] = s1; }
    __syncthreads();
    if (threadIdx.x < 4) {
        double v = 0.0;
        for (int k = 0; k < (int)(blockDim.x >> 5); ++k) v += r[threadIdx.x][k];
        part[(size_t)blockIdx.x * 4 + threadIdx.x] = v;
    }
}

// Adds the partials (one warp of every CTA, all in the same order, so that no launch of its own is needed for
// it), sets the exponents and quantises; CTA 0 also stores the exponents and the sums.
__global__ void __launch_bounds__(256)
k_weight_quant(int W, const double *__restrict__ t, const double *__restrict__ e, int mode, int n_parts,
               const double *__restrict__ part, int *__restrict__ sexp, double *__restrict__ sums,
               long long *__restrict__ cq) {
    __shared__ int s_exp[2];
    if (threadIdx.x < 32) {
        double v[4] = {0.0, 0.0, 0.0, 0.0};
        for (int b = threadIdx.x; b < n_parts; b += 32)
#pragma unroll
            for (int q = 0; q < 4; ++q) v[q] += part[(size_t)b * 4 + q];
#pragma unroll
        for (int q = 0; q < 4; ++q) v[q] = warp_sum_f64(v[q]);
        if (threadIdx.x == 0) {
            s_exp[0] = v[0] > 0.0 ? 61 - ilogb(v[0]) : 0;
            s_exp[1] = v[1] > 0.0 ? 61 - ilogb(v[1]) : 0;
            if (blockIdx.x == 0) {
                sexp[0] = s_exp[0];
                sexp[1] = s_exp[1];
                if (sums) { sums[0] += v[2]; sums[1] += v[3]; }
            }
        }
    }
    __syncthreads();
    const int e0 = s_exp[0], e1 = s_exp[1];
    for (int w = blockIdx.x * blockDim.x + threadIdx.x; w < W; w += gridDim.x * blockDim.x) {
        double c0, c1;
        weights(mode, t, e, w, c0, c1);
        cq[w] = __double2ll_rn(scalbn(c0, e0));
        if (mode) cq[W + w] = __double2ll_rn(scalbn(c1, e1));
    }
}

// dJ partials: tile (P, Q) of 32 x 32 spin orbitals with P <= Q, walker chunk blockIdx.y.
// Exact 64-bit integer sums of the fixed-point weights.  part layout: [n_out][chunk][N2][N2].
// The chunk's 32-orbital occupation windows and weights are staged in shared memory; lane l of
// warp v owns p = 32P + l and q = 32Q + 4v .. 4v + 3, so the q bits are warp-uniform (a branch)
// and the p bit is a mask.
__global__ void __launch_bounds__(256)
k_grad_J(int W, int M, const uint32_t *__restrict__ bits, const long long *__restrict__ cq, int mode,
         long long *__restrict__ part) {
    const int N2 = 2 * M, nw = (M + 31) / 32, T = (N2 + 31) / 32;
    int t = blockIdx.x, P = 0;
    while (t >= T - P) { t -= T - P; ++P; }
    const int Q = P + t;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarp = blockDim.x >> 5;
    __shared__ uint2 s_b[kChunkJ];
    __shared__ longlong2 s_c[kChunkJ];
    const int w0 = blockIdx.y * kChunkJ, nwk = min(W, w0 + kChunkJ) - w0;
    if ((M & 31) == 0) {   // windows are whole words of one spin
        const int wp = P * 32 < M ? P : nw + (P * 32 - M) / 32, wq = Q * 32 < M ? Q : nw + (Q * 32 - M) / 32;
        for (int i = tid; i < nwk; i += blockDim.x) {
            const uint32_t *bw = bits + (size_t)(w0 + i) * 2 * nw;
            s_b[i] = make_uint2(bw[wp], bw[wq]);
        }
    } else {
        for (int i = warp; i < nwk; i += nwarp) {
            const uint32_t *bw = bits + (size_t)(w0 + i) * 2 * nw;
            const uint32_t bp = window_bits(bw, M, nw, P * 32, lane);
            const uint32_t bq = window_bits(bw, M, nw, Q * 32, lane);
            if (lane == 0) s_b[i] = make_uint2(bp, bq);
        }
    }
    for (int i = tid; i < nwk; i += blockDim.x) {
        longlong2 c;
        c.x = cq[w0 + i];
        c.y = mode ? cq[W + w0 + i] : 0;
        s_c[i] = c;
    }
    __syncthreads();
    const int qb = warp * 4;
    long long acc[4] = {0, 0, 0, 0}, acc2[4] = {0, 0, 0, 0};
    if (mode) {
        for (int i = 0; i < nwk; ++i) {
            const uint2 b = s_b[i];
            const longlong2 c = s_c[i];
            const long long m = -(long long)((b.x >> lane) & 1u);
            const long long c0 = c.x & m, c1 = c.y & m;
#pragma unroll
            for (int k = 0; k < 4; ++k)
                if ((b.y >> (qb + k)) & 1u) { acc[k] += c0; acc2[k] += c1; }
        }
    } else {
        for (int i = 0; i < nwk; ++i) {
            const uint2 b = s_b[i];
            const long long c0 = s_c[i].x & -(long long)((b.x >> lane) & 1u);
#pragma unroll
            for (int k = 0; k < 4; ++k)
                if ((b.y >> (qb + k)) & 1u) acc[k] += c0;
        }
    }
    const size_t chunk_sz = (size_t)N2 * N2;
    long long *dst = part + (size_t)blockIdx.y * chunk_sz;
    long long *dst2 = part + ((size_t)gridDim.y + blockIdx.y) * chunk_sz;
    const int p = P * 32 + lane;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const int q = Q * 32 + qb + k;
        if (p < N2 && q < N2 && p <= q) {
            dst[(size_t)p * N2 + q] = acc[k];
            if (mode) dst2[(size_t)p * N2 + q] = acc2[k];
        }
    }
}

// Sum of the dJ partials over walker chunks (integers: any order).  CTA = 32 consecutive outputs (lanes) x 8 warps over
// interleaved chunks: a small system has few outputs and as many chunks as the SMs leave it (H20: 76), which one
// thread per output added one after the other (4,096 walkers: 12.0 -> 4.0 us; H80, 16,384 walkers: 7.3 -> 3.4 us; H160,
// 32,768 walkers, where outputs are many: 5.6 -> 6.1 us).
__global__ void __launch_bounds__(256)
k_reduce_J(int M, int n_chunks, const long long *__restrict__ part, const int *__restrict__ sexp,
           double *__restrict__ dJ, double *__restrict__ dJ2) {
    __shared__ long long red[2][8][32];
    const int N2 = 2 * M, lane = threadIdx.x & 31, v = threadIdx.x >> 5;
    const size_t csz = (size_t)N2 * N2;
    const int t = blockIdx.x * 32 + lane, p = t / N2, q = t - p * N2;
    const bool mine = t < N2 * N2 && p <= q;
    long long s = 0, s2 = 0;
    if (mine)
        for (int c = v; c < n_chunks; c += 8) {
            s += part[(size_t)c * csz + t];
            if (dJ2) s2 += part[((size_t)n_chunks + c) * csz + t];
        }
    red[0][v][lane] = s;
    red[1][v][lane] = s2;
    __syncthreads();
    if (v < (dJ2 ? 2 : 1) && mine) {
        long long sum = 0;
#pragma unroll
        for (int k = 0; k < 8; ++k) sum += red[v][k][lane];
        (v ? dJ2 : dJ)[t] += scalbn((double)sum, -sexp[v]);
    }
}

// dC partials: sum_w c_w AinvT_w[col(k)][x] for occupied k.  CTA = (spin, range of k) x walker chunk, with the
// accumulators [k][x] of one or two weight sets in shared memory.  A warp owns a block of columns x
// (kXL lanes of VE elements) and goes through every walker's rows c in order, 32 / kXL rows at a time; row c
// belongs to orbital k = occ[c], so rows of one walker never meet and no other warp touches the warp's
// columns.  AinvT is read once, contiguously and with kDepth to 2 kDepth loads per lane in flight, and nothing is
// done for unoccupied orbitals (a thread per x with register accumulators for 16 orbitals spends half of its
// multiply-adds on zeros, and leaves 24 of 64 lanes idle at n = 40).  Per accumulator the walkers of a chunk
// are added in order.  Bound: latency and shared-memory
// read-modify-writes; H80, 16,384 walkers, FP64: 672 -> 195 us (its FP64 multiply-adds alone 167 us).
// part layout: [n_out][chunk][2][M][nmax].  acc_t = float (mixed) or double.
constexpr int kXL = 4, kDepth = 8;

template <typename real, int VE> struct __align__(sizeof(real) * VE) RowVec { real v[VE]; };

template <typename real, int VE, int kMode>
__global__ void __launch_bounds__(1024 / VE)          // (at most 32 warps of kXL VE columns: n <= 128)
k_grad_C(int W, int M, int na, int nb, int chunk, int n_k, const uint16_t *__restrict__ occ, const real *__restrict__ AinvT,
         const double *__restrict__ wgt, const double *__restrict__ e, double *__restrict__ part) {
    constexpr int kCL = 32 / kXL;                    // rows per step
    typedef RowVec<real, VE> vec;
    const int s = blockIdx.x & 1, k0 = (blockIdx.x >> 1) * n_k, nk = min(n_k, M - k0);
    const int n = s ? nb : na, ne = na + nb, nmax = na > nb ? na : nb;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nt = blockDim.x;
    extern __shared__ __align__(16) unsigned char sm[];
    real *acc0 = (real *)sm, *acc1 = acc0 + (size_t)n_k * nmax;           // [k][x], rows of n
    real *s_w = acc0 + (size_t)(kMode + 1) * n_k * nmax;                  // [kWalkC][2] weights
    uint16_t *s_occ = (uint16_t *)(s_w + 2 * kWalkC);                     // [kWalkC][n]
    for (int t = tid; t < (kMode + 1) * n_k * nmax; t += nt) acc0[t] = real(0);
    const size_t astride = (size_t)na * na + (size_t)nb * nb;
    const int w_begin = blockIdx.y * chunk, w_end = min(W, w_begin + chunk);
    const int x = (warp * kXL + lane % kXL) * VE, cl = lane / kXL, G = (n + kCL - 1) / kCL;
    const bool xin = x < n;                          // (n is a multiple of VE)
    for (int wb = w_begin; wb < w_end; wb += kWalkC) {
        const int nw = min(kWalkC, w_end - wb);
        __syncthreads();
        for (int t = tid; t < nw * n; t += nt) {
            const int i = t / n, c = t - i * n;
            s_occ[t] = occ[(size_t)(wb + i) * ne + (s ? na : 0) + c];
        }
        for (int i = tid; i < nw; i += nt) {
            double c0, c1;
            weights(kMode, wgt, e, wb + i, c0, c1);
            s_w[2 * i] = (real)c0;
            s_w[2 * i + 1] = (real)c1;
        }
        __syncthreads();
        const real *A = AinvT + (size_t)wb * astride + (s ? (size_t)na * na : 0);
        int wl = 0, gl = 0;                          // walker and row step of the next load
        struct Step {
            vec v;
            int at, w;                               // accumulator offset (-1: none), walker
        } cur[kDepth], nxt[kDepth];
        auto load = [&](Step (&p)[kDepth]) {
#pragma unroll
            for (int u = 0; u < kDepth; ++u) {
                const int c = gl * kCL + cl;
                p[u].at = -1;
                p[u].w = wl;
                if (wl < nw && c < n && xin) {
                    const int k = (int)s_occ[wl * n + c] - k0;
                    if ((unsigned)k < (unsigned)nk) {
                        p[u].at = k * n + x;
                        p[u].v = *(const vec *)(A + (size_t)wl * astride + (size_t)c * n + x);
                    }
                }
                if (++gl == G) { gl = 0; ++wl; }
            }
        };
        load(cur);
        for (int f0 = 0; f0 < nw * G; f0 += kDepth) {
            load(nxt);                               // in flight while the previous ones are added
#pragma unroll
            for (int u = 0; u < kDepth; ++u) {
                if (cur[u].at >= 0) {
                    const real c0 = s_w[2 * cur[u].w], c1 = kMode ? s_w[2 * cur[u].w + 1] : real(0);
                    vec p = *(const vec *)(acc0 + cur[u].at);
#pragma unroll
                    for (int q = 0; q < VE; ++q) p.v[q] += c0 * cur[u].v.v[q];
                    *(vec *)(acc0 + cur[u].at) = p;
                    if (kMode) {
                        vec r = *(const vec *)(acc1 + cur[u].at);
#pragma unroll
                        for (int q = 0; q < VE; ++q) r.v[q] += c1 * cur[u].v.v[q];
                        *(vec *)(acc1 + cur[u].at) = r;
                    }
                }
                __syncwarp();                        // the next step may be another walker's
                cur[u] = nxt[u];
            }
        }
    }
    __syncthreads();
    const size_t blk = (size_t)M * nmax;
    double *dst = part + ((size_t)blockIdx.y * 2 + s) * blk + (size_t)k0 * n;
    double *dst2 = part + (((size_t)gridDim.y + blockIdx.y) * 2 + s) * blk + (size_t)k0 * n;
    for (int t = tid; t < nk * n; t += nt) {
        dst[t] = (double)acc0[t];
        if (kMode) dst2[t] = (double)acc1[t];
    }
}

// The mixed form's dC partials for n_sigma > kRegC: CTA = (spin, block of kRowsC orbital rows) x walker chunk;
// thread x owns the accumulators dC[k][x] of its rows in registers: acc[k][x] += c_w AinvT_w[pos_w(k)][x] for
// occupied k.  Its chunks of 64 walkers are too short for the shared-memory kernel above to fill the SMs with the few
// CTAs that its accumulators leave (H160: 798 us there, 679 us here; H61, 8,192 walkers: 141 and 131 us a call;
// at n = 10 it is 117 us here and 90 us there).
constexpr int kRegC = 24;
__global__ void __launch_bounds__(128)
k_grad_C_reg(int W, int M, int na, int nb, const uint16_t *__restrict__ pos, const float *__restrict__ AinvT,
         const double *__restrict__ wgt, const double *__restrict__ e, int mode, double *__restrict__ part) {
    const int nrb = (M + kRowsC - 1) / kRowsC;
    const int s = blockIdx.x / nrb, rb = blockIdx.x - s * nrb;
    const int n = s ? nb : na, x = threadIdx.x;
    const int k0 = rb * kRowsC;
    float acc[kRowsC], acc2[kRowsC];
#pragma unroll
    for (int r = 0; r < kRowsC; ++r) { acc[r] = 0; acc2[r] = 0; }
    const size_t astride = (size_t)na * na + (size_t)nb * nb;
    const size_t aoff = s ? (size_t)na * na : 0;
    const int w0 = blockIdx.y * kChunkC, w1 = min(W, w0 + kChunkC);
    const bool xin = x < n;
    // the kRowsC map entries of a walker: two 16-byte loads when aligned (M % 8 == 0 and the caller's array)
    const bool vec = (M & 7) == 0 && k0 + kRowsC <= M && (uintptr_t)pos % 16 == 0;
    auto map_of = [&](int w, uint4 &lo, uint4 &hi) {
        const uint16_t *pw = pos + (size_t)w * 2 * M + (size_t)s * M + k0;
        if (vec) {
            lo = __ldg((const uint4 *)pw);
            hi = __ldg((const uint4 *)pw + 1);
        } else {
            uint16_t t[kRowsC];
#pragma unroll
            for (int r = 0; r < kRowsC; ++r) t[r] = k0 + r < M ? pw[r] : (uint16_t)0x8000;
            uint32_t q[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) q[k] = (uint32_t)t[2 * k] | ((uint32_t)t[2 * k + 1] << 16);
            lo = make_uint4(q[0], q[1], q[2], q[3]);
            hi = make_uint4(q[4], q[5], q[6], q[7]);
        }
    };
    uint4 nlo = make_uint4(0, 0, 0, 0), nhi = nlo;
    if (w0 < w1) map_of(w0, nlo, nhi);
    for (int w = w0; w < w1; ++w) {
        const uint4 lo = nlo, hi = nhi;
        if (w + 1 < w1) map_of(w + 1, nlo, nhi);    // prefetch the next walker's map
        double c0d, c1d;
        weights(mode, wgt, e, w, c0d, c1d);
        const float c0 = (float)c0d, c1 = (float)c1d;
        const float *A = AinvT + (size_t)w * astride + aoff;
        const uint32_t words[8] = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, hi.w};
        float a[kRowsC];
#pragma unroll
        for (int r = 0; r < kRowsC; ++r) {         // all row loads in flight together
            const uint32_t pc = (words[r >> 1] >> ((r & 1) * 16)) & 0xFFFFu;
            a[r] = (xin && k0 + r < M && !(pc & 0x8000u)) ? A[(size_t)pc * n + x] : float(0);
        }
#pragma unroll
        for (int r = 0; r < kRowsC; ++r) {
            acc[r] += c0 * (float)a[r];
            if (mode) acc2[r] += c1 * (float)a[r];
        }
    }
    if (!xin) return;
    const size_t blk = (size_t)M * (na > nb ? na : nb);
    double *dst = part + ((size_t)blockIdx.y * 2 + s) * blk;
    double *dst2 = part + (((size_t)gridDim.y + blockIdx.y) * 2 + s) * blk;
#pragma unroll
    for (int r = 0; r < kRowsC; ++r) {
        const int k = k0 + r;
        if (k >= M) break;
        dst[(size_t)k * n + x] = (double)acc[r];
        if (mode) dst2[(size_t)k * n + x] = (double)acc2[r];
    }
}

// Sum of the dC partials over walker chunks.  CTA = 32 consecutive outputs (lanes, coalesced) x 8
// warps; warp v adds chunks v, v + 8, ... into four running sums (more loads in flight), then the
// eight warp sums are added in warp order: a fixed order, so the result is deterministic.
__global__ void __launch_bounds__(256)
k_reduce_C(int M, int na, int nb, int n_chunks, int n_out, const double *__restrict__ part,
           double *__restrict__ dCa, double *__restrict__ dCb, double *__restrict__ dCa2, double *__restrict__ dCb2) {
    __shared__ double red[8][33];
    const int nmax = na > nb ? na : nb;
    const int tot = M * na + M * nb, total = n_out * tot;
    const int lane = threadIdx.x & 31, v = threadIdx.x >> 5;
    const int t = blockIdx.x * 32 + lane;
    const int o = t / tot, r = t - o * tot;
    const int s = r >= M * na;
    const int u = s ? r - M * na : r;
    double acc[4] = {0.0, 0.0, 0.0, 0.0};
    if (t < total) {
        const size_t mn = (size_t)M * nmax, stride = 2 * mn;
        const double *src = part + ((size_t)o * n_chunks * 2 + s) * mn + u;
        int c = v;
        for (; c + 24 < n_chunks; c += 32) {
            acc[0] += src[(size_t)c * stride];
            acc[1] += src[(size_t)(c + 8) * stride];
            acc[2] += src[(size_t)(c + 16) * stride];
            acc[3] += src[(size_t)(c + 24) * stride];
        }
        if (c < n_chunks) acc[0] += src[(size_t)c * stride];            // at most three left
        if (c + 8 < n_chunks) acc[1] += src[(size_t)(c + 8) * stride];
        if (c + 16 < n_chunks) acc[2] += src[(size_t)(c + 16) * stride];
    }
    red[v][lane] = (acc[0] + acc[1]) + (acc[2] + acc[3]);
    __syncthreads();
    if (v == 0 && t < total) {
        double sum = 0.0;
#pragma unroll
        for (int k = 0; k < 8; ++k) sum += red[k][lane];
        double *dst = o == 0 ? (s ? dCb : dCa) : (s ? dCb2 : dCa2);
        dst[u] += sum;
    }
}

__global__ void k_amsgrad(double *p, const double *g, double *m, double *v, size_t np, double alpha,
                          double b1, double b2) {
    for (size_t k = blockIdx.x * (size_t)blockDim.x + threadIdx.x; k < np; k += (size_t)gridDim.x * blockDim.x) {
        const double gk = g[k];
        const double mk = (1.0 - b1) * m[k] + b1 * gk;
        const double cand = (1.0 - b2) * v[k] + b2 * (gk * gk);
        const double vk = v[k] > cand ? v[k] : cand;
        m[k] = mk;
        v[k] = vk;
        if (vk > 0.0) p[k] -= alpha * mk / sqrt(vk);
    }
}

__global__ void k_energy_gradient(size_t n, const double *__restrict__ sums, const double *__restrict__ aO,
                                  const double *__restrict__ aEO, double *__restrict__ g) {
    const double T = sums[0], E = sums[1] / T;
    for (size_t k = blockIdx.x * (size_t)blockDim.x + threadIdx.x; k < n; k += (size_t)gridDim.x * blockDim.x)
        g[k] = 2.0 * (aEO[k] / T - E * (aO[k] / T));
}

__global__ void __launch_bounds__(1024)
k_walker_reduce(int W, const double *__restrict__ t, const double *__restrict__ e, double *out) {
    __shared__ double r0[32], r1[32];
    double a = 0.0, b = 0.0;
    for (int w = threadIdx.x; w < W; w += blockDim.x) {
        a += t[w];
        b += t[w] * e[w];
    }
    a = warp_sum_f64(a);
    b = warp_sum_f64(b);
    if ((threadIdx.x & 31) == 0) { r0[threadIdx.x >> 5] = a; r1[threadIdx.x >> 5] = b; }
    __syncthreads();
    if (threadIdx.x == 0) {
        double sa = 0.0, sb = 0.0;
        for (int k = 0; k < (int)(blockDim.x >> 5); ++k) { sa += r0[k]; sb += r1[k]; }
        out[0] += sa;
        out[1] += sb;
    }
}

}  // namespace

// Work split of k_grad_C: orbitals per CTA so that the accumulators take at most half of an SM's shared
// memory (two CTAs, or more), walkers per CTA: 64 in the mixed form (the FP32 sums' length), in FP64 one
// wave of CTAs, but 16 or more.
struct PlanC {
    int n_k, parts, chunk, chunks;
    size_t smem;
};
static PlanC plan_grad_C(int W, int M, int na, int nb, int esz, int nout) {
    const int nmax = na > nb ? na : nb;
    PlanC p;
    const size_t fixed = 2 * (size_t)esz * kWalkC + sizeof(uint16_t) * (size_t)kWalkC * nmax, room = 112 * 1024 - fixed;
    const size_t per_k = (size_t)nout * nmax * esz;
    int parts = 1;
    while (parts < M && per_k * (size_t)((M + parts - 1) / parts) > room) ++parts;
    p.n_k = (M + parts - 1) / parts;
    p.parts = (M + p.n_k - 1) / p.n_k;
    p.smem = (per_k * (size_t)p.n_k + fixed + 15) & ~(size_t)15;
    p.chunk = kChunkC;
    if (esz == 8) {
        const int warps = (nmax + kXL * 2 - 1) / (kXL * 2);
        const int per_sm = (int)std::max<size_t>(1, std::min<size_t>(227 * 1024 / (p.smem + 1024), 64 / std::max(1, warps)));
        const int ctas = std::max(1, 152 * std::min(per_sm, 8) / (2 * p.parts));
        p.chunk = std::max(16, (W + ctas - 1) / ctas);
    }
    p.chunks = (W + p.chunk - 1) / p.chunk;
    return p;
}

template <typename real, int VE>
static cudaError_t grad_C_launch_v(vmc_ctx *ctx, const vmc_walkers *Wk, const PlanC &p, const double *t, const double *e,
                                   int mode, double *part) {
    const int na = Wk->n_alpha, nb = Wk->n_beta, nmax = na > nb ? na : nb;
    const int threads = 32 * ((nmax + kXL * VE - 1) / (kXL * VE));
    const dim3 grid(2 * p.parts, p.chunks);
    auto *k = mode ? k_grad_C<real, VE, 1> : k_grad_C<real, VE, 0>;
    cudaError_t err = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)p.smem);
    if (err == cudaSuccess)
        k<<<grid, threads, p.smem, ctx->stream>>>(Wk->W, Wk->M, na, nb, p.chunk, p.n_k, Wk->occ_list,
                                                  (const real *)Wk->AinvT, t, e, part);
    return err == cudaSuccess ? cudaGetLastError() : err;
}

// 16-byte, 8-byte or single elements: rows start at multiples of n_alpha and n_beta elements
template <typename real>
static cudaError_t grad_C_launch(vmc_ctx *ctx, const vmc_walkers *Wk, const PlanC &p, const double *t, const double *e,
                                 int mode, double *part) {
    const int na = Wk->n_alpha, nb = Wk->n_beta;
    const uintptr_t a = (uintptr_t)Wk->AinvT;
    constexpr int most = 16 / (int)sizeof(real);
    if (na % most == 0 && nb % most == 0 && a % 16 == 0) return grad_C_launch_v<real, most>(ctx, Wk, p, t, e, mode, part);
    if (most == 4 && na % 2 == 0 && nb % 2 == 0 && a % 8 == 0) return grad_C_launch_v<real, 2>(ctx, Wk, p, t, e, mode, part);
    return grad_C_launch_v<real, 1>(ctx, Wk, p, t, e, mode, part);
}

static cudaError_t grad_C_reg_launch(vmc_ctx *ctx, const vmc_walkers *Wk, const PlanC &p, const double *t, const double *e,
                                     int mode, double *part) {
    const int M = Wk->M, na = Wk->n_alpha, nb = Wk->n_beta, nmax = na > nb ? na : nb;
    const dim3 grid(2 * ((M + kRowsC - 1) / kRowsC), p.chunks);
    k_grad_C_reg<<<grid, (nmax + 31) / 32 * 32, 0, ctx->stream>>>(Wk->W, M, na, nb, Wk->pos, (const float *)Wk->AinvT, t, e,
                                                                  mode, part);
    return cudaGetLastError();
}

static vmc_status grad_impl(vmc_ctx *ctx, const vmc_walkers *Wk, const double *t, const double *e, int mode,
                            double *const out0[3], double *const out1[3], double *sums) {
    const int W = Wk->W, M = Wk->M, na = Wk->n_alpha, nb = Wk->n_beta, N2 = 2 * M;
    const int T = (N2 + 31) / 32, ntile = T * (T + 1) / 2;
    const bool jtc = ctx->grad_j_tc != 0 && out0[0] != nullptr;
    int cj = (W + kChunkJ - 1) / kChunkJ, chunk_j = kChunkJ;
    if (jtc) {
        int dev = 0, nsm = 0;
        cudaError_t err = cudaGetDevice(&dev);
        if (err == cudaSuccess) err = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
        if (err != cudaSuccess) return cuda_check(ctx, err, "device attributes");
        grad_j_umma_chunks(W, M, nsm, &chunk_j, &cj);
    }
    const int nmax = na > nb ? na : nb, nout = mode + 1;
    if (nmax > 128) return set_err(ctx, VMC_ERR_ARG, "n_sigma > 128 is not supported by the gradient kernel");
    // workspace: [exponents | pad to 256] [partial weight sums] [cq: 2 W int64] [gradient partials]
    const size_t parts = 256 + sizeof(double) * 4 * kWeightParts;
    const size_t head = parts + sizeof(long long) * 2 * (size_t)W;
    const size_t bytes_J = sizeof(long long) * (size_t)nout * cj * N2 * N2;
    const PlanC pc = plan_grad_C(W, M, na, nb, Wk->precision == VMC_FP64 ? 8 : 4, nout);
    const int cc = pc.chunks;
    const size_t bytes_C = sizeof(double) * (size_t)nout * cc * 2 * M * nmax;
    vmc_status st = ensure_workspace(ctx, head + (bytes_J > bytes_C ? bytes_J : bytes_C));
    if (st) return st;
    int *sexp = (int *)ctx->ws;
    double *wpart = (double *)((char *)ctx->ws + 256);
    long long *cq = (long long *)((char *)ctx->ws + parts);
    void *part = (char *)ctx->ws + head;
    {
        const int wchunk = std::max(kWeightChunk, (W + kWeightParts - 1) / kWeightParts);
        const int n_parts = (W + wchunk - 1) / wchunk;
        k_weight_partial<<<n_parts, 256, 0, ctx->stream>>>(W, wchunk, t, e, mode, wpart);
        k_weight_quant<<<(W + 255) / 256 < 1216 ? (W + 255) / 256 : 1216, 256, 0, ctx->stream>>>(W, t, e, mode, n_parts, wpart,
                                                                                                 sexp, sums, cq);
        ctx->launches += 2;
    }
    if (out0[0]) {
        if (jtc) {
            st = launch_grad_J_umma(ctx, W, M, Wk->occ_bits, cq, mode, (long long *)part, chunk_j, cj);
            if (st) return st;     // (the launch is counted there)
        } else {
            k_grad_J<<<dim3(ntile, cj), 256, 0, ctx->stream>>>(W, M, Wk->occ_bits, cq, mode, (long long *)part);
            ctx->launches += 1;
        }
        k_reduce_J<<<(N2 * N2 + 31) / 32, 256, 0, ctx->stream>>>(M, cj, (const long long *)part, sexp, out0[0],
                                                                   mode ? out1[0] : nullptr);
        ctx->launches += 1;
        cudaError_t err = cudaGetLastError();
        if (err != cudaSuccess) return cuda_check(ctx, err, "k_grad_J");
    }
    if (out0[1] && out0[2]) {
        cudaError_t err = Wk->precision == VMC_FP64
                              ? grad_C_launch<double>(ctx, Wk, pc, t, e, mode, (double *)part)
                              : (nmax > kRegC ? grad_C_reg_launch(ctx, Wk, pc, t, e, mode, (double *)part)
                                              : grad_C_launch<float>(ctx, Wk, pc, t, e, mode, (double *)part));
        if (err != cudaSuccess) return cuda_check(ctx, err, "k_grad_C");
        const int tot = nout * (M * na + M * nb);
        k_reduce_C<<<(tot + 31) / 32, 256, 0, ctx->stream>>>(M, na, nb, cc, nout, (const double *)part, out0[1],
                                                               out0[2], mode ? out1[1] : nullptr, mode ? out1[2] : nullptr);
        ctx->launches += 2;
        err = cudaGetLastError();
        if (err != cudaSuccess) return cuda_check(ctx, err, "k_grad_C");
    }
    return VMC_OK;
}

vmc_status launch_grad(vmc_ctx *ctx, const vmc_walkers *Wk, const double *w, double *dJ, double *dCa,
                       double *dCb) {
    double *const o0[3] = {dJ, dCa, dCb};
    double *const o1[3] = {nullptr, nullptr, nullptr};
    return grad_impl(ctx, Wk, w, nullptr, 0, o0, o1, nullptr);
}

vmc_status launch_accumulate(vmc_ctx *ctx, const vmc_walkers *Wk, const double *t, const double *e,
                             double *const aO[3], double *const aEO[3], double *sums) {
    return grad_impl(ctx, Wk, t, e, 1, aO, aEO, sums);
}

vmc_status launch_amsgrad(vmc_ctx *ctx, double *p, const double *g, double *m, double *n, size_t np,
                          double alpha, double b1, double b2) {
    if (np == 0) return VMC_OK;
    const int blocks = (int)((np + 255) / 256 < 152 * 8 ? (np + 255) / 256 : 152 * 8);
    k_amsgrad<<<blocks, 256, 0, ctx->stream>>>(p, g, m, n, np, alpha, b1, b2);
    ctx->launches += 1;
    return cuda_check(ctx, cudaGetLastError(), "k_amsgrad");
}

vmc_status launch_energy_gradient(vmc_ctx *ctx, size_t n, const double *sums, const double *aO,
                                  const double *aEO, double *g) {
    if (n == 0) return VMC_OK;
    const int blocks = (int)((n + 255) / 256 < 152 * 8 ? (n + 255) / 256 : 152 * 8);
    k_energy_gradient<<<blocks, 256, 0, ctx->stream>>>(n, sums, aO, aEO, g);
    ctx->launches += 1;
    return cuda_check(ctx, cudaGetLastError(), "k_energy_gradient");
}

vmc_status launch_walker_reduce(vmc_ctx *ctx, int W, const double *t, const double *e, double *out) {
    k_walker_reduce<<<1, 1024, 0, ctx->stream>>>(W, t, e, out);
    ctx->launches += 1;
    return cuda_check(ctx, cudaGetLastError(), "k_walker_reduce");
}
