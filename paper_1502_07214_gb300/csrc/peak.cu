// peak.cu -- the pseudo-transition point Delta*_L of Sec. III: the crystal
// field where C(Delta) of Eq. 6 is largest, found as the zero crossing of
// dC/dDelta by bisection with time-series reweighting (Eq. 3), for the full
// series and for w jackknife subsets that each leave out one block of
// consecutive measurements; C*_L = C(Delta*_L).
//
// Differentiating a reweighted mean, d<O>/dDelta = -beta (<O E_Delta> - <O><E_Delta>);
// applied to Eq. 6,
//   dC/dDelta = beta^2 <(E_J - <E_J>)(E_Delta - <E_Delta>)^2>.
// A sample enters C and dC/dDelta only through its E_Delta bin and its E_J,
// and (E_Delta - <E_Delta>) is constant within a bin, so both need per bin
// only the number of samples n and their mean E_J:
//   C = -beta / Z sum_E w(E) n(E) (mj(E) - <E_J>)(E - <E_Delta>),
//   dC/dDelta / beta^2 = 1 / Z sum_E w(E) n(E) (mj(E) - <E_J>)(E - <E_Delta>)^2,
// with w(E) = exp(-beta Delta E - lnW(E)) taken relative to its largest value.
//
// GPU layout: one pass over the series forms exact integer sums (count, sum
// E_J) per bin and per jackknife block; each data set's sums are all blocks'
// sums minus the left-out block's (integers, exact); the weighted sums over
// blocks of consecutive bins become polynomials in the field once per call; one
// thread-block cluster per data set then runs the whole bisection, each CTA
// over its own slice of the blocks, the CTAs' parts combined through
// distributed shared memory in rank order (so that every CTA holds the same
// numbers and takes the same bisection step), one cluster barrier per step.
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <string>
#include <vector>

#include "../../include/muca.h"
#include "muca_internal.h"

namespace {

namespace cg = cooperative_groups;

// Integer sums per jackknife block: cnt[b][E], sej[b][E].  bnd[i] is the first
// row of block i (bnd[n_blocks] = n_rows).
template <bool SEJ>
__global__ void jk_bin_kernel(const int32_t *__restrict__ ej, const int32_t *__restrict__ ed,
                              int64_t n_rows, int row_len, int64_t row_stride, int e_min, int nE,
                              const int64_t *__restrict__ bnd, int n_blocks,
                              unsigned long long *cnt, unsigned long long *sej, int *err)
{
    for (int64_t r = blockIdx.y; r < n_rows; r += gridDim.y) {
        int b = 0;
        while (b + 1 < n_blocks && bnd[b + 1] <= r) ++b;
        unsigned long long *cb = cnt + (size_t)b * nE, *sb = sej + (size_t)b * nE;
        for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < row_len;
             c += gridDim.x * blockDim.x) {
            const int64_t o = r * row_stride + c;
            const int e = (int)((unsigned)__ldg(ed + o) - (unsigned)e_min);
            if ((unsigned)e >= (unsigned)nE) {
                atomicOr(err, 1);
                continue;
            }
            atomicAdd(cb + e, 1ull);
            if (SEJ) atomicAdd(sb + e, (unsigned long long)(long long)__ldg(ej + o));
        }
    }
}

// Per data set d (0: every block; 1 + i: every block but i) and bin: the
// sample count and the mean E_J.
__global__ void jk_stats_kernel(const unsigned long long *__restrict__ cnt,
                                const unsigned long long *__restrict__ sej, int n_blocks, int nE,
                                double *n_out, double *mj_out)
{
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    const int d = blockIdx.y;
    if (e >= nE) return;
    unsigned long long n = 0, s = 0;
    for (int b = 0; b < n_blocks; ++b) {
        n += cnt[(size_t)b * nE + e];
        s += sej[(size_t)b * nE + e];
    }
    if (d > 0) {
        n -= cnt[(size_t)(d - 1) * nE + e];
        s -= sej[(size_t)(d - 1) * nE + e];
    }
    n_out[(size_t)d * nE + e] = (double)n;
    mj_out[(size_t)d * nE + e] = n ? (double)(long long)s / (double)n : 0.0;
}

constexpr int kPkThreads = 256;

// ------------------------------------------------------------- blocks of bins
// The bisection evaluates the same sums at some sixty fields of a narrow
// interval.  Over a block of B consecutive bins the weight factorises: with s
// the interval's middle field beta Delta, E_b the block's heaviest bin (the
// largest n exp(-s E - lnW)), E_mid its middle and r = E - E_b,
//   exp(-c E - lnW(E)) = exp(a_b - (c - s) (E_mid - E_r)) exp(-(c - s) (E - E_mid)) V(E),
//   a_b = -s (E_b - E_r) - (lnW(E_b) - lnW(E_r)),   V = exp(-s r - (lnW(E) - lnW(E_b))),
// and |c - s| B / 2 is small in the whole interval, so the middle factor is its
// Taylor polynomial in x = -(c - s) B / 2 and each weighted sum over the block
// is a polynomial in x, its coefficients formed once per call.  A step then
// takes one exponential and 6 deg multiply-adds per block, where the bins took
// an exponential and some hundred FP64 instructions each (FP64 runs at two
// multiply-adds per clock and SM).
// Sums are taken about bins that hold weight (inside a block its heaviest bin
// and weighted mean E_J, then the heaviest block's of the CTA) and moved to the
// common mean at the end of the step.  a_b is kept as a pair (its magnitude
// is that of beta Delta V, the differences between blocks that count are
// small).  C* of a series that fills 61 of 262145 bins, against binary128:
// 1e-15, as with compensated sums over the bins; with a_b rounded once 8e-13.
// Measured: 21 data sets of 4.1e7 samples, 32769 bins, 60 steps: the bisection
// kernel took 8.7 ms bin by bin, now 0.73 ms.
constexpr int kPkStats = 6;    // n, n r, n r^2, n J, n J r, n J r^2 (J about the block's mean)
constexpr int kPkDegMax = 20;
constexpr int kPkMaxB = 512;
constexpr int kPkFew = 64, kPkMany = 256;  // threads per CTA of a step
constexpr int kPkMaxCta = 8;   // CTAs per cluster

struct PkPlan {
    int B, nblk, deg, ncta, threads, per, slots;  // slots = ncta threads per
    double slope;
};

// Bins per block and degree for fields [c_lo, c_hi]: the largest power of 2 with
// |x| <= 1.2 (the polynomial's alternating terms stay within e^2.4 of their
// sum), the first degree whose remainder is below a sixteenth of the rounding;
// single bins when not even blocks of 16 allow it.
PkPlan pk_plan(double c_lo, double c_hi, int nE)
{
    PkPlan p{};
    p.slope = c_lo + 0.5 * (c_hi - c_lo);
    const double w = 0.5 * (c_hi - c_lo);
    for (int B = kPkMaxB; B >= 16 && !p.B; B /= 2)
        if (w * (B / 2) <= 1.2) p.B = B;
    if (!p.B) p.B = 1;
    const double x = w * (p.B / 2);
    double term = 1.0;
    for (p.deg = 0; p.deg < kPkDegMax; ++p.deg) {
        term *= x / (p.deg + 1);
        if (term <= 0x1p-57) break;
    }
    p.nblk = (nE + p.B - 1) / p.B;
    return p;
}

// Thread g of a set's ncta threads takes blocks g per .. g per + per - 1, the
// i-th at slot i ncta threads + g.
__host__ __device__ inline int pk_slot(const PkPlan &p, int b)
{
    return (b % p.per) * (p.ncta * p.threads) + b / p.per;
}

// Per set and slot: coefficients [deg + 1][kPkStats], a_b = ah + al, the
// block's weighted mean E_J, ln of the samples in its heaviest bin (-inf for a
// block without samples), that bin (relative to e_min).
struct PkBlocks {
    double *coef, *ah, *al, *mj, *ln;
    int *E;
};

// Coefficients per block: of a single bin n alone, its other sums are zero.
int pk_coefs(const PkPlan &p) { return p.B == 1 ? 1 : kPkStats * (p.deg + 1); }

size_t pk_block_bytes(const PkPlan &p, int n_sets)
{
    return (size_t)n_sets * p.slots * ((pk_coefs(p) + 4) * sizeof(double) + sizeof(int));
}

PkBlocks pk_block_layout(const PkPlan &p, int n_sets, char *mem)
{
    const size_t n = (size_t)n_sets * p.slots;
    PkBlocks b;
    b.coef = (double *)mem;
    b.ah = b.coef + n * pk_coefs(p);
    b.al = b.ah + n;
    b.mj = b.al + n;
    b.ln = b.mj + n;
    b.E = (int *)(b.ln + n);
    return b;
}

__constant__ double pk_inv[kPkDegMax + 1] = {
    0.0, 1.0, 1.0 / 2, 1.0 / 3, 1.0 / 4, 1.0 / 5, 1.0 / 6, 1.0 / 7, 1.0 / 8, 1.0 / 9, 1.0 / 10,
    1.0 / 11, 1.0 / 12, 1.0 / 13, 1.0 / 14, 1.0 / 15, 1.0 / 16, 1.0 / 17, 1.0 / 18, 1.0 / 19, 1.0 / 20};

// Middle bin of block b (relative to e_min).
__device__ __forceinline__ int pk_mid(const PkPlan &p, int b, int nE)
{
    return min(b * p.B + p.B / 2, nE - 1);
}

// a_b of the bin `ref` relative to the bin `er`, as a pair: the product and the
// differences without rounding.
__device__ __forceinline__ void pk_exponent(double slope, int ref, int er, const double *lnW,
                                            double &ah, double &al)
{
    const double lref = lnW[ref], l0 = lnW[er];
    const double x = (double)(ref - er), a1 = -__dmul_rn(slope, x), pe = fma(slope, x, a1);
    const double l = __dsub_rn(lref, l0), bb = __dsub_rn(l, lref);
    const double le = __dsub_rn(__dsub_rn(lref, __dsub_rn(l, bb)), __dadd_rn(l0, bb));
    const double h = __dsub_rn(a1, l), u = __dsub_rn(h, a1);
    const double he = __dsub_rn(__dsub_rn(a1, __dsub_rn(h, u)), __dadd_rn(l, u));
    ah = h;
    al = he - (pe + le);
}

// Blocks of one bin, a thread each: n is their only statistic.
__global__ void pk_single_kernel(const double *__restrict__ n_all, const double *__restrict__ mj_all,
                                 const double *__restrict__ lnW, int nE, PkPlan p, PkBlocks out)
{
    const int e = blockIdx.x * blockDim.x + threadIdx.x, d = blockIdx.y;
    if (e >= nE) return;
    const double n = n_all[(size_t)d * nE + e];
    const size_t slot = (size_t)d * p.slots + pk_slot(p, e);
    out.ln[slot] = n > 0.0 ? log(n) : -INFINITY;
    out.coef[slot] = n;
    out.mj[slot] = mj_all[(size_t)d * nE + e];
    pk_exponent(p.slope, e, nE / 2, lnW, out.ah[slot], out.al[slot]);
}

// One (block, data set) per CTA of 128 threads.
__global__ void __launch_bounds__(128)
pk_coef_kernel(const double *__restrict__ n_all, const double *__restrict__ mj_all,
               const double *__restrict__ lnW, int nE, PkPlan p, PkBlocks out)
{
    __shared__ double f[kPkStats][64], t[kPkDegMax + 1][64], sv[kPkMaxB];
    __shared__ double red[2][4];
    __shared__ int ired[4];
    const int b = blockIdx.x, d = blockIdx.y, i = threadIdx.x, lane = i & 31, wid = i >> 5;
    const double *n = n_all + (size_t)d * nE, *mj = mj_all + (size_t)d * nE;
    const int e0 = b * p.B, e1 = min(e0 + p.B, nE), mid = pk_mid(p, b, nE);
    const size_t slot = (size_t)d * p.slots + pk_slot(p, b), stride = (size_t)gridDim.y * p.slots;
    // the heaviest bin (to the precision of an FP32 logarithm: any bin near it serves)
    double best = -INFINITY;
    int ref = -1;
    for (int e = e0 + i; e < e1; e += 128)
        if (n[e] > 0.0) {
            const double v = (-(p.slope * (double)(e - mid)) - (lnW[e] - lnW[mid])) +
                             (double)__logf((float)n[e]);
            if (ref < 0 || v > best) {
                best = v;
                ref = e;
            }
        }
    for (int o = 16; o > 0; o >>= 1) {
        const double v2 = __shfl_xor_sync(0xFFFFFFFFu, best, o);
        const int r2 = __shfl_xor_sync(0xFFFFFFFFu, ref, o);
        if (r2 >= 0 && (ref < 0 || v2 > best || (v2 == best && r2 < ref))) {
            best = v2;
            ref = r2;
        }
    }
    if (lane == 0) {
        red[0][wid] = best;
        ired[wid] = ref;
    }
    __syncthreads();
    best = red[0][0];
    ref = ired[0];
    for (int k = 1; k < 4; ++k)
        if (ired[k] >= 0 && (ref < 0 || red[0][k] > best)) {
            best = red[0][k];
            ref = ired[k];
        }
    if (ref < 0) {  // no samples: the whole CTA
        if (i == 0) out.ln[slot] = -INFINITY;
        return;
    }
    __syncthreads();
    const double lref = lnW[ref], jref = mj[ref];
    double sn = 0.0, sj = 0.0;
    for (int e = e0 + i; e < e1; e += 128) {
        // near the heaviest bin the exponents are differences of near numbers
        const double vn = n[e] > 0.0 ? exp(-(p.slope * (double)(e - ref)) - (lnW[e] - lref)) * n[e] : 0.0;
        sv[e - e0] = vn;
        sn += vn;
        sj += n[e] > 0.0 ? vn * (mj[e] - jref) : 0.0;
    }
    for (int o = 16; o > 0; o >>= 1) {
        sn += __shfl_xor_sync(0xFFFFFFFFu, sn, o);
        sj += __shfl_xor_sync(0xFFFFFFFFu, sj, o);
    }
    if (lane == 0) {
        red[0][wid] = sn;
        red[1][wid] = sj;
    }
    __syncthreads();
    sn = (red[0][0] + red[0][1]) + (red[0][2] + red[0][3]);
    sj = (red[1][0] + red[1][1]) + (red[1][2] + red[1][3]);
    const double jb = jref + sj / sn;
    if (i == 0) {
        pk_exponent(p.slope, ref, nE / 2, lnW, out.ah[slot], out.al[slot]);
        out.mj[slot] = jb;
        out.ln[slot] = log(n[ref]);
        out.E[slot] = ref;
    }
    double c[2] = {0.0, 0.0};  // this thread's coefficients i and i + 128
    for (int k0 = e0; k0 < e1; k0 += 64) {
        __syncthreads();
        if (i < 64) {
            const int e = k0 + i;
            const bool in = e < e1 && n[e] > 0.0;
            const double r = (double)(e - ref), dj = in ? mj[e] - jb : 0.0;
            const double vn = in ? sv[e - e0] : 0.0;
            f[0][i] = vn;
            f[1][i] = vn * r;
            f[2][i] = vn * (r * r);
            f[3][i] = vn * dj;
            f[4][i] = vn * (dj * r);
            f[5][i] = vn * (dj * r * r);
            const double rho = (double)(e - mid) * (2.0 / p.B);  // exact: B is a power of 2
            double pw = 1.0;
            t[0][i] = 1.0;
            for (int q = 1; q <= p.deg; ++q) {
                pw *= rho * pk_inv[q];
                t[q][i] = pw;
            }
        }
        __syncthreads();
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int q = i + 128 * u;
            if (q >= kPkStats * (p.deg + 1)) continue;
            const double *ff = f[q % kPkStats], *tt = t[q / kPkStats];
            for (int k = 0; k < 64; ++k) c[u] = fma(ff[k], tt[k], c[u]);
        }
    }
#pragma unroll
    for (int u = 0; u < 2; ++u) {
        const int q = i + 128 * u;
        if (q < kPkStats * (p.deg + 1)) out.coef[(size_t)q * stride + slot] = c[u];
    }
}

// A block as the reference of a CTA's sums (E < 0: none).
struct PkRef {
    double ah, al, ln, J;
    int mid, E;
};

// One CTA's part of a step: its sums R relative to the exponent of its reference
// block, about (E, J) of that block, then (in a step that finds it) the block's
// ah, al, ln, J, (E, mid).
constexpr int kPkWords = kPkStats + 5;
constexpr int kPkSums = kPkMany / 32 * kPkStats;
struct PkPart {
    double w[kPkWords];
};

// Move the sums R of n, n E, n E^2, n J, n J E, n J E^2 to references that lie
// dE and dJ lower (E and J grow by them).
__device__ __forceinline__ void pk_shift(double (&R)[kPkStats], double dE, double dJ)
{
    const double e1 = fma(dE, R[0], R[1]), e2 = fma(dE, R[1] + e1, R[2]);
    const double j1 = fma(dE, R[3], R[4]), j2 = fma(dE, R[4] + j1, R[5]);
    R[3] = fma(dJ, R[0], R[3]);
    R[4] = fma(dJ, e1, j1);
    R[5] = fma(dJ, e2, j2);
    R[1] = e1;
    R[2] = e2;
}

// Covariance <(E_J - <E_J>)(E_Delta - <E_Delta>)> and third moment
// <(E_J - <E_J>)(E_Delta - <E_Delta>)^2> of data set d at field c = beta Delta.
// The CTAs hand their parts to one another in slot `slot` of each one's `part`
// (slots alternate, so one cluster barrier per step suffices); every thread gets
// the result.
// ref: the heaviest of the CTA's blocks, found anew when `find` is set, else kept
// as a fixed reference; peer: that of rank lane % 8, in warp 0.
// SINGLE: blocks of one bin, whose only statistic is n.
// Results: the moments times z = sum n (the sign of the third is all that a
// step needs).
template <int NT, bool SINGLE>
__device__ void pk_moments(cg::cluster_group &cl, PkPart *part, int &slot, const PkBlocks &bl,
                           const PkPlan &p, int d, int nE, double c, bool find, PkRef &ref,
                           PkRef &peer, double *sh, int *shi, double &cov, double &third, double &z0)
{
    const int q = (int)cl.block_rank(), t = (int)threadIdx.x, lane = t & 31, wid = t >> 5;
    const int g = q * NT + t, gs = p.ncta * NT;
    const size_t base = (size_t)d * p.slots, stride = (size_t)(gridDim.x / p.ncta) * p.slots;
    const double dc = c - p.slope, x = -dc * (0.5 * p.B);
    const int er = nE / 2;
    if (find) {
        double mx = -INFINITY;
        int at = -1;
        for (int i = 0; i < p.per; ++i) {
            const int b = g * p.per + i;
            const size_t k = base + (size_t)i * gs + g;
            if (b >= p.nblk || bl.ln[k] == -INFINITY) continue;
            const double v = fma(-dc, (double)(pk_mid(p, b, nE) - er), bl.ah[k]) + bl.ln[k];
            if (v > mx) {
                mx = v;
                at = b;
            }
        }
        for (int o = 16; o > 0; o >>= 1) {
            const double v2 = __shfl_xor_sync(0xFFFFFFFFu, mx, o);
            const int a2 = __shfl_xor_sync(0xFFFFFFFFu, at, o);
            if (v2 > mx || (v2 == mx && a2 > at)) {
                mx = v2;
                at = a2;
            }
        }
        __syncthreads();
        if (lane == 0) {
            sh[wid] = mx;
            shi[wid] = at;
        }
        __syncthreads();
        for (int i = 0; i < NT / 32; ++i)
            if (sh[i] > mx || (sh[i] == mx && shi[i] > at)) {
                mx = sh[i];
                at = shi[i];
            }
        ref = PkRef{0.0, 0.0, -INFINITY, 0.0, er, -1};
        if (at >= 0) {
            const size_t k = base + pk_slot(p, at);
            ref = PkRef{bl.ah[k], bl.al[k], bl.ln[k], bl.mj[k], pk_mid(p, at, nE),
                        SINGLE ? at : bl.E[k]};
        }
    }
    double S[kPkStats];
#pragma unroll
    for (int j = 0; j < kPkStats; ++j) S[j] = 0.0;
    for (int i = 0; i < p.per; ++i) {
        const int b = g * p.per + i;
        const size_t k = base + (size_t)i * gs + g;
        // loaded together (slots past the last block are allocated, and not used)
        const double ln = bl.ln[k], ah = bl.ah[k], al = bl.al[k], mj = bl.mj[k];
        const double n = SINGLE ? bl.coef[k] : 0.0;
        const int E = SINGLE ? b : bl.E[k];
        if (b >= p.nblk || ln == -INFINITY) continue;
        const double A = exp(fma(-dc, (double)(pk_mid(p, b, nE) - ref.mid), (ah - ref.ah) + (al - ref.al)));
        if (!(A > 0.0)) continue;
        if constexpr (SINGLE) {
            const double dE = (double)(E - ref.E), dJ = mj - ref.J, w = A * n;
            const double we = w * dE, wee = we * dE;
            S[0] += w;
            S[1] += we;
            S[2] += wee;
            S[3] = fma(w, dJ, S[3]);
            S[4] = fma(we, dJ, S[4]);
            S[5] = fma(wee, dJ, S[5]);
        } else {
            double R[kPkStats];
#pragma unroll
            for (int j = 0; j < kPkStats; ++j)
                R[j] = bl.coef[(size_t)(p.deg * kPkStats + j) * stride + k];
            // (unrolled: the coefficients of several orders are on their way at once)
#pragma unroll 4
            for (int u = p.deg - 1; u >= 0; --u)
#pragma unroll
                for (int j = 0; j < kPkStats; ++j)
                    R[j] = fma(R[j], x, bl.coef[(size_t)(u * kPkStats + j) * stride + k]);
            pk_shift(R, (double)(E - ref.E), mj - ref.J);
#pragma unroll
            for (int j = 0; j < kPkStats; ++j) S[j] = fma(A, R[j], S[j]);
        }
    }
#pragma unroll
    for (int j = 0; j < kPkStats; ++j)
        for (int o = 16; o > 0; o >>= 1) S[j] += __shfl_xor_sync(0xFFFFFFFFu, S[j], o);
    __syncthreads();
    if (lane == 0)
#pragma unroll
        for (int j = 0; j < kPkStats; ++j) sh[wid * kPkStats + j] = S[j];
    __syncthreads();
    // this CTA's part to every CTA of the cluster, a word per thread (reading the
    // others' parts instead waits for distributed shared memory once more)
    const int words = find ? kPkWords : kPkStats;
    for (int i = t; i < 8 * words; i += NT) {
        const int r = i & 7, w = i >> 3;
        if (r >= p.ncta) continue;
        double v = 0.0;
        if (w < kPkStats)
            for (int k = 0; k < NT / 32; ++k) v += sh[k * kPkStats + w];
        else
            v = w == kPkStats       ? ref.ah
                : w == kPkStats + 1 ? ref.al
                : w == kPkStats + 2 ? ref.ln
                : w == kPkStats + 3 ? ref.J
                                    : __hiloint2double(ref.E, ref.mid);
        cl.map_shared_rank(part, r)[slot * kPkMaxCta + q].w[w] = v;
    }
    cl.sync();
    // lane r of each eight of warp 0 takes rank r's part
    if (wid == 0) {
        const bool in = (lane & 7) < p.ncta;
        const double *pw = part[slot * kPkMaxCta + (in ? lane & 7 : 0)].w;
        if (find) {
            const double ei = pw[kPkStats + 4];
            peer = PkRef{pw[kPkStats], pw[kPkStats + 1], pw[kPkStats + 2], pw[kPkStats + 3],
                         __double2loint(ei), __double2hiint(ei)};
        }
        const PkRef &rr = peer;
        double R[kPkStats];
#pragma unroll
        for (int j = 0; j < kPkStats; ++j) R[j] = pw[j];
        const bool on = in && rr.E >= 0;
        const double m = on ? fma(-dc, (double)(rr.mid - er), rr.ah) + rr.ln : -INFINITY;
        double M = m;
        for (int o = 4; o > 0; o >>= 1) M = fmax(M, __shfl_xor_sync(0xFFFFFFFFu, M, o));
        const int top = __ffs((int)__ballot_sync(0xFFFFFFFFu, m == M)) - 1;
        // relative to the leading CTA's reference
        const double h0 = __shfl_sync(0xFFFFFFFFu, rr.ah, top), l0 = __shfl_sync(0xFFFFFFFFu, rr.al, top);
        const int mid0 = __shfl_sync(0xFFFFFFFFu, rr.mid, top);
        const int E0 = __shfl_sync(0xFFFFFFFFu, rr.E, top);
        const double J0 = __shfl_sync(0xFFFFFFFFu, rr.J, top);
        const double f = exp(fma(-dc, (double)(rr.mid - mid0), (rr.ah - h0) + (rr.al - l0)));
#pragma unroll
        for (int j = 0; j < kPkStats; ++j) R[j] = on ? f * R[j] : 0.0;
        const int Er = on ? rr.E : E0;
        const double Jr = on ? rr.J : J0;
        // the means about the leading CTA's references
        double z[3] = {R[0], fma(R[0], (double)(Er - E0), R[1]), fma(R[0], Jr - J0, R[3])};
#pragma unroll
        for (int j = 0; j < 3; ++j)
            for (int o = 4; o > 0; o >>= 1) z[j] += __shfl_xor_sync(0xFFFFFFFFu, z[j], o);
        const double iz = 1.0 / z[0];
        pk_shift(R, (double)(Er - E0) - z[1] * iz, (Jr - J0) - z[2] * iz);
        double cv = R[4], th = R[5];
        for (int o = 4; o > 0; o >>= 1) {
            cv += __shfl_xor_sync(0xFFFFFFFFu, cv, o);
            th += __shfl_xor_sync(0xFFFFFFFFu, th, o);
        }
        if (lane == 0) {
            sh[kPkSums] = cv;
            sh[kPkSums + 1] = th;
            sh[kPkSums + 2] = z[0];
        }
    }
    slot ^= 1;
    __syncthreads();
    cov = sh[kPkSums];
    third = sh[kPkSums + 1];
    z0 = sh[kPkSums + 2];
}

// One cluster per data set: bisection on the sign of dC/dDelta in [lo, hi].
// Every CTA of a cluster holds the same combined sums, so all take the same
// steps.  A cluster barrier before the first step: a CTA's shared memory may be
// written by the others only once it runs.
template <int NT, bool SINGLE>
__global__ void __launch_bounds__(NT)
peak_kernel(PkBlocks bl, PkPlan p, int nE, double beta, double lo, double hi, int n_iter,
            double *res, int *bad)
{
    __shared__ double sh[kPkSums + 3];  // the warps' sums, then the results
    __shared__ int shi[kPkMany / 32];
    __shared__ PkPart part[2 * kPkMaxCta];  // [slot][rank]
    cg::cluster_group cl = cg::this_cluster();
    cl.sync();
    const int q = (int)cl.block_rank(), d = blockIdx.x / p.ncta;
    int slot = 0;
    // Exponents move by at most beta (hi - lo) |E - E'| in what is left of the
    // interval: once that is 2, the heaviest block of the step before holds at least
    // e^-2 of the weight that the heaviest has, and is not looked for again.  (At the
    // ends of a wider interval it may hold next to nothing: the sums about it would
    // be differences of large numbers, down to the sign of the third moment.)
    // (Looked for in some seven steps of 63 instead of one: about 1.5 % of the kernel.)
    PkRef ref, peer;
    double z0;
    bool first = true;
    auto third_at = [&](double delta, double &cov) {
        double t;
        const bool find = first || beta * (hi - lo) * nE > 2.0;
        first = false;
        pk_moments<NT, SINGLE>(cl, part, slot, bl, p, d, nE, beta * delta, find, ref, peer, sh, shi,
                               cov, t, z0);
        return t;
    };
    double cov;
    const double t_lo = third_at(lo, cov), t_hi = third_at(hi, cov);
    if (!(t_lo > 0.0 && t_hi < 0.0)) {
        if (q == 0 && threadIdx.x == 0) bad[d] = 1;
        return;
    }
    for (int i = 0; i < n_iter; ++i) {
        const double mid = lo + 0.5 * (hi - lo);
        if (third_at(mid, cov) > 0.0) lo = mid;
        else hi = mid;
    }
    const double ds = lo + 0.5 * (hi - lo);
    third_at(ds, cov);
    if (q == 0 && threadIdx.x == 0) {
        res[2 * d] = ds;
        res[2 * d + 1] = -beta * (cov / z0);
    }
}

// ---------------------------------------------------- equal height, barrier
// The reweighted E_Delta distribution at field Delta, from the series' count
// n(E) per bin: ln P(E) = ln n(E) - beta Delta E - lnW(E) (+ const).  Delta_eqh
// is where its highest bins below and at or above split are equally high;
// B = ln(P_max / P_min) / (2 beta Delta_eqh), P_min the lowest occupied bin
// between the two peaks.

// Per data set d and bin: ln of the sample count (-inf when empty).
__global__ void jk_lncount_kernel(const unsigned long long *__restrict__ cnt, int n_blocks, int nE,
                                  double *lnn)
{
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    const int d = blockIdx.y;
    if (e >= nE) return;
    unsigned long long n = 0;
    for (int b = 0; b < n_blocks; ++b) n += cnt[(size_t)b * nE + e];
    if (d > 0) n -= cnt[(size_t)(d - 1) * nE + e];
    lnn[(size_t)d * nE + e] = n ? log((double)n) : -INFINITY;
}

// ln P(E) at Delta, evaluated in the order (ln n - (beta Delta) E) - lnW.
__device__ __forceinline__ double eqh_lnp(double lnn, double bd, int E, double lnw)
{
    return __dsub_rn(__dsub_rn(lnn, __dmul_rn(bd, (double)E)), lnw);
}

// Larger (want_max) or smaller value wins, ties to the smaller bin, bin -1 is empty.
__device__ __forceinline__ bool eqh_better(double v2, int a2, double v, int a, bool want_max)
{
    if (a2 < 0) return false;
    if (a < 0) return true;
    if (want_max ? v2 > v : v2 < v) return true;
    return v2 == v && a2 < a;
}

// Block-wide best of K (value, bin) pairs; every thread gets the result.
template <int K>
__device__ void eqh_best(double (&v)[K], int (&a)[K], bool want_max, double *sh, int *shi)
{
#pragma unroll
    for (int k = 0; k < K; ++k)
        for (int o = 16; o > 0; o >>= 1) {
            const double v2 = __shfl_xor_sync(0xFFFFFFFFu, v[k], o);
            const int a2 = __shfl_xor_sync(0xFFFFFFFFu, a[k], o);
            if (eqh_better(v2, a2, v[k], a[k], want_max)) {
                v[k] = v2;
                a[k] = a2;
            }
        }
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    __syncthreads();
    if (lane == 0)
#pragma unroll
        for (int k = 0; k < K; ++k) {
            sh[K * wid + k] = v[k];
            shi[K * wid + k] = a[k];
        }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < K; ++k) {
        v[k] = sh[k];
        a[k] = shi[k];
        for (int i = 1; i < nw; ++i)
            if (eqh_better(sh[K * i + k], shi[K * i + k], v[k], a[k], want_max)) {
                v[k] = sh[K * i + k];
                a[k] = shi[K * i + k];
            }
    }
}

// The bins of a thread that can still hold a peak, bit i for its i-th bin
// (bins from the 64th on always count).  A bin drops out when it lies below its
// side's peak of the step before by more than the interval that is left can
// make up: ln P of two bins moves apart by beta |E - E'| per unit of Delta.
// The interval halves with every step, so after some ten steps a few bins per
// side are left, and the others are not read again.  Measured: 21 data sets x
// 32769 bins, 60 steps: 1.20 -> 0.46 ms.
struct EqLive {
    unsigned long long mask = ~0ull;
    bool have = false;  // peaks of a step before: bins p, values v at field bd
    int p[2];
    double v[2], bd;
};

// The two peak bins at beta Delta = bd among bins [e0, e1) (relative to e_min,
// -1 when a side is empty); reach: beta times the width of the interval that
// holds every field still to come, bd among them; slack: above the rounding of
// the values that are compared.
__device__ void eqh_peaks(const double *lnn, const double *lnW, int e0, int e1, int e_min,
                          int split, double bd, double reach, double slack, EqLive &live,
                          int (&p)[2],
                          double (&v)[2], double *sh, int *shi)
{
    v[0] = v[1] = -INFINITY;
    p[0] = p[1] = -1;
    double top[2] = {0.0, 0.0};
    if (live.have)
        for (int s = 0; s < 2; ++s)
            top[s] = live.v[s] - (bd - live.bd) * (double)(e_min + live.p[s]);
    int i = 0;
    for (int e = e0 + (int)threadIdx.x; e < e1; e += blockDim.x, ++i) {
        const unsigned long long bit = i < 64 ? 1ull << i : 0ull;
        if (bit && !(live.mask & bit)) continue;
        const double n = lnn[e];
        if (n == -INFINITY) {
            live.mask &= ~bit;
            continue;
        }
        const double w = eqh_lnp(n, bd, e_min + e, lnW[e]);
        const int s = e_min + e < split ? 0 : 1;
        if (live.have && (w - top[s]) + reach * (double)abs(e - live.p[s]) < -slack) {
            live.mask &= ~bit;
            continue;
        }
        if (p[s] < 0 || w > v[s]) {
            v[s] = w;
            p[s] = e;
        }
    }
    eqh_best<2>(v, p, true, sh, shi);
}

// One CTA's best (value, bin) pairs for the two peaks, or its lowest bin.
struct EqPart {
    double vl, vr;
    int pl, pr;
};

// The cluster's peaks from its CTAs' block results, combined in rank order
// through the slot `slot` of every CTA's parts (slots alternate, so one
// cluster barrier per combination suffices).
__device__ double eqh_cluster_peaks(cg::cluster_group &cl, EqPart *part, int &slot, int &pl, int &pr,
                                    double &vl, double &vr)
{
    if (threadIdx.x == 0) part[slot] = EqPart{vl, vr, pl, pr};
    cl.sync();
    double bl = -INFINITY, br = -INFINITY;
    int al = -1, ar = -1;
    for (int r = 0; r < (int)cl.num_blocks(); ++r) {
        const EqPart q = cl.map_shared_rank(part, r)[slot];
        if (eqh_better(q.vl, q.pl, bl, al, true)) {
            bl = q.vl;
            al = q.pl;
        }
        if (eqh_better(q.vr, q.pr, br, ar, true)) {
            br = q.vr;
            ar = q.pr;
        }
    }
    slot ^= 1;
    vl = bl;
    vr = br;
    pl = al;
    pr = ar;
    return vl - vr;
}

// One cluster per data set (each CTA over its slice [e0, e1) of the bins):
// bisection on g = ln P_low - ln P_high, then the barrier at Delta_eqh.
__global__ void __launch_bounds__(kPkThreads)
eqh_kernel(const double *__restrict__ lnn_all, const double *__restrict__ lnW, int nE, int e_min,
           int split, double beta, double lo, double hi, int n_iter, double slack, double *res,
           int *bad)
{
    __shared__ double sh[64];
    __shared__ int shi[64];
    __shared__ EqPart part[2];
    cg::cluster_group cl = cg::this_cluster();
    const int ncta = (int)cl.num_blocks(), q = (int)cl.block_rank();
    const int d = blockIdx.x / ncta;
    const int e0 = (int)((int64_t)nE * q / ncta), e1 = (int)((int64_t)nE * (q + 1) / ncta);
    const double *lnn = lnn_all + (size_t)d * nE;
    int slot = 0;
    EqLive live;
    auto peaks = [&](double bd, int &pl, int &pr, double &vl, double &vr) {
        double v[2];
        int p[2];
        eqh_peaks(lnn, lnW, e0, e1, e_min, split, bd, beta * (hi - lo), slack, live, p, v, sh,
                  shi);
        vl = v[0];
        vr = v[1];
        pl = p[0];
        pr = p[1];
        const double g = eqh_cluster_peaks(cl, part, slot, pl, pr, vl, vr);
        live.have = pl >= 0 && pr >= 0;
        live.p[0] = pl;
        live.p[1] = pr;
        live.v[0] = vl;
        live.v[1] = vr;
        live.bd = bd;
        return g;
    };
    int pl, pr;
    double vl, vr;
    const double g_lo = peaks(beta * lo, pl, pr, vl, vr);
    const bool ok_lo = pl >= 0 && pr >= 0;
    const double g_hi = peaks(beta * hi, pl, pr, vl, vr);
    if (!ok_lo || pl < 0 || pr < 0 || !(g_lo < 0.0 && g_hi > 0.0)) {
        if (q == 0 && threadIdx.x == 0) bad[d] = 1;
        cl.sync();
        return;
    }
    for (int i = 0; i < n_iter; ++i) {
        const double mid = lo + 0.5 * (hi - lo);
        if (peaks(beta * mid, pl, pr, vl, vr) < 0.0) lo = mid;
        else hi = mid;
    }
    const double dq = lo + 0.5 * (hi - lo);
    const double bd = beta * dq;
    peaks(bd, pl, pr, vl, vr);
    const double vmax = vl > vr ? vl : vr;
    double vmin = INFINITY;
    int pm = -1;
    for (int e = max(pl, e0) + (int)threadIdx.x; e <= min(pr, e1 - 1); e += blockDim.x) {
        if (lnn[e] == -INFINITY) continue;
        const double v = eqh_lnp(lnn[e], bd, e_min + e, lnW[e]);
        if (pm < 0 || v < vmin) {
            vmin = v;
            pm = e;
        }
    }
    {
        double v[1] = {vmin};
        int a[1] = {pm};
        eqh_best<1>(v, a, false, sh, shi);
        vmin = v[0];
        pm = a[0];
    }
    if (threadIdx.x == 0) part[slot] = EqPart{vmin, 0.0, pm, -1};
    cl.sync();
    double bm = INFINITY;
    int am = -1;
    for (int r = 0; r < ncta; ++r) {
        const EqPart qq = cl.map_shared_rank(part, r)[slot];
        if (eqh_better(qq.vl, qq.pl, bm, am, false)) {
            bm = qq.vl;
            am = qq.pl;
        }
    }
    vmin = bm;
    pm = am;
    if (q == 0 && threadIdx.x == 0) {
        double *o = res + 5 * (size_t)d;
        o[0] = dq;
        o[1] = (vmax - vmin) / (2.0 * beta * dq);
        o[2] = (double)(e_min + pl);
        o[3] = (double)(e_min + pr);
        o[4] = (double)(e_min + pm);
    }
    cl.sync();
}

int pk_fail(int code, const std::string &msg)
{
    muca::set_last_error(msg.c_str());
    return code;
}

}  // namespace

// Launch configuration of a per-data-set cluster kernel: one cluster per data
// set and one CTA per SM (the CTAs reserve unused dynamic shared memory above
// half an SM's); the cluster size is the largest of min(8, max_cta) .. 1 for which every
// data set's cluster can be resident at once (clusters live within a GPC, so
// the SM count alone does not tell).  attr must outlive cfg.
static cudaError_t cluster_config(const void *kernel, int n_sets, int threads, int max_cta,
                                  cudaStream_t st, cudaLaunchConfig_t &cfg,
                                  cudaLaunchAttribute (&attr)[1])
{
    int dev = 0, nsm = 152, smem_sm = 0;
    cudaError_t ce = cudaGetDevice(&dev);
    if (ce != cudaSuccess) return ce;
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    cudaDeviceGetAttribute(&smem_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev);
    const size_t one_per_sm = smem_sm > 0 ? (size_t)smem_sm / 2 + 1024 : 0;
    ce = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)one_per_sm);
    if (ce != cudaSuccess) return ce;
    cfg = cudaLaunchConfig_t{};
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = one_per_sm;
    cfg.stream = st;
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int ncta = std::max(1, std::min(std::min(kPkMaxCta, max_cta), nsm / std::max(n_sets, 1)));
    for (; ncta > 1; --ncta) {
        attr[0].val.clusterDim.x = (unsigned)ncta;
        cfg.gridDim = dim3((unsigned)(n_sets * ncta));
        int nc = 0;
        if (cudaOccupancyMaxActiveClusters(&nc, kernel, &cfg) == cudaSuccess && nc >= n_sets) break;
    }
    (void)cudaGetLastError();
    attr[0].val.clusterDim.x = (unsigned)ncta;
    cfg.gridDim = dim3((unsigned)(n_sets * ncta));
    return cudaSuccess;
}

extern "C" int muca_find_peak(const int32_t *e_j, const int32_t *e_d, int64_t n_rows,
                              int32_t row_len, int64_t row_stride, const double *lnW,
                              int32_t e_min, int32_t n_e, double beta, double delta_lo,
                              double delta_hi, int32_t n_iter, int32_t n_jack, double *out,
                              void *stream)
{
    if (!e_j || !e_d || !lnW || !out)
        return pk_fail(MUCA_ERR_INVALID_ARG, "muca_find_peak: null pointer");
    if (n_rows < 1 || row_len < 1 || (n_rows > 1 && row_stride < row_len) || n_e < 1 ||
        n_iter < 0 || n_iter > 200 || n_jack < 0 || n_jack == 1 || n_jack > n_rows ||
        n_jack > 1024)
        return pk_fail(MUCA_ERR_INVALID_ARG, "muca_find_peak: bad sizes");
    if ((int64_t)e_min + n_e - 1 > INT32_MAX)
        return pk_fail(MUCA_ERR_INVALID_ARG, "muca_find_peak: e_min + n_e - 1 exceeds int32");
    if (!(beta > 0.0) || !std::isfinite(beta) || !std::isfinite(delta_lo) ||
        !std::isfinite(delta_hi) || !(delta_lo < delta_hi))
        return pk_fail(MUCA_ERR_INVALID_ARG, "muca_find_peak: need beta > 0 and delta_lo < delta_hi");
    for (int e = 0; e < n_e; ++e)
        if (!std::isfinite(lnW[e])) return pk_fail(MUCA_ERR_INVALID_ARG, "muca_find_peak: lnW not finite");
    cudaStream_t st = (cudaStream_t)stream;
    const int n_blocks = n_jack > 0 ? n_jack : 1, n_sets = 1 + n_jack;
    std::vector<int64_t> bnd(n_blocks + 1);
    for (int i = 0; i <= n_blocks; ++i) bnd[i] = (int64_t)i * n_rows / n_blocks;
    auto al = [](size_t x) { return (x + 255) & ~(size_t)255; };
    const size_t b_sums = al((size_t)2 * n_blocks * n_e * sizeof(unsigned long long));
    const size_t b_sets = al((size_t)2 * n_sets * n_e * sizeof(double));
    const size_t b_lnw = al((size_t)n_e * sizeof(double));
    const size_t b_bnd = al(bnd.size() * sizeof(int64_t));
    const size_t b_res = al((size_t)2 * n_sets * sizeof(double));
    const size_t b_bad = al((size_t)(n_sets + 1) * sizeof(int));
    // blocks of bins, spread over the CTAs of each set's cluster: at least 16
    // blocks per CTA (below that a step is its barriers), and 256 threads per CTA
    // instead of 64 where those would take more than two blocks each (latency:
    // 101 sets of 4097 bins in blocks of 32 2.5 -> 1.5 ms, of 1729 single bins
    // on 8 CTAs 0.81 -> 0.71 ms; 513 single bins on 8 CTAs 0.60 on 64 threads,
    // 0.68 on 256)
    PkPlan plan = pk_plan(beta * delta_lo, beta * delta_hi, n_e);
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr[1];
    const bool single = plan.B == 1;
    auto kernel = single ? &peak_kernel<kPkFew, true> : &peak_kernel<kPkFew, false>;
    plan.threads = kPkFew;
    cudaError_t ce = cluster_config((const void *)kernel, n_sets, plan.threads,
                                    (plan.nblk + 15) / 16, st, cfg, attr);
    if (ce == cudaSuccess && plan.nblk > 2 * kPkFew * (int)attr[0].val.clusterDim.x) {
        kernel = single ? &peak_kernel<kPkMany, true> : &peak_kernel<kPkMany, false>;
        plan.threads = kPkMany;
        ce = cluster_config((const void *)kernel, n_sets, plan.threads, kPkMaxCta, st, cfg, attr);
    }
    if (ce != cudaSuccess)
        return pk_fail(MUCA_ERR_CUDA, std::string("cluster configuration: ") + cudaGetErrorString(ce));
    plan.ncta = (int)attr[0].val.clusterDim.x;
    plan.per = (plan.nblk + plan.ncta * plan.threads - 1) / (plan.ncta * plan.threads);
    plan.slots = plan.ncta * plan.threads * plan.per;
    const size_t b_w = al(pk_block_bytes(plan, n_sets));
    char *p = nullptr;
    cudaMemPool_t pool = nullptr;
    const int rp = muca::scratch_pool(muca::ScratchPool::peak, &pool);
    if (rp != MUCA_OK) return rp;
    ce = cudaMallocFromPoolAsync((void **)&p, b_sums + b_sets + b_lnw + b_bnd + b_res + b_bad + b_w,
                                 pool, st);
    if (ce != cudaSuccess)
        return pk_fail(ce == cudaErrorMemoryAllocation ? MUCA_ERR_OOM : MUCA_ERR_CUDA,
                       std::string("cudaMallocAsync: ") + cudaGetErrorString(ce));
    unsigned long long *cnt = (unsigned long long *)p, *sej = cnt + (size_t)n_blocks * n_e;
    double *n_all = (double *)(p + b_sums), *mj_all = n_all + (size_t)n_sets * n_e;
    double *d_lnW = (double *)(p + b_sums + b_sets);
    int64_t *d_bnd = (int64_t *)(p + b_sums + b_sets + b_lnw);
    double *d_res = (double *)(p + b_sums + b_sets + b_lnw + b_bnd);
    int *d_bad = (int *)(p + b_sums + b_sets + b_lnw + b_bnd + b_res);  // [0]: window, [1 + d]
    const PkBlocks blocks =
        pk_block_layout(plan, n_sets, p + b_sums + b_sets + b_lnw + b_bnd + b_res + b_bad);
    std::vector<double> res(2 * (size_t)n_sets, 0.0);
    std::vector<int> bad(n_sets + 1, 0);
    int rc = MUCA_OK;
#define PCK(call)                                                                         \
    do {                                                                                  \
        ce = (call);                                                                      \
        if (ce != cudaSuccess) {                                                          \
            rc = pk_fail(MUCA_ERR_CUDA, std::string(#call) + ": " + cudaGetErrorString(ce)); \
            goto done;                                                                    \
        }                                                                                 \
    } while (0)
    PCK(cudaMemsetAsync(p, 0, b_sums, st));
    PCK(cudaMemsetAsync(d_bad, 0, b_bad, st));
    PCK(cudaMemcpyAsync(d_lnW, lnW, (size_t)n_e * sizeof(double), cudaMemcpyHostToDevice, st));
    PCK(cudaMemcpyAsync(d_bnd, bnd.data(), bnd.size() * sizeof(int64_t), cudaMemcpyHostToDevice, st));
    {
        dim3 g((unsigned)std::min<int64_t>((row_len + 255) / 256, 1024),
               (unsigned)std::min<int64_t>(n_rows, 4096));
        jk_bin_kernel<true><<<g, 256, 0, st>>>(e_j, e_d, n_rows, row_len, row_stride, e_min, n_e,
                                               d_bnd, n_blocks, cnt, sej, d_bad);
        PCK(cudaGetLastError());
        dim3 g2((unsigned)((n_e + 255) / 256), (unsigned)n_sets);
        jk_stats_kernel<<<g2, 256, 0, st>>>(cnt, sej, n_blocks, n_e, n_all, mj_all);
        PCK(cudaGetLastError());
        if (single)
            pk_single_kernel<<<g2, 256, 0, st>>>(n_all, mj_all, d_lnW, n_e, plan, blocks);
        else
            pk_coef_kernel<<<dim3((unsigned)plan.nblk, (unsigned)n_sets), 128, 0, st>>>(
                n_all, mj_all, d_lnW, n_e, plan, blocks);
        PCK(cudaGetLastError());
        PCK(cudaLaunchKernelEx(&cfg, kernel, blocks, plan, (int)n_e, beta, delta_lo, delta_hi,
                               (int)n_iter, d_res, d_bad + 1));
    }
    PCK(cudaMemcpyAsync(res.data(), d_res, res.size() * sizeof(double), cudaMemcpyDeviceToHost, st));
    PCK(cudaMemcpyAsync(bad.data(), d_bad, bad.size() * sizeof(int), cudaMemcpyDeviceToHost, st));
    PCK(cudaStreamSynchronize(st));
#undef PCK
    if (bad[0]) {
        rc = pk_fail(MUCA_ERR_WINDOW, "a sample's E_Delta lies outside [e_min, e_min + n_e)");
        goto done;
    }
    for (int d = 0; d < n_sets; ++d)
        if (bad[1 + d]) {
            rc = pk_fail(MUCA_ERR_INVALID_ARG,
                         "muca_find_peak: [delta_lo, delta_hi] does not bracket the maximum of C "
                         "for data set " + std::to_string(d) +
                         " (dC/dDelta must be > 0 at delta_lo and < 0 at delta_hi)");
            goto done;
        }
    {
        // jackknife errors: var = (w - 1) / w sum_i (x_i - mean_i x_i)^2
        double err[2] = {0.0, 0.0};
        if (n_jack > 0) {
            for (int q = 0; q < 2; ++q) {
                double mean = 0.0;
                for (int i = 0; i < n_jack; ++i) mean += res[2 * (1 + i) + q];
                mean /= n_jack;
                double ss = 0.0;
                for (int i = 0; i < n_jack; ++i) {
                    const double dv = res[2 * (1 + i) + q] - mean;
                    ss += dv * dv;
                }
                err[q] = std::sqrt((double)(n_jack - 1) / n_jack * ss);
            }
        }
        out[0] = res[0];
        out[1] = err[0];
        out[2] = res[1];
        out[3] = err[1];
        for (int i = 0; i < n_jack; ++i) {
            out[4 + 2 * i] = res[2 * (1 + i)];
            out[5 + 2 * i] = res[2 * (1 + i) + 1];
        }
    }
done:
    cudaFreeAsync(p, st);
    cudaStreamSynchronize(st);
    return rc;
}

extern "C" int muca_equal_height(const int32_t *e_d, int64_t n_rows, int32_t row_len,
                                 int64_t row_stride, const double *lnW, int32_t e_min,
                                 int32_t n_e, double beta, int32_t split, double delta_lo,
                                 double delta_hi, int32_t n_iter, int32_t n_jack, double *out,
                                 void *stream)
{
    if (!e_d || !lnW || !out) return pk_fail(MUCA_ERR_INVALID_ARG, "muca_equal_height: null pointer");
    if (n_rows < 1 || row_len < 1 || (n_rows > 1 && row_stride < row_len) || n_e < 1 ||
        n_iter < 0 || n_iter > 200 || n_jack < 0 || n_jack == 1 || n_jack > n_rows ||
        n_jack > 1024)
        return pk_fail(MUCA_ERR_INVALID_ARG, "muca_equal_height: bad sizes");
    if ((int64_t)e_min + n_e - 1 > INT32_MAX)
        return pk_fail(MUCA_ERR_INVALID_ARG, "muca_equal_height: e_min + n_e - 1 exceeds int32");
    if (!(beta > 0.0) || !std::isfinite(beta) || !std::isfinite(delta_lo) ||
        !std::isfinite(delta_hi) || !(delta_lo < delta_hi))
        return pk_fail(MUCA_ERR_INVALID_ARG,
                       "muca_equal_height: need beta > 0 and delta_lo < delta_hi");
    double lnw_max = 0.0;
    for (int e = 0; e < n_e; ++e) {
        if (!std::isfinite(lnW[e]))
            return pk_fail(MUCA_ERR_INVALID_ARG, "muca_equal_height: lnW not finite");
        lnw_max = std::max(lnw_max, std::fabs(lnW[e]));
    }
    // ln P and its prediction from the step before are some ten operations on
    // numbers of this size, of at most half a unit in the last place (2^-53) each
    const double e_max = std::max(std::fabs((double)e_min), std::fabs((double)e_min + n_e));
    const double slack =
        1e-3 + 0x1p-48 * (beta * std::max(std::fabs(delta_lo), std::fabs(delta_hi)) * e_max + lnw_max);
    cudaStream_t st = (cudaStream_t)stream;
    const int n_blocks = n_jack > 0 ? n_jack : 1, n_sets = 1 + n_jack;
    std::vector<int64_t> bnd(n_blocks + 1);
    for (int i = 0; i <= n_blocks; ++i) bnd[i] = (int64_t)i * n_rows / n_blocks;
    auto al = [](size_t x) { return (x + 255) & ~(size_t)255; };
    const size_t b_cnt = al((size_t)n_blocks * n_e * sizeof(unsigned long long));
    const size_t b_lnn = al((size_t)n_sets * n_e * sizeof(double));
    const size_t b_lnw = al((size_t)n_e * sizeof(double));
    const size_t b_bnd = al(bnd.size() * sizeof(int64_t));
    const size_t b_res = al((size_t)5 * n_sets * sizeof(double));
    const size_t b_bad = al((size_t)(n_sets + 1) * sizeof(int));
    char *p = nullptr;
    cudaMemPool_t pool = nullptr;
    const int rp = muca::scratch_pool(muca::ScratchPool::peak, &pool);
    if (rp != MUCA_OK) return rp;
    cudaError_t ce = cudaMallocFromPoolAsync(
        (void **)&p, b_cnt + b_lnn + b_lnw + b_bnd + b_res + b_bad, pool, st);
    if (ce != cudaSuccess)
        return pk_fail(ce == cudaErrorMemoryAllocation ? MUCA_ERR_OOM : MUCA_ERR_CUDA,
                       std::string("cudaMallocAsync: ") + cudaGetErrorString(ce));
    unsigned long long *cnt = (unsigned long long *)p;
    double *lnn = (double *)(p + b_cnt);
    double *d_lnW = (double *)(p + b_cnt + b_lnn);
    int64_t *d_bnd = (int64_t *)(p + b_cnt + b_lnn + b_lnw);
    double *d_res = (double *)(p + b_cnt + b_lnn + b_lnw + b_bnd);
    int *d_bad = (int *)(p + b_cnt + b_lnn + b_lnw + b_bnd + b_res);
    std::vector<double> res(5 * (size_t)n_sets, 0.0);
    std::vector<int> bad(n_sets + 1, 0);
    int rc = MUCA_OK;
#define PCK(call)                                                                         \
    do {                                                                                  \
        ce = (call);                                                                      \
        if (ce != cudaSuccess) {                                                          \
            rc = pk_fail(MUCA_ERR_CUDA, std::string(#call) + ": " + cudaGetErrorString(ce)); \
            goto done;                                                                    \
        }                                                                                 \
    } while (0)
    PCK(cudaMemsetAsync(p, 0, b_cnt, st));
    PCK(cudaMemsetAsync(d_bad, 0, b_bad, st));
    PCK(cudaMemcpyAsync(d_lnW, lnW, (size_t)n_e * sizeof(double), cudaMemcpyHostToDevice, st));
    PCK(cudaMemcpyAsync(d_bnd, bnd.data(), bnd.size() * sizeof(int64_t), cudaMemcpyHostToDevice, st));
    {
        dim3 g((unsigned)std::min<int64_t>((row_len + 255) / 256, 1024),
               (unsigned)std::min<int64_t>(n_rows, 4096));
        jk_bin_kernel<false><<<g, 256, 0, st>>>(e_d, e_d, n_rows, row_len, row_stride, e_min, n_e,
                                                d_bnd, n_blocks, cnt, nullptr, d_bad);
        PCK(cudaGetLastError());
        dim3 g2((unsigned)((n_e + 255) / 256), (unsigned)n_sets);
        jk_lncount_kernel<<<g2, 256, 0, st>>>(cnt, n_blocks, n_e, lnn);
        PCK(cudaGetLastError());
        cudaLaunchConfig_t cfg;
        cudaLaunchAttribute attr[1];
        PCK(cluster_config((const void *)eqh_kernel, n_sets, kPkThreads, 8, st, cfg, attr));
        PCK(cudaLaunchKernelEx(&cfg, eqh_kernel, (const double *)lnn, (const double *)d_lnW,
                               (int)n_e, (int)e_min, (int)split, beta, delta_lo, delta_hi,
                               (int)n_iter, slack, d_res, d_bad + 1));
    }
    PCK(cudaMemcpyAsync(res.data(), d_res, res.size() * sizeof(double), cudaMemcpyDeviceToHost, st));
    PCK(cudaMemcpyAsync(bad.data(), d_bad, bad.size() * sizeof(int), cudaMemcpyDeviceToHost, st));
    PCK(cudaStreamSynchronize(st));
#undef PCK
    if (bad[0]) {
        rc = pk_fail(MUCA_ERR_WINDOW, "a sample's E_Delta lies outside [e_min, e_min + n_e)");
        goto done;
    }
    for (int d = 0; d < n_sets; ++d)
        if (bad[1 + d]) {
            rc = pk_fail(MUCA_ERR_INVALID_ARG,
                         "muca_equal_height: [delta_lo, delta_hi] does not bracket the equal-height "
                         "field for data set " + std::to_string(d) +
                         " (the peak below split must be lower at delta_lo and higher at delta_hi)");
            goto done;
        }
    {
        double err[2] = {0.0, 0.0};
        if (n_jack > 0) {
            for (int q = 0; q < 2; ++q) {
                double mean = 0.0;
                for (int i = 0; i < n_jack; ++i) mean += res[5 * (1 + i) + q];
                mean /= n_jack;
                double ss = 0.0;
                for (int i = 0; i < n_jack; ++i) {
                    const double dv = res[5 * (1 + i) + q] - mean;
                    ss += dv * dv;
                }
                err[q] = std::sqrt((double)(n_jack - 1) / n_jack * ss);
            }
        }
        out[0] = res[0];
        out[1] = err[0];
        out[2] = res[1];
        out[3] = err[1];
        out[4] = res[2];
        out[5] = res[3];
        out[6] = res[4];
        for (int i = 0; i < n_jack; ++i) {
            out[7 + 2 * i] = res[5 * (1 + i)];
            out[8 + 2 * i] = res[5 * (1 + i) + 1];
        }
    }
done:
    cudaFreeAsync(p, st);
    cudaStreamSynchronize(st);
    return rc;
}
