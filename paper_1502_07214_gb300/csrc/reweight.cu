// reweight.cu -- time-series reweighting of a multicanonical run to a grid of
// crystal fields Delta_k (Eq. 3), with C(Delta) from Eq. 6, chi and U4.
//
// The multicanonical weight of a sample depends on the sample only through its
// E_Delta (Eq. 3: exp(-beta Delta E_Delta) / W(E_Delta)).  The GPU path therefore
// works in two stages:
//   A. one streaming pass over the samples accumulates, per E_Delta bin, exact
//      integer sums: count, sum E_J, sum |M|, sum M^2 and sum M^4 (128-bit);
//   B. for every Delta_k, the weighted sums over the occupied bins, the exponents
//      shifted by their maximum; C and chi are taken about the means, or about
//      a bin that holds a good share of the weight, so no difference of large
//      moments is ever formed.
// Stage B runs in FP64 (blocks of bins, wide grids bin by bin), or in FP32 where
// the exponent -beta Delta_k E - lnW(E) is carried as a float pair (hi + lo,
// error-free products and sums) so that its O(10^5) magnitude does not eat the
// 24-bit mantissa, and all sums are Kahan-compensated.
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <mutex>
#include <string>
#include <vector>

#include "../../include/muca.h"
#include "muca_internal.h"

namespace {

int rw_fail(int code, const std::string &msg)
{
    muca::set_last_error(msg.c_str());
    return code;
}

// Integer bin sums of stage A (device scratch).
struct Bins {
    unsigned long long *cnt;   // samples per bin
    unsigned long long *sej;   // sum E_J (two's complement)
    unsigned long long *sam;   // sum |M|
    unsigned long long *sm2;   // sum M^2
    unsigned long long *sm4lo; // sum M^4, low 64 bits
    unsigned long long *sm4hi; // sum M^4, high 64 bits
};

// Per-bin statistics consumed by stage B.
template <typename F>
struct BinStats {
    F *n;    // count
    F *mej;  // mean E_J in the bin
    F *cm;   // mean |m| in the bin, m = M / V
    F *vb;   // sum over the bin of (|m| - cm)^2
    F *q2;   // sum m^2
    F *q4;   // sum m^4
    F *lw;   // lnW (FP64) or its high float (FP32)
    F *lwlo; // FP32 only: lnW - hi
};

// Offset of a sample's E_Delta from the window start, formed in unsigned
// arithmetic so that it is defined for every int32 value; a sample lies in the
// window iff (unsigned)offset < nE (the argument check keeps e_min + nE - 1
// inside int32, so the window does not wrap).
__device__ __forceinline__ int bin_offset(int v, int e_min)
{
    return (int)((unsigned)v - (unsigned)e_min);
}

// Stage A, one sample at a time: every sum of every sample is a 64-bit
// atomic add into the global bin sums; M^4 is a 128-bit sum whose low word's
// returned old value gives the carry into the high word.
__global__ void bin_kernel(const int32_t *__restrict__ ej, const int32_t *__restrict__ ed,
                           const int32_t *__restrict__ m, int64_t n_rows, int row_len,
                           int64_t row_stride, int e_min, int nE, Bins b, int *err)
{
    for (int64_t r = blockIdx.y; r < n_rows; r += gridDim.y) {
        const int64_t base = r * row_stride;
        for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < row_len;
             c += gridDim.x * blockDim.x) {
            const int64_t o = base + c;
            const int e = bin_offset(__ldg(ed + o), e_min);
            if ((unsigned)e >= (unsigned)nE) {
                atomicOr(err, 1);
                continue;
            }
            const long long j = __ldg(ej + o);
            const long long mm = __ldg(m + o);
            const unsigned long long am = (unsigned long long)(mm < 0 ? -mm : mm);
            const unsigned long long m2 = am * am;
            const unsigned long long m4lo = m2 * m2, m4hi = __umul64hi(m2, m2);
            atomicAdd(b.cnt + e, 1ull);
            atomicAdd(b.sej + e, (unsigned long long)j);
            atomicAdd(b.sam + e, am);
            atomicAdd(b.sm2 + e, m2);
            const unsigned long long old = atomicAdd(b.sm4lo + e, m4lo);
            const unsigned long long carry = (old + m4lo < old) ? 1ull : 0ull;
            if (m4hi + carry) atomicAdd(b.sm4hi + e, m4hi + carry);
        }
    }
}

// ------------------------------------------------- stage A through buckets
// The same integer bin sums, formed without one global atomic per sample and
// without one shared atomic per sum.  Bins are grouped into buckets of kBkt
// consecutive bins.  Four launches per pass:
//   1. count: each block counts its samples per bucket and writes one counter
//      per (bucket, block);
//   2. scan: one block gives every (bucket, block) segment two places: where
//      its records are stored (block-major: a block's records of every bucket
//      in one region, so that a block writes to one neighbourhood of memory)
//      and where they stand in bucket order (bucket-major), the order the sums
//      walk in;
//   3. scatter: each block re-reads the same samples, takes places from its
//      own shared cursors and writes 8-byte records;
//   4. sums: each block takes an equal share of the records in bucket order,
//      gathering a bucket's segments through a table in shared memory,
//      counting-sorts tiles of them by bin in shared memory (one 32-bit shared
//      atomic per record), and every thread sums the run of its own bin in
//      registers; a bucket's sums go to the global bins once per block.
// A record holds the bin offset, E_J (|E_J| < 2^20) and |M| (<= 2^18, so
// M^4 <= 2^72); a sample outside those ranges is added straight to the global
// sums instead and leaves a null record.  Every sum stays an exact integer, so
// the result does not depend on the order in which records are summed.
constexpr int kBktBits = 10;
constexpr int kBkt = 1 << kBktBits;
constexpr unsigned kNullRec = 0xFFFFFFFFu;
constexpr int kMaxBk = 1024;      // buckets of the bucketed path (n_e <= 2^20)
constexpr int kMaxG = 1024;       // blocks of the count and scatter launches
constexpr int kCsThreads = 1024;  // threads of a count or scatter block
constexpr int kCsPer = 4;         // samples per thread and chunk
constexpr int kChunk = kCsThreads * kCsPer;  // samples of one row per chunk

__device__ __forceinline__ void direct_add(const Bins &b, int e, long long j, unsigned long long am)
{
    const unsigned long long m2 = am * am;
    const unsigned long long m4lo = m2 * m2, m4hi = __umul64hi(m2, m2);
    atomicAdd(b.cnt + e, 1ull);
    atomicAdd(b.sej + e, (unsigned long long)j);
    atomicAdd(b.sam + e, am);
    atomicAdd(b.sm2 + e, m2);
    const unsigned long long old = atomicAdd(b.sm4lo + e, m4lo);
    const unsigned long long carry = (old + m4lo < old) ? 1ull : 0ull;
    if (m4hi + carry) atomicAdd(b.sm4hi + e, m4hi + carry);
}

__device__ __forceinline__ unsigned warp_incl_scan(unsigned v)
{
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const unsigned u = __shfl_up_sync(0xffffffffu, v, d);
        if (lane >= d) v += u;
    }
    return v;
}

// Chunks of one block: chunk t is columns [(t % cpr) kChunk, + kChunk) of row
// t / cpr, and block i takes chunks [n i / G, n (i+1) / G) of the n = rows x
// cpr chunks.  The count and scatter launches share this partition; a block
// walks its chunks as (row, chunk of the row) without dividing per chunk.
struct ChunkWalk {
    int64_t t, t1, row;
    int ci;
    __device__ __forceinline__ ChunkWalk(int64_t n_rows, int cpr)
    {
        const int64_t n = n_rows * cpr;
        t = n * blockIdx.x / gridDim.x;
        t1 = n * (blockIdx.x + 1) / gridDim.x;
        row = t / cpr;
        ci = (int)(t - row * cpr);
    }
    __device__ __forceinline__ void next(int cpr)
    {
        ++t;
        if (++ci == cpr) {
            ci = 0;
            ++row;
        }
    }
};

// This thread's kCsPer values of one column in columns [col0, col0 + kChunk)
// of a row (0 past the row's end).
__device__ __forceinline__ void load_chunk(const int32_t *__restrict__ row, int col0, int row_len,
                                           int (&v)[kCsPer])
{
#pragma unroll
    for (int q = 0; q < kCsPer; ++q) {
        const int c = col0 + q * kCsThreads + threadIdx.x;
        v[q] = c < row_len ? __ldg(row + c) : 0;
    }
}

// Samples per (bucket, block), written to cnt[bucket * gridDim.x + block];
// flags a sample outside [e_min, e_min + nE).
__global__ void __launch_bounds__(kCsThreads)
bucket_count_kernel(const int32_t *__restrict__ ed, int64_t n_rows, int row_len,
                    int64_t row_stride, int e_min, int nE, int nbk, int cpr,
                    unsigned *__restrict__ cnt, int *err)
{
    __shared__ unsigned sc[kMaxBk];
    for (int i = threadIdx.x; i < nbk; i += blockDim.x) sc[i] = 0u;
    __syncthreads();
    // two chunks per step, so that twice the loads are in flight
    for (ChunkWalk w(n_rows, cpr); w.t < w.t1;) {
        int col[2];
        int v[2][kCsPer];
        col[0] = w.ci * kChunk;
        load_chunk(ed + w.row * row_stride, col[0], row_len, v[0]);
        w.next(cpr);
        const bool two = w.t < w.t1;
        col[1] = two ? w.ci * kChunk : row_len;
        if (two) {
            load_chunk(ed + w.row * row_stride, col[1], row_len, v[1]);
            w.next(cpr);
        }
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int q = 0; q < kCsPer; ++q) {
                const int c = col[h] + q * kCsThreads + threadIdx.x;
                const int e = bin_offset(v[h][q], e_min);
                const bool in = c < row_len, ok = in && (unsigned)e < (unsigned)nE;
                if (in && !ok) atomicOr(err, 1);
                if (ok) atomicAdd(&sc[(unsigned)e >> kBktBits], 1u);
            }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < nbk; i += blockDim.x) cnt[(size_t)i * gridDim.x + blockIdx.x] = sc[i];
}

// One block of 1024 threads.  In: cnt[k * g + b], the samples of bucket k in
// count block b (g <= 1024 blocks).  Out: lst[k * g + b], the segment's first
// place in bucket order; cnt[k * g + b] (in place), its first place in the
// record buffer (block b's segments of buckets 0, 1, ... one after another,
// after those of blocks 0 .. b-1); bstart / bcnt, each bucket's first place in
// bucket order and its size.
__global__ void __launch_bounds__(1024)
bucket_scan_kernel(unsigned *cnt, unsigned *lst, int nbk, int g, unsigned *bstart, unsigned *bcnt)
{
    __shared__ unsigned tot[kMaxBk];
    __shared__ unsigned ws[32];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int k = w; k < nbk; k += 32) {
        unsigned s = 0u;
        for (int b = lane; b < g; b += 32) s += cnt[(size_t)k * g + b];
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) s += __shfl_xor_sync(0xffffffffu, s, d);
        if (lane == 0) tot[k] = s;
    }
    __syncthreads();
    // bucket order: exclusive scan of the bucket totals
    {
        const unsigned v = (int)threadIdx.x < nbk ? tot[threadIdx.x] : 0u;
        const unsigned incl = warp_incl_scan(v);
        if (lane == 31) ws[w] = incl;
        __syncthreads();
        const unsigned wv = ws[lane];
        const unsigned wi = warp_incl_scan(wv);
        const unsigned wex = __shfl_sync(0xffffffffu, wi - wv, w);
        __syncthreads();
        if ((int)threadIdx.x < nbk) {
            tot[threadIdx.x] = wex + incl - v;
            bstart[threadIdx.x] = wex + incl - v;
            bcnt[threadIdx.x] = v;
        }
        __syncthreads();
    }
    for (int k = w; k < nbk; k += 32) {
        unsigned run = tot[k];
        for (int b0 = 0; b0 < g; b0 += 32) {
            const int b = b0 + lane;
            const unsigned x = b < g ? cnt[(size_t)k * g + b] : 0u;
            const unsigned xi = warp_incl_scan(x);
            if (b < g) lst[(size_t)k * g + b] = run + xi - x;
            run += __shfl_sync(0xffffffffu, xi, 31);
        }
    }
    // storage order: thread b sums its block's counts, scans them over the
    // blocks, then lays its segments out bucket after bucket
    const int b = threadIdx.x;
    unsigned bt = 0u;
    if (b < g)
        for (int k = 0; k < nbk; ++k) bt += cnt[(size_t)k * g + b];
    const unsigned incl = warp_incl_scan(bt);
    if (lane == 31) ws[w] = incl;
    __syncthreads();
    const unsigned wv = ws[lane];
    const unsigned wi = warp_incl_scan(wv);
    unsigned run = __shfl_sync(0xffffffffu, wi - wv, w) + incl - bt;
    if (b < g)
        for (int k = 0; k < nbk; ++k) {
            const unsigned x = cnt[(size_t)k * g + b];
            cnt[(size_t)k * g + b] = run;
            run += x;
        }
}

// Records: the block's samples of bucket k take places off[k * gridDim.x +
// block], +1, ... (the scan's storage places), handed out by shared cursors.
// A record is
// (bin offset in its bucket | (E_J + 2^20) << kBktBits, |M|).
__global__ void __launch_bounds__(kCsThreads)
bucket_scatter_kernel(const int32_t *__restrict__ ej, const int32_t *__restrict__ ed,
                      const int32_t *__restrict__ m, int64_t n_rows, int row_len,
                      int64_t row_stride, int e_min, int nE, int nbk, int cpr,
                      const unsigned *__restrict__ off, uint2 *__restrict__ rec, Bins b)
{
    __shared__ unsigned cur[kMaxBk];
    for (int i = threadIdx.x; i < nbk; i += blockDim.x)
        cur[i] = off[(size_t)i * gridDim.x + blockIdx.x];
    __syncthreads();
    for (ChunkWalk w(n_rows, cpr); w.t < w.t1; w.next(cpr)) {
        const int col0 = w.ci * kChunk;
        const int64_t base = w.row * row_stride;
        int vd[kCsPer], vj[kCsPer], vm[kCsPer];
        load_chunk(ed + base, col0, row_len, vd);
        load_chunk(ej + base, col0, row_len, vj);
        load_chunk(m + base, col0, row_len, vm);
#pragma unroll
        for (int q = 0; q < kCsPer; ++q) {
            const int c = col0 + q * kCsThreads + threadIdx.x;
            const int e = bin_offset(vd[q], e_min);
            const bool ok = c < row_len && (unsigned)e < (unsigned)nE;
            if (!ok) continue;
            const unsigned pos = atomicAdd(&cur[(unsigned)e >> kBktBits], 1u);
            const int j = vj[q], mm = vm[q];
            const unsigned am = mm < 0 ? 0u - (unsigned)mm : (unsigned)mm;
            uint2 rr;
            if (j > -(1 << 20) && j < (1 << 20) && am <= (1u << 18)) {
                rr.x = ((unsigned)e & (kBkt - 1)) | ((unsigned)(j + (1 << 20)) << kBktBits);
                rr.y = am;
            } else {
                direct_add(b, e, j, am);
                rr.x = 0u;
                rr.y = kNullRec;
            }
            rec[pos] = rr;
        }
    }
}

// Stage A sums.  Block i takes places [total i / G, total (i+1) / G) of
// bucket order; within each bucket it gathers tiles of kHS records through the
// bucket's segment table (place in bucket order -> place in the buffer), sorts
// each tile by bin in shared memory, and thread t sums bin t of the bucket in
// registers (count, E_J + 2^20, |M|, M^2 and M^4), which go to the global sums
// at the end of the bucket.  The sort buffers are double buffered, so a tile
// needs four barriers.
constexpr int kHT = kBkt;
constexpr int kHS = 8192;
constexpr int kHRpt = kHS / kHT;
constexpr size_t kHistSmem = 2 * (size_t)kHS * sizeof(uint2) + 3 * (size_t)kBkt * sizeof(unsigned) +
                             32 * sizeof(unsigned) + (2 * (size_t)kMaxG + 1) * sizeof(unsigned);

// Sums of one bin.  M^4 is kept as three 64-bit sums of 36-bit products: with
// M^2 = h 2^18 + l (h, l < 2^18), M^4 = h^2 2^36 + 2 h l 2^18 + l^2, exact for
// up to 2^28 records; the 128-bit value is formed once, at the flush.
struct BinAcc {
    unsigned n = 0u;
    unsigned long long j = 0ull, a = 0ull, q = 0ull, s0 = 0ull, s1 = 0ull, s2 = 0ull;
    __device__ __forceinline__ void add(uint2 r)
    {
        const unsigned am = r.y;
        const unsigned long long m2 = (unsigned long long)am * am;
        const unsigned h = (unsigned)(m2 >> 18), l = (unsigned)m2 & 0x3FFFFu;
        n += 1u;
        j += r.x >> kBktBits;
        a += am;
        q += m2;
        s0 += (unsigned long long)l * l;
        s1 += (unsigned long long)h * l;
        s2 += (unsigned long long)h * h;
    }
    __device__ __forceinline__ void flush(const Bins &b, int e)
    {
        if (!n) return;
        atomicAdd(b.cnt + e, (unsigned long long)n);
        atomicAdd(b.sej + e, j - ((unsigned long long)n << 20));
        atomicAdd(b.sam + e, a);
        atomicAdd(b.sm2 + e, q);
        const unsigned __int128 m4 = ((unsigned __int128)s2 << 36) + ((unsigned __int128)s1 << 19) + s0;
        const unsigned long long lo = (unsigned long long)m4, hi = (unsigned long long)(m4 >> 64);
        const unsigned long long old = atomicAdd(b.sm4lo + e, lo);
        const unsigned long long carry = (old + lo < old) ? 1ull : 0ull;
        if (hi + carry) atomicAdd(b.sm4hi + e, hi + carry);
        n = 0u;
        j = a = q = s0 = s1 = s2 = 0ull;
    }
};

__global__ void __launch_bounds__(kHT, 1)
bucket_hist_kernel(const uint2 *__restrict__ rec, const unsigned *__restrict__ pst,
                   const unsigned *__restrict__ lst, int g, const unsigned *__restrict__ bstart,
                   const unsigned *__restrict__ bcnt, int nbk, unsigned total, Bins b)
{
    extern __shared__ __align__(16) unsigned char hsm[];
    uint2 *srt0 = (uint2 *)hsm;                                  // [2][kHS]
    unsigned *scnt0 = (unsigned *)(hsm + 2 * kHS * sizeof(uint2)); // [2][kBkt]
    unsigned *soff = scnt0 + 2 * kBkt;                           // [kBkt]
    unsigned *wsum = soff + kBkt;                                // [32]
    unsigned *segL = wsum + 32;                                  // [g + 1] bucket order
    unsigned *segP = segL + kMaxG + 1;                           // [g] buffer
    const unsigned lo = (unsigned)((unsigned long long)total * blockIdx.x / gridDim.x);
    const unsigned hi = (unsigned)((unsigned long long)total * (blockIdx.x + 1) / gridDim.x);
    if (lo >= hi) return;
    const int tid = threadIdx.x, w = tid >> 5, lane = tid & 31;
    for (int i = tid; i < 2 * kBkt; i += kHT) scnt0[i] = 0u;
    int k = 0;
    while (k < nbk && bstart[k] + bcnt[k] <= lo) ++k;
    BinAcc acc;
    int buf = 0;
    for (; k < nbk && bstart[k] < hi; ++k) {
        const unsigned s_lo = max(lo, bstart[k]), s_hi = min(hi, bstart[k] + bcnt[k]);
        // the bucket's segment table (the previous bucket's last reads are done)
        __syncthreads();
        for (int i = tid; i < g; i += kHT) {
            segL[i] = lst[(size_t)k * g + i];
            segP[i] = pst[(size_t)k * g + i];
        }
        if (tid == 0) segL[g] = bstart[k] + bcnt[k];
        __syncthreads();
        // record j of the tile at s0: place s0 + j kHT + tid in bucket order,
        // in segment sg (segL[sg] <= place < segL[sg + 1]); places only grow
        // (the segment's end in bucket order and its buffer offset are kept in
        // registers; unsigned wrap-around makes i + dlt the buffer place)
        int sg = 0;
        unsigned send = segL[1], dlt = segP[0] - segL[0];
        auto load = [&](unsigned s0, uint2 (&r)[kHRpt]) {
#pragma unroll
            for (int q = 0; q < kHRpt; ++q) {
                const unsigned i = s0 + q * kHT + tid;
                if (i < s_hi) {
                    while (send <= i) {
                        ++sg;
                        send = segL[sg + 1];
                        dlt = segP[sg] - segL[sg];
                    }
                    r[q] = rec[i + dlt];
                } else {
                    r[q] = make_uint2(0u, kNullRec);
                }
            }
        };
        uint2 r[kHRpt];
        load(s_lo, r);
        for (unsigned s0 = s_lo; s0 < s_hi; s0 += kHS) {
            unsigned *scnt = scnt0 + buf * kBkt;
            uint2 *srt = srt0 + buf * kHS;
            unsigned rk[kHRpt];
#pragma unroll
            for (int q = 0; q < kHRpt; ++q)
                rk[q] = r[q].y != kNullRec ? atomicAdd(&scnt[r[q].x & (kBkt - 1)], 1u) : 0u;
            __syncthreads();
            const unsigned c = scnt[tid];
            const unsigned incl = warp_incl_scan(c);
            if (lane == 31) wsum[w] = incl;
            __syncthreads();
            const unsigned wv = wsum[lane];
            const unsigned wi = warp_incl_scan(wv);
            const unsigned o = __shfl_sync(0xffffffffu, wi - wv, w) + incl - c;
            soff[tid] = o;
            __syncthreads();
#pragma unroll
            for (int q = 0; q < kHRpt; ++q)
                if (r[q].y != kNullRec) srt[soff[r[q].x & (kBkt - 1)] + rk[q]] = r[q];
            // the next tile's records, loaded while this tile is summed
            load(s0 + kHS, r);
            __syncthreads();
            unsigned i = o;
            for (; i + 1 < o + c; i += 2) {
                const uint2 x = srt[i], y = srt[i + 1];
                acc.add(x);
                acc.add(y);
            }
            if (i < o + c) acc.add(srt[i]);
            scnt[tid] = 0u;
            buf ^= 1;
        }
        acc.flush(b, k * kBkt + tid);
    }
}

__device__ __forceinline__ double u128_to_double(unsigned long long hi, unsigned long long lo)
{
    return (double)hi * 18446744073709551616.0 + (double)lo;
}

__device__ __forceinline__ float u128_to_float(unsigned long long hi, unsigned long long lo)
{
    return (float)hi * 18446744073709551616.0f + (float)lo;
}

// Stage A2: integer sums -> per-bin statistics.  vb uses the exact integer
// n sum M^2 - (sum |M|)^2 (128-bit) before any rounding.
__global__ void stats_kernel_f64(Bins b, int nE, int V, const double *__restrict__ lnW,
                                 BinStats<double> s)
{
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= nE) return;
    const unsigned long long n = b.cnt[e];
    s.lw[e] = lnW[e];
    if (n == 0) {
        s.n[e] = 0;
        return;
    }
    const double dn = (double)n, dV = (double)V;
    const long long sej = (long long)b.sej[e];
    const unsigned long long sam = b.sam[e], sm2 = b.sm2[e];
    const unsigned __int128 a = (unsigned __int128)n * sm2;
    const unsigned __int128 c = (unsigned __int128)sam * sam;
    const unsigned __int128 v = a - c;
    s.n[e] = dn;
    s.mej[e] = (double)sej / dn;
    s.cm[e] = (double)sam / dn / dV;
    s.vb[e] = u128_to_double((unsigned long long)(v >> 64), (unsigned long long)v) / dn / dV / dV;
    s.q2[e] = (double)sm2 / dV / dV;
    s.q4[e] = u128_to_double(b.sm4hi[e], b.sm4lo[e]) / dV / dV / dV / dV;
}

__global__ void stats_kernel_f32(Bins b, int nE, int V, const double *__restrict__ lnW,
                                 BinStats<float> s)
{
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= nE) return;
    const unsigned long long n = b.cnt[e];
    // lnW as a float pair (hi + lo)
    s.lw[e] = (float)lnW[e];
    s.lwlo[e] = (float)(lnW[e] - (double)s.lw[e]);
    if (n == 0) {
        s.n[e] = 0.f;
        return;
    }
    const float fn = (float)n, fV = (float)V;
    const long long sej = (long long)b.sej[e];
    const unsigned long long sam = b.sam[e], sm2 = b.sm2[e];
    const unsigned __int128 a = (unsigned __int128)n * sm2;
    const unsigned __int128 c = (unsigned __int128)sam * sam;
    const unsigned __int128 v = a - c;
    s.n[e] = fn;
    s.mej[e] = (float)sej / fn;
    s.cm[e] = (float)sam / fn / fV;
    s.vb[e] = u128_to_float((unsigned long long)(v >> 64), (unsigned long long)v) / fn / fV / fV;
    s.q2[e] = (float)sm2 / fV / fV;
    s.q4[e] = u128_to_float(b.sm4hi[e], b.sm4lo[e]) / fV / fV / fV / fV;
}

// ---------------------------------------------------------------- reductions
template <typename F>
struct KSum {  // Kahan-compensated accumulator
    F s, c;
    __device__ void init() { s = c = F(0); }
    __device__ void add(F x)
    {
        const F y = x - c;
        const F t = s + y;
        c = (t - s) - y;
        s = t;
    }
};

template <typename F>
__device__ __forceinline__ F block_max(F v, F *sh)
{
    for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xFFFFFFFFu, v, o));
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    __syncthreads();
    if (lane == 0) sh[wid] = v;
    __syncthreads();
    F r = sh[0];
    for (int i = 1; i < nw; ++i) r = fmax(r, sh[i]);
    return r;
}

// Sum of K compensated accumulators over the block; every thread gets the sums.
template <typename F, int K>
__device__ __forceinline__ void block_sum(KSum<F> (&a)[K], F (&out)[K], F *sh)
{
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
#pragma unroll
    for (int k = 0; k < K; ++k) {
        F s = a[k].s, c = -a[k].c;
        for (int o = 16; o > 0; o >>= 1) {
            const F s2 = __shfl_xor_sync(0xFFFFFFFFu, s, o);
            const F c2 = __shfl_xor_sync(0xFFFFFFFFu, c, o);
            // two-sum of s and s2 keeps the rounding error in c
            const F t = s + s2;
            const F bp = t - s;
            const F err = (s - (t - bp)) + (s2 - bp);
            s = t;
            c = c + c2 + err;
        }
        __syncthreads();
        if (lane == 0) {
            sh[2 * wid] = s;
            sh[2 * wid + 1] = c;
        }
        __syncthreads();
        KSum<F> tot;
        tot.init();
        F cc = F(0);
        for (int i = 0; i < nw; ++i) {
            tot.add(sh[2 * i]);
            cc += sh[2 * i + 1];
        }
        out[k] = tot.s + (cc - tot.c);
    }
}

// Block-wide argmax of (value, bin); ties go to the smaller bin.
__device__ __forceinline__ void block_argmax(double &v, int &e, double *shv, int *she)
{
    for (int o = 16; o > 0; o >>= 1) {
        const double v2 = __shfl_xor_sync(0xFFFFFFFFu, v, o);
        const int e2 = __shfl_xor_sync(0xFFFFFFFFu, e, o);
        if (v2 > v || (v2 == v && e2 < e)) {
            v = v2;
            e = e2;
        }
    }
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    __syncthreads();
    if (lane == 0) {
        shv[wid] = v;
        she[wid] = e;
    }
    __syncthreads();
    v = shv[0];
    e = she[0];
    for (int i = 1; i < nw; ++i)
        if (shv[i] > v || (shv[i] == v && she[i] < e)) {
            v = shv[i];
            e = she[i];
        }
}

// ------------------------------------------------------------ FP32 stage B
// a = -(c_hi + c_lo) E - (lw_hi + lw_lo) as an unevaluated float pair.
struct F2 {
    float hi, lo;
};

__device__ __forceinline__ F2 expo32(float chi, float clo, int E, float lwh, float lwl)
{
    const float fe = (float)E;                  // exact: E < 2^24
    // the _rn intrinsics keep the compiler from fusing the error-free steps
    const float p = __fmul_rn(chi, fe);         // two-product: p + pe = chi E exactly
    const float pe = fmaf(chi, fe, -p);
    const float s = __fsub_rn(-p, lwh);         // two-sum of -p and -lwh
    const float bp = __fadd_rn(s, p);
    const float se = __fadd_rn(__fsub_rn(-p, __fsub_rn(s, bp)), __fsub_rn(-lwh, bp));
    const float lo = se - pe - fmaf(clo, fe, lwl);
    return {s, lo};
}

// One block serves kGridD consecutive Delta points, so that every bin's
// statistics are read once per kGridD points; per point, the arithmetic and the
// order of every sum are those of a block serving that point alone.
constexpr int kGridD = 4;

template <int D>
__global__ void __launch_bounds__(256, 4)  // four blocks per SM: more warps hide the latencies
grid_kernel_f32(BinStats<float> s, int nE, int e_min, float beta, int V,
                const double *__restrict__ cgrid, int n_grid, double *__restrict__ out)
{
    __shared__ float sh[64];
    const int k0 = blockIdx.x * D;
    float ch[D], cl[D], amax[D];
#pragma unroll
    for (int d = 0; d < D; ++d) {
        const int k = min(k0 + d, n_grid - 1);
        ch[d] = (float)cgrid[k];
        cl[d] = (float)(cgrid[k] - (double)ch[d]);
        amax[d] = -INFINITY;
    }
    for (int e = threadIdx.x; e < nE; e += blockDim.x)
        if (s.n[e] > 0.f) {
            const float lh = s.lw[e], ll = s.lwlo[e];
#pragma unroll
            for (int d = 0; d < D; ++d)
                amax[d] = fmaxf(amax[d], expo32(ch[d], cl[d], e_min + e, lh, ll).hi);
        }
#pragma unroll
    for (int d = 0; d < D; ++d) amax[d] = block_max(amax[d], sh);
    KSum<float> acc[D][6];
#pragma unroll
    for (int d = 0; d < D; ++d)
#pragma unroll
        for (int i = 0; i < 6; ++i) acc[d][i].init();
    for (int e = threadIdx.x; e < nE; e += blockDim.x) {
        const float n = s.n[e];
        if (n <= 0.f) continue;
        const float lh = s.lw[e], ll = s.lwlo[e], mej = s.mej[e], cm = s.cm[e], q2 = s.q2[e],
                    q4 = s.q4[e];
        const float fe = (float)(e_min + e);
#pragma unroll
        for (int d = 0; d < D; ++d) {
            const F2 a = expo32(ch[d], cl[d], e_min + e, lh, ll);
            const float x = (a.hi - amax[d]) + a.lo;
            if (x < -104.f) continue;
            const float w = expf(x);
            const float wn = w * n;
            acc[d][0].add(wn);
            acc[d][1].add(wn * fe);
            acc[d][2].add(wn * mej);
            acc[d][3].add(wn * cm);
            acc[d][4].add(w * q2);
            acc[d][5].add(w * q4);
        }
    }
    float Z[D], mE[D], mJ[D], mu[D], m2[D], m4[D];
#pragma unroll
    for (int d = 0; d < D; ++d) {
        float S[6];
        block_sum<float, 6>(acc[d], S, sh);
        Z[d] = S[0];
        mE[d] = S[1] / Z[d];
        mJ[d] = S[2] / Z[d];
        mu[d] = S[3] / Z[d];
        m2[d] = S[4] / Z[d];
        m4[d] = S[5] / Z[d];
    }
    KSum<float> acc2[D][2];
#pragma unroll
    for (int d = 0; d < D; ++d) {
        acc2[d][0].init();
        acc2[d][1].init();
    }
    for (int e = threadIdx.x; e < nE; e += blockDim.x) {
        const float n = s.n[e];
        if (n <= 0.f) continue;
        const float lh = s.lw[e], ll = s.lwlo[e], mej = s.mej[e], cm = s.cm[e], vb = s.vb[e];
        const float fe = (float)(e_min + e);
#pragma unroll
        for (int d = 0; d < D; ++d) {
            const F2 a = expo32(ch[d], cl[d], e_min + e, lh, ll);
            const float x = (a.hi - amax[d]) + a.lo;
            if (x < -104.f) continue;
            const float w = expf(x);
            const float wn = w * n;
            acc2[d][0].add(wn * ((mej - mJ[d]) * (fe - mE[d])));
            const float dm = cm - mu[d];
            acc2[d][1].add(w * vb + wn * (dm * dm));
        }
    }
#pragma unroll
    for (int d = 0; d < D; ++d) {
        float S2[2];
        block_sum<float, 2>(acc2[d], S2, sh);
        if (threadIdx.x == 0 && k0 + d < n_grid) {
            double *o = out + 5 * (int64_t)(k0 + d);
            o[0] = mJ[d];
            o[1] = mE[d];
            o[2] = -beta * (S2[0] / Z[d]);
            o[3] = beta * (float)V * (S2[1] / Z[d]);
            o[4] = 1.f - m4[d] / (3.f * m2[d] * m2[d]);
        }
    }
}

constexpr int kStats = 8;

// Sums of K values over the block (of NW warps if given); every thread gets them.
template <int K, int NW = 0>
__device__ __forceinline__ void block_sum_plain(double (&v)[K], double *sh)
{
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = NW ? NW : blockDim.x >> 5;
#pragma unroll
    for (int k = 0; k < K; ++k)
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v[k] += __shfl_xor_sync(0xFFFFFFFFu, v[k], o);
    __syncthreads();
    if (lane == 0)
#pragma unroll
        for (int k = 0; k < K; ++k) sh[wid * K + k] = v[k];
    __syncthreads();
#pragma unroll
    for (int k = 0; k < K; ++k) {
        double a = sh[k];
        for (int i = 1; i < nw; ++i) a += sh[i * K + k];
        v[k] = a;
    }
}

// C, chi and the means of one field from its sums T about the reference bin's or
// block's (E0, J0, M0): weight, E, E_J, |m|, m^2, m^4, (E_J - J0)(E - E0), the
// variance of |m| about M0.
__device__ __forceinline__ void put_field(const double (&T)[kStats], int E0, double J0, double M0,
                                          double beta, int V, double *o)
{
    const double Z = T[0], mE = T[1] / Z, mJ = T[2] / Z, mu = T[3] / Z;
    const double m2 = T[4] / Z, m4 = T[5] / Z;
    o[0] = J0 + mJ;
    o[1] = (double)E0 + mE;
    o[2] = -beta * (T[6] / Z - mE * mJ);
    o[3] = beta * (double)V * (T[7] / Z - mu * mu);
    o[4] = 1.0 - m4 / (3.0 * m2 * m2);
}

// ------------------------------------------- FP64 stage B, bin by bin
// Grids that are too wide for blocks of bins (below), one field per CTA.  The
// sums are taken about the field's heaviest bin (to the precision of an FP32
// logarithm of its samples: any bin near it serves), which holds at least
// 1 / n_e of the weight or so; so one pass gives the centred sums too.
// Exponents are formed as -c (E - E0) - (lnW(E) - lnW(E0)), c = beta Delta_k,
// so that two O(beta Delta V) numbers are never subtracted.  Each thread adds up
// 32 bins at a time, and those sums.
//   4096 fields, beta = 0.7, half width 1, 6.4e5 samples: 4097 bins 1.47 ms a call,
//   32769 bins 5.0, 262145 bins 29.4 (three passes of compensated sums: 3.6, 8.9,
//   41.1; polynomials over blocks of one bin: 2.1, 15.1, 102)
__global__ void __launch_bounds__(512)
grid_kernel_f64(BinStats<double> s, int nE, int e_min, double beta, int V,
                const double *__restrict__ cgrid, double *__restrict__ out)
{
    __shared__ double shv[32];
    __shared__ int she[32];
    __shared__ double sh[16 * kStats];
    const double c = cgrid[blockIdx.x];
    double best = -INFINITY;
    int at = 0x7FFFFFFF;
#pragma unroll 4
    for (int e = threadIdx.x; e < nE; e += blockDim.x) {
        const double n = s.n[e], lw = s.lw[e];
        if (n > 0.0) {
            const double a = (-(c * (double)(e_min + e)) - lw) + (double)__logf((float)n);
            if (a > best) {
                best = a;
                at = e;
            }
        }
    }
    block_argmax(best, at, shv, she);
    if (at >= nE) at = 0;  // no sample lies in the window (the call fails)
    const double l0 = s.lw[at], J0 = s.mej[at], M0 = s.cm[at];
    double T[kStats];
#pragma unroll
    for (int j = 0; j < kStats; ++j) T[j] = 0.0;
    for (int e0 = threadIdx.x; e0 < nE; e0 += 32 * blockDim.x) {
        double S[kStats];
#pragma unroll
        for (int j = 0; j < kStats; ++j) S[j] = 0.0;
        const int e1 = min(nE, e0 + 32 * (int)blockDim.x);
#pragma unroll 4
        for (int e = e0; e < e1; e += blockDim.x) {
            const double n = s.n[e], lw = s.lw[e];
            if (!(n > 0.0)) continue;
            const double dE = (double)(e - at), d = __dsub_rn(-__dmul_rn(c, dE), __dsub_rn(lw, l0));
            if (d < -800.0) continue;
            const double w = exp(d), wn = w * n;
            const double dJ = s.mej[e] - J0, dM = s.cm[e] - M0, wj = wn * dJ, wm = wn * dM;
            S[0] += wn;
            S[1] = fma(wn, dE, S[1]);
            S[2] += wj;
            S[3] += wm;
            S[4] = fma(w, s.q2[e], S[4]);
            S[5] = fma(w, s.q4[e], S[5]);
            S[6] = fma(wj, dE, S[6]);
            S[7] += fma(w, s.vb[e], wm * dM);
        }
#pragma unroll
        for (int j = 0; j < kStats; ++j) T[j] += S[j];
    }
    block_sum_plain<kStats>(T, sh);
    if (threadIdx.x == 0) put_field(T, e_min + at, J0, M0, beta, V, out + 5 * (int64_t)blockIdx.x);
}

// ------------------------------------------- FP64 stage B, blocks of bins
// The weight of Eq. 3 factorises over a block of B consecutive bins: with
// E_b the block's heaviest bin (the largest n exp(-s E - lnW), s a slope common
// to the grid) and r = E - E_b,
//   exp(-c E - lnW(E)) = A(c, b) exp(-(c - s) (E - E_mid)) V(E),   c = beta Delta_k,
//   A = exp(-c E_b - lnW(E_b) - (c - s) (E_mid - E_b)),
//   V = exp(-s r - (lnW(E) - lnW(E_b))).
// V does not depend on the field, and |c - s| B / 2 is small for a grid of
// fields around a transition.  So the middle factor is its Taylor polynomial in
// x = -(c - s) B / 2 (E_mid: the block's middle), and each weighted sum over
// the block is a polynomial in x whose coefficients sum
// V f(E) (2 (E - E_mid) / B)^p / p! over the block once per call: one
// exponential and 8 deg multiply-adds per (field, block).  FP64 runs at two
// multiply-adds per clock and SM here, so FP64 instructions are the time: bin
// by bin, with two exponentials and eight compensated sums, they were about a
// hundred per (field, bin); in blocks of 64 bins they are four.
// The exponent of A is formed with error-free products and differences.  Sums
// are taken about bins that hold weight, so that no difference of large moments
// is formed, however narrow the distribution: inside a block about its heaviest
// bin and its weighted mean E_J and |m|, across blocks about the heaviest
// block's of the field.  (A reference that holds a share p of the weight lies
// within 1 / sqrt(p) standard deviations of the mean.)
//   C of a distribution pinned at one end of E_Delta (weights -ln of the binomial
//   density of states, beta Delta = -25 .. 25) against binary128: within 7e-15,
//   as with compensated sums about the mean; about the blocks' middle bins and
//   the first blocks that count it was up to 1e-4
//   4.1e7 samples, 32769 bins, 4096 fields: 21.8 -> 1.69 ms per call (bin by bin,
//   then this), of which stage A 0.42, the coefficients 0.03, the fields 1.0 ms
// FP32 keeps one evaluation per bin: its pipe is 64 times wider, and sums about
// a block's reference bin cost the covariance of a narrow distribution a
// decimal digit that FP32 does not have to spare (3e-5 to 5e-5 where 1e-5 is
// asked, on a rough 262145-bin window).
constexpr int kDegMax = 20;
constexpr int kRgThreads = 128;
constexpr double kXMax = 1.2;

struct BlockPlan {
    int B, nblk, per, deg;  // bins per block, blocks, blocks per thread, degree
    double slope;           // s
};

// Block size and degree for fields c in [lo, hi].  |x| <= 1.2 keeps the
// polynomial's alternating terms within e^2.4 of their sum.  The degree is the
// first whose remainder |x|^(deg+1) / (deg+1)! is below a sixteenth of the
// rounding.  B = 0: the grid is too wide for blocks, its fields go bin by bin.
// The smallest block is 8 bins, beyond 2^17 bins 16: 4096 fields of half width
// 0.42 (beta = 0.7) take 1.27, 5.5 and 39 ms in blocks of 8 for 4097, 32769 and
// 262145 bins; of half width 0.5, bin by bin, 1.68, 5.7 and 30.6 ms.
BlockPlan block_plan(double lo, double hi, int nE)
{
    BlockPlan p{};
    p.slope = lo + 0.5 * (hi - lo);
    const double w = 0.5 * (hi - lo);
    for (int B = 64; B >= (nE <= 1 << 17 ? 8 : 16) && !p.B; B /= 2)
        if (w * (B / 2) <= kXMax) p.B = B;
    if (!p.B) return p;
    const double x = w * (p.B / 2), eps = 0x1p-57;
    double term = 1.0;
    for (p.deg = 0; p.deg < kDegMax; ++p.deg) {
        term *= x / (p.deg + 1);
        if (term <= eps) break;
    }
    p.nblk = (nE + p.B - 1) / p.B;
    p.per = (p.nblk + kRgThreads - 1) / kRgThreads;
    return p;
}

BlockPlan grid_plan(const double *c, int n_grid, int nE)
{
    if (n_grid < 1) return BlockPlan{};
    double lo = c[0], hi = c[0];
    for (int k = 1; k < n_grid; ++k) {
        lo = std::min(lo, c[k]);
        hi = std::max(hi, c[k]);
    }
    return block_plan(lo, hi, nE);
}

// Where a block's numbers stand: thread t of the grid kernel takes blocks
// t per .. t per + per - 1, its i-th at slot i kRgThreads + t.
__host__ __device__ inline int block_slot(const BlockPlan &p, int b)
{
    return (b % p.per) * kRgThreads + b / p.per;
}

// Per slot: polynomial coefficients [deg + 1][kStats][slots]; the block's
// heaviest bin, its weighted mean E_J and |m|.
struct Blocks {
    double *coef, *mj, *mm;
    double *lw;  // lnW at the heaviest bin
    double *ln;  // ln of its samples, -inf for a block without samples
    int *E;      // its E_Delta
    int *mid;    // E_mid - E_b
};

size_t block_bytes(const BlockPlan &p)
{
    const size_t slots = (size_t)p.per * kRgThreads;  // 0 without blocks
    return slots * ((kStats * (p.deg + 1) + 4) * sizeof(double) + 2 * sizeof(int));
}

Blocks block_layout(const BlockPlan &p, char *mem)
{
    const size_t slots = (size_t)p.per * kRgThreads;
    Blocks b;
    b.lw = (double *)mem;
    b.ln = b.lw + slots;
    b.coef = b.ln + slots;
    b.mj = b.coef + slots * kStats * (p.deg + 1);
    b.mm = b.mj + slots;
    b.E = (int *)(b.mm + slots);
    b.mid = b.E + slots;
    return b;
}

// 1 / q: a division is some twenty FP64 instructions.
__constant__ double inv_q[kDegMax + 1] = {
    0.0, 1.0, 1.0 / 2, 1.0 / 3, 1.0 / 4, 1.0 / 5, 1.0 / 6, 1.0 / 7, 1.0 / 8, 1.0 / 9, 1.0 / 10,
    1.0 / 11, 1.0 / 12, 1.0 / 13, 1.0 / 14, 1.0 / 15, 1.0 / 16, 1.0 / 17, 1.0 / 18, 1.0 / 19, 1.0 / 20};

// One block of bins per CTA: its heaviest bin, the statistics about that bin
// and the block's weighted means, times V, then thread (p, j) sums its
// coefficient.
__global__ void __launch_bounds__(192)
block_coef_kernel(BinStats<double> s, int nE, int e_min, BlockPlan p, Blocks out)
{
    __shared__ double f[kStats][64], t[kDegMax + 1][64];
    __shared__ double red[3][2];
    __shared__ int ra[2];
    const int b = blockIdx.x, e0 = b * p.B, len = min(p.B, nE - e0), i = threadIdx.x;
    const int mid = min(e0 + p.B / 2, nE - 1), slot = block_slot(p, b);
    const double n = i < len ? s.n[e0 + i] : 0.0;  // bins in the first two warps
    if (i < 64) {
        double v = -INFINITY;
        int a = i;
        if (n > 0.0) v = (-(p.slope * (double)(e0 + i - mid)) - (s.lw[e0 + i] - s.lw[mid])) + log(n);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const double v2 = __shfl_xor_sync(0xFFFFFFFFu, v, o);
            const int a2 = __shfl_xor_sync(0xFFFFFFFFu, a, o);
            if (v2 > v || (v2 == v && a2 < a)) {
                v = v2;
                a = a2;
            }
        }
        if ((i & 31) == 0) {
            red[0][i >> 5] = v;
            ra[i >> 5] = a;
        }
    }
    __syncthreads();
    const int first = red[0][1] > red[0][0] ? 1 : 0;
    if (red[0][first] == -INFINITY) {  // no samples: the whole CTA
        if (i == 0) out.ln[slot] = -INFINITY;
        return;
    }
    const int ref = e0 + ra[first];
    const double r = (double)(e0 + i - ref);
    double v = 0.0, vn = 0.0, mej = 0.0, cm = 0.0;
    __syncthreads();
    if (n > 0.0) {
        // near the heaviest bin these are differences of near numbers
        v = exp(-(p.slope * r) - (s.lw[e0 + i] - s.lw[ref]));
        vn = v * n;
        mej = s.mej[e0 + i] - s.mej[ref];
        cm = s.cm[e0 + i] - s.cm[ref];
    }
    if (i < 64) {
        double z[3] = {vn, vn * mej, vn * cm};
#pragma unroll
        for (int k = 0; k < 3; ++k) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) z[k] += __shfl_xor_sync(0xFFFFFFFFu, z[k], o);
            if ((i & 31) == 0) red[k][i >> 5] = z[k];
        }
    }
    __syncthreads();
    const double z = red[0][0] + red[0][1];
    const double mj = s.mej[ref] + (red[1][0] + red[1][1]) / z, mm = s.cm[ref] + (red[2][0] + red[2][1]) / z;
    if (i == 0) {
        out.ln[slot] = log(s.n[ref]);
        out.E[slot] = e_min + ref;
        out.mid[slot] = mid - ref;
        out.lw[slot] = s.lw[ref];
        out.mj[slot] = mj;
        out.mm[slot] = mm;
    }
    if (i < p.B) {
        const double rho = (double)(e0 + i - mid) * (2.0 / p.B);  // exact: B is a power of 2
        const double dj = n > 0.0 ? s.mej[e0 + i] - mj : 0.0, dm = n > 0.0 ? s.cm[e0 + i] - mm : 0.0;
        f[0][i] = vn;
        f[1][i] = vn * r;
        f[2][i] = vn * dj;
        f[3][i] = vn * dm;
        f[4][i] = n > 0.0 ? v * s.q2[e0 + i] : 0.0;
        f[5][i] = n > 0.0 ? v * s.q4[e0 + i] : 0.0;
        f[6][i] = vn * (dj * r);
        f[7][i] = n > 0.0 ? v * s.vb[e0 + i] + vn * (dm * dm) : 0.0;
        double pw = 1.0;
        t[0][i] = 1.0;
        for (int q = 1; q <= p.deg; ++q) {
            pw *= rho * inv_q[q];
            t[q][i] = pw;
        }
    }
    __syncthreads();
    for (int q = i; q < kStats * (p.deg + 1); q += blockDim.x) {
        const double *ff = f[q % kStats], *tt = t[q / kStats];
        double c = 0.0;
        for (int k = 0; k < p.B; ++k) c = fma(ff[k], tt[k], c);
        out.coef[(size_t)q * (p.per * kRgThreads) + slot] = c;
    }
}

// -c e - (lw - l0), e the distance from the reference bin: the product and the
// difference without rounding, their sum rounded once.
__device__ __forceinline__ double block_exponent(double c, double e, double lw, double l0)
{
    const double p = __dmul_rn(c, e), pe = fma(c, e, -p);
    const double l = __dsub_rn(lw, l0), bb = __dsub_rn(l, lw);
    const double le = __dsub_rn(__dsub_rn(lw, __dsub_rn(l, bb)), __dadd_rn(l0, bb));
    return (-p - l) - (pe + le);
}

// KK consecutive fields per CTA; thread t takes the blocks at slots
// i kRgThreads + t, whose coefficients are read once for the KK fields.
template <int KK>
__global__ void __launch_bounds__(kRgThreads)
block_grid_kernel(Blocks bl, BlockPlan p, double beta, int V, const double *__restrict__ cgrid,
                  int n_grid, double *__restrict__ out)
{
    __shared__ double shv[32];
    __shared__ int she[32];
    __shared__ double sh[kRgThreads / 32 * kStats];
    const int t = threadIdx.x, k0 = blockIdx.x * KK;
    const size_t slots = (size_t)p.per * kRgThreads;
    double c[KK], x[KK], u[KK], l0[KK], J0[KK], M0[KK];
    int E0[KK];
    // the reference of each field: its heaviest block
#pragma unroll
    for (int k = 0; k < KK; ++k) {
        c[k] = cgrid[min(k0 + k, n_grid - 1)];
        u[k] = -(c[k] - p.slope);
        x[k] = u[k] * (0.5 * p.B);
        double best = -INFINITY;
        int at = 0x7FFFFFFF;
        for (int i = 0; i < p.per; ++i) {
            // loaded together (slots without a block are allocated, and not used)
            const int q = i * kRgThreads + t, E = bl.E[q];
            const double ln = bl.ln[q], lw = bl.lw[q];
            if (t * p.per + i < p.nblk && ln > -INFINITY) {
                const double a = (-(c[k] * (double)E) - lw) + ln;
                if (a > best) {
                    best = a;
                    at = q;
                }
            }
        }
        block_argmax(best, at, shv, she);
        const bool none = at >= (int)slots;  // no sample lies in the window (the call fails)
        E0[k] = none ? 0 : bl.E[at];
        l0[k] = none ? 0.0 : bl.lw[at];
        J0[k] = none ? 0.0 : bl.mj[at];
        M0[k] = none ? 0.0 : bl.mm[at];
    }
    double S[KK][kStats];
#pragma unroll
    for (int k = 0; k < KK; ++k)
#pragma unroll
        for (int j = 0; j < kStats; ++j) S[k][j] = 0.0;
    for (int i = 0; i < p.per; ++i) {
        const int q = i * kRgThreads + t, Eb = bl.E[q];
        const double ln = bl.ln[q], lb = bl.lw[q], mid = (double)bl.mid[q];
        if (t * p.per + i >= p.nblk || ln == -INFINITY) continue;
        double A[KK];
        bool any = false;
#pragma unroll
        for (int k = 0; k < KK; ++k) {
            A[k] = exp(fma(u[k], mid, block_exponent(c[k], (double)(Eb - E0[k]), lb, l0[k])));
            any = any || A[k] > 0.0;
        }
        if (!any) continue;
        double a[kStats][KK];
#pragma unroll
        for (int j = 0; j < kStats; ++j) {
            const double *cf = bl.coef + (size_t)j * slots + q;
            const double top = cf[(size_t)p.deg * kStats * slots];
#pragma unroll
            for (int k = 0; k < KK; ++k) a[j][k] = top;
            for (int g = p.deg - 1; g >= 0; --g) {
                const double cg = cf[(size_t)g * kStats * slots];
#pragma unroll
                for (int k = 0; k < KK; ++k) a[j][k] = fma(a[j][k], x[k], cg);
            }
        }
        const double Jb = bl.mj[q], Mb = bl.mm[q];
#pragma unroll
        for (int k = 0; k < KK; ++k) {
            const double dE = (double)(Eb - E0[k]), dJ = Jb - J0[k], dM = Mb - M0[k];
            const double n0 = A[k] * a[0][k], e1 = A[k] * a[1][k], j1 = A[k] * a[2][k], m1 = A[k] * a[3][k];
            const double e2 = fma(n0, dE, e1), j2 = fma(n0, dJ, j1);
            S[k][0] += n0;
            S[k][1] += e2;
            S[k][2] += j2;
            S[k][3] += fma(n0, dM, m1);
            S[k][4] += A[k] * a[4][k];
            S[k][5] += A[k] * a[5][k];
            // sum n (J - J0)(E - E0) and sum (vb + n (m - M0)^2)
            S[k][6] += fma(A[k], a[6][k], fma(j1, dE, e2 * dJ));
            S[k][7] += fma(A[k], a[7][k], dM * fma(n0, dM, m1 + m1));
        }
    }
#pragma unroll
    for (int k = 0; k < KK; ++k) {
        double (&T)[kStats] = S[k];
        block_sum_plain<kStats, kRgThreads / 32>(T, sh);
        if (t == 0 && k0 + k < n_grid)
            put_field(T, E0[k], J0[k], M0[k], beta, V, out + 5 * (int64_t)(k0 + k));
    }
}

cudaError_t launch_blocks(const BinStats<double> &s, int nE, int e_min, double beta, int V,
                          const BlockPlan &p, char *mem, const double *d_c, int n_grid,
                          double *d_out, int nsm, cudaStream_t st)
{
    const Blocks bl = block_layout(p, mem);
    block_coef_kernel<<<p.nblk, 192, 0, st>>>(s, nE, e_min, p, bl);
    // four fields per CTA share the coefficients' reads; with few fields one
    // each, so that they spread over the SMs
    if (n_grid >= 4 * nsm)
        block_grid_kernel<4><<<(n_grid + 3) / 4, kRgThreads, 0, st>>>(bl, p, beta, V, d_c, n_grid,
                                                                      d_out);
    else
        block_grid_kernel<1><<<n_grid, kRgThreads, 0, st>>>(bl, p, beta, V, d_c, n_grid, d_out);
    return cudaGetLastError();
}

// Scratch layout of one call (bytes), all 256-byte aligned.
struct Scratch {
    size_t bins, stats, grid, out, err, total;
    size_t lnw;  // lnW's place in stats
};

Scratch scratch_layout(int nE, int n_grid, int precision)
{
    auto al = [](size_t x) { return (x + 255) & ~(size_t)255; };
    Scratch s{};
    s.bins = al((size_t)6 * nE * sizeof(unsigned long long));
    s.lnw = (size_t)(precision == 32 ? 8 * sizeof(float) : 7 * sizeof(double)) * nE;
    s.stats = al((size_t)(precision == 32 ? 10 * sizeof(float) : 9 * sizeof(double)) * nE);
    s.grid = al((size_t)2 * n_grid * sizeof(double));
    s.out = al((size_t)5 * n_grid * sizeof(double));
    s.err = al(sizeof(int));
    s.total = s.bins + s.stats + s.grid + s.out + s.err;
    return s;
}

// Buckets of a window of nE bins.
int bucket_count_of(int nE) { return (int)(((int64_t)nE + kBkt - 1) >> kBktBits); }

// Bytes of the bucket counters at the start of a record buffer (256-byte
// aligned): [nbk][kMaxG] storage places, [nbk][kMaxG] places in bucket order,
// then each bucket's start and size.
size_t bucket_counter_bytes(int nE)
{
    const size_t nbk = (size_t)bucket_count_of(nE);
    return ((2 * nbk * kMaxG + 2 * nbk) * sizeof(unsigned) + 255) & ~(size_t)255;
}

}  // namespace

namespace muca {

size_t reweight_record_bytes(int32_t n_e, int64_t n_samples)
{
    // windows of more than kMaxBk buckets take the direct path: no records
    if (bucket_count_of(n_e) > kMaxBk) return 0;
    const int64_t cap = std::min<int64_t>(n_samples, (int64_t)1 << 26);
    return bucket_counter_bytes(n_e) + (size_t)std::max<int64_t>(cap, 0) * sizeof(uint2);
}


// The whole reweighting on a caller-provided scratch region of
// scratch_layout(...).total bytes (device memory).
int reweight_on_scratch(const int32_t *e_j, const int32_t *e_d, const int32_t *m, int64_t n_rows,
                        int32_t row_len, int64_t row_stride, const double *lnW, int32_t e_min,
                        int32_t n_e, double beta, int32_t V, const double *delta_grid,
                        int32_t n_grid, int32_t precision, double *out, cudaStream_t st,
                        char *scratch, char *records, size_t records_bytes, char *blocks,
                        size_t blocks_bytes)
{
    const Scratch L = scratch_layout(n_e, n_grid, precision);
    char *p = scratch;
    Bins b;
    b.cnt = (unsigned long long *)p;
    b.sej = b.cnt + n_e;
    b.sam = b.sej + n_e;
    b.sm2 = b.sam + n_e;
    b.sm4lo = b.sm2 + n_e;
    b.sm4hi = b.sm4lo + n_e;
    char *ps = p + L.bins;
    char *pg = ps + L.stats;
    double *d_out = (double *)(pg + L.grid);
    int *d_err = (int *)((char *)d_out + L.out);
    cudaError_t ce;
#define RCK(call)                                                                   \
    do {                                                                            \
        ce = (call);                                                                \
        if (ce != cudaSuccess)                                                      \
            return rw_fail(MUCA_ERR_CUDA, std::string(#call) + ": " + cudaGetErrorString(ce)); \
    } while (0)
    RCK(cudaMemsetAsync(p, 0, L.bins, st));
    RCK(cudaMemsetAsync(d_err, 0, sizeof(int), st));
    int dev = 0, nsm = 152;
    if (cudaGetDevice(&dev) == cudaSuccess)
        cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    const int nbk = bucket_count_of(n_e);
    const size_t rec_cap =
        (records && nbk <= kMaxBk)
            ? (records_bytes - std::min(records_bytes, bucket_counter_bytes(n_e))) / sizeof(uint2)
            : 0;
    if (n_rows > 0 && row_len > 0 && (size_t)row_len <= rec_cap) {
        // stage A through buckets, a pass of at most rec_cap samples at a time
        unsigned *d_cnt = (unsigned *)records;  // [nbk][g], g <= kMaxG
        unsigned *d_lst = d_cnt + (size_t)nbk * kMaxG;
        unsigned *d_bstart = d_lst + (size_t)nbk * kMaxG, *d_bcnt = d_bstart + nbk;
        uint2 *d_rec = (uint2 *)(records + bucket_counter_bytes(n_e));
        RCK(cudaFuncSetAttribute(bucket_hist_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)kHistSmem));
        const int cpr = (int)(((int64_t)row_len + kChunk - 1) / kChunk);
        const int64_t rows_pass = std::min<int64_t>(n_rows, (int64_t)(rec_cap / (size_t)row_len));
        for (int64_t r0 = 0; r0 < n_rows; r0 += rows_pass) {
            const int64_t nr = std::min(rows_pass, n_rows - r0);
            const int64_t off = r0 * row_stride;
            // one 1024-thread block per SM
            const int g = (int)std::min<int64_t>(nr * cpr, std::min(nsm, kMaxG));
            bucket_count_kernel<<<g, kCsThreads, 0, st>>>(e_d + off, nr, row_len, row_stride,
                                                          e_min, n_e, nbk, cpr, d_cnt,
                                                          d_err);
            RCK(cudaGetLastError());
            bucket_scan_kernel<<<1, 1024, 0, st>>>(d_cnt, d_lst, nbk, g, d_bstart, d_bcnt);
            RCK(cudaGetLastError());
            bucket_scatter_kernel<<<g, kCsThreads, 0, st>>>(
                e_j + off, e_d + off, m + off, nr, row_len, row_stride, e_min, n_e, nbk, cpr,
                d_cnt, d_rec, b);
            RCK(cudaGetLastError());
            bucket_hist_kernel<<<nsm, kHT, kHistSmem, st>>>(d_rec, d_cnt, d_lst, g, d_bstart,
                                                           d_bcnt, nbk, (unsigned)(nr * row_len),
                                                           b);
            RCK(cudaGetLastError());
        }
    } else if (n_rows > 0 && row_len > 0) {
        dim3 grid((unsigned)std::min<int64_t>((row_len + 255) / 256, 1024),
                  (unsigned)std::min<int64_t>(n_rows, 4096));
        bin_kernel<<<grid, 256, 0, st>>>(e_j, e_d, m, n_rows, row_len, row_stride, e_min, n_e, b,
                                         d_err);
        RCK(cudaGetLastError());
    }
    const int sb = (n_e + 255) / 256;
    // the fields c = beta Delta
    std::vector<double> c(n_grid);
    for (int k = 0; k < n_grid; ++k) c[k] = beta * delta_grid[k];
    const BlockPlan plan = grid_plan(c.data(), n_grid, n_e);
    if (precision == 64 && n_grid > 0 && block_bytes(plan) > blocks_bytes)
        return rw_fail(MUCA_ERR_OOM, "muca_reweight: no room for the blocks of bins");
    if (precision == 64) {
        BinStats<double> s;
        double *q = (double *)ps;
        s.n = q;
        s.mej = q + n_e;
        s.cm = q + 2 * (size_t)n_e;
        s.vb = q + 3 * (size_t)n_e;
        s.q2 = q + 4 * (size_t)n_e;
        s.q4 = q + 5 * (size_t)n_e;
        s.lw = q + 6 * (size_t)n_e;
        s.lwlo = nullptr;
        double *d_lnW = (double *)(ps + L.lnw);
        double *d_c = (double *)pg;
        RCK(cudaMemcpyAsync(d_lnW, lnW, (size_t)n_e * sizeof(double), cudaMemcpyHostToDevice, st));
        RCK(cudaMemcpyAsync(d_c, c.data(), (size_t)n_grid * sizeof(double),
                            cudaMemcpyHostToDevice, st));
        stats_kernel_f64<<<sb, 256, 0, st>>>(b, n_e, V, d_lnW, s);
        RCK(cudaGetLastError());
        if (n_grid > 0 && plan.B)
            RCK(launch_blocks(s, n_e, e_min, beta, V, plan, blocks, d_c, n_grid, d_out, nsm, st));
        else if (n_grid > 0) {
            // few fields leave SMs idle: more threads for each; no more than bins
            int threads = n_grid < nsm ? 512 : 256;
            while (threads > 64 && threads / 2 >= n_e) threads /= 2;
            grid_kernel_f64<<<n_grid, threads, 0, st>>>(s, n_e, e_min, beta, V, d_c, d_out);
        }
        RCK(cudaGetLastError());
    } else {
        BinStats<float> s;
        float *q = (float *)ps;
        s.n = q;
        s.mej = q + n_e;
        s.cm = q + 2 * (size_t)n_e;
        s.vb = q + 3 * (size_t)n_e;
        s.q2 = q + 4 * (size_t)n_e;
        s.q4 = q + 5 * (size_t)n_e;
        s.lw = q + 6 * (size_t)n_e;
        s.lwlo = q + 7 * (size_t)n_e;
        double *d_lnW = (double *)(ps + L.lnw);
        double *d_c = (double *)pg;
        RCK(cudaMemcpyAsync(d_lnW, lnW, (size_t)n_e * sizeof(double), cudaMemcpyHostToDevice, st));
        RCK(cudaMemcpyAsync(d_c, c.data(), (size_t)n_grid * sizeof(double),
                            cudaMemcpyHostToDevice, st));
        stats_kernel_f32<<<sb, 256, 0, st>>>(b, n_e, V, d_lnW, s);
        RCK(cudaGetLastError());
        if (n_grid > 0)
            grid_kernel_f32<kGridD><<<(n_grid + kGridD - 1) / kGridD, 256, 0, st>>>(
                s, n_e, e_min, (float)beta, V, d_c, n_grid, d_out);
        RCK(cudaGetLastError());
        RCK(cudaStreamSynchronize(st));
    }
    int h_err = 0;
    RCK(cudaMemcpyAsync(&h_err, d_err, sizeof(int), cudaMemcpyDeviceToHost, st));
    RCK(cudaMemcpyAsync(out, d_out, (size_t)5 * n_grid * sizeof(double), cudaMemcpyDeviceToHost,
                        st));
    RCK(cudaStreamSynchronize(st));
#undef RCK
    if (h_err) return rw_fail(MUCA_ERR_WINDOW, "a sample's E_Delta lies outside [e_min, e_min + n_e)");
    return MUCA_OK;
}

size_t reweight_block_bytes(double beta, const double *delta_grid, int32_t n_grid, int32_t n_e,
                            int32_t precision)
{
    if (precision != 64 || n_grid < 1) return 0;
    std::vector<double> c(n_grid);
    for (int k = 0; k < n_grid; ++k) c[k] = beta * delta_grid[k];
    return block_bytes(grid_plan(c.data(), n_grid, n_e));
}

size_t reweight_scratch_bytes(int32_t n_e, int32_t n_grid, int32_t precision)
{
    return scratch_layout(n_e, n_grid, precision).total;
}

int reweight_check_args(const int32_t *e_j, const int32_t *e_d, const int32_t *m, int64_t n_rows,
                        int32_t row_len, int64_t row_stride, const double *lnW, int32_t e_min,
                        int32_t n_e,
                        double beta, int32_t V, const double *delta_grid, int32_t n_grid,
                        int32_t precision, double *out)
{
    if (!e_j || !e_d || !m || !lnW || !out || (n_grid > 0 && !delta_grid))
        return rw_fail(MUCA_ERR_INVALID_ARG, "muca_reweight: null pointer");
    if (n_rows < 0 || row_len < 0 || (n_rows > 1 && row_stride < row_len) || n_e < 1 || V < 1 ||
        n_grid < 0)
        return rw_fail(MUCA_ERR_INVALID_ARG, "muca_reweight: bad sizes");
    if (n_rows * (int64_t)row_len < 1)
        return rw_fail(MUCA_ERR_INVALID_ARG, "muca_reweight: no samples");
    if ((int64_t)e_min + n_e - 1 > INT32_MAX)
        return rw_fail(MUCA_ERR_INVALID_ARG, "muca_reweight: e_min + n_e - 1 exceeds int32");
    if (precision != 32 && precision != 64)
        return rw_fail(MUCA_ERR_INVALID_ARG, "muca_reweight: precision must be 32 or 64");
    if (!(beta > 0.0) || !std::isfinite(beta))
        return rw_fail(MUCA_ERR_INVALID_ARG, "muca_reweight: beta must be > 0");
    for (int e = 0; e < n_e; ++e)
        if (!std::isfinite(lnW[e])) return rw_fail(MUCA_ERR_INVALID_ARG, "muca_reweight: lnW not finite");
    for (int k = 0; k < n_grid; ++k)
        if (!std::isfinite(delta_grid[k]))
            return rw_fail(MUCA_ERR_INVALID_ARG, "muca_reweight: Delta grid not finite");
    return MUCA_OK;
}

}  // namespace muca

// Device memory pools of the analysis calls on the current device, created on
// first use, so that repeated calls do not map and unmap their working memory
// each time.  muca_reweight's keeps what it has once held (release threshold:
// all); that of muca_find_peak and muca_equal_height keeps 256 MiB between calls
// (20 data sets of 262145 bins) and gives the rest back when a call ends.
int muca::scratch_pool(ScratchPool which, cudaMemPool_t *out)
{
    static std::mutex mu;
    static cudaMemPool_t all[2][64] = {};
    cudaMemPool_t *const pools = all[which == ScratchPool::peak];
    int dev = -1;
    cudaError_t ce = cudaGetDevice(&dev);
    if (ce != cudaSuccess)
        return rw_fail(MUCA_ERR_CUDA, std::string("cudaGetDevice: ") + cudaGetErrorString(ce));
    if (dev < 0 || dev >= 64) return rw_fail(MUCA_ERR_NOT_SUPPORTED, "device index out of range");
    std::lock_guard<std::mutex> lk(mu);
    if (!pools[dev]) {
        cudaMemPoolProps props = {};
        props.allocType = cudaMemAllocationTypePinned;
        props.location.type = cudaMemLocationTypeDevice;
        props.location.id = dev;
        cudaMemPool_t p = nullptr;
        ce = cudaMemPoolCreate(&p, &props);
        if (ce != cudaSuccess)
            return rw_fail(MUCA_ERR_CUDA, std::string("cudaMemPoolCreate: ") + cudaGetErrorString(ce));
        uint64_t keep = which == ScratchPool::peak ? (uint64_t)256 << 20 : ~0ull;
        ce = cudaMemPoolSetAttribute(p, cudaMemPoolAttrReleaseThreshold, &keep);
        if (ce != cudaSuccess) {
            cudaMemPoolDestroy(p);
            return rw_fail(MUCA_ERR_CUDA, std::string("cudaMemPoolSetAttribute: ") +
                                              cudaGetErrorString(ce));
        }
        pools[dev] = p;
    }
    *out = pools[dev];
    return MUCA_OK;
}

extern "C" int muca_reweight(const int32_t *e_j, const int32_t *e_d, const int32_t *m,
                             int64_t n_rows, int32_t row_len, int64_t row_stride,
                             const double *lnW, int32_t e_min, int32_t n_e, double beta, int32_t V,
                             const double *delta_grid, int32_t n_grid, int32_t precision,
                             double *out, void *stream)
{
    int rc = muca::reweight_check_args(e_j, e_d, m, n_rows, row_len, row_stride, lnW, e_min, n_e,
                                       beta, V, delta_grid, n_grid, precision, out);
    if (rc != MUCA_OK) return rc;
    cudaStream_t st = (cudaStream_t)stream;
    const size_t bytes = muca::reweight_scratch_bytes(n_e, n_grid, precision);
    const size_t rbytes = muca::reweight_record_bytes(n_e, n_rows * (int64_t)row_len);
    cudaMemPool_t pool = nullptr;
    rc = muca::scratch_pool(muca::ScratchPool::reweight, &pool);
    if (rc != MUCA_OK) return rc;
    void *scratch = nullptr;
    const size_t bbytes = muca::reweight_block_bytes(beta, delta_grid, n_grid, n_e, precision);
    const size_t blocks_at = (bytes + rbytes + 255) & ~(size_t)255;
    cudaError_t ce = cudaMallocFromPoolAsync(&scratch, blocks_at + bbytes, pool, st);
    if (ce != cudaSuccess)
        return rw_fail(ce == cudaErrorMemoryAllocation ? MUCA_ERR_OOM : MUCA_ERR_CUDA,
                       std::string("cudaMallocAsync: ") + cudaGetErrorString(ce));
    rc = muca::reweight_on_scratch(e_j, e_d, m, n_rows, row_len, row_stride, lnW, e_min, n_e, beta,
                                   V, delta_grid, n_grid, precision, out, st, (char *)scratch,
                                   (char *)scratch + bytes, rbytes, (char *)scratch + blocks_at,
                                   bbytes);
    cudaFreeAsync(scratch, st);
    cudaStreamSynchronize(st);
    return rc;
}
