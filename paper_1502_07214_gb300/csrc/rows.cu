// rows.cu -- the site-per-lane sweep kernel: typewriter Metropolis sweeps
// (Sec. II) in which the lanes of a warp hold the sites of a walker's row and
// resolve the row together, for the clean model and for couplings per bond.
//
// A site's decision needs three things that the row itself changes: whether
// its left neighbour was accepted, E_Delta when the site is visited, and, for
// the last site, whether site 0 was.  Given the row's acceptance bits all
// three follow at once: the neighbours' bits, and E_Delta at the row start
// plus the accepted moves with d = +1 minus those with d = -1 among the sites
// before it (two population counts).  So the lanes guess the bits (none
// accepted), decide every site with them, collect the new bits by a ballot
// and repeat until they reproduce themselves.  After pass t the first t sites
// are right, whatever the guess, so the row converges to the site-by-site
// result, bit for bit; it takes as many passes as accepted moves that change
// a later decision of the same row, about two or three, not one per site.
//
// Why this layout: a walker is one serial chain of rows, and a program runs
// 64 to some thousand walkers on 608 schedulers, so the time of a sweep is
// the latency of a row times the rows, not the arithmetic.  One site per lane
// makes a row's latency independent of its length (up to 32 sites) and a
// walker's bits warp-uniform; a chain kernel pays a dependent table load per
// site instead.  Longer rows are cut into SEG segments of A lanes that follow one
// another (the segment before is final); 32 / A walkers lie side by side in a
// warp.
//
// Memory: the planes that a row reads lie in shared memory, rows at a fixed
// pitch; behind the row being resolved, finished rows go back to the lattice
// and the rows of the plane after next come in (cp.async), four rows at a time.
// Thresholds are read through L1: a walker stays within a few table rows for
// many rows.  Random numbers: four rows of L sites are L Philox blocks, for
// every L (one more where a row starts inside a block), so the lanes draw one
// block per site of a row for four rows and pass the words through shared
// memory.
//
// What bounds it: the latency of a row, about 200 cycles of dependent
// instructions without an accepted move and 100 more for each further pass
// (three or four warps per scheduler at most); 110 to 170 warp instructions
// per row of up to 32 sites.  Nothing moves through HBM but each spin once in
// and once out per sweep.
//
// Measured on GB300 against the kernels that the autotuner picked before
// (sweep.cu's split kernel for L = 8 .. 32, scan.cu's for L = 48, one thread
// per walker for L % 4 != 0 and for couplings), time per call:
//   L = 8, T = 2, 64 walkers, 200 sweeps and merge    11.8 -> 4.4 ms
//   L = 16, T = 1, 1024 walkers, 500 sweeps and merge 94.8 -> 25.0 ms
//   L = 32, T = 0.9, 2048 walkers, 150 and merge      157 -> 43.4 ms
//   L = 8 .. 32 in one context, 12288 walkers, 60     112 -> 42.2 ms
//   L = 22, T = 1.4182, 1000 walkers, 50 and merge    76.9 -> 6.8 ms
//   L = 28, T = 1, 1024 walkers, 100 recorded         74.4 -> 26.0 ms
//   L = 48, T = 0.9, 4096 walkers, 60 recorded        248 -> 115 ms
//   couplings, L = 24, 4096 walkers, 50 and merge     120 -> 23.4 ms
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "muca_internal.h"
#include "philox.cuh"

namespace muca {
namespace {

// Byte lookup by t = 2 (s + 1) + proposal bit (0 .. 5), sign-extended: the
// selector takes byte t and replicates its sign into the other bytes (the
// instruction itself: __byte_perm masks the selector's sign bits away).
__device__ __forceinline__ uint32_t lut_sel(int t) { return (uint32_t)t * 0x1111u + 0x8880u; }
__device__ __forceinline__ int lut(uint32_t lo, uint32_t hi, uint32_t sel)
{
    int r;
    asm("prmt.b32 %0, %1, %2, %3;" : "=r"(r) : "r"(lo), "r"(hi), "r"(sel));
    return r;
}
// t:               0    1    2    3    4    5
// delta = s' - s  +1   +2   -1   +1   -2   -1
// d               -1    0   +1   +1    0   -1
constexpr uint32_t kDeltaLo = 0x01FF0201u, kDeltaHi = 0x0000FFFEu;
constexpr uint32_t kDLo = 0x010100FFu, kDHi = 0x0000FF00u;
// clean columns 19 + 13 d + k h: k = -sign(delta)
constexpr uint32_t kStepLo = 0xFF01FFFFu, kStepHi = 0x00000101u;

// Memory operations under a predicate, without a branch: a branch that the
// compiler takes for divergent splits the code around it into small blocks,
// each warp-wide operation behind a convergence check of its own.
__device__ __forceinline__ uint32_t shared_addr(const void *p)
{
    return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void st_shared_u8(uint32_t a, int v, bool p)
{
    asm volatile("{.reg .pred q; setp.ne.s32 q, %2, 0; @q st.shared.u8 [%0], %1;}" ::"r"(a), "r"(v),
                 "r"((int)p)
                 : "memory");
}
__device__ __forceinline__ void st_shared_v4(uint32_t a, uint4 v, bool p)
{
    asm volatile("{.reg .pred q; setp.ne.s32 q, %5, 0; @q st.shared.v4.b32 [%0], {%1, %2, %3, %4};}" ::"r"(a),
                 "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w), "r"((int)p)
                 : "memory");
}
__device__ __forceinline__ void st_global_v4(void *a, uint4 v, bool p)
{
    asm volatile("{.reg .pred q; setp.ne.s32 q, %5, 0; @q st.global.v4.b32 [%0], {%1, %2, %3, %4};}" ::"l"(a),
                 "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w), "r"((int)p)
                 : "memory");
}
__device__ __forceinline__ void cp4(void *smem, const void *gmem)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(shared_addr(smem)), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp16(uint32_t smem, const void *gmem, bool p)
{
    asm volatile("{.reg .pred q; setp.ne.s32 q, %2, 0; @q cp.async.cg.shared.global [%0], [%1], 16;}" ::"r"(smem),
                 "l"(gmem), "r"((int)p)
                 : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_wait_1() { asm volatile("cp.async.wait_group 1;" ::: "memory"); }
__device__ __forceinline__ void cp_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// How a walker's rows pass through shared memory:
//   planes: up to 12 sites all L; else the three that a row reads (z - 1, z, z + 1);
//   row L of a plane repeats row 0, the y + 1 neighbour of the last row, but for
//     three segments, where a select takes its place;
//   random words: two buffers for one or two segments, so that the next rows' words are
//     stored as they are drawn; else one, the words waiting in registers.
// The differences buy room: 48-site rows of three segments take 15.5 KB per warp, 14
// warps per SM, so that the benchmark's 2048 warps run in one wave (17.4 KB left 72
// of them to a second one: 157 -> 116 ms for 60 sweeps of 4096 walkers).
// Rows are PITCH bytes apart, so a row's addresses are a register and a
// constant.
__host__ __device__ constexpr int rows_slots(int L) { return L <= 12 ? L : 3; }
__host__ __device__ constexpr bool rows_repeat0(int seg) { return seg != 3; }
__host__ __device__ constexpr int rows_buffers(int seg) { return seg <= 2 ? 2 : 1; }
// Words of a buffer: four rows touch at most L + 1 Philox blocks (rows that
// start inside a block, L odd, one more than L).
__host__ __device__ constexpr int rows_random_words(int L) { return 4 * (L + 1); }
// Words from one walker to the next: 16-byte aligned, and spread over the
// banks so that the walkers of a warp read a row without conflicts.  With one
// or two segments the rows after a plane's last are read, and not used: two rows of
// slack.
__host__ __device__ inline int rows_walker_words(int L, int seg, int per_warp, int pitch)
{
    const int rows = rows_slots(L) * (L + rows_repeat0(seg)) + (seg <= 2 ? 2 : 0);
    const int n = rows_buffers(seg) * rows_random_words(L) + rows * (pitch / 4);
    const int want = per_warp <= 1 ? 0 : per_warp == 2 ? 16 : per_warp <= 4 ? 8 : 4;
    return want ? n + ((want - n) % 32 + 32) % 32 : (n + 3) / 4 * 4;
}

// Copies of the rows y0 .. y0 + n - 1 of a plane between the lattice and shared
// memory, a word per lane and row, for any layout of the lattice.
template <int PITCH>
struct RowCopy {
    uint32_t *g;   // word 0 of the walker's lattice
    int64_t wstr;  // its word stride
    int L, Lw, rw, h;
    __device__ __forceinline__ void in(int8_t *sm, int z, int y0, int n) const
    {
        if (h < Lw)
            for (int i = 0; i < n; ++i)
                cp4(sm + i * PITCH + 4 * h, g + ((ptrdiff_t)(z * L + y0 + i) * rw + h) * wstr);
    }
    __device__ __forceinline__ void out(const int8_t *sm, int z, int y0, int n) const
    {
        if (h < Lw)
            for (int i = 0; i < n; ++i)
                g[((ptrdiff_t)(z * L + y0 + i) * rw + h) * wstr] =
                    *reinterpret_cast<const uint32_t *>(sm + i * PITCH + 4 * h);
    }
    // a whole plane, and row 0 once more as row L
    __device__ __forceinline__ void plane_in(int8_t *sm, int z, bool repeat0) const
    {
        in(sm, z, 0, L);
        if (repeat0) in(sm + L * PITCH, z, 0, 1);
    }
};

// What a site's decision needs that no earlier site of its row changes.
struct Site {
    uint32_t u;             // uniform draw, ~0 without a site
    int s, delta, d, step;  // old spin, s' - s, s'^2 - s^2, column step per unit of h
    int h;                  // neighbour sum without the y - 1 neighbour
    uint32_t j;             // couplings to the x and y neighbours
    // from the row's other lanes: the left site's delta, site 0's, and which
    // sites' moves have d = +1 and d = -1
    int dl, d0;
    unsigned Pm, Mm;
};

// The sweeps of one warp's walkers w0 .. w0 + nw - 1 (a block).  Lane h of a
// walker's A lanes holds sites q A + h, q < SEG, of every row.  Everything but
// the lane's own quantities comes from kernel parameters, so that the loop
// control and the branches stay uniform.
//
// The steps (row, segment) of four rows are pipelined: while the first
// thresholds of a step are on their way, the next step's Site is formed, and
// in the second row the random words of the next four rows are drawn.
template <int SEG, int PITCH, bool BONDS>
__device__ __forceinline__ void rows_sweeps(const GroupDev &g, int A, int per_warp, int w0,
                                            uint32_t *smem, uint32_t seed, uint64_t sweep0,
                                            int n_sweeps, int64_t ts_pos, int record)
{
    const int lane = (int)(threadIdx.x & 31);
    const int L = g.L, nw = min(per_warp, g.W - w0);
    // lanes without a walker run along on the block's first walker, with no
    // site: they never accept and store nothing
    const int slot0 = lane / A, slot = slot0 < nw ? slot0 : 0;
    const int h = lane - slot0 * A, sbase = slot * A;
    const bool used = slot0 < nw;
    const int w = w0 + slot;
    int xo[SEG], xl_o[SEG], xr_o[SEG];  // the lane's byte of a row, its x neighbours' bytes
    uint32_t idle[SEG];
#pragma unroll
    for (int q = 0; q < SEG; ++q) {
        const bool act = used && q * A + h < L;
        idle[q] = act ? 0u : ~0u;
        xo[q] = act ? q * A + h : 0;
        xl_o[q] = xo[q] == 0 ? L - 1 : xo[q] - 1;
        xr_o[q] = xo[q] == L - 1 ? 0 : xo[q] + 1;
    }
    uint32_t *const mem = smem + slot * rows_walker_words(L, SEG, per_warp, PITCH);
    int8_t *const sp = reinterpret_cast<int8_t *>(mem + rows_buffers(SEG) * rows_random_words(L));
    constexpr bool REPEAT0 = rows_repeat0(SEG), TWO = rows_buffers(SEG) == 2;
    const int pb = (L + REPEAT0) * PITCH;  // bytes per plane
    const bool ring = rows_slots(L) < L;
    const RowCopy<PITCH> copy{g.spins + (ptrdiff_t)w * g.cstr, g.wstr, L, g.Lw, g.rw, h};
    // a lattice whose rows lie as in shared memory is copied 16 bytes per lane
    const bool wide = g.wstr == 1 && g.rw * 4 == PITCH;
    char *const lat = reinterpret_cast<char *>(copy.g) + 16 * h;
    const uint32_t sp_a = shared_addr(sp);
    if (used) {
        if (ring) {
            copy.plane_in(sp, L - 1, REPEAT0);
            copy.plane_in(sp + pb, 0, REPEAT0);
            copy.plane_in(sp + 2 * pb, 1, REPEAT0);
        } else {
            for (int z = 0; z < L; ++z) copy.plane_in(sp + z * pb, z, REPEAT0);
        }
    }
    cp_commit();
    // the table from kPad rows below its first, at the middle of the columns
    const int nj = BONDS ? 24 * g.jmax + 1 : kBlk;
    const int trow = BONDS ? 3 * nj : kRow;
    const uint32_t *__restrict__ thr = (BONDS ? g.thrJ : g.thrE) - (ptrdiff_t)kPad * trow +
                                       (BONDS ? nj + 12 * g.jmax : 19);
    const unsigned lanes = (A == 32 ? ~0u : ((1u << A) - 1u)) << sbase;  // the walker's
    const unsigned lower = ((1u << lane) - 1u) & lanes;
    const int last_lane = sbase + (L - 1) - (SEG - 1) * A;  // holds site L - 1
    const unsigned bitL = h > 0 ? 1u << (lane - 1) : 0u;
    const unsigned bit0 = SEG == 1 && lane == last_lane ? 1u << sbase : 0u;
    const PhiloxKeys keys = philox_keys(g.walker0 + (uint32_t)w, seed);
    const unsigned lmask = __ballot_sync(~0u, used && h == 0);
    // E_Delta as the word offset of its table row
    int eo = (g.tal[g.Wpad + w] - g.e_min + kPad) * trow;
    int EJ = g.tal[w], Mg = g.tal[2 * g.Wpad + w];
    // byte offsets of planes z - 1, z, z + 1 in shared memory
    int am = ring ? 0 : (L - 1) * pb, az = ring ? pb : 0, ap = ring ? 2 * pb : pb;
    // random words of the four rows from site `site` on: block b of the walker
    auto draw = [&](int site, int b, uint64_t sw) {
        return philox4x32_10(
            make_uint4((uint32_t)((site >> 2) + b), (uint32_t)sw, (uint32_t)(sw >> 32), 0u), keys);
    };
    auto keep = [&](uint32_t *to, uint4 v, int n_blk, int b) {
        st_shared_v4(shared_addr(to + 4 * b), v, used && b < n_blk);
    };
    uint32_t *buf = mem, *buf1 = TWO ? mem + rows_random_words(L) : mem;
    auto blocks_of = [&](int site, int y0) {
        return ((site & 3) + min(4, L - y0) * L + 3) >> 2;
    };
    for (int b = h; b < blocks_of(0, 0); b += A) keep(mem, draw(0, b, sweep0), blocks_of(0, 0), b);
    cp_wait_all();
    __syncwarp();

    for (int k = 0; k < n_sweeps; ++k) {
        const uint64_t sw = sweep0 + (uint64_t)k;
        int dJ = 0, dM = 0;
#pragma unroll 1
        for (int z = 0; z < L; ++z) {
            const uint2 *jrow = reinterpret_cast<const uint2 *>(g.J6) + z * L * L;
            const int dm = am - az, dp = ap - az;
            // per segment: the old spin of the next row to form, the new spin of
            // the row before the current one
            int own[SEG], ym[SEG];
#pragma unroll
            for (int q = 0; q < SEG; ++q) {
                own[q] = sp[az + xo[q]];
                ym[q] = sp[az + (L - 1) * PITCH + xo[q]];
            }
#pragma unroll 1
            for (int y0 = 0; y0 < L; y0 += 4) {
                const int site0 = (z * L + y0) * L;
                // the next four rows: of this plane, the next, or the next sweep
                const int y_n = y0 + 4 < L ? y0 + 4 : 0;
                const int site_n = y_n ? site0 + 4 * L : z + 1 < L ? (z + 1) * L * L : 0;
                const int blk_n = blocks_of(site_n, y_n);
                const uint64_t sw_n = site_n ? sw : sw + 1;
                int8_t *const row = sp + az + y0 * PITCH;
                const uint32_t row_a = sp_a + az + y0 * PITCH;
                const uint32_t *const rnd = buf + (site0 & 3);
                uint4 drawn[SEG];
                // The Site of row j, segment q, in two parts: the loads, and the
                // rest.  x neighbours are the old spins (a step adds what the
                // row changed), but for site L - 1 of a row of three segments,
                // whose right neighbour, site 0, is final by then.
                struct Raw {
                    uint32_t rw;
                    int zm, zp, xl, xr, up;
                    uint2 j;
                };
                auto load = [&](int j, int q) {
                    Raw r;
                    // rows past the plane's last are formed (where there is no slack,
                    // from its first row) and not used
                    const int8_t *const rj = SEG <= 2 || y0 + j < L ? row + j * PITCH : sp + az;
                    const int8_t *const ru = SEG <= 2 || y0 + j + 1 < L ? row + (j + 1) * PITCH
                                             : sp + az + (REPEAT0 ? L * PITCH : 0);
                    r.rw = rnd[j * L + xo[q]];
                    r.zm = (rj + dm)[xo[q]];
                    r.zp = (rj + dp)[xo[q]];
                    r.xl = rj[xl_o[q]];
                    r.xr = rj[xr_o[q]];
                    r.up = ru[xo[q]];
                    r.j = make_uint2(0u, 0u);
                    if (BONDS) r.j = __ldg(jrow + (y0 + j < L ? (y0 + j) * L : 0) + xo[q]);
                    return r;
                };
                auto form = [&](const Raw &r, int q) {
                    Site t;
                    t.s = own[q];
                    own[q] = r.up;
                    int xr = r.xr;
                    if (SEG > 2 && q == SEG - 1) {
                        const int er = __shfl_sync(~0u, ym[0], sbase);
                        xr = lane == last_lane ? er : xr;
                    }
                    t.u = (r.rw & 0x7FFFFFFFu) | idle[q];
                    const uint32_t sel = lut_sel(2 * t.s + 2 + (int)(r.rw >> 31));
                    t.delta = lut(kDeltaLo, kDeltaHi, sel);
                    t.d = lut(kDLo, kDHi, sel);
                    t.j = r.j.x;
                    if (BONDS) {
                        // neighbours in the order of the couplings' bytes: x + 1, x - 1,
                        // y + 1, y - 1 (left out), z + 1, z - 1 (bytes 6, 7 are zero)
                        const uint32_t lo =
                            __byte_perm(__byte_perm((uint32_t)xr, (uint32_t)r.xl, 0x0040),
                                        (uint32_t)r.up, 0x0410) & 0x00FFFFFFu;
                        const uint32_t hi = __byte_perm((uint32_t)r.zp, (uint32_t)r.zm, 0x0040);
                        t.step = -t.delta;
                        t.h = __dp4a((int)r.j.x, (int)lo, __dp4a((int)r.j.y, (int)hi, 0));
                    } else {
                        t.step = lut(kStepLo, kStepHi, sel);
                        t.h = (r.up + r.zm + r.zp) + (r.xl + xr);
                    }
                    return t;
                };
                // what a Site takes from the other lanes: issued beside the ballot
                // of the step before, since every warp-wide operation ends a
                // stretch of code that the compiler can interleave
                auto gather = [&](Site &t) {
                    t.dl = __shfl_sync(~0u, t.delta, (lane - 1) & 31);
                    t.d0 = SEG == 1 ? __shfl_sync(~0u, t.delta, sbase) : 0;
                    t.Pm = __ballot_sync(~0u, t.d > 0);
                    t.Mm = __ballot_sync(~0u, t.d < 0);
                };
                // couplings to the y - 1, x - 1 and x + 1 neighbours
                auto j_ym = [](const Site &t) { return BONDS ? (int)t.j >> 24 : 1; };
                auto j_xl = [](const Site &t) { return BONDS ? (int)(int8_t)(t.j >> 8) : 1; };
                auto j_xr = [](const Site &t) { return BONDS ? (int)(int8_t)t.j : 1; };
                Site c = form(load(0, 0), 0);
                gather(c);
                // changes of the last site of the segment before, of site 0
                int edge = 0, first = 0;
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    if (j > 0 && y0 + j >= L) break;
#pragma unroll
                    for (int q = 0; q < SEG; ++q) {
                        const int qn = q + 1 < SEG ? q + 1 : 0, jn = q + 1 < SEG ? j : j + 1;
                        Raw r;
                        if (jn < 4) r = load(jn, qn);
                        // first pass: nothing accepted before the site
                        int hh = c.h + ym[q] * j_ym(c);
                        if (SEG > 1 && q > 0) hh += (h == 0 ? edge : 0) * j_xl(c);
                        if (SEG == 2 && q == 1) hh += (lane == last_lane ? first : 0) * j_xr(c);
                        const int hk0 = c.step * hh, row0 = eo + c.d * nj;
                        const uint32_t t0 = __ldg(thr + (row0 + hk0));
                        // meanwhile the next step's Site and the next four rows'
                        // random words
                        if (j == 0) {
                            drawn[q] = draw(site_n, q * A + h, sw_n);
                            if (TWO) keep(buf1, drawn[q], blk_n, q * A + h);
                        }
                        Site n = c;
                        if (jn < 4) n = form(r, qn);
                        bool mine = c.u < t0;
                        unsigned acc = __ballot_sync(~0u, mine);
                        const bool some = __any_sync(~0u, mine);
                        if (jn < 4) gather(n);
                        edge = 0;
                        if (q == 0) first = 0;
                        int s_new = c.s;
                        if (some) {
                            // hk0 changes by cL when the left neighbour is accepted, for
                            // site L - 1 by cW when site 0 is, which the first pass
                            // decided for good
                            const int cL = c.step * c.dl * j_xl(c);
                            int hb = hk0, hk;
                            if (SEG == 1) hb += (acc & bit0) ? c.step * c.d0 * j_xr(c) : 0;
                            bool was;
                            do {
                                was = mine;
                                hk = hb + ((acc & bitL) ? cL : 0);
                                // E_Delta moves by the accepted d before the site
                                const int nd = __popc(acc & c.Pm & lower) - __popc(acc & c.Mm & lower);
                                mine = c.u < __ldg(thr + (row0 + hk + nd * trow));
                                acc = __ballot_sync(~0u, mine);
                            } while (__any_sync(~0u, mine != was));
                            // E_J changes by |delta| k h (clean), -delta h (couplings)
                            const int da = mine ? c.delta : 0;
                            dJ += BONDS ? (mine ? hk : 0) : hk * abs(da);
                            dM += da;
                            s_new += da;
                            st_shared_u8(row_a + j * PITCH + xo[q], s_new, mine);
                            if (j == 0 && REPEAT0)
                                st_shared_u8(row_a + L * PITCH + xo[q], s_new, mine && y0 == 0);
                            eo += trow * (__popc(acc & c.Pm & lanes) - __popc(acc & c.Mm & lanes));
                            if (SEG > 1 && q + 1 < SEG) edge = __shfl_sync(~0u, da, sbase + A - 1);
                            if (SEG == 2 && q == 0) first = __shfl_sync(~0u, da, sbase);
                        }
                        ym[q] = s_new;
                        c = n;
                    }
                }
                if (!TWO) {
                    __syncwarp();
#pragma unroll
                    for (int q = 0; q < SEG; ++q) keep(buf1, drawn[q], blk_n, q * A + h);
                }
                if (blk_n > SEG * A)
                    keep(buf1, draw(site_n, SEG * A + h, sw_n), blk_n, SEG * A + h);
                __syncwarp();
                // the finished rows back to the lattice, and the same rows of plane
                // z + 2 over those of plane z - 1
                if (ring) {
                    const int n = min(4, L - y0), z2 = z + 2 < L ? z + 2 : z + 2 - L;
                    if (wide) {
                        // n PITCH bytes, 16 per lane and turn
                        const ptrdiff_t o = (ptrdiff_t)(z * L + y0) * PITCH;
                        const ptrdiff_t i = (ptrdiff_t)(z2 * L + y0) * PITCH;
#pragma unroll
                        for (int t = 0; t < (SEG <= 2 ? 1 : 2); ++t) {
                            const int at = t * 16 * A;
                            const bool p = used && 16 * h + at < n * PITCH;
                            const uint4 v =
                                *reinterpret_cast<const uint4 *>(row + (p ? 16 * h + at : 0));
                            st_global_v4(lat + o + at, v, p);
                            cp16(row_a + dm + 16 * h + at, lat + i + at, p);
                            if (t == 0 && REPEAT0)
                                cp16(row_a + dm + L * PITCH + 16 * h, lat + i,
                                     used && y0 == 0 && 16 * h < PITCH);
                        }
                    } else if (used) {
                        copy.out(row, z, y0, n);
                        copy.in(row + dm, z2, y0, n);
                        if (REPEAT0 && y0 == 0) copy.in(row + dm + L * PITCH, z2, 0, 1);
                    }
                    cp_commit();
                    cp_wait_1();
                    __syncwarp();
                }
                if (TWO) {
                    uint32_t *const t = buf;
                    buf = buf1;
                    buf1 = t;
                }
            }
            // the next plane
            const int t = am;
            am = az;
            az = ap;
            ap = ring ? t : (ap + pb == L * pb ? 0 : ap + pb);
        }
        // sums over the walker's lanes
        int tJ = dJ, tM = dM;
        for (int v = 1; v < A; ++v) {
            const int src = sbase + (h + v) % A;
            tJ += __shfl_sync(~0u, dJ, src);
            tM += __shfl_sync(~0u, dM, src);
        }
        EJ += tJ;
        Mg += tM;
        if (used && h == 0) {
            const int E = eo / trow - kPad;
            const unsigned peers = __match_any_sync(lmask, E);
            if (lane == __ffs(peers) - 1)
                atomicAdd(g.hist + E, (unsigned long long)__popc(peers));
            if (record) {
                int32_t *ts = g.ts + (ts_pos + k) * 3 * (int64_t)g.W + w;
                ts[0] = EJ;
                ts[g.W] = E + g.e_min;
                ts[2 * g.W] = Mg;
            }
        }
        __syncwarp();
    }
    cp_wait_all();
    __syncwarp();
    if (used && !ring)
        for (int z = 0; z < L; ++z)
            for (int y0 = 0; y0 < L; y0 += 4)
                copy.out(sp + z * pb + y0 * PITCH, z, y0, min(4, L - y0));
    if (used && h == 0) {
        g.tal[w] = EJ;
        g.tal[g.Wpad + w] = eo / trow - kPad + g.e_min;
        g.tal[2 * g.Wpad + w] = Mg;
    }
}

template <int SEG, int PITCH, bool BONDS>
__global__ void __launch_bounds__(32, 16)
sweep_rows_kernel(const __grid_constant__ GroupDev g, int lanes, uint32_t seed, uint64_t sweep0,
                  int n_sweeps, int64_t ts_pos, int record)
{
    extern __shared__ __align__(16) uint32_t s_rows[];
    const int per_warp = 32 / lanes;
    rows_sweeps<SEG, PITCH, BONDS>(g, lanes, per_warp, (int)blockIdx.x * per_warp, s_rows, seed,
                                   sweep0, n_sweeps, ts_pos, record);
}

// The groups of one launch, in kernel parameters (32764 bytes at most; from there
// every block reads its group's values uniformly): group i's blocks are
// first[i] .. first[i + 1] - 1.  One launch for up to 128 groups of a kind: a
// launch per group keeps at most 32 of them on the GPU at a time (one per stream).
//   us per sweep of 128 groups of 32 walkers, L = 8: 66 -> 16, of 256: 132 -> 22;
//   100 groups of 8 walkers, L = 32: 905 -> 274; 24 groups of 512, L = 8 .. 32, 60
//   sweeps and merge 43.5 -> 42.1 ms
struct RowsList {
    GroupDev g[kRowsMaxGroups];
    int first[kRowsMaxGroups + 1], lanes[kRowsMaxGroups];
    int n;
};
static_assert(sizeof(RowsList) <= 32000, "kernel parameters");

template <int SEG, int PITCH, bool BONDS>
__global__ void __launch_bounds__(32, 16)
sweep_rows_list_kernel(const __grid_constant__ RowsList list, uint32_t seed, uint64_t sweep0,
                       int n_sweeps, int64_t ts_pos, int record)
{
    extern __shared__ __align__(16) uint32_t s_rows[];
    // the last group with first <= block
    int i = 0;
#pragma unroll
    for (int step = kRowsMaxGroups / 2; step > 0; step /= 2)
        i += i + step < list.n && list.first[i + step] <= (int)blockIdx.x ? step : 0;
    const int per_warp = 32 / list.lanes[i];
    rows_sweeps<SEG, PITCH, BONDS>(list.g[i], list.lanes[i], per_warp,
                                   ((int)blockIdx.x - list.first[i]) * per_warp, s_rows, seed,
                                   sweep0, n_sweeps, ts_pos, record);
}

}  // namespace

// Segments of rows of 33 to 48 sites, for all the walkers with such rows that are
// swept together.  Two segments are one walker per warp; three, of up to 16
// lanes, two walkers per warp, so half the warps, each slower (a step's passes
// go on to the slower walker's last).  Two while the GPU holds all the walkers at
// once (16 warps per SM); beyond that neither is ahead everywhere.
// us per sweep, L = 48, T = 1, two and three segments:
//   transition weights: 640 walkers 1398, 2521;  2048 1924, 3382;  4096 3699, 3963
//   weights soon after a random start: 4096 walkers 2110, 1930
// Rows of more than 48 sites are two segments, however many walkers there are (L = 64,
// transition weights: 1024 walkers 3.46 ms a sweep, 4096 8.3; in four segments
// 7.42 and 9.6).
int rows_long_segments(int64_t walkers)
{
    int dev = 0, nsm = 152;
    if (cudaGetDevice(&dev) == cudaSuccess)
        (void)cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    return walkers <= (int64_t)16 * nsm ? 2 : 3;
}

RowShape rows_shape(int L, int long_seg)
{
    RowShape s{0, 0, 0};
    if (L < 3 || L > 64) return s;
    s.seg = L <= 32 ? 1 : L <= 48 ? long_seg : 2;
    s.lanes = (L + s.seg - 1) / s.seg;
    s.per_warp = 32 / s.lanes;
    return s;
}

// Bytes between a walker's rows in shared memory, and in the lattice of a group
// kept walker by walker whose planes pass through it (rows_lattice_words).
static int rows_pitch(int L) { return L <= 16 ? 16 : L <= 32 ? 32 : L <= 48 ? 48 : 64; }

int rows_lattice_words(int L) { return L > 12 ? rows_pitch(L) / 4 : (L + 3) / 4; }

static size_t rows_bytes_for(int L, const RowShape &s)
{
    return (size_t)s.per_warp * rows_walker_words(L, s.seg, s.per_warp, rows_pitch(L)) *
           sizeof(uint32_t);
}

namespace {
template <int SEG, int PITCH, bool BONDS>
void launch(const GroupDev *const *g, const RowShape *sh, int n, size_t smem, uint32_t seed,
            uint64_t sweep0, int n_sweeps, int64_t ts_pos, int rec, cudaStream_t st)
{
    auto blocks = [&](int i) { return (g[i]->W + sh[i].per_warp - 1) / sh[i].per_warp; };
    if (n == 1) {
        sweep_rows_kernel<SEG, PITCH, BONDS><<<blocks(0), 32, smem, st>>>(
            *g[0], sh[0].lanes, seed, sweep0, n_sweeps, ts_pos, rec);
        return;
    }
    RowsList list;
    list.n = n;
    list.first[0] = 0;
    for (int i = 0; i < n; ++i) {
        list.g[i] = *g[i];
        list.lanes[i] = sh[i].lanes;
        list.first[i + 1] = list.first[i] + blocks(i);
    }
    sweep_rows_list_kernel<SEG, PITCH, BONDS><<<list.first[n], 32, smem, st>>>(
        list, seed, sweep0, n_sweeps, ts_pos, rec);
}
}  // namespace

int rows_kind(const GroupDev &g)
{
    return (rows_shape(g.L, g.rows_seg).seg * 100 + rows_pitch(g.L)) * 2 + (g.jmax > 0);
}

cudaError_t launch_sweeps_rows(const GroupDev *const *g, int n, uint32_t seed, uint64_t sweep0,
                               int n_sweeps, int64_t ts_pos, bool record, cudaStream_t st)
{
    if (n_sweeps <= 0) return cudaSuccess;
    if (n < 1 || n > kRowsMaxGroups) return cudaErrorInvalidValue;
    RowShape sh[kRowsMaxGroups];
    size_t smem = 0;  // at most 16 KB: no opt-in
    const int kind = rows_kind(*g[0]);
    for (int i = 0; i < n; ++i) {
        sh[i] = rows_shape(g[i]->L, g[i]->rows_seg);
        if (sh[i].seg == 0 || rows_kind(*g[i]) != kind) return cudaErrorInvalidValue;
        smem = std::max(smem, rows_bytes_for(g[i]->L, sh[i]));
    }
    const int rec = record ? 1 : 0;
    switch (kind) {
#define MUCA_ROWS_LAUNCH(S, P)                                                                \
    case (S * 100 + P) * 2:                                                                   \
        launch<S, P, false>(g, sh, n, smem, seed, sweep0, n_sweeps, ts_pos, rec, st);         \
        break;                                                                                \
    case (S * 100 + P) * 2 + 1:                                                               \
        launch<S, P, true>(g, sh, n, smem, seed, sweep0, n_sweeps, ts_pos, rec, st);          \
        break;
        MUCA_ROWS_LAUNCH(1, 16)
        MUCA_ROWS_LAUNCH(1, 32)
        MUCA_ROWS_LAUNCH(2, 48)
        MUCA_ROWS_LAUNCH(2, 64)
        MUCA_ROWS_LAUNCH(3, 48)
#undef MUCA_ROWS_LAUNCH
        default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

}  // namespace muca
