// Block product over GF(p): C = A B mod p, A m x k, B k x nb (row-major
// uint32 residues), the dense contraction at the heart of block methods.
//
// Tensor-core path (p <= 65791, the centred residues of Section 3.2.2 then
// fit two balanced 8-bit digits):
//   a in [0, p) is centred to s in [-(p-1)/2, (p-1)/2] and split exactly as
//   s = 256 h + l with l in [-128, 127], h in [-128, 128].  Every digit is an
//   exact fp16 value and every digit product is an integer of magnitude at
//   most 2^14.  The digit products go through tcgen05.mma kind::f16 into fp32
//   accumulators in TMEM, three per output: hh, hl + lh and ll.  The middle
//   one takes two products per term, so 512 terms sum to at most 2^24: exact
//   (Eq. (1) read with m = 24 for the fp32 significand).  After each such
//   chunk the accumulators are recombined as (hh 256 + (hl + lh)) 256 + ll mod
//   p and added to the output's residue sum.  Nothing is approximated.
//
//   A work unit is one 128-row tile of A times one K range of at most 512
//   terms (eight 64-deep k-blocks) of one 64-column tile of B.  Units are
//   ordered with the row tiles innermost and split evenly over one persistent
//   CTA per SM, so a CTA works through many row tiles against the same K
//   range: that range's B digits (128 KiB) are copied to shared memory once and
//   stay, and A alone streams.  A's digits go to TMEM, from where
//   the MMAs read them: shared memory sees only B, and the rest of its 256 KiB
//   per SM stays L1, which is where loads in flight land.  Roles per CTA:
//     warps 0-15   load A with 16-byte loads (64 KiB in flight per SM), centre
//                  and split the words in registers and store the fp16 digits
//                  (tcgen05.st) to TMEM: two groups of eight warps with a slot
//                  each take alternate k-blocks.  No warp waits for another:
//                  slots pass through mbarriers alone
//     warps 16-23  drain the accumulators (tcgen05.ld), recombine, reduce and
//                  add the residues to the partial sums
//     warp 24      owns TMEM and issues the MMAs
//     warp 25      bulk-copies B's digit tiles, split once by a small kernel
//                  before this one, each as soon as the MMAs of the K range
//                  before have read its place for the last time
//   The residues of a unit are added to a u32 workspace, two columns in one
//   64-bit addition, and a small kernel behind this one reduces the sums mod p,
//   writes C through a shared-memory transpose and clears the workspace; a product
//   with a single K range writes C directly.
//
//   What bounds it (16384 x 16384 x 64 over GF(65521), calls back to back, before
//   -> now; before: A through in-place shared-memory slots, B's tiles re-read for
//   every row tile):  uint32 A 215 -> 176 us, HBM at 6.1 TB/s of the 6.5-7.0 that
//   loads in this pattern reach alone; prepared A 172 -> 128 us, the hand-over of
//   TMEM slots between converters and MMAs (0.5 us per k-block against 0.37 us of
//   HBM).  In the order they were taken, with a flushed L2
//   (uint32 / prepared): digits in shared-memory slots beside the resident B
//   366 / 304 us (28 KiB of L1 left: the loads in flight did not fit), digits in
//   TMEM 253 / 206, fewer instructions per k-block 213 / 177, B's tiles split by a
//   kernel of its own instead of by each CTA 201 / 156, MMAs issued from a converged
//   warp 196 / 135, two converter groups 184 / 114, 64-bit additions 185 / 111.
//   Not kept: half-k-block hand-overs (125 prepared), a look ahead at the next
//   slot's barrier (116), L2 prefetch of the next unit (197 uint32), 32-byte loads
//   (186), more half k-blocks in registers (199 / 121), remainders of the drain in
//   fp32 (117 prepared).
//
// Larger moduli on the tensor cores (p > 65791): the exact integer products
// sum_t A[i][t] B[t][j] are below k (p-1)^2, so they are fixed by their
// residues modulo a few small primes p' <= 65536 whose product exceeds that
// bound (a residue number system).  Each pass runs the tensor-core kernel
// above modulo one p', reducing every input a < 2^32 to a mod p' while it is
// split into digits (B's digits for all passes are made by one launch); a last
// kernel recombines the residues with Garner's mixed-radix method and evaluates
// the integer modulo p.
//
// CUDA-core path (any p <= 2^32-1): shared-memory tiled product with the
// per-thread unreduced accumulators of the dot-product kernels.
#include <cuda_fp16.h>

#include <algorithm>
#include <atomic>
#include <cstring>
#include <mutex>

#include "gfp_internal.h"
#include "gfp_tc.cuh"

namespace gfp {
namespace blk {

constexpr int BM = 128;            // rows per tile (MMA M)
constexpr int BK = 64;             // K per k-block: one 128-byte swizzle row of fp16
constexpr int NT = 64;             // output columns per n-tile
constexpr int B_ROWS = 2 * NT;     // low and high digits of B, one below the other
constexpr int RK = 8;              // k-blocks per K range at most: 512 terms, the exact chunk
constexpr int B_TILE_BYTES = B_ROWS * BK * 2;                 // 16 KiB
// A's digits live in TMEM: two slots of one k-block each
constexpr int SLOTS = 2;
constexpr uint32_t SLOT_COLS = 64;                            // 32 columns per digit
constexpr uint32_t ACC_COLS = 3 * NT;                         // ll, middle, hh
constexpr uint32_t A_COL0 = 2 * ACC_COLS;                     // behind two accumulator sets
constexpr int CONV_GROUPS = 2, CONV_WARPS = 8, EPI_WARPS = 8;   // converter warps of a group
constexpr int W_EPI0 = CONV_GROUPS * CONV_WARPS, W_MMA = W_EPI0 + EPI_WARPS, W_BPROD = W_MMA + 1;
static_assert(CONV_GROUPS == SLOTS, "each group has a slot of its own");
constexpr int THREADS = 32 * (W_MMA + 4);                     // 896: two warps of the last group idle
// registers per thread: 72 at launch, then shared out by role (warpgroups)
constexpr int REGS_LAUNCH = 72, REGS_CONV = 88, REGS_EPI = 56, REGS_MMA = 40;
static_assert(REGS_LAUNCH * THREADS ==
                  32 * (REGS_CONV * CONV_GROUPS * CONV_WARPS + REGS_EPI * EPI_WARPS + REGS_MMA * 4),
              "the roles' registers are exactly those the block is launched with");
static_assert(REGS_LAUNCH * THREADS <= 65536, "one CTA per SM");
static_assert(W_EPI0 % 4 == 0 && W_MMA % 4 == 0, "the shares go to whole warpgroups");
static_assert(W_EPI0 % 4 == 0, "an epilogue warp reads the TMEM lanes of its index modulo 4");
constexpr uint32_t TMEM_COLS = 512;
static_assert(A_COL0 + SLOTS * SLOT_COLS == TMEM_COLS, "accumulators and A digits fill TMEM");
constexpr uint64_t WAIT_NS = 2000000000ull;   // bounded waits: 2 s
// Every MMA is 128 x 64 x 16 and adds into one of three accumulators that do not
// overlap: MMAs in flight are ordered among themselves only where accumulator and
// shape are the same, and the middle sum takes two MMAs per 16 K.  (One 128-wide
// MMA for each digit of A, over ll | middle and middle | hh, took 108.6 us for the
// prepared 16384 x 16384 x 64 against 122.5 us, the same for uint32 A; its middle
// sum would rest on an order that nothing promises.)
constexpr uint32_t IDESC = ptx::idesc_f16_f32(BM, NT);
constexpr uint64_t B_HIGH = (NT * 128) >> 4;   // from a tile's low to its high digits, in descriptor units
// terms of one launch: 2^24 / 512 partial sums below p <= 65791, and one more
// (the sums of earlier launches, folded below p), stay below 2^32
constexpr uint64_t SLAB_K = 1ull << 24;

struct Bars {
    uint64_t conv[SLOTS];      // digits of a slot written (one arrival per converter warp)
    uint64_t a_empty[SLOTS];   // MMAs reading the slot completed (tcgen05.commit)
    uint64_t b_full[RK];       // B digit tile landed (1 arrival + tx bytes)
    uint64_t b_empty[RK];      // last MMAs reading the tile completed (tcgen05.commit)
    uint64_t acc_full[2];      // accumulator set ready (tcgen05.commit)
    uint64_t acc_empty[2];     // accumulator set drained (one arrival per epilogue warp)
    uint64_t drain;            // all MMAs issued by this CTA completed
    uint32_t tmem_base;
    uint32_t abort;
};
constexpr size_t SMEM_BYTES = 1024 /*alignment slack*/ + (size_t)RK * B_TILE_BYTES + 1024;
static_assert(sizeof(Bars) <= 1024, "barriers fit their reserve");
static_assert(SMEM_BYTES <= 232448, "shared memory per block");

// How A arrives: uint32 rows that 16-byte loads can take, uint32 rows of any
// alignment, or prepared 8-bit digit planes.
enum AMode : int { A_VEC = 0, A_ANY = 1, A_PREP = 2 };

// Prepared A (gfp_block_prepare): per (m-tile, k-block) the 8-bit digits of
// 128 rows x 64 K, in the order the converter lanes of the product take them:
// for each of the eight converter warps 1 KiB of high and 1 KiB of low
// digits, 16 bytes a lane at a time (AWords), every digit stored with a bias of 128.  A
// residue a of p <= 65536 is represented by s = a or a - p in
// [-32896, 32639] (s = a when a <= min((p-1)/2, 32639)), split as
// s = 256 h + l with h, l in [-128, 127]: u = s + 32896 in [0, 65535] holds
// h + 128 in its high byte and l + 128 in its low byte.  Every digit is still
// at most 128 in magnitude, so the 512-term fp32 chunks stay exact.
constexpr int A8_TILE_BYTES = 2 * BM * BK;        // 16 KiB per (m-tile, k-block)
constexpr uint32_t DIGIT8_MAX_P = 65536;

struct Args {
    uint64_t m, k, nb;        // k: terms of this launch
    const uint32_t *A;
    uint64_t lda;
    const uint8_t *Aimg;      // prepared A: [m_tiles][img_kblocks] tiles of A8_TILE_BYTES
    uint32_t img_kblocks, img_kb0;   // k-blocks of the whole image, first one of this launch
    const uint8_t *Bimg;      // [n_tiles][kblocks] tiles of B_TILE_BYTES
    uint32_t *C;
    uint64_t ldc;
    uint32_t *Cacc;           // (n_tiles*NT) x m u32 partial residue sums, by pairs of columns:
                              // row i of columns 2 j and 2 j + 1 at 2 (j m + i) and the next
                              // word (zero outside calls)
    uint32_t *err;            // bit 0: a bounded wait expired
    uint32_t p, half;         // half = (p-1)/2
    uint32_t magic;           // floor(2^32 / p)
    int32_t smagic;           // the same, at most 2^31 - 1
    uint32_t magic47;         // floor(2^47 / p) of a residue-pass modulus (p > 65000)
    uint32_t backward;        // each CTA takes its units in reverse order
    uint32_t direct;          // one K range: residues go to C, not to the workspace
    uint32_t m_tiles, n_tiles, kblocks;
    uint32_t ranges, r_base, r_rem;   // K ranges of r_base k-blocks, the first r_rem one more
    uint32_t bsets;           // K ranges whose B tiles fit the RK tiles at once,
    uint32_t bset_tiles;      // the distance between their tiles
    uint32_t edge_m, edge_k;  // last row tile, last k-block where ragged (else none: ~0)
    uint64_t units;
};

// Bounded wait on an mbarrier phase: gives up after limit_ns (or as soon as
// another role of the CTA has given up), sets the CTA abort flag and bit 0 of
// the error word, and returns false.
__device__ __forceinline__ bool wait_bar(uint32_t bar, uint32_t parity, volatile uint32_t *abort,
                                         uint32_t *err, uint64_t limit_ns = WAIT_NS)
{
    uint64_t t0 = 0;
    for (uint32_t i = 0;; ++i) {
        if (ptx::mbar_try_wait(bar, parity)) return true;
        if ((i & 255u) == 255u) {
            if (*abort) return false;
            const uint64_t t = ptx::globaltimer();
            if (t0 == 0) t0 = t;
            else if (t - t0 > limit_ns) {
                *abort = 1u;
                atomicOr(err, 1u);
                return false;
            }
        }
    }
}

// The same for a converged warp: every lane polls (a lone polling lane adds
// the cost of leaving and rejoining the warp, 506 against 318 cycles for a
// hand-over of 16 warps to one and back), and all lanes agree on the result.
__device__ __forceinline__ bool wait_bar_warp(uint32_t bar, uint32_t parity, volatile uint32_t *abort,
                                              uint32_t *err)
{
    return __all_sync(0xffffffffu, wait_bar(bar, parity, abort, err));
}

// Failure-detection self test: one thread waits on an mbarrier that nothing
// arrives on; the bounded wait must expire and report it in *err.
__global__ void k_wait_selftest(uint64_t limit_ns, uint32_t *err)
{
    __shared__ __align__(8) uint64_t bar;
    __shared__ uint32_t abort;
    if (threadIdx.x == 0) {
        ptx::mbar_init(ptx::smem_u32(&bar), 1);
        abort = 0;
        ptx::fence_barrier_init();
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        if (!wait_bar(ptx::smem_u32(&bar), 0, &abort, err, limit_ns)) atomicOr(err, 2u);
    }
}

__device__ uint32_t g_selftest_err;

// Walks a CTA's units in order (row tiles innermost, then K ranges, then
// column tiles), or backwards.
struct Walk {
    uint32_t mt, rg, nt;
    uint32_t kb0, kbs;   // first k-block and number of k-blocks of the K range
    uint32_t left;       // units not finished, the current one included
    __device__ __forceinline__ void range(const Args &a)
    {
        kb0 = rg * a.r_base + min(rg, a.r_rem);
        kbs = a.r_base + (rg < a.r_rem ? 1u : 0u);
    }
    __device__ __forceinline__ void start(const Args &a, uint64_t u0, uint64_t u1)
    {
        const uint64_t u = a.backward ? u1 - 1 : u0;
        left = (uint32_t)(u1 - u0);
        mt = (uint32_t)(u % a.m_tiles);
        const uint64_t t = u / a.m_tiles;
        rg = (uint32_t)(t % a.ranges);
        nt = (uint32_t)(t / a.ranges);
        range(a);
    }
    // the last of its K range's units, in walking order
    __device__ __forceinline__ bool last_of_range(const Args &a) const
    {
        return left == 1 || (a.backward ? mt == 0 : mt + 1 == a.m_tiles);
    }
    // to the next unit; true when its K range or column tile is another one
    __device__ __forceinline__ bool next(const Args &a)
    {
        const bool turn = last_of_range(a);
        --left;
        if (!turn) {
            mt += a.backward ? ~0u : 1u;
            return false;
        }
        if (!a.backward) {
            mt = 0;
            if (++rg == a.ranges) {
                rg = 0;
                ++nt;
            }
        } else {
            mt = a.m_tiles - 1;
            if (rg-- == 0) {
                rg = a.ranges - 1;
                --nt;
            }
        }
        range(a);
        return true;
    }
};

// Two values u = s + 32896 (s the representative, in [-32896, 32895]) to the
// balanced 8-bit digits l = (u & 255) - 128 and h = (u >> 8) - 128 of
// s = 256 h + l, as packed fp16 pairs (element 0 in the low half).  The fp16
// encoding of 1024 + b for an integer 0 <= b <= 256 is the 16-bit integer
// 0x6400 + b, so with U_BIAS added to u (0x64 in its two upper bytes; u = 2^16
// and above carries into the lower of them, as 0x6400 + 256 wants it) one byte
// permute builds 1024 + b for both lanes and one exact fp16 subtraction of
// 1152 leaves the digits.
constexpr uint32_t U_BIAS = 0x64640000u + 32896u;

__device__ __forceinline__ uint32_t sub_half2(uint32_t x, uint32_t half_bits)
{
    const __half2 b = __halves2half2(__ushort_as_half((unsigned short)half_bits),
                                     __ushort_as_half((unsigned short)half_bits));
    const __half2 r = __hsub2(*reinterpret_cast<const __half2 *>(&x), b);
    return *reinterpret_cast<const uint32_t *>(&r);
}

__device__ __forceinline__ void split_u(uint32_t u0, uint32_t u1, uint32_t &hi2, uint32_t &lo2)
{
    lo2 = sub_half2(__byte_perm(u0, u1, 0x7430), 0x6480u);   // bytes 0 and 3 of each
    hi2 = sub_half2(__byte_perm(u0, u1, 0x6521), 0x6480u);   // bytes 1 and 2 of each
}

// a mod p for any 32-bit a and p <= 65791: q = floor(a * floor(2^32/p) / 2^32)
// is floor(a/p) or one less, so one conditional subtraction finishes it
__device__ __forceinline__ uint32_t reduce_small(uint32_t a, uint32_t p, uint32_t magic)
{
    const uint32_t r = a - __umulhi(a, magic) * p;
    return min(r, r - p);
}

// u = s + U_BIAS for the centred representative s of a residue a < p
__device__ __forceinline__ uint32_t centre_u(uint32_t a, const Args &g)
{
    return a + (a > g.half ? U_BIAS - g.p : U_BIAS);
}

// u = s + U_BIAS with s = a (mod p) for any 32-bit a and a residue-pass modulus
// 65000 < p < 65536: q = a / p rounded to nearest from the quotient to 15
// fractional bits.  That quotient is low by less than two units of 2^-15
// (magic47 by less than one part in 2^31, the multiply-high by less than one
// unit), so |s| <= p/2 + 2 p / 32768 < 32896 - 100.
__device__ __forceinline__ uint32_t reduce_u(uint32_t a, const Args &g)
{
    const uint32_t q = (__umulhi(a, g.magic47) + 16384u) >> 15;
    return a + U_BIAS - q * g.p;
}

template <bool PRE>
__device__ __forceinline__ void split4(const uint4 &w, const Args &a, uint32_t &hi01, uint32_t &hi23,
                                       uint32_t &lo01, uint32_t &lo23)
{
    const uint32_t u0 = PRE ? reduce_u(w.x, a) : centre_u(w.x, a);
    const uint32_t u1 = PRE ? reduce_u(w.y, a) : centre_u(w.y, a);
    const uint32_t u2 = PRE ? reduce_u(w.z, a) : centre_u(w.z, a);
    const uint32_t u3 = PRE ? reduce_u(w.w, a) : centre_u(w.w, a);
    split_u(u0, u1, hi01, lo01);
    split_u(u2, u3, hi23, lo23);
}

// Four biased 8-bit digits to fp16 pairs: a byte b under 0x64 is 1024 + b
__device__ __forceinline__ void widen4(uint32_t w, uint32_t &d01, uint32_t &d23)
{
    d01 = sub_half2(__byte_perm(w, 0x64646464u, 0x4140), 0x6480u);
    d23 = sub_half2(__byte_perm(w, 0x64646464u, 0x4342), 0x6480u);
}

// What one converter lane holds of a k-block of A.  Warp w writes the TMEM
// lanes (rows) 32 (w mod 4) + 16 (w / 4) .. + 15; with the 16x256b store shape
// lane l holds, per 16 K, four consecutive K (l mod 4) of rows l / 4 and
// l / 4 + 8.  v[i] are those pieces: K group i / 2, row l / 4 + 8 (i mod 2); for
// uint32 A 16 bytes each (the four groups of a row are 256 consecutive bytes),
// for a prepared A the four bytes of one word: v[0], v[1] the high digits of K
// groups 0, 1 and 2, 3, v[2], v[3] the low ones.  Rows and columns outside the
// matrix are zero.
template <int MODE>
struct AWords {
    uint4 v[MODE == A_PREP ? 4 : 8];
};

// Runs ahead of the conversion: where the next k-block's words are.
template <int MODE, bool PRE>
struct ALoads {
    Walk w;
    uint32_t j;           // k-block within the K range
    const uint8_t *src;   // this lane's first piece of that k-block
    bool end;             // no k-block left
    static constexpr uint32_t STRIDE = MODE == A_PREP ? A8_TILE_BYTES : BK * 4;
    __device__ __forceinline__ void locate(const Args &a, int warp, int lane)
    {
        if constexpr (MODE == A_PREP) {
            src = a.Aimg + ((uint64_t)w.mt * a.img_kblocks + a.img_kb0 + w.kb0 + j) * A8_TILE_BYTES + warp * 2048 +
                  lane * 16;
        } else {
            const uint64_t row = (uint64_t)w.mt * BM + (warp & 3) * 32 + (warp >> 2) * 16 + (lane >> 2);
            const uint64_t col = (uint64_t)(w.kb0 + j) * BK + (lane & 3) * 4;
            src = reinterpret_cast<const uint8_t *>(a.A + row * a.lda + col);
        }
    }
    // n k-blocks on
    __device__ __forceinline__ void advance(const Args &a, int warp, int lane, uint32_t n)
    {
        j += n;
        if (j < w.kbs) {
            src += n * STRIDE;
            return;
        }
        do {
            j -= w.kbs;
            if (w.left <= 1) {
                end = true;
                return;
            }
            w.next(a);
        } while (j >= w.kbs);
        locate(a, warp, lane);
    }
    __device__ __forceinline__ void load(const Args &a, int warp, int lane, AWords<MODE> &r) const
    {
        if constexpr (MODE == A_PREP) {
#pragma unroll
            for (int i = 0; i < 4; ++i) ptx::ld_stream4(r.v[i], src + i * 512);
        } else if (w.mt != a.edge_m && w.kb0 + j != a.edge_k) {
            const uint8_t *src8 = src + 32 * a.lda;   // eight rows further
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const uint8_t *q = ((i & 1) ? src8 : src) + (i >> 1) * 64;
                if constexpr (MODE == A_VEC) {
                    // a residue pass leaves A in L2 for the pass behind it
                    if constexpr (PRE) ptx::ld_l2_4(r.v[i], q);
                    else ptx::ld_stream4(r.v[i], q);
                } else {
                    const uint32_t *q1 = reinterpret_cast<const uint32_t *>(q);
                    ptx::ld_if(r.v[i].x, q1, true);
                    ptx::ld_if(r.v[i].y, q1 + 1, true);
                    ptx::ld_if(r.v[i].z, q1 + 2, true);
                    ptx::ld_if(r.v[i].w, q1 + 3, true);
                }
            }
        } else {
            const uint64_t row = (uint64_t)w.mt * BM + (warp & 3) * 32 + (warp >> 2) * 16 + (lane >> 2);
            const uint64_t col = (uint64_t)(w.kb0 + j) * BK + (lane & 3) * 4;
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const uint32_t *q = reinterpret_cast<const uint32_t *>(src + (i & 1) * 32 * a.lda + (i >> 1) * 64);
                const uint64_t c = col + (i >> 1) * 16;
                // columns of this piece inside A
                const uint64_t n = row + 8 * (i & 1) < a.m && c < a.k ? a.k - c : 0;
                r.v[i] = make_uint4(0u, 0u, 0u, 0u);
                ptx::ld_if(r.v[i].x, q, n > 0);
                ptx::ld_if(r.v[i].y, q + 1, n > 1);
                ptx::ld_if(r.v[i].z, q + 2, n > 2);
                ptx::ld_if(r.v[i].w, q + 3, n > 3);
            }
        }
    }
};

// Splits (or widens) the lane's words into the digits of its 16 rows x 64 K,
// in the order of the 16x256b store
template <int MODE, bool PRE>
__device__ __forceinline__ void convert_a(const Args &a, const AWords<MODE> &r, uint32_t (&hi)[16],
                                          uint32_t (&lo)[16])
{
    if constexpr (MODE == A_PREP) {
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            widen4(r.v[i].x, hi[8 * i], hi[8 * i + 1]);
            widen4(r.v[i].y, hi[8 * i + 2], hi[8 * i + 3]);
            widen4(r.v[i].z, hi[8 * i + 4], hi[8 * i + 5]);
            widen4(r.v[i].w, hi[8 * i + 6], hi[8 * i + 7]);
            widen4(r.v[2 + i].x, lo[8 * i], lo[8 * i + 1]);
            widen4(r.v[2 + i].y, lo[8 * i + 2], lo[8 * i + 3]);
            widen4(r.v[2 + i].z, lo[8 * i + 4], lo[8 * i + 5]);
            widen4(r.v[2 + i].w, lo[8 * i + 6], lo[8 * i + 7]);
        }
    } else {
#pragma unroll
        for (int i = 0; i < 8; ++i)
            split4<PRE>(r.v[i], a, hi[2 * i], hi[2 * i + 1], lo[2 * i], lo[2 * i + 1]);
    }
}

// PRE: reduce each entry of A modulo p while splitting it (the residue passes).
template <int MODE, bool PRE>
__global__ void __launch_bounds__(THREADS, 1) k_block_tc(const __grid_constant__ Args a)
{
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint8_t *btiles = smem;                                    // RK digit tiles of B
    Bars *bars = reinterpret_cast<Bars *>(btiles + (size_t)RK * B_TILE_BYTES);
    // one lane's value for the whole warp: the compiler may then keep what
    // depends on it in uniform registers, where tcgen05 takes its addresses from
    const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;

    const uint64_t u0 = a.units * blockIdx.x / gridDim.x;
    const uint64_t u1 = a.units * (blockIdx.x + 1) / gridDim.x;

    if (threadIdx.x == 0) {
        for (int s = 0; s < SLOTS; ++s) {
            ptx::mbar_init(ptx::smem_u32(&bars->conv[s]), CONV_WARPS);
            ptx::mbar_init(ptx::smem_u32(&bars->a_empty[s]), 1);
        }
        for (int t = 0; t < RK; ++t) {
            ptx::mbar_init(ptx::smem_u32(&bars->b_full[t]), 1);
            ptx::mbar_init(ptx::smem_u32(&bars->b_empty[t]), 1);
        }
        for (int b = 0; b < 2; ++b) {
            ptx::mbar_init(ptx::smem_u32(&bars->acc_full[b]), 1);
            ptx::mbar_init(ptx::smem_u32(&bars->acc_empty[b]), EPI_WARPS);
        }
        ptx::mbar_init(ptx::smem_u32(&bars->drain), 1);
        bars->abort = 0;
        ptx::fence_barrier_init();
    }
    if (warp == W_MMA) {
        ptx::tmem_alloc(ptx::smem_u32(&bars->tmem_base), TMEM_COLS);
        ptx::tmem_relinquish();
    }
    ptx::tc_fence_before();
    __syncthreads();
    ptx::tc_fence_after();
    const uint32_t tmem = __shfl_sync(0xffffffffu, bars->tmem_base, 0);   // uniform, as above
    volatile uint32_t *abort = &bars->abort;
    // registers by role, each share by one instruction for all warps of a
    // warpgroup (the .aligned form wants that), so ahead of the roles: the last
    // warpgroup holds several
    if (warp < W_EPI0) ptx::regs_inc<REGS_CONV>();
    else if (warp < W_MMA) ptx::regs_dec<REGS_EPI>();
    else ptx::regs_dec<REGS_MMA>();
    // Programmatic dependent launch: this grid may be placed, and sets itself up,
    // while the previous kernel of the stream, the one that makes B's digits or
    // reduces the partial sums of the pass before, is still running.  What it and
    // the kernels before it wrote is visible behind griddepcontrol.wait only, so
    // every role that touches global memory starts with it.  (Converters that load
    // A ahead of it, on the ground that A's writer completed before the previous
    // kernel went on, gained 0.6 of 174 us and nothing of 20 us; one wait ahead of
    // the roles made the compiler spill, 750 us.)

    if (warp < W_EPI0) {
        // ---------------- converters: A to fp16 digits ----------------
        // each group takes every second k-block: while one waits for its slot's
        // MMAs the other converts
        const int group = warp / CONV_WARPS, gw = warp % CONV_WARPS;
        // k-blocks in flight in registers: 64 KiB per SM over both groups
        constexpr int D = MODE == A_PREP ? 2 : 1;
        AWords<MODE> buf[D];
        ALoads<MODE, PRE> ld;
        ld.w.start(a, u0, u1);
        ld.j = 0;
        ld.end = false;
        ld.locate(a, gw, lane);
        if (group) ld.advance(a, gw, lane, 1);
        uint32_t loaded = 0;
        asm volatile("griddepcontrol.wait;" ::: "memory");
#pragma unroll
        for (int d = 0; d < D; ++d) {
            if (!ld.end) {
                ld.load(a, gw, lane, buf[d]);
                ld.advance(a, gw, lane, CONV_GROUPS);
                ++loaded;
            }
        }
        const uint32_t tslot = tmem + A_COL0 + (uint32_t)group * SLOT_COLS +
                               ((uint32_t)((gw & 3) * 32 + (gw >> 2) * 16) << 16);
        const uint32_t bar_empty = ptx::smem_u32(&bars->a_empty[group]), bar_conv = ptx::smem_u32(&bars->conv[group]);
        uint32_t ph = 1;
        bool run = true;
        while (run) {
#pragma unroll
            for (int d = 0; d < D; ++d) {
                if (loaded == 0) {
                    run = false;
                    break;
                }
                uint32_t hi[16], lo[16];
                convert_a<MODE, PRE>(a, buf[d], hi, lo);
                if (!ld.end) {
                    ld.load(a, gw, lane, buf[d]);
                    ld.advance(a, gw, lane, CONV_GROUPS);
                } else {
                    --loaded;
                }
                if (!wait_bar_warp(bar_empty, ph, abort, a.err)) {
                    run = false;
                    break;
                }
                ptx::tc_fence_after();
                ptx::tmem_st_16x256b_x4(tslot, hi);
                ptx::tmem_st_16x256b_x4(tslot + SLOT_COLS / 2, lo);
                ptx::tmem_st_wait();
                ptx::tc_fence_before();
                __syncwarp();
                if (lane == 0) ptx::mbar_arrive(bar_conv);
                ph ^= 1u;
            }
        }
    } else if (warp == W_MMA) {
        // ---------------- MMA issue ----------------
        // The whole warp walks the loop, so that addresses and descriptors stay
        // in uniform registers, and one elected lane issues: with a lone lane in
        // the loop every operand of every MMA was moved there first, and the
        // eight MMAs of a k-block took 750-1000 cycles to issue against the 503
        // they need
        const uint32_t lead = ptx::elect_one();
        Walk w;
        w.start(a, u0, u1);
        uint32_t s = 0, ph = 0, bset = 0, used = 0, b = 0, bph = 1;
        bool ok = true, fresh = true;   // fresh: the K range's first unit
        while (w.left && ok) {
            // the accumulator set was drained by the unit before the last
            if (!wait_bar_warp(ptx::smem_u32(&bars->acc_empty[b]), bph, abort, a.err)) break;
            ptx::tc_fence_after();
            const uint32_t d_ll = tmem + b * ACC_COLS, d_md = d_ll + NT, d_hh = d_md + NT;
            const bool final = w.last_of_range(a);
            uint32_t t = bset * a.bset_tiles;
            uint64_t db = ptx::sdesc_k_sw128(ptx::smem_u32(btiles + t * B_TILE_BYTES));
            for (uint32_t j = 0; j < w.kbs; ++j, ++t, db += B_TILE_BYTES >> 4) {
                ok = wait_bar_warp(ptx::smem_u32(&bars->conv[s]), ph, abort, a.err);
                if (ok && fresh) {
                    ok = wait_bar_warp(ptx::smem_u32(&bars->b_full[t]), (used >> t) & 1u, abort, a.err);
                    used ^= 1u << t;
                }
                if (!ok) break;
                ptx::tc_fence_after();
                const uint32_t ah = tmem + A_COL0 + s * SLOT_COLS, al = ah + SLOT_COLS / 2;
                // 16 K: eight TMEM columns of A, 32 bytes of B inside the swizzle atom.
                // Two such steps an accumulator at a time: 122.5 us for the prepared
                // 16384 x 16384 x 64, one at a time 125.3, four 141.2
#pragma unroll
                for (uint32_t kk = 0; kk < 4; kk += 2) {
                    const uint32_t more = kk || j ? 1u : 0u;
                    const auto two = [&](uint32_t d, uint32_t at, uint64_t bd, uint32_t accumulate) {
                        ptx::mma_f16_ts(lead, d, at + 8 * kk, bd + 2 * kk, IDESC, accumulate);
                        ptx::mma_f16_ts(lead, d, at + 8 * kk + 8, bd + 2 * kk + 2, IDESC, 1u);
                    };
                    two(d_ll, al, db, more);
                    two(d_md, al, db + B_HIGH, more);
                    two(d_md, ah, db, 1u);
                    two(d_hh, ah, db + B_HIGH, more);
                }
                ptx::mma_commit(lead, ptx::smem_u32(&bars->a_empty[s]));
                if (final) ptx::mma_commit(lead, ptx::smem_u32(&bars->b_empty[t]));
                s ^= 1u;
                if (s == 0) ph ^= 1u;
            }
            if (!ok) break;
            ptx::mma_commit(lead, ptx::smem_u32(&bars->acc_full[b]));
            b ^= 1u;
            if (b == 0) bph ^= 1u;
            fresh = w.next(a);
            if (fresh && ++bset == a.bsets) bset = 0;
        }
        // every MMA issued by this CTA has completed before TMEM is freed
        ptx::mma_commit(lead, ptx::smem_u32(&bars->drain));
        const uint64_t t0 = ptx::globaltimer();
        while (!ptx::mbar_try_wait(ptx::smem_u32(&bars->drain), 0) && ptx::globaltimer() - t0 < WAIT_NS) {
        }
        __syncwarp();
    } else if (warp > W_MMA) {
        // ---------------- B digit tiles, once per K range (bulk copies) ----------------
        if (warp == W_BPROD && lane == 0) {
            asm volatile("griddepcontrol.wait;" ::: "memory");
            Walk w;
            w.start(a, u0, u1);
            uint32_t bset = 0, used = 0, landing = 0;   // bit t: tile t's phase; tiles copied to
            bool ok = true;
            while (w.left && ok) {
                for (uint32_t j = 0; j < w.kbs; ++j) {
                    const uint32_t t = bset * a.bset_tiles + j, bit = 1u << t;
                    // free once the last unit of the range before has read it
                    ok = wait_bar(ptx::smem_u32(&bars->b_empty[t]), used & bit ? 0u : 1u, abort, a.err);
                    if (!ok) break;
                    used ^= bit;
                    landing |= bit;
                    const uint32_t fb = ptx::smem_u32(&bars->b_full[t]);
                    ptx::mbar_arrive_expect_tx(fb, B_TILE_BYTES);
                    ptx::bulk_g2s(ptx::smem_u32(btiles + t * B_TILE_BYTES),
                                  a.Bimg + ((uint64_t)w.nt * a.kblocks + w.kb0 + j) * B_TILE_BYTES, B_TILE_BYTES,
                                  fb);
                }
                if (++bset == a.bsets) bset = 0;
                while (w.left && !w.next(a)) {
                }
            }
            // copies already issued must land before the CTA can exit
            for (uint32_t t = 0; t < RK; ++t) {
                if (!((landing >> t) & 1u)) continue;
                const uint64_t t0 = ptx::globaltimer();
                while (!ptx::mbar_try_wait(ptx::smem_u32(&bars->b_full[t]), ((used >> t) & 1u) ^ 1u) &&
                       ptx::globaltimer() - t0 < WAIT_NS) {
                }
            }
        }
    } else {
        // ---------------- epilogue: TMEM -> residues ----------------
        asm volatile("griddepcontrol.wait;" ::: "memory");
        const int quarter = warp & 3;               // TMEM lanes 32*quarter .. +31
        const uint32_t c_first = (uint32_t)((warp - W_EPI0) >> 2) * 32u;   // this warp's 32 columns
        const uint32_t taddr = tmem + ((uint32_t)(quarter * 32) << 16) + c_first;
        Walk w;
        w.start(a, u0, u1);
        uint32_t b = 0, ph = 0;
        while (w.left && wait_bar_warp(ptx::smem_u32(&bars->acc_full[b]), ph, abort, a.err)) {
            ptx::tc_fence_after();
            const uint64_t grow = (uint64_t)w.mt * BM + quarter * 32 + lane;
            const uint64_t col0 = (uint64_t)w.nt * NT + c_first;
            // columns of this warp's 32 that exist (none for a row outside)
            const int ncols = grow < a.m && col0 < a.nb ? (int)min(a.nb - col0, (uint64_t)32) : 0;
            uint32_t *dst = a.direct ? a.C + grow * a.ldc + col0 : a.Cacc + col0 * a.m + 2 * grow;
#pragma unroll 1
            for (int g = 0; g < 32; g += 8) {
                uint32_t hh[8], md[8], ll[8];
                ptx::tmem_ld8(taddr + b * ACC_COLS + g, ll);
                ptx::tmem_ld8(taddr + b * ACC_COLS + NT + g, md);
                ptx::tmem_ld8(taddr + b * ACC_COLS + 2 * NT + g, hh);
                ptx::tmem_ld_wait();
                if (g == 24) {
                    ptx::tc_fence_before();
                    __syncwarp();
                    if (lane == 0) ptx::mbar_arrive(ptx::smem_u32(&bars->acc_empty[b]));
                }
                // Horner's rule modulo p in 32 bits, t - floor(t smagic / 2^32) p:
                // every accumulator is at most 2^24 in magnitude, so |t| stays
                // below 2^26, the quotient is that of t / p but for less than
                // |t| / 2^32 < 1/64, and the remainder lies in (-p/64, p + p/64);
                // adding p and taking it off again where the result stays
                // non-negative leaves [0, p + p/64]
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const int p = (int)a.p;
                    int t = __float2int_rn(__uint_as_float(hh[j]));
                    t -= __mulhi(t, a.smagic) * p;
                    t = t * 256 + __float2int_rn(__uint_as_float(md[j]));
                    t -= __mulhi(t, a.smagic) * p;
                    t = t * 256 + __float2int_rn(__uint_as_float(ll[j]));
                    t -= __mulhi(t, a.smagic) * p;
                    hh[j] = min((uint32_t)t, (uint32_t)(t + p));
                }
                if (a.direct) {
#pragma unroll
                    for (int j = 0; j < 8; ++j)
                        if (g + j < ncols) dst[g + j] = min(hh[j], hh[j] - a.p);
                } else {
                    // two columns in one 64-bit addition (neither sum reaches
                    // 2^32, so nothing carries between them; columns past the
                    // last add their zero), the 32 lanes of a warp, consecutive
                    // rows, to 256 consecutive bytes
#pragma unroll
                    for (int j = 0; j < 8; j += 2) {
                        if (g + j < ncols)
                            atomicAdd(reinterpret_cast<unsigned long long *>(dst),
                                      (unsigned long long)hh[j] | (unsigned long long)hh[j + 1] << 32);
                        dst += 2 * a.m;
                    }
                }
            }
            b ^= 1u;
            if (b == 0) ph ^= 1u;
            w.next(a);
        }
        // the kernel that reduces the partial sums may be launched now (it
        // waits for this grid to complete before reading them)
        asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    }

    ptx::tc_fence_before();
    __syncthreads();
    if (warp == W_MMA) {
        ptx::tc_fence_after();
        ptx::tmem_dealloc(tmem, TMEM_COLS);
    }
}

// B (k x nb, row-major) -> per (modulus, n-tile, k-block) tiles of 128 rows x
// 64 K fp16 digits in the 128-byte swizzled K-major layout: rows 0..63 hold the
// low digits of output columns nt*64 + r, rows 64..127 the high digits.  One
// pass over B serves every residue pass.
struct PrepB {
    uint32_t n;                        // moduli
    uint32_t reduce;                   // B's entries are not below them yet
    uint32_t p[RNS_MAX], magic[RNS_MAX];
    uint4 *clear;                      // scratch that is to be zero for the product (or none)
    uint64_t clear_n;
};
constexpr int PREPB_THREADS = 256;
__global__ void __launch_bounds__(PREPB_THREADS)
    k_block_prep_b(const uint32_t *__restrict__ B, uint64_t ldb, uint64_t k, uint64_t nb, uint32_t kblocks,
                   const __grid_constant__ PrepB pb, uint8_t *img)
{
    // everything before this kernel is complete from here on, so the product
    // kernel may be placed (it waits for this grid where it reads the tiles)
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const uint32_t tile = blockIdx.x;            // nt * kblocks + kb
    const uint32_t nt = tile / kblocks, kb = tile % kblocks;
    constexpr int PER = 64 * 8 / PREPB_THREADS;  // (column, 8 K) items of a thread
    uint32_t v[PER][8];
#pragma unroll
    for (int i = 0; i < PER; ++i) {
        const int t = threadIdx.x + i * PREPB_THREADS;
        // consecutive threads: consecutive columns of one row of B
        const uint64_t col = (uint64_t)nt * NT + (t & 63), k0 = (uint64_t)kb * BK + (t >> 6) * 8;
#pragma unroll
        for (int e = 0; e < 8; ++e) v[i][e] = (col < nb && k0 + e < k) ? __ldg(B + (k0 + e) * ldb + col) : 0u;
    }
    for (uint64_t i = (uint64_t)blockIdx.x * PREPB_THREADS + threadIdx.x; i < pb.clear_n;
         i += (uint64_t)gridDim.x * PREPB_THREADS)
        pb.clear[i] = make_uint4(0u, 0u, 0u, 0u);
    for (uint32_t l = 0; l < pb.n; ++l) {
        const uint32_t p = pb.p[l], half = (p - 1) / 2;
        uint8_t *out = img + ((uint64_t)l * gridDim.x + tile) * B_TILE_BYTES;
#pragma unroll
        for (int i = 0; i < PER; ++i) {
            const int t = threadIdx.x + i * PREPB_THREADS;
            uint32_t u[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const uint32_t b = pb.reduce ? reduce_small(v[i][e], p, pb.magic[l]) : v[i][e];
                u[e] = b + (b > half ? U_BIAS - p : U_BIAS);
            }
            uint4 h, lo;
            split_u(u[0], u[1], h.x, lo.x);
            split_u(u[2], u[3], h.y, lo.y);
            split_u(u[4], u[5], h.z, lo.z);
            split_u(u[6], u[7], h.w, lo.w);
            // 128-byte swizzle: 16-byte chunk j of row r sits at chunk j ^ (r & 7)
            const int row = t & 63, j = t >> 6;
            const uint32_t off = (uint32_t)row * 128u + ((uint32_t)(j ^ (row & 7)) << 4);
            *reinterpret_cast<uint4 *>(out + off) = lo;
            *reinterpret_cast<uint4 *>(out + 64 * 128 + off) = h;
        }
    }
}

// Partial sums to residues: C = sums mod p (and the sums back to zero), or,
// with C null, the sums themselves reduced below p in place (between the
// launches of a product with more than SLAB_K terms).
constexpr int FIN_THREADS = 512;
__global__ void __launch_bounds__(FIN_THREADS)
    k_block_finish(uint32_t *__restrict__ Cacc, uint64_t m, uint64_t nb, uint32_t *__restrict__ C,
                   uint64_t ldc, uint32_t p, uint32_t magic)
{
    __shared__ uint32_t t[NT][BM + 1];   // [column][row], padded against bank conflicts
    constexpr int PER = NT * BM / FIN_THREADS;
    // the next product of the stream may be placed now; it waits for this grid
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const uint64_t r0 = (uint64_t)blockIdx.x * BM, c0 = (uint64_t)blockIdx.y * NT;
    // all of a thread's loads are issued before any is used or cleared (one
    // memory latency, not one per element); consecutive threads take
    // consecutive rows of one column
    constexpr int PAIRS = PER / 2;
    uint2 v[PAIRS];
    uint2 *acc = reinterpret_cast<uint2 *>(Cacc);
#pragma unroll
    for (int e = 0; e < PAIRS; ++e) {
        const int i = threadIdx.x + e * FIN_THREADS, c = i / BM * 2, r = i % BM;
        v[e] = (r0 + r < m && c0 + c < nb) ? __ldcg(&acc[(c0 + c) / 2 * m + r0 + r]) : make_uint2(0u, 0u);
    }
#pragma unroll
    for (int e = 0; e < PAIRS; ++e) {
        const int i = threadIdx.x + e * FIN_THREADS, c = i / BM * 2, r = i % BM;
        v[e].x = reduce_small(v[e].x, p, magic);   // the sums are below 2^32
        v[e].y = reduce_small(v[e].y, p, magic);
        if (r0 + r < m && c0 + c < nb) __stcg(&acc[(c0 + c) / 2 * m + r0 + r], C ? make_uint2(0u, 0u) : v[e]);
        t[c][r] = v[e].x;
        t[c + 1][r] = v[e].y;
    }
    if (!C) return;
    __syncthreads();
    for (int i = threadIdx.x; i < NT * BM; i += FIN_THREADS) {
        const int r = i / NT, c = i % NT;   // consecutive threads: consecutive columns of one row
        if (r0 + r < m && c0 + c < nb) C[(r0 + r) * ldc + c0 + c] = t[c][r];
    }
}

// A (m x k, row-major uint32 residues, leading dimension lda) -> prepared
// tiles for one modulus p <= 65536 (A8_TILE_BYTES): thread t of a tile writes
// the 32 high and 32 low digits that converter lane t of the product reads.
// Entries outside the matrix are 0 (bytes 0x80, 0x80).  With pre != 0 each
// entry is first reduced modulo p (a residue pass).
__global__ void __launch_bounds__(32 * CONV_WARPS)
    k_block_prep_a(const uint32_t *__restrict__ A, uint64_t lda, uint64_t m, uint64_t k, uint32_t p,
                   uint32_t magic, int pre, int vec, uint32_t kblocks, uint8_t *img)
{
    const uint64_t tile = blockIdx.x;   // mt * kblocks + kb
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint64_t row = tile / kblocks * BM + (warp & 3) * 32 + (warp >> 2) * 16 + (lane >> 2);
    const uint64_t col = tile % kblocks * BK + (lane & 3) * 4;
    const uint32_t thr = min((p - 1) / 2, 32639u);   // largest residue kept as itself
    uint4 w[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const uint64_t r = row + 8 * (i & 1), c = col + (i >> 1) * 16;
        const uint32_t *q = A + r * lda + c;
        const uint64_t n = r < m && c < k ? k - c : 0;
        if (vec && n >= 4)
            w[i] = __ldcs(reinterpret_cast<const uint4 *>(q));
        else
            w[i] = make_uint4(n > 0 ? __ldg(q) : 0u, n > 1 ? __ldg(q + 1) : 0u, n > 2 ? __ldg(q + 2) : 0u,
                              n > 3 ? __ldg(q + 3) : 0u);
    }
    uint32_t hb[8], lb[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const uint32_t e[4] = {w[i].x, w[i].y, w[i].z, w[i].w};
        hb[i] = lb[i] = 0;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const uint32_t v = pre ? reduce_small(e[j], p, magic) : e[j];
            const uint32_t u = v + 32896u - (v > thr ? p : 0u);   // in [0, 65535]
            hb[i] |= (u >> 8) << (8 * j);
            lb[i] |= (u & 255u) << (8 * j);
        }
    }
    uint8_t *out = img + tile * A8_TILE_BYTES + warp * 2048 + lane * 16;
    *reinterpret_cast<uint4 *>(out) = make_uint4(hb[0], hb[1], hb[2], hb[3]);
    *reinterpret_cast<uint4 *>(out + 512) = make_uint4(hb[4], hb[5], hb[6], hb[7]);
    *reinterpret_cast<uint4 *>(out + 1024) = make_uint4(lb[0], lb[1], lb[2], lb[3]);
    *reinterpret_cast<uint4 *>(out + 1536) = make_uint4(lb[4], lb[5], lb[6], lb[7]);
}

// Garner recombination of L residue matrices R[l] (m x nb, dense) into
// C = X mod p, where X is the unique integer in [0, prod m_l) with X = R[l]
// mod m_l: mixed-radix digits v_l in [0, m_l), X = v_0 + m_0 (v_1 + m_1 (v_2
// + ...)), evaluated modulo p from the innermost term out.  The moduli are
// the largest primes <= 65536, all above 65000, so a digit v_j < m_j is below
// 2 m_l and reduces modulo m_l by one conditional subtraction.
__global__ void k_block_crt(const uint32_t *R, uint64_t m, uint64_t nb, uint32_t *C, uint64_t ldc, RnsConst rc)
{
    const uint64_t count = m * nb;
    for (uint64_t e = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; e < count;
         e += (uint64_t)gridDim.x * blockDim.x) {
        uint32_t v[RNS_MAX];
#pragma unroll
        for (int l = 0; l < RNS_MAX; ++l) {
            if (l >= rc.L) break;
            const uint32_t ml = rc.mod[l];
            uint32_t t = R[(uint64_t)l * count + e];   // below ml
#pragma unroll
            for (int j = 0; j < RNS_MAX; ++j) {
                if (j >= l) break;
                const uint32_t vj = v[j] >= ml ? v[j] - ml : v[j];
                t = t >= vj ? t - vj : t + ml - vj;     // (t - v_j) mod m_l
                t = reduce_small(t * rc.inv[l][j], ml, rc.magic[l]);   // both below 2^16
            }
            v[l] = t;
        }
        uint64_t acc = reduce64(v[rc.L - 1], rc.modp);
        for (int l = rc.L - 2; l >= 0; --l) acc = reduce64(acc * rc.mod[l] + v[l], rc.modp);
        C[(e / nb) * ldc + e % nb] = (uint32_t)acc;
    }
}

// ---------------- CUDA-core path ----------------
constexpr int CC_TM = 64, CC_TN = 64, CC_TK = 32, CC_THREADS = 256;

template <class Acc>
__global__ void __launch_bounds__(CC_THREADS)
    k_block_cc(Mod mod, uint64_t kk_bound, uint64_t m, uint64_t k, uint64_t nb,
               const uint32_t *__restrict__ A, uint64_t lda, const uint32_t *__restrict__ B,
               uint64_t ldb, uint32_t *__restrict__ C, uint64_t ldc)
{
    __shared__ __align__(16) uint32_t As[CC_TK][CC_TM];   // transposed: [k][row]
    __shared__ __align__(16) uint32_t Bs[CC_TK][CC_TN];
    const int t = threadIdx.x, tx = t & 15, ty = t >> 4;
    const uint64_t row0 = (uint64_t)blockIdx.y * CC_TM, col0 = (uint64_t)blockIdx.x * CC_TN;
    Acc acc[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j].init(mod, kk_bound);
    for (uint64_t k0 = 0; k0 < k; k0 += CC_TK) {
        // A tile: 64 rows x 32 K; thread -> row t/4, 8 consecutive K
        {
            const int r = t >> 2, kc = (t & 3) * 8;
            const uint64_t gr = row0 + r;
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const uint64_t gk = k0 + kc + e;
                As[kc + e][r] = (gr < m && gk < k) ? __ldg(A + gr * lda + gk) : 0u;
            }
        }
        // B tile: 32 K x 64 columns; thread -> K t/8, 8 consecutive columns
        {
            const int r = t >> 3, cc = (t & 7) * 8;
            const uint64_t gk = k0 + r;
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const uint64_t gc = col0 + cc + e;
                Bs[r][cc + e] = (gk < k && gc < nb) ? __ldg(B + gk * ldb + gc) : 0u;
            }
        }
        __syncthreads();
        const int kmax = (int)min((uint64_t)CC_TK, k - k0);
        for (int kk = 0; kk < kmax; ++kk) {
            const uint4 av = *reinterpret_cast<const uint4 *>(&As[kk][ty * 4]);
            const uint4 bv = *reinterpret_cast<const uint4 *>(&Bs[kk][tx * 4]);
            const uint32_t ar[4] = {av.x, av.y, av.z, av.w};
            const uint32_t br[4] = {bv.x, bv.y, bv.z, bv.w};
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[i][j].add(ar[i], br[j], mod);
        }
        __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const uint64_t gr = row0 + ty * 4 + i;
        if (gr >= m) continue;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const uint64_t gc = col0 + tx * 4 + j;
            if (gc < nb) C[gr * ldc + gc] = acc[i][j].residue(mod);
        }
    }
}

}  // namespace blk

// ---------------- launchers ----------------

bool block_tc_layout_ok(const uint32_t *A, uint64_t lda)
{
    return ((((uintptr_t)A) & 15u) == 0) && (lda % 4 == 0);
}

static uint32_t pow_mod_small(uint64_t b, uint64_t e, uint32_t m)
{
    uint64_t r = 1 % m;
    b %= m;
    while (e) {
        if (e & 1) r = r * b % m;
        b = b * b % m;
        e >>= 1;
    }
    return (uint32_t)r;
}

bool block_rns_plan(uint32_t p, uint64_t k, RnsConst *rc)
{
    // the RNS_MAX largest primes not above 65536, by trial division: every
    // residue modulus then also fits the 8-bit digit planes of a prepared A
    static uint32_t primes[RNS_MAX];
    static bool ready = false;
    static std::mutex mu;
    {
        std::lock_guard<std::mutex> g(mu);
        if (!ready) {
            int found = 0;
            for (uint32_t c = RNS_PRIME_MAX; found < RNS_MAX; --c) {
                bool prime = c > 1;
                for (uint32_t d = 2; prime && d * d <= c; ++d) prime = (c % d) != 0;
                if (prime) primes[found++] = c;
            }
            ready = true;
        }
    }
    if (p < 2) return false;
    // every exact entry sum_t a_t b_t lies in [0, k (p-1)^2]; the moduli's
    // product must exceed that to fix it
    const unsigned __int128 bound = (unsigned __int128)k * (uint64_t)(p - 1) * (uint64_t)(p - 1);
    unsigned __int128 M = 1;
    int L = 0;
    while (L < RNS_MAX && M <= bound) M *= primes[L++];
    if (M <= bound) return false;
    rc->L = L;
    rc->p = p;
    for (int l = 0; l < RNS_MAX; ++l) {
        rc->mod[l] = l < L ? primes[l] : 1;
        for (int j = 0; j < RNS_MAX; ++j)
            rc->inv[l][j] = (l < L && j < l) ? pow_mod_small(primes[j], primes[l] - 2, primes[l]) : 0;
        rc->magic[l] = (uint32_t)((1ull << 32) / std::max<uint32_t>(rc->mod[l], 2));
    }
    rc->modp = make_mod(p);
    return true;
}

size_t block_tc_workspace_bytes(uint64_t m, uint64_t nb)
{
    const uint64_t n_tiles = (nb + blk::NT - 1) / blk::NT;
    return (m * n_tiles * blk::NT * 4 + 255) & ~(size_t)255;
}

size_t block_tc_bimg_bytes(uint64_t k, uint64_t nb, int at_once)
{
    const uint64_t kblocks = (std::min<uint64_t>(k, blk::SLAB_K) + blk::BK - 1) / blk::BK;
    const uint64_t n_tiles = (nb + blk::NT - 1) / blk::NT;
    return n_tiles * kblocks * (uint64_t)blk::B_TILE_BYTES * at_once;
}

// One launch for all of them saves the others' (4.7 us each) and their reads of B,
// next to nothing once B is large; what B's tiles may take is bounded by it.
int block_tc_moduli_at_once(uint64_t k, uint64_t nb, int n_mod)
{
    constexpr size_t TILES_MAX = (size_t)1 << 30;
    return k <= blk::SLAB_K && block_tc_bimg_bytes(k, nb, n_mod) <= TILES_MAX ? n_mod : 1;
}

size_t block_prep_a_bytes(uint64_t m, uint64_t k)
{
    const uint64_t kblocks = (k + blk::BK - 1) / blk::BK;
    const uint64_t m_tiles = (m + blk::BM - 1) / blk::BM;
    return (size_t)(m_tiles * kblocks) * blk::A8_TILE_BYTES;
}

cudaError_t launch_block_prep_a(const Mod &mod, uint64_t m, uint64_t k, const uint32_t *A,
                                uint64_t lda, bool reduce_inputs, uint8_t *img, cudaStream_t s)
{
    using namespace blk;
    const uint64_t kblocks = (k + BK - 1) / BK, m_tiles = (m + BM - 1) / BM;
    if (m_tiles * kblocks == 0) return cudaSuccess;
    if (m_tiles * kblocks > 0x7FFFFFFFull) return cudaErrorInvalidValue;
    if (mod.p > DIGIT8_MAX_P) return cudaErrorInvalidValue;
    k_block_prep_a<<<(unsigned)(m_tiles * kblocks), 32 * CONV_WARPS, 0, s>>>(
        A, lda, m, k, mod.p, (uint32_t)((1ull << 32) / mod.p), reduce_inputs ? 1 : 0,
        block_tc_layout_ok(A, lda) ? 1 : 0, (uint32_t)kblocks, img);
    return cudaGetLastError();
}

// K ranges of a product with `tiles` output tiles and `kblocks` k-blocks on
// `sms` CTAs: at least enough for the exact chunk of RK k-blocks, more where
// units would not fill the CTAs or would leave them uneven.  A unit costs its
// k-blocks plus its drain; the CTA with the most units sets the time.
static uint32_t block_ranges(uint64_t tiles, uint32_t kblocks, int sms)
{
    const uint32_t lo = (kblocks + blk::RK - 1) / blk::RK;
    uint32_t best = lo;
    double best_cost = 0;
    for (uint32_t r = lo; r <= kblocks && r <= 8 * lo; ++r) {
        const double per_cta = (double)((tiles * r + sms - 1) / (uint64_t)sms);
        const double cost = per_cta * ((double)((kblocks + r - 1) / r) + 1.5);
        if (r == lo || cost < 0.97 * best_cost) {
            best = r;
            best_cost = cost;
        }
        if (tiles * r > 8 * (uint64_t)sms) break;
    }
    return best;
}

// One product (n_mod = 1: modulus mods[0]; C = A B mod it) or all residue
// passes (n_mod moduli; pass l writes the dense m x nb matrix C + l m nb).
cudaError_t launch_block_tc(const uint32_t *mods, int n_mod, uint64_t m, uint64_t k, uint64_t nb,
                            const uint32_t *A, uint64_t lda, const uint32_t *B, uint64_t ldb, uint32_t *C,
                            uint64_t ldc, const BlockScratch &sc, int sm_count, cudaStream_t s,
                            int *launches, const uint8_t *Aimg, size_t img_bytes)
{
    using namespace blk;
    typedef void (*Kernel)(const Args);
    static const Kernel kernels[5] = {k_block_tc<A_VEC, false>, k_block_tc<A_VEC, true>,
                                      k_block_tc<A_ANY, false>, k_block_tc<A_ANY, true>,
                                      k_block_tc<A_PREP, false>};
    static std::atomic<bool> attr{false};   // products of several threads may be the first
    if (!attr) {
        for (Kernel f : kernels) {
            cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                 (int)SMEM_BYTES);
            // the rest of the 256 KiB stays L1: the loads in flight land there
            if (e == cudaSuccess)
                e = cudaFuncSetAttribute(f, cudaFuncAttributePreferredSharedMemoryCarveout, 58);
            // a warpgroup that asks for more registers than the block was launched
            // with waits forever: nothing but the planned number is launched
            cudaFuncAttributes fa;
            if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, f);
            if (e == cudaSuccess && fa.numRegs != REGS_LAUNCH) e = cudaErrorInvalidDeviceFunction;
            if (e != cudaSuccess) return e;
        }
        attr = true;
    }
    const bool reduce = n_mod > 1;
    // prepared digits: 16-byte aligned tiles of a device allocation
    if (Aimg && (((uintptr_t)Aimg) & 15u)) return cudaErrorInvalidValue;
    const Kernel kernel = Aimg ? kernels[4] : kernels[(block_tc_layout_ok(A, lda) ? 0 : 2) + (reduce ? 1 : 0)];
    static_assert(BLOCK_TC_MAX_NB == 65535ull * NT, "grid y of the finishing kernel");
    if (nb > BLOCK_TC_MAX_NB) return cudaErrorInvalidValue;
    Args a;
    memset(&a, 0, sizeof a);
    a.m = m;
    a.nb = nb;
    a.lda = lda;
    a.img_kblocks = (uint32_t)((k + BK - 1) / BK);
    a.err = sc.err;
    a.Cacc = (uint32_t *)sc.ws;
    a.n_tiles = (uint32_t)((nb + NT - 1) / NT);
    a.m_tiles = (uint32_t)((m + BM - 1) / BM);
    a.edge_m = m % BM ? a.m_tiles - 1 : ~0u;
    const uint64_t tiles = (uint64_t)a.m_tiles * a.n_tiles;
    cudaLaunchAttribute pdl[1];
    pdl[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    pdl[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t bcfg = {}, cfg = {}, fcfg = {};
    bcfg.blockDim = dim3(PREPB_THREADS);
    cfg.blockDim = dim3(THREADS);
    cfg.dynamicSmemBytes = SMEM_BYTES;
    fcfg.gridDim = dim3(a.m_tiles, a.n_tiles);
    fcfg.blockDim = dim3(FIN_THREADS);
    bcfg.stream = cfg.stream = fcfg.stream = s;
    bcfg.attrs = cfg.attrs = fcfg.attrs = pdl;
    bcfg.numAttrs = cfg.numAttrs = fcfg.numAttrs = 1;
    PrepB pb;
    memset(&pb, 0, sizeof pb);
    bool dirty = sc.dirty;
    for (int l0 = 0; l0 < n_mod; l0 += sc.at_once) {
        const int l1 = std::min(n_mod, l0 + sc.at_once);
        for (uint64_t k0 = 0; k0 < k; k0 += SLAB_K) {
            a.k = std::min<uint64_t>(SLAB_K, k - k0);
            const bool last = k - k0 <= SLAB_K;
            a.A = A ? A + k0 : nullptr;
            a.img_kb0 = (uint32_t)(k0 / BK);
            a.kblocks = (uint32_t)((a.k + BK - 1) / BK);
            a.ranges = block_ranges(tiles, a.kblocks, sm_count);
            a.r_base = a.kblocks / a.ranges;
            a.r_rem = a.kblocks % a.ranges;
            a.bsets = RK / (a.r_base + (a.r_rem ? 1 : 0));
            a.bset_tiles = RK / a.bsets;
            a.edge_k = a.k % BK ? a.kblocks - 1 : ~0u;
            a.units = tiles * a.ranges;
            a.direct = a.ranges == 1 && k <= SLAB_K ? 1 : 0;
            const uint32_t btiles = a.n_tiles * a.kblocks;
            pb.n = (uint32_t)(l1 - l0);
            pb.reduce = reduce ? 1 : 0;
            for (int l = l0; l < l1; ++l) {
                pb.p[l - l0] = mods[l];
                pb.magic[l - l0] = (uint32_t)((1ull << 32) / mods[l]);
            }
            pb.clear = dirty && !a.direct ? (uint4 *)sc.ws : nullptr;
            pb.clear_n = pb.clear ? block_tc_workspace_bytes(m, nb) / 16 : 0;
            dirty = false;
            bcfg.gridDim = dim3(btiles);
            cudaError_t e = cudaLaunchKernelEx(&bcfg, k_block_prep_b, B + k0 * ldb, ldb, a.k, nb, a.kblocks, pb,
                                               sc.bimg);
            if (e != cudaSuccess) return e;
            ++*launches;
            cfg.gridDim = dim3((unsigned)std::min<uint64_t>(a.units, (uint64_t)sm_count));
            for (int l = l0; l < l1; ++l) {
                const uint32_t p = mods[l];
                a.p = p;
                a.half = (p - 1) / 2;
                a.magic = (uint32_t)((1ull << 32) / p);
                a.smagic = (int32_t)std::min<uint64_t>((1ull << 32) / p, 0x7FFFFFFFull);
                a.magic47 = reduce ? (uint32_t)((1ull << 47) / p) : 0;
                a.C = C + (reduce ? (uint64_t)l * m * nb : 0);
                a.ldc = ldc;
                a.Aimg = Aimg ? Aimg + (size_t)l * img_bytes : nullptr;
                a.Bimg = sc.bimg + (uint64_t)(l - l0) * btiles * B_TILE_BYTES;
                // residue passes over a uint32 A alternate direction: what a CTA
                // read last is what L2 still holds, and every second pass
                // begins there
                a.backward = reduce && !Aimg ? (uint32_t)(l & 1) : 0;
                e = cudaLaunchKernelEx(&cfg, kernel, a);
                if (e != cudaSuccess) return e;
                ++*launches;
                if (a.direct) continue;
                e = cudaLaunchKernelEx(&fcfg, k_block_finish, a.Cacc, m, nb, last ? a.C : (uint32_t *)nullptr,
                                       ldc, p, a.magic);
                if (e != cudaSuccess) return e;
                ++*launches;
            }
        }
    }
    return cudaGetLastError();
}

cudaError_t launch_block_crt(const uint32_t *R, uint64_t m, uint64_t nb, uint32_t *C, uint64_t ldc,
                             const RnsConst &rc, int sm_count, cudaStream_t s)
{
    const uint64_t count = m * nb;
    const uint64_t blocks = std::max<uint64_t>(1, std::min<uint64_t>((count + 255) / 256, (uint64_t)sm_count * 8));
    blk::k_block_crt<<<(unsigned)blocks, 256, 0, s>>>(R, m, nb, C, ldc, rc);
    return cudaGetLastError();
}

template <class Acc>
static cudaError_t cc_launch(const Mod &mod, uint64_t kb, uint64_t m, uint64_t k, uint64_t nb,
                             const uint32_t *A, uint64_t lda, const uint32_t *B, uint64_t ldb,
                             uint32_t *C, uint64_t ldc, cudaStream_t s)
{
    using namespace blk;
    dim3 grid((unsigned)((nb + CC_TN - 1) / CC_TN), (unsigned)((m + CC_TM - 1) / CC_TM));
    k_block_cc<Acc><<<grid, CC_THREADS, 0, s>>>(mod, kb, m, k, nb, A, lda, B, ldb, C, ldc);
    return cudaGetLastError();
}

cudaError_t wait_selftest(uint64_t limit_ns, cudaStream_t s, uint32_t *status_bits)
{
    uint32_t zero = 0;
    cudaError_t e = cudaMemcpyToSymbolAsync(blk::g_selftest_err, &zero, 4, 0, cudaMemcpyHostToDevice, s);
    if (e != cudaSuccess) return e;
    uint32_t *dptr = nullptr;
    e = cudaGetSymbolAddress((void **)&dptr, blk::g_selftest_err);
    if (e != cudaSuccess) return e;
    blk::k_wait_selftest<<<1, 32, 0, s>>>(limit_ns, dptr);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    e = cudaMemcpyFromSymbolAsync(status_bits, blk::g_selftest_err, 4, 0, cudaMemcpyDeviceToHost, s);
    if (e != cudaSuccess) return e;
    return cudaStreamSynchronize(s);
}

cudaError_t launch_block_cc(Repr r, const Mod &mod, uint64_t kbound, uint64_t m, uint64_t k,
                            uint64_t nb, const uint32_t *A, uint64_t lda, const uint32_t *B,
                            uint64_t ldb, uint32_t *C, uint64_t ldc, cudaStream_t s)
{
    switch (r) {
    case U64_BLOCK: return cc_launch<AccBlock>(mod, kbound, m, k, nb, A, lda, B, ldb, C, ldc, s);
    case U64_CARRY: return cc_launch<AccCarry>(mod, kbound, m, k, nb, A, lda, B, ldb, C, ldc, s);
    case FP64: return cc_launch<AccF64>(mod, kbound, m, k, nb, A, lda, B, ldb, C, ldc, s);
    case CENTERED: return cc_launch<AccCentered>(mod, kbound, m, k, nb, A, lda, B, ldb, C, ldc, s);
    case MONTGOMERY: return cc_launch<AccMontgomery>(mod, kbound, m, k, nb, A, lda, B, ldb, C, ldc, s);
    default: return cc_launch<AccPerTerm>(mod, kbound, m, k, nb, A, lda, B, ldb, C, ldc, s);
    }
}

}  // namespace gfp
