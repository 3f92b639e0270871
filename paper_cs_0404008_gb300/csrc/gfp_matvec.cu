// Dense matrix-vector product over GF(p): y_i = (sum_j A_ij x_j) mod p.
//
// Each CTA owns a contiguous range of rows (ranges differ by at most one row
// over the grid, one CTA per SM).  x is staged once per CTA in shared memory.
// Inside a CTA the warps form G groups of W warps: a group works on one row at
// a time and warp s of the group streams column segment s of that row with
// 128-bit loads, accumulating unreduced (Section 3 of the paper) and leaving
// one residue per (row, segment) in shared memory.  After a window of rows
// the CTA sums the W segment residues of each row and writes y.  No atomics,
// no per-row barrier; A is read exactly once.
//
// HBM bound, so what counts is that loads stay in flight.  A warp keeps two
// batches of U vectors a lane: while it adds one up (and reduces at the end of a
// row) the next, of the same row or of its next one, is already loading.  A
// ragged end is part of a batch, not a loop of its own.  64 iterations of
// 32768^2 over GF(2^31 - 1): 39.1 -> 37.7 ms (7.29 TB/s) against one batch of
// four vectors in flight in 32 warps; 9001 x 7003 with packed, odd rows: 54.9 ->
// 41.6 us (6.1 TB/s).  Batches of four or six vectors were slower (70 and 66
// against 52 us for the latter with a flushed L2): more batches a row.
//
// Rows of at most 256 columns are bound by the latency of a row (load, add, reduce
// by shuffles): twice the warps with batches of two vectors; 200000 x 64 over
// GF(65521) 64.8 -> 36.5 us, 45 with one batch of four in flight.  Above 51200
// columns x is read through L1 and L2 beside A, in 32 warps with one batch of four
// in flight: two batches of eight in 16 warps took 82.2 against 55.9 us for
// 700 x 100000 over GF(65521), and 286 against 87.1 where rows are not 16-byte
// aligned.
//
// Rows need not be 16-byte aligned.  A row that starts r words past a 16-byte
// boundary is read as the aligned vectors inside it; x is then kept in shared
// memory as four planes of every fourth element, so that the four elements a
// vector multiplies are one conflict-free read each (from a plain x the lanes'
// words would lie four apart, a four-way bank conflict).  The fewer than four
// elements before the first and after the last vector are added by themselves.  Such
// rows of at most 64 columns, a word or two a lane, are read word by word (200000 x
// 16 over GF(65521): 44 against 55 us), in FP64, where each pass over the lanes
// costs, up to 256 (200000 x 200: 360 against 408 us).
#include <algorithm>
#include <type_traits>

#include "gfp_internal.h"

namespace gfp {

// Threads and vectors a lane loads at a time, two batches in flight: for rows of
// more than MV_SHORT columns, for shorter ones, for a remainder at every term (which
// bounds the time: 32 warps, 3000 x 5000 23.4 us, 30.4 in 16); and, one batch in
// flight, for rows whose x is not in shared memory.
constexpr int MV_THREADS = 512, MV_U = 8;
constexpr int MV_SHORT_THREADS = 1024, MV_SHORT_U = 2;
constexpr int MV_TERM_THREADS = 1024, MV_TERM_U = 4;
constexpr int MV_GLOBAL_THREADS = 1024, MV_GLOBAL_U = 4;
constexpr uint64_t MV_SHORT = 256, MV_WORDS = 64;   // columns
constexpr uint32_t MV_GLOBAL_WINDOW = 64;           // rows
constexpr int MV_PREFETCH_ROWS = 4;   // rows of A requested into L2 before the dependency wait

// Sum of one uint64 per thread over the CTA, valid in thread 0.
__device__ __forceinline__ uint64_t cta_sum_mv(uint64_t v)
{
    __shared__ uint64_t sh[32];
#pragma unroll
    for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    if (l == 0) sh[w] = v;
    __syncthreads();
    if (w == 0) {
        v = (l < (int)(blockDim.x >> 5)) ? sh[l] : 0;
#pragma unroll
        for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    }
    __syncthreads();
    return v;
}

// Projection of the product onto a vector u, fused into the epilogue (the
// scalar sequence u^T A^t x of a Wiedemann-style iteration): every CTA adds
// the residue of sum_i u_i y_i over its rows to a slot; the last CTA reduces
// it into *sout.  Inactive when u is null.
struct MvProj {
    const uint32_t *u;
    unsigned long long *slot;
    uint32_t *ticket;
    uint32_t *sout;
};

// Where x is read from: global memory (16-byte aligned, or 4-byte reads),
// shared memory as it is, or shared memory in four planes for rows of any
// alignment.
enum XMode : int { X_GLOBAL = 0, X_SMEM = 1, X_PLANES = 2 };

// One warp's part [c0, c1) of a row; columns are counted from c0.
struct RowPart {
    const uint4 *av;   // first 16-byte vector inside it, this lane's
    uint32_t nv;       // vectors
    uint32_t head;     // column of the first one
    uint32_t ecol;     // column of the lane's element outside the vectors, or ~0
    uint32_t eval;     // that element
};

template <class Acc, int XM, int U, int T>
__global__ void __launch_bounds__(T, 1)
    k_matvec(Mod m, uint64_t k, uint64_t rows, uint64_t cols, const uint32_t *__restrict__ A,
             uint64_t lda, const uint32_t *__restrict__ x, uint32_t *__restrict__ y, int W, uint32_t window,
             MvProj proj)
{
    extern __shared__ __align__(16) uint32_t smem[];
    const uint64_t colsp = (cols + 3) & ~3ull;
    // Programmatic dependent launch: the next kernel of the stream may be
    // scheduled on SMs this grid has left (its tail).  A never changes, so
    // before waiting for the previous kernel (which may have produced x) the
    // CTA asks L2 for the first rows it will stream; everything that reads
    // x or writes y comes after the wait.
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const uint64_t r_begin = rows * blockIdx.x / gridDim.x;
    const uint64_t r_end = rows * (blockIdx.x + 1) / gridDim.x;
    {
        const uint64_t row_bytes = cols * 4;
        if (threadIdx.x < MV_PREFETCH_ROWS && r_begin + threadIdx.x < r_end &&
            ((((uintptr_t)A) | (lda * 4) | row_bytes) & 15u) == 0 && row_bytes <= 0xFFFFFFF0ull)
            asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(A + (r_begin + threadIdx.x) * lda),
                         "r"((uint32_t)row_bytes)
                         : "memory");
    }
    asm volatile("griddepcontrol.wait;" ::: "memory");
    uint32_t *xs = smem;
    const uint32_t plane = (uint32_t)(colsp >> 2);   // words of a plane of x
    uint32_t *part = smem + (XM != X_GLOBAL ? colsp : 0);
    const int nw = T / 32, w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int G = nw / W, sgm = w % W;
    const uint32_t g = w < G * W ? (uint32_t)(w / W) : ~0u;   // ~0: no group, where W does not divide the warps

    // column segment of this warp: [c0, c1), c0 a multiple of 4
    const uint64_t seg = ((cols + W - 1) / W + 3) & ~3ull;
    const uint64_t c0 = min((uint64_t)sgm * seg, cols);
    const uint64_t c1 = min(c0 + seg, cols);
    // batches that cover any row's part (at least one: it carries the elements outside the vectors)
    const uint32_t nq = max(1u, (uint32_t)((((c1 - c0) >> 2) + U * 32 - 1) / (U * 32)));

    const uint32_t cs = (uint32_t)c0;   // where x is in shared memory
    const auto xat = [&](uint32_t j) -> uint32_t {
        if constexpr (XM == X_PLANES) return xs[(j & 3) * plane + ((cs + j) >> 2)];   // c0 is a multiple of 4
        else return xs[cs + j];
    };
    const auto locate = [&](uint64_t row, RowPart &p) {
        const uint32_t *Ar = A + row * lda + c0;
        const uint32_t len = (uint32_t)(c1 - c0);
        uint32_t head = 0;   // words before the first boundary
        if constexpr (XM == X_PLANES) head = min((uint32_t)(-(int)((uintptr_t)Ar >> 2) & 3), len);
        p.nv = (len - head) >> 2;
        p.head = head;
        p.av = reinterpret_cast<const uint4 *>(Ar + head) + lane;
        const uint32_t after = head + (p.nv << 2);   // first element past the vectors
        const uint32_t e = (uint32_t)lane < head ? (uint32_t)lane : after + (uint32_t)lane - 4u;
        const bool has = (uint32_t)lane < head || (lane >= 4 && e < len);
        p.ecol = has ? e : ~0u;
        p.eval = has ? __ldcs(Ar + e) : 0u;
    };
    const auto load = [&](const RowPart &p, uint32_t q, uint4 (&buf)[U]) {
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const uint32_t v = q * (U * 32) + u * 32;
            if (v + lane < p.nv) buf[u] = __ldcs(p.av + v);
        }
    };
    Acc acc;
    acc.init(m, k);
    const auto consume = [&](const RowPart &p, uint32_t q, const uint4 (&buf)[U]) {
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const uint32_t v = q * (U * 32) + u * 32 + lane;
            if (v < p.nv) {
                uint4 xv;
                if constexpr (XM == X_PLANES) {
                    const uint32_t j = p.head, i = (cs >> 2) + v;   // element e: plane (j + e) mod 4
                    const uint32_t i1 = i + (j > 2), i2 = i + (j > 1), i3 = i + (j > 0);
                    xv = make_uint4(xs[j * plane + i], xs[((j + 1) & 3) * plane + i1],
                                    xs[((j + 2) & 3) * plane + i2], xs[((j + 3) & 3) * plane + i3]);
                } else {
                    xv = reinterpret_cast<const uint4 *>(xs + cs)[v];
                }
                acc.add4(buf[u], xv, m);
            }
        }
    };

    uint64_t pacc = 0;   // projection partial (sum of residues)
    bool staged = XM == X_GLOBAL;
    for (uint64_t rb = r_begin; rb < r_end; rb += window) {
        const uint32_t rcount = (uint32_t)min(r_end - rb, (uint64_t)window);
        const auto finish = [&](uint32_t i) {
            uint64_t s = acc.residue(m);
#pragma unroll
            for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            if (lane == 0) part[i * W + sgm] = reduce64(s, m);
            acc.init(m, k);
        };
        if constexpr (XM != X_GLOBAL) {
            uint4 b0[U], b1[U];
            RowPart cur, nxt;
            uint32_t i = g, q = 0;
            if (i < rcount) {
                locate(rb + i, cur);
                load(cur, 0, b0);
            }
            if (!staged) {   // the first loads are under way
                for (uint64_t j = threadIdx.x; j < colsp; j += T)
                    xs[XM == X_PLANES ? (j & 3) * plane + (j >> 2) : j] = (j < cols) ? x[j] : 0u;
                __syncthreads();
                staged = true;
            }
            // one batch: start the next, add this one up, end the row
            const auto step = [&](uint4 (&bc)[U], uint4 (&bn)[U]) {
                uint32_t ni = i, n = q + 1;
                nxt = cur;
                if (n == nq) {
                    n = 0;
                    ni += G;
                    if (ni < rcount) locate(rb + ni, nxt);
                }
                if (ni < rcount) load(nxt, n, bn);
                consume(cur, q, bc);
                if (n == 0) {
                    if (cur.ecol != ~0u) acc.add(cur.eval, xat(cur.ecol), m);
                    finish(i);
                }
                cur = nxt;
                i = ni;
                q = n;
            };
            while (i < rcount) {
                step(b0, b1);
                if (i < rcount) step(b1, b0);
            }
        } else {
            // rows that 16-byte loads take as they are
            const bool vec = ((((uintptr_t)A) | (uintptr_t)(lda * 4) | ((uintptr_t)x)) & 15u) == 0;
            for (uint32_t i = g; i < rcount; i += G) {
                const uint32_t *Ar = A + (rb + i) * lda;
                if (vec) {
                    const uint4 *av = reinterpret_cast<const uint4 *>(Ar + c0);
                    const uint4 *xv = reinterpret_cast<const uint4 *>(x + c0);
                    const uint64_t nv = (c1 - c0) >> 2;
                    uint64_t v = lane;
                    for (; v + (U - 1) * 32 < nv; v += U * 32) {
                        uint4 a[U];
#pragma unroll
                        for (int u = 0; u < U; ++u) a[u] = __ldcs(av + v + u * 32);
#pragma unroll
                        for (int u = 0; u < U; ++u) acc.add4(a[u], __ldg(xv + v + u * 32), m);
                    }
                    for (; v < nv; v += 32) acc.add4(__ldcs(av + v), __ldg(xv + v), m);
                    const uint64_t j = c0 + (nv << 2) + lane;
                    if (j < c1) acc.add(__ldcs(Ar + j), __ldg(x + j), m);
                } else {
                    for (uint64_t j = c0 + lane; j < c1; j += 32) acc.add(__ldcs(Ar + j), __ldg(x + j), m);
                }
                finish(i);
            }
        }
        __syncthreads();
        for (uint32_t i = threadIdx.x; i < rcount; i += T) {
            uint64_t s = 0;
            for (int q = 0; q < W; ++q) s += part[i * W + q];
            const uint32_t yi = reduce64(s, m);
            y[rb + i] = yi;
            if (proj.u) pacc += reduce64((uint64_t)yi * __ldg(proj.u + rb + i), m);
        }
        __syncthreads();
    }
    if (proj.u) {
        const uint64_t s = cta_sum_mv(pacc);
        if (threadIdx.x == 0) {
            atomicAdd(proj.slot, (unsigned long long)reduce64(s, m));
            __threadfence();
            if (atomicAdd(proj.ticket, 1u) == gridDim.x - 1) {
                __threadfence();
                const unsigned long long v = atomicExch(proj.slot, 0ull);
                atomicExch(proj.ticket, 0u);
                *proj.sout = reduce64((uint64_t)v, m);
            }
        }
    }
}

// Shared memory above which x is read through the L1/L2 path instead, and the
// part kept for the segment residues of a window of rows.
constexpr size_t MV_XS_MAX = 200 * 1024, MV_PART_MAX = 16 * 1024;

template <class Acc, int XM, int U, int T>
static cudaError_t mv_launch(const Mod &m, uint64_t k, uint64_t rows, uint64_t cols,
                             const uint32_t *A, uint64_t lda, const uint32_t *x, uint32_t *y,
                             int sm_count, cudaStream_t s, const MvProj &proj)
{
    const int nw = T / 32;
    const uint64_t grid = std::min<uint64_t>((uint64_t)sm_count, rows ? rows : 1);
    const uint64_t per_cta = (rows + grid - 1) / grid;
    const uint64_t nv = cols / 4;
    int W = 1;
    if constexpr (XM == X_GLOBAL) {
        // at least one batch a warp
        while (W < nw && nv / (uint64_t)(2 * W) >= (uint64_t)U * 32) W *= 2;
    } else {
        // warps per row: the power of two that takes a row in one batch of U vectors a
        // lane (more would reduce more often for the same bytes), another number where
        // its batches fill more of all lanes (a row of 1125 vectors: eight warps fill
        // 55 % of them, three groups of five 82 %; 3000 x 4500 over GF(65521) 12.2 ->
        // 10.2 us, 10.6 in eight warps with batches of four), and more where a CTA's
        // rows would leave half of its warps without one, while each has a vector a
        // lane (64 rows of 64: 3.1 us an iteration in 32 warps a row, 2.7 in one)
        const auto filled = [&](int c) {
            const uint64_t batch = (uint64_t)c * U * 32;
            return (double)(nw / c * c) / nw * (double)nv / (double)((nv + batch - 1) / batch * batch);
        };
        while (W < nw && nv > (uint64_t)W * U * 32) W *= 2;
        for (int c = 1; nv && c <= nw; ++c)
            if (nv <= (uint64_t)c * U * 32 && filled(c) > 1.05 * filled(W)) W = c;
        while (2 * W <= nw && nv >= 2 * (uint64_t)W * 32 && (uint64_t)(nw / W) >= 2 * per_cta) W *= 2;
    }
    const size_t colsp = (cols + 3) & ~3ull;
    const uint32_t window = (uint32_t)std::min<uint64_t>(per_cta, XM == X_GLOBAL ? MV_GLOBAL_WINDOW : MV_PART_MAX / (4 * W));
    const size_t smem = (XM != X_GLOBAL ? colsp * 4 : 0) + (size_t)window * W * 4;
    static bool attr_set = false;
    if (!attr_set) {
        cudaError_t e = cudaFuncSetAttribute(k_matvec<Acc, XM, U, T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)(MV_XS_MAX + MV_PART_MAX));
        if (e != cudaSuccess) return e;
        attr_set = true;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3(T);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, k_matvec<Acc, XM, U, T>, m, k, rows, cols, A, lda, x,
                                             y, W, window, proj);
    return e != cudaSuccess ? e : cudaGetLastError();
}

template <class Acc>
static cudaError_t mv_dispatch(const Mod &m, uint64_t k, uint64_t rows, uint64_t cols,
                               const uint32_t *A, uint64_t lda, const uint32_t *x, uint32_t *y,
                               int sm_count, cudaStream_t s, const MvProj &proj)
{
    // rows that 16-byte loads take as they are, or not
    const bool vec = (((uintptr_t)A) & 15u) == 0 && lda % 4 == 0;
    const bool words = !vec && cols <= (std::is_same<Acc, AccF64>::value ? MV_SHORT : MV_WORDS);
    if (words || ((cols + 3) & ~3ull) * 4 > MV_XS_MAX)
        return mv_launch<Acc, X_GLOBAL, MV_GLOBAL_U, MV_GLOBAL_THREADS>(m, k, rows, cols, A, lda, x, y, sm_count, s,
                                                                        proj);
    if constexpr (std::is_same<Acc, AccPerTerm>::value)
        return vec ? mv_launch<Acc, X_SMEM, MV_TERM_U, MV_TERM_THREADS>(m, k, rows, cols, A, lda, x, y, sm_count, s,
                                                                        proj)
                   : mv_launch<Acc, X_PLANES, MV_TERM_U, MV_TERM_THREADS>(m, k, rows, cols, A, lda, x, y, sm_count, s,
                                                                          proj);
    else if (cols <= MV_SHORT)
        return vec ? mv_launch<Acc, X_SMEM, MV_SHORT_U, MV_SHORT_THREADS>(m, k, rows, cols, A, lda, x, y, sm_count, s,
                                                                          proj)
                   : mv_launch<Acc, X_PLANES, MV_SHORT_U, MV_SHORT_THREADS>(m, k, rows, cols, A, lda, x, y, sm_count,
                                                                            s, proj);
    else
        return vec ? mv_launch<Acc, X_SMEM, MV_U, MV_THREADS>(m, k, rows, cols, A, lda, x, y, sm_count, s, proj)
                   : mv_launch<Acc, X_PLANES, MV_U, MV_THREADS>(m, k, rows, cols, A, lda, x, y, sm_count, s, proj);
}

cudaError_t launch_matvec(Repr r, const Mod &m, uint64_t k, uint64_t rows, uint64_t cols,
                          const uint32_t *A, uint64_t lda, const uint32_t *x, uint32_t *y,
                          int sm_count, cudaStream_t s, const uint32_t *u,
                          unsigned long long *slot, uint32_t *ticket, uint32_t *sout)
{
    const MvProj proj{u, slot, ticket, sout};
    switch (r) {
    case U64_BLOCK: return mv_dispatch<AccBlock>(m, k, rows, cols, A, lda, x, y, sm_count, s, proj);
    case U64_CARRY: return mv_dispatch<AccCarry>(m, k, rows, cols, A, lda, x, y, sm_count, s, proj);
    case FP64: return mv_dispatch<AccF64>(m, k, rows, cols, A, lda, x, y, sm_count, s, proj);
    case CENTERED: return mv_dispatch<AccCentered>(m, k, rows, cols, A, lda, x, y, sm_count, s, proj);
    case MONTGOMERY: return mv_dispatch<AccMontgomery>(m, k, rows, cols, A, lda, x, y, sm_count, s, proj);
    default: return mv_dispatch<AccPerTerm>(m, k, rows, cols, A, lda, x, y, sm_count, s, proj);
    }
}

}  // namespace gfp
