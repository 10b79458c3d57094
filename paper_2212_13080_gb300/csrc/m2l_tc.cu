// Bilinear forms of the interaction lists (§2.2 step 3, eq. bilinear) on the
// 5th-generation tensor cores (tcgen05): operands split into 16-bit parts (half or
// bfloat16), FP32 accumulation.
//
// Only cells that hold charges get a functional (step 4 reads no other).
// After the sort, a list of the occupied cells of every (level, target
// parity) segment is built in coarse Morton order; one CTA takes 128 of them
// (the MMA's M).  For each of the 189 interaction-list offsets o, the tile's
// contribution L[cell][a] += sum_b Phi[cell + o][b] K_o[a][b] is a
// 128 x N x K GEMM (N = p^3 padded to a multiple of 32, K to a multiple of
// 16): A holds the tile's 128 source vectors, B the unit-cell kernel K_o, both
// in K chunks staged in shared memory with the swizzle of their width; one thread
// issues the MMAs into tensor memory.  A arrives in one of two ways:
//   - box tiles (a segment whose cells nearly all hold charges): the tile is
//     128 consecutive Morton cells, an 8 x 4 x 4 box of the padded parity-major
//     layout, one box copy a chunk;
//   - gathered tiles: producer warps copy the rows with 16-byte cp.async
//     straight into the swizzled layout, complete and fence them for the async
//     proxy before they arrive on the stage.  A lane's rows and places are fixed
//     for the whole tile, so a row costs one address and two or three copies a
//     stage; TMA row gathers (four rows each) took 65 cycles each: 79.7 against
//     51 ms on 8M clustered charges at p = 6.
//
// Operands, after an exact power-of-two scaling (per cell for the grid charges, one
// factor for the kernels) that puts the largest value near the half type's maximum:
//   two parts (split TF32; plain FP32 plans of p = 3, 4): x = hi + lo, two halves of
//     11 significant bits each, so that x is off by at most 2^-23 of itself, and
//     D = Alo Bhi + Ahi Blo + Ahi Bhi leaves out a product of up to 2^-22 of a term:
//     less than FP32's 24 bits, in sums of at most 64 terms whose rounding outweighs it.
//     Twice TF32's MMA rate and half its bytes.
//   three parts (plain FP32 plans of p = 5, 6): all of FP32's bits of values down to
//     2^-9 of their cell's largest (smaller ones to 2^-32 of it), six products, and the
//     leading products' sum is exact (KSplit).  The tensor cores' FP32 additions do
//     not round to nearest, and two parts summed that way over 125 and 216 terms were
//     up to 7% further from the 64-bit results than FP32 multiply-adds where the terms
//     cancel.  Contraction of 1M clustered charges at p = 6: 7.3 ms with two parts, 10.8
//     with three, 243 with multiply-adds.
//   BF16: two parts of 8 bits, unscaled; the 1-pass form: Ahi Bhi alone, 11 bits.
//
// Accuracy.  The kernel is split as K_o = Kbar_o[a] + Kt_o[a,b] (row mean): the
// tensor cores contract Kt_o, the CUDA cores add Kbar_o[a] Q (Q = the source
// cell's total charge).  Each offset accumulates into fresh TMEM regions, small
// products first; the epilogue warps read them out and add the offsets in FP32
// registers, for plain FP32 plans with Kahan compensation: without it these 189
// additions are the largest error of the form (potentials of a depth-4 system at
// p = 6: 3.2e-7 against 2.8e-7 for FP32 multiply-adds), and it costs the
// reduced-precision plans more than they need (uniform1m: 0.36 against 0.24 ms).
// Plain FP32 plans against FP32 multiply-adds, distance from the 64-bit results in
// 74 systems of 2,001 to 1M charges, open and periodic, p = 3..6: potentials 0.94
// times (at most 1.00), forces 0.91 (at most 1.001); with octants charged in turn,
// where the terms cancel, 0.97 to 1.00 in the mean of 24 systems.
// A row's functional depends on its own A rows only, so it is the same, bit for
// bit, whichever tile form computes it.
#include <algorithm>
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <type_traits>

#include "fmm_internal.cuh"
#include "launch.cuh"
#include "tc_ptx.cuh"

namespace fmm {

#define TC_M 128
#define TC_WAIT_CYCLES (4LL << 30)  // about 2 s of SM clock
#define TC_NOFF 189

// records the first wait of the launch that gave up (diagnostics in the header)
__device__ __forceinline__ void tc_wait_failed(int *status, int site, int level, int iter) {
    WsHeader *h = reinterpret_cast<WsHeader *>(status);
    if (atomicCAS(&h->wait_site, 0, site) == 0) {
        h->wait_block = blockIdx.x;
        h->wait_level = level;
        h->wait_iter = iter;
    }
}

// The interaction list of every target parity (bx, by, bz): offsets o in
// [-2 - b, 3 - b]^3 without [-1, 1]^3, in one of two orders.  An entry packs the
// index of the offset in the 7^3 kernel tables, the source's parity block and its
// coarse shift (-1..1 per axis).
//   0: z, y, x order: neighbouring source cells follow one another, and what they
//      cancel of each other leaves the sum at once.
//   1: by the source's parity, then by its coarse shift: a tile's source cells of
//      one parity (a few hundred cells, used by up to 27 offsets) are read in one
//      stretch of the walk, so that the tiles in flight find them in L2 (152 tiles x
//      0.3 MB at p = 6, against 2.6 MB a tile for all eight parities).
// Order 1 only where a level's operand copy may exceed the L2 (level 6: 282 MB at
// p = 6, level 5: 42 MB): the contraction of 8M clustered charges takes 38 ms so, 55
// in order 0.  On coarse levels it would cost digits: the 27 sources of one parity
// are the 27 images of a single cell at level 1 of the periodic form, and their
// sum, several times the result, rounds before the other parities cancel it
// (water, 66,669 charges: potentials up to 1.17 times as far from the 64-bit results
// as in order 0).
struct OffTable {
    uint32_t v[2][8][TC_NOFF];
};
__host__ __device__ constexpr int off_order(int l) { return l >= 6; }
constexpr uint32_t off_entry(const int (&b)[3], int ox, int oy, int oz) {
    const int s[3] = {b[0] + ox, b[1] + oy, b[2] + oz};  // the source in children of the target's parent
    uint32_t v = (uint32_t)(((oz + 3) * 7 + (oy + 3)) * 7 + (ox + 3));
    for (int a = 0; a < 3; a++) {
        const int h = s[a] & 1, d = (s[a] - h) / 2;
        v |= (uint32_t)h << (9 + a) | (uint32_t)(d + 1) << (12 + 2 * a);
    }
    return v;
}
constexpr bool off_near(int ox, int oy, int oz) {
    return ox >= -1 && ox <= 1 && oy >= -1 && oy <= 1 && oz >= -1 && oz <= 1;
}
constexpr OffTable make_off_table() {
    OffTable t{};
    for (int par = 0; par < 8; par++) {
        const int b[3] = {par & 1, (par >> 1) & 1, par >> 2};
        int n = 0;
        for (int oz = -2 - b[2]; oz <= 3 - b[2]; oz++)
            for (int oy = -2 - b[1]; oy <= 3 - b[1]; oy++)
                for (int ox = -2 - b[0]; ox <= 3 - b[0]; ox++)
                    if (!off_near(ox, oy, oz)) t.v[0][par][n++] = off_entry(b, ox, oy, oz);
        n = 0;
        for (int sp = 0; sp < 8; sp++)
            for (int d = 0; d < 27; d++) {
                const int ox = 2 * (d % 3 - 1) + (sp & 1) - b[0], oy = 2 * (d / 3 % 3 - 1) + ((sp >> 1) & 1) - b[1],
                          oz = 2 * (d / 9 - 1) + (sp >> 2) - b[2];
                if (!off_near(ox, oy, oz)) t.v[1][par][n++] = off_entry(b, ox, oy, oz);
            }
    }
    return t;
}
struct Off {
    int oi, spar, dX, dY, dZ;
};
__host__ __device__ constexpr Off unpack_off(uint32_t v) {
    return Off{(int)(v & 511u), (int)((v >> 9) & 7u), (int)((v >> 12) & 3u) - 1, (int)((v >> 14) & 3u) - 1,
               (int)(v >> 16) - 1};
}
// both orders hold every offset of every target parity's list once, each with the
// source cell it leads to; order 1 goes by source parity
constexpr bool off_table_ok(const OffTable &t) {
    for (int ord = 0; ord < 2; ord++)
        for (int par = 0; par < 8; par++) {
            const int b[3] = {par & 1, (par >> 1) & 1, par >> 2};
            bool seen[343] = {};
            int last = 0;
            for (int i = 0; i < TC_NOFF; i++) {
                const Off f = unpack_off(t.v[ord][par][i]);
                const int o[3] = {f.oi % 7 - 3, f.oi / 7 % 7 - 3, f.oi / 49 - 3}, d[3] = {f.dX, f.dY, f.dZ};
                if (f.oi >= 343 || seen[f.oi] || off_near(o[0], o[1], o[2])) return false;
                seen[f.oi] = true;
                for (int a = 0; a < 3; a++) {
                    if (o[a] < -2 - b[a] || o[a] > 3 - b[a] || d[a] < -1 || d[a] > 1) return false;
                    if (2 * d[a] + ((f.spar >> a) & 1) != b[a] + o[a]) return false;
                }
                if (ord == 1 && f.spar < last) return false;
                last = f.spar;
            }
        }
    return true;
}
static_assert(off_table_ok(make_off_table()), "the interaction lists of the eight target parities");
__constant__ const OffTable c_off = make_off_table();
__device__ __forceinline__ Off list_offset(int ord, int par, int i) { return unpack_off(c_off.v[ord][par][i]); }

#define TC_F16X3 FMM_TC_F16X3
#define TC_F16X1 FMM_TC_F16X1
#define TC_BF16X3 FMM_TC_BF16X3
#define TC_F32 FMM_TC_F32

// A cell vector (and a kernel row) in chunks.
// Two parts: 128-byte chunks of 64 values, the hi and the lo part of every 64
// values in two chunks; a tail of at most 32 values has both in one (hi in its
// first half).  p = 3: 27 values, one chunk; 4: 64, two; 5: 125, four; 6: 216, seven.
// Three parts: 64-byte chunks, the three parts of every 32 values one after another.
template <int N, int MODE>
struct TcShape {
    static constexpr int CH = N > 64 || (N == 64 && MODE == TC_F32) ? 2 : 1;  // epilogue column groups
    static constexpr int EPI = 4 * CH;                  // epilogue warps
    static constexpr bool LO = MODE != TC_F16X1;        // lo parts loaded and used
    static constexpr bool SCALED = MODE != TC_BF16X3;   // operands scaled by powers of two
    static constexpr bool COMP = MODE == TC_F32;        // compensated sum over the offsets
    static constexpr bool P3 = COMP && N > 64;          // three parts per operand
    static constexpr int KS = N == 32 ? 2 : (N == 64 ? 4 : (N == 128 ? 8 : 14));  // MMA steps of 16 values
    static constexpr int FC = KS / 4;                   // two parts: stages of whole chunks (hi, lo)
    static constexpr int KC = P3 ? KS / 2 : (KS + 3) / 4;  // stages per offset
    static constexpr int RC = P3 ? 3 * KC : 2 * FC + (KC - FC);  // chunks per cell vector
    static constexpr int UB = P3 ? 64 : 128;            // bytes of a chunk's row
    static constexpr int ABYTES = TC_M * UB;            // one chunk of the tile's rows
    static constexpr int BBYTES = N * UB;               // one chunk of K_o
    static constexpr int NCH = P3 ? 3 : (FC ? 2 : 1);   // chunks of a stage (two parts: a tail stage has one)
    static constexpr int NCX = P3 ? 3 : 2;              // chunks from one stage to the next in a cell vector
    static constexpr int ACC = P3 ? 2 : 1;              // accumulators per offset
    // cross-system tiles keep the totals of their runs of offsets in TMEM, the
    // widest tile (two accumulators fill it) in the output
    static constexpr bool RMW = N == 224;
    static constexpr int TUSED = RMW ? 2 * N : 4 * N;  // two accumulators, and two rows of totals or accumulators
    static constexpr int TCOLS = TUSED <= 128 ? 128 : (TUSED <= 256 ? 256 : 512);
    static constexpr int COLS = N / CH;                 // columns per epilogue thread
};

// ---------------------------------------------------------------------------
// Occupied cells.  Only the functionals of cells that hold a charge are read
// (step 4 evaluates a cell's functional at its own charges, and a cell with
// charges has a parent with charges), so the contraction forms those alone:
// its 128-row tiles are cut from a list of the occupied cells of each (level,
// target parity) segment, in coarse Morton order, built after the sort.
// ---------------------------------------------------------------------------
struct OccParams {
    const int *leaf_start;
    int *occ;  // the workspace region (layout in fmm_internal.cuh)
    int depth, lmin, nseg, nblk;
    int N;     // tile width of the contraction (box or gathered tiles per segment)
    int bfirst[8 * (FMM_MAXDEPTH + 1) + 1];  // first block of each segment
};

// block -> segment, level, parity and its first coarse cell
__device__ __forceinline__ int occ_block_segment(const OccParams &op, int bid, int &l, int &par, int64_t &c0) {
    int s = 0;
    while (s + 1 < op.nseg && bid >= op.bfirst[s + 1]) s++;
    l = op.lmin + s / 8;
    par = s & 7;
    c0 = (int64_t)(bid - op.bfirst[s]) * OCC_BLOCK;
    return s;
}

// Occupancy of the four consecutive coarse cells of this thread (bit k: cell
// c0 + 4 threadIdx.x + k) and the block's exclusive prefix of their count.
__device__ __forceinline__ unsigned occ_flags(const OccParams &op, int l, int par, int64_t c0, int &pre,
                                              int &total) {
    __shared__ int wsum[OCC_BLOCK / 4 / 32];
    const int64_t ncs = occ_seg_cells(op.lmin, 8 * (l - op.lmin));
    unsigned f = 0;
#pragma unroll
    for (int k = 0; k < 4; k++) {
        const int64_t kc = c0 + 4 * threadIdx.x + k;
        if (kc < ncs && cell_occupied(op.leaf_start, op.depth, l, kc * 8 + par)) f |= 1u << k;
    }
    const int v = __popc(f), lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int inc = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += y;
    }
    if (lane == 31) wsum[warp] = inc;
    __syncthreads();
    int before = 0;
    total = 0;
#pragma unroll
    for (int w = 0; w < OCC_BLOCK / 4 / 32; w++) {
        before += w < warp ? wsum[w] : 0;
        total += wsum[w];
    }
    pre = before + inc - v;
    return f;
}

struct KOccCount {
    static constexpr int BS = OCC_BLOCK / 4, MINB = 0;  // bounds on the block size only
    OccParams op;
    __device__ __forceinline__ void run(const int bid_, const int nblk_) const {
        int l, par, pre, total;
        int64_t c0;
        occ_block_segment(op, bid_, l, par, c0);
        occ_flags(op, l, par, c0, pre, total);
        if (threadIdx.x == 0) op.occ[bid_] = total;
    }
};
__global__ void __launch_bounds__(KOccCount::BS) k_occ_count(const __grid_constant__ KOccCount k) {
    k.run(blockIdx.x, gridDim.x);
}

// per segment (one warp each): the blocks' exclusive prefix and the segment's count
struct KOccOffsets {
    static constexpr int BS = 0, MINB = 0;
    OccParams op;
    __device__ __forceinline__ void run(const int bid_, const int nblk_) const {
        int *bcnt = op.occ, *cnt = op.occ + op.nblk;
        const int s = (bid_ * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
        if (s >= op.nseg) return;
        int run = 0;
        for (int b0 = op.bfirst[s]; b0 < op.bfirst[s + 1]; b0 += 32) {
            const int b = b0 + lane;
            const int c = b < op.bfirst[s + 1] ? bcnt[b] : 0;
            int inc = c;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, inc, o);
                if (lane >= o) inc += y;
            }
            if (b < op.bfirst[s + 1]) bcnt[b] = run + inc - c;
            run += __shfl_sync(0xffffffffu, inc, 31);
        }
        if (lane == 0) cnt[s] = run;
    }
};
__global__ void k_occ_offsets(const __grid_constant__ KOccOffsets k) {
    k.run(blockIdx.x, gridDim.x);
}

// the list entries: coarse coordinates X | Y << 10 | Z << 20 of each occupied
// cell; block 0 also writes the prefix of the segments' blocks
struct KOccScatter {
    static constexpr int BS = OCC_BLOCK / 4, MINB = 0;  // bounds on the block size only
    OccParams op;
    __device__ __forceinline__ void run(const int bid_, const int nblk_) const {
        int l, par, pre, total;
        int64_t c0;
        const int s = occ_block_segment(op, bid_, l, par, c0);
        unsigned f = occ_flags(op, l, par, c0, pre, total);
        int *dst = op.occ + occ_list_offset(op.depth, op.lmin) + occ_seg_first(op.lmin, s) + op.occ[bid_] + pre;
        for (int k = 0; k < 4; k++) {
            if (f & (1u << k)) {
                int X, Y, Z;
                morton_decode((uint32_t)(c0 + 4 * threadIdx.x + k), X, Y, Z);
                *dst++ = X | (Y << 10) | (Z << 20);
            }
        }
        if (bid_ == 0 && threadIdx.x == 0) {
            const int *cnt = op.occ + op.nblk;
            int *tiles = op.occ + op.nblk + op.nseg;
            int t = 0;
            for (int k = 0; k < op.nseg; k++) {  // the deepest level's blocks first
                const int sg = op.nseg - 1 - k, lv = op.lmin + sg / 8;
                tiles[k] = t;
                t += occ_seg_tiles(1 << (lv - 1), cnt[sg], op.N) * tc_parts(lv, op.depth);
            }
            tiles[op.nseg] = t;
        }
    }
};
__global__ void __launch_bounds__(KOccScatter::BS) k_occ_scatter(const __grid_constant__ KOccScatter k) {
    k.run(blockIdx.x, gridDim.x);
}

// ---------------------------------------------------------------------------
// The contraction over the occupied-cell lists.  A block takes one 128-row tile
// of a segment (level l, target parity b): row r is the tile's r-th occupied
// target cell, and its A operand row for offset o is the source cell (target +
// o), gathered with cp.async (or one box copy); the kernel matrix B arrives by
// TMA box copies.  Levels with few tiles split the 189 offsets over tc_parts
// blocks, whose partial functionals k_tc_reduce adds.
//
// What bounds it (GB300): p = 4 the shared-memory traffic of operands and MMAs
// (N = 64 reads 6 KB per 32-cycle MMA), p = 5 and 6 the tensor pipe and the
// operand copies; with three parts at p = 6 also the wait for the epilogue, since
// one offset's two accumulators fill the tensor memory.
// ---------------------------------------------------------------------------
struct TcgParams {
    CUtensorMap k;                        // kernel tables: [343][N] rows of chunks
    CUtensorMap phi[FMM_MAXDEPTH + 1];    // box maps of the operand copy, per level
    const char *op;                       // the operand copy
    int lmin, depth, p3, spow, nseg;
    const int *occ;             // occupied-cell lists
    long long loc_off[FMM_MAXDEPTH + 1];
    long long q_off[FMM_MAXDEPTH + 1];    // first cell of a level in the padded layout
    long long part_off[FMM_MAXDEPTH + 1], part_stride[FMM_MAXDEPTH + 1];  // partials of levels with tc_parts > 1
    float *loc;
    float *part;
    const float2 *qsc;  // per cell: total charge, factor of its scaled operands (see KSplit)
    const float *kbar;  // [343][N], zero padded
    int *status;
    int inject_stall;   // test hook: the first stage's kernel copies are withheld
    // Cross-system tiles (batched evaluations; xsys != nullptr): the levels
    // lmin..depth of many systems whose levels have fewer than 8 coarse cells
    // per axis, every cell of every system one row, gathered.  xseg: [nseg]
    // rows per segment, [nseg + 1] prefix of their tiles, [nseg] first list
    // entry, then the list (system << 12 | Z << 8 | Y << 4 | X); xsys: per
    // system its operand copy, charges and functionals (qsc, loc above are
    // unused; op is the start of the batch's workspace).
    const TcXSys *xsys;
    const int *xseg;
};

// Ring depths per tile shape.  N >= 128: the A stages (32 KB) and the kernel
// stages (N 256 bytes) are separate rings with their own producers, one CTA per
// SM (N = 224: 3 A + 2 B stages, 208 KB; N = 128: 3 + 3, 192 KB; three parts: stages
// of 24 KB and N 192 bytes, 3 + 3 and 4 + 4, 198 and 192 KB).  Dynamic plus static
// shared memory stays below 227 KB.  N <= 64 (UNI): one ring whose
// stages hold A and B, six warps and two CTAs per SM (each CTA's barrier round
// trips and epilogue hide under the other's MMAs).  The three-part shapes need about
// 210 registers per epilogue thread (N = 224: 112 sums and their compensations): the
// other warpgroup gives its share up (216 x 256 + 72 x 128 = 168 x 384).
template <int N, int MODE>
struct TcgShape {
    typedef TcShape<N, MODE> B;
    static constexpr bool UNI = N <= 64;
    static constexpr int SA = N == 32 || (N == 128 && B::P3) ? 4 : (N == 64 ? 2 : 3);
    static constexpr int SB = N == 224 && !B::P3 ? 2 : SA;
    static constexpr int ASTAGE = B::NCH * B::ABYTES;
    static constexpr int BSTAGE = B::NCH * B::BBYTES;
    static constexpr int PW = UNI ? 1 : 2;           // A warps
    static constexpr int G = SA - 1;                 // stages of copies in flight per gathering thread
    static constexpr int WA = B::EPI;
    static constexpr int WB = WA + PW;               // kernel-matrix warp (split rings)
    static constexpr int WM = UNI ? WB : WB + 1;     // MMA warp
    static constexpr bool SETREG = B::P3;
    static constexpr int THREADS = 32 * (WM + 1);
    static_assert(!SETREG || THREADS == 384, "three warpgroups");
    static constexpr int MINB = UNI ? 2 : 1;
    // rings, barriers, two offsets' row means, the rows' tables
    static constexpr int SMEM = 1024 + SA * ASTAGE + SB * BSTAGE + 256 + 2 * N * 4 + 4 * TC_M * 4;
    static_assert(SMEM + 1024 <= 227 * 1024, "shared memory of one CTA");
};

// One step of a compensated sum of pairs: run += y, where y holds the new term and
// the rounding error of the last step, which comp carried; comp takes this step's.
__device__ __forceinline__ float2 kahan_error(float2 &run, float2 y) {
    const float2 m1 = make_float2(-1.0f, -1.0f);
    const float2 s = __fadd2_rn(run, y);
    const float2 e = __ffma2_rn(__ffma2_rn(run, m1, s), m1, y);
    run = s;
    return e;
}
__device__ __forceinline__ float2 comp_value(float2 c) { return c; }
__device__ __forceinline__ void kahan_add(float2 &run, float2 &comp, float2 y) { comp = kahan_error(run, y); }
__device__ __forceinline__ void comp_keep(float2 &comp, float2 y) { comp = y; }
__device__ __forceinline__ void comp_keep(uint32_t &, float2) {}
// N = 224, where 112 sums and as many floats do not fit a thread's registers: the
// error's leading eight bits (two bfloat16), so that a sum is carried with 24 + 8
// bits; what is left out is below 2^-33 of a partial sum each step
__device__ __forceinline__ float2 comp_value(uint32_t c) {
    return make_float2(__uint_as_float(c << 16), __uint_as_float(c & 0xFFFF0000u));
}
__device__ __forceinline__ void kahan_add(float2 &run, uint32_t &comp, float2 y) {
    const float2 e = kahan_error(run, y);
    const __nv_bfloat162 c = __floats2bfloat162_rn(e.x, e.y);
    comp = *reinterpret_cast<const uint32_t *>(&c);
}

// The next part of a sum of several runs: (h, w) += t with the rounding error
// of the addition kept in w; after the last part h is the sum.
__device__ __forceinline__ void part_add(float &h, float &w, float t, bool last) {
    const float s = h + t, b = s - h;
    w += (h - (s - b)) + (t - b);
    h = last ? s + w : s;
}

template <int N, int MODE, bool CROSS = false>
struct KM2LTcg {
    static constexpr int BS = TcgShape<N, MODE>::THREADS, MINB = TcgShape<N, MODE>::MINB;
    static constexpr int SMEM = TcgShape<N, MODE>::SMEM;
    TcgParams prm;
    __device__ __forceinline__ void run(const int bid_, const int nblk_) const {
        typedef TcShape<N, MODE> Sh;
        typedef TcgShape<N, MODE> Gh;
        // the segments' counts and block prefix, read once into shared memory
        __shared__ int seg_cnt[8 * (FMM_MAXDEPTH + 1)], seg_first[8 * (FMM_MAXDEPTH + 1) + 1];
        constexpr bool cross = CROSS;
        {
            const int *cnt_g = cross ? prm.xseg : prm.occ + occ_nblk(prm.depth, prm.lmin), *first_g = cnt_g + prm.nseg;
            if ((int)threadIdx.x <= prm.nseg) seg_first[threadIdx.x] = first_g[threadIdx.x];
            if ((int)threadIdx.x < prm.nseg) seg_cnt[threadIdx.x] = cnt_g[threadIdx.x];
            __syncthreads();
        }
        if ((int)bid_ >= seg_first[prm.nseg]) return;  // past the last occupied tile
        int k = 0;
        while (k + 1 < prm.nseg && (int)bid_ >= seg_first[k + 1]) k++;
        const int sg = cross ? k : prm.nseg - 1 - k;  // a system's own blocks: the deepest level first
        const int l = prm.lmin + sg / 8, par = sg & 7;
        const int H = 1 << (l - 1), P = H + 2, ord = off_order(l);
        const int count = seg_cnt[sg];
        const int parts = cross ? 1 : tc_parts(l, prm.depth);
        const int tile = ((int)bid_ - seg_first[k]) / parts, part = ((int)bid_ - seg_first[k]) % parts;
        const int i0 = part * (TC_NOFF / parts), i1 = i0 + TC_NOFF / parts;  // this block's offsets
        const int r0 = tile * TC_M;  // first list entry of the tile
        const int *lst = cross ? prm.xseg + 3 * prm.nseg + 1 + prm.xseg[2 * prm.nseg + 1 + sg]
                               : prm.occ + occ_list_offset(prm.depth, prm.lmin) + occ_seg_first(prm.lmin, sg);

        extern __shared__ unsigned char smraw[];
        const uint32_t raw = tc::smem_u32(smraw);
        const uint32_t abase = (raw + 1023u) & ~1023u;           // A ring
        const uint32_t bbase = abase + Gh::SA * Gh::ASTAGE;       // B ring
        const uint32_t bars = bbase + Gh::SB * Gh::BSTAGE;
        const uint32_t afull0 = bars, aempty0 = afull0 + 8 * Gh::SA;
        const uint32_t bfull0 = aempty0 + 8 * Gh::SA, bempty0 = bfull0 + 8 * Gh::SB;
        const uint32_t rfull0 = bempty0 + 8 * Gh::SB, rfree0 = rfull0 + 32;
        const uint32_t done = rfree0 + 32;
        const uint32_t tslot = done + 8;
        volatile uint32_t *tslot_ptr = reinterpret_cast<volatile uint32_t *>(smraw + (tslot - raw));
        float *kbs = reinterpret_cast<float *>(smraw + (bars - raw) + 256);  // row means of two offsets
        // per row: first chunk of its own cell in the operand copy, cell in the
        // padded layout, target cell in the L layout (-1: past the list), system
        int *rowG = reinterpret_cast<int *>(kbs + 2 * N);
        int *rowQ = rowG + TC_M, *rowL = rowQ + TC_M, *rowS = rowL + TC_M;

        // chunks of an offset's kc-th stage (two parts: a tail holds hi and lo in one)
        auto stage_chunks = [](int kc) { return Sh::P3 ? 3 : (kc < Sh::FC && Sh::LO ? 2 : 1); };
        // Box tiles (occ_box_segment): tile t is the 128 consecutive Morton cells
        // [128 t, 128 t + 128), one 8 x 4 x 4 box, and each chunk's A operand is
        // one TMA box copy (row r = x + 8 y + 32 z of the box).
        const bool box = !cross && occ_box_segment(H, count, N);
        // gathers: lanes per row (16 bytes each) and rows per group; rows past the list
        // hold no operand, and groups of such rows are not copied
        constexpr int LPR = Sh::UB / 16, RPG = 32 / LPR;
        const int ngroups = (min(TC_M, count - r0) + RPG - 1) / RPG;
        // accumulators in tensor memory: those of two offsets, but of one for the pairs
        // of the widest tile, and of a cross-system tile beside its totals.  The i-th
        // accumulator of the block, in the order they are read, is region i mod NR.
        constexpr int NR = Sh::P3 && N == 128 && !cross ? 4 : 2;
        int X0 = 0, Y0 = 0, Z0 = 0;
        if (box) morton_decode((uint32_t)r0, X0, Y0, Z0);
        const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
        if (threadIdx.x < TC_M) {
            const int r = threadIdx.x;
            int X, Y, Z, sys = 0;
            bool in = true;
            if (box) {
                X = X0 + (r & 7);
                Y = Y0 + ((r >> 3) & 3);
                Z = Z0 + (r >> 5);
            } else {
                in = r0 + r < count;
                const int pk = lst[in ? r0 + r : r0];  // rows past the list repeat the tile's first cell
                if (cross) {
                    X = pk & 15;
                    Y = (pk >> 4) & 15;
                    Z = (pk >> 8) & 15;
                    sys = pk >> 12;
                } else {
                    X = pk & 1023;
                    Y = (pk >> 10) & 1023;
                    Z = pk >> 20;
                }
            }
            rowQ[r] = ((Z + 1) * P + Y + 1) * P + X + 1;
            rowL[r] = in ? ((par * H + Z) * H + Y) * H + X : -1;
            rowS[r] = sys;
            rowG[r] = (cross ? prm.xsys[sys].op_chunk : 0) + (int)(prm.q_off[l] + rowQ[r]) * Sh::RC;
        }
        if (threadIdx.x == 0) {
            for (int s = 0; s < Gh::SA; s++) {
                // arrivals: the copies' issuer (box), or every gathering thread (and
                // the issuer of the B copies that share the ring)
                tc::mbar_init(afull0 + 8 * s, box ? 1 : 32 * Gh::PW + (Gh::UNI ? 1 : 0));
                tc::mbar_init(aempty0 + 8 * s, 1);
            }
            for (int s = 0; s < Gh::SB; s++) {
                tc::mbar_init(bfull0 + 8 * s, 1);
                tc::mbar_init(bempty0 + 8 * s, 1);
            }
            for (int r = 0; r < NR; r++) {
                tc::mbar_init(rfull0 + 8 * r, 1);
                tc::mbar_init(rfree0 + 8 * r, 32 * Sh::EPI);
            }
            tc::mbar_init(done, 1);
            tc::fence_barrier_init();
        }
        if (warp == 0) tc::tmem_alloc(tslot, Sh::TCOLS);
        tc::fence_before_sync();
        __syncthreads();
        tc::fence_after_sync();
        const uint32_t tmem = *tslot_ptr;
        // Register shares (SETREG): whole warpgroups 0-3 and 4-7 (epilogue) and 8-11,
        // each group's change one instruction, its role inside the branch.
        if (warp < Sh::EPI) {
            if constexpr (Gh::SETREG) tc::setmaxnreg_inc<216>();
            // ---- epilogue: TMEM lane = row; columns [c0, c0 + COLS) ----
            const int sub = warp & 3, cgrp = warp >> 2;
            const int c0 = cgrp * Sh::COLS;
            const int row = sub * 32 + lane;
            const int lrow = rowL[row];
            const bool valid = lrow >= 0;
            const float2 *q = (cross ? prm.xsys[rowS[row]].qsc : prm.qsc) + prm.q_off[l] + rowQ[row];
            const int p3 = prm.p3;
            float *out = (cross ? prm.xsys[rowS[row]].loc + prm.loc_off[l]
                          : parts > 1 ? prm.part + prm.part_off[l] + part * prm.part_stride[l] : prm.loc + prm.loc_off[l]) +
                         (int64_t)(valid ? lrow : 0) * p3 + c0;
            // the totals' low parts of the widest cross-system tile
            float *out_lo = cross && Sh::RMW
                                ? prm.xsys[rowS[row]].part + prm.loc_off[l] + (int64_t)(valid ? lrow : 0) * p3 + c0 : nullptr;
            const float scale = (float)(1 << (l * prm.spow));
            // where the totals of a cross-system tile's runs wait (this thread's columns)
            const uint32_t ttot = tmem + ((uint32_t)(sub * 32) << 16) + (uint32_t)(2 * N + c0);
            float2 run[Sh::COLS / 2];
            typedef typename std::conditional<N == 224, uint32_t, float2>::type Comp;
            Comp comp[Sh::COMP ? Sh::COLS / 2 : 1];
#pragma unroll
            for (int j = 0; j < Sh::COLS / 2; j++) {
                run[j] = make_float2(0.0f, 0.0f);
                if (Sh::COMP) comp[j] = Comp{};
            }
            constexpr int LDC = Sh::COMP && N == 64 ? 8 : 16;  // columns per read
            bool ok = true;
            // the row's source charge and factor, and the row means Kbar_o, are
            // fetched one offset ahead: the charge into registers, the means by the
            // epilogue's threads into a shared row
            auto source = [&](int i) {
                const Off f = list_offset(ord, par, i);
                return valid ? q[((f.spar * P + f.dZ) * P + f.dY) * P + f.dX] : make_float2(0.0f, 0.0f);
            };
            const int et = threadIdx.x;  // epilogue thread (the epilogue warps come first)
            float2 qs = source(i0);
            if (et < N) kbs[et] = prm.kbar[list_offset(ord, par, i0).oi * N + et];
            asm volatile("bar.sync 1, %0;" ::"n"(32 * Sh::EPI) : "memory");
            for (int i = i0; i < i1; i++) {
                const int j = i - i0, in = i + 1 < i1 ? i + 1 : i;
                const float2 qn = source(in);
                const float kn = et < N ? prm.kbar[list_offset(ord, par, in).oi * N + et] : 0.0f;
                const float2 Q2 = make_float2(qs.x, qs.x), inv2 = make_float2(qs.y, qs.y);
                const float *kb = kbs + (j & 1) * N + c0;
#pragma unroll 1
                for (int h = 0; h < Sh::ACC; h++) {
                const int r = (j * Sh::ACC + h) % NR;
                const uint32_t u = (uint32_t)((j * Sh::ACC + h) / NR) & 1u;
                if (ok && !tc::mbar_wait(rfull0 + 8 * r, u, TC_WAIT_CYCLES)) {
                    if (lane == 0) tc_wait_failed(prm.status, 4, l, j);
                    ok = false;
                }
                tc::fence_after_sync();
                const uint32_t taddr = tmem + ((uint32_t)(sub * 32) << 16) + (uint32_t)(r * N + c0);
#pragma unroll
                for (int c = 0; c < Sh::COLS / LDC; c++) {
                    uint32_t v[LDC];
                    if constexpr (LDC == 8) tc::tmem_ld8(taddr + c * LDC, v);
                    else tc::tmem_ld16(taddr + c * LDC, v);
#pragma unroll
                    for (int e = 0; e < LDC; e += 2) {
                        // the offset's contribution, with its monopole term Kbar Q in the last
                        // accumulator (the factor is a power of two: the sum is rounded once, and
                        // once with the error that the last addition left)
                        const int x = (c * LDC + e) / 2;
                        const float2 m = *reinterpret_cast<const float2 *>(kb + c * LDC + e);
                        float2 d = make_float2(__uint_as_float(v[e]), __uint_as_float(v[e + 1]));
                        if constexpr (Sh::COMP) {
                            d = __ffma2_rn(d, inv2, comp_value(comp[x]));
                            if (h == Sh::ACC - 1) d = __ffma2_rn(m, Q2, d);
                            if (h < Sh::ACC - 1 && N != 224) comp_keep(comp[x], d);  // joins the sum with the next term
                            else kahan_add(run[x], comp[x], d);
                        } else {
                            run[x] = __fadd2_rn(run[x], __ffma2_rn(m, Q2, Sh::SCALED ? __fmul2_rn(d, inv2) : d));
                        }
                    }
                }
                tc::fence_before_sync();
                tc::mbar_arrive(rfree0 + 8 * r);
                }
                qs = qn;
                if (et < N) kbs[((j + 1) & 1) * N + et] = kn;
                asm volatile("bar.sync 1, %0;" ::"n"(32 * Sh::EPI) : "memory");
                // a cross-system tile adds its offsets in the same runs as a system's
                // own blocks of these levels do (one run per block, added by
                // k_tc_reduce in order), for the same sums bit for bit
                if (cross && (j + 1) % (TC_NOFF / TC_PARTS_SMALL) == 0) {
                    const bool first = j + 1 == TC_NOFF / TC_PARTS_SMALL, last = j + 1 == TC_NOFF;
                    if constexpr (Sh::RMW) {  // p^3 = 216 values: rows of whole, aligned float4
                        if (ok && valid) {
#pragma unroll
                            for (int e = 0; e < Sh::COLS; e += 4) {
                                if (c0 + e >= p3) break;
                                float4 *h4 = reinterpret_cast<float4 *>(out + e), *w4 = reinterpret_cast<float4 *>(out_lo + e);
                                const float4 z = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                                float4 h = first ? z : *h4, w = first ? z : *w4;
                                part_add(h.x, w.x, scale * run[e / 2].x, last);
                                part_add(h.y, w.y, scale * run[e / 2].y, last);
                                part_add(h.z, w.z, scale * run[e / 2 + 1].x, last);
                                part_add(h.w, w.w, scale * run[e / 2 + 1].y, last);
                                *h4 = h;
                                if (!last) *w4 = w;
                            }
                        }
                    } else {
#pragma unroll
                        for (int c = 0; c < Sh::COLS / 8; c++) {
                            uint32_t h[8], w[8];
#pragma unroll
                            for (int e = 0; e < 8; e++) h[e] = w[e] = 0u;
                            if (!first) {
                                tc::tmem_ld8(ttot + c * 8, h);
                                tc::tmem_ld8(ttot + N + c * 8, w);
                            }
#pragma unroll
                            for (int e = 0; e < 8; e++) {
                                float &t = e & 1 ? run[c * 4 + e / 2].y : run[c * 4 + e / 2].x;
                                float hf = __uint_as_float(h[e]), wf = __uint_as_float(w[e]);
                                part_add(hf, wf, t, last);
                                if (last) t = hf;
                                h[e] = __float_as_uint(hf);
                                w[e] = __float_as_uint(wf);
                            }
                            if (!last) {
                                tc::tmem_st8(ttot + c * 8, h);
                                tc::tmem_st8(ttot + N + c * 8, w);
                            }
                        }
                        tc::tmem_wait_st();
                    }
                    if (j + 1 < TC_NOFF) {
#pragma unroll
                        for (int e = 0; e < Sh::COLS / 2; e++) {
                            run[e] = make_float2(0.0f, 0.0f);
                            if (Sh::COMP) comp[e] = Comp{};
                        }
                    }
                }
            }
            if (ok) {
                if (!(cross && Sh::RMW) && valid) {
#pragma unroll
                    for (int e = 0; e < Sh::COLS; e++)
                        if (c0 + e < p3) out[e] = scale * (e & 1 ? run[e / 2].y : run[e / 2].x);
                }
            } else if (lane == 0) {
                atomicOr(prm.status, ST_TIMEOUT);
            }
        } else {
            if constexpr (Gh::SETREG) tc::setmaxnreg_dec<72>();
            if (warp < Gh::WA + Gh::PW) {
                // ---- A producers; with one ring (UNI) the first lane also issues the
                //      stage's B copies.  Gather: lane = LPR (row within a group) + 16-byte
                //      piece; warp pw takes the groups pw + PW i.  A stage is signalled once
                //      its copies are complete and fenced, G - 1 stages later. ----
                const int pw = warp - Gh::WA;
                const bool lead = pw == 0 && lane == 0;
                if (lead) {
                    if (box) tc::tensormap_acquire(&prm.phi[l]);
                    if (Gh::UNI) tc::tensormap_acquire(&prm.k);
                }
                constexpr int RI = TC_M / RPG / Gh::PW;
                const int piece = lane % LPR, rsub = lane / LPR;
                // groups of this warp that hold rows of the tile
                const int ni = box ? 0 : (ngroups - pw + Gh::PW - 1) / Gh::PW;
                int g[RI];
                // shared-memory places of the first NPL groups, the further ones 1 KB a pair
                // of four-row groups (128-byte rows), 1 KB a group here (64-byte rows, PW = 2)
                constexpr int NPL = Sh::P3 ? 1 : 2 / Gh::PW;
                static_assert(!Sh::P3 || Gh::PW == 2, "places of the 64-byte rows");
                uint32_t place[NPL];
                if (!box) {
#pragma unroll
                    for (int i = 0; i < RI; i++) g[i] = rowG[RPG * (pw + Gh::PW * i) + rsub];
#pragma unroll
                    for (int i = 0; i < NPL; i++) {
                        const int r = RPG * (pw + Gh::PW * i) + rsub;
                        // 128-byte swizzle: piece ^ (row mod 8); 64-byte: piece ^ (row / 2 mod 4)
                        place[i] = (uint32_t)(r * Sh::UB + ((piece ^ (Sh::P3 ? (r >> 1) & 3 : r & 7)) << 4));
                    }
                }
                const char *src0 = prm.op + 16 * piece;
                bool failed = false;
                int last_phase[4] = {-1, -1, -1, -1};
                int it = 0, sig = 0;  // sig: next gathered stage to signal
                for (int i = i0; i < i1 && !failed; i++) {
                    const Off f = list_offset(ord, par, i);
                    const int delta = (((f.spar * P + f.dZ) * P + f.dY) * P + f.dX) * Sh::RC;
#pragma unroll 1
                    for (int kc = 0; kc < Sh::KC; kc++, it++) {
                        const int s = it % Gh::SA;
                        const uint32_t ph = (uint32_t)(it / Gh::SA) & 1u;
                        if (!tc::mbar_wait(aempty0 + 8 * s, ph ^ 1u, TC_WAIT_CYCLES)) {
                            if (lane == 0) tc_wait_failed(prm.status, 1, l, it);
                            failed = true;
                            break;
                        }
                        const uint32_t st = abase + s * Gh::ASTAGE, fb = afull0 + 8 * s;
                        const int nch = stage_chunks(kc);
                        if (lead && (box || Gh::UNI)) {
                            tc::mbar_expect_tx(fb, (uint32_t)(nch * ((box ? Sh::ABYTES : 0) + (Gh::UNI ? Sh::BBYTES : 0))));
                            last_phase[s] = (int)ph;
                            if (box) {
                                const int cX = X0 + 1 + f.dX, cY = Y0 + 1 + f.dY, cZ = Z0 + 1 + f.dZ;
#pragma unroll
                                for (int t = 0; t < Sh::NCH; t++)
                                    if (t < nch)
                                        tc::tma_load_5d(st + t * Sh::ABYTES, &prm.phi[l], fb, (Sh::NCX * kc + t) * (Sh::UB / 2), cX,
                                                        cY, cZ, f.spar);
                            }
                            if (Gh::UNI && !(prm.inject_stall && it == 0)) {  // inject: armed, never filled
                                const uint32_t stb = bbase + s * Gh::BSTAGE;
#pragma unroll
                                for (int t = 0; t < Sh::NCH; t++)
                                    if (t < nch)
                                        tc::tma_load_3d(stb + t * Sh::BBYTES, &prm.k, fb, (Sh::NCX * kc + t) * (Sh::UB / 2), 0, f.oi);
                            }
                        }
                        if (box) continue;
                        const int d = delta + Sh::NCX * kc;
#pragma unroll
                        for (int i = 0; i < RI; i++) {
                            if (i >= ni) break;
                            const char *src = src0 + (int64_t)(g[i] + d) * Sh::UB;
                            const uint32_t to = st + place[i % NPL] + 1024 * (i / NPL);
#pragma unroll
                            for (int t = 0; t < Sh::NCH; t++)
                                if (t < nch) tc::cp_async16(to + t * Sh::ABYTES, src + t * Sh::UB);
                        }
                        tc::cp_async_commit();
                        tc::cp_async_wait_pending<Gh::G - 1>();  // stages <= it - G + 1 have landed
                        if (it - Gh::G + 1 >= sig) {
                            tc::fence_proxy_async_smem();
                            for (; sig <= it - Gh::G + 1; sig++) tc::mbar_arrive(afull0 + 8 * (sig % Gh::SA));
                        }
                    }
                }
                if (!box) {
                    tc::cp_async_wait_all();  // no copy outlives the CTA
                    if (!failed) {
                        tc::fence_proxy_async_smem();
                        for (; sig < it; sig++) tc::mbar_arrive(afull0 + 8 * (sig % Gh::SA));
                    }
                }
                if (failed) {
                    if (lane == 0) atomicOr(prm.status, ST_TIMEOUT);
                    if (lead)  // the TMA copies already issued land before the CTA can exit
                        for (int s = 0; s < Gh::SA; s++)
                            if (last_phase[s] >= 0) tc::mbar_wait(afull0 + 8 * s, (uint32_t)last_phase[s], TC_WAIT_CYCLES);
                }
            } else if (!Gh::UNI && warp == Gh::WB) {
                // ---- kernel-matrix producer (split rings): the chunks of K_o by TMA ----
                if (lane == 0) {
                    tc::tensormap_acquire(&prm.k);
                    bool failed = false;
                    int last_phase[4] = {-1, -1, -1, -1};
                    int it = 0;
                    for (int i = i0; i < i1 && !failed; i++) {
                        const int oi = list_offset(ord, par, i).oi;
                        for (int kc = 0; kc < Sh::KC; kc++, it++) {
                            const int s = it % Gh::SB;
                            const uint32_t ph = (uint32_t)(it / Gh::SB) & 1u;
                            if (!tc::mbar_wait(bempty0 + 8 * s, ph ^ 1u, TC_WAIT_CYCLES)) {
                                tc_wait_failed(prm.status, 1, l, it);
                                failed = true;
                                break;
                            }
                            const uint32_t st = bbase + s * Gh::BSTAGE, fb = bfull0 + 8 * s;
                            const int nch = stage_chunks(kc);
                            tc::mbar_expect_tx(fb, (uint32_t)(nch * Sh::BBYTES));
                            last_phase[s] = (int)ph;
                            if (prm.inject_stall && it == 0) continue;  // armed, never filled (test hook)
#pragma unroll
                            for (int t = 0; t < Sh::NCH; t++)
                                if (t < nch) tc::tma_load_3d(st + t * Sh::BBYTES, &prm.k, fb, (Sh::NCX * kc + t) * (Sh::UB / 2), 0, oi);
                        }
                    }
                    if (failed) {
                        atomicOr(prm.status, ST_TIMEOUT);
                        // the copies already issued land before the CTA can exit
                        for (int s = 0; s < Gh::SB; s++)
                            if (last_phase[s] >= 0) tc::mbar_wait(bfull0 + 8 * s, (uint32_t)last_phase[s], TC_WAIT_CYCLES);
                    }
                }
            } else if (warp == Gh::WM) {
                // ---- MMA issuer: the j-th offset of the block accumulates into regions ACC j mod NR and up ----
                if (lane == 0) {
                    const uint32_t idesc = MODE == TC_BF16X3 ? tc::idesc_bf16(TC_M, N) : tc::idesc_f16(TC_M, N);
                    bool failed = false;
                    for (int j = 0; j < i1 - i0 && !failed; j++) {
                        // the accumulators of the offset: d0 of the leading (or all) products, read
                        // last, d1 of the others
                        const int u0 = j * Sh::ACC, u1 = u0 + Sh::ACC - 1;
                        const uint32_t d1 = tmem + (uint32_t)(u0 % NR * N), d0 = tmem + (uint32_t)(u1 % NR * N);
                        auto region_free = [&](int i) {
                            if (tc::mbar_wait(rfree0 + 8 * (i % NR), ((uint32_t)(i / NR) & 1u) ^ 1u, TC_WAIT_CYCLES)) return true;
                            tc_wait_failed(prm.status, 2, l, j);
                            return false;
                        };
                        if (!region_free(u0)) {
                            failed = true;
                            break;
                        }
#pragma unroll (Sh::P3 ? 1 : Sh::KC)
                        for (int kc = 0; kc < Sh::KC; kc++) {
                            const int it = Sh::KC * j + kc;
                            const int sa = it % Gh::SA, sb = it % Gh::SB;
                            if (!tc::mbar_wait(afull0 + 8 * sa, (uint32_t)(it / Gh::SA) & 1u, TC_WAIT_CYCLES) ||
                                (!Gh::UNI && !tc::mbar_wait(bfull0 + 8 * sb, (uint32_t)(it / Gh::SB) & 1u, TC_WAIT_CYCLES))) {
                                tc_wait_failed(prm.status, 3, l, it);
                                failed = true;
                                break;
                            }
                            tc::fence_after_sync();
                            const uint32_t a0 = abase + sa * Gh::ASTAGE, b0 = bbase + sb * Gh::BSTAGE;
                            // 32 bytes of K (16 values) per MMA
                            if constexpr (Sh::P3) {
                                // the smaller products into one accumulator, smallest first; the
                                // leading ones into another, where every sum is exact (KSplit) and
                                // which may still be read while the first stage's others run
#pragma unroll
                                for (int s = 0; s < 2; s++) {
                                    uint64_t A[3], B[3];
#pragma unroll
                                    for (int t = 0; t < 3; t++) {
                                        A[t] = tc::desc_sw64(a0 + t * Sh::ABYTES + 32 * s);
                                        B[t] = tc::desc_sw64(b0 + t * Sh::BBYTES + 32 * s);
                                    }
                                    tc::mma_f16(d1, A[2], B[0], idesc, (kc | s) != 0);
                                    tc::mma_f16(d1, A[0], B[2], idesc, 1u);
                                    tc::mma_f16(d1, A[1], B[1], idesc, 1u);
                                    tc::mma_f16(d1, A[1], B[0], idesc, 1u);
                                    tc::mma_f16(d1, A[0], B[1], idesc, 1u);
                                }
                                if (kc == 0) {
                                    if (!region_free(u1)) {
                                        failed = true;
                                        break;
                                    }
                                    tc::fence_after_sync();
                                }
#pragma unroll
                                for (int s = 0; s < 2; s++)
                                    tc::mma_f16(d0, tc::desc_sw64(a0 + 32 * s), tc::desc_sw64(b0 + 32 * s), idesc, (kc | s) != 0);
                            } else {
                                // the stage's hi and lo parts: two chunks, or the halves of a tail
                                // chunk; the small products of the stage first, so that they meet an
                                // accumulator of their own size
                                const bool full = kc < Sh::FC;
                                const uint32_t al = a0 + (full ? Sh::ABYTES : 64), bl = b0 + (full ? Sh::BBYTES : 64);
                                if (Sh::LO) {
#pragma unroll
                                    for (int s = 0; s < 4; s++) {
                                        if (s >= 2 && !full) break;
                                        tc::mma_f16(d0, tc::desc_sw128(a0 + 32 * s), tc::desc_sw128(bl + 32 * s), idesc, (kc | s) != 0);
                                        tc::mma_f16(d0, tc::desc_sw128(al + 32 * s), tc::desc_sw128(b0 + 32 * s), idesc, 1u);
                                    }
                                }
#pragma unroll
                                for (int s = 0; s < 4; s++)
                                    if (s < 2 || full)
                                        tc::mma_f16(d0, tc::desc_sw128(a0 + 32 * s), tc::desc_sw128(b0 + 32 * s), idesc,
                                                    Sh::LO || (kc | s) != 0);
                            }
                            tc::mma_commit(aempty0 + 8 * sa);
                            if (!Gh::UNI) tc::mma_commit(bempty0 + 8 * sb);
                        }
                        for (int i = u0; i <= u1 && !failed; i++) tc::mma_commit(rfull0 + 8 * (i % NR));
                    }
                    if (failed) atomicOr(prm.status, ST_TIMEOUT);
                    tc::mma_commit(done);  // always: the deallocation waits on it
                }
            }
        }
        tc::fence_before_sync();
        __syncthreads();
        if (warp == 0) {
            tc::mbar_wait(done, 0, TC_WAIT_CYCLES);
            tc::fence_after_sync();
            tc::tmem_dealloc(tmem, Sh::TCOLS);
        }
    }
};
template <int N, int MODE>
__global__ void __launch_bounds__(KM2LTcg<N, MODE>::BS, KM2LTcg<N, MODE>::MINB) k_m2l_tcg(const __grid_constant__ KM2LTcg<N, MODE> k) {
    k.run(blockIdx.x, gridDim.x);
}
// cross-system tiles: launched merged only (their functor lives in the batch's table)
template <int N, int MODE>
__global__ void __launch_bounds__(KM2LTcg<N, MODE, true>::BS, KM2LTcg<N, MODE, true>::MINB)
    k_m2l_tcx(const __grid_constant__ KM2LTcg<N, MODE, true> k) {
    k.run(blockIdx.x, gridDim.x);
}

// The partials of the levels whose offsets are split over blocks, added in
// order of the offsets (every cell of those levels; cells without charges hold
// no partials and their sums are never read).
struct KTcReduce {
    static constexpr int BS = 256, MINB = 0;
    const float *__restrict__ part;
    float *__restrict__ loc;
    int nlev;
    int parts[4];
    long long first[5];  // prefix of the levels' values
    long long part_off[4], part_stride[4], loc_off[4];
    __device__ __forceinline__ void run(const int bid_, const int nblk_) const {
        for (int64_t i = (int64_t)bid_ * BS + threadIdx.x; i < first[nlev]; i += (int64_t)nblk_ * BS) {
            int v = 0;
            while (i >= first[v + 1]) v++;
            const int64_t e = i - first[v];
            const float *p = part + part_off[v] + e;
            float h = 0.0f, w = 0.0f;
            for (int k = 0; k < parts[v]; k++) part_add(h, w, p[k * part_stride[v]], k + 1 == parts[v]);
            loc[loc_off[v] + e] = h;
        }
    }
};
__global__ void __launch_bounds__(KTcReduce::BS) k_tc_reduce(const __grid_constant__ KTcReduce k) {
    k.run(blockIdx.x, gridDim.x);
}

// Split of the grid charges into 16-bit parts, one warp per cell of the padded
// layout (cells [c0, c1), all levels in one stretch).
// F16: x s = hi + lo with hi = half(x s), lo = half(x s - hi), both rounded to
// nearest, s the power of two that takes the cell's largest |x| into [2^14,
// 2^15): the remainder is at most 2^-11 of x and keeps 11 bits, so that a value is
// off by at most 2^-23 of itself, or 2^-39 of the cell's largest (the type's
// subnormal floor).  The accumulated products are scaled back by the cell's
// factor 1/(s TC_KSCALE) where they are added up, all exact powers of two.
// Three parts (P3): x s = x0 + x1 + x2, x0 the multiple of 2^7 next to x s (an
// integer of at most 8 bits, times 2^7), x1 and x2 the remainder's two halves: all of
// an FP32 value's bits where it is at least 2^6, 2^-9 of the cell's largest; a smaller
// one is off by at most 2^-23 of itself, 2^-32 of the largest.  The leading
// parts' products are integers below 2^16 of one unit (2^7 times the kernel row's),
// so that their sum over up to 224 values stays below 2^24 units: whatever the order
// and the rounding of the tensor cores' additions, it is exact.
// BF16: hi = bf16(x), lo = bf16(x - hi), unscaled (the type has FP32's range).
// qsc: per cell (total charge, factor).  Infinite or NaN grid charges stay so.
template <int MODE, bool P3>
struct KSplit {
    static constexpr int BS = 256, MINB = 0;
    const float *__restrict__ phi;   // the cells' values from cell 0 of the layout
    const float *__restrict__ qlev;
    float2 *__restrict__ qsc;
    char *__restrict__ op;
    long long c0, c1;
    int p3;
    int fc;     // whole stages (64 values) of a row
    int tail;   // values of the last, shorter stage (0 or 32)
    __device__ __forceinline__ void run(const int bid_, const int nblk_) const {
        typedef typename std::conditional<MODE == TC_BF16X3, __nv_bfloat162, __half2>::type T2;
        const int lane = threadIdx.x & 31;
        const int row_bytes = P3 ? 6 * ((p3 + 31) / 32 * 32) : 256 * fc + (tail ? 128 : 0);
        for (int64_t c = c0 + ((bid_ * (int64_t)BS + threadIdx.x) >> 5); c < c1; c += ((int64_t)nblk_ * BS) >> 5) {
            const float *src = phi + c * p3;
            float2 v[4];
            uint32_t m = 0;
#pragma unroll
            for (int k = 0; k < 4; k++) {
                const int b = 2 * lane + 64 * k;
                v[k].x = b < p3 ? src[b] : 0.0f;
                v[k].y = b + 1 < p3 ? src[b + 1] : 0.0f;
                m = max(m, max(__float_as_uint(v[k].x) & 0x7FFFFFFFu, __float_as_uint(v[k].y) & 0x7FFFFFFFu));
            }
            float s = 1.0f, inv = 1.0f;
            if (MODE != TC_BF16X3) {
                // biased exponent e of the largest: s = 2^(14 - (e - 127)), capped at 2^127
                const int e = (int)(__reduce_max_sync(0xffffffffu, m) >> 23);
                const int f = min(268 - e, 254);
                s = __uint_as_float((uint32_t)f << 23);
                // 2^(127 - f) / TC_KSCALE, subnormal for the smallest cells: two exact factors
                inv = __uint_as_float((uint32_t)(254 - min(f, 253)) << 23) * (f > 253 ? 0.5f / TC_KSCALE : 1.0f / TC_KSCALE);
            }
            if (lane == 0) qsc[c] = make_float2(qlev[c], inv);
            if constexpr (P3) {
                // values 2 lane + 64 k: stage 2 k + lane / 16 of 32 values, 192 bytes each
                char *dst = op + c * row_bytes + 192 * (lane >> 4) + 4 * (lane & 15);
#pragma unroll
                for (int k = 0; k < 4; k++) {
                    if (2 * lane + 64 * k >= (p3 + 31) / 32 * 32) break;
                    const float x = v[k].x * s, y = v[k].y * s;
                    const float x0 = rintf(x * 0x1p-7f) * 0x1p7f, y0 = rintf(y * 0x1p-7f) * 0x1p7f;
                    const __half2 a = __floats2half2_rn(x0, y0), b = __floats2half2_rn(x - x0, y - y0);
                    const float2 f = __half22float2(b);
                    char *to = dst + 384 * k;
                    *reinterpret_cast<__half2 *>(to) = a;
                    *reinterpret_cast<__half2 *>(to + 64) = b;
                    *reinterpret_cast<__half2 *>(to + 128) = __floats2half2_rn((x - x0) - f.x, (y - y0) - f.y);
                }
                continue;
            }
            char *dst = op + c * row_bytes + 4 * lane;
#pragma unroll
            for (int k = 0; k < 4; k++) {
                const bool full = k < fc;
                if (!full && !(k == fc && tail && lane < 16)) break;
                T2 a, r;
                const float x = v[k].x * s, y = v[k].y * s;
                if constexpr (MODE == TC_BF16X3) {
                    a = __floats2bfloat162_rn(x, y);
                    const float2 f = __bfloat1622float2(a);
                    r = __floats2bfloat162_rn(x - f.x, y - f.y);
                } else {
                    a = __floats2half2_rn(x, y);
                    const float2 f = __half22float2(a);
                    r = __floats2half2_rn(x - f.x, y - f.y);
                }
                *reinterpret_cast<T2 *>(dst + 256 * k) = a;
                *reinterpret_cast<T2 *>(dst + 256 * k + (full ? 128 : 64)) = r;
            }
        }
    }
};
template <int MODE, bool P3>
__global__ void __launch_bounds__(KSplit<MODE, P3>::BS) k_split(const __grid_constant__ KSplit<MODE, P3> k) {
    k.run(blockIdx.x, gridDim.x);
}

// Kernel tables of a plan, K_o[a,b] of eq. (bilinear) at unit cells with its row
// mean split off, computed in FP64: one warp per (offset, a).  KtT: Kt_o^T
// [o][b][a] and Kbar [o][a] in the plan's type (SIMT contraction); row: the
// row's chunks for the tensor cores (hi, lo as the operand copy's, scaled by
// TC_KSCALE or in bfloat16; three parts: the leading one in at most 8 bits of a unit
// of the row's own), kbar_tc [o][p3s].  Offsets of adjacent cells stay
// zero (the tables are cleared first).
template <typename real>
struct KTables {
    double tau[FMM_MAXP];
    int p, power, ncomp, bf16, three, p3s, fc, tail;
    real *KtT, *Kbar;
    char *row;       // nullptr: no tensor-core tables
    float *kbar_tc;
};
__device__ __forceinline__ double table_value(int comp, int power, double dx, double dy, double dz) {
    // comp 0: 1/r^power; comps 1..3: the components of its force kernel
    const double r2 = dx * dx + dy * dy + dz * dz, r = sqrt(r2);
    const double d = comp == 1 ? dx : comp == 2 ? dy : dz;
    if (power == 2) return comp == 0 ? 1.0 / r2 : 2.0 * d / (r2 * r2);
    return comp == 0 ? 1.0 / r : d / (r2 * r);
}
template <typename real>
__global__ void __launch_bounds__(256) k_tables(const __grid_constant__ KTables<real> t) {
    const int p = t.p, p3 = p * p * p, lane = threadIdx.x & 31;
    const int a = blockIdx.y * 8 + (threadIdx.x >> 5), oc = blockIdx.x, c = oc / 343, oi = oc % 343;
    const int ox = oi % 7 - 3, oy = (oi / 7) % 7 - 3, oz = oi / 49 - 3;
    if (a >= p3 || (abs(ox) <= 1 && abs(oy) <= 1 && abs(oz) <= 1)) return;
    const double ax = t.tau[a % p] - ox, ay = t.tau[(a / p) % p] - oy, az = t.tau[a / (p * p)] - oz;
    auto value = [&](int b) {
        return table_value(c, t.power, ax - t.tau[b % p], ay - t.tau[(b / p) % p], az - t.tau[b / (p * p)]);
    };
    double mean = 0.0;
    for (int b = lane; b < p3; b += 32) mean += value(b);
    for (int o = 16; o >= 1; o >>= 1) mean += __shfl_xor_sync(0xffffffffu, mean, o);
    mean /= p3;
    if (lane == 0) t.Kbar[(int64_t)oc * p3 + a] = (real)mean;
    for (int b = lane; b < p3; b += 32) t.KtT[((int64_t)oc * p3 + b) * p3 + a] = (real)(value(b) - mean);
    if (!t.row) return;
    if (lane == 0) t.kbar_tc[oc * t.p3s + a] = (float)mean;
    if (t.three) {
        double m = 0.0;
        for (int b = lane; b < p3; b += 32) m = fmax(m, fabs(value(b) - mean));
        for (int o = 16; o >= 1; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
        int e;
        frexp(m * (double)TC_KSCALE, &e);
        const double unit = ldexp(1.0, e - 8);  // the row's largest: 128 to 256 units
        char *row = t.row + ((int64_t)oc * t.p3s + a) * 6 * t.p3s;
        for (int b = lane; b < p3; b += 32) {
            const double u = (value(b) - mean) * (double)TC_KSCALE, u0 = rint(u / unit) * unit;
            const __half x = __float2half_rn((float)(u - u0));
            char *to = row + 192 * (b / 32) + 2 * (b % 32);
            *reinterpret_cast<__half *>(to) = __float2half_rn((float)u0);
            *reinterpret_cast<__half *>(to + 64) = x;
            *reinterpret_cast<__half *>(to + 128) = __float2half_rn((float)(u - u0 - (double)__half2float(x)));
        }
        return;
    }
    char *row = t.row + ((int64_t)oc * t.p3s + a) * (256 * t.fc + (t.tail ? 128 : 0));
    for (int b = lane; b < p3; b += 32) {
        const double v = value(b) - mean;
        const bool full = b < 64 * t.fc;
        char *h = row + (b / 64) * 256 + (b % 64) * 2, *w = h + (full ? 128 : 64);
        if (t.bf16) {
            const __nv_bfloat16 x = __float2bfloat16_rn((float)v);
            *reinterpret_cast<__nv_bfloat16 *>(h) = x;
            *reinterpret_cast<__nv_bfloat16 *>(w) = __float2bfloat16_rn((float)(v - (double)__bfloat162float(x)));
        } else {
            const double u = v * (double)TC_KSCALE;
            const __half x = __float2half_rn((float)u);
            *reinterpret_cast<__half *>(h) = x;
            *reinterpret_cast<__half *>(w) = __float2half_rn((float)(u - (double)__half2float(x)));
        }
    }
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
static PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    if (!fn) {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault,
                                             &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = (PFN_cuTensorMapEncodeTiled_v12000)p;
    }
    return fn;
}

int tc_padded(int p3) { return (p3 + 31) / 32 * 32; }
// a cell vector's (and kernel row's) chunks: stages of 64 values (two chunks),
// a rest of at most 32 values in one chunk
static int tc_full(int p3) { return p3 % 64 == 0 || p3 % 64 > 32 ? (p3 + 63) / 64 : p3 / 64; }
static int tc_tail(int p3) { return p3 > 64 * tc_full(p3) ? 32 : 0; }
static bool tc_three(int p3, int mode) { return mode == FMM_TC_F32 && p3 > 64; }
int tc_row_bytes(int p3, int mode) {
    return tc_three(p3, mode) ? 6 * tc_padded(p3) : 256 * tc_full(p3) + (tc_tail(p3) ? 128 : 0);
}
int tc_chunk_bytes(int p3, int mode) { return tc_three(p3, mode) ? 64 : 128; }

static CUtensorMapDataType op_type(int mode) {
    return mode == FMM_TC_BF16X3 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT16;
}
static int encode(CUtensorMap *m, int p3, int mode, int rank, const void *base, const cuuint64_t *dims,
                  const cuuint64_t *strides, const cuuint32_t *box) {
    auto enc = encode_fn();
    if (!enc) return FMM_ERR_CUDA;
    const cuuint32_t es[5] = {1, 1, 1, 1, 1};
    CUresult r = enc(m, op_type(mode), rank, (void *)base, dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
                     tc_three(p3, mode) ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_128B,
                     CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                     CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? FMM_OK : FMM_ERR_CUDA;
}

// Box map of level l of the operand copy: dims (row values, P x, P y, P z, 8
// parity), box (one chunk, 8, 4, 4, 1).  Every box the kernel loads lies inside.
static int encode_phi_map(CUtensorMap *m, const void *base, int l, int p3, int mode) {
    const cuuint64_t P = ((cuuint64_t)1 << (l - 1)) + 2, rb = (cuuint64_t)tc_row_bytes(p3, mode);
    const cuuint64_t dims[5] = {rb / 2, P, P, P, 8}, strides[4] = {rb, rb * P, rb * P * P, rb * P * P * P};
    const cuuint32_t box[5] = {(cuuint32_t)tc_chunk_bytes(p3, mode) / 2, 8, 4, 4, 1};
    return encode(m, p3, mode, 5, base, dims, strides, box);
}

// Kernel-table map: dims (row values, p3s a, 343 offsets), box (one chunk, p3s, 1).
int tc_encode_kernel_map(void *map, const void *base, int p3, int mode) {
    const cuuint64_t rb = (cuuint64_t)tc_row_bytes(p3, mode), p3s = (cuuint64_t)tc_padded(p3);
    const cuuint64_t dims[3] = {rb / 2, p3s, 343}, strides[2] = {rb, rb * p3s};
    const cuuint32_t box[3] = {(cuuint32_t)tc_chunk_bytes(p3, mode) / 2, (cuuint32_t)p3s, 1};
    return encode((CUtensorMap *)map, p3, mode, 3, base, dims, strides, box);
}

size_t tc_map_bytes() { return sizeof(CUtensorMap); }

template <typename real>
int build_tables(int p, double grid_scale, int power, int ncomp, int mode, real *KtT, real *Kbar, void *rows,
                 float *kbar_tc) {
    KTables<real> t;
    memset(&t, 0, sizeof(t));
    const int p3 = p * p * p;
    // §2.1.2: the p-division points; §4.1's reduced arrangement
    for (int i = 0; i < p; i++) t.tau[i] = 0.5 + grid_scale * ((double)i / (double)(p - 1) - 0.5);
    t.p = p;
    t.power = power;
    t.ncomp = ncomp;
    t.bf16 = mode == FMM_TC_BF16X3;
    t.three = tc_three(p3, mode);
    t.p3s = tc_padded(p3);
    t.fc = tc_full(p3);
    t.tail = tc_tail(p3);
    t.KtT = KtT;
    t.Kbar = Kbar;
    t.row = (char *)rows;
    t.kbar_tc = kbar_tc;
    const size_t no = (size_t)343 * ncomp;
    if (cudaMemset(KtT, 0, no * p3 * p3 * sizeof(real)) != cudaSuccess ||
        cudaMemset(Kbar, 0, no * p3 * sizeof(real)) != cudaSuccess)
        return FMM_ERR_CUDA;
    if (rows && (cudaMemset(rows, 0, no * t.p3s * tc_row_bytes(p3, mode)) != cudaSuccess ||
                 cudaMemset(kbar_tc, 0, no * t.p3s * sizeof(float)) != cudaSuccess))
        return FMM_ERR_CUDA;
    k_tables<real><<<dim3((unsigned)no, (p3 + 7) / 8), 256>>>(t);
    return cudaGetLastError() == cudaSuccess ? FMM_OK : FMM_ERR_CUDA;
}
template int build_tables<float>(int, double, int, int, int, float *, float *, void *, float *);
template int build_tables<double>(int, double, int, int, int, double *, double *, void *, float *);

template <int N, int MODE>
static int launch_tcg_kernel(const TcgParams &prm, int blocks, int comp, cudaStream_t st, Tracer &tr) {
    typedef TcgShape<N, MODE> Gh;
    launch_k(tr, FMM_TAG(S_M2L_TC, comp), k_m2l_tcg<N, MODE>, KM2LTcg<N, MODE>{prm}, blocks, Gh::THREADS, Gh::SMEM,
             st);
    return FMM_OK;
}

// the record of a cross-system launch (batched evaluations)
template <int N, int MODE>
static int record_tcx(const TcgParams &prm, int blocks, int comp, Tracer &tr) {
    typedef KM2LTcg<N, MODE, true> K;
    kb_set_smem<K>(K::SMEM);
    launch_k(tr, FMM_TAG(S_M2L_TCX, comp), k_m2l_tcx<N, MODE>, K{prm}, blocks, K::BS, K::SMEM, nullptr);
    return FMM_OK;
}
template <int MODE>
static int record_tcx_mode(int p3s, const TcgParams &prm, int blocks, int comp, Tracer &tr) {
    switch (p3s) {
    case 32: return record_tcx<32, MODE>(prm, blocks, comp, tr);
    case 64: return record_tcx<64, MODE>(prm, blocks, comp, tr);
    case 128: return record_tcx<128, MODE>(prm, blocks, comp, tr);
    case 224: return record_tcx<224, MODE>(prm, blocks, comp, tr);
    default: return FMM_ERR_UNSUPPORTED;
    }
}

template <int N, int MODE>
static int set_attributes() {
    typedef TcgShape<N, MODE> Gh;
    if (cudaFuncSetAttribute(k_m2l_tcg<N, MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize, Gh::SMEM) != cudaSuccess)
        return FMM_ERR_CUDA;
    kb_set_smem<KM2LTcg<N, MODE>>(Gh::SMEM);
    return cudaGetLastError() == cudaSuccess ? FMM_OK : FMM_ERR_CUDA;
}
template <int MODE>
static int set_attributes_mode(int p3s) {
    switch (p3s) {
    case 32: return set_attributes<32, MODE>();
    case 64: return set_attributes<64, MODE>();
    case 128: return set_attributes<128, MODE>();
    case 224: return set_attributes<224, MODE>();
    default: return FMM_ERR_UNSUPPORTED;
    }
}
int tc_set_attributes(int p3, int mode) {
    const int p3s = tc_padded(p3);
    return mode == FMM_TC_BF16X3  ? set_attributes_mode<TC_BF16X3>(p3s)
           : mode == FMM_TC_F16X1 ? set_attributes_mode<TC_F16X1>(p3s)
           : mode == FMM_TC_F32 ? set_attributes_mode<TC_F32>(p3s)
                                  : set_attributes_mode<TC_F16X3>(p3s);
}

template <int MODE>
static int launch_tcg_mode(int p3s, const TcgParams &prm, int blocks, int comp, cudaStream_t st, Tracer &tr) {
    switch (p3s) {
    case 32: return launch_tcg_kernel<32, MODE>(prm, blocks, comp, st, tr);
    case 64: return launch_tcg_kernel<64, MODE>(prm, blocks, comp, st, tr);
    case 128: return launch_tcg_kernel<128, MODE>(prm, blocks, comp, st, tr);
    case 224: return launch_tcg_kernel<224, MODE>(prm, blocks, comp, st, tr);
    default: return FMM_ERR_UNSUPPORTED;
    }
}

template <int MODE, bool P3 = false>
static void launch_split(const Ptrs<float> &P, int64_t c0, int64_t c1, int p3, int blocks, cudaStream_t st, Tracer &tr) {
    typedef KSplit<MODE, P3> K;
    launch_k(tr, FMM_TAG(S_SPLIT_TC, 0), k_split<MODE, P3>,
             K{P.phi, P.qlev, P.qsc, P.op, c0, c1, p3, tc_full(p3), tc_tail(p3)}, blocks, K::BS, 0, st);
}

int launch_m2l_tc(const Geom &g, const Ptrs<float> &P, const WsLayout &W, const void *k_map, const float *kbar,
                  int lmin, int mode, int inject, float *loc, int spow, bool split, int comp, cudaStream_t st,
                  Tracer &tr) {
    const int depth = g.depth, p3 = g.p3, p3s = tc_padded(p3), rb = tc_row_bytes(p3, mode);
    tr.begin(FMM_STAGE_M2L, st);
    if (split) {
        // grid-stride over the cells, a warp each; small systems take a small
        // grid, so that other work keeps the SMs
        const int64_t c0 = W.q_level[lmin], c1 = W.q_level[depth + 1];
        const int nbs = (int)std::min<int64_t>(152 * 8, std::max<int64_t>(1, (c1 - c0 + 7) / 8));
        if (mode == FMM_TC_BF16X3) launch_split<TC_BF16X3>(P, c0, c1, p3, nbs, st, tr);
        else if (tc_three(p3, mode)) launch_split<TC_F32, true>(P, c0, c1, p3, nbs, st, tr);
        else launch_split<TC_F16X3>(P, c0, c1, p3, nbs, st, tr);
        tr.count();
    }
    // a batch whose small levels run as cross-system tiles: this system's own
    // launch takes the levels from tr.tc_lbig up
    if (tr.rec && tr.tc_lbig > lmin) {
        lmin = tr.tc_lbig;
        if (depth < lmin) {
            tr.end();
            return FMM_OK;
        }
    }
    // the occupied cells of every (level, parity) segment, once per evaluation
    OccParams op;
    memset(&op, 0, sizeof(op));
    op.leaf_start = P.leaf_start;
    op.occ = P.occ;
    op.depth = depth;
    op.lmin = lmin;
    op.nseg = occ_nseg(depth, lmin);
    op.N = p3s;
    int nb = 0, blocks = 0;
    for (int s = 0; s < op.nseg; s++) {
        op.bfirst[s] = nb;
        nb += (int)((occ_seg_cells(lmin, s) + OCC_BLOCK - 1) / OCC_BLOCK);
        // blocks if every cell holds charges
        blocks += (int)((occ_seg_cells(lmin, s) + TC_M - 1) / TC_M) * tc_parts(lmin + s / 8, depth);
    }
    op.bfirst[op.nseg] = nb;
    op.nblk = nb;
    if (split) {
        launch_k(tr, FMM_TAG(S_OCC_COUNT, 0), k_occ_count, KOccCount{op}, nb, OCC_BLOCK / 4, 0, st);
        launch_k(tr, FMM_TAG(S_OCC_OFFSETS, 0), k_occ_offsets, KOccOffsets{op}, (op.nseg + 7) / 8, 256, 0, st);
        launch_k(tr, FMM_TAG(S_OCC_SCATTER, 0), k_occ_scatter, KOccScatter{op}, nb, OCC_BLOCK / 4, 0, st);
        tr.count(3);
    }
    TcgParams prm;
    memset(&prm, 0, sizeof(prm));
    memcpy(&prm.k, k_map, sizeof(CUtensorMap));
    prm.lmin = lmin;
    prm.depth = depth;
    prm.p3 = p3;
    prm.spow = spow;
    prm.nseg = op.nseg;
    prm.occ = P.occ;
    prm.op = P.op;
    int rc = FMM_OK;
    KTcReduce red;
    memset(&red, 0, sizeof(red));
    for (int l = lmin; l <= depth && !rc; l++) {
        prm.loc_off[l] = W.loc_level[l];
        prm.q_off[l] = W.q_level[l];
        if (l >= 4) rc = encode_phi_map(&prm.phi[l], P.op + W.q_level[l] * rb, l, p3, mode);
        if (tc_parts(l, depth) > 1) {
            const int v = red.nlev++;
            tc_part_place(l, p3, &prm.part_off[l], &prm.part_stride[l]);
            red.parts[v] = tc_parts(l, depth);
            red.first[v + 1] = red.first[v] + ((long long)p3 << (3 * l));
            red.part_off[v] = prm.part_off[l];
            red.part_stride[v] = prm.part_stride[l];
            red.loc_off[v] = W.loc_level[l];
        }
    }
    if (rc) return rc;
    prm.loc = loc;
    prm.part = P.tc_part;
    prm.qsc = P.qsc;
    prm.kbar = kbar;
    prm.status = &P.hdr->status;
    prm.inject_stall = inject == FMM_INJECT_TC_STALL;
    rc = mode == FMM_TC_BF16X3  ? launch_tcg_mode<TC_BF16X3>(p3s, prm, blocks, comp, st, tr)
         : mode == FMM_TC_F16X1 ? launch_tcg_mode<TC_F16X1>(p3s, prm, blocks, comp, st, tr)
         : mode == FMM_TC_F32 ? launch_tcg_mode<TC_F32>(p3s, prm, blocks, comp, st, tr)
                                : launch_tcg_mode<TC_F16X3>(p3s, prm, blocks, comp, st, tr);
    tr.count();
    if (!rc && red.nlev > 0) {
        red.part = P.tc_part;
        red.loc = loc;
        const int nbr = (int)std::min<int64_t>(152 * 4, (red.first[red.nlev] + KTcReduce::BS - 1) / KTcReduce::BS);
        launch_k(tr, FMM_TAG(S_TC_REDUCE, comp), k_tc_reduce, red, nbr, KTcReduce::BS, 0, st);
        tr.count();
    }
    tr.end();
    return rc;
}

int tc_cross_records(const std::vector<TcXSys> &sys, const std::vector<int> &depth, int ncomp, int lmin,
                     int lmax, int p3, int mode, int spow0, const void *const *k_maps, const float *const *kbars,
                     const WsLayout &W, const char *ws, size_t ws_bytes, int *status, void **dx, size_t *dx_bytes,
                     std::vector<LaunchRec> &out) {
    const int ns = (int)depth.size();
    const int p3s = tc_padded(p3);
    const int nseg = 8 * (lmax - lmin + 1);
    // coordinates and systems fit the list's entries, chunks of the workspace a gather's row index
    if (lmax >= 5 || ns >= (1 << 19) || ws_bytes / tc_chunk_bytes(p3, mode) > INT32_MAX) return FMM_ERR_UNSUPPORTED;
    // the lists: every cell of every system with that level, system-major
    std::vector<int> cnt(nseg, 0), tiles(nseg + 1, 0), first(nseg, 0), list;
    for (int sg = 0; sg < nseg; sg++) {
        const int l = lmin + sg / 8, H = 1 << (l - 1);
        first[sg] = (int)list.size();
        for (int i = 0; i < ns; i++) {
            if (depth[i] < l) continue;
            for (int Z = 0; Z < H; Z++)
                for (int Y = 0; Y < H; Y++)
                    for (int X = 0; X < H; X++) list.push_back(i << 12 | Z << 8 | Y << 4 | X);
        }
        cnt[sg] = (int)list.size() - first[sg];
        tiles[sg + 1] = tiles[sg] + (cnt[sg] + TC_M - 1) / TC_M;
    }
    // device buffer: the segment table and list, then the systems' table per component
    std::vector<int> seg;
    seg.insert(seg.end(), cnt.begin(), cnt.end());
    seg.insert(seg.end(), tiles.begin(), tiles.end());
    seg.insert(seg.end(), first.begin(), first.end());
    seg.insert(seg.end(), list.begin(), list.end());
    const size_t seg_bytes = (seg.size() * sizeof(int) + 255) / 256 * 256;
    const size_t need = seg_bytes + sizeof(TcXSys) * sys.size();
    if (need > *dx_bytes) {
        if (*dx) cudaFree(*dx);
        *dx = nullptr;
        *dx_bytes = 0;
        if (cudaMalloc(dx, need) != cudaSuccess) return FMM_ERR_OOM;
        *dx_bytes = need;
    }
    char *d = reinterpret_cast<char *>(*dx);
    if (cudaMemcpy(d, seg.data(), seg.size() * sizeof(int), cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemcpy(d + seg_bytes, sys.data(), sizeof(TcXSys) * sys.size(), cudaMemcpyHostToDevice) != cudaSuccess)
        return FMM_ERR_CUDA;
    out.clear();
    for (int c = 0; c < ncomp; c++) {
        TcgParams prm;
        memset(&prm, 0, sizeof(prm));
        memcpy(&prm.k, k_maps[c], sizeof(CUtensorMap));
        prm.op = ws;
        prm.lmin = lmin;
        prm.depth = lmax;
        prm.p3 = p3;
        prm.spow = c == 0 ? spow0 : spow0 + 1;
        prm.nseg = nseg;
        for (int l = lmin; l <= lmax; l++) {
            prm.loc_off[l] = W.loc_level[l];
            prm.q_off[l] = W.q_level[l];
        }
        prm.kbar = kbars[c];
        prm.status = status;
        prm.xsys = reinterpret_cast<const TcXSys *>(d + seg_bytes) + (size_t)c * ns;
        prm.xseg = reinterpret_cast<const int *>(d);
        Tracer t;
        std::vector<LaunchRec> one;
        t.rec = &one;
        int rc = mode == FMM_TC_BF16X3  ? record_tcx_mode<TC_BF16X3>(p3s, prm, tiles[nseg], c, t)
             : mode == FMM_TC_F16X1 ? record_tcx_mode<TC_F16X1>(p3s, prm, tiles[nseg], c, t)
             : mode == FMM_TC_F32 ? record_tcx_mode<TC_F32>(p3s, prm, tiles[nseg], c, t)
                                    : record_tcx_mode<TC_F16X3>(p3s, prm, tiles[nseg], c, t);
        if (rc) return rc;
        out.push_back(std::move(one[0]));
    }
    return FMM_OK;
}

}  // namespace fmm
