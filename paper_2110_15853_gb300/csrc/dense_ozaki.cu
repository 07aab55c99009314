// FP64-accurate dense products on the BF16 tensor cores (Ozaki-scheme splitting),
// for the large products of the ChFSI closure (Algorithm 1 steps 2, 3 and 5,
// Sec. 3.4): the Gram matrix Y^T Y of the Cholesky-QR, X_F = Y R^-1, the projection
// X_F^T (H X_F) and the rotation X_F Q.  GB300's FP64 pipe runs about 1.2 TFLOP/s;
// its BF16 tensor cores about 1.9 PFLOP/s.
//
// Splitting.  The product is C = A_hat B_hat^T with both operands K-major: for
// C = A^T B (Gram form) A_hat = A^T, B_hat = B^T; for C = A B, A_hat = A, B_hat =
// B^T.  Each row r of an operand gets a power-of-two scale 2^{e_r} with
// |A_hat[r][k]| 2^{-e_r} < 1/2 for all k, and the scaled value a is rounded to a
// 56-bit fixed-point number and written as seven balanced base-256 digits
//     a = sum_{t=1..7} d_t 2^{-8t},   d_t integer, |d_t| <= 128,
// (integer arithmetic on the FP64 bit pattern; no FP64 instructions).  Slice t stores the
// integers d_t in BF16, which is exact (8 significant bits).  Then
//     C_ij = 2^{e_i + f_j} sum_{t + u <= 8} 2^{-8(t+u)} sum_k a_t[i][k] b_u[j][k]
// keeps every digit product of weight 2^{-64} and above (28 slice pairs; the
// dropped pairs and the 56-bit rounding are below about 2^{-55} of the row scales
// per term, i.e. about 2^{-48} of a typical term).
//
// Exact accumulation.  A product of two digits is an integer of at most 2^14.  Every level
// l = t + u = 2 .. 8 has its own FP32 accumulator E_l in TMEM, and each is drained before
// its sums can pass 2^24 (see Groups), so the tensor-core accumulation -- which truncates
// rather than rounds -- never rounds at all: the sums are exact integers.  The drains add
// them to one 96-bit integer per output element in units of 2^{-64}.  A work item spans at
// most 8192 K (longer sums are split over items and the FP64 partial tiles added), which
// bounds that integer by 2^76.  It is rounded to a double once at the end, so the only
// errors are the 56-bit rounding of the inputs and the dropped pairs (weights 2^{-72} and
// below).
//
// Five-slice steps.  A filter step may also use only the first five digits of each
// operand (a 40-bit fixed-point value, truncation below 2^{-41} of the row scale) and
// the 15 pairs of weight 2^{-48} and above (levels 2 .. 6): about 2^{-40} of the row
// scales per term, some 2^{16} times finer than FP32, for 15 slice products instead
// of 28.  The digits are the same as above, so the same slices serve both step kinds.
//
// Layout.  An operand is stored as [row tile][K chunk of 8][7 planes][rows of the tile][8]:
// 16 bytes a row, plane and chunk, the core-matrix order that an unswizzled K-major
// shared-memory operand has.  So a chunk of a tile is one contiguous copy of 14 KB (128
// rows) or 7 KB (64 rows; its first five planes for a five-slice step), and any chunks can
// be put side by side: the BSR step copies only the chunks of Y_cur that meet a nonzero
// column of H.  (Tensor-map boxes of 128 rows x 64 bytes, 14 a stage, took the producer 87
// cycles each.)
//
// Kernel.  Persistent, warp-specialised, one CTA per SM, 128 x 64 output tiles; NS = 7
// slices per operand (or 5 for the 40-bit filter steps):
//   warp 0    : producer, K = 16 of both operands per ring slot (42 KB, five slots; or 30
//               KB, seven);
//   warp 1    : MMA issuer, owns 512 TMEM columns; stages of K = 32 (two slots);
//   warps 2-3 : BSR mode, the recurrence on the finished products;
//   warps 4-11: epilogue; warp w reads TMEM lanes 32 (w % 4) .. + 31 (one output row per
//               thread), columns 32 ((w - 4) / 4) .. + 31, and keeps their sums in registers.
// Every mbarrier wait is bounded; on a timeout the CTA flags DEV_TIMEOUT, stops, waits
// (bounded) for its copies and MMAs in flight, frees TMEM and exits.
//
// What bounds it: the tensor pipe, at 908 cycles per K = 16 of the 28 slice products (their
// work is 896) when nothing else runs on the SM; over a launch 1240 in a Gram product and
// 1350 in the filter step (pipe 74% and 66% active), since the warps share the issue slots
// with the drains' conversions (6 of 60 ms), a drained group's MMAs come in narrower
// pieces, and an item ends with three drains in turn.  The 40-bit step takes 915 for 480.  20 FP64-accurate steps at 40^3, w = 3, 1024
// states: 98.0 -> 60.0 ms (0.83 of the chunks, and 1.35 x the rate); 20 40-bit and 4
// FP64-accurate steps at 48^3, w = 4, 1500 states: 266 -> 161 ms.
#include <algorithm>
#include <type_traits>

#include "common.cuh"
#include "kernels.cuh"
#include "tcgen05.cuh"

namespace chfsi {

namespace {

using namespace tc;

constexpr int kSlices = 7;                            // digit planes stored per operand
constexpr int kTileM = 128;                           // output rows per tile (TMEM lanes)
constexpr int kTileN = 64;                            // output columns per tile
constexpr int kChunk = 8;                             // K columns per chunk: 8 BF16 = 16 bytes per row
constexpr int kKB = 32;                               // K per stage: two ring slots of 16
constexpr int kStageChunks = kKB / kChunk;
constexpr int kSlotChunks = 2;                        // chunks per ring slot (K = 16, one MMA step)
constexpr int kStageSlots = kStageChunks / kSlotChunks;
constexpr int kMaxItemKB = 8192 / kKB;                // stages per work item (8192 K)
constexpr int kBlockChunks = 64 / kChunk;             // chunks per 64-wide BSR block
constexpr int kPlaneA = kTileM * 16;                  // bytes of one chunk and digit plane of a 128-row tile
constexpr int kPlaneB = kTileN * 16;                  // the same for a 64-row tile
constexpr int kEpiWarps = 8;                          // two warpgroups
constexpr int kColsPerThread = kTileN / (kEpiWarps / 4);   // 32
constexpr int kThreads = 32 * (4 + kEpiWarps);        // a warpgroup for the producer and the issuer
// Registers a thread: launched with 168 (three warps on each scheduler's 16,384), of which
// the first warpgroup gives 80 away to the other two: 88 + 2 x 208 = 3 x 168.
constexpr int kRegsIssue = 88, kRegsEpilogue = 208;
constexpr uint32_t kTmemCols = 512;
constexpr int kMaxSlots = 7;
constexpr int kEvents = 4;                            // barrier pairs of the drains
static_assert(kColsPerThread == 32, "TMEM loads of 8 columns, batches of 8 and 16");

// Shape of a product with NS digit slices per operand (7: FP64-accurate; 5: the
// 40-bit steps): a ring slot holds the NS slices of K = 16 of both operands; level l = 2
// .. NS + 1 has an accumulator E_l (index a = l - 2, 64 TMEM columns).
template <int NS>
struct OzShape {
    static constexpr int kChunkA = NS * kPlaneA, kChunkB = NS * kPlaneB;   // chunk strides in a slot
    static constexpr int kSlotBytes = kSlotChunks * (kChunkA + kChunkB);
    static constexpr int kSlots = (216 * 1024) / kSlotBytes;
    static constexpr int kSmemBytes = kSlots * kSlotBytes + 128;
    static_assert(NS == 7 || NS == 5, "seven or five slices");
    static_assert(kSlots > 2 * kStageSlots && kSlots <= kMaxSlots, "two stages and more in the ring");
    static_assert(kSmemBytes + 1024 <= 227 * 1024, "shared memory per CTA");
};

// Drains.  The accumulators are drained in groups, one group after a stage, so that the
// MMAs of the others cover it: seven slices E7-E8 (index 5, 6), E5-E6 (3, 4) and E2-E4
// (0 .. 2); five slices E4-E6 (2 .. 4) and E2-E3 (0, 1), E4-E6 in two alternating sets of
// columns, so that its drain holds up nothing.  A product of two digits is at most 2^14 and
// E_l takes l - 1 pairs, so l - 1 <= 2^10 / K keeps |E_l| <= 2^24 between drains:
//   seven slices: E7-E8 after stages 3, 7, 11 .. (K = 128), E5-E6 after 4, 10, 16 .. (160,
//   192), E2-E4 after 9, 17 .. (320, 256); at the end of an item all three in turn.
//   five slices: E4-E6 after 3, 7, 11 .. (128), E2-E3 after 9, 25 .. (320, 512); at the end
//   E2-E3, then E4-E6.
// (Drained in two groups, E2-E5 and E6-E8, the tensor pipe waited 1200 of 3800 cycles a
// stage for them and for the outputs.)
template <int NS>
struct Groups;
template <>
struct Groups<7> {
    static constexpr int kCount = 3;
    __host__ __device__ static constexpr int lo(int g) { return g == 0 ? 5 : (g == 1 ? 3 : 0); }
    __host__ __device__ static constexpr int hi(int g) { return g == 0 ? 7 : (g == 1 ? 5 : 3); }
    __host__ __device__ static constexpr int column(int g, int) { return lo(g) * kTileN; }
    // the group drained after stage kb (not the item's last), or -1
    __device__ static int event(int kb) { return kb % 4 == 3 ? 0 : (kb % 6 == 4 ? 1 : (kb % 8 == 1 && kb > 1 ? 2 : -1)); }
};
template <>
struct Groups<5> {
    static constexpr int kCount = 2;
    __host__ __device__ static constexpr int lo(int g) { return g == 0 ? 0 : 2; }
    __host__ __device__ static constexpr int hi(int g) { return g == 0 ? 2 : 5; }
    // E2 E3 | E4 E5 E6 | E4 E5 E6 (second set)
    __host__ __device__ static constexpr int column(int g, int set) { return g == 0 ? 0 : (2 + 3 * set) * kTileN; }
    __device__ static int event(int kb) { return kb % 4 == 3 ? 1 : (kb % 16 == 9 ? 0 : -1); }
};

// The slice pairs (t, u), 0-based, t + u <= NS - 1, go to accumulator t + u.  For one slice
// t of A consecutive slices u of B fall into consecutive accumulators, so they run as one
// MMA with the B slices stacked along N (N = 64 c <= 256).  The pairs of the accumulators
// LO .. HI - 1 take, for every t, the slices u = max(LO - t, 0) .. HI - 1 - t, in one MMA or
// (five to seven slices) two; the t = 0 MMAs cover every accumulator of the range and come
// first, so they overwrite when its sums start fresh; then the last slices of A (narrow
// MMAs) down to the first (wide ones), because the tensor pipe queues only a few MMAs and
// the wide ones last cover the waits between two ranges.  All of it is known at compile time:
// the unrolled sequence has immediate descriptor offsets.  The whole warp runs it on
// warp-uniform values and the MMAs are predicated on the leader lane (issued from a branch
// that one lane takes, 10 MMAs took 1016-1146 cycles instead of 951-1030, their work being
// 908).  `mid` runs before the MMAs of the last two slices.
template <int NS, int LO, int HI, typename Mid>
__device__ __forceinline__ void issue_range(uint32_t leader, uint64_t da0, uint64_t db0, uint32_t dcol, bool fresh,
                                            Mid&& mid) {
    static_assert(0 <= LO && LO < HI && HI <= NS, "accumulator range");
#pragma unroll
    for (int k = 0; k < HI; k++) {
        const int t = k == 0 ? 0 : HI - k;
        if (k == HI - 2) mid();
        const int u0 = LO > t ? LO - t : 0, n = HI - t - u0;
        const int first = n > 4 ? n / 2 : n;
#pragma unroll
        for (int part = 0; part < (n > 4 ? 2 : 1); part++) {
            const int u = part ? u0 + first : u0, c = part ? n - first : first;
            constexpr uint32_t kIdesc1 = idesc_bf16(kTileM, kTileN);
            // an offset stays inside the low word's 14-bit start address below 256 KB
            const uint32_t da = (uint32_t)da0 + (uint32_t)((t * kPlaneA) >> 4);
            const uint32_t db = (uint32_t)db0 + (uint32_t)((u * kPlaneB) >> 4);
            const uint32_t dt = dcol + (uint32_t)((t + u - LO) * kTileN);
            const uint32_t idesc = kIdesc1 + (uint32_t)(((kTileN * (c - 1)) >> 3) << 17);
            const uint32_t accumulate = fresh && t == 0 ? 0u : 1u;
            asm volatile(
                "{\n\t.reg .pred p, q;\n\t.reg .b64 a, b;\n\tsetp.ne.b32 p, %6, 0;\n\tsetp.ne.b32 q, %7, 0;\n\t"
                "mov.b64 a, {%1, %2};\n\tmov.b64 b, {%3, %4};\n\t"
                "@q tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %5, p;\n\t}\n"
                :: "r"(dt), "r"(da), "r"((uint32_t)(da0 >> 32)), "r"(db), "r"((uint32_t)(db0 >> 32)), "r"(idesc),
                   "r"(accumulate), "r"(leader));
        }
    }
}

// Shared-memory descriptor of a K-major operand tile without swizzle: core matrices of 8
// rows x 16 bytes (128 contiguous bytes), 8-row groups 128 bytes apart, the two 8-wide
// K chunks of a step `chunk_stride` bytes apart.
__device__ __forceinline__ uint64_t desc_chunks(uint32_t addr, int chunk_stride) {
    uint64_t d = 0;
    d |= (uint64_t)((addr & 0x3FFFF) >> 4);             // start address
    d |= (uint64_t)(chunk_stride >> 4) << 16;           // leading byte offset: next K chunk
    d |= (uint64_t)(128 >> 4) << 32;                    // stride byte offset: next 8 rows
    d |= (uint64_t)1 << 46;                             // descriptor version
    return d;
}

struct OzArgs {
    // operands: [row tile][K chunk][7][rows of the tile][8] digits (128-row tiles of A_hat,
    // 64-row tiles of B_hat; b_in_a: B_hat is A_hat, its 64-row tiles halves of A's)
    const unsigned char* A;
    const unsigned char* B;
    int b_in_a;               // then loaded through the tensor map tmA
    int64_t chunksA, chunksB; // K chunks per row tile
    int64_t M, Nc;            // output rows / columns
    int64_t ldc;
    double* C;                // output (direct mode), or
    double* part;             // split-K partial tiles [splits][Mp][Np] (split mode)
    int64_t Mp, Np;           // partial-tile extents: tilesM * 128, tilesN * 64
    const int* expA;          // biased exponent field of each row's largest |value| (0: zero row)
    const int* expB;
    int tilesM, tilesN;
    int kb_total;             // stages (32 K)
    int kb_split;             // stages per split
    int splits;
    int symmetric;            // only tiles that reach the upper triangle (j >= i)
    int b_upper;              // B_hat[j][k] = 0 for k > j: K limited to the tile's last column
    int64_t pairs;            // tiles per split and batch
    int nbatch;               // independent products (diagonal blocks of the split layout)
    int64_t m_batch;          // output rows per batch (M when nbatch = 1)
    int64_t a_batch_tiles, b_batch_tiles;   // row tiles per batch in the operands
    uint64_t wait_ns;         // limit of the waits on the other roles (drains keep kDrainNs)
    unsigned* status;
    // BSR filter-step mode (bsr != 0): A_hat = Y_cur^T (states x grid points), B_hat = the
    // non-zero 8-column chunks of H's 64-row block rows; a work item is one block row
    // (the 64 output columns, grid rows R * 64 ..) against one tile of 128 states, its K
    // the row's chunks; the epilogue leaves the products in C (ldc), where the output warps
    // apply the recurrence Y_out = alpha (H Y_cur - c Y_cur) - beta Y_prev in FP64.
    int bsr;
    int slices;               // digit slices per operand in the products: 7, or 5 (BSR mode)
    const int32_t* brow_ptr;
    const int32_t* hchunk;    // Y_cur chunk of each stored chunk of H (row R from brow_ptr[R] * 8 on)
    const int32_t* hcount;    // stored chunks of each block row (a multiple of kStageChunks),
                              // kUnfolded set where c is not in H's digits
    int64_t nblocks;
    const int* expH;          // exponent field of each grid row of H (over its block row)
    const double* Ycur;
    int64_t ldcur;
    const double* Yprev;      // nullptr: no beta term
    int64_t ldprev;
    double alpha, cshift, beta;
    int* expNext;             // largest exponent field of each state of Y_out (zeroed before)
};

constexpr int kUnfolded = 1 << 30;

struct Item {
    int batch, tm, tn, kb0, KB;
    bool unfolded;            // BSR mode: the output warps subtract c Y_cur
    int64_t qc;               // BSR mode: first stored chunk of the row
};

// Stored block range of block row R, clamped to [0, nblocks] and to 128 blocks (the host
// rejects longer rows); `bad` is set for a malformed row pointer.
__device__ __forceinline__ void bsr_row_range(const int32_t* brow_ptr, int64_t nblocks, int64_t R, int& qb, int& nq,
                                              bool& bad) {
    constexpr int kMaxBlocks = kMaxItemKB * kKB / 64;
    int b0 = brow_ptr[R], b1 = brow_ptr[R + 1];
    if (b0 < 0) { b0 = 0; bad = true; }
    if (b0 > nblocks) { b0 = (int)nblocks; bad = true; }
    if (b1 > nblocks) { b1 = (int)nblocks; bad = true; }
    if (b1 < b0) { b1 = b0; bad = true; }
    if (b1 - b0 > kMaxBlocks) { b1 = b0 + kMaxBlocks; bad = true; }
    qb = b0;
    nq = b1 - b0;
}

// First column tile of row tile tm that reaches the upper triangle (j >= i).
__device__ __host__ __forceinline__ int first_upper_tn(int tm) { return (tm * kTileM) / kTileN; }

template <bool kBsr>
__device__ __forceinline__ Item decode(const OzArgs& g, int64_t item) {
    Item it;
    if (kBsr) {
        // the state tiles of a block row are consecutive, so its H chunks are shared
        // through L2
        const int64_t R = item / g.tilesM;
        bool bad = false;
        int qb, nq;
        bsr_row_range(g.brow_ptr, g.nblocks, R, qb, nq, bad);
        it.batch = 0;
        it.tm = (int)(item - R * g.tilesM);
        it.tn = (int)R;
        it.kb0 = 0;
        const int packed = g.hcount[R], cnt = packed & ~kUnfolded;
        it.unfolded = (packed & kUnfolded) != 0;
        it.KB = (cnt < nq * kBlockChunks ? cnt : nq * kBlockChunks) / kStageChunks;
        it.qc = (int64_t)qb * kBlockChunks;
        return it;
    }
    it.qc = 0;
    const int64_t per_split = g.pairs * g.nbatch;
    const int z = (int)(item / per_split);
    it.batch = (int)((item % per_split) / g.pairs);
    int64_t p = item % g.pairs;
    if (g.symmetric) {
        int tm = 0;
        while (tm < g.tilesM - 1 && p >= g.tilesN - first_upper_tn(tm)) { p -= g.tilesN - first_upper_tn(tm); tm++; }
        it.tm = tm;
        it.tn = first_upper_tn(tm) + (int)p;
    } else {
        it.tm = (int)(p / g.tilesN);
        it.tn = (int)(p % g.tilesN);
    }
    int kend = g.kb_total;
    if (g.b_upper) {
        const int lim = (int)(((int64_t)(it.tn + 1) * kTileN + kKB - 1) / kKB);
        if (lim < kend) kend = lim;
    }
    it.kb0 = z * g.kb_split;
    const int k1 = it.kb0 + g.kb_split < kend ? it.kb0 + g.kb_split : kend;
    it.KB = k1 > it.kb0 ? k1 - it.kb0 : 0;
    return it;
}

// Eight accumulator columns of this warp's 32 TMEM lanes (one row per lane).
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t (&r)[8]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(taddr));
}

// Output sum of an element in units of 2^-64, 96 bits (|T| < 2^76): three registers where
// one 64-bit sum per accumulator group takes four (with those the epilogue spilled).
struct Sum96 {
    uint32_t w0, w1, w2;
};
// t += x 2^kShift
template <int kShift>
__device__ __forceinline__ void add96(Sum96& t, long long x) {
    if constexpr (kShift < 32) {
        const uint32_t a0 = (uint32_t)x << kShift;
        const uint32_t a1 = (uint32_t)(x >> (kShift == 0 ? 32 : 32 - kShift));
        const uint32_t a2 = (uint32_t)(x >> (kShift == 0 ? 63 : 64 - kShift));
        asm("add.cc.u32 %0, %0, %3;\n\taddc.cc.u32 %1, %1, %4;\n\taddc.u32 %2, %2, %5;"
            : "+r"(t.w0), "+r"(t.w1), "+r"(t.w2) : "r"(a0), "r"(a1), "r"(a2));
    } else {
        const uint32_t a1 = (uint32_t)x << (kShift - 32), a2 = (uint32_t)(x >> (64 - kShift));
        asm("add.cc.u32 %0, %0, %2;\n\taddc.u32 %1, %1, %3;" : "+r"(t.w1), "+r"(t.w2) : "r"(a1), "r"(a2));
    }
}

// umma_commit by the leader lane of a convergent warp.
__device__ __forceinline__ void commit_by(uint32_t leader, uint64_t* b) {
    asm volatile(
        "{\n\t.reg .pred q;\n\tsetp.ne.b32 q, %1, 0;\n\t"
        "@q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t}"
        :: "r"(sa(b)), "r"(leader) : "memory");
}

// One lane of the warp, always the same one.
__device__ __forceinline__ bool elect_one() {
    uint32_t p;
    asm volatile("{\n\t.reg .pred e;\n\telect.sync _|e, 0xffffffff;\n\tselp.u32 %0, 1, 0, e;\n\t}" : "=r"(p));
    return p != 0;
}

// Whether the phase of `parity` has completed, without waiting.
__device__ __forceinline__ bool mbar_test(uint32_t addr, uint32_t parity) {
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}\n"
        : "=r"(done) : "r"(addr), "r"(parity) : "memory");
    return done != 0;
}

// Contiguous copy of `bytes` (a multiple of 16) into shared memory.
__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
        :: "r"(dst), "l"(src), "r"(bytes), "r"(bar) : "memory");
}

__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap* map, int x, int y, int z, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
        :: "r"(dst), "l"((uint64_t)map), "r"(x), "r"(y), "r"(z), "r"(bar) : "memory");
}

// acc + v * mul (32 x 32 -> 64-bit multiply-add).
__device__ __forceinline__ long long mad_wide(int v, int mul, long long acc) {
    long long r;
    asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(v), "r"(mul), "l"(acc));
    return r;
}

// 2^{e - 64} T rounded to nearest once, from the exact sum T of an output element; results
// below the normal range flush to signed zero, above it to infinity.  Integer
// instructions only: the FP64 pipe runs two operations a cycle and SM, so that its
// conversions of two 64-bit sums, their addition and scaling cost an item of 128 x 64
// outputs 16,000 cycles and more.
__device__ __forceinline__ double combine(const Sum96& t, int e) {
    const uint32_t neg = (uint32_t)((int)t.w2 >> 31);
    uint32_t a0 = t.w0 ^ neg, a1 = t.w1 ^ neg, a2 = t.w2 ^ neg;      // |T|
    asm("sub.cc.u32 %0, %0, %3;\n\tsubc.cc.u32 %1, %1, %3;\n\tsubc.u32 %2, %2, %3;"
        : "+r"(a0), "+r"(a1), "+r"(a2) : "r"(neg));
    // leading bit to bit 31 of a2
    int ex = 1023 + 95 - 64 + e;
#pragma unroll
    for (int k = 0; k < 2; k++) {
        const bool z = a2 == 0;
        a2 = z ? a1 : a2;
        a1 = z ? a0 : a1;
        a0 = z ? 0u : a0;
        ex -= z ? 32 : 0;
    }
    const int lz = __clz((int)a2) & 31;
    a2 = __funnelshift_l(a1, a2, lz);
    a1 = __funnelshift_l(a0, a1, lz);
    a0 <<= lz;
    ex -= lz;                                                        // biased exponent of the leading bit
    // 53 bits, rounded to nearest even; the implicit bit adds one to the exponent field, as
    // does a mantissa that rounds up to 2^53
    uint32_t lo = __funnelshift_r(a1, a2, 11), hi = a2 >> 11;
    const uint32_t rest = ((a1 & 0x7ffu) << 1) | (a0 != 0 ? 1u : 0u);
    const uint32_t up = rest + (lo & 1u) > 0x800u ? 1u : 0u;
    hi += (uint32_t)(ex - 1) << 20;
    asm("add.cc.u32 %0, %0, %2;\n\taddc.u32 %1, %1, 0;" : "+r"(lo), "+r"(hi) : "r"(up));
    if (ex <= 0 || ex >= 0x7ff || hi >= 0x7ff00000u || a2 == 0) {
        lo = 0;
        hi = (a2 == 0 || ex <= 0) ? 0u : 0x7ff00000u;
        if (a2 == 0) return 0.0;
    }
    return __hiloint2double((int)(hi | (neg & 0x80000000u)), (int)lo);
}

// One CTA of 12 warps per SM.  kBsr: the BSR filter-step mode (its own instantiation, so
// that neither mode carries the other's epilogue registers).  NS: digit slices per operand
// (7, or 5 for the 40-bit steps).
template <bool kBsr, int NS>
__global__ void __launch_bounds__(kThreads, 1) oz_gemm_kernel(const __grid_constant__ OzArgs g,
                                                              const __grid_constant__ CUtensorMap tmA, int64_t total) {
    using Sh = OzShape<NS>;
    using Gr = Groups<NS>;
    constexpr int kSlots = Sh::kSlots, kSlotBytes = Sh::kSlotBytes;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    unsigned char* smem = (unsigned char*)(((uintptr_t)smem_raw + 127) & ~(uintptr_t)127);
    __shared__ __align__(8) uint64_t full[kMaxSlots], empty[kMaxSlots], efull[kEvents], eempty[kEvents], done;
    __shared__ __align__(8) uint64_t dfull[2], dempty[2];
    __shared__ uint32_t tmem_slot;
    __shared__ int abort_flag;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    bool nonfinite = false, bad_pattern = false;
    if (threadIdx.x == 0) {
        for (int s = 0; s < kSlots; s++) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        for (int e = 0; e < kEvents; e++) {
            mbar_init(&efull[e], 1);
            mbar_init(&eempty[e], kEpiWarps);
        }
        for (int d = 0; d < 2; d++) {
            mbar_init(&dfull[d], kEpiWarps);
            mbar_init(&dempty[d], 2);
        }
        mbar_init(&done, 1);
        asm volatile("fence.mbarrier_init.release.cluster;");
        asm volatile("fence.proxy.async.shared::cta;");
        abort_flag = 0;
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" :: "r"(sa(&tmem_slot)),
                     "r"(kTmemCols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
    const uint32_t tmem = tmem_slot;
    volatile int* abort_v = &abort_flag;

    if (warp < 4) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" :: "n"(kRegsIssue));
    if (warp == 0) {
        // ---------------- producer: lane 0 waits for the slot and announces its bytes, then
        // the lanes issue its copies
        int64_t sc = 0;
        int s = 0;
        uint32_t ph = 1;        // parity of the previous pass over the ring
        bool ok = true;
        // BSR mode: entry p of an item's list of Y_cur chunks, always a valid chunk
        auto list_entry = [&](const Item& it, int64_t p) -> int {
            int yc = kBsr && p < (int64_t)it.KB * kStageChunks ? g.hchunk[it.qc + p] : 0;
            if (yc < 0 || yc >= g.chunksA) { yc = 0; bad_pattern = true; }
            return yc;
        };
        Item it{}, next{};
        int list0 = 0, list1 = 0, next0 = 0;   // this lane's entries of the current 32, the next 32, the next item's first
        if (blockIdx.x < total) {
            next = decode<kBsr>(g, blockIdx.x);
            next0 = list_entry(next, lane);
        }
        for (int64_t item = blockIdx.x; ok && item < total; item += gridDim.x) {
            if (__any_sync(0xffffffffu, *abort_v)) break;
            it = next;
            list0 = next0;
            list1 = list_entry(it, 32 + lane);
            const int slots = it.KB * kStageSlots;
            if (item + gridDim.x < total) {    // the next item's sizes and list, a whole item ahead of their use
                next = decode<kBsr>(g, item + gridDim.x);
                next0 = list_entry(next, lane);
            }
            if (kBsr) {
                int qb, nq;
                bsr_row_range(g.brow_ptr, g.nblocks, it.tn, qb, nq, bad_pattern);
            }
            const unsigned char* At = g.A + ((int64_t)(it.batch * g.a_batch_tiles + it.tm) * g.chunksA) *
                                                (kSlices * kPlaneA);
            const unsigned char* Bt =
                kBsr ? g.B + it.qc * (kSlices * kPlaneB)
                     : g.B + ((int64_t)(it.batch * g.b_batch_tiles + it.tn) * g.chunksB) * (kSlices * kPlaneB);
            for (int sl = 0; sl < slots; sl++, sc++) {
                if (kBsr && sl % (32 / kSlotChunks) == 0 && sl > 0) {
                    list0 = list1;
                    list1 = list_entry(it, (int64_t)sl * kSlotChunks + 32 + lane);
                }
                const int64_t c0 = (int64_t)(it.kb0 * kStageSlots + sl) * kSlotChunks;
                bool got = true;
                if (lane == 0) {
                    if (sc >= kSlots) got = mbar_wait(sa(&empty[s]), ph, g.wait_ns);
                    if (got) mbar_expect_tx(&full[s], kSlotBytes);
                }
                if (!__all_sync(0xffffffffu, got)) { ok = false; break; }
                const uint32_t st = sa(smem + (size_t)s * kSlotBytes), bar = sa(&full[s]);
                if (kBsr) {
                    const int64_t yc = __shfl_sync(0xffffffffu, list0, (sl * kSlotChunks + lane) & 31);
                    if (lane < kSlotChunks) {       // chunks of Y_cur, and of H
                        bulk_load(st + lane * Sh::kChunkA, At + yc * (kSlices * kPlaneA), Sh::kChunkA, bar);
                        bulk_load(st + kSlotChunks * Sh::kChunkA + lane * Sh::kChunkB,
                                  Bt + (c0 + lane) * (kSlices * kPlaneB), Sh::kChunkB, bar);
                    }
                } else {
                    const uint32_t sb = st + kSlotChunks * Sh::kChunkA;
                    if (g.b_in_a) {
                        // columns 64 tn ..: the half (tn & 1) of every plane of 128-row tile tn / 2
                        if (lane == 0)
                            tma_load_3d(sb, &tmA, (it.tn & 1) * (kPlaneB / 4), 0,
                                        (int)((it.tn >> 1) * g.chunksA + c0), bar);
                    } else if (lane < kSlotChunks) {
                        bulk_load(sb + lane * Sh::kChunkB, Bt + (c0 + lane) * (kSlices * kPlaneB), Sh::kChunkB, bar);
                    }
                    if (lane >= 30)
                        bulk_load(st + (lane - 30) * Sh::kChunkA, At + (c0 + lane - 30) * (kSlices * kPlaneA),
                                  Sh::kChunkA, bar);
                }
                if (++s == kSlots) { s = 0; ph ^= 1; }
            }
        }
        if (!ok && lane == 0) *abort_v = 1;
        // every copy issued has landed before the CTA can exit
        __syncwarp();
        if (lane == 0)
            for (int q = 0; q < kSlots && q < sc; q++) {
                const int64_t last = q + ((sc - 1 - q) / kSlots) * kSlots;
                mbar_wait(sa(&full[q]), (uint32_t)((last / kSlots) & 1), kDrainNs);
            }
    } else if (warp == 1) {
        // ---------------- MMA issuer: the whole warp runs the loop on warp-uniform values, one
        // elected lane issues.
        // Drain number e uses barrier pair e % kEvents; pend_g is the last drain of group g
        // (five slices: pend1 and pend2 of the two sets of E4-E6), -1 once waited for, so that
        // at most three drains are on the way.
        const uint32_t tm = __shfl_sync(0xffffffffu, tmem, 0);
        const uint32_t ring = __shfl_sync(0xffffffffu, sa(smem), 0);
        const uint32_t leader = elect_one() ? 1u : 0u;
        int ev = 0, pend0 = -1, pend1 = -1, pend2 = -1;
        int set = 0;            // five slices: the set of E4-E6 in use
        int s = 0;
        uint32_t ph = 0;
        bool issued = false, ok = true;
        bool ready = false;     // slot s is known to be full
        int kb_next = blockIdx.x < total ? decode<kBsr>(g, blockIdx.x).KB : 0;
        for (int64_t item = blockIdx.x; ok && item < total; item += gridDim.x) {
            if (__any_sync(0xffffffffu, *abort_v)) break;
            const int KB = __shfl_sync(0xffffffffu, kb_next, 0);
            if (item + gridDim.x < total) kb_next = decode<kBsr>(g, item + gridDim.x).KB;   // an item ahead of its use
            int fresh = -1;     // the group drained after the last stage
            for (int kb = 0; kb < KB; kb++) {
                // the stage's two slots and their descriptors (each slot's first A and B plane)
                const int s0 = s, s1 = s + 1 == kSlots ? 0 : s + 1;
                const uint32_t ph0 = ph, ph1 = s + 1 == kSlots ? ph ^ 1 : ph;
                s = s1 + 1 == kSlots ? 0 : s1 + 1;
                ph = s1 + 1 == kSlots ? ph1 ^ 1 : ph1;
                const uint32_t st0 = ring + (uint32_t)(s0 * kSlotBytes), st1 = ring + (uint32_t)(s1 * kSlotBytes);
                const uint64_t da0 = desc_chunks(st0, Sh::kChunkA), da1 = desc_chunks(st1, Sh::kChunkA);
                const uint64_t db0 = desc_chunks(st0 + kSlotChunks * Sh::kChunkA, Sh::kChunkB);
                const uint64_t db1 = desc_chunks(st1 + kSlotChunks * Sh::kChunkA, Sh::kChunkB);
                auto wait_full = [&](int sl, uint32_t p) -> bool {
                    const bool w = ready || __all_sync(0xffffffffu, mbar_wait(sa(&full[sl]), p, g.wait_ns));
                    ready = false;
                    asm volatile("tcgen05.fence::after_thread_sync;");
                    return w;
                };
                // looks at a slot without waiting, while MMAs are queued
                auto test_full = [&](int sl, uint32_t p) { ready = __all_sync(0xffffffffu, mbar_test(sa(&full[sl]), p)); };
                // the drain that a group (or set) still waits for; after a wait that gave up,
                // nothing more is issued into accumulators that the epilogue may be reading
                auto test_drain = [&](int& pend) {
                    if (pend >= 0 && __all_sync(0xffffffffu, mbar_test(sa(&eempty[pend % kEvents]),
                                                                       (uint32_t)((pend / kEvents) & 1))))
                        pend = -1;
                };
                auto wait_drain = [&](int& pend) -> bool {
                    if (pend < 0) {
                        asm volatile("tcgen05.fence::after_thread_sync;");
                        return true;
                    }
                    const int e = pend;
                    pend = -1;
                    const bool w = __all_sync(0xffffffffu, mbar_wait(sa(&eempty[e % kEvents]),
                                                                     (uint32_t)((e / kEvents) & 1), g.wait_ns));
                    asm volatile("tcgen05.fence::after_thread_sync;");
                    return w;
                };
                bool w = true;
                issued = true;
                auto none = []() {};
                auto test1 = [&]() { test_full(s1, ph1); };
                auto test_next = [&]() { test_full(s, ph); };   // the next stage's (or item's) first slot
                if (!wait_full(s0, ph0)) { ok = false; break; }
                if constexpr (NS == 7) {
                    const uint32_t c0 = tm + Gr::column(0, 0), c1 = tm + Gr::column(1, 0), c2 = tm + Gr::column(2, 0);
                    if (kb == 0) {                     // each group when the last item's sums have left it
                        w = wait_full(s1, ph1) && wait_drain(pend0);
                        if (w) {
                            issue_range<NS, 5, 7>(leader, da0, db0, c0, true, none);
                            issue_range<NS, 5, 7>(leader, da1, db1, c0, false, none);
                            w = wait_drain(pend1);
                        }
                        if (w) {
                            issue_range<NS, 3, 5>(leader, da0, db0, c1, true, none);
                            issue_range<NS, 3, 5>(leader, da1, db1, c1, false, none);
                            w = wait_drain(pend2);
                        }
                        if (w) {
                            issue_range<NS, 0, 3>(leader, da0, db0, c2, true, none);
                            commit_by(leader, &empty[s0]);
                            issue_range<NS, 0, 3>(leader, da1, db1, c2, false, test_next);
                        }
                    } else if (fresh < 0) {
                        issue_range<NS, 0, 7>(leader, da0, db0, tm, false, test1);
                        commit_by(leader, &empty[s0]);
                        if ((w = wait_full(s1, ph1))) issue_range<NS, 0, 7>(leader, da1, db1, tm, false, test_next);
                    } else if (fresh == 0) {           // the other groups, then the drained one
                        issue_range<NS, 0, 5>(leader, da0, db0, tm, false, test1);
                        if ((w = wait_full(s1, ph1))) {
                            issue_range<NS, 0, 5>(leader, da1, db1, tm, false, [&]() { test_drain(pend0); });
                            w = wait_drain(pend0);
                        }
                        if (w) {
                            issue_range<NS, 5, 7>(leader, da0, db0, c0, true, none);
                            commit_by(leader, &empty[s0]);
                            issue_range<NS, 5, 7>(leader, da1, db1, c0, false, test_next);
                        }
                    } else if (fresh == 1) {
                        issue_range<NS, 5, 7>(leader, da0, db0, c0, false, test1);
                        issue_range<NS, 0, 3>(leader, da0, db0, c2, false, none);
                        if ((w = wait_full(s1, ph1))) {
                            issue_range<NS, 5, 7>(leader, da1, db1, c0, false, [&]() { test_drain(pend1); });
                            issue_range<NS, 0, 3>(leader, da1, db1, c2, false, none);
                            w = wait_drain(pend1);
                        }
                        if (w) {
                            issue_range<NS, 3, 5>(leader, da0, db0, c1, true, none);
                            commit_by(leader, &empty[s0]);
                            issue_range<NS, 3, 5>(leader, da1, db1, c1, false, test_next);
                        }
                    } else {
                        issue_range<NS, 3, 7>(leader, da0, db0, c1, false, test1);
                        if ((w = wait_full(s1, ph1))) {
                            issue_range<NS, 3, 7>(leader, da1, db1, c1, false, [&]() { test_drain(pend2); });
                            w = wait_drain(pend2);
                        }
                        if (w) {
                            issue_range<NS, 0, 3>(leader, da0, db0, c2, true, none);
                            commit_by(leader, &empty[s0]);
                            issue_range<NS, 0, 3>(leader, da1, db1, c2, false, test_next);
                        }
                    }
                } else {
                    const bool fresh0 = kb == 0 || fresh == 0, fresh1 = kb == 0 || fresh == 1;
                    const uint32_t d0 = tm + Gr::column(0, 0), d1 = tm + Gr::column(1, set);
                    if (fresh1) w = set ? wait_drain(pend2) : wait_drain(pend1);   // this set's drain before the last
                    if (w && !fresh0) {
                        issue_range<NS, 0, 2>(leader, da0, db0, d0, false, none);
                        issue_range<NS, 2, 5>(leader, da0, db0, d1, fresh1, test1);
                        commit_by(leader, &empty[s0]);
                        if ((w = wait_full(s1, ph1))) {
                            issue_range<NS, 0, 2>(leader, da1, db1, d0, false, none);
                            issue_range<NS, 2, 5>(leader, da1, db1, d1, false, test_next);
                        }
                    } else if (w) {
                        issue_range<NS, 2, 5>(leader, da0, db0, d1, fresh1, test1);
                        if ((w = wait_full(s1, ph1))) {
                            issue_range<NS, 2, 5>(leader, da1, db1, d1, false, [&]() { test_drain(pend0); });
                            w = wait_drain(pend0);
                        }
                        if (w) {
                            issue_range<NS, 0, 2>(leader, da0, db0, d0, true, none);
                            commit_by(leader, &empty[s0]);
                            issue_range<NS, 0, 2>(leader, da1, db1, d0, false, test_next);
                        }
                    }
                }
                commit_by(leader, &empty[s1]);
                if (!w) { ok = false; break; }
                auto event = [&](int& pend) {
                    commit_by(leader, &efull[ev % kEvents]);
                    pend = ev++;
                };
                fresh = Gr::event(kb);
                const bool last = kb == KB - 1;
                if (last || fresh == 0) event(pend0);
                if (last || fresh == 1) {
                    if (NS == 5 && set) event(pend2);
                    else event(pend1);
                    if (NS == 5) set ^= 1;
                }
                if (NS == 7 && (last || fresh == 2)) event(pend2);
            }
        }
        if (!ok && lane == 0) *abort_v = 1;
        // every MMA issued has completed before TMEM is released
        if (issued) {
            commit_by(leader, &done);
            mbar_wait(sa(&done), 0, kDrainNs);
        }
    } else if (kBsr) {
        // ---------------- output of the BSR mode (two warps, 64 states each): Y_out = alpha D -
        // beta Y_prev from the products D that the epilogue has left in Y_out, with D already
        // of H - c unless the row is unfolded.  Warps of their own: the two FP64 operations an
        // element take 8200 cycles an item at least and wait for Y_prev; done by the epilogue
        // warps (at once, or in pieces between the drains) they kept the drains and so
        // the MMAs waiting for a fifth of the time, and no registers or shared memory are left
        // to hold an item's products for later, but L2 is.  They also leave the exponents that the
        // next step's slices need (a pass over Y_out otherwise: 75 us of 3.1 ms at 40^3 x 1024).
        int n = 0;
        bool ok = true;
        for (int64_t item = blockIdx.x; ok && item < total; item += gridDim.x, n++) {
            if (__any_sync(0xffffffffu, *abort_v)) break;
            const Item it = decode<kBsr>(g, item);
            ok = __all_sync(0xffffffffu, mbar_wait(sa(&dfull[n & 1]), (uint32_t)((n >> 1) & 1), g.wait_ns));
            if (!ok) break;
            constexpr int kStep = 4;
            const int64_t i0 = (int64_t)it.tn * kTileN;
#pragma unroll 1
            for (int half = 0; half < 2; half++) {
                const int64_t j = (int64_t)it.tm * kTileM + 64 * (warp - 2) + 32 * half + lane;
                if (j >= g.M) continue;
                double* out = g.C + i0 * g.ldc + j;
                const double* prev = g.Yprev ? g.Yprev + i0 * g.ldprev + j : nullptr;
                double d[2][kStep], p[2][kStep];
                int emax = 0;
                auto load = [&](int b, int r) {
#pragma unroll
                    for (int c = 0; c < kStep; c++) {
                        d[b][c] = out[(r + c) * g.ldc];
                        p[b][c] = prev ? prev[(r + c) * g.ldprev] : 0.0;
                    }
                };
                load(0, 0);
#pragma unroll 2
                for (int r = 0; r < kTileN; r += kStep) {
                    const int b = (r / kStep) & 1;
                    if (r + kStep < kTileN) load(b ^ 1, r + kStep);   // on the way before this step's stores
#pragma unroll
                    for (int c = 0; c < kStep; c++) {
                        double D = d[b][c];
                        if (it.unfolded) D = fma(-g.cshift, g.Ycur[(i0 + r + c) * g.ldcur + j], D);
                        double y = g.alpha * D;
                        if (prev) y = fma(-g.beta, p[b][c], y);
                        const int ef = (__double2hiint(y) >> 20) & 0x7ff;
                        emax = ef > emax ? ef : emax;
                        out[(r + c) * g.ldc] = y;
                    }
                }
                nonfinite |= emax == 0x7ff;
                if (emax) atomicMax(g.expNext + j, emax);
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&dempty[n & 1]);
        }
        if (!ok && lane == 0) *abort_v = 1;
    }
    } else {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" :: "n"(kRegsEpilogue));
        // ---------------- epilogue: exact drains into 96-bit integers, then the output
        const int q = warp & 3, h = (warp - 4) >> 2;
        const uint32_t lane_base = (uint32_t)(32 * q) << 16;
        int ev = 0, set = 0;
        Sum96 sum[kColsPerThread];
        // drain number ev, of group GI: its accumulators are given back as soon as they are in
        // registers, the last conversions (16 lanes a cycle and SM) overlap the next MMAs
        auto drain = [&](auto gc) -> bool {
            constexpr int GI = decltype(gc)::value, LO = Gr::lo(GI), HI = Gr::hi(GI), kAccs = HI - LO;
            constexpr int kBatch = kAccs > 2 ? 16 : 32;       // columns read before they are converted
            constexpr int kShift = 64 - 8 * (HI + 1);         // unit of E_{HI + 1}
            const int slot = ev % kEvents;
            if (!__all_sync(0xffffffffu,
                            !*abort_v && mbar_wait(sa(&efull[slot]), (uint32_t)((ev / kEvents) & 1), g.wait_ns)))
                return false;
            asm volatile("tcgen05.fence::after_thread_sync;");
            const uint32_t at = tmem + lane_base + (uint32_t)(Gr::column(GI, set) + h * kColsPerThread);
#pragma unroll
            for (int c0 = 0; c0 < kColsPerThread; c0 += kBatch) {
                uint32_t v[kAccs][kBatch / 8][8];
#pragma unroll
                for (int a = 0; a < kAccs; a++)
#pragma unroll
                    for (int k = 0; k < kBatch / 8; k++) tmem_ld8(at + (uint32_t)(a * kTileN + c0 + 8 * k), v[a][k]);
                asm volatile("tcgen05.wait::ld.sync.aligned;");
                if (c0 + kBatch == kColsPerThread) {
                    asm volatile("tcgen05.fence::before_thread_sync;");
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&eempty[slot]);
                }
#pragma unroll
                for (int c = 0; c < kBatch; c++) {
                    // E_l holds an integer of at most 2^24, in units of 2^-8l
                    long long x = __float2int_rn(__uint_as_float(v[kAccs - 1][c / 8][c % 8]));
#pragma unroll
                    for (int a = kAccs - 2; a >= 0; a--)
                        x = mad_wide(__float2int_rn(__uint_as_float(v[a][c / 8][c % 8])), 1 << (8 * (kAccs - 1 - a)), x);
                    add96<kShift>(sum[c0 + c], x);
                }
            }
            if (NS == 5 && GI == 1) set ^= 1;
            ev++;
            return true;
        };
        auto drain_group = [&](int gi) -> bool {
            if (gi == 0) return drain(std::integral_constant<int, 0>{});
            if (NS == 5 || gi == 1) return drain(std::integral_constant<int, 1>{});
            return drain(std::integral_constant<int, Gr::kCount - 1>{});
        };
        int n = 0;
        for (int64_t item = blockIdx.x; item < total; item += gridDim.x, n++) {
            const Item it = decode<kBsr>(g, item);
#pragma unroll
            for (int c = 0; c < kColsPerThread; c++) sum[c] = Sum96{0, 0, 0};
            if (kBsr && *abort_v) break;
            // exponents of the item's state and (one a lane) of its grid rows
            int ea = 0, eh = 0;
            if (kBsr && it.KB > 0) {
                const int j = it.tm * kTileM + 32 * q + lane;
                if (j < g.M) ea = g.expA[j];
                eh = g.expH[it.tn * kTileN + h * kColsPerThread + lane];
            }
            bool ok = true;
            for (int kb = 0; ok && kb < it.KB; kb++) {
                const bool end = kb == it.KB - 1;
                const int gi0 = end ? 0 : Gr::event(kb);
                if (gi0 < 0) continue;
                for (int gi = gi0; ok && (gi == gi0 || (end && gi < Gr::kCount)); gi++) ok = drain_group(gi);
            }
            if (!ok) { *abort_v = 1; break; }
            if constexpr (kBsr) {
                // the products (zero for an empty block row) for the output warps
                const int64_t j = (int64_t)it.tm * kTileM + 32 * q + lane;
                double* out = g.C + ((int64_t)it.tn * kTileN + h * kColsPerThread) * g.ldc + j;
#pragma unroll
                for (int c = 0; c < kColsPerThread; c++) {
                    const int eb = __shfl_sync(0xffffffffu, eh, c);
                    const double D = (ea != 0 && eb != 0) ? combine(sum[c], (ea - 1021) + (eb - 1021)) : 0.0;
                    if (j < g.M) out[c * g.ldc] = D;
                }
                if (n >= 2 && !__all_sync(0xffffffffu, mbar_wait(sa(&dempty[n & 1]), (uint32_t)(((n - 2) >> 1) & 1),
                                                                 g.wait_ns))) {
                    *abort_v = 1;
                    break;
                }
                __syncwarp();
                if (lane == 0) mbar_arrive(&dfull[n & 1]);
            } else if (it.KB > 0) {
                const int64_t row = (int64_t)it.tm * kTileM + 32 * q + lane;        // within the batch
                const int64_t orow = it.batch * g.m_batch + row;                     // output row
                const int64_t col0 = (int64_t)it.tn * kTileN + h * kColsPerThread;
                const bool valid = row < g.m_batch && orow < g.M;
                const int ea = valid ? g.expA[it.batch * g.a_batch_tiles * kTileM + row] : 0;
                const int* expB = g.expB + it.batch * g.b_batch_tiles * kTileN;
                double* dst = g.part ? g.part + ((int64_t)(it.kb0 / g.kb_split) * g.Mp + row) * g.Np + col0
                                     : g.C + orow * g.ldc + col0;
                const bool whole = g.part || (valid && col0 + kColsPerThread <= g.Nc &&
                                              (reinterpret_cast<uintptr_t>(dst) & 31u) == 0);
#pragma unroll
                for (int c0 = 0; c0 < kColsPerThread; c0 += 4) {
                    double v[4];
#pragma unroll
                    for (int c = 0; c < 4; c++) {
                        const int eb = (col0 + c0 + c < g.Nc) ? expB[col0 + c0 + c] : 0;
                        v[c] = (ea != 0 && eb != 0) ? combine(sum[c0 + c], (ea - 1021) + (eb - 1021)) : 0.0;
                    }
                    if (whole) {     // a thread's columns as whole 32-byte sectors
                        asm volatile("st.global.v4.f64 [%0], {%1, %2, %3, %4};"
                                     :: "l"(dst + c0), "d"(v[0]), "d"(v[1]), "d"(v[2]), "d"(v[3]) : "memory");
                    } else if (valid) {
#pragma unroll
                        for (int c = 0; c < 4; c++)
                            if (col0 + c0 + c < g.Nc) dst[c0 + c] = v[c];
                    }
                }
            }
        }
    }

    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    if (warp == 1) {
        asm volatile("tcgen05.fence::after_thread_sync;");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" :: "r"(tmem), "r"(kTmemCols));
    }
    if (threadIdx.x == 0 && abort_flag) raise_status(g.status, DEV_TIMEOUT);
    if (nonfinite) raise_status(g.status, DEV_NONFINITE);
    if (bad_pattern) raise_status(g.status, DEV_PATTERN);
}

// Largest biased exponent field of each row of A_hat (A_hat[r][k] = src[k * ld + r]
// when trans, else src[r * ld + k]); 0 for a row of zeros (subnormals count as zero).
// Batch z = blockIdx.z reads src + z * src_bstride over K_z = min(Kb, Ktot - z Kb) and
// writes exps + z * rows_pad.  exps must be zeroed first.
// kTrans: a thread per column of src, span of its rows per block row, eight loads in
// flight.  Short spans where K is small: the loads of a span follow one another (64 rows
// in one span, four at a time, took 13 us).
inline int exponent_span(int64_t K) { return K <= 4096 ? 32 : 256; }

template <bool kTrans>
__global__ void oz_exponents_kernel(const double* __restrict__ src, int64_t ld, int64_t rows, int64_t Kb,
                                    int64_t Ktot, int64_t src_bstride, int64_t rows_pad, int span, int* exps,
                                    unsigned* status) {
    const int64_t z = blockIdx.z;
    src += z * src_bstride;
    exps += z * rows_pad;
    const int64_t K = Ktot - z * Kb < Kb ? Ktot - z * Kb : Kb;
    int m = 0;
    bool bad = false;
    if (kTrans) {
        const int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
        const int64_t k0 = (int64_t)blockIdx.y * span;
        if (r >= rows) return;
        const int64_t k1 = k0 + span < K ? k0 + span : K;
        for (int64_t k = k0; k < k1; k += 8) {
            double x[8];
#pragma unroll
            for (int u = 0; u < 8; u++) x[u] = k + u < k1 ? src[(k + u) * ld + r] : 0.0;
#pragma unroll
            for (int u = 0; u < 8; u++) {
                const int ef = (__double2hiint(x[u]) >> 20) & 0x7ff;
                m = ef > m ? ef : m;
            }
        }
        bad = m == 0x7ff;
        if (m) atomicMax(exps + r, m);
    } else {
        // warp per row
        const int64_t r = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
        const int lane = threadIdx.x & 31;
        if (r >= rows) return;
        for (int64_t k = lane; k < K; k += 32) {
            const int ef = (int)((__double_as_longlong(src[r * ld + k]) >> 52) & 0x7ff);
            bad |= ef == 0x7ff;
            m = ef > m ? ef : m;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
        if (lane == 0) exps[r] = m;
    }
    if (bad) raise_status(status, DEV_NONFINITE);
}

// Fixed-point form of x in a row whose largest exponent field is efm: sign(x) |x| 2^{-e}
// 2^{56} rounded to nearest, e = efm - 1021, below 2^55 in magnitude.
__device__ __forceinline__ long long fixed_point(double x, int efm) {
    const long long b = __double_as_longlong(x);
    const int ef = (int)((b >> 52) & 0x7ff);
    if (ef == 0 || efm == 0 || ef == 0x7ff) return 0;
    const long long mant = (b & ((1ll << 52) - 1)) | (1ll << 52);
    const int sh = efm - ef - 2;
    long long F;
    if (sh <= 0) F = mant << (-sh);
    else F = sh < 60 ? (mant + (1ll << (sh - 1))) >> sh : 0;
    return b < 0 ? -F : F;
}

// The seven digit planes of eight consecutive K entries of a row, 16 bytes per plane.
// Balanced base-256 digits in [-128, 127] (the top one keeps the carry): adding 128 to
// each of the six low digits at once turns them into the bytes of G, so digit = byte -
// 128 without a carry chain; bytes become floats by placing them under 2^23, and an exact
// BF16 is the upper half of its float.
__device__ __forceinline__ void digits8(const long long (&F)[kChunk], uint4 (&out)[kSlices]) {
    uint32_t w[kSlices][4];
#pragma unroll
    for (int pr = 0; pr < kChunk / 2; pr++) {
        float f[2][kSlices];
#pragma unroll
        for (int k = 0; k < 2; k++) {
            const long long G = F[2 * pr + k] + 0x0000808080808080ll;
            const uint32_t glo = (uint32_t)G, ghi = (uint32_t)((unsigned long long)G >> 32);
            f[k][0] = __int_as_float(0x4B400000 + ((int)ghi >> 16)) - 12582912.0f;
#pragma unroll
            for (int t = 1; t < kSlices; t++) {
                const int byte = kSlices - 1 - t;
                const uint32_t u = __byte_perm(byte < 4 ? glo : ghi, 0x4B000000u, 0x7440u + (uint32_t)(byte & 3));
                f[k][t] = __uint_as_float(u) - 8388736.0f;
            }
        }
#pragma unroll
        for (int t = 0; t < kSlices; t++)
            w[t][pr] = __byte_perm(__float_as_uint(f[0][t]), __float_as_uint(f[1][t]), 0x7632);
    }
#pragma unroll
    for (int t = 0; t < kSlices; t++) out[t] = make_uint4(w[t][0], w[t][1], w[t][2], w[t][3]);
}

// Digit planes of A_hat in tiles of kRows rows: [batch z][row tile][K chunk][7][kRows][8],
// zero in the padding; batch z = blockIdx.z as in oz_exponents_kernel.  Only the first
// nplanes planes are written (the five-slice steps read no others).  A thread makes the
// eight digits of one row and chunk, so that each plane is written 16 bytes a thread and
// 512 contiguous bytes a warp: bounded by the reads of src and those writes.
// kTrans (A_hat[r][k] = src[k * ld + r]): a warp reads 32 consecutive columns of each of
// the chunk's src rows, straight into the threads that need them.  Otherwise 32 rows x 64
// columns pass through shared memory.
template <bool kTrans, int kRows>
__global__ void __launch_bounds__(256) oz_slice_kernel(const double* __restrict__ src, int64_t ld, int64_t rows,
                                                       int64_t Kb, int64_t Ktot, int64_t src_bstride,
                                                       const int* __restrict__ exps, int64_t tiles, int64_t chunks,
                                                       int nplanes, unsigned char* __restrict__ slices) {
    const int64_t z = blockIdx.z;
    src += z * src_bstride;
    exps += z * tiles * kRows;
    slices += (size_t)(z * tiles * chunks) * (kSlices * kRows * 16);
    const int64_t K = Ktot - z * Kb < Kb ? Ktot - z * Kb : Kb;
    auto store = [&](const double (&x)[kChunk], int64_t r, int64_t ch, int efm) {
        long long F[kChunk];
#pragma unroll
        for (int k = 0; k < kChunk; k++) F[k] = fixed_point(x[k], efm);
        uint4 dg[kSlices];
        digits8(F, dg);
        uint4* dst = reinterpret_cast<uint4*>(slices) + ((r / kRows) * chunks + ch) * (kSlices * kRows) + r % kRows;
#pragma unroll
        for (int t = 0; t < kSlices; t++)
            if (t < nplanes) dst[t * kRows] = dg[t];
    };
    if (kTrans) {
        // blocks of 256 / kRows chunks x one row tile
        const int64_t ch = (int64_t)blockIdx.x * (256 / kRows) + threadIdx.x / kRows;
        if (ch >= chunks) return;
        const int64_t k0 = ch * kChunk;
        for (int64_t rt = blockIdx.y; rt < tiles; rt += gridDim.y) {
            const int64_t r = rt * kRows + threadIdx.x % kRows;
            double x[kChunk];
#pragma unroll
            for (int k = 0; k < kChunk; k++) x[k] = (r < rows && k0 + k < K) ? src[(k0 + k) * ld + r] : 0.0;
            store(x, r, ch, r < rows ? exps[r] : 0);
        }
    } else {
        __shared__ double tile[32][65];
        const int64_t k0 = (int64_t)blockIdx.x * 64;
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
        for (int64_t rt = blockIdx.y; rt < tiles * (kRows / 32); rt += gridDim.y) {
            const int64_t r0 = rt * 32;
            __syncthreads();   // the previous tile has been read
            for (int i = warp; i < 32; i += 8)
#pragma unroll
                for (int e = 0; e < 2; e++) {
                    const int64_t k = k0 + 32 * e + lane;
                    tile[i][32 * e + lane] = (r0 + i < rows && k < K) ? src[(r0 + i) * ld + k] : 0.0;
                }
            __syncthreads();
            const int64_t ch = (int64_t)blockIdx.x * 8 + warp, r = r0 + lane;
            if (ch < chunks) {
                double x[kChunk];
#pragma unroll
                for (int k = 0; k < kChunk; k++) x[k] = tile[lane][warp * kChunk + k];
                store(x, r, ch, r < rows ? exps[r] : 0);
            }
        }
    }
}

// C (= C - when subtract) the sum over splits of the partial tiles; for a symmetric product
// an element below the diagonal takes its mirror above it (always in a computed tile).  A
// block per 256 columns of a row: with the row and column from a 64-bit division per element
// the pass took twice as long.
__global__ void __launch_bounds__(256) oz_reduce_kernel(const double* __restrict__ part, int splits, int64_t Mp,
                                                        int64_t Np, int64_t M, int64_t Nc, double* C, int64_t ldc,
                                                        int symmetric, int subtract) {
    const int64_t c = (int64_t)blockIdx.x * 256 + threadIdx.x;
    if (c >= Nc) return;
    for (int64_t r = blockIdx.y; r < M; r += gridDim.y) {
        const bool below = symmetric && r > c;
        const double* p = part + (below ? c * Np + r : r * Np + c);
        double s = 0.0;
        for (int z = 0; z < splits; z++) s += p[(int64_t)z * Mp * Np];
        double* d = C + r * ldc + c;
        *d = subtract ? *d - s : s;
    }
}

inline int64_t round_up(int64_t x, int64_t m) { return (x + m - 1) / m * m; }

// Arena stand-in that only counts bytes.
struct CountAr {
    Sizer s;
    template <typename T>
    T* take(size_t n) {
        s.take<T>(n);
        return nullptr;
    }
};

// Workspace pieces of one operand: exponents (int32 per padded row) and digit planes
// [nbatch][row tile][K chunk][7][tile_rows][8]; tile_rows 128 for A_hat, 64 for B_hat.
struct OzOperand {
    int* exps = nullptr;
    unsigned char* slices = nullptr;
    int64_t rows = 0, K = 0, tiles = 0, chunks = 0;
    int tile_rows = kTileM;
    int nbatch = 1;
    int64_t padded_rows() const { return (int64_t)nbatch * tiles * tile_rows; }
};

template <typename Ar>
void oz_operand_layout(Ar& ar, int64_t rows, int64_t K, int nbatch, int tile_rows, OzOperand* op) {
    OzOperand o;
    o.rows = rows;
    o.K = K;
    o.nbatch = nbatch;
    o.tile_rows = tile_rows;
    o.tiles = (rows + tile_rows - 1) / tile_rows;
    o.chunks = round_up(K, kKB) / kChunk;
    o.exps = ar.template take<int>((size_t)o.padded_rows());
    o.slices = ar.template take<unsigned char>((size_t)o.padded_rows() * o.chunks * (kSlices * 16));
    if (op) *op = o;
}

template <bool kTrans, int kRows>
int launch_slices(const double* src, int64_t ld, const OzOperand& o, int64_t Ktot, int64_t src_bstride, int nplanes,
                  cudaStream_t s) {
    const int64_t per = kTrans ? 256 / kRows : 8, ytiles = kTrans ? o.tiles : o.tiles * (kRows / 32);
    const dim3 grid((unsigned)((o.chunks + per - 1) / per), (unsigned)std::min<int64_t>(ytiles, 65535),
                    (unsigned)o.nbatch);
    oz_slice_kernel<kTrans, kRows><<<grid, 256, 0, s>>>(src, ld, o.rows, o.K, Ktot, src_bstride, o.exps, o.tiles,
                                                        o.chunks, nplanes, o.slices);
    CHFSI_LAUNCH_CHECK();
    return CHFSI_OK;
}

// Exponents (unless have_exps) and digit planes of an operand; batch b reads src + b * src_bstride over
// min(o.K, Ktot - b o.K) of the K dimension.  nplanes: digit planes written.
int oz_prepare(const double* src, int64_t ld, bool trans, const OzOperand& o, int64_t Ktot, int64_t src_bstride,
               unsigned* status, cudaStream_t s, int nplanes = kSlices, bool have_exps = false) {
    const int64_t brows = o.tiles * o.tile_rows;
    if (!have_exps) CHFSI_CUDA_TRY(cudaMemsetAsync(o.exps, 0, sizeof(int) * (size_t)o.padded_rows(), s));
    if (have_exps) {
        // the exponents are there (left by the step that made src)
    } else if (trans) {
        const int span = exponent_span(o.K);
        dim3 grid((unsigned)((o.rows + 255) / 256), (unsigned)((o.K + span - 1) / span), (unsigned)o.nbatch);
        oz_exponents_kernel<true><<<grid, 256, 0, s>>>(src, ld, o.rows, o.K, Ktot, src_bstride, brows, span, o.exps,
                                                      status);
        CHFSI_LAUNCH_CHECK();
    } else {
        dim3 grid((unsigned)((o.rows * 32 + 255) / 256), 1, (unsigned)o.nbatch);
        oz_exponents_kernel<false><<<grid, 256, 0, s>>>(src, ld, o.rows, o.K, Ktot, src_bstride, brows, 0, o.exps,
                                                       status);
        CHFSI_LAUNCH_CHECK();
    }
    if (o.tile_rows == kTileM)
        return trans ? launch_slices<true, kTileM>(src, ld, o, Ktot, src_bstride, nplanes, s)
                     : launch_slices<false, kTileM>(src, ld, o, Ktot, src_bstride, nplanes, s);
    return trans ? launch_slices<true, kTileN>(src, ld, o, Ktot, src_bstride, nplanes, s)
                 : launch_slices<false, kTileN>(src, ld, o, Ktot, src_bstride, nplanes, s);
}

// Split-K count for a product whose output has `tiles` tiles: at most kMaxItemKB
// K-blocks per work item (the range of the 96-bit sums), and enough items
// for about one per SM while each split keeps at least 2048 K.
int oz_splits(int64_t tiles, int kb_total, int sms) {
    const int64_t need = (kb_total + kMaxItemKB - 1) / kMaxItemKB;
    int64_t want = (sms + tiles - 1) / tiles;
    constexpr int64_t kMinSplitKB = 2048 / kKB;
    const int64_t maxs = (kb_total + kMinSplitKB - 1) / kMinSplitKB;
    if (want > maxs) want = maxs;
    const int64_t sp = want > need ? want : need;
    return (int)(sp < 1 ? 1 : sp);
}

struct OzPlan {
    OzOperand A, B;
    double* part = nullptr;
    int splits = 1;
    bool same = false;        // B_hat is A_hat (a Gram matrix)
};

// M x Nc output, K reduction; tn_form: C = A^T B (split over K), else C = A B.
template <typename Ar>
void oz_layout(Ar& ar, bool tn_form, int64_t M, int64_t Nc, int64_t K, bool same, OzPlan* plan) {
    OzPlan p;
    p.same = same;
    oz_operand_layout(ar, M, K, 1, kTileM, &p.A);
    if (same) p.B = p.A;
    else oz_operand_layout(ar, Nc, K, 1, kTileN, &p.B);
    if (tn_form) {
        const int64_t tm = (M + kTileM - 1) / kTileM, tn = (Nc + kTileN - 1) / kTileN;
        p.splits = oz_splits(tm * tn, (int)(p.A.chunks / kStageChunks), (int)sm_count_or_default());
        p.part = ar.template take<double>((size_t)p.splits * (tm * kTileM) * (tn * kTileN));
    }
    if (plan) *plan = p;
}

// One persistent CTA per SM (or per work item, if fewer).
int launch_oz(const OzArgs& g, const CUtensorMap& tmA, int64_t total, cudaStream_t s) {
    if (total <= 0) return CHFSI_OK;
    const int dev = current_device();
    if (dev < 0) return CHFSI_ERR_CUDA;
    if (g.slices != 7 && !(g.slices == 5 && g.bsr)) return CHFSI_ERR_ARG;
    static bool attr[kMaxDevices] = {};
    if (!attr[dev]) {
        CHFSI_CUDA_TRY(cudaFuncSetAttribute(oz_gemm_kernel<false, 7>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                            OzShape<7>::kSmemBytes));
        CHFSI_CUDA_TRY(cudaFuncSetAttribute(oz_gemm_kernel<true, 7>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                            OzShape<7>::kSmemBytes));
        CHFSI_CUDA_TRY(cudaFuncSetAttribute(oz_gemm_kernel<true, 5>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                            OzShape<5>::kSmemBytes));
        attr[dev] = true;
    }
    const int sms = sm_count();
    if (sms <= 0) return CHFSI_ERR_CUDA;
    const unsigned grid = (unsigned)(total < sms ? total : sms);
    if (g.bsr && g.slices == 5)
        oz_gemm_kernel<true, 5><<<grid, kThreads, OzShape<5>::kSmemBytes, s>>>(g, tmA, total);
    else if (g.bsr)
        oz_gemm_kernel<true, 7><<<grid, kThreads, OzShape<7>::kSmemBytes, s>>>(g, tmA, total);
    else
        oz_gemm_kernel<false, 7><<<grid, kThreads, OzShape<7>::kSmemBytes, s>>>(g, tmA, total);
    CHFSI_LAUNCH_CHECK();
    return CHFSI_OK;
}

// Tensor map over the planes of an operand with 128-row tiles, [tile and chunk][7][512
// words]: a box is 64 rows of the seven planes of a slot's two chunks.
int make_map_planes(CUtensorMap* map, const OzOperand& o) {
    EncodeTiledFn enc = encode_fn();
    if (!enc) return CHFSI_ERR_CUDA;
    const cuuint64_t dims[3] = {kPlaneA / 4, kSlices, (cuuint64_t)(o.nbatch * o.tiles * o.chunks)};
    const cuuint64_t strides[2] = {kPlaneA, kSlices * kPlaneA};
    const cuuint32_t box[3] = {kPlaneB / 4, kSlices, kSlotChunks}, es[3] = {1, 1, 1};
    const CUresult r = enc(map, CU_TENSOR_MAP_DATA_TYPE_UINT32, 3, o.slices, dims, strides, box, es,
                           CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                           CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? CHFSI_OK : CHFSI_ERR_CUDA;
}

// The product of prepared operands.  nbatch > 1: independent products, batch b of the
// output at rows b * m_batch (m_batch rows each, the last one clipped at M).
int oz_run(const OzPlan& p, bool tn_form, double* C, int64_t ldc, int64_t M, int64_t Nc, bool symmetric,
           bool b_upper, unsigned* status, cudaStream_t s, int nbatch = 1, int64_t m_batch = 0, bool subtract = false) {
    if (M <= 0 || Nc <= 0) return CHFSI_OK;
    const int64_t K_pad = p.A.chunks * kChunk;
    if (K_pad > (int64_t)1 << 21 || p.A.padded_rows() * kSlices > INT32_MAX || p.B.padded_rows() * kSlices > INT32_MAX)
        return CHFSI_ERR_UNSUPPORTED;
    if (!tn_form && K_pad > (int64_t)kMaxItemKB * kKB) return CHFSI_ERR_UNSUPPORTED;   // no split-K in the nn form
    if (nbatch > 1 && (tn_form || symmetric || p.A.nbatch != nbatch || p.B.nbatch != nbatch || m_batch <= 0 ||
                       m_batch > p.A.tiles * kTileM))
        return CHFSI_ERR_ARG;
    int rc;
    CUtensorMap tmA{};
    if (p.same && (rc = make_map_planes(&tmA, p.A))) return rc;
    OzArgs g{};
    const int64_t mb = nbatch > 1 ? m_batch : M;
    g.M = M;
    g.Nc = Nc;
    g.ldc = ldc;
    g.nbatch = nbatch;
    g.m_batch = mb;
    g.A = p.A.slices;
    g.B = p.B.slices;
    g.b_in_a = p.same ? 1 : 0;
    g.chunksA = p.A.chunks;
    g.chunksB = p.B.chunks;
    g.a_batch_tiles = p.A.tiles;
    g.b_batch_tiles = p.B.tiles;
    g.tilesM = (int)((mb + kTileM - 1) / kTileM);
    g.tilesN = (int)((Nc + kTileN - 1) / kTileN);
    g.Mp = (int64_t)g.tilesM * kTileM;
    g.Np = (int64_t)g.tilesN * kTileN;
    g.expA = p.A.exps;
    g.expB = p.B.exps;
    g.kb_total = (int)(K_pad / kKB);
    g.splits = tn_form ? p.splits : 1;
    g.kb_split = (g.kb_total + g.splits - 1) / g.splits;
    g.splits = (g.kb_total + g.kb_split - 1) / g.kb_split;   // no empty split
    g.symmetric = symmetric ? 1 : 0;
    g.b_upper = b_upper ? 1 : 0;
    g.slices = kSlices;
    g.wait_ns = pipeline_wait_ns();
    g.status = status;
    g.C = tn_form ? nullptr : C;
    g.part = tn_form ? p.part : nullptr;
    int64_t pairs = 0;
    if (symmetric) {
        for (int tm = 0; tm < g.tilesM; tm++) {
            const int first = first_upper_tn(tm);
            if (first < g.tilesN) pairs += g.tilesN - first;
        }
    } else {
        pairs = (int64_t)g.tilesM * g.tilesN;
    }
    g.pairs = pairs;
    const int64_t total = pairs * g.splits * nbatch;
    if ((rc = launch_oz(g, tmA, total, s))) return rc;
    if (tn_form) {
        const dim3 grid((unsigned)((Nc + 255) / 256), (unsigned)std::min<int64_t>(M, 65535));
        oz_reduce_kernel<<<grid, 256, 0, s>>>(p.part, g.splits, g.Mp, g.Np, M, Nc, C, ldc, g.symmetric,
                                              subtract ? 1 : 0);
        CHFSI_LAUNCH_CHECK();
    }
    return CHFSI_OK;
}

// Block-diagonal product of the split layout: D slices (prepared once) and the slices
// of the multiplied block (prepared per product).
struct OzBlockDiag {
    OzOperand D, Y;
};

template <typename Ar>
void oz_blockdiag_layout(Ar& ar, int64_t N, int B, int64_t n, OzBlockDiag* out) {
    OzBlockDiag b;
    const int nblk = (int)((N + B - 1) / B);
    oz_operand_layout(ar, (int64_t)nblk * B, B, 1, kTileM, &b.D);   // rows of all blocks, K = B
    oz_operand_layout(ar, n, B, nblk, kTileN, &b.Y);                 // per block: n rows (Y columns), K = B
    if (out) *out = b;
}

// BSR filter step: digit planes of the chunks of H (made once per filter call) and of
// Y_cur^T (made per step; rows = states, K = grid points).  H is stored by block rows:
// of a row's blocks only the chunks of eight columns with a nonzero entry are kept, in
// order, [chunk][7][64 rows][8], from chunk brow_ptr[R] * 8 on; chunk[] names the chunk of
// Y_cur that each multiplies, count[] how many a row has (rounded up to a whole stage by
// zero chunks).  Every grid row has one scale over its whole block row, so that the
// products of all its chunks share it.
struct OzBsr {
    OzOperand Y;
    int* exps[2] = {nullptr, nullptr};   // exponents of Y_cur and of the step's output, alternating
    unsigned char* H = nullptr;
    int32_t *chunk = nullptr, *count = nullptr;
    int* expH = nullptr;      // per grid row
};

template <typename Ar>
void oz_bsr_layout(Ar& ar, int64_t nbr, int64_t nblocks, int64_t n, OzBsr* out) {
    OzBsr b;
    const size_t stored = (size_t)(nblocks > 0 ? nblocks : 1) * kBlockChunks;
    b.H = ar.template take<unsigned char>(stored * (kSlices * kPlaneB));
    b.chunk = ar.template take<int32_t>(stored);
    b.count = ar.template take<int32_t>((size_t)nbr);
    oz_operand_layout(ar, n, nbr * 64, 1, kTileM, &b.Y);
    b.exps[0] = b.Y.exps;
    b.exps[1] = ar.template take<int>((size_t)b.Y.padded_rows());
    b.expH = ar.template take<int>((size_t)(nbr * 64));
    if (out) *out = b;
}

// Exponents, chunk list and digit planes of one block row per CTA.  The first pass reads
// the row's blocks with a warp per grid row (512 contiguous bytes a load) for the row's
// largest exponent and the chunks' nonzero flags, the second makes the kept chunks'
// digits, a thread per grid row: bounded by reading H twice and writing 14 bytes an entry.
// A chunk whose entries are all zero (as on the faces of a block that the stencil does
// not reach) adds nothing to the product and is left out of it.
// The shift c goes into the digits of the diagonal (of H_ii - c as a two-float sum), so that
// the step's output need not read Y_cur again nor spend a third FP64 operation an element
// (8192 outputs an item at two operations a cycle) on it -- where, for every grid row of the
// block row, no scale grows and |H_ii - c| <= 2 |H_ii|, so that the rounding of Y_cur to 56
// (40) bits is multiplied by at most twice the diagonal that it meets without the shift
// (c within -1 .. 3 times the diagonal: all rows of the grid operators, whose errors against
// 64 bits fell with the fold); other block rows, and those without a stored diagonal
// block, are marked kUnfolded, and their shift is an FP64 multiply-add on Y_cur itself.
__global__ void __launch_bounds__(256) oz_bsr_prepare_kernel(const double* __restrict__ val,
                                                             const int32_t* __restrict__ brow_ptr,
                                                             const int32_t* __restrict__ bcol, int64_t nblocks,
                                                             double c, int* expH, int32_t* chunk, int32_t* count,
                                                             unsigned char* __restrict__ H, unsigned* status) {
    constexpr int kMaxChunks = kMaxItemKB * kStageChunks;
    __shared__ int rowmax[64];
    __shared__ unsigned char flag[kMaxChunks];
    __shared__ int16_t list[kMaxChunks + kStageChunks];
    __shared__ int kept, padded, larger;
    const int64_t R = blockIdx.x;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int qb, nq;
    bool bad_ptr = false, bad = false;
    bsr_row_range(brow_ptr, nblocks, R, qb, nq, bad_ptr);
    for (int p = threadIdx.x; p < nq * kBlockChunks; p += 256) flag[p] = 0;
    if (threadIdx.x == 0) larger = 0;
    __syncthreads();
    int qd = -1;        // the first diagonal block of the row
    int m[8] = {};      // largest exponent fields, without that block's diagonal
    for (int q = 0; q < nq; q++) {
        const bool diag = qd < 0 && bcol[qb + q] == (int)R;
        if (diag) qd = q;
        const double* blk = val + (int64_t)(qb + q) * 4096;
        bool any0 = false, any1 = false;
#pragma unroll
        for (int i = 0; i < 8; i++) {       // grid rows warp, warp + 8, ...
            const double* row = blk + (warp + 8 * i) * 64;
            const int e0 = (__double2hiint(row[lane]) >> 20) & 0x7ff;
            const int e1 = (__double2hiint(row[32 + lane]) >> 20) & 0x7ff;
            bad |= e0 == 0x7ff || e1 == 0x7ff;
            any0 |= e0 != 0;
            any1 |= e1 != 0;
            const int d = diag ? warp + 8 * i : -1;      // column of the diagonal entry
            if (lane != d && e0 > m[i]) m[i] = e0;
            if (32 + lane != d && e1 > m[i]) m[i] = e1;
        }
        const unsigned b0 = __ballot_sync(0xffffffffu, any0), b1 = __ballot_sync(0xffffffffu, any1);
        if (lane < kBlockChunks && (((lane < 4 ? b0 : b1) >> (8 * (lane & 3))) & 255u)) flag[q * kBlockChunks + lane] = 1;
    }
#pragma unroll
    for (int i = 0; i < 8; i++) {
        const int e = __reduce_max_sync(0xffffffffu, m[i]);
        if (lane == 0) rowmax[warp + 8 * i] = e;
    }
    __syncthreads();
    // H_ii of this thread's grid row, and its scale without and with the shift
    const int r = threadIdx.x & 63;
    const double hii = qd >= 0 ? val[(int64_t)(qb + qd) * 4096 + r * 65] : 0.0;
    const double sd = hii - c, back = sd + c, err = (hii - back) + ((back - sd) - c);   // hii - c = sd + err
    const int ed = (__double2hiint(hii) >> 20) & 0x7ff, es = (__double2hiint(sd) >> 20) & 0x7ff;
    const int em = rowmax[r];
    if (threadIdx.x < 64 && (!(fabs(sd) <= 2.0 * fabs(hii)) || es > (em > ed ? em : ed))) larger = 1;
    __syncthreads();
    const bool fold = qd >= 0 && c != 0.0 && !larger;
    const int efd = fold ? es : ed, efm = em > efd ? em : efd;
    if (fold && threadIdx.x < kBlockChunks) flag[qd * kBlockChunks + threadIdx.x] = 1;
    __syncthreads();
    if (warp == 0) {
        int k = 0;
        for (int c0 = 0; c0 < nq * kBlockChunks; c0 += 32) {
            const int p = c0 + lane;
            const bool f = p < nq * kBlockChunks && flag[p];
            const unsigned b = __ballot_sync(0xffffffffu, f);
            if (f) list[k + __popc(b & ((1u << lane) - 1))] = (int16_t)p;
            k += __popc(b);
        }
        const int up = (k + kStageChunks - 1) / kStageChunks * kStageChunks;   // at most nq * 8
        if (lane < up - k) list[k + lane] = -1;
        if (lane == 0) {
            kept = k;
            padded = up;
            count[R] = up | (fold || c == 0.0 ? 0 : kUnfolded);
        }
    }
    __syncthreads();
    const int64_t base = (int64_t)qb * kBlockChunks;
    if (threadIdx.x < 64) expH[R * 64 + r] = efm;
    for (int p = threadIdx.x >> 6; p < padded; p += 4) {
        const int l = p < kept ? list[p] : 0, blk = l / kBlockChunks, k0 = (l % kBlockChunks) * kChunk;
        double x[kChunk];
        const double* src = val + (int64_t)(qb + blk) * 4096 + r * 64 + k0;
#pragma unroll
        for (int k = 0; k < kChunk; k++) x[k] = p < kept ? src[k] : 0.0;
        long long F[kChunk];
#pragma unroll
        for (int k = 0; k < kChunk; k++) {
            F[k] = fixed_point(x[k], efm);
            if (fold && p < kept && blk == qd && k0 + k == r) F[k] = fixed_point(sd, efm) + fixed_point(err, efm);
        }
        uint4 dg[kSlices];
        digits8(F, dg);
        uint4* dst = reinterpret_cast<uint4*>(H) + (base + p) * (kSlices * 64) + r;
#pragma unroll
        for (int t = 0; t < kSlices; t++) dst[t * 64] = dg[t];
        if (r == 0) {
            const int C = p < kept ? bcol[qb + blk] : 0;
            const bool in = C >= 0 && C < (int64_t)gridDim.x;
            bad_ptr |= !in;
            chunk[base + p] = p < kept && in ? C * kBlockChunks + l % kBlockChunks : 0;   // always a valid chunk
        }
    }
    if (bad) raise_status(status, DEV_NONFINITE);
    if (bad_ptr) raise_status(status, DEV_PATTERN);
}

}  // namespace

size_t ozaki_bsr_bytes(int64_t nbr, int64_t nblocks, int64_t n) {
    CountAr ar;
    oz_bsr_layout(ar, nbr, nblocks, n, nullptr);
    return ar.s.used;
}

int ozaki_bsr_prepare(const BsrDev& h, int64_t n, double c, void* ws, size_t ws_bytes, unsigned* status, cudaStream_t s) {
    if (h.bdim != 64 || h.nbr <= 0) return CHFSI_ERR_UNSUPPORTED;
    if (ws_bytes < ozaki_bsr_bytes(h.nbr, h.nblocks, n)) return CHFSI_ERR_NOMEM;
    Arena ar(ws, ws_bytes);
    OzBsr b;
    oz_bsr_layout(ar, h.nbr, h.nblocks, n, &b);
    if (std::max<int64_t>(h.nblocks, 2) * 64 * kSlices > INT32_MAX || b.Y.padded_rows() * kSlices > INT32_MAX)
        return CHFSI_ERR_UNSUPPORTED;
    oz_bsr_prepare_kernel<<<(unsigned)h.nbr, 256, 0, s>>>(static_cast<const double*>(h.val), h.brow_ptr, h.bcol,
                                                          h.nblocks, c, b.expH, b.chunk, b.count, b.H, status);
    CHFSI_LAUNCH_CHECK();
    return CHFSI_OK;
}

int ozaki_bsr_step(const BsrDev& h, int64_t n, const double* Yc, int64_t ldc, const double* Yp, int64_t ldp,
                   double* Yo, int64_t ldo, double alpha, double c, double beta, void* ws, size_t ws_bytes,
                   unsigned* status, cudaStream_t s, int slices, int pass) {
    if (slices != 7 && slices != 5) return CHFSI_ERR_ARG;
    if (n <= 0 || h.nbr <= 0) return CHFSI_OK;
    if (ws_bytes < ozaki_bsr_bytes(h.nbr, h.nblocks, n)) return CHFSI_ERR_NOMEM;
    Arena ar(ws, ws_bytes);
    OzBsr b;
    oz_bsr_layout(ar, h.nbr, h.nblocks, n, &b);
    const int64_t N = h.nbr * 64;
    int rc;
    b.Y.exps = b.exps[pass & 1];
    int* next = b.exps[(pass + 1) & 1];
    if ((rc = oz_prepare(Yc, ldc, true, b.Y, N, 0, status, s, slices, pass > 0))) return rc;
    CHFSI_CUDA_TRY(cudaMemsetAsync(next, 0, sizeof(int) * (size_t)b.Y.padded_rows(), s));
    OzArgs g{};
    g.A = b.Y.slices;
    g.B = b.H;
    g.chunksA = b.Y.chunks;
    g.M = n;
    g.Nc = N;
    g.ldc = ldo;
    g.C = Yo;
    g.nbatch = 1;
    g.m_batch = n;
    g.tilesM = (int)((n + kTileM - 1) / kTileM);
    g.tilesN = (int)h.nbr;
    g.expA = b.Y.exps;
    g.kb_total = kMaxItemKB;
    g.kb_split = kMaxItemKB;
    g.splits = 1;
    g.pairs = (int64_t)g.tilesM * h.nbr;
    g.wait_ns = pipeline_wait_ns();
    g.status = status;
    g.bsr = 1;
    g.slices = slices;
    g.brow_ptr = h.brow_ptr;
    g.hchunk = b.chunk;
    g.hcount = b.count;
    g.nblocks = h.nblocks;
    g.expH = b.expH;
    g.Ycur = Yc;
    g.ldcur = ldc;
    g.Yprev = Yp;
    g.ldprev = ldp;
    g.alpha = alpha;
    g.cshift = c;
    g.beta = beta;
    g.expNext = next;
    return launch_oz(g, CUtensorMap{}, g.pairs, s);
}

size_t ozaki_workspace_bytes(bool tn_form, int64_t M, int64_t Nc, int64_t K, bool same) {
    CountAr ar;
    oz_layout(ar, tn_form, M, Nc, K, same, nullptr);
    return ar.s.used;
}

int ozaki_gemm_tn(const double* A, int64_t lda, const double* B, int64_t ldb, int64_t K, int64_t M, int64_t Nc,
                  double* C, int64_t ldc, bool symmetric, void* ws, size_t ws_bytes, unsigned* status,
                  cudaStream_t s, bool subtract) {
    if (M <= 0 || Nc <= 0) return CHFSI_OK;
    // the same operand twice (a Gram matrix) is sliced once; `symmetric` says that the
    // product is known to be symmetric (a Gram matrix, or X^T (H X) for symmetric H):
    // only the tiles on and above the diagonal are computed and the others mirrored
    const bool same = (A == B) && (lda == ldb) && (M == Nc);
    if (symmetric && M != Nc) return CHFSI_ERR_ARG;
    if (ws_bytes < ozaki_workspace_bytes(true, M, Nc, K, same)) return CHFSI_ERR_NOMEM;
    Arena ar(ws, ws_bytes);
    OzPlan p;
    oz_layout(ar, true, M, Nc, K, same, &p);
    int rc;
    if ((rc = oz_prepare(A, lda, true, p.A, K, 0, status, s))) return rc;
    if (!same && (rc = oz_prepare(B, ldb, true, p.B, K, 0, status, s))) return rc;
    return oz_run(p, true, C, ldc, M, Nc, symmetric, false, status, s, 1, 0, subtract);
}

int ozaki_gemm_nn(const double* A, int64_t lda, const double* B, int64_t ldb, int64_t M, int64_t K, int64_t Nc,
                  double* C, int64_t ldc, bool b_upper, void* ws, size_t ws_bytes, unsigned* status,
                  cudaStream_t s) {
    if (M <= 0 || Nc <= 0) return CHFSI_OK;
    if (ws_bytes < ozaki_workspace_bytes(false, M, Nc, K, false)) return CHFSI_ERR_NOMEM;
    Arena ar(ws, ws_bytes);
    OzPlan p;
    oz_layout(ar, false, M, Nc, K, false, &p);
    int rc;
    if ((rc = oz_prepare(A, lda, false, p.A, K, 0, status, s))) return rc;
    if ((rc = oz_prepare(B, ldb, true, p.B, K, 0, status, s))) return rc;   // B_hat = B^T: rows are B's columns
    return oz_run(p, false, C, ldc, M, Nc, false, b_upper, status, s);
}

size_t ozaki_blockdiag_bytes(int64_t N, int B, int64_t n) {
    CountAr ar;
    oz_blockdiag_layout(ar, N, B, n, nullptr);
    return ar.s.used;
}

int ozaki_blockdiag_prepare(const double* diag, int64_t N, int B, int64_t n, void* ws, size_t ws_bytes,
                            unsigned* status, cudaStream_t s) {
    if (B <= 0 || B % kTileM || B > kMaxItemKB * kKB) return CHFSI_ERR_UNSUPPORTED;
    if (ws_bytes < ozaki_blockdiag_bytes(N, B, n)) return CHFSI_ERR_NOMEM;
    Arena ar(ws, ws_bytes);
    OzBlockDiag bd;
    oz_blockdiag_layout(ar, N, B, n, &bd);
    // every block is B x B row-major, the blocks stacked: one direct operand of nblk * B rows
    return oz_prepare(diag, B, false, bd.D, B, 0, status, s);
}

int ozaki_blockdiag_apply(const double* Y, int64_t ldy, int64_t N, int B, int64_t n, double* T, int64_t ldt,
                          void* ws, size_t ws_bytes, unsigned* status, cudaStream_t s) {
    if (n <= 0 || N <= 0) return CHFSI_OK;
    if (B <= 0 || B % kTileM || B > kMaxItemKB * kKB) return CHFSI_ERR_UNSUPPORTED;
    if (ws_bytes < ozaki_blockdiag_bytes(N, B, n)) return CHFSI_ERR_NOMEM;
    Arena ar(ws, ws_bytes);
    OzBlockDiag bd;
    oz_blockdiag_layout(ar, N, B, n, &bd);
    // Y_hat of block k = (rows kB .. kB + B - 1 of Y)^T: n rows, K = B (the last block clipped at N)
    int rc;
    if ((rc = oz_prepare(Y, ldy, true, bd.Y, N, (int64_t)B * ldy, status, s))) return rc;
    OzPlan p;
    p.A = bd.D;
    p.A.nbatch = bd.Y.nbatch;
    p.A.tiles = B / kTileM;      // row tiles per batch in the stacked D operand
    p.B = bd.Y;
    return oz_run(p, false, T, ldt, N, n, false, false, status, s, bd.Y.nbatch, B);
}

}  // namespace chfsi

// ------------------------------------------------------------------ C ABI

namespace {

int oz_abi_check(int32_t op, int64_t M, int64_t Nc, int64_t K, int32_t flags) {
    if (op != CHFSI_OP_TN && op != CHFSI_OP_NN) return CHFSI_ERR_ARG;
    if (M < 0 || Nc < 0 || K < 0) return CHFSI_ERR_ARG;
    if (flags & ~(CHFSI_GEMM_SYMMETRIC | CHFSI_GEMM_B_UPPER)) return CHFSI_ERR_ARG;
    if ((flags & CHFSI_GEMM_SYMMETRIC) && (op != CHFSI_OP_TN || M != Nc)) return CHFSI_ERR_ARG;
    if ((flags & CHFSI_GEMM_B_UPPER) && op != CHFSI_OP_NN) return CHFSI_ERR_ARG;
    if (K > ((int64_t)1 << 21) || M > INT32_MAX / 8 || Nc > INT32_MAX / 8) return CHFSI_ERR_UNSUPPORTED;
    if (op == CHFSI_OP_NN && K > 8192) return CHFSI_ERR_UNSUPPORTED;
    return CHFSI_OK;
}

}  // namespace

int chfsi_ozaki_gemm_workspace_size(int32_t op, int64_t M, int64_t Nc, int64_t K, int32_t flags, size_t* bytes) {
    if (!bytes) return CHFSI_ERR_ARG;
    const int rc = oz_abi_check(op, M, Nc, K, flags);
    if (rc) return rc;
    // the tn form with one operand twice is smaller; size for two distinct operands
    *bytes = chfsi::align_up(chfsi::kStatusBytes) + chfsi::ozaki_workspace_bytes(op == CHFSI_OP_TN, M, Nc, K, false);
    return CHFSI_OK;
}

int chfsi_ozaki_gemm(int32_t op, const double* A, int64_t lda, const double* B, int64_t ldb, double* C, int64_t ldc,
                     int64_t M, int64_t Nc, int64_t K, int32_t flags, void* ws, size_t ws_bytes, void* stream) {
    int rc = oz_abi_check(op, M, Nc, K, flags);
    if (rc) return rc;
    if (M == 0 || Nc == 0) return CHFSI_OK;
    if (!C || ldc < Nc || (reinterpret_cast<uintptr_t>(C) & 7u)) return CHFSI_ERR_ARG;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (K == 0) {
        for (int64_t i = 0; i < M; i++)
            CHFSI_CUDA_TRY(cudaMemsetAsync(C + i * ldc, 0, sizeof(double) * (size_t)Nc, s));
        return CHFSI_OK;
    }
    if (!A || !B || (reinterpret_cast<uintptr_t>(A) & 7u) || (reinterpret_cast<uintptr_t>(B) & 7u)) return CHFSI_ERR_ARG;
    const bool tn = op == CHFSI_OP_TN;
    if (tn ? (lda < M || ldb < Nc) : (lda < K || ldb < Nc)) return CHFSI_ERR_ARG;
    size_t need = 0;
    if ((rc = chfsi_ozaki_gemm_workspace_size(op, M, Nc, K, flags, &need))) return rc;
    if (!ws || (reinterpret_cast<uintptr_t>(ws) & 255u) || ws_bytes < need) return ws ? CHFSI_ERR_NOMEM : CHFSI_ERR_ARG;
    unsigned* st = chfsi::status_word(ws);
    CHFSI_CUDA_TRY(cudaMemsetAsync(st, 0, sizeof(unsigned), s));
    char* rest = static_cast<char*>(ws) + chfsi::align_up(chfsi::kStatusBytes);
    const size_t rest_bytes = ws_bytes - chfsi::align_up(chfsi::kStatusBytes);
    if (tn)
        return chfsi::ozaki_gemm_tn(A, lda, B, ldb, K, M, Nc, C, ldc, (flags & CHFSI_GEMM_SYMMETRIC) != 0, rest,
                                    rest_bytes, st, s);
    return chfsi::ozaki_gemm_nn(A, lda, B, ldb, M, K, Nc, C, ldc, (flags & CHFSI_GEMM_B_UPPER) != 0, rest,
                                rest_bytes, st, s);
}
