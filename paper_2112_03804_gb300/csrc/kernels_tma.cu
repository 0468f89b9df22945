// Kronecker-form payoff products, TMA-staged (sm_103a): single game, FP32,
// BF16 or FP16 storage, FP32 arithmetic.
//
// Mathematics (Prop. 1, Sec. 3; the fold block is the card-removal
// compatibility of Sec. 4's eq. for C, the showdown block the strength sign
// times compatibility, whose inverse-D prefix sums are Technique B's):
//   out / lambda_out = K_F(w) + S (2 Lo(b) + TieC(b)),
//   a = lambda_in * y_f,  b = lambda_in * y_s,  w = F a - S b,
// with y_f / y_s the input rows of the output sequence's fold and showdown
// terminals (payoffs F and S), K_F(w)[h] = Tot - P[c1] - P[c2] + w[h]
// (P[c] the per-card totals; one-card hands: Tot - P[c1]), Lo the
// compatible strictly weaker mass and TieC the compatible tied mass.
//
// Ties without tie-aligned tiles.  The scan walks hands in library order
// (strength, then canonical index) and accumulates the compatible mass of
// every hand *before* the current one, Lo_ord.  With TB / TA the compatible
// tied mass before / after a hand in that order, Lo = Lo_ord - TB and
// TieC = TB + TA, so
//   2 Lo + TieC = 2 Lo_ord - TB + TA.
// Every tie group has at most 4 hands (the host checks it): a hand's tied
// partners are at most 3 positions away, and the two corrections are made in
// registers (the current 16-hand box and the previous one are held there).
//
// Organisation.  A CTA = one item (an output sequence, or two that share one
// input row, see below) and 32 consecutive vectors (lane j = vector b0 + j):
// all its columns share their input rows, payoffs and column kind (fold only,
// showdown only, both).  Four warps scan
// four chunks of the hand order (chunk boundaries at 16-hand boxes that cut
// no tie group).  For each box one lane issues cp.async.bulk.tensor copies
// of the box's [32 vectors][16 hands] from each input row into a 64-byte
// swizzled slot of the warp's ring (an mbarrier per slot); lanes read their
// row four hands at a time (conflict free under the swizzle).  Per-card sums
// live in shared memory [card][lane] (float2: mass of b for Lo, total of w
// for K_F), addressed by per-hand byte offsets from the box's hand records
// (copied by cp.async.bulk with the box into a record ring).  Two hands per
// step: all four per-card loads are issued together; when the second hand
// holds a card of the first, its loaded sums get the first hand's update in
// registers; the two hands' arithmetic (and the two halves of a float2 sum)
// runs as packed FP32x2 instructions.  Partial results stay on chip: the
// first 16 boxes of a chunk in tensor memory (lane = column, a column per
// hand, one tcgen05.st per box), later boxes in shared memory.  After a
// barrier the four chunks' per-card sums are combined into
// -Q[c] = -(Pall[c] + 2 S R_before[c]) at the start of each warp's ring, and
// each warp finishes its boxes: out = lambda_out ((partial + C) - (Q[c1] +
// Q[c2])) with C = Tot + 2 S G_before, the finishing records read from the
// record ring (copied one box ahead by cp.async), written into a swizzled
// box and stored with one cp.async.bulk.tensor per box.  No atomics:
// results are bit-reproducible.
//
// Pairs.  Where a player answers a bet by folding or calling, the two answers
// are output sequences with the same input row y (the bet's): with b = lambda_in
// y and one scan of b,
//   out_call / lambda_out = S (2 Lo(b) + TieC(b) - K_F(b)),
//   out_fold / lambda_out = F K_F(b),
// so one item makes both: its finishing pass also gathers the totals P[c] (a
// second table, in the idle half of warp 0's per-card table) and reads the
// row's boxes once more (L2) for the b[h] of K_F.  A third of a game's items
// go (43 sequences of the 1081-hand river game: 29 items), with their scans
// and table traffic: 1024 FP32 vectors 134 -> 124 us, 250 vectors of the
// 247-sequence tree 185 -> 168 us (single against paired items, same build;
// 121 and 163 us since the finishing pass counts its staging slots).
//
// 16-bit storage (1000 BF16 vectors of the river game: 284 us on the
// tensor-memory kernel, 118 us here) differs in the boxes alone.  Both storage
// types are bound by the scan's and the finishing pass's short dependent
// steps at eight resident warps per SM, not by memory (floor 55 / 27 us).
//
// Waits are bounded: a wait that gives up sets *err; the warp scans no
// further box and finishes nothing, the CTA runs to its end without waiting
// again (its results are not valid), waits (bounded) for its copies still in
// flight and frees its tensor memory.
#include "kernels.h"
#include "game.h"
#include "scan_records.h"

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstdlib>
#include <cstring>
#include <mutex>
#include <new>
#include <string>
#include <vector>

namespace kps {

constexpr int kTmaMaxExtra = 2;    // boxes of a chunk past the 256 tensor-memory columns
constexpr int kMaxNw = 8;          // warps (chunks) of a CTA: 4, or 8 for few CTAs

// An item, with all that a CTA needs to begin: one load instead of a chain of
// two (128 FP32 vectors of the river game, 172 CTAs).
struct alignas(32) TmaItem {
    int sigma, sigma2;             // output sequence, and the fold-only sequence of its pair or -1
    int rf, rs;                    // its fold / showdown input sequence or -1
    float F, S, F2;                // their payoffs (0 without), the pair's fold payoff
    int pad;
};

// Kernel arguments (__grid_constant__).
struct alignas(128) TmaArgs {
    CUtensorMap tin;               // input  [batch][n_in][H], box 16 x 1 x 32, rows of a box swizzled (64 or 32 bytes)
    CUtensorMap tout;              // output [batch][n_out][hs] fp32, same box
    int H, hs, nc, k, n_out, n_in, batch, nbb, nbox, extra;
    int stall_test;                // test hook: warp 0's first box expects 16 bytes that never come
    int bchunk[kMaxNw + 1];        // warp k scans boxes [bchunk[k], bchunk[k+1])
    int nitems;
    const TmaItem *items;
    const unsigned char *rscan;    // [nbox][kScanBlock]
    const TmaFinRec *rfin;         // [nbox * 8]
    unsigned int *err;             // set to 1 when a wait gives up
};

// Host side of one direction: the arguments and the record tables.
struct TmaParams {
    TmaArgs a;
    void *dev = nullptr;           // device copy of the records (scan blocks, then finishing records)
    std::vector<unsigned char> host;   // records, the paired items, the single ones
    size_t o_items = 0;
    int npaired = 0, nsingle = 0;
    int chunk4[5] = {}, chunk8[kMaxNw + 1] = {};
    bool eight = false;            // the eight-warp shape fits
    bool alone = false;            // one CTA of the four-warp shape fills an SM
    int extra4 = 0;                // overflow boxes of the four-warp shape
    int sms = 1;                   // of the device
    int device = -1;
};

namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kRingBytes = 12288;          // per warp: 3 slots of 4 KB or 6 of 2 KB (half of it for 16-bit storage)
constexpr int kFewBoxes = 4;               // boxes up to which eight warps only add to the fixed part
constexpr int kSmallBoxes = 24;            // boxes up to which an item is mostly fixed part (kSmall)
constexpr int kPairMinCards = 48;          // per-card rows from which half a table holds three FP32 boxes
constexpr int kRecRing = 6 * kScanBlock;   // per warp: one scan block per slot
constexpr int kTmemCols = 256;             // per four warps (two CTAs of four or one of eight per SM)
constexpr unsigned long long kWaitNs = 2000000000ull;   // give up after 2 s

enum Kind { kKindF = 1, kKindS = 2, kKindFS = 3 };
// What a launch's items are: single sequences, pairs (four warps), or single
// sequences of a game of few boxes.  Each runs a kernel without the code of the
// others.
enum Form { kSingle, kPaired, kSmall };

// Shared memory (from a 1 KB aligned base) with nw warps: the warps' rings,
// their per-card tables (nc rows of 256 bytes), their overflow boxes of partial
// results, their record rings, then the header (tensor-memory slot at +0,
// nw x 8 mbarriers at +16, per-warp sums [2][nw][32] floats after them).
__host__ __device__ inline size_t ring_off(int w) { return (size_t)w * kRingBytes; }
__host__ __device__ inline size_t state_off(int nw, int w, int nc) { return (size_t)nw * kRingBytes + (size_t)w * nc * 256; }
__host__ __device__ inline size_t extra_off(int nw, int w, int nc, int extra) {
    return state_off(nw, nw, nc) + (size_t)w * extra * kTmaBox * 32 * 4;
}
__host__ __device__ inline size_t rec_off(int nw, int w, int nc, int extra) {
    return extra_off(nw, nw, nc, extra) + (size_t)w * kRecRing;
}
__host__ __device__ inline size_t hdr_off(int nw, int nc, int extra) { return rec_off(nw, nw, nc, extra); }
__host__ __device__ constexpr int sums_at(int nw) { return 16 + 64 * nw; }
__host__ __device__ constexpr int hdr_bytes(int nw) { return sums_at(nw) + 256 * nw; }

// ---- PTX wrappers ------------------------------------------------------------
__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count));
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}
__device__ __forceinline__ unsigned long long gtime() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}
// Bounded wait for phase `parity` of a barrier; false when it gave up.
__device__ __noinline__ bool mbar_wait(uint32_t bar, uint32_t parity) {
    if (mbar_try(bar, parity)) return true;
    const unsigned long long t0 = gtime();
    for (int i = 0; i < (1 << 26); ++i) {
        if (mbar_try(bar, parity)) return true;
        if ((i & 63) == 63 && gtime() - t0 > kWaitNs) break;
    }
    return false;
}
__device__ __forceinline__ void fence_barrier_init() {
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void fence_proxy_async() {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
__device__ __forceinline__ void tma_load3(uint32_t dst, const CUtensorMap *map, int x, int y, int z, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], "
        "[%5];" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(z), "r"(bar)
        : "memory");
}
__device__ __forceinline__ void bulk_load(uint32_t dst, const void *src, uint32_t bytes, uint32_t bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
                 "l"(reinterpret_cast<uint64_t>(src)), "r"(bytes), "r"(bar)
                 : "memory");
}
// 16-byte copy global -> shared by this thread (cp.async, L2 only)
__device__ __forceinline__ void cp16(uint32_t dst, const void *src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}
__device__ __forceinline__ void tma_store3(const CUtensorMap *map, int x, int y, int z, uint32_t src) {
    asm volatile("cp.async.bulk.tensor.3d.global.shared::cta.tile.bulk_group [%0, {%1, %2, %3}], [%4];" ::"l"(
                     reinterpret_cast<uint64_t>(map)),
                 "r"(x), "r"(y), "r"(z), "r"(src)
                 : "memory");
}
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void bulk_wait_read() {
    asm volatile("cp.async.bulk.wait_group.read %0;" ::"n"(N) : "memory");
}
// the same with a run-time count of at most 5 groups still reading
__device__ __forceinline__ void bulk_wait_read_n(int n) {
    if (n <= 0) bulk_wait_read<0>();
    else if (n == 1) bulk_wait_read<1>();
    else if (n == 2) bulk_wait_read<2>();
    else if (n == 3) bulk_wait_read<3>();
    else if (n == 4) bulk_wait_read<4>();
    else bulk_wait_read<5>();
}

__device__ __forceinline__ void tm_alloc(uint32_t dst_smem, uint32_t ncols) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(dst_smem), "r"(ncols));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
}
__device__ __forceinline__ void tm_dealloc(uint32_t taddr, uint32_t ncols) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols));
}
__device__ __forceinline__ void tm_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tm_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tm_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tm_st16(uint32_t taddr, const float *r) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};" ::"r"(
            taddr),
        "f"(r[0]), "f"(r[1]), "f"(r[2]), "f"(r[3]), "f"(r[4]), "f"(r[5]), "f"(r[6]), "f"(r[7]), "f"(r[8]), "f"(r[9]),
        "f"(r[10]), "f"(r[11]), "f"(r[12]), "f"(r[13]), "f"(r[14]), "f"(r[15])
        : "memory");
}
__device__ __forceinline__ void tm_ld16(uint32_t taddr, float *r) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=f"(r[0]), "=f"(r[1]), "=f"(r[2]), "=f"(r[3]), "=f"(r[4]), "=f"(r[5]), "=f"(r[6]), "=f"(r[7]), "=f"(r[8]),
          "=f"(r[9]), "=f"(r[10]), "=f"(r[11]), "=f"(r[12]), "=f"(r[13]), "=f"(r[14]), "=f"(r[15])
        : "r"(taddr)
        : "memory");
}
// waits for this thread's tensor-memory loads; names the 16 destination
// registers so that no use of them is scheduled before the data arrive
__device__ __forceinline__ void tm_wait_ld16(float *r) {
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+f"(r[0]), "+f"(r[1]), "+f"(r[2]), "+f"(r[3]), "+f"(r[4]), "+f"(r[5]), "+f"(r[6]), "+f"(r[7]),
                   "+f"(r[8]), "+f"(r[9]), "+f"(r[10]), "+f"(r[11]), "+f"(r[12]), "+f"(r[13]), "+f"(r[14]), "+f"(r[15])::"memory");
}

// Packed FP32x2 arithmetic (each component rounded to nearest, as the
// scalar instruction would be).
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }

// A box of [32 vectors][16 hands] in shared memory: rows of 64 (FP32) or 32
// bytes, their 16-byte chunks swizzled by the copy (chunk bits XORed with the
// row's: address bits 4-5 with 7-8, or bit 4 with bit 7), so that the lanes'
// accesses of one chunk are conflict free.
template <typename T> struct Box;
template <> struct Box<float> {
    static constexpr int kBytes = 2048;
    __device__ static uint32_t at(int row, int q) { return (uint32_t)(row * 64 + ((q ^ ((row >> 1) & 3)) << 4)); }
    // lane's 16 values as hand pairs (2i, 2i + 1)
    __device__ static void load(const unsigned char *slot, int lane, float2 *y) {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const float4 v = *reinterpret_cast<const float4 *>(slot + at(lane, q));
            y[2 * q] = make_float2(v.x, v.y);
            y[2 * q + 1] = make_float2(v.z, v.w);
        }
    }
    __device__ static void store(unsigned char *slot, int lane, const float2 *o) {
#pragma unroll
        for (int q = 0; q < 4; ++q)
            *reinterpret_cast<float4 *>(slot + at(lane, q)) =
                make_float4(o[2 * q].x, o[2 * q].y, o[2 * q + 1].x, o[2 * q + 1].y);
    }
};
__device__ __forceinline__ float2 widen(uint32_t w, __nv_bfloat16) {
    return make_float2(__uint_as_float(w << 16), __uint_as_float(w & 0xffff0000u));
}
__device__ __forceinline__ float2 widen(uint32_t w, __half) {
    return __half22float2(*reinterpret_cast<const __half2 *>(&w));
}
__device__ __forceinline__ uint32_t narrow(float2 v, __nv_bfloat16) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(v.x, v.y);
    return *reinterpret_cast<const uint32_t *>(&h);
}
__device__ __forceinline__ uint32_t narrow(float2 v, __half) {
    const __half2 h = __floats2half2_rn(v.x, v.y);
    return *reinterpret_cast<const uint32_t *>(&h);
}
template <typename T> struct Box {
    static constexpr int kBytes = 1024;
    __device__ static uint32_t at(int row, int q) { return (uint32_t)(row * 32 + ((q ^ ((row >> 2) & 1)) << 4)); }
    __device__ static void load(const unsigned char *slot, int lane, float2 *y) {
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const uint4 v = *reinterpret_cast<const uint4 *>(slot + at(lane, q));
            y[4 * q] = widen(v.x, T());
            y[4 * q + 1] = widen(v.y, T());
            y[4 * q + 2] = widen(v.z, T());
            y[4 * q + 3] = widen(v.w, T());
        }
    }
    __device__ static void store(unsigned char *slot, int lane, const float2 *o) {
#pragma unroll
        for (int q = 0; q < 2; ++q)
            *reinterpret_cast<uint4 *>(slot + at(lane, q)) =
                make_uint4(narrow(o[4 * q], T()), narrow(o[4 * q + 1], T()), narrow(o[4 * q + 2], T()),
                           narrow(o[4 * q + 3], T()));
    }
};

// The CTA's column set, its warp's chunk and its shared-memory regions.
struct Ctx {
    unsigned char *sm;
    int lane, warp;
    int bb, sigma, rf, rs;
    int sigma2;                // fold-only sequence of a pair, or -1
    float F, S;                // a pair's F: sigma2's
    int b0, nb;                // first box of the chunk, boxes in it
    uint32_t tmem;             // the warp's tensor-memory lanes, column 0
    bool ok;                   // no wait gave up
};

// Scan and combination of one column kind; returns this warp's C.  A
// showdown-only column is scanned with S = 1 (finishing multiplies by S), but in
// small games with its own.
template <typename T, int KIND, int K2, int NW, Form FORM>
__device__ __forceinline__ float tma_scan(const TmaArgs &P, Ctx &c) {
    constexpr bool HF = (KIND & kKindF) != 0, HS = (KIND & kKindS) != 0, FS = KIND == kKindFS;
    constexpr int NS = FS ? 3 : 6;                    // ring slots
    constexpr int BB = Box<T>::kBytes, SLOT = FS ? 2 * BB : BB;   // bytes per box, per slot
    const int lane = c.lane, warp = c.warp, nc = P.nc;
    unsigned char *ring = c.sm + ring_off(warp);
    const uint32_t ring_s = smem_u32(ring);
    unsigned char *hdr = c.sm + hdr_off(NW, nc, P.extra);
    const uint32_t bar0 = smem_u32(hdr + 16) + 8u * 8u * (uint32_t)warp;
    unsigned char *rring = c.sm + rec_off(NW, warp, nc, P.extra);
    const uint32_t rring_s = smem_u32(rring);
    // per-card table of the chunk, [card][lane]: float2 {b mass, w total}
    // for columns of both kinds (rows of 256 bytes, row offset 2 * off),
    // one float otherwise (rows of 128 bytes, offset off)
    unsigned char *stb = c.sm + state_off(NW, warp, nc);
    unsigned char *lb = stb + (FS ? 8 : 4) * lane;
    float *xpart = reinterpret_cast<float *>(c.sm + extra_off(NW, warp, nc, P.extra));
    float *sums = reinterpret_cast<float *>(hdr + sums_at(NW));
    const float F = c.F, S = FS || FORM == kSmall ? c.S : 1.f, S2 = 2.f * S;
    const int nb = c.nb;
    const int z0 = 32 * c.bb;
    auto row = [&](uint32_t off) -> unsigned char * { return lb + (FS ? 2 * off : off); };

    for (int q = lane; q < nc * (FS ? 64 : 32); q += 32) reinterpret_cast<float *>(stb)[q] = 0.f;

    auto issue = [&](int m) {
        const int sl = m % NS;
        const uint32_t bar = bar0 + 8u * (uint32_t)sl;
        const uint32_t dst = ring_s + (uint32_t)(sl * SLOT);
        const int x = kTmaBox * (c.b0 + m);
        mbar_expect_tx(bar, (uint32_t)(SLOT + kScanBlock) + (P.stall_test && m == 0 && warp == 0 ? 16u : 0u));
        if (HF) tma_load3(dst, &P.tin, x, c.rf, z0, bar);
        if (HS) tma_load3(dst + (HF ? (uint32_t)BB : 0u), &P.tin, x, c.rs, z0, bar);
        bulk_load(rring_s + (uint32_t)(sl * kScanBlock), P.rscan + (size_t)(c.b0 + m) * kScanBlock, kScanBlock, bar);
    };
    if (lane == 0) {
        for (int sl = 0; sl < NS; ++sl) mbar_init(bar0 + 8u * (uint32_t)sl, 1);
        fence_barrier_init();
        for (int m = 0; m < NS && m < nb; ++m) issue(m);
    }
    __syncwarp();
    int nissued = min(NS, nb), nwaited = 0;   // boxes copied in / waited for (warp-uniform)

    // ---- scan (lane = column)
    float G2 = 0.f;               // twice the b mass before the current hand
    float2 pp[8];                 // the previous box's partial results (stored one box late)
    float bq1 = 0.f, bq2 = 0.f, bq3 = 0.f;   // b of the previous box's hands 15, 14, 13
    const float2 F2 = make_float2(F, F), S2v = make_float2(S, S), nS2 = make_float2(-S, -S);
#pragma unroll
    for (int k = 0; k < 8; ++k) pp[k] = make_float2(0.f, 0.f);
    auto store_box = [&](int m, const float2 *r) {
        if (m < 16) {
            tm_st16(c.tmem + (uint32_t)(16 * m), reinterpret_cast<const float *>(r));
        } else {
            float *xp = xpart + (m - 16) * (kTmaBox * 32);
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                xp[(2 * k) * 32 + lane] = r[k].x;
                xp[(2 * k + 1) * 32 + lane] = r[k].y;
            }
        }
    };
    for (int m = 0; m < nb; ++m) {
        const int sl = m % NS;
        if (c.ok) {
            // the first try inline (the box is usually there), then the
            // bounded loop
            const uint32_t bar = bar0 + 8u * (uint32_t)sl, par = (uint32_t)((m / NS) & 1);
            const bool got = mbar_try(bar, par) || mbar_wait(bar, par);
            c.ok = __all_sync(kFull, got);
            if (c.ok) nwaited = m + 1;
        }
        // after a wait gave up, the slot's records (shared-memory offsets)
        // may never have arrived: scan no further
        if (!c.ok) break;
        const unsigned char *slot = ring + sl * SLOT;
        // the box's inputs as hand pairs (2i, 2i+1)
        float2 yf[8], ys[8];
        if (HF) Box<T>::load(slot, lane, yf);
        if (HS) Box<T>::load(slot + (HF ? BB : 0), lane, ys);
        // the box's records: the next pair's are read before this pair's
        // per-card stores (program order keeps them ahead)
        const unsigned char *rs = rring + sl * kScanBlock;
        const uint32_t tw0 = reinterpret_cast<const uint32_t *>(rs + 256)[0];
        const uint32_t tw1 = reinterpret_cast<const uint32_t *>(rs + 256)[1];
        TmaScanRec rn = *reinterpret_cast<const TmaScanRec *>(rs);
        // two hands per step; the arithmetic of the two hands (or of the two
        // halves of a per-card float2) runs as packed FP32x2 instructions,
        // each component rounded as the scalar operation would be
        float2 p[8], bv[8];
#pragma unroll
        for (int i = 0; i < 16; i += 2) {
            const int k = i / 2;
            const TmaScanRec r = rn;
            if (i + 2 < 16) rn = reinterpret_cast<const TmaScanRec *>(rs)[k + 1];
            unsigned char *A1 = row(r.oa1), *A2 = row(r.oa2), *B1 = row(r.ob1), *B2 = row(r.ob2);
            const float2 lin = make_float2(r.lin1, r.lin2);
            // the two hands' inputs: a (fold side), b (showdown side), w
            const float2 bb = HS ? mul2(lin, ys[k]) : make_float2(0.f, 0.f);
            bv[k] = bb;
            float2 ww;
            if (FS) ww = fma2(F2, mul2(lin, yf[k]), mul2(nS2, bb));   // F a - S b
            else if (HF) ww = mul2(F2, mul2(lin, yf[k]));
            else ww = make_float2(0.f, 0.f);   // a showdown-only column tracks b alone
            float cs1, cs2;   // b mass of the hands' cards before them
            if (FS) {
                // per-card rows {b mass, w total}
                float2 sa1 = *reinterpret_cast<const float2 *>(A1);
                float2 sa2 = *reinterpret_cast<const float2 *>(A2);
                float2 sb1 = make_float2(0.f, 0.f), sb2 = make_float2(0.f, 0.f);
                if (K2 == 2) {
                    sb1 = *reinterpret_cast<const float2 *>(B1);
                    sb2 = *reinterpret_cast<const float2 *>(B2);
                }
                const float2 h1 = make_float2(bb.x, ww.x), h2 = make_float2(bb.y, ww.y);
                // the first hand's update, seen by the second hand's sums
                // when they share a card (ma, mb are 0 or 1)
                sa2 = fma2(make_float2(r.ma, r.ma), h1, sa2);
                if (K2 == 2) sb2 = fma2(make_float2(r.mb, r.mb), h1, sb2);
                cs1 = sa1.x + sb1.x;
                cs2 = sa2.x + sb2.x;
                *reinterpret_cast<float2 *>(A1) = add2(sa1, h1);
                if (K2 == 2) *reinterpret_cast<float2 *>(B1) = add2(sb1, h1);
                *reinterpret_cast<float2 *>(A2) = add2(sa2, h2);
                if (K2 == 2) *reinterpret_cast<float2 *>(B2) = add2(sb2, h2);
            } else {
                // one float per card: {first card, second card} of each hand
                float2 s1 = make_float2(*reinterpret_cast<const float *>(A1), 0.f);
                float2 s2 = make_float2(*reinterpret_cast<const float *>(A2), 0.f);
                if (K2 == 2) {
                    s1.y = *reinterpret_cast<const float *>(B1);
                    s2.y = *reinterpret_cast<const float *>(B2);
                }
                const float d1 = HS ? bb.x : ww.x, d2 = HS ? bb.y : ww.y;
                s2 = fma2(make_float2(r.ma, r.mb), make_float2(d1, d1), s2);
                cs1 = s1.x + s1.y;
                cs2 = s2.x + s2.y;
                const float2 u1 = add2(s1, make_float2(d1, d1)), u2 = add2(s2, make_float2(d2, d2));
                *reinterpret_cast<float *>(A1) = u1.x;
                if (K2 == 2) *reinterpret_cast<float *>(B1) = u1.y;
                *reinterpret_cast<float *>(A2) = u2.x;
                if (K2 == 2) *reinterpret_cast<float *>(B2) = u2.y;
            }
            if (HS) {
                // t = 2 Lo_ord - TB (b units), from the running 2G;
                // partial = w + S t, the w only for two-card hands (see K_F)
                const float gA = G2, gB = fmaf(2.f, bb.x, G2);
                G2 = fmaf(2.f, bb.y, gB);
                const float2 t = fma2(make_float2(-2.f, -2.f), make_float2(cs1, cs2), make_float2(gA, gB));
                if (HF) p[k] = fma2(S2v, t, K2 == 2 ? ww : make_float2(0.f, 0.f));
                else if (FORM == kSmall) p[k] = K2 == 2 ? fma2(S2v, t, mul2(nS2, bb)) : mul2(S2v, t);
                else p[k] = K2 == 2 ? fma2(nS2, bb, t) : t;   // showdown only: S = 1, w = -b
            } else {
                p[k] = K2 == 2 ? ww : make_float2(0.f, 0.f);
            }
        }
        // tie corrections of the box (partial = w + S (2 Lo_ord - TB + TA)):
        // TB leaves each tied hand's partial, TA enters the earlier
        // partner's; partners before the box are the previous box's last
        // three hands (their partials are stored one box late)
        if (HS && (tw0 | tw1)) {
            auto hb = [&](int j) -> float { return (j & 1) ? bv[j >> 1].y : bv[j >> 1].x; };
            auto bat = [&](int j) { return j >= 0 ? hb(j) : (j == -1 ? bq1 : j == -2 ? bq2 : bq3); };
            auto pat = [&](int j) -> float & {
                float2 &v = j >= 0 ? p[j >> 1] : pp[(16 + j) >> 1];
                return (j & 1) ? v.y : v.x;
            };
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const uint32_t tb = ((k < 4 ? tw0 : tw1) >> (8 * (k & 3))) & 0xfcu;
                if (tb) {
                    const int i = 2 * k;
#pragma unroll
                    for (int d = 1; d <= 3; ++d)
                        if (tb & (1u << (1 + d))) {
                            p[k].x = fmaf(-S, bat(i - d), p[k].x);
                            pat(i - d) = fmaf(S, bv[k].x, pat(i - d));
                        }
#pragma unroll
                    for (int d = 1; d <= 3; ++d)
                        if (tb & (1u << (4 + d))) {
                            p[k].y = fmaf(-S, bat(i + 1 - d), p[k].y);
                            pat(i + 1 - d) = fmaf(S, bv[k].y, pat(i + 1 - d));
                        }
                }
            }
        }
        // every lane has used the slot's values: refill it
        __syncwarp();
        if (c.ok && m + NS < nb) {
            if (lane == 0) {
                fence_proxy_async();
                issue(m + NS);
            }
            nissued = m + NS + 1;
        }
        if (m > 0) store_box(m - 1, pp);
#pragma unroll
        for (int k = 0; k < 8; ++k) pp[k] = p[k];
        bq1 = bv[7].y;
        bq2 = bv[7].x;
        bq3 = bv[6].y;
    }
    if (nb > 0) store_box(nb - 1, pp);
    tm_wait_st();
    if (!c.ok && lane == 0) {
        // a wait gave up: wait (bounded) for the copies still in flight
        // before the ring is reused or the CTA exits
        for (int m = nwaited; m < nissued; ++m)
            if (!mbar_wait(bar0 + 8u * (uint32_t)(m % NS), (uint32_t)((m / NS) & 1))) break;
    }
    __syncwarp();

    // per-warp totals: G (b mass) and Tot (w total; K_F's Tot)
    float tot = 0.f;
    if (HF) {
        for (int q = 0; q < nc; ++q)
            tot += FS ? reinterpret_cast<const float2 *>(stb)[q * 32 + lane].y
                      : reinterpret_cast<const float *>(stb)[q * 32 + lane];
        if (K2 == 2) tot *= 0.5f;
    } else {
        tot = -S * (0.5f * G2);
    }
    sums[(0 * NW + warp) * 32 + lane] = 0.5f * G2;
    sums[(1 * NW + warp) * 32 + lane] = tot;
    __syncthreads();

    // ---- combination: -Q_k[c] with Q_k[c] = Pall[c] + 2 S (mass of card c
    // in chunks < k), [card][lane] floats at the start of warp k's ring (free
    // now: every copy in has been consumed)
    for (int q = warp; q < nc; q += NW) {
        float rr[NW], pw[NW];
#pragma unroll
        for (int k = 0; k < NW; ++k) {
            const unsigned char *sk = c.sm + state_off(NW, k, nc);
            if (FS) {
                const float2 v = reinterpret_cast<const float2 *>(sk)[q * 32 + lane];
                rr[k] = v.x;
                pw[k] = v.y;
            } else {
                const float v = reinterpret_cast<const float *>(sk)[q * 32 + lane];
                rr[k] = HS ? v : 0.f;
                pw[k] = HS ? -S * v : v;
            }
        }
        const float pall = NW == 4 ? (pw[0] + pw[1]) + (pw[2] + pw[3])
                                   : ((pw[0] + pw[1]) + (pw[2] + pw[3])) + ((pw[4 % NW] + pw[5 % NW]) + (pw[6 % NW] + pw[7 % NW]));
        float run = 0.f;
#pragma unroll
        for (int k = 0; k < NW; ++k) {
            reinterpret_cast<float *>(c.sm + ring_off(k))[q * 32 + lane] = -(pall + S2 * run);
            run += rr[k];
        }
        // a pair's fold side: -P of b, past warp 0's per-card table
        if (HS && !HF && c.sigma2 >= 0)
            reinterpret_cast<float *>(c.sm + state_off(NW, 0, nc) + (size_t)nc * 128)[q * 32 + lane] = pall;
    }
    float Cw;
    {
        float tall = 0.f, gb = 0.f;
#pragma unroll
        for (int k = 0; k < NW; ++k) {
            tall += sums[(1 * NW + k) * 32 + lane];
            if (k < warp) gb += sums[(0 * NW + k) * 32 + lane];
        }
        Cw = tall + S2 * gb;
    }
    __syncthreads();

    return Cw;
}

// Finishing pass (the same for every column kind): out = scale lambda_out
// ((partial + C) - (Q[c1] + Q[c2])), staged in swizzled boxes (the rest of the
// ring) and stored by TMA; scale is S for showdown-only columns, else 1.  A
// box's finishing records (256 bytes) are copied one box ahead by cp.async
// into two buffers in the warp's record ring (idle after the scan).  PAIR: the
// fold side too, F lambda_out (Tot + b - (P[c1] + P[c2])), the row's boxes
// copied one box ahead into two buffers in the warp's own (idle) per-card
// table, whose rest is one more staging slot.  (Copied by the lanes, with
// cp.async, a 1024-vector FP32 launch takes 6 % longer.)  A warp whose scan gave
// up finishes nothing: a copy into its ring may still be in flight.
template <typename T, int K2, int NW, bool PAIR, bool SCALED>
__device__ __forceinline__ void tma_finish(const TmaArgs &P, Ctx &c, float Cw, float scale) {
    if (!c.ok) return;
    constexpr int BB = Box<T>::kBytes;
    const int lane = c.lane, nc = P.nc, nb = c.nb, z0 = 32 * c.bb;
    unsigned char *ring = c.sm + ring_off(c.warp);
    const float *xpart = reinterpret_cast<const float *>(c.sm + extra_off(NW, c.warp, nc, P.extra));
    const unsigned char *qb = ring + 4 * lane;
    const int qbytes = (nc * 128 + 1023) & ~1023;
    const int nring = min((kRingBytes - qbytes) / BB, 5), nbuf = nring + (PAIR ? 1 : 0);   // staging slots
    unsigned char *frb = c.sm + rec_off(NW, c.warp, nc, P.extra);
    const uint32_t frb_s = smem_u32(frb);
    // pairs: -P table, input boxes and a staging slot, their barriers (the
    // ring's last two), Tot
    const unsigned char *fb = c.sm + state_off(NW, 0, nc) + (size_t)nc * 128 + 4 * lane;
    unsigned char *yb = c.sm + ((state_off(NW, c.warp, nc) + 1023) & ~(size_t)1023), *xst = yb + 2 * BB;
    const uint32_t ybar = smem_u32(c.sm + hdr_off(NW, nc, P.extra) + 16) + 8u * (8u * (uint32_t)c.warp + 6u);
    float Tb = 0.f;
    if (PAIR) {
        const float *sums = reinterpret_cast<const float *>(c.sm + hdr_off(NW, nc, P.extra) + sums_at(NW));
#pragma unroll
        for (int k = 0; k < NW; ++k) Tb += sums[(0 * NW + k) * 32 + lane];
    }
    const float2 F2 = make_float2(c.F, c.F), S2 = make_float2(scale, scale);
    int ny = 0;                   // lane 0: boxes of the row copied
    auto fetch_y = [&](int m) {   // lane 0: box m of the row
        ny = m + 1;
        const uint32_t bar = ybar + 8u * (uint32_t)(m & 1);
        mbar_expect_tx(bar, BB);
        tma_load3(smem_u32(yb) + (uint32_t)((m & 1) * BB), &P.tin, kTmaBox * (c.b0 + m), c.rs, z0, bar);
    };
    if (PAIR) {
        if (lane == 0) {
            mbar_init(ybar, 1);
            mbar_init(ybar + 8u, 1);
            fence_barrier_init();
            fence_proxy_async();
            if (nb > 0) fetch_y(0);
        }
        __syncwarp();
    }
    auto fetch_fin = [&](int m) {
        if (m < nb && lane < 16)
            cp16(frb_s + (uint32_t)((m & 1) * 256 + 16 * lane),
                 reinterpret_cast<const unsigned char *>(P.rfin + (size_t)kTmaBox / 2 * (c.b0 + m)) + 16 * lane);
        cp_commit();
    };
    float cur[16], nxt[16];
    auto load_box = [&](int m, float *r) {
        if (m < 16) {
            tm_ld16(c.tmem + (uint32_t)(16 * m), r);
        } else {
            const float *xp = xpart + (m - 16) * (kTmaBox * 32);
#pragma unroll
            for (int i = 0; i < 16; ++i) r[i] = xp[i * 32 + lane];
        }
    };
    int nst = 0, next = 0;   // boxes staged, the next one's slot
    auto put = [&](int m, int sigma, const float2 *o) {
        const int sl = next;
        next = sl + 1 == nbuf ? 0 : sl + 1;
        unsigned char *buf = PAIR && sl == nring ? xst : ring + qbytes + sl * BB;
        // (a group per box: before a slot's second use all but the newest
        // nbuf - 1 have been read)
        if (nst >= nbuf) {
            if (lane == 0) {
                if (nbuf == 3) bulk_wait_read<2>();
                else bulk_wait_read_n(nbuf - 1);
            }
            __syncwarp();
        }
        ++nst;
        Box<T>::store(buf, lane, o);
        fence_proxy_async();
        // every lane has staged its outputs
        __syncwarp();
        if (lane == 0) {
            tma_store3(&P.tout, kTmaBox * (c.b0 + m), sigma, z0, smem_u32(buf));
            bulk_commit();
        }
    };
    // box m of the chunk: its partials in pc, box m + 1's loaded into pn
    // (the two arrays alternate, so no copy between boxes)
    auto box = [&](int m, const float *pc, float *pn) {
        if (m + 1 < nb) load_box(m + 1, pn);
        fetch_fin(m + 1);
        cp_wait<1>();   // this lane's copy of box m's records
        float2 y[8];
        if (PAIR) {
            if (lane == 0 && m + 1 < nb && c.ok) {
                fence_proxy_async();   // box m - 1's values were read before its staging barrier
                fetch_y(m + 1);
            }
            if (c.ok) {
                const uint32_t bar = ybar + 8u * (uint32_t)(m & 1), par = (uint32_t)((m >> 1) & 1);
                c.ok = __all_sync(kFull, mbar_try(bar, par) || mbar_wait(bar, par));
            }
            Box<T>::load(yb + (m & 1) * BB, lane, y);
        }
        __syncwarp();
        const TmaFinRec *fr = reinterpret_cast<const TmaFinRec *>(frb + (m & 1) * 256);
        float2 o[8];
#pragma unroll
        for (int i = 0; i < 16; i += 2) {
            const TmaFinRec r = fr[i / 2];
            // the table holds -Q: nq = -(Q[c1] + Q[c2]) for both hands
            float2 nq = make_float2(*reinterpret_cast<const float *>(qb + r.oa1),
                                    *reinterpret_cast<const float *>(qb + r.oa2));
            if (K2 == 2)
                nq = add2(nq, make_float2(*reinterpret_cast<const float *>(qb + r.ob1),
                                          *reinterpret_cast<const float *>(qb + r.ob2)));
            const float2 lo = make_float2(r.lout1, r.lout2);
            o[i / 2] = mul2(SCALED ? mul2(S2, lo) : lo, add2(add2(make_float2(pc[i], pc[i + 1]), make_float2(Cw, Cw)), nq));
            if (PAIR) {
                float2 np = make_float2(*reinterpret_cast<const float *>(fb + r.oa1),
                                        *reinterpret_cast<const float *>(fb + r.oa2));
                float2 b = make_float2(Tb, Tb);
                if (K2 == 2) {
                    np = add2(np, make_float2(*reinterpret_cast<const float *>(fb + r.ob1),
                                              *reinterpret_cast<const float *>(fb + r.ob2)));
                    b = fma2(make_float2(r.lin1, r.lin2), y[i / 2], b);
                }
                y[i / 2] = mul2(mul2(F2, lo), add2(b, np));
            }
        }
        put(m, c.sigma, o);
        if (PAIR) put(m, c.sigma2, y);
        if (m + 1 < nb) tm_wait_ld16(pn);
    };
    fetch_fin(0);
    if (nb > 0) {
        load_box(0, cur);
        tm_wait_ld16(cur);
    }
    for (int m = 0; m < nb; m += 2) {
        box(m, cur, nxt);
        if (m + 1 < nb) box(m + 1, nxt, cur);
    }
    cp_wait<0>();
    if (lane == 0) {
        bulk_wait_read<0>();
        // a wait gave up: the row's last two copies may be in flight
        if (PAIR && !c.ok)
            for (int m = max(0, ny - 2); m < ny; ++m)
                if (!mbar_wait(ybar + 8u * (uint32_t)(m & 1), (uint32_t)((m >> 1) & 1))) break;
    }
    __syncwarp();
}

template <typename T, int K2, int NW, Form FORM>
__global__ void __launch_bounds__(32 * NW, NW == 4 ? 2 : 1) tma_scan_kernel(const __grid_constant__ TmaArgs P) {
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    // the swizzled boxes need 1 KB alignment (one KB of slack is allocated)
    unsigned char *sm = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
    Ctx c;
    c.sm = sm;
    c.lane = threadIdx.x & 31;
    c.warp = threadIdx.x >> 5;
    c.bb = blockIdx.x / P.nitems;
    const TmaItem item = P.items[blockIdx.x - c.bb * P.nitems];
    c.sigma = item.sigma;
    c.sigma2 = item.sigma2;
    c.rf = item.rf;
    c.rs = item.rs;
    c.F = item.F;
    c.S = item.S;
    c.b0 = P.bchunk[c.warp];
    c.nb = P.bchunk[c.warp + 1] - c.b0;
    c.ok = true;
    uint32_t *tslot = reinterpret_cast<uint32_t *>(sm + hdr_off(NW, P.nc, P.extra));
    if (c.warp == 0) tm_alloc(smem_u32(tslot), NW * 64);
    tm_fence_before();
    __syncthreads();
    tm_fence_after();
    const uint32_t tbase = *tslot;
    c.tmem = tbase + ((uint32_t)(32 * (c.warp & 3)) << 16) + (uint32_t)(kTmemCols * (c.warp >> 2));
    const int kind = (c.rf >= 0 ? kKindF : 0) | (c.rs >= 0 ? kKindS : 0);
    float Cw;
    if (kind == kKindFS) Cw = tma_scan<T, kKindFS, K2, NW, FORM>(P, c);
    else if (kind == kKindF) Cw = tma_scan<T, kKindF, K2, NW, FORM>(P, c);
    else Cw = tma_scan<T, kKindS, K2, NW, FORM>(P, c);
    if (FORM == kPaired && c.sigma2 >= 0) {
        c.F = item.F2;
        tma_finish<T, K2, NW, true, true>(P, c, Cw, c.S);
    } else if (FORM != kSmall && kind == kKindS) {
        tma_finish<T, K2, NW, false, true>(P, c, Cw, c.S);
    } else {
        tma_finish<T, K2, NW, false, false>(P, c, Cw, 1.f);
    }
    if (!c.ok && c.lane == 0) atomicExch(P.err, 1u);
    tm_fence_before();
    __syncthreads();
    tm_fence_after();
    if (c.warp == 0) tm_dealloc(tbase, NW * 64);
}

// ---- host ------------------------------------------------------------------
using EncodeFn = CUresult (*)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                              const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                              CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeFn encode_fn(cudaError_t *err) {
    static std::once_flag once;
    static EncodeFn fn = nullptr;
    static cudaError_t status = cudaSuccess;
    std::call_once(once, [] {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q = cudaDriverEntryPointSymbolNotFound;
        status = cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q);
        if (status == cudaSuccess && (q != cudaDriverEntryPointSuccess || !p)) status = cudaErrorSymbolNotFound;
        if (status == cudaSuccess) fn = reinterpret_cast<EncodeFn>(p);
    });
    *err = status;
    return fn;
}

cudaError_t encode3(CUtensorMap *map, int storage, const void *base, int x, int y, int z, int pitch) {
    cudaError_t e;
    EncodeFn fn = encode_fn(&e);
    if (!fn) return e;
    const bool f32 = storage == kStoreF32;
    const cuuint64_t es = f32 ? 4 : 2;
    const cuuint64_t dims[3] = {(cuuint64_t)x, (cuuint64_t)y, (cuuint64_t)z};
    const cuuint64_t strides[2] = {(cuuint64_t)pitch * es, (cuuint64_t)pitch * es * (cuuint64_t)y};
    const cuuint32_t box[3] = {(cuuint32_t)kTmaBox, 1, 32};
    const cuuint32_t estr[3] = {1, 1, 1};
    auto encode = [&]() {
        return fn(map,
                  f32 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32
                  : storage == kStoreBF16 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT16,
                  3, const_cast<void *>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                  f32 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_32B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    };
    CUresult r = encode();
    if (r != CUDA_SUCCESS) {
        // a thread that has not used the device yet has no current context, which
        // a driver call (unlike the runtime's) does not make
        int dev = 0;
        e = cudaGetDevice(&dev);
        if (e == cudaSuccess) e = cudaSetDevice(dev);
        if (e != cudaSuccess) return e;
        r = encode();
    }
    return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

__device__ unsigned int g_tma_err;

template <typename T>
auto pick(bool one, int nw, Form form) {
    if (nw == 8) return one ? tma_scan_kernel<T, 1, 8, kSingle> : tma_scan_kernel<T, 2, 8, kSingle>;
    if (form == kPaired) return one ? tma_scan_kernel<T, 1, 4, kPaired> : tma_scan_kernel<T, 2, 4, kPaired>;
    if (form == kSmall) return one ? tma_scan_kernel<T, 1, 4, kSmall> : tma_scan_kernel<T, 2, 4, kSmall>;
    return one ? tma_scan_kernel<T, 1, 4, kSingle> : tma_scan_kernel<T, 2, 4, kSingle>;
}

}  // namespace

static size_t tma_smem_bytes(int nw, int nc, int extra) { return hdr_off(nw, nc, extra) + hdr_bytes(nw) + 1024; }

// Chunks, records and eligibility of one direction; fills p.a (but the
// tensor maps, pointers and batch) and p.host.  Empty string on success.
static std::string tma_prepare(const HostGame &h, const double *lam_in, const double *lam_out, TmaParams &p) {
    ScanRecords r;
    const std::string why = build_scan_records(h, lam_in, lam_out, kTmaMaxExtra, false, &r);
    if (!why.empty()) return why;
    TmaArgs &A = p.a;
    A.H = r.H;
    A.hs = r.hs;
    A.nc = r.nc;
    A.k = r.k;
    A.nbox = r.nbox;
    for (int k = 0; k <= kTmaWarps; ++k) p.chunk4[k] = r.bchunk[k];
    // eight chunks: each cut in two at the box boundary nearest its middle that
    // cuts no tie group
    auto clean = [&](int bx) { return bx <= 0 || bx >= r.nbox || 16 * bx >= r.H || h.group_lo[16 * bx] == 16 * bx; };
    p.eight = true;
    for (int k = 0; k < kTmaWarps; ++k) {
        const int lo = r.bchunk[k], hi = r.bchunk[k + 1], mid = (lo + hi) / 2;
        int cut = -1;
        for (int d = 0; d <= hi - lo && cut < 0; ++d) {
            if (mid - d >= lo && clean(mid - d)) cut = mid - d;
            else if (mid + d <= hi && clean(mid + d)) cut = mid + d;
        }
        p.chunk8[2 * k] = lo;
        p.chunk8[2 * k + 1] = cut;
        p.eight = p.eight && cut >= 0 && cut - lo <= 16 && hi - cut <= 16;
    }
    p.chunk8[2 * kTmaWarps] = r.nbox;
    p.eight = p.eight && tma_smem_bytes(kMaxNw, r.nc, 0) <= (size_t)max_dyn_smem();
    // (an SM has the largest CTA's shared memory and its reserved 1 KB)
    p.alone = 2 * (tma_smem_bytes(kTmaWarps, r.nc, r.extra) + 1024) > (size_t)max_dyn_smem() + 1024;
    p.extra4 = r.extra;
    p.host = std::move(r.bytes);
    return "";
}

// Items after the records: first the pairs and what is left alone, then every
// sequence alone.
std::string tma_items(int n_out, const int *hfcol, const int *hscol, const double *fcoef, const double *scoef,
                      TmaParams &p) {
    std::vector<TmaItem> items;
    auto add = [&](int r, int q) {
        items.push_back(TmaItem{r, q, hfcol[r], hscol[r], hfcol[r] >= 0 ? (float)fcoef[r] : 0.f,
                                hscol[r] >= 0 ? (float)scoef[r] : 0.f, q >= 0 ? (float)fcoef[q] : 0.f, 0});
    };
    for (int r = 0; r < n_out; ++r)
        if (hfcol[r] < 0 && hscol[r] < 0) return "an output sequence without terminals";
    std::vector<int> mate(n_out, -1);
    if (p.a.nc >= kPairMinCards) mate = fold_mates(n_out, hfcol, hscol);
    for (int r = 0; r < n_out; ++r)
        if (mate[r] != kMate) add(r, mate[r]);
    p.npaired = (int)items.size();
    p.nsingle = n_out;
    for (int r = 0; r < n_out; ++r) add(r, -1);
    p.o_items = (p.host.size() + 31) / 32 * 32;
    p.host.resize(p.o_items + sizeof(TmaItem) * items.size());
    if (!items.empty()) std::memcpy(p.host.data() + p.o_items, items.data(), sizeof(TmaItem) * items.size());
    return "";
}

}  // namespace kps

namespace kps {

TmaParams *tma_create(const HostGame &h, const double *lam_in, const double *lam_out, int n_out, int n_in,
                      const int *hfcol, const int *hscol, const double *fcoef, const double *scoef, std::string *why) {
    TmaParams *p = new (std::nothrow) TmaParams();
    if (!p) {
        *why = "host allocation";
        return nullptr;
    }
    std::string w;
    try {
        w = tma_prepare(h, lam_in, lam_out, *p);
        if (w.empty()) w = tma_items(n_out, hfcol, hscol, fcoef, scoef, *p);
    } catch (const std::bad_alloc &) {
        w = "host allocation";
    }
    if (w.empty() && std::max<size_t>(tma_smem_bytes(kTmaWarps, p->a.nc, p->extra4), 80 * 1024) > (size_t)max_dyn_smem())
        w = "shared memory";
    if (!w.empty()) {
        delete p;
        *why = w;
        return nullptr;
    }
    p->a.n_out = n_out;
    p->a.n_in = n_in;
    p->a.err = nullptr;
    return p;
}

cudaError_t tma_take_error(bool *set) {
    unsigned int v = 0, zero = 0;
    cudaError_t e = cudaMemcpyFromSymbol(&v, g_tma_err, sizeof(v));
    if (e == cudaSuccess && v) e = cudaMemcpyToSymbol(g_tma_err, &zero, sizeof(zero));
    *set = v != 0;
    return e;
}

void tma_destroy(TmaParams *p) {
    if (!p) return;
    if (p->dev) cudaFree(p->dev);
    delete p;
}

cudaError_t tma_upload(TmaParams *pp, cudaStream_t stream) {
    TmaParams &p = *pp;
    if (p.dev) return cudaSuccess;
    cudaError_t e = cudaGetSymbolAddress(reinterpret_cast<void **>(&p.a.err), g_tma_err);
    if (e != cudaSuccess) return e;
    int dev = 0;
    e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&p.sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    e = upload_table(&p.dev, p.host.data(), p.host.size(), stream);
    if (e != cudaSuccess) return e;
    p.a.rscan = static_cast<const unsigned char *>(p.dev);
    p.a.rfin = reinterpret_cast<const TmaFinRec *>(static_cast<const unsigned char *>(p.dev) +
                                                   (size_t)p.a.nbox * kScanBlock);
    p.device = dev;
    return cudaSuccess;
}

cudaError_t launch_tma_scan(TmaParams *pp, int storage, const void *vin, void *vout, int batch, cudaStream_t stream) {
    const TmaParams &p = *pp;
    cudaError_t e;
    TmaArgs A = p.a;   // a copy: other threads may launch the same game's products (the first ones under
                       // its lock until the tables are there)
    A.batch = batch;
    A.nbb = (batch + 31) / 32;
    // test hook (KPS_TEST_STALL_WAIT=1): one barrier per CTA never completes,
    // so that its bounded wait gives up and sets the error flag
    const char *st = std::getenv("KPS_TEST_STALL_WAIT");
    A.stall_test = st && std::atoi(st) > 0 ? 1 : 0;
    e = encode3(&A.tin, storage, vin, A.H, A.n_in, batch, A.hs);
    if (e == cudaSuccess) e = encode3(&A.tout, storage, vout, A.hs, A.n_out, batch, A.hs);
    if (e != cudaSuccess) return e;
    const int sms = p.sms;
    // Shape.  Eight warps (half as long a scan per warp) while every single item
    // has an SM to itself: 1 FP32 vector 26.6 -> 20.5 us, 96 vectors 28.8 ->
    // 22.6 us.  Else four warps, and pairs where they save a wave of two CTAs
    // per SM, since a paired item alone takes longer (41 against 35 us a wave):
    // 192 vectors (0.85 / 0.57 waves) single 34.9, paired 41.0 us; 256 (1.13 /
    // 0.76) 54.0, 41.2; 384 (1.70 / 1.14) 60.4, 67.6; 512 (2.26 / 1.53) 80.6, 72.0.
    // Where one CTA of four warps fills an SM's shared memory (1128 hands and up)
    // eight warps always: 100 FP32 vectors 46.6 -> 32.5 us, 384 95.7 -> 65.2.
    // Games of few boxes: up to kFewBoxes four warps (5.2 -> 4.6 us for one vector
    // of a 47-card one-card game), and up to kSmallBoxes the kernel whose finishing
    // pass is one for every kind (its instructions are fetched once: 1000 vectors of
    // a 6-card game 12.3 -> 11.1 us, 300 of a one-card game 6.5 -> 5.8).
    const long long single = (long long)p.nsingle * A.nbb, paired = (long long)p.npaired * A.nbb, slots = 2 * sms;
    const int nw = p.eight && A.nbox > kFewBoxes && (single <= sms || p.alone) ? 8 : 4;
    const bool pair = nw == 4 && (paired + slots - 1) / slots < (single + slots - 1) / slots;
    const Form form = pair ? kPaired : A.nbox <= kSmallBoxes ? kSmall : kSingle;
    const unsigned char *items = static_cast<const unsigned char *>(p.dev) + p.o_items;
    A.items = reinterpret_cast<const TmaItem *>(items) + (pair ? 0 : p.npaired);
    A.nitems = pair ? p.npaired : p.nsingle;
    A.extra = nw == 4 ? p.extra4 : 0;
    for (int k = 0; k <= nw; ++k) A.bchunk[k] = nw == 4 ? p.chunk4[k] : p.chunk8[k];
    // at least 80 KB: never more than two CTAs per SM, so that their tensor
    // memory (256 columns each) always fits
    const size_t smem = std::max<size_t>(tma_smem_bytes(nw, A.nc, A.extra), nw == 4 ? 80 * 1024 : 120 * 1024);
    const long long blocks = pair ? paired : single;
    if (blocks <= 0) return cudaSuccess;
    if (blocks > 0x7fffffffLL) return cudaErrorInvalidValue;
    void (*fn)(TmaArgs) = nullptr;
    const bool one = A.k == 1;
    switch (storage) {
        case kStoreF32: fn = pick<float>(one, nw, form); break;
        case kStoreBF16: fn = pick<__nv_bfloat16>(one, nw, form); break;
        case kStoreF16: fn = pick<__half>(one, nw, form); break;
        default: return cudaErrorInvalidValue;
    }
    e = ensure_dyn_smem(reinterpret_cast<const void *>(fn), smem);
    if (e != cudaSuccess) return e;
    fn<<<(unsigned)blocks, 32 * nw, smem, stream>>>(A);
    return cudaGetLastError();
}

}  // namespace kps
