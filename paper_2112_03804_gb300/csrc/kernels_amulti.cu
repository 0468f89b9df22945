// Kronecker-form payoff products of many games in one persistent launch
// (sm_103a), one vector per game and player, FP32 / BF16 / FP16 storage with
// FP32 arithmetic.
//
// Mathematics as in kernels_tma.cu (Prop. 1, Sec. 3):
//   out / lambda_out = K_F(w) + S (2 Lo_ord(b) - TB(b) + TA(b)),
//   a = lambda_in * y_f,  b = lambda_in * y_s,  w = F a - S b,
// K_F(w)[h] = Tot - P[c1] - P[c2] + w[h] (one-card hands: Tot - P[c1]).
//
// Organisation.  A work item is one game and up to 32 of its rows: lane j owns
// row row0 + j, an output sequence with its own fold and showdown input rows
// and payoffs (a sequence without a fold or a showdown terminal reads a zero
// row and has a zero payoff for it), or the pair of a call and a fold that
// share an input row: one scan of b (S = 1) gives both, as in kernels_tma.cu.  The
// four warps of a CTA scan four chunks of the game's hand order in boxes
// of 16 hands (the chunks and per-box hand records of scan_records.h,
// built once per game and direction).  For each box every lane copies its
// own two 64-byte row segments with cp.async into its own 16-byte slots of
// the warp's ring ([chunk of 4 hands][lane]: conflict-free reads), and
// lanes 0-16 copy the box's 272-byte record block; a ring of three boxes
// keeps two in flight while one is scanned, and each lane waits only for
// its own copy groups (plus a warp barrier before reading the records and
// before a slot is refilled).  Per-card sums are float2 [card][lane]
// tables, one per warp.  Partial results of the first 16 boxes of a chunk
// stay in tensor memory (lane = column, a column per hand); later boxes go
// to a per-CTA scratch area in global memory (L2-resident).  The four
// chunks are combined in shared memory exactly as in the single-game
// kernel; the finishing pass reads each box's finishing records from the
// record ring (copied one box ahead with cp.async, 256 bytes per half-warp),
// and each lane writes its finished row segments with 16-byte stores.  Ties:
// groups of up to 4 hands in registers, longer ones pair by pair from the
// entry lists of scan_records.h.  CTAs are persistent: they take work items from an atomic ticket
// or a static stride.  No spin-waits (cp.async groups complete in
// hardware), no atomics on results: bit-reproducible.
#include "kernels.h"
#include "game.h"
#include "host_parallel.h"
#include "scan_records.h"

#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <array>
#include <cstdint>
#include <cstring>
#include <new>
#include <string>
#include <vector>

namespace kps {

namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kNS = 3;                     // ring slots per warp
constexpr int kSlot = 4096;                // bytes per slot: fold rows, then showdown rows
constexpr int kRing = kNS * kSlot;         // per warp
constexpr int kRecRing = 2 * kNS * kScanBlock; // per warp: two record blocks per slot (split items)
constexpr int kTmemCols = 256;             // per CTA (two CTAs per SM)
constexpr int kMaxExtra = 8;               // chunk boxes past tensor memory (scratch)

// One game in one direction (device).
struct alignas(16) AmGame {
    int H, hs, nc, nbox;
    int bchunk[kTmaWarps + 1];
    int pad3[3];
    int bchunk8[2 * kTmaWarps + 1];   // split items: each chunk cut in two at a tie-free box boundary
    int pad4[3];
    long long in_off, out_off;     // element offsets of the game's input / output vectors
    const int2 *rows;              // of pairs: output sequence, the fold-only sequence of its pair or -1
    const int *fcol, *scol;        // per output sequence: its fold / showdown input sequence or -1
    const float *fcoef, *scoef;    // and the payoffs
    const unsigned char *rscan;    // [nbox][kScanBlock]
    const TmaFinRec *rfin;         // [nbox * 8]
    const TieEntry *ent;           // pairs of long tie groups
};

struct AmArgs {
    const AmGame *games;
    const int4 *items;             // (game, first row, split, last row + 1)
    int nitems, nc, schedule;
    const void *vin;               // element type: the kernel's storage type
    void *vout;
    float *scratch;                // [grid][4 warps][kMaxExtra][16][32]
    int *ticket;
};

// Shared memory: the four rings, the four record rings, the four per-card
// tables (nc rows of 256 bytes), then the header (tensor-memory slot at
// +0, work item at +4, per-warp sums [2][4][32] floats at +16).
__host__ __device__ inline size_t am_ring_off(int w) { return (size_t)w * kRing; }
__host__ __device__ inline size_t am_rec_off(int w) { return (size_t)kTmaWarps * kRing + (size_t)w * kRecRing; }
__host__ __device__ inline size_t am_state_off(int w, int nc) { return am_rec_off(kTmaWarps) + (size_t)w * nc * 256; }
__host__ __device__ inline size_t am_hdr_off(int nc) { return am_state_off(kTmaWarps, nc); }
inline size_t am_smem_bytes(int nc) { return am_hdr_off(nc) + 16 + 2 * kTmaWarps * 32 * 4; }

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }
// 16 bytes from global memory; the bytes past `src_bytes` (0 to 16) are zero
__device__ __forceinline__ void cp16(uint32_t dst, const void *src, uint32_t src_bytes) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(src_bytes) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
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
__device__ __forceinline__ void tm_wait_ld16(float *r) {
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+f"(r[0]), "+f"(r[1]), "+f"(r[2]), "+f"(r[3]), "+f"(r[4]), "+f"(r[5]), "+f"(r[6]), "+f"(r[7]),
                   "+f"(r[8]), "+f"(r[9]), "+f"(r[10]), "+f"(r[11]), "+f"(r[12]), "+f"(r[13]), "+f"(r[14]), "+f"(r[15])::"memory");
}

// Storage types: a 16-byte chunk holds 4 FP32 or 8 BF16 / FP16 values.
template <typename T> struct Store;
template <> struct Store<float> {
    static constexpr int kPer = 4;
    __device__ static void load(const unsigned char *p, float *v) {
        const float4 u = *reinterpret_cast<const float4 *>(p);
        v[0] = u.x; v[1] = u.y; v[2] = u.z; v[3] = u.w;
    }
    __device__ static uint4 pack(const float *v) {
        return make_uint4(__float_as_uint(v[0]), __float_as_uint(v[1]), __float_as_uint(v[2]), __float_as_uint(v[3]));
    }
};
template <> struct Store<__nv_bfloat16> {
    static constexpr int kPer = 8;
    __device__ static void load(const unsigned char *p, float *v) {
        const uint4 u = *reinterpret_cast<const uint4 *>(p);
        const uint32_t w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            v[2 * i] = __uint_as_float(w[i] << 16);
            v[2 * i + 1] = __uint_as_float(w[i] & 0xffff0000u);
        }
    }
    __device__ static uint4 pack(const float *v) {
        uint32_t w[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            __nv_bfloat162 h = __floats2bfloat162_rn(v[2 * i], v[2 * i + 1]);
            w[i] = *reinterpret_cast<uint32_t *>(&h);
        }
        return make_uint4(w[0], w[1], w[2], w[3]);
    }
};
template <> struct Store<__half> {
    static constexpr int kPer = 8;
    __device__ static void load(const unsigned char *p, float *v) {
        const uint4 u = *reinterpret_cast<const uint4 *>(p);
        const uint32_t w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float2 f = __half22float2(*reinterpret_cast<const __half2 *>(&w[i]));
            v[2 * i] = f.x;
            v[2 * i + 1] = f.y;
        }
    }
    __device__ static uint4 pack(const float *v) {
        uint32_t w[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            __half2 h = __floats2half2_rn(v[2 * i], v[2 * i + 1]);
            w[i] = *reinterpret_cast<uint32_t *>(&h);
        }
        return make_uint4(w[0], w[1], w[2], w[3]);
    }
};

// Bytes of a 16-byte chunk that hold hands when `left` hands of the row remain
// from its first (none when it is all padding).
template <typename T>
__device__ __forceinline__ uint32_t hand_bytes(int left) {
    return (uint32_t)(max(0, min(left, Store<T>::kPer)) * (int)sizeof(T));
}

// One work item, one warp: scan of the warp's chunk, combination of the
// four chunks (two CTA barriers), finishing pass.  A split item has at most
// 16 output sequences: lanes 16-31 take the same sequences as lanes 0-15 over
// the second half of the warp's chunk (eight sub-chunks in all), and the half
// with fewer boxes runs zero-filled boxes to the other's count, so that the
// warp's tensor-memory operations stay uniform.
// PAIRS: the rows are pairs and what is left alone, showdown-only rows scanned
// with S = 1.  TIES: a game of the batch lists ties of more than 4 hands.  A plan
// without them runs code without them (184 to 205 registers instead of 240): 512
// uneven games with single rows and no long ties 168 -> 158 us, 256 river games in
// pairs 64.6 -> 62.
template <typename T, int K2, bool PAIRS, bool TIES>
__device__ __forceinline__ void am_item(const AmArgs &P, const AmGame &G, int row0, int row1, int split,
                                        unsigned char *sm, uint32_t tmem, float *xs) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int nc = P.nc, hs = G.hs, H = G.H;
    const int half = split ? lane >> 4 : 0, col = split ? lane & 15 : lane;
    const int sub = split ? 2 * warp + half : warp;   // this lane's (sub-)chunk
    const int b0 = split ? G.bchunk8[sub] : G.bchunk[warp];
    const int nbl = (split ? G.bchunk8[sub + 1] : G.bchunk[warp + 1]) - b0;   // this lane's boxes
    const int b0h0 = __shfl_sync(kFull, b0, 0), b0h1 = __shfl_sync(kFull, b0, 16);
    const int nbh0 = __shfl_sync(kFull, nbl, 0), nbh1 = __shfl_sync(kFull, nbl, 16);
    const int nb = split ? max(nbh0, nbh1) : nbl;   // the warp's box count
    const bool act = row0 + col < row1;
    // without pairs a row is the sequence of its number
    const int2 sq = !act ? make_int2(0, -1) : PAIRS ? G.rows[row0 + col] : make_int2(row0 + col, -1);
    const int sigma = sq.x;
    const int rf = act ? G.fcol[sigma] : -1, rs = act ? G.scol[sigma] : -1;
    const float F = rf >= 0 ? G.fcoef[sigma] : 0.f;
    // a showdown-only row is scanned with S = 1 and finished with its payoff;
    // Fm: the payoff of its fold-only mate
    const bool unit = PAIRS && rf < 0 && rs >= 0;
    const float S = unit ? 1.f : rs >= 0 ? G.scoef[sigma] : 0.f;
    const float So = unit ? G.scoef[sigma] : 1.f, Fm = sq.y >= 0 ? G.fcoef[sq.y] : 0.f;
    const bool pairs = PAIRS && __any_sync(kFull, sq.y >= 0);
    const float S2 = 2.f * S;
    constexpr int NQ = 16 / Store<T>::kPer;   // 16-byte chunks per 16-hand row segment
    const T *vin = static_cast<const T *>(P.vin) + G.in_off;
    const T *pa = vin + (size_t)(rf >= 0 ? rf : 0) * hs;
    const T *pb = vin + (size_t)(rs >= 0 ? rs : 0) * hs;
    const uint32_t na = rf >= 0 ? 16u : 0u, nbytes_b = rs >= 0 ? 16u : 0u;
    unsigned char *ring = sm + am_ring_off(warp);
    const uint32_t ring_s = smem_u32(ring);
    unsigned char *rring = sm + am_rec_off(warp);
    const uint32_t rring_s = smem_u32(rring);
    unsigned char *stb = sm + am_state_off(warp, nc);
    unsigned char *lb = stb + 8 * lane;
    float *sums = reinterpret_cast<float *>(sm + am_hdr_off(nc) + 16);
    auto row = [&](uint32_t off) -> unsigned char * { return lb + 2 * off; };

    for (int q = lane; q < nc * 64; q += 32) reinterpret_cast<float *>(stb)[q] = 0.f;

    // copies of box m into slot m % kNS (an empty group past the chunk)
    auto issue = [&](int m) {
        if (m < nb) {
            const int sl = m % kNS;
            const bool real = m < nbl;   // past its half's boxes a lane copies zeros
            const int x = kTmaBox * (b0 + (real ? m : 0));
            const uint32_t dst = ring_s + (uint32_t)(sl * kSlot) + 16u * (uint32_t)lane;
            if (x + kTmaBox <= H) {
#pragma unroll
                for (int q = 0; q < NQ; ++q) {
                    const int h0 = x + Store<T>::kPer * q;
                    cp16(dst + 512u * q, pa + h0, real ? na : 0u);
                    cp16(dst + 2048u + 512u * q, pb + h0, real ? nbytes_b : 0u);
                }
            } else {   // the last boxes: padding hands hold anything, zeros take their place
#pragma unroll
                for (int q = 0; q < NQ; ++q) {
                    const int h0 = x + Store<T>::kPer * q;
                    const bool in = real && h0 < hs;   // hs is a multiple of 8: a chunk is all in or all out
                    const uint32_t n = in ? hand_bytes<T>(H - h0) : 0u;
                    cp16(dst + 512u * q, in ? pa + h0 : pa, min(n, na));
                    cp16(dst + 2048u + 512u * q, in ? pb + h0 : pb, min(n, nbytes_b));
                }
            }
            // the record block of each half's box (zeros for a zero-filled box)
            if (lane < kScanBlock / 16) {
                const bool r0 = m < nbh0;
                cp16(rring_s + (uint32_t)(2 * sl * kScanBlock) + 16u * (uint32_t)lane,
                     G.rscan + (size_t)(b0h0 + (r0 ? m : 0)) * kScanBlock + 16 * lane, r0 ? 16u : 0u);
                if (split) {
                    const bool r1 = m < nbh1;
                    cp16(rring_s + (uint32_t)((2 * sl + 1) * kScanBlock) + 16u * (uint32_t)lane,
                         G.rscan + (size_t)(b0h1 + (r1 ? m : 0)) * kScanBlock + 16 * lane, r1 ? 16u : 0u);
                }
            }
        }
        cp_commit();
    };
    for (int m = 0; m < kNS; ++m) issue(m);
    __syncwarp();

    float Gm = 0.f;
    float pp[16];
    float bq1 = 0.f, bq2 = 0.f, bq3 = 0.f;
#pragma unroll
    for (int i = 0; i < 16; ++i) pp[i] = 0.f;
    auto store_box = [&](int m, const float *r) {
        if (m < 16) {
            tm_st16(tmem + (uint32_t)(16 * m), r);
        } else {
            float *xp = xs + (m - 16) * (kTmaBox * 32);
#pragma unroll
            for (int i = 0; i < 16; ++i) xp[i * 32 + lane] = r[i];
        }
    };
    for (int m = 0; m < nb; ++m) {
        const int sl = m % kNS;
        cp_wait<kNS - 1>();
        __syncwarp();
        const unsigned char *slot = ring + sl * kSlot + 16 * lane;
        float yf[16], ys[16];
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
            Store<T>::load(slot + 512 * q, yf + Store<T>::kPer * q);
            Store<T>::load(slot + 2048 + 512 * q, ys + Store<T>::kPer * q);
        }
        const unsigned char *rsb = rring + (2 * sl + half) * kScanBlock;
        const uint32_t tw0 = reinterpret_cast<const uint32_t *>(rsb + 256)[0];
        const uint32_t tw1 = reinterpret_cast<const uint32_t *>(rsb + 256)[1];
        TmaScanRec rn = *reinterpret_cast<const TmaScanRec *>(rsb);
        float p[16], bv[16];
#pragma unroll
        for (int i = 0; i < 16; i += 2) {
            const TmaScanRec r = rn;
            if (i + 2 < 16) rn = reinterpret_cast<const TmaScanRec *>(rsb)[i / 2 + 1];
            unsigned char *A1 = row(r.oa1), *A2 = row(r.oa2), *B1 = row(r.ob1), *B2 = row(r.ob2);
            float2 sa1 = *reinterpret_cast<const float2 *>(A1);
            float2 sa2 = *reinterpret_cast<const float2 *>(A2);
            float2 sb1 = make_float2(0.f, 0.f), sb2 = make_float2(0.f, 0.f);
            if (K2 == 2) {
                sb1 = *reinterpret_cast<const float2 *>(B1);
                sb2 = *reinterpret_cast<const float2 *>(B2);
            }
            const float b1 = r.lin1 * ys[i], b2 = r.lin2 * ys[i + 1];
            bv[i] = b1;
            bv[i + 1] = b2;
            const float w1 = fmaf(F, r.lin1 * yf[i], -(S * b1));
            const float w2 = fmaf(F, r.lin2 * yf[i + 1], -(S * b2));
            // the first hand's update, seen by the second hand's sums when
            // they share a card (ma, mb are 0 or 1)
            sa2.x = fmaf(r.ma, b1, sa2.x);
            sa2.y = fmaf(r.ma, w1, sa2.y);
            if (K2 == 2) {
                sb2.x = fmaf(r.mb, b1, sb2.x);
                sb2.y = fmaf(r.mb, w1, sb2.y);
            }
            // partial = w + S (2 Lo_ord - TB), the w only for two-card hands
            const float t1 = 2.f * (Gm - (sa1.x + sb1.x));
            const float g1 = Gm + b1;
            const float t2 = 2.f * (g1 - (sa2.x + sb2.x));
            Gm = g1 + b2;
            p[i] = fmaf(S, t1, K2 == 2 ? w1 : 0.f);
            p[i + 1] = fmaf(S, t2, K2 == 2 ? w2 : 0.f);
            *reinterpret_cast<float2 *>(A1) = make_float2(sa1.x + b1, sa1.y + w1);
            if (K2 == 2) *reinterpret_cast<float2 *>(B1) = make_float2(sb1.x + b1, sb1.y + w1);
            *reinterpret_cast<float2 *>(A2) = make_float2(sa2.x + b2, sa2.y + w2);
            if (K2 == 2) *reinterpret_cast<float2 *>(B2) = make_float2(sb2.x + b2, sb2.y + w2);
        }
        // tie corrections of the box (TB leaves each tied hand's partial,
        // TA enters the earlier partner's; partners before the box are the
        // previous box's last three hands, stored one box late)
        if (tw0 | tw1) {
            auto bat = [&](int j) { return j >= 0 ? bv[j] : (j == -1 ? bq1 : j == -2 ? bq2 : bq3); };
            auto pat = [&](int j) -> float & { return j >= 0 ? p[j] : pp[16 + j]; };
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const uint32_t tb = ((k < 4 ? tw0 : tw1) >> (8 * (k & 3))) & 0xfcu;
                if (tb) {
                    const int i = 2 * k;
#pragma unroll
                    for (int d = 1; d <= 3; ++d)
                        if (tb & (1u << (1 + d))) {
                            p[i] = fmaf(-S, bat(i - d), p[i]);
                            pat(i - d) = fmaf(S, bv[i], pat(i - d));
                        }
#pragma unroll
                    for (int d = 1; d <= 3; ++d)
                        if (tb & (1u << (4 + d))) {
                            p[i + 1] = fmaf(-S, bat(i + 1 - d), p[i + 1]);
                            pat(i + 1 - d) = fmaf(S, bv[i + 1], pat(i + 1 - d));
                        }
                }
            }
        }
        // tie groups of more than 4 hands, pair by pair (rare: 1 in 270 of the
        // 1081-hand games).  The game stays on this kernel: in a launch of its own
        // on the tensor-memory kernel it cost a 256-game product 51 us more.
        const uint32_t nent = reinterpret_cast<const uint32_t *>(rsb + 256)[3];
        if (TIES && nent && rs >= 0) {
            // A hand's entries follow one another: they are added up first (sixteen
            // compares and additions a hand, not an entry), with the next two inputs
            // and the entry after them under way: 64 games with 924 entries each
            // 89 -> 58 us, 128 games with 810 90 -> 68.
            const TieEntry *te = G.ent + reinterpret_cast<const uint32_t *>(rsb + 256)[2];
            const uint32_t last = nent - 1;
            TieEntry t = te[0], t1 = te[min(1u, last)], t2 = te[min(2u, last)];
            float y = float(pb[t.q]), y1 = float(pb[t1.q]), sum = 0.f;
#pragma unroll 1
            for (uint32_t e = 0; e < nent; ++e) {
                const TieEntry t3 = te[min(e + 3, last)];
                const float y2 = float(pb[t2.q]);
                sum = fmaf(t.lin, y, sum);
                if (e == last || t1.i != t.i) {
#pragma unroll
                    for (int i = 0; i < 16; ++i)
                        if (i == t.i) p[i] = fmaf(S, sum, p[i]);
                    sum = 0.f;
                }
                t = t1;
                t1 = t2;
                t2 = t3;
                y = y1;
                y1 = y2;
            }
        }
        // every lane has read the slot's records: refill it
        __syncwarp();
        issue(m + kNS);
        if (m > 0) store_box(m - 1, pp);
#pragma unroll
        for (int i = 0; i < 16; ++i) pp[i] = p[i];
        bq1 = bv[15];
        bq2 = bv[14];
        bq3 = bv[13];
    }
    if (nb > 0) store_box(nb - 1, pp);
    cp_wait<0>();
    tm_wait_st();
    __syncwarp();

    // per-warp totals: b mass and K_F's Tot (every two-card hand is in two rows)
    float tot = 0.f;
    for (int q = 0; q < nc; ++q) tot += reinterpret_cast<const float2 *>(stb)[q * 32 + lane].y;
    if (K2 == 2) tot *= 0.5f;
    sums[(0 * kTmaWarps + warp) * 32 + lane] = Gm;
    sums[(1 * kTmaWarps + warp) * 32 + lane] = tot;
    __syncthreads();

    // combination: Q_k[c] = Pall[c] + 2 S (mass of card c in chunks < k),
    // [card][lane] floats at the start of warp k's ring; a split item's
    // sub-chunk k lives in warp k / 2, lanes 16 (k & 1) + column
    if (!split) {
        for (int q = warp; q < nc; q += kTmaWarps) {
            float rr[kTmaWarps], pw[kTmaWarps];
#pragma unroll
            for (int k = 0; k < kTmaWarps; ++k) {
                const float2 v = reinterpret_cast<const float2 *>(sm + am_state_off(k, nc))[q * 32 + lane];
                rr[k] = v.x;
                pw[k] = v.y;
            }
            const float pall = (pw[0] + pw[1]) + (pw[2] + pw[3]);
            float run = 0.f;
#pragma unroll
            for (int k = 0; k < kTmaWarps; ++k) {
                reinterpret_cast<float *>(sm + am_ring_off(k))[q * 32 + lane] = pall + S2 * run;
                run += rr[k];
            }
            // pairs: P in place of every warp's sums (this lane alone read them)
            if (pairs)
#pragma unroll
                for (int k = 0; k < kTmaWarps; ++k)
                    reinterpret_cast<float2 *>(sm + am_state_off(k, nc))[q * 32 + lane].x = pall;
        }
    } else if (lane < 16) {
        for (int q = warp; q < nc; q += kTmaWarps) {
            float rr[2 * kTmaWarps], pw[2 * kTmaWarps];
#pragma unroll
            for (int k = 0; k < 2 * kTmaWarps; ++k) {
                const float2 v =
                    reinterpret_cast<const float2 *>(sm + am_state_off(k >> 1, nc))[q * 32 + lane + 16 * (k & 1)];
                rr[k] = v.x;
                pw[k] = v.y;
            }
            const float pall = ((pw[0] + pw[1]) + (pw[2] + pw[3])) + ((pw[4] + pw[5]) + (pw[6] + pw[7]));
            float run = 0.f;
#pragma unroll
            for (int k = 0; k < 2 * kTmaWarps; ++k) {
                reinterpret_cast<float *>(sm + am_ring_off(k >> 1))[q * 32 + lane + 16 * (k & 1)] = pall + S2 * run;
                run += rr[k];
            }
            if (pairs)
#pragma unroll
                for (int k = 0; k < 2 * kTmaWarps; ++k)
                    reinterpret_cast<float2 *>(sm + am_state_off(k >> 1, nc))[q * 32 + lane + 16 * (k & 1)].x = pall;
        }
    }
    float Cw, tall = 0.f;
    {
        float gb = 0.f;
        if (!split) {
#pragma unroll
            for (int k = 0; k < kTmaWarps; ++k) {
                tall += sums[(1 * kTmaWarps + k) * 32 + lane];
                if (k < warp) gb += sums[(0 * kTmaWarps + k) * 32 + lane];
            }
        } else {
#pragma unroll
            for (int k = 0; k < 2 * kTmaWarps; ++k) {
                const int at = (k >> 1) * 32 + col + 16 * (k & 1);
                tall += sums[1 * kTmaWarps * 32 + at];
                if (k < sub) gb += sums[at];
            }
        }
        Cw = tall + S2 * gb;
    }
    __syncthreads();

    // finishing: out = So lambda_out (partial + C - Q[c1] - Q[c2]), and a pair's
    // fold side Fm lambda_out (b - Tot + P[c1] + P[c2]) (P and Tot of w = -b),
    // its row read once more, box by box, into the rest of the ring
    const unsigned char *qb = ring + 4 * lane;
    const unsigned char *pq = stb + 8 * lane;
    const uint32_t yb = (uint32_t)kRing - 4096u + 16u * (uint32_t)lane;
    T *orow2 = static_cast<T *>(P.vout) + G.out_off + (size_t)(sq.y >= 0 ? sq.y : 0) * hs;
    T *orow = static_cast<T *>(P.vout) + G.out_off + (size_t)(act ? sigma : 0) * hs;
    float cur[16], nxt[16];
    auto load_box = [&](int m, float *r) {
        if (m < 16) {
            tm_ld16(tmem + (uint32_t)(16 * m), r);
        } else {
            const float *xp = xs + (m - 16) * (kTmaBox * 32);
#pragma unroll
            for (int i = 0; i < 16; ++i) r[i] = xp[i * 32 + lane];
        }
    };
    // each half's finishing records of box m (256 bytes) are copied one box
    // ahead by its 16 lanes into two buffers in the record ring (idle after
    // the scan): [m & 1][half]
    const uint32_t frb_s = smem_u32(rring);
    auto fetch_fin = [&](int m) {
        if (m < nb && (split || lane < 16)) {
            // a zero-filled box reads the game's first records: its half may be empty
            // at the very end of the order
            const int bm = m < nbl ? b0 + m : 0;
            cp16(frb_s + (uint32_t)((((m & 1) * 2 + half) * 256) + 16 * (lane & 15)),
                 reinterpret_cast<const unsigned char *>(G.rfin + (size_t)kTmaBox / 2 * bm) + 16 * (lane & 15), 16u);
        }
        if (pairs && sq.y >= 0 && m < nbl) {
            const int x = kTmaBox * (b0 + m);
#pragma unroll
            for (int q = 0; q < NQ; ++q)
                if (x + Store<T>::kPer * q < hs)
                    cp16(ring_s + yb + (uint32_t)((m & 1) * 2048) + 512u * q, pb + x + Store<T>::kPer * q,
                         hand_bytes<T>(H - x - Store<T>::kPer * q));
        }
        cp_commit();
    };
    // box m: its partials in pc, box m + 1's loaded into pn (the two arrays
    // alternate, so no copy between boxes)
    auto box = [&](int m, const float *pc, float *pn) {
        if (m + 1 < nb) load_box(m + 1, pn);
        const bool real = m < nbl;   // a zero-filled box of the shorter half writes nothing
        __syncwarp();   // every lane has read box m - 1's records: refill their buffer
        fetch_fin(m + 1);
        cp_wait<1>();   // this lane's copy of box m's records
        __syncwarp();
        const TmaFinRec *fr = reinterpret_cast<const TmaFinRec *>(rring + ((m & 1) * 2 + half) * 256);
        float o[16], y[16];
        if (pairs) {
#pragma unroll
            for (int q = 0; q < NQ; ++q) Store<T>::load(ring + yb + (m & 1) * 2048 + 512 * q, y + Store<T>::kPer * q);
        }
#pragma unroll
        for (int i = 0; i < 16; i += 2) {
            const TmaFinRec r = fr[i / 2];
            if (pairs) {
                float p1 = *reinterpret_cast<const float *>(pq + 2 * r.oa1);
                float p2 = *reinterpret_cast<const float *>(pq + 2 * r.oa2);
                if (K2 == 2) {
                    p1 += *reinterpret_cast<const float *>(pq + 2 * r.ob1);
                    p2 += *reinterpret_cast<const float *>(pq + 2 * r.ob2);
                }
                y[i] = (r.lout1 * Fm) * ((K2 == 2 ? fmaf(r.lin1, y[i], -tall) : -tall) + p1);
                y[i + 1] = (r.lout2 * Fm) * ((K2 == 2 ? fmaf(r.lin2, y[i + 1], -tall) : -tall) + p2);
            }
            float q1 = *reinterpret_cast<const float *>(qb + r.oa1);
            float q2 = *reinterpret_cast<const float *>(qb + r.oa2);
            if (K2 == 2) {
                q1 += *reinterpret_cast<const float *>(qb + r.ob1);
                q2 += *reinterpret_cast<const float *>(qb + r.ob2);
            }
            o[i] = (PAIRS ? r.lout1 * So : r.lout1) * ((pc[i] + Cw) - q1);
            o[i + 1] = (PAIRS ? r.lout2 * So : r.lout2) * ((pc[i + 1] + Cw) - q2);
        }
        if (act && real) {
            const int x = kTmaBox * (b0 + m);
#pragma unroll
            for (int q = 0; q < NQ; ++q)
                if (x + Store<T>::kPer * q < hs)
                    *reinterpret_cast<uint4 *>(orow + x + Store<T>::kPer * q) = Store<T>::pack(o + Store<T>::kPer * q);
            if (pairs && sq.y >= 0) {
#pragma unroll
                for (int q = 0; q < NQ; ++q)
                    if (x + Store<T>::kPer * q < hs)
                        *reinterpret_cast<uint4 *>(orow2 + x + Store<T>::kPer * q) =
                            Store<T>::pack(y + Store<T>::kPer * q);
            }
        }
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
    __syncwarp();
}

template <typename T, int K2, bool PAIRS, bool TIES>
__global__ void __launch_bounds__(128, 2) async_multi_kernel(const __grid_constant__ AmArgs P) {
    extern __shared__ __align__(16) unsigned char sm[];
    const int warp = threadIdx.x >> 5;
    unsigned char *hdr = sm + am_hdr_off(P.nc);
    uint32_t *tslot = reinterpret_cast<uint32_t *>(hdr);
    int *sitem = reinterpret_cast<int *>(hdr + 4);
    if (warp == 0) tm_alloc(smem_u32(tslot), kTmemCols);
    tm_fence_before();
    __syncthreads();
    tm_fence_after();
    const uint32_t tbase = *tslot;
    const uint32_t tmem = tbase + ((uint32_t)(32 * warp) << 16);
    float *xs = P.scratch + ((size_t)blockIdx.x * kTmaWarps + warp) * kMaxExtra * (kTmaBox * 32);
    int next = blockIdx.x;
    for (;;) {
        int item;
        if (P.schedule == 0) {
            if (threadIdx.x == 0) *sitem = atomicAdd(P.ticket, 1);
            __syncthreads();
            item = *sitem;
        } else {
            item = next;
            next += gridDim.x;
        }
        if (item >= P.nitems) break;
        const int4 it = P.items[item];
        am_item<T, K2, PAIRS, TIES>(P, P.games[it.x], it.y, it.w, it.z, sm, tmem, xs);
        // the next ticket is written only after every thread has read this one
        // (am_item ends its combination with a CTA barrier)
    }
    tm_fence_before();
    __syncthreads();
    tm_fence_after();
    if (warp == 0) tm_dealloc(tbase, kTmemCols);
}

}  // namespace

// Time (us) of an item [single rows, pairs][full, split] of a 1081-hand game in
// FP32, {alone on its SM, two per SM}, measured on 1 to 600 river games and 20 games
// of 247 sequences (a full item of pairs alone: 39.3 and 44.2; two per SM 62 where
// every row is a pair, less in uneven games): what am_create's choice of rows and
// items goes by.  16-bit vectors take 0.75 to 0.8
// of every entry, and 1128 and 1176 hands a few percent more, so the choice is the
// same; games of some ten hands, whose items are bound by their fixed parts,
// take single rows in full items by it too, which is the fastest there (300
// one-card games of 47 hands 9.4 us; pairs 10.1, split items 18.4).  Uneven games (3 to
// 5 board cards): 200 games take 81 us by it (75 with pairs in split items), 512
// 155 (161 with pairs), 1500 404 and 4096 1055 with pairs (406 and 1077 without).
constexpr double kItemTime[2][2][2] = {{{29.5, 45.5}, {19.5, 27.8}}, {{42, 60}, {26.5, 39.6}}};

namespace {
template <typename T>
auto pick(int k, bool pairs, bool ties) {
    if (k == 1)
        return pairs ? (ties ? async_multi_kernel<T, 1, true, true> : async_multi_kernel<T, 1, true, false>)
                     : (ties ? async_multi_kernel<T, 1, false, true> : async_multi_kernel<T, 1, false, false>);
    return pairs ? (ties ? async_multi_kernel<T, 2, true, true> : async_multi_kernel<T, 2, true, false>)
                 : (ties ? async_multi_kernel<T, 2, false, true> : async_multi_kernel<T, 2, false, false>);
}
}  // namespace

// One direction of a batch.  Two lists of items over the same records and scratch
// area: the fastest ones (0), and plain rows (1).
struct AmPlan {
    AmArgs a{};
    struct {
        const int4 *items = nullptr;
        int n = 0;
        bool pairs = false;
    } list[2];
    bool ties = false;             // a game lists ties of more than 4 hands
    void *blob = nullptr;          // games, items, rows, records
    float *scratch = nullptr;
    int grid_cap = 0;              // CTAs the scratch area holds
    int k = 2;
    int device = -1;
};

namespace {
AmPlan *build_plan(const std::vector<AmGameDesc> &games, int grid_cap, cudaStream_t stream, std::vector<char> *taken,
                   std::string *why, size_t *need) {
    if (games.empty() || grid_cap < 1) {
        *why = "no games";
        return nullptr;
    }
    const int ng = (int)games.size();
    std::vector<ScanRecords> rec(ng);
    taken->assign(ng, 0);
    int nc = 0, ntaken = 0;
    size_t rbytes = 0;
    const int k = games[0].h->k;
    for (int i = 0; i < ng; ++i)
        if (games[i].h->k != k) {
            *why = "games with different hand sizes";
            return nullptr;
        }
    std::vector<std::string> refused(ng);
    long long hands = 0;
    for (int i = 0; i < ng; ++i) hands += games[i].h->H;
    parallel_for(ng, hands, [&](int i) {
        const AmGameDesc &d = games[i];
        refused[i] = build_scan_records(*d.h, d.lam_in, d.lam_out, kMaxExtra, true, &rec[i]);
        if (refused[i].empty() && rec[i].hs % 8 != 0) refused[i] = "hand stride not a multiple of 8";
        if (!refused[i].empty()) rec[i] = ScanRecords();
    });
    for (int i = 0; i < ng; ++i) {
        if (!refused[i].empty()) {
            // left to another kernel
            if (why->empty()) *why = "game " + std::to_string(i) + ": " + refused[i];
            continue;
        }
        (*taken)[i] = 1;
        ++ntaken;
        nc = std::max(nc, rec[i].nc);
        rbytes += (rec[i].bytes.size() + 255) / 256 * 256;
    }
    if (ntaken == 0) return nullptr;
    // Rows and items of every game: pairs or single sequences, items of 32 rows
    // (a tail of at most 16 as a split item) or split items alone.  Pairs leave
    // fewer items, split items half as long a scan: one A product of 600 river
    // games takes 132 us with pairs in full items, 164 without pairs, of
    // 100 games 28 us with single rows in split items, 46 in full ones, 40 with pairs.
    std::vector<char> can_split(ng, 0);
    std::vector<std::array<int, 2 * kTmaWarps + 1>> sub(ng);
    std::vector<std::vector<int2>> paired(ng);
    parallel_for(ng, hands, [&](int i) {
        if (!(*taken)[i]) return;
        const AmGameDesc &d = games[i];
        const ScanRecords &r = rec[i];
        // sub-chunks of split items: each chunk cut at the tie-free box
        // boundary nearest its middle (an empty second half if there is none)
        const HostGame &h = *d.h;
        auto clean = [&](int bx) {
            return bx <= 0 || bx >= r.nbox || 16 * bx >= r.H || h.group_lo[16 * bx] == 16 * bx;
        };
        can_split[i] = 1;
        for (int w = 0; w < kTmaWarps; ++w) {
            const int lo = r.bchunk[w], hi = r.bchunk[w + 1], ideal = (lo + hi) / 2;
            int mid = hi;
            for (int dd = 0; dd <= hi - lo && mid == hi; ++dd) {
                if (ideal - dd >= lo && clean(ideal - dd)) mid = ideal - dd;
                else if (ideal + dd <= hi && clean(ideal + dd)) mid = ideal + dd;
            }
            sub[i][2 * w] = lo;
            sub[i][2 * w + 1] = mid;
            can_split[i] = can_split[i] && mid - lo <= 16 && hi - mid <= 16;
        }
        sub[i][2 * kTmaWarps] = r.nbox;
        const std::vector<int> mate = fold_mates(d.n_out, d.hfcol, d.hscol);
        paired[i].reserve(d.n_out);
        for (int s = 0; s < d.n_out; ++s)
            if (d.hfcol[s] < 0) paired[i].push_back(make_int2(s, mate[s]));
        for (int s = 0; s < d.n_out; ++s)
            if (d.hfcol[s] >= 0 && mate[s] != kMate) paired[i].push_back(make_int2(s, -1));
    });
    // estimated time of a layout (see kItemTime), its items in *out
    auto layout = [&](bool pairs, bool halves, std::vector<int4> *out) {
        double sum = 0.0, alone = 0.0, longest = 0.0;
        long long n_items = 0;
        for (int i = 0; i < ng; ++i) {
            const int n = !(*taken)[i] ? 0 : pairs ? (int)paired[i].size() : games[i].n_out;
            for (int r0 = 0; r0 < n;) {
                const bool half = can_split[i] && (halves || n - r0 <= 16);
                const int r1 = std::min(n, r0 + (half ? 16 : 32));
                if (out) out->push_back(make_int4(i, r0, half ? 1 : 0, r1));
                const double *c = kItemTime[pairs ? 1 : 0][half ? 1 : 0];
                sum += c[1];
                alone = std::max(alone, c[0]);
                longest = std::max(longest, c[1]);
                ++n_items;
                r0 = r1;
            }
        }
        if (2 * n_items <= grid_cap) return alone;
        return n_items <= grid_cap ? longest : sum / grid_cap + 0.45 * longest;
    };
    double best = 0.0;
    int choice = -1;   // bit 0: single rows, bit 1: split items alone
    for (int v = 0; v < 4; ++v) {
        const double t = layout((v & 1) == 0, (v & 2) != 0, nullptr);
        if (choice < 0 || t < best) {
            best = t;
            choice = v;
        }
    }
    const bool pairs = (choice & 1) == 0, same = choice == 1;   // same: plain rows are the fastest
    std::vector<int4> items[2];
    layout(pairs, (choice & 2) != 0, &items[0]);
    if (!same) layout(false, false, &items[1]);
    const size_t nitems = items[0].size() + items[1].size();
    size_t nrows = 0;
    for (int i = 0; i < ng && pairs; ++i) nrows += paired[i].size();
    if (std::max(items[0].size(), items[1].size()) > 0x7fffffffULL) {
        *why = "too many work items";
        return nullptr;
    }
    if (std::max<size_t>(am_smem_bytes(nc), 80 * 1024) > (size_t)max_dyn_smem()) {
        *why = "shared memory";
        return nullptr;
    }
    auto al = [](size_t x) { return (x + 255) / 256 * 256; };
    const size_t o_games = 0, o_items = al(sizeof(AmGame) * ng), o_rows = o_items + al(sizeof(int4) * nitems),
                 o_rec = o_rows + al(sizeof(int2) * nrows);
    const size_t total = o_rec + rbytes;
    std::vector<unsigned char> host(total, 0);
    std::vector<AmGame> g(ng);
    std::vector<size_t> rec_at(ng), rows_at(ng);
    for (size_t i = 0, ro = o_rec, rowo = o_rows; i < (size_t)ng; ++i) {
        rec_at[i] = ro;
        rows_at[i] = rowo;
        if (!(*taken)[i]) continue;
        ro += al(rec[i].bytes.size());
        if (pairs) rowo += sizeof(int2) * paired[i].size();
    }
    const size_t scratch = (size_t)grid_cap * kTmaWarps * kMaxExtra * kTmaBox * 32 * sizeof(float);
    AmPlan *p = new AmPlan();
    cudaError_t e = device_malloc(&p->blob, total);
    if (e == cudaSuccess) e = device_malloc(&p->scratch, scratch);
    if (e != cudaSuccess) {
        if (p->blob) cudaFree(p->blob);
        delete p;
        *need = total + scratch;
        *why = "device memory for the launch tables";
        return nullptr;
    }
    p->grid_cap = grid_cap;
    unsigned char *dev = static_cast<unsigned char *>(p->blob);
    parallel_for(ng, hands, [&](int i) {
        const AmGameDesc &d = games[i];
        const ScanRecords &r = rec[i];
        AmGame &x = g[i];
        std::memset(&x, 0, sizeof(x));
        if (!(*taken)[i]) return;
        const size_t ro = rec_at[i];
        x.H = r.H;
        x.hs = r.hs;
        x.nc = r.nc;
        if (pairs) {
            std::memcpy(host.data() + rows_at[i], paired[i].data(), sizeof(int2) * paired[i].size());
            x.rows = reinterpret_cast<const int2 *>(dev + rows_at[i]);
        }
        for (int w = 0; w <= 2 * kTmaWarps; ++w) x.bchunk8[w] = sub[i][w];
        x.nbox = r.nbox;
        for (int w = 0; w <= kTmaWarps; ++w) x.bchunk[w] = r.bchunk[w];
        x.in_off = d.in_off;
        x.out_off = d.out_off;
        x.fcol = d.fcol;
        x.scol = d.scol;
        x.fcoef = d.fcoef;
        x.scoef = d.scoef;
        std::memcpy(host.data() + ro, r.bytes.data(), r.bytes.size());
        x.rscan = dev + ro;
        x.rfin = reinterpret_cast<const TmaFinRec *>(dev + ro + (size_t)r.nbox * kScanBlock);
        x.ent = reinterpret_cast<const TieEntry *>(dev + ro + r.entries_at);
    });
    std::memcpy(host.data() + o_games, g.data(), sizeof(AmGame) * ng);
    for (int l = 0, at = 0; l < 2; at += (int)items[l].size(), ++l)
        if (!items[l].empty())
            std::memcpy(host.data() + o_items + sizeof(int4) * at, items[l].data(), sizeof(int4) * items[l].size());
    e = cudaMemcpyAsync(p->blob, host.data(), total, cudaMemcpyHostToDevice, stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(stream);
    if (e != cudaSuccess) {
        cudaFree(p->blob);
        cudaFree(p->scratch);
        delete p;
        *need = total + scratch;
        *why = "uploading the launch tables";
        return nullptr;
    }
    p->a.games = reinterpret_cast<const AmGame *>(dev + o_games);
    p->list[0] = {reinterpret_cast<const int4 *>(dev + o_items), (int)items[0].size(), pairs};
    if (same) p->list[1] = p->list[0];
    else p->list[1] = {p->list[0].items + items[0].size(), (int)items[1].size(), false};
    for (int i = 0; i < ng; ++i) p->ties = p->ties || ((*taken)[i] && rec[i].bytes.size() > rec[i].entries_at);
    p->a.nc = nc;
    p->k = k;
    cudaGetDevice(&p->device);
    return p;
}
}  // namespace

AmPlan *am_create(const std::vector<AmGameDesc> &games, int grid_cap, cudaStream_t stream, std::vector<char> *taken,
                  std::string *why, size_t *need) {
    *need = 0;
    try {
        return build_plan(games, grid_cap, stream, taken, why, need);
    } catch (const std::bad_alloc &) {
        *need = 1;
        *why = "host allocation";
        return nullptr;
    }
}

void am_destroy(AmPlan *p) {
    if (!p) return;
    if (p->blob) cudaFree(p->blob);
    if (p->scratch) cudaFree(p->scratch);
    delete p;
}

// At least 80 KB of shared memory per CTA: never more than two CTAs per SM,
// so that their tensor memory (256 columns each) always fits.
static size_t am_launch_smem(int nc) { return std::max<size_t>(am_smem_bytes(nc), 80 * 1024); }

int am_grid_cap(const AmPlan *p) { return p->grid_cap; }

int am_items(const AmPlan *p, bool plain) { return p->list[plain ? 1 : 0].n; }

int am_ctas_per_sm(const AmPlan *p) {
    const size_t smem = am_launch_smem(p->a.nc);
    int dev = 0, per_sm = 0, reserved = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&per_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev);
    cudaDeviceGetAttribute(&reserved, cudaDevAttrReservedSharedMemoryPerBlock, dev);
    const int by_smem = (int)((size_t)per_sm / (smem + (size_t)reserved));
    return std::max(0, std::min(2, by_smem));
}

cudaError_t launch_async_multi(AmPlan *p, bool plain, int storage, const void *vin, void *vout, int *ticket,
                               int schedule, int grid, cudaStream_t stream) {
    // the scratch area holds the chunk boxes past tensor memory of grid_cap CTAs
    if (grid <= 0 || grid > p->grid_cap) return cudaErrorInvalidValue;
    AmArgs a = p->a;
    const auto &l = p->list[plain ? 1 : 0];
    a.items = l.items;
    a.nitems = l.n;
    a.vin = vin;
    a.vout = vout;
    a.scratch = p->scratch;
    a.ticket = ticket;
    a.schedule = schedule;
    if (a.nitems == 0) return cudaSuccess;
    const size_t smem = am_launch_smem(a.nc);
    void (*fn)(AmArgs) = nullptr;
    switch (storage) {
        case kStoreF32: fn = pick<float>(p->k, l.pairs, p->ties); break;
        case kStoreBF16: fn = pick<__nv_bfloat16>(p->k, l.pairs, p->ties); break;
        case kStoreF16: fn = pick<__half>(p->k, l.pairs, p->ties); break;
        default: return cudaErrorInvalidValue;
    }
    cudaError_t e = ensure_dyn_smem(reinterpret_cast<const void *>(fn), smem);
    if (e != cudaSuccess) return e;
    fn<<<grid, 32 * kTmaWarps, smem, stream>>>(a);
    return cudaGetLastError();
}

}  // namespace kps
