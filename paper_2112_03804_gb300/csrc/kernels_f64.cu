// Kronecker-form payoff products in FP64 (sm_103a): one game and many vectors,
// or many games with one vector each.
//
// Mathematics as in kernels_tma.cu (Prop. 1, Sec. 3):
//   out / lambda_out = K_F(w) + S (2 Lo_ord(b) - TB(b) + TA(b)),
//   a = lambda_in y_f,  b = lambda_in y_s,  w = F a - S b,
// Lo_ord the compatible mass of b before a hand in library order, TB / TA the
// compatible tied mass before / after it.
//
// What bounds it: the FP64 pipe, which starts one warp instruction per SM about
// every 16 cycles.  So every FP64 instruction counts (rows by kind, a fold and a
// call of one bet as one row scanned with S = 1, weights and card offsets from
// records, the second hand of a pair fixed up by selects instead of multiplies),
// and the pipe must never wait: six warps per SM, each with its own per-card
// table.  The kernel it replaces (kernels_vec.cu, still taken where this one
// does not apply) had three warps per SM and several times the instructions:
// 100 vectors of the 1081-hand river game 432 -> 214 us, one product of 64 such
// games 514 -> 122 us.
//
// Organisation.  A CTA = one item: up to 32 columns (row, vector) of one game
// and one kind, lane = column; or up to 16 (8) columns, their two (four) groups
// of lanes on two (four) parts of every warp's chunk: where 32 columns are not
// there, or where shorter items fill the SMs better.  The NW warps scan NW
// chunks of the hand order in boxes of 8 hands.  Every lane copies its own
// 64-byte row segments with cp.async one box ahead ([16 bytes][lane]: conflict
// free), a group's lanes together its box's records.  Partial results go to
// the output row and come back in the finishing pass (the lane's own, L2), so
// that shared memory holds the tables only.  Combination: Q_k[c] = P[c] + 2 S
// (mass of card c in earlier chunks) takes the place of chunk k's sums in its
// table, P (for the fold side of pairs) their second component.  Ties are
// corrected pair by pair from entry lists (two FP64 instructions each), so
// chunks may cut tie groups.  No atomics: results are bit-reproducible.
#include "kernels.h"
#include "game.h"
#include "host_parallel.h"
#include "scan_records.h"

#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <cstring>
#include <functional>
#include <new>
#include <queue>
#include <string>
#include <vector>

namespace kps {

namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kBox = 8;                    // hands per box
constexpr int kNW = kF64Warps;             // warps per CTA
constexpr int kNS = 2;                     // ring slots
constexpr int kParts = 4;                  // most parts of a chunk
constexpr int kRow = 2048;                 // bytes of one row's box (32 lanes x 64)
constexpr int kSlot = 2 * kRow;

struct alignas(16) Rec {                   // hands 2i, 2i + 1 of a box
    uint32_t oa1, ob1, oa2, ob2;           // card rows * 16
    double lin1, lin2, lout1, lout2;
    uint32_t ma, mb;                       // the second hand's first / second card is one of the first hand's
    uint32_t pad[2];
};
struct alignas(16) Tie {
    int i, q;                              // hand i of the box, its tied partner q
    double lin;                            // lambda_in[q], negative when q is earlier
};
constexpr int kInline = 2;                 // tie entries in the record itself (a tied pair inside a box makes two)
struct alignas(16) RecBox {
    Rec r[kBox / 2];
    Tie t[kInline];
    uint32_t first, count, pad[2];         // the others in the game's list; count of all
};
static_assert(sizeof(Rec) == 64 && sizeof(RecBox) == 304, "record layout");

// One game in one direction (device).
struct alignas(16) Game {
    int H, hs, nbox, n_in, n_out;
    int nunit, nrows, pad;                 // rows: nunit showdown-only ones (pairs among them), then the others
    long long in_off, out_off;
    const int2 *rows;
    const int *fcol, *scol;
    const double *fcoef, *scoef;
    const RecBox *rec;
    const Tie *ties;
};

struct Args {
    const Game *games;
    const int4 *items;                     // (game, first column, end, parts | unit << 3), or null: one game
    const double *vin;
    double *vout;
    int batch, nc, parts, nother;          // one game: vectors, and its items: nother of the other rows first
};

// Shared memory of a warp: table [card][lane] {b mass, w total}, ring, records.
__host__ __device__ inline size_t table_bytes(int nc) { return (size_t)nc * 512; }
__host__ __device__ inline size_t warp_bytes(int nc) { return table_bytes(nc) + kNS * kSlot + kNS * kParts * sizeof(RecBox); }
inline size_t smem_bytes(int nc) { return kNW * warp_bytes(nc) + 2 * kNW * 32 * 8; }

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }
// 16 bytes; those past `src_bytes` (0 or 16) are zero
__device__ __forceinline__ void cp16(uint32_t dst, const void *src, uint32_t src_bytes) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(src_bytes) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// UNIT: every column is showdown-only (S = 1, w = -b; a table's second
// components unused), its fold-only mate finished with it.
template <bool UNIT>
__device__ __forceinline__ void f64_item(const Args &P, const Game &G, int col0, int col1, int parts,
                                         unsigned char *smem) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nc = P.nc, hs = G.hs;
    const int width = 32 / parts, part = lane / width, slot = lane & (width - 1), col = col0 + slot;
    const bool act = col < col1;
    const int row = (UNIT ? 0 : G.nunit) + (act ? col / P.batch : 0), vec = act ? col % P.batch : 0;
    const int2 sq = act ? G.rows[row] : make_int2(0, -1);
    const int sigma = sq.x;
    const int rf = act && !UNIT ? G.fcol[sigma] : -1, rs = act ? G.scol[sigma] : -1;
    const double F = rf >= 0 ? G.fcoef[sigma] : 0.0, Sc = rs >= 0 ? G.scoef[sigma] : 0.0;
    const double S = UNIT ? 1.0 : Sc, S2 = 2.0 * S;
    const bool pairs = UNIT && __any_sync(kFull, sq.y >= 0);
    const double Fm = UNIT && sq.y >= 0 ? G.fcoef[sq.y] : 0.0;
    const double *vin = P.vin + G.in_off + (long long)vec * G.n_in * hs;
    const double *pa = vin + (long long)(rf >= 0 ? rf : 0) * hs, *pb = vin + (long long)(rs >= 0 ? rs : 0) * hs;
    double *vout = P.vout + G.out_off + (long long)vec * G.n_out * hs;
    double *po = vout + (long long)sigma * hs, *po2 = vout + (long long)(sq.y >= 0 ? sq.y : 0) * hs;
    // this lane's boxes, and the warp's longest part
    const int nk = kNW * parts, sub = parts * warp + part;
    auto bound = [&](int k) { return (int)((long long)G.nbox * k / nk); };
    const int b0 = bound(sub), nbl = bound(sub + 1) - b0, nb = __reduce_max_sync(kFull, nbl);

    unsigned char *mine = smem + (size_t)warp * warp_bytes(nc);
    double2 *tab = reinterpret_cast<double2 *>(mine) + lane;   // [card * 32]; a record offset is card * 16
    unsigned char *lt = mine + 16 * lane;
    unsigned char *ring = mine + table_bytes(nc), *recs = ring + kNS * kSlot;
    const uint32_t ring_s = smem_u32(ring) + 16u * (uint32_t)lane, recs_s = smem_u32(recs);
    double *sums = reinterpret_cast<double *>(smem + (size_t)kNW * warp_bytes(nc));   // [2][NW][32]
    auto at = [&](uint32_t off) { return reinterpret_cast<double2 *>(lt + 32 * off); };

    for (int c = 0; c < nc; ++c) tab[c * 32] = make_double2(0.0, 0.0);

    auto fetch = [&](int m, bool rows) {
        if (m < nb) {
            const int sl = m & 1;
            const bool real = act && m < nbl;
            const long long x = (long long)kBox * (b0 + (real ? m : 0));
            if (rows) {
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    if (!UNIT) cp16(ring_s + (uint32_t)(sl * kSlot + 512 * q), pa + x + 2 * q, real && rf >= 0 ? 16u : 0u);
                    cp16(ring_s + (uint32_t)(sl * kSlot + kRow + 512 * q), pb + x + 2 * q, real && rs >= 0 ? 16u : 0u);
                }
            }
            // records of each part's box (zeros past its last)
            const bool rec = m < nbl;
            for (int j = slot; j < (int)sizeof(RecBox) / 16; j += width)
                cp16(recs_s + (uint32_t)((kParts * sl + part) * sizeof(RecBox)) + 16u * (uint32_t)j,
                     reinterpret_cast<const unsigned char *>(rec ? G.rec + b0 + m : G.rec) + 16 * j, rec ? 16u : 0u);
        }
        cp_commit();
    };
    auto values = [&](const unsigned char *p, int x, double *y) {   // hands past H hold anything
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const double2 v = *reinterpret_cast<const double2 *>(p + 512 * q);
            y[2 * q] = x + 2 * q < G.H ? v.x : 0.0;
            y[2 * q + 1] = x + 2 * q + 1 < G.H ? v.y : 0.0;
        }
    };

    // ---- scan
    double Gm = 0.0;
    fetch(0, true);
    for (int m = 0; m < nb; ++m) {
        fetch(m + 1, true);
        cp_wait<1>();
        __syncwarp();
        const int sl = m & 1, x = kBox * (b0 + m);
        const RecBox *rb = reinterpret_cast<const RecBox *>(recs) + kParts * sl + part;
        double ys[kBox], yf[kBox], p[kBox];
        if (!UNIT) values(ring + sl * kSlot + 16 * lane, x, yf);
        values(ring + sl * kSlot + kRow + 16 * lane, x, ys);
#pragma unroll
        for (int i = 0; i < kBox; i += 2) {
            const Rec &r = rb->r[i / 2];
            double2 *A1 = at(r.oa1), *B1 = at(r.ob1), *A2 = at(r.oa2), *B2 = at(r.ob2);
            const double b1 = r.lin1 * ys[i], b2 = r.lin2 * ys[i + 1];
            if (UNIT) {
                const double a1 = A1->x, c1 = B1->x;
                double a2 = A2->x, c2 = B2->x;
                const double u1 = a1 + b1, v1 = c1 + b1;
                // the second hand sees the first one's update of a shared card
                if (r.ma) a2 = r.oa2 == r.oa1 ? u1 : v1;
                if (r.mb) c2 = r.ob2 == r.oa1 ? u1 : v1;
                const double t1 = Gm - (a1 + c1);
                const double g1 = Gm + b1;
                const double t2 = g1 - (a2 + c2);
                Gm = g1 + b2;
                A1->x = u1;
                B1->x = v1;
                A2->x = a2 + b2;
                B2->x = c2 + b2;
                p[i] = fma(2.0, t1, -b1);
                p[i + 1] = fma(2.0, t2, -b2);
            } else {
                const double w1 = fma(F, r.lin1 * yf[i], -(S * b1)), w2 = fma(F, r.lin2 * yf[i + 1], -(S * b2));
                const double2 a1 = *A1, c1 = *B1;
                double2 a2 = *A2, c2 = *B2;
                const double2 u1 = make_double2(a1.x + b1, a1.y + w1), v1 = make_double2(c1.x + b1, c1.y + w1);
                if (r.ma) a2 = r.oa2 == r.oa1 ? u1 : v1;
                if (r.mb) c2 = r.ob2 == r.oa1 ? u1 : v1;
                const double t1 = Gm - (a1.x + c1.x);
                const double g1 = Gm + b1;
                const double t2 = g1 - (a2.x + c2.x);
                Gm = g1 + b2;
                *A1 = u1;
                *B1 = v1;
                *A2 = make_double2(a2.x + b2, a2.y + w2);
                *B2 = make_double2(c2.x + b2, c2.y + w2);
                p[i] = fma(S2, t1, w1);
                p[i + 1] = fma(S2, t2, w2);
            }
        }
        if (rb->count && rs >= 0) {
            for (uint32_t e = 0; e < rb->count; ++e) {
                const Tie t = e < kInline ? rb->t[e] : G.ties[rb->first + e - kInline];
                double y = 0.0;
                if ((unsigned)(t.q - x) < (unsigned)kBox) {   // most partners are in the box itself
#pragma unroll
                    for (int i = 0; i < kBox; ++i)
                        if (i == t.q - x) y = ys[i];
                } else {
                    y = pb[t.q];
                }
                const double d = S * (t.lin * y);
#pragma unroll
                for (int i = 0; i < kBox; ++i)
                    if (i == t.i) p[i] += d;
            }
        }
        if (act && m < nbl) {
#pragma unroll
            for (int q = 0; q < 4; ++q)
                reinterpret_cast<double2 *>(po + x)[q] = make_double2(p[2 * q], p[2 * q + 1]);
        }
        __syncwarp();   // every lane has read the slot's records
    }
    cp_wait<0>();

    // ---- combination, in place
    double tot = 0.0;
    if (!UNIT)
        for (int c = 0; c < nc; ++c) tot += tab[c * 32].y;
    sums[warp * 32 + lane] = Gm;
    sums[(kNW + warp) * 32 + lane] = UNIT ? -Gm : 0.5 * tot;   // every hand is in two card rows
    __syncthreads();
    {
        // a row of the tables by the lanes of one part, for its columns
        for (int c = sub; c < nc; c += nk) {
            double pall = 0.0, run = 0.0;
            auto cell = [&](int k) {
                return reinterpret_cast<double2 *>(smem + (size_t)(k / parts) * warp_bytes(nc)) + c * 32 + slot +
                       width * (k % parts);
            };
            for (int k = 0; k < nk; ++k) pall += UNIT ? -cell(k)->x : cell(k)->y;
            for (int k = 0; k < nk; ++k) {
                double2 *v = cell(k);
                const double rr = v->x;
                *v = make_double2(fma(S2, run, pall), pall);
                run += rr;
            }
        }
    }
    double C, tall = 0.0, gb = 0.0;
    for (int k = 0; k < nk; ++k) {
        const int i = k / parts * 32 + slot + width * (k % parts);
        tall += sums[kNW * 32 + i];
        if (k < sub) gb += sums[i];
    }
    C = fma(S2, gb, tall);
    __syncthreads();

    // ---- finishing: out = So lambda_out (partial + C - Q[c1] - Q[c2]); the fold
    // side of a pair: Fm lambda_out (b - Tot + P[c1] + P[c2]) (P, Tot of w = -b)
    const double So = UNIT ? Sc : 1.0;
    double2 cur[4], nxt[4], yc[4], yn[4];
    auto load = [&](int m, double2 *pp, double2 *yy) {
        const bool real = act && m < nbl;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            pp[q] = real ? reinterpret_cast<const double2 *>(po + kBox * (b0 + m))[q] : make_double2(0.0, 0.0);
            if (UNIT)
                yy[q] = real && sq.y >= 0 ? reinterpret_cast<const double2 *>(pb + kBox * (b0 + m))[q]
                                          : make_double2(0.0, 0.0);
        }
    };
    fetch(0, false);
    load(0, cur, yc);
    for (int m = 0; m < nb; ++m) {
        fetch(m + 1, false);
        load(m + 1, nxt, yn);
        cp_wait<1>();
        __syncwarp();
        const RecBox *rb = reinterpret_cast<const RecBox *>(recs) + kParts * (m & 1) + part;
        const int x = kBox * (b0 + m);
        if (act && m < nbl) {
#pragma unroll
            for (int i = 0; i < kBox; i += 2) {
                const Rec &r = rb->r[i / 2];
                const double2 a1 = *at(r.oa1), c1 = *at(r.ob1), a2 = *at(r.oa2), c2 = *at(r.ob2);
                const double2 pc = cur[i / 2];
                const double o1 = (pc.x + C) - (a1.x + c1.x), o2 = (pc.y + C) - (a2.x + c2.x);
                reinterpret_cast<double2 *>(po + x)[i / 2] =
                    UNIT ? make_double2((r.lout1 * So) * o1, (r.lout2 * So) * o2) : make_double2(r.lout1 * o1, r.lout2 * o2);
                if (UNIT && pairs && sq.y >= 0) {
                    const double y1 = x + i < G.H ? yc[i / 2].x : 0.0, y2 = x + i + 1 < G.H ? yc[i / 2].y : 0.0;
                    const double f1 = fma(r.lin1, y1, -tall) + (a1.y + c1.y);
                    const double f2 = fma(r.lin2, y2, -tall) + (a2.y + c2.y);
                    reinterpret_cast<double2 *>(po2 + x)[i / 2] = make_double2((r.lout1 * Fm) * f1, (r.lout2 * Fm) * f2);
                }
            }
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            cur[q] = nxt[q];
            if (UNIT) yc[q] = yn[q];
        }
        __syncwarp();
    }
    cp_wait<0>();
}

__global__ void __launch_bounds__(32 * kNW, 1) f64_scan_kernel(const __grid_constant__ Args P) {
    extern __shared__ __align__(16) unsigned char smem[];
    int4 it;
    if (P.items) {
        it = P.items[blockIdx.x];
    } else {
        // one game: the items of the other rows (the longer ones), then the showdown-only ones
        const Game &G = P.games[0];
        const int w = 32 / P.parts, b = (int)blockIdx.x;
        const bool unit = b >= P.nother;
        const int c0 = w * (unit ? b - P.nother : b), n = (unit ? G.nunit : G.nrows - G.nunit) * P.batch;
        it = make_int4(0, c0, min(n, c0 + w), P.parts | (unit ? 8 : 0));
    }
    const Game &G = P.games[it.x];
    if (it.w & 8) f64_item<true>(P, G, it.y, it.z, it.w & 7, smem);
    else f64_item<false>(P, G, it.y, it.z, it.w & 7, smem);
}

}  // namespace

struct F64Plan {
    Args a{};
    void *blob = nullptr;
    int nitems = 0;                // many games
    int nunit = 0, nother = 0;     // one game: rows by kind
    int nbox = 0;                  // and its boxes
    int sms = 1;                   // of the device
};

namespace {
// Time (us) of an item of `parts` parts: the tables are cleared and combined row
// by row, and the longest part goes box by box.  Fitted to games of 15 to 1176
// hands (one wave of items: 11.7 us at 2 boxes and 9 card rows, 48 / 33 / 26 at 27
// and 22 for 1, 2 and 4 parts, 207 / 119 / 72 at 136 and 48); with it the time of
// 20 to 1500 uneven games comes out within 3 %.
double item_time(int nc, int nbox, int parts) {
    return 0.5 * nc + 8.0 * ((nbox + kNW * parts - 1) / (kNW * parts));
}
}  // namespace

F64Plan *f64_create(const std::vector<F64GameDesc> &games, bool multi, cudaStream_t stream, std::string *why,
                    size_t *need) {
    *need = 0;
    const int ng = (int)games.size();
    std::vector<std::vector<int2>> rows(ng);
    std::vector<Game> g(ng);
    std::vector<int4> items;
    auto al = [](size_t x) { return (x + 255) / 256 * 256; };
    int nc = 0, dev = 0, sms = 1;
    if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    size_t rbytes = 0, nrows = 0;
    long long hands = 0;
    for (int i = 0; i < ng; ++i) {
        nc = std::max(nc, games[i].h->ncards + 1);
        hands += games[i].h->H;
    }
    std::vector<std::vector<RecBox>> rec(ng);
    std::vector<std::vector<Tie>> listed(ng);
    std::vector<std::string> refused(ng);
    std::atomic<bool> fits{true};
    parallel_for(ng, hands, [&](int i) {
        const F64GameDesc &d = games[i];
        const HostGame &h = *d.h;
        auto refuse = [&](const char *w) {
            refused[i] = w;
            fits = false;
        };
        if (!fits) return;   // another game is refused: so is the batch
        if (h.k != 2) return refuse("one-card hands");
        if (h.hs % kBox != 0) return refuse("hand stride");
        const int nbox = h.hs / kBox;
        std::vector<RecBox> &rb = rec[i];
        rb.resize(nbox);     // (zeros)
        std::vector<Tie> &ties = listed[i];
        ties.reserve(h.H / 4);
        auto card = [&](int x, int j) { return h.hand_slots[2 * x + j]; };
        // a hand's cards as bits (a deck has at most 63)
        auto cards = [&](int x) { return 1ull << card(x, 0) | 1ull << card(x, 1); };
        for (int b = 0; b < nbox; ++b) {
            for (int k = 0; k < kBox / 2; ++k) {
                Rec &r = rb[b].r[k];
                const int x = kBox * b + 2 * k;
                // padding hands: weight 0, the spare card row
                auto off = [&](int hand, int j) { return (uint32_t)(hand < h.H ? card(hand, j) : h.ncards) * 16u; };
                r.oa1 = off(x, 0);
                r.ob1 = off(x, 1);
                r.oa2 = off(x + 1, 0);
                r.ob2 = off(x + 1, 1);
                if (x < h.H) { r.lin1 = d.lam_in[x]; r.lout1 = d.lam_out[x]; }
                if (x + 1 < h.H) {
                    r.lin2 = d.lam_in[x + 1];
                    r.lout2 = d.lam_out[x + 1];
                    r.ma = r.oa2 == r.oa1 || r.oa2 == r.ob1;
                    r.mb = r.ob2 == r.oa1 || r.ob2 == r.ob1;
                }
            }
            rb[b].first = (uint32_t)ties.size();
            uint32_t n = 0;
            for (int x = kBox * b; x < std::min(h.H, kBox * b + kBox); ++x)
                for (int q = h.group_lo[x]; q <= h.group_hi[x]; ++q)
                    if (q != x && (cards(x) & cards(q)) == 0) {
                        const Tie t{x - kBox * b, q, q > x ? d.lam_in[q] : -d.lam_in[q]};
                        if (n < kInline) rb[b].t[n] = t;
                        else ties.push_back(t);
                        ++n;
                    }
            rb[b].count = n;
        }
        // on average at most two corrections a hand
        if (ties.size() > 2 * (size_t)h.H) return refuse("many tied hands");
        // rows: showdown-only sequences with the fold-only one of their input row, then the others
        for (int s = 0; s < d.n_out; ++s)
            if (d.hfcol[s] < 0 && d.hscol[s] < 0) return refuse("an output sequence without terminals");
        const std::vector<int> mate = fold_mates(d.n_out, d.hfcol, d.hscol);
        for (int s = 0; s < d.n_out; ++s)
            if (d.hfcol[s] < 0) rows[i].push_back(make_int2(s, mate[s]));
        g[i].nunit = (int)rows[i].size();
        for (int s = 0; s < d.n_out; ++s)
            if (d.hfcol[s] >= 0 && mate[s] != kMate) rows[i].push_back(make_int2(s, -1));
        g[i].nrows = (int)rows[i].size();
    });
    for (int i = 0; i < ng; ++i) {
        if (!refused[i].empty()) {
            *why = refused[i];
            return nullptr;
        }
        rbytes += al(sizeof(RecBox) * rec[i].size() + sizeof(Tie) * listed[i].size());
        nrows += rows[i].size();
    }
    if (smem_bytes(nc) > (size_t)max_dyn_smem()) { *why = "shared memory"; return nullptr; }
    if (multi) {
        // items of at least `least` parts, more where the columns left fill
        // only one of the groups; returns their time, one after another on the
        // SM that is free first
        auto build = [&](int least, std::vector<int4> *out) {
            std::priority_queue<double, std::vector<double>, std::greater<double>> free_at;
            for (int k = 0; k < sms; ++k) free_at.push(0.0);
            double last = 0.0;
            for (int unit = 0; unit < 2; ++unit)     // the longer items first
                for (int i = 0; i < ng; ++i) {
                    const int n = unit ? g[i].nunit : g[i].nrows - g[i].nunit;
                    for (int c = 0; c < n;) {
                        int parts = least;
                        while (parts < kParts && n - c <= 16 / parts) parts *= 2;
                        const int e = std::min(n, c + 32 / parts);
                        if (out) out->push_back(make_int4(i, c, e, parts | (unit ? 8 : 0)));
                        const double t = free_at.top() + item_time(nc, games[i].h->hs / kBox, parts);
                        last = std::max(last, t);
                        free_at.pop();
                        free_at.push(t);
                        c = e;
                    }
                }
            return last;
        };
        int least = 1;
        double best = build(1, nullptr);
        for (int j = 2; j <= kParts; j *= 2) {
            const double t = build(j, nullptr);
            if (t < best) {
                best = t;
                least = j;
            }
        }
        build(least, &items);
    }
    const size_t o_items = al(sizeof(Game) * ng), o_rows = o_items + al(sizeof(int4) * items.size()),
                 o_rec = o_rows + al(sizeof(int2) * nrows), total = o_rec + rbytes;
    std::vector<unsigned char> host(total, 0);
    std::vector<size_t> rec_at(ng), rows_at(ng);
    for (size_t i = 0, ro = o_rec, rowo = o_rows; i < (size_t)ng; ++i) {
        rec_at[i] = ro;
        rows_at[i] = rowo;
        ro += al(sizeof(RecBox) * rec[i].size() + sizeof(Tie) * listed[i].size());
        rowo += sizeof(int2) * rows[i].size();
    }
    F64Plan *p = new F64Plan();
    cudaError_t e = device_malloc(&p->blob, total);
    if (e != cudaSuccess) {
        delete p;
        *need = total;
        *why = "device memory for the launch tables";
        return nullptr;
    }
    unsigned char *b = static_cast<unsigned char *>(p->blob);
    parallel_for(ng, hands, [&](int i) {
        const F64GameDesc &d = games[i];
        Game &x = g[i];
        x.H = d.h->H;
        x.hs = d.h->hs;
        x.nbox = d.h->hs / kBox;
        x.n_in = d.n_in;
        x.n_out = d.n_out;
        x.in_off = d.in_off;
        x.out_off = d.out_off;
        x.fcol = d.fcol;
        x.scol = d.scol;
        x.fcoef = d.fcoef;
        x.scoef = d.scoef;
        if (!rows[i].empty()) std::memcpy(host.data() + rows_at[i], rows[i].data(), sizeof(int2) * rows[i].size());
        x.rows = reinterpret_cast<const int2 *>(b + rows_at[i]);
        const size_t ties_at = rec_at[i] + sizeof(RecBox) * rec[i].size();
        std::memcpy(host.data() + rec_at[i], rec[i].data(), sizeof(RecBox) * rec[i].size());
        if (!listed[i].empty()) std::memcpy(host.data() + ties_at, listed[i].data(), sizeof(Tie) * listed[i].size());
        x.rec = reinterpret_cast<const RecBox *>(b + rec_at[i]);
        x.ties = reinterpret_cast<const Tie *>(b + ties_at);
    });
    std::memcpy(host.data(), g.data(), sizeof(Game) * ng);
    if (!items.empty()) std::memcpy(host.data() + o_items, items.data(), sizeof(int4) * items.size());
    e = cudaMemcpyAsync(p->blob, host.data(), total, cudaMemcpyHostToDevice, stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(stream);
    if (e != cudaSuccess) {
        f64_destroy(p);
        *need = total;
        *why = "uploading the launch tables";
        return nullptr;
    }
    p->a.games = reinterpret_cast<const Game *>(b);
    p->a.items = multi ? reinterpret_cast<const int4 *>(b + o_items) : nullptr;
    p->a.nc = nc;
    p->sms = sms;
    p->nitems = (int)items.size();
    if (!multi) {
        p->nunit = g[0].nunit;
        p->nother = g[0].nrows - g[0].nunit;
        p->nbox = g[0].nbox;
    }
    return p;
}

void f64_destroy(F64Plan *p) {
    if (!p) return;
    if (p->blob) cudaFree(p->blob);
    delete p;
}

int f64_items(const F64Plan *p) { return p->nitems; }

cudaError_t launch_f64_scan(F64Plan *p, const double *vin, double *vout, int batch, cudaStream_t stream) {
    Args a = p->a;
    a.vin = vin;
    a.vout = vout;
    a.batch = batch;
    long long n = p->nitems;
    if (!a.items) {
        const int sms = p->sms;
        const long long cu = (long long)p->nunit * batch, co = (long long)p->nother * batch;
        if (std::max(cu, co) > 0x7fffffe0LL) return cudaErrorInvalidValue;
        // the parts whose waves of items are shortest: 60 vectors of the river
        // game 119 us in items of 16 columns, 207 of 32, 141 of 8; 300 vectors of a
        // 6-card game (two boxes) 20 us of 32, 66 of 8
        auto items = [&](int j) { return (co + 32 / j - 1) / (32 / j) + (cu + 32 / j - 1) / (32 / j); };
        auto time = [&](int j) { return (double)((items(j) + sms - 1) / sms) * item_time(a.nc, p->nbox, j); };
        a.parts = 1;
        for (int j = 2; j <= kParts; j *= 2)
            if (time(j) < time(a.parts)) a.parts = j;
        const int w = 32 / a.parts;
        a.nother = (int)((co + w - 1) / w);
        n = a.nother + (cu + w - 1) / w;
    }
    if (n <= 0) return cudaSuccess;
    if (n > 0x7fffffffLL) return cudaErrorInvalidValue;
    const size_t smem = smem_bytes(a.nc);
    cudaError_t e = ensure_dyn_smem(reinterpret_cast<const void *>(f64_scan_kernel), smem);
    if (e != cudaSuccess) return e;
    f64_scan_kernel<<<(unsigned)n, 32 * kNW, smem, stream>>>(a);
    return cudaGetLastError();
}

}  // namespace kps
