// Per-box hand records of the staged scan kernels (kernels_tma.cu for one
// game and many vectors, kernels_amulti.cu for many games), built on the
// host once per game and direction (scan_records.cpp).
//
// The scan walks hands in library order (strength, then canonical index) in
// boxes of 16 hands; a chunk of consecutive boxes goes to each of four warps.
// For every pair of hands (2i, 2i+1) the scan reads a TmaScanRec and the
// finishing pass a TmaFinRec:
//   oa*, ob*  byte offsets of the hands' card rows in a warp's per-card table
//             (card * 128; the spare row ncards * 128 for padding hands and
//             for the second card of one-card hands),
//   lin*      input weights lambda_in (0 for padding hands),
//   ma, mb    1 when the first / second card of hand 2i+1 is a card of hand
//             2i, else 0,
//   lout*     output weights lambda_out; the finishing records repeat lin*.
// A box's scan block is its 8 pair records followed by two tie words: byte
// 8j + (k - 4j) of word j (pair k) has
//   bits 2-4  hand 2k has a compatible tied hand 1, 2, 3 positions before it
//   bits 5-7  the same for hand 2k+1.
// Chunk boundaries fall on box boundaries that cut no tie group of up to 4
// hands.  Longer groups are refused, or (long_ties) listed: the last 8 bytes of
// a box's scan block are {first, count} into the TieEntry list, one entry per
// ordered pair of compatible hands of such a group; those hands have no tie
// bits, and chunk boundaries may cut the group (the scan counts every earlier
// hand as weaker, whichever chunk it is in, and an entry undoes that).
#pragma once

#include <cstdint>
#include <string>
#include <vector>

#include "game.h"

namespace kps {

constexpr int kTmaBox = 16;        // hands per box
constexpr int kTmaWarps = 4;       // chunks per CTA

struct alignas(16) TmaScanRec {
    uint32_t oa1, ob1, oa2, ob2;
    float lin1, lin2, ma, mb;
};
constexpr int kScanBlock = 8 * 32 + 16;   // bytes per box
struct alignas(16) TieEntry {
    int i, q;                      // hand 16 box + i, its tied partner q
    float lin;                     // lambda_in[q] when q comes later, - lambda_in[q] when earlier
    int pad;
};
constexpr int kMaxTieEntries = 256;       // per chunk of a box row
struct alignas(16) TmaFinRec {
    uint32_t oa1, ob1, oa2, ob2;
    float lout1, lout2, lin1, lin2;
};

// Records of one game and direction.  bytes = nbox scan blocks, nbox * 8
// finishing records, the tie entries.
struct ScanRecords {
    int H = 0, hs = 0, nc = 0, k = 0, nbox = 0;
    int extra = 0;                 // boxes of the longest chunk past 16
    int bchunk[kTmaWarps + 1] = {0, 0, 0, 0, 0};
    size_t entries_at = 0;         // byte offset of the tie entries
    std::vector<unsigned char> bytes;
};

// Pairs of output sequences with one input row: where a player answers a bet by a
// fold or a call, both answers read the bet's row, one as a fold-only and one as
// a showdown-only sequence (hfcol, hscol: a sequence's fold / showdown input row or
// -1).  Returns for every sequence the fold-only one of its pair (a showdown-only
// sequence takes the first fold-only one of its row that is not taken), kMate
// for a fold-only sequence that is in one, and -1 for one left alone.
constexpr int kMate = -2;
std::vector<int> fold_mates(int n_out, const int *hfcol, const int *hscol);

// Empty string on success, else why the game does not fit these kernels
// (tie group over 4 hands or, with long_ties, more than kMaxTieEntries pairs in a
// chunk; more than 64 card rows; a chunk longer than 16 + max_extra boxes).
std::string build_scan_records(const HostGame &h, const double *lam_in, const double *lam_out, int max_extra,
                               bool long_ties, ScanRecords *out);

}  // namespace kps
