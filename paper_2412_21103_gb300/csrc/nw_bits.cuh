// Bit-sliced fills (nw_bits.cu: score-only batches; nw_bits_band.cu: the
// certified band with pointers): shared declarations and device helpers.
#pragma once

#include <string>
#include <vector>

#include "nw_internal.cuh"

namespace nw {

constexpr int64_t kPlanePad = 64;  // bases of padding in front of base 0 of the planar pool
constexpr int kBitsWarps = 8;      // warps per CTA

// Three-input logic operation with the truth table LUT (PTX lop3).
template <uint32_t LUT>
__device__ __forceinline__ uint32_t lop3(uint32_t a, uint32_t b, uint32_t c) {
    uint32_t d;
    asm("lop3.b32 %0, %1, %2, %3, %4;" : "=r"(d) : "r"(a), "r"(b), "r"(c), "n"(LUT));
    return d;
}
// Truth tables from the canonical inputs a = 0xF0, b = 0xCC, c = 0xAA.
constexpr uint32_t kA = 0xF0, kB = 0xCC, kC = 0xAA;
constexpr uint32_t lut(uint32_t v) { return v & 0xFFu; }
constexpr uint32_t kLutEq = lut(~(kA ^ kB) & ~kC);           // ~(a ^ b) & ~c
constexpr uint32_t kLutAndOrNot = lut(kA & (kB | ~kC));      // a & (b | ~c)
constexpr uint32_t kLutXor3 = lut(kA ^ kB ^ kC);             // a ^ b ^ c
constexpr uint32_t kLutAndNot = lut(kA & ~kB);               // a & ~b
constexpr uint32_t kLutXorAnd = lut((kA ^ kB) & kC);         // (a ^ b) & c
constexpr uint32_t kLutSel = lut((kA & kB) | (~kA & kC));    // a ? b : c
constexpr uint32_t kLutAndNotOr = lut(kA & (~kB | kC));      // a & (~b | c)
constexpr uint32_t kLutOrAndNot = lut((kA | kB) & ~kC);      // (a | b) & ~c

// The cell update for the scoring s' = 3 (match) / 1 (mismatch), the paper's
// +1/-1/-1, on 32 cells: inputs e (bases equal), a (dH of the cell above), b
// (dV of the cell to the left), outputs dV = T - a and dH = T - b with
// T = max(s', a, b).  A match acts like b = 3 on dV and like a = 3 on dH, so
// with f = "b acts as 3" and g the choice that orders a against b, each
// output bit is one three-input operation: 8 in all, where computing T and
// subtracting with borrows takes 12.  (Found by exhaustive search over pairs
// of intermediates; the truth tables were checked on all 32 inputs.)  The
// update is symmetric: swapping a and b swaps the outputs.  The outputs may
// name the inputs' registers.
constexpr uint32_t kLutF = 0xF8;  // e | (x & y)
constexpr uint32_t kLutG = 0x98;  // of (b1, a1, f)
constexpr uint32_t kLut1 = 0x46;  // high bit, of (a0, f, g)
constexpr uint32_t kLut0 = 0x29;  // low bit, of (a0, a1, g)
__device__ __forceinline__ void bits_cell(uint32_t e, uint32_t a0, uint32_t a1, uint32_t b0, uint32_t b1, uint32_t &H0,
                                          uint32_t &H1, uint32_t &V0, uint32_t &V1) {
    const uint32_t f = lop3<kLutF>(e, b0, b1), ft = lop3<kLutF>(e, a0, a1);
    const uint32_t g = lop3<kLutG>(b1, a1, f), gt = lop3<kLutG>(a1, b1, ft);
    V1 = lop3<kLut1>(a0, f, g);
    V0 = lop3<kLut0>(a0, a1, g);
    H1 = lop3<kLut1>(b0, ft, gt);
    H0 = lop3<kLut0>(b0, b1, gt);
}

// x * k + c as an integer multiply-add.  On sm_103 it issues on another pipe
// than the logic and shift operations (measured, lanes per clock and SM:
// LOP3, SHF, PRMT or add-max alone 60; multiply-add alone 60; LOP3 and
// multiply-adds 1:1 together 110), so a shift by a constant or a choice
// between a value and 0 costs the logic pipe nothing in this form.
__device__ __forceinline__ uint32_t muladd(uint32_t x, uint32_t k, uint32_t c) {
    uint32_t d;
    asm("mad.lo.u32 %0, %1, %2, %3;" : "=r"(d) : "r"(x), "r"(k), "r"(c));
    return d;
}
__device__ __forceinline__ uint32_t mul(uint32_t x, uint32_t k) { return muladd(x, k, 0u); }

// 32 bits of a planar sequence plane starting at global base index g.
__device__ __forceinline__ uint32_t plane_window(const uint32_t *pl, int64_t g) {
    const uint64_t x = (uint64_t)(g + kPlanePad);
    return __funnelshift_r(__ldg(pl + (x >> 5)), __ldg(pl + (x >> 5) + 1), (uint32_t)x & 31u);
}

// The two planes of s' for a general scoring with 0 <= s'x <= s'm <= 3:
// bit k of s'(match) / s'(mismatch) as all-ones or zero words.
struct BitsScoring {
    uint32_t M1, M0, X1, X0;
};

// One pair of a score-only launch: byte offsets in the pool, the first words
// of its sequences' planar slots, and its score's destinations.
struct BitsTask {
    uint64_t a_off, b_off;
    uint32_t aw, bw;
    uint32_t m, n;
    uint32_t out0, out1;  // out1 == ~0u: none
};

// All-vs-all launches name their pairs instead of listing them.  The
// sequences are sorted longest first; a class holds the rows [r0, r1) of
// equal shape (words a lane, stripes), and its pairs are all (column c < row r), by c and then
// r, so that 32 consecutive pairs have one shape and nearly one width.
struct BitsSeq {
    uint32_t w, len, id;  // first word of the planar slot, bases, index in the caller's list
};
struct BitsClass {
    uint32_t r0, r1;
};

struct BitsJob {
    uint64_t T;        // chunks in all (of the job's widest pair)
    uint32_t t0, cnt;  // tasks (or pairs of the class) [t0, t0 + cnt), cnt <= 32, one per lane
    uint32_t S, C;     // stripes, chunks from one to the next
    uint32_t K;        // words a lane
    uint32_t cls;      // all-vs-all: the class
};

struct BitsArgs {
    const uint32_t *pl0, *pl1;  // planar sequences: bit k of global base g at word (g+64)>>5, bit (g+64)&31
    const BitsTask *tasks;      // or, all-vs-all:
    const BitsSeq *seqs;
    const BitsClass *classes;
    uint32_t nseq;
    const BitsJob *jobs;
    uint32_t njobs;
    uint32_t *counter;
    uint2 *rows;          // per warp: rows_chunks x 32 lanes of (plane 0, plane 1) words
    uint32_t rows_chunks;
    int32_t *scores;
    uint32_t score_cap;
    int32_t unit, gap;  // score = unit * W + gap * (m + n)
    BitsScoring g;
    uint32_t *err;
};

// Planar copy of the sequences a launch reads.  Each distinct sequence
// (pool byte offset, length) gets a slot of whole 32-base words, two words
// apart; a kernel addresses base i of the sequence as global base index
// slot + i.  Only the launch's own sequences are copied, wherever they lie
// in the pool.
struct PlaneSeg {
    uint64_t src;      // pool byte offset of the sequence (its device address when the pool is null)
    uint32_t nbytes;   // its packed bytes
    uint32_t dst;      // first word of its slot
};
class PlaneSet {
  public:
    // Room for n sequences without regrowing.
    void reserve(size_t n);
    // Slot (global base index of base 0) of the sequence at pool byte `off`
    // with `len` bases, added on first use.
    int64_t add(uint64_t off, uint32_t len);
    // Scratch that a sequence of `len` bases takes: its words in both planes and its segment.
    static uint64_t bytes_of(uint32_t len) { return ((uint64_t)(len + 31) / 32 + 2) * 8 + sizeof(PlaneSeg); }
    // First word of a slot that add() returned.
    static uint32_t word_of(int64_t slot) { return (uint32_t)((slot + kPlanePad) / 32); }
    // Room for `words` words of slots laid out by the caller from word 2 on.
    void reserve_words(uint64_t words) { words_ += words; }
    // Enqueues the copy (one H2D table, one kernel); pl0 / pl1 receive the
    // two planes, max_base the largest base index a 32-bit window may start at.
    // With a null pool the offsets given to add() are device addresses.
    int launch(nw_ctx *ctx, const uint8_t *pool, const std::string &prefix);
    // Uploads the segment table and sizes the planes without copying (the
    // copy can then be enqueued, also into a graph, by enqueue()).
    int prepare(nw_ctx *ctx, const std::string &prefix);
    int enqueue(nw_ctx *ctx, const uint8_t *pool) const;
    const uint32_t *pl0 = nullptr, *pl1 = nullptr;
    int64_t max_base = 0;
    uint32_t *planes() const { return planes_; }
    uint64_t plane_words() const { return words_ + 4; }  // words from one plane to the next

  private:
    // open addressing (linear probing, at most half full): one table of
    // entries instead of a node per sequence
    struct Entry {
        uint64_t off;
        uint32_t len, used;
        int64_t slot;
    };
    std::vector<Entry> table_;
    size_t count_ = 0;
    void rehash(size_t size);
    std::vector<PlaneSeg> segs_;
    uint64_t words_ = 2;  // kPlanePad bases in front of the first slot
    PlaneSeg *dsegs_ = nullptr;
    uint32_t *planes_ = nullptr;
};

// Everything a launch needs, prepared (sorted, uploaded, scratch sized)
// ahead of the launch so that the launch itself only enqueues kernels.
struct BitsPlan {
    BitsArgs ba{};
    uint32_t blocks = 0;
    uint32_t wide = 0;        // leading jobs of 2^32 chunks or more
    const uint8_t *pool = nullptr;
    uint32_t ntasks = 0;      // tasks whose sequences have slots of their own
    PlaneSet planes;          // or the distinct sequences
    bool gen = false;
};

// A scoring's two values s' = s - 2*gap in units of their greatest common
// divisor: every W is a multiple of it, so the recurrence, its ties and its
// pointers are the same on W / unit, and only the scores are scaled back.
struct BitsUnits {
    int32_t sm, sx, unit;
    bool gen() const { return !(sm == 3 && sx == 1); }
    BitsScoring planes() const {
        return BitsScoring{(sm & 2) ? ~0u : 0u, (sm & 1) ? ~0u : 0u, (sx & 2) ? ~0u : 0u, (sx & 1) ? ~0u : 0u};
    }
};
BitsUnits bits_units(const nw_scoring &sc);
// 0 <= s'(mismatch) <= s'(match) <= 3: every difference fits two bits.
bool bits_scoring_ok(const nw_scoring &sc);
// The same in units, for batches: +2/-1/-2 (s' = 6, 3) runs as 2, 1 in units
// of 3.  1,001 pairs of 300 to 2,500 bases with alignments: 0.57 against 2.80 ms of
// fill on the scalar kernel.  Single pairs and all-vs-all matrices keep the
// rule above: their scalar kernels' shapes are what saved tunings hold for
// such scorings.
bool bits_batch_ok(const nw_scoring &sc);
// Orients, groups and uploads the tasks, sizes the scratch; scores[out0] (and
// scores[out1]) receive each task's score.
int bits_prepare(nw_ctx *ctx, const uint8_t *pool, const std::vector<BatchTask> &tasks, const nw_scoring &sc,
                 int32_t *scores, uint32_t score_cap, const std::string &prefix, BitsPlan *plan);
// Hands a plan's scratch back (after a plan that did not fit).
void bits_release(nw_ctx *ctx, const std::string &prefix);
// The same for every pair of nseq sequences (the off-diagonal entries of the
// nseq x nseq matrix `scores`).
int bits_prepare_all(nw_ctx *ctx, const uint8_t *pool, const uint64_t *off, const uint32_t *len, uint32_t nseq,
                     const nw_scoring &sc, int32_t *scores, const std::string &prefix, BitsPlan *plan);
// Enqueues the planar copy of the pool and the fill (no host copies: it can
// be captured into a graph).
int bits_launch(nw_ctx *ctx, const BitsPlan &plan);

// ---- one long pair on the bit-sliced stripes (nw_bits_pair.cu)
// Whether the pair runs there (the paper's scoring, long enough to spread
// over several warps, every warp co-resident, pointers within the budget).
bool bits_pair_takes(nw_ctx *ctx, uint32_t m, uint32_t n, const nw_scoring &sc, bool want);
// Score (and with `want` the CIGAR, written by the CIGAR assembly) of one pair.
int bits_pair(nw_ctx *ctx, const uint8_t *a2b, uint32_t m, const uint8_t *b2b, uint32_t n, const nw_scoring &sc,
              bool want, uint32_t mflag, int32_t *score, char *cigar, uint64_t *cigar_len);
// Many pairs, each on its own warps: waves of pairs whose warps are all
// resident at once, longest chains first.  a_off / b_off: byte offsets into
// `pool` (device addresses when it is null).  Every job must pass
// bits_pair_takes.
struct PairJob {
    uint64_t a_off, b_off;
    uint32_t m, n;
    int32_t *score;
    char *cigar;
    uint64_t *cigar_len;
};
int bits_pairs(nw_ctx *ctx, const uint8_t *pool, const std::vector<PairJob> &jobs, const nw_scoring &sc, bool want,
               uint32_t mflag);

// Many pairs with alignments, each on a group of lanes of one warp, in waves
// whose records fit the budget (any lengths, also 0; want is implied).
int bits_groups(nw_ctx *ctx, const uint8_t *pool, const std::vector<PairJob> &pairs, const nw_scoring &sc,
                uint32_t mflag);
double bits_group_seconds(uint32_t m, uint32_t n);  // estimated time of a pair on one warp there
uint64_t bits_group_bytes(uint32_t m, uint32_t n);  // its records on a whole warp

// ---- the certified band on the bit-sliced window (nw_bits_band.cu)
// Window of one pair: g lanes (a power of two) x Q words of 32 rows, its
// anchor diagonal hi (the band's upper diagonal raised to the parity of
// m+n), and its anti-diagonals a_first .. m+n in chunks of 64.
struct BandBitsShape {
    uint32_t g = 1, Q = 1, nchunks = 0;
    int32_t hi = 0, a_first = 0;
    uint32_t words = 1;  // the band needs this many 32-row words (g * Q >= words)
};
// One banded pair of a round: pool offsets, sizes, score slot, window, and
// its first kept planes (16 bytes per word, every 64 anti-diagonals).
struct BandBitsItem {
    uint64_t a_off, b_off, ptr_off;  // pool byte offsets (the CIGARs), first kept planes
    int64_t a_slot, b_slot;          // the sequences' planar slots (the fill and the walk)
    uint32_t m, n, out0;
    BandBitsShape shape;
};
// Most words per lane of the throughput shape: 4, or NW_BBAND_MAXQ (1..4)
// when set (read on each call; a round reads it once).
int band_bits_max_q();
// The window of the band of diagonals [lo, hi] on the fewest lanes of at
// most max_q words each; false when it needs more than 128 words (4,096
// rows).
bool band_bits_shape(uint32_t m, uint32_t n, int32_t lo, int32_t hi, BandBitsShape *s, int max_q);
// The same window spread over twice the lanes: fewer instructions per lane and
// step, so a shorter time for the pair; false when it cannot be spread further.
bool band_bits_spread(BandBitsShape *s);
uint64_t band_bits_cells(const BandBitsShape &s);  // cells of the pair's window, over all its chunks
uint64_t band_bits_kept(const BandBitsShape &s);   // its kept planes (16-byte units)
// Bytes an alignment takes there beside the planar copy: kept planes, moves and
// its entries in the tables of fill and walk.
uint64_t band_bits_scratch(uint32_t m, uint32_t n, const BandBitsShape &s);
// The widest half-width whose band fits the window of an m x n pair.
uint32_t band_bits_max_width(uint32_t m, uint32_t n);
double band_bits_seconds(const BandBitsShape &s);    // estimated time of the pair on one warp
// Fills the items (the paper's scoring: s' = 3 on a match, 1 on a
// mismatch), writes scores[out0], returns the banded scores in item order,
// and with `want` the kept planes at ptr + ptr_off (`kept` units in all).
int band_bits_fill(nw_ctx *ctx, const PlaneSet &planes, const std::vector<BandBitsItem> &items, bool want, int32_t gap, int32_t *scores, uint32_t score_cap,
                   void *ptr, uint64_t kept, std::vector<int32_t> &banded);
// Walks the items `which` of a filled wave and writes their CIGARs.
int band_bits_walk(nw_ctx *ctx, const PlaneSet &planes, const void *ptr, const std::vector<BandBitsItem> &items,
                   const std::vector<uint32_t> &which, const uint8_t *pool, char *cigar_pool,
                   const uint64_t *cigar_off, uint64_t *cigar_len, uint32_t mflag);

}  // namespace nw
