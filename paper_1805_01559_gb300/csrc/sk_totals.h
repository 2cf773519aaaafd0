// The counted totals of the persistent solver's sweeps: words that several CTAs add to and all
// of them wait for.  Plain C++ apart from the function qualifiers, so that the protocol can be
// stepped on the host.
//
// A sweep's row of totals has a 64-bit word per column and two for the row residual.  The words
// carry their own completion: every addition includes 1 << 56, and a reader, which knows what
// the word held when the row was last complete, has the sweep's total once the difference
// counts all additions that are due.  So no barrier stands between the sweep and the column
// update, and nothing is cleared.  Each of the V partitions adds to every word of the row; the
// values of a sweep stay below 2^56 together.
//
// Sweep s adds into row s mod 2, so a row is added to again two sweeps later.  A CTA does that
// only after it has seen the other row's residual words complete, and to those EVERY CTA has
// added after it read this row: the owners of partitions with their residuals, and a CTA
// without a partition (a group of more CTAs than its instance has partitions) with a bare
// count.  Without the latter nothing would keep the owners from adding sweep s + 2 to a row that
// such a CTA is still reading.
#pragma once

#include <stdint.h>

#ifdef __CUDACC__
#define OTA_HD __host__ __device__ __forceinline__
#else
#define OTA_HD inline
#endif

namespace ota {

static constexpr int FX_BITS = 40;   // a column total of q^_j is about 2^40 units
static constexpr int FX_TOP = 48;    // partials (and totals) from 2^48 on go to the exact path
static constexpr int FX_ERR = 50;    // row residuals in units of 2^-50
static constexpr int FX_COUNT = 56;  // bit position of the count of additions
static constexpr uint64_t FX_ONE = 1ull << FX_COUNT;

// Partitions [v0, v1) of CTA b of nb; none when there are fewer partitions than CTAs before it.
OTA_HD void cta_parts(int V, int b, int nb, int* v0, int* v1) {
    *v0 = (int)((int64_t)V * b / nb);
    *v1 = (int)((int64_t)V * (b + 1) / nb);
}
// Additions due to a column's word, and to a residual word: one a partition, and one for each
// of the nb - V CTAs that own none (with nb <= V every CTA owns one).  At most 255 fit the count.
OTA_HD int fx_due_col(int V) { return V; }
OTA_HD int fx_due_err(int V, int nb) { return V > nb ? V : nb; }
// What was added to a word since it held `was`: complete when `due` additions have arrived.
OTA_HD bool fx_complete(uint64_t now, uint64_t was, int due) { return ((now - was) >> FX_COUNT) == (uint64_t)due; }
OTA_HD uint64_t fx_value(uint64_t now, uint64_t was) { return (now - was) & (FX_ONE - 1); }

// The row residual sum p^ |r - 1|, in units of 2^-FX_ERR.  That of a plan of unit mass is at most
// 2, that is 2^51 units, and may come from one partition, so V of them do not fit below the
// count; each adds its low 48 bits to one word and the rest to another.  A row whose residual
// is 4 or more, infinite or not a number counts as FX_BROKEN units, and a total from there on never
// passes the loop test: no plan of unit mass has it, whatever tolerance was asked for.
static constexpr uint64_t FX_BROKEN = 1ull << (FX_ERR + 2);
OTA_HD uint64_t fx_err_low(uint64_t e) { return e & ((1ull << FX_TOP) - 1); }
OTA_HD uint64_t fx_err_high(uint64_t e) { return e >> FX_TOP; }
OTA_HD uint64_t fx_err(uint64_t low, uint64_t high) { return low + (high << FX_TOP); }
// The loop test's bound for a tolerance in units.
OTA_HD uint64_t fx_stop_units(double t) { return t < (double)FX_BROKEN ? (uint64_t)t : FX_BROKEN - 1; }

}  // namespace ota
