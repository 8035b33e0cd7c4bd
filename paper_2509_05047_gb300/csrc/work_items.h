// work_items.h -- how a batch's requests are cut into work items (host code,
// no CUDA: also compiled by the CPU tests).
//
// A CTA that ends an item drains its slots before it takes the next one (about
// 30 us beside its neighbours), and items left over after whole rounds of the
// grid run on an idle chip.  So each request is cut into the fewest equal
// items that fill whole rounds (chunks_per_cta of them at least, at most
// max_chunk histories each).  Against two or more items a CTA of at least 1024
// histories: small scanner, 1e6 histories 121 -> 88 us, 2e4 39 -> 32 us; 1e8
// through the gaps scanner (5.02 rounds of 65536 before, now 6 of 54826) 7.82 ->
// 7.13 ms; six uneven requests 7.35 -> 7.25 ms.
//
// A batch's requests share the rounds.  Cut each for itself, 32 requests of
// 20,000 histories gave a CTA 17 items of 128 to drain (376 us, and 711 us for
// 32 of 60,000; 181 and 356 us with items of 1024), so an item of a batch is
// at least the batch's share of a CTA over the rounds that pay: one while the
// share is below two items of kRoundHistories, and never more than kBatchItems
// (32 uneven requests: 7.66 ms, with 128 7.79 ms).
#ifndef PSC_WORK_ITEMS_H
#define PSC_WORK_ITEMS_H

#include <algorithm>

namespace psc {

constexpr unsigned long long kMaxChunk = 1ull << 16;  // histories of a work item (a slot holds 16 bits of the index)
constexpr unsigned long long kMinChunk = 128, kRoundHistories = 1024, kBatchItems = 32;

// chunk[j]: histories per item of request j, of n[j] >= 1 histories
inline void work_items(const unsigned long long* n, int jobs, unsigned long long grid, unsigned long long chunks_per_cta,
                       unsigned long long max_chunk, unsigned long long* chunk) {
  const unsigned long long most = std::min(kMaxChunk, std::max<unsigned long long>(1024, max_chunk));
  unsigned long long least = kMinChunk;
  if (jobs > 1) {
    unsigned long long share = 0, rest = 0;  // (per CTA: the sum of all histories may exceed 64 bits)
    for (int j = 0; j < jobs; ++j) {
      share += n[j] / grid;
      rest += n[j] % grid;
    }
    share += rest / grid + (rest % grid != 0);
    const unsigned long long rounds = std::min(kBatchItems, std::max(1ull, share / kRoundHistories));
    least = std::max(kMinChunk, share / rounds + (share % rounds != 0));
  }
  for (int j = 0; j < jobs; ++j) {
    const unsigned long long per_cta = n[j] / grid + (n[j] % grid != 0);
    const unsigned long long rounds = std::max(chunks_per_cta, per_cta / most + (per_cta % most != 0));
    const unsigned long long per = std::min(most, std::max(least, per_cta / rounds + (per_cta % rounds != 0)));
    const unsigned long long items = n[j] / per + (n[j] % per != 0);
    chunk[j] = n[j] / items + (n[j] % items != 0);
  }
}

}  // namespace psc

#endif
