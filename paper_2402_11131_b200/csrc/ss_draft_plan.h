// How the next draft cuts its rows into CTAs.  Host code without CUDA, so that the rule and its ways out can be checked without a GPU.
#pragma once

namespace ss {

constexpr int kDraftThreads = 512;    // few rows: a segment of up to 16384 logits is one batch of loads (eight float4 a thread)
constexpr int kDraftBatch = kDraftThreads * 32;
constexpr int kPortableCtas = 8;      // of a cluster
constexpr int kMaxClusterCtas = 16;   // what sm_100a takes besides

// words that the longest segment of a row of `vocab` logits spans when n CTAs take it (see make_segment): whole vectors, and up to three words
// before an unaligned start
inline int draft_segment_words(int vocab, int n) { return (((vocab + n - 1) / n + 3) & ~3) + (vocab % 4 != 0 ? 3 : 0); }

// CTAs per row, all rows of a sequence in one cluster.  Up to 8 CTAs, and up to 16 (`most`) for a few sequences where a CTA's segment is then one
// batch of loads instead of two (whose candidates would be read again).  One sequence and six, 8 / 16: three rows of 51200 logits 5.2 / 4.2 and
// 5.9 / 4.8 us, of 32769 5.15 / 4.75 and 5.9 / 5.45, four rows of 50257 5.9 / 4.6 and 6.5 / 5.3; but of sixteen sequences the clusters no
// longer run all at once, 7.75 / 10.3; four rows of 32000, one batch already, 4.0 / 4.0.  Not for a single row, whose 16 lists one warp would rank:
// 131100 logits 4.65 / 5.25, eight best of 140000 6.55 / 9.4, 200000 5.55 / 5.4.
inline int draft_ctas(int batch, int gamma, int vocab, int most) {
    int n = 1;
    while (vocab / (n * 2) >= kDraftThreads * 4 &&
           (gamma * n * 2 <= kPortableCtas || (batch <= 6 && gamma > 1 && draft_segment_words(vocab, n) > kDraftBatch && gamma * n * 2 <= most))) n *= 2;
    return n;
}

// launch(CTAs per row), which gives 0 or an error.  More than 8 CTAs cannot be placed on every part of a GPU: then 8 at most take the sequence, whether
// fits(CTAs) says so beforehand or the launch.
template <typename Fits, typename Launch>
inline auto launch_draft(int batch, int gamma, int vocab, Fits&& fits, Launch&& launch) -> decltype(launch(1)) {
    const int narrow = draft_ctas(batch, gamma, vocab, kPortableCtas);
    int n = draft_ctas(batch, gamma, vocab, kMaxClusterCtas);
    if (n != narrow && !fits(gamma * n)) n = narrow;
    const auto err = launch(n);
    return err != decltype(err)(0) && n != narrow ? launch(narrow) : err;
}

}  // namespace ss
