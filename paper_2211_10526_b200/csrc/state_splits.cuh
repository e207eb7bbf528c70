// How many CTAs share the tokens of a plane in the state kernel of the tensor-core path (csrc/tc_state.cu), and how their sums meet.  Host
// arithmetic only.  A tile is a stage of that kernel: 128 rows of 128 bytes.
#pragma once

namespace castling {
namespace tc {

constexpr int kMaxSplits = 64, kMaxCluster = 8;

// The number of splits of at most P, all of equal size but the last, that leaves none of them empty.
inline int even_splits(int tiles, int P) {
    const int per = (tiles + P - 1) / P;
    return (tiles + per - 1) / per;
}

// Two state CTAs fit on a multiprocessor: as many splits as keep all CTAs of the launch resident at once.  The workspace is sized for these.
inline int most_splits(int planes, int tiles, int sms) {
    if (tiles < 1) return 1;
    int P = 2 * sms / planes;
    if (P > tiles) P = tiles;
    if (P > kMaxSplits) P = kMaxSplits;
    return even_splits(tiles, P < 1 ? 1 : P);
}

struct StateSplits {
    int P;            // at most most_splits
    bool clustered;   // the splits of a plane are one cluster and add their states through distributed shared memory; else they meet in memory
};

// fit(P): clusters of P that the device holds at once while it is empty; a few less find room at once.
//
// Meeting in memory costs about 3 us where it takes two levels (from five splits on), 0.5 us where it takes one; a cluster costs less, but it
// starts only where P CTAs find room in one part of the device.  Us per forward from a graph, memory / cluster:
//   clusters that all fit at once: width 64, 42 planes of 12 tiles, P = 6 20.5 / 17.9, 66 of 12, P = 4 22.3 / 21.8, 128 of 6, P = 2 21.2 / 20.8;
//     some that do not (72 against 71): 72 planes of 12 tiles, P = 4 22.8 / 25.5, 37 of 16, P = 8 19.9 / 22.6, 49 of 32, P = 6 36.3 / 40.8; those that
//     fit in number, but not at once: 92 against 93, P = 3 27.2 / 31.5, 87 34.0 / 35.1 (84 25.2 / 24.7);
//   width 32, whose CTAs have more work to overlap: P = 5 to 8 as above (49 planes of 15 tiles, P = 5 19.3 / 17.8), P = 2 to 4 only where each CTA has a
//     multiprocessor of its own: 16 planes of 4 tiles 9.4 / 8.7, 37 9.6 / 9.8, 64 of 15 tiles 21.8 / 22.1.
// More than eight splits become eight that meet in a cluster unless that gives a CTA many more tiles in a row (0.55 us each at width 64):
// 16 planes of 128 tiles, 8 tiles more, 43.9 / 42.3, one plane of 64 tiles, 7 more, 14.2 / 12.8, one of 94 tiles, 10 more, 14.1 / 15.5, 9 of 128, 12 more,
// 32.0 / 32.3; width 32: 16 planes of 32 tiles, 2 more, 17.4 / 16.5, of 64 tiles, 4 more, 24.1 / 24.7.
template <typename Fit>
inline StateSplits state_splits(int planes, int tiles, int sms, bool narrow, Fit fit) {
    int P = most_splits(planes, tiles, sms);
    auto room = [&](int n) { return 100 * planes <= (n > 4 ? 94 : 93) * fit(n); };   // up to four there is less to gain
    if (P > kMaxCluster) {
        const int more = (tiles + kMaxCluster - 1) / kMaxCluster - (tiles + P - 1) / P;
        if (more > (narrow ? 3 : 8) || !room(kMaxCluster)) return {P, false};
        P = even_splits(tiles, kMaxCluster);
    }
    return {P, P > 1 && (P > 4 || !narrow || planes * P < sms) && room(P)};
}

}  // namespace tc
}  // namespace castling
