// How a block of the level-2 kernel shares the columns of a row of C out to its
// threads. Plain C++, so that a host program can go through every thread and size.
#pragma once

namespace msp {

// A row of SP columns as SP / 2 pairs of neighbours over Threads threads: groups
// of SP / 2 threads take every groups-th row where that many fit, and a thread
// takes per_thread pairs, those at u + k Threads, where they do not.
template <int SP, int Threads>
struct L2Columns {
    static constexpr int pairs = SP / 2;
    static constexpr int groups = pairs >= Threads ? 1 : Threads / pairs;
    static constexpr int per_thread = (pairs + Threads - 1) / Threads;
    // row group of thread t; threads at or past `groups` groups have no columns
    static constexpr int group(int t) { return groups > 1 ? t / pairs : 0; }
    // first pair of thread t
    static constexpr int first(int t) { return groups > 1 ? t % pairs : t; }
    static constexpr bool active(int t) { return group(t) < groups && first(t) < pairs; }
    // whether an active thread's pair k lies in the row (1536 columns: 768 pairs, of
    // which only the first 256 of 512 threads have a second one)
    static constexpr bool has(int u, int k) {
        return pairs % Threads == 0 || per_thread == 1 || u + k * Threads < pairs;
    }
};

}  // namespace msp
