// unit_split.h -- how the CTAs of a column tile share the units of a matrix
// (rnn_step.cuh): a unit is a row of a product, or a hidden unit of a cell with
// all its gate rows, and every CTA ("member") owns a contiguous range of them.
// Host only, plain C++.
//
// Equal numbers of units are equal work only where the block sizes are mixed.
// Where rows of one block size lie together, as in a matrix whose first tenth
// keeps a weight in 4 and whose rest keeps one in 64, the member with the dense
// rows has 6 times the mean.  The ranges then follow the units' cost instead.
#pragma once

#include <algorithm>
#include <atomic>
#include <cstdint>
#include <new>
#include <vector>

namespace darb {

constexpr int kMaxMembers = 160;   // members, at most (a GB300 has 152 SMs)

// Two ways to give `members` members their ranges: equal numbers, member q
// owning units [units * q / members, units * (q + 1) / members), or by cost,
// [start[q], start[q + 1]).
struct UnitRanges {
    int64_t busiest;      // cost of the busiest member
    int32_t most_units;   // units of the member that has most
};
struct UnitSplit {
    UnitRanges equal, by_cost;
    bool prefer_by_cost;
    int32_t start[kMaxMembers + 1];
};

class UnitSplits {
public:
    UnitSplits() = default;
    UnitSplits(const UnitSplits &) = delete;
    UnitSplits &operator=(const UnitSplits &) = delete;
    ~UnitSplits() {
        for (auto &s : kept_) delete s.load(std::memory_order_relaxed);
    }

    // cost(u): of unit u, at least 1
    template <class Cost>
    void build(int64_t units, Cost cost) {
        prefix_.resize(static_cast<size_t>(units) + 1);
        prefix_[0] = 0;
        for (int64_t u = 0; u < units; ++u)
            prefix_[static_cast<size_t>(u) + 1] = prefix_[static_cast<size_t>(u)] + cost(u);
    }

    int64_t units() const { return static_cast<int64_t>(prefix_.size()) - 1; }
    int64_t total() const { return prefix_.back(); }

    // The split over `members` (1 .. min(units, kMaxMembers)).  Worked out by the
    // first call that asks for it (some microseconds) and kept; any thread may
    // call.  Without memory to keep it, it is worked out in `local`.
    const UnitSplit &get(int members, UnitSplit &local) const {
        std::atomic<UnitSplit *> &slot = kept_[members];
        if (const UnitSplit *s = slot.load(std::memory_order_acquire)) return *s;
        UnitSplit *s = new (std::nothrow) UnitSplit;
        if (s == nullptr) {
            work_out(members, local);
            return local;
        }
        work_out(members, *s);
        UnitSplit *first = nullptr;
        if (slot.compare_exchange_strong(first, s, std::memory_order_acq_rel)) return *s;
        delete s;   // another thread was faster
        return *first;
    }

private:
    void work_out(int members, UnitSplit &s) const {
        const int64_t n = units(), all = total();
        const int64_t *const p = prefix_.data();
        s.equal = {0, static_cast<int32_t>((n + members - 1) / members)};
        for (int q = 0; q < members; ++q)
            s.equal.busiest = std::max(s.equal.busiest, p[n * (q + 1) / members] - p[n * q / members]);
        // by cost: a member ends with the unit that brings the running sum nearest
        // to its share, and leaves one unit for every later member
        s.by_cost = {0, 0};
        s.start[0] = 0;
        for (int q = 0; q < members; ++q) {
            const int64_t from = s.start[q], last = n - (members - 1 - q);
            int64_t to = last;
            if (q + 1 < members) {
                const int64_t share = all / members * (q + 1) + all % members * (q + 1) / members;
                to = std::lower_bound(p + from + 1, p + last, share) - p;
                if (to > from + 1 && p[to] - share > share - p[to - 1]) --to;
            }
            s.start[q + 1] = static_cast<int32_t>(to);
            s.by_cost.busiest = std::max(s.by_cost.busiest, p[to] - p[from]);
            s.by_cost.most_units = std::max(s.by_cost.most_units, static_cast<int32_t>(to - from));
        }
        // Equal numbers unless the busiest member gets 5% less: their members have
        // equally many outputs to form at the end, and their ranges need no table
        s.prefer_by_cost = s.by_cost.busiest * 20 < s.equal.busiest * 19;
    }

    std::vector<int64_t> prefix_ = {0};
    mutable std::atomic<UnitSplit *> kept_[kMaxMembers + 1] = {};
};

}  // namespace darb
