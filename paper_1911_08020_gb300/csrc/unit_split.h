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

    // Units of `gates` rows, unit u rows u, units + u, 2 units + u ...; prefix[r]:
    // the cost of rows [0, r), at least 1 each, kept by the caller.
    void set(const int64_t *prefix, int64_t units, int gates) {
        prefix_ = prefix;
        units_ = units;
        gates_ = gates;
    }

    int64_t total() const { return prefix_[units_ * gates_]; }

    // The split over `members` (1 .. min(units, kMaxMembers)).  Worked out by the
    // first call that asks for it (about a microsecond) and kept; any thread may
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
        const int64_t n = units_, all = total();
        auto p = [&](int64_t u) {   // the cost of units [0, u)
            int64_t c = prefix_[u];
            for (int q = 1; q < gates_; ++q) c += prefix_[q * n + u] - prefix_[q * n];
            return c;
        };
        s.equal = {0, static_cast<int32_t>((n + members - 1) / members)};
        for (int64_t q = 0, before = 0; q < members; ++q) {
            const int64_t upto = p(n * (q + 1) / members);
            s.equal.busiest = std::max(s.equal.busiest, upto - before);
            before = upto;
        }
        // by cost: a member ends with the unit that brings the running sum nearest
        // to its share, and leaves one unit for every later member
        s.by_cost = {0, 0};
        s.start[0] = 0;
        int64_t before = 0;
        int64_t length = n / members;   // of the range before: about that of the next
        for (int q = 0; q < members; ++q) {
            const int64_t from = s.start[q], last = n - (members - 1 - q);
            int64_t to = last;
            if (q + 1 < members) {
                const int64_t share = all / members * (q + 1) + all % members * (q + 1) / members;
                to = std::min(from + std::max<int64_t>(length, 1), last);   // the first unit past the share
                while (to < last && p(to) < share) ++to;
                while (to > from + 1 && p(to - 1) >= share) --to;
                if (to > from + 1 && p(to) - share > share - p(to - 1)) --to;
            }
            length = to - from;
            s.start[q + 1] = static_cast<int32_t>(to);
            const int64_t upto = p(to);
            s.by_cost.busiest = std::max(s.by_cost.busiest, upto - before);
            before = upto;
            s.by_cost.most_units = std::max(s.by_cost.most_units, static_cast<int32_t>(to - from));
        }
        // Equal numbers unless the busiest member gets 5% less: their members have
        // equally many outputs to form at the end, and their ranges need no table
        s.prefer_by_cost = s.by_cost.busiest * 20 < s.equal.busiest * 19;
    }

    const int64_t *prefix_ = nullptr;
    int64_t units_ = 0;
    int gates_ = 1;
    mutable std::atomic<UnitSplit *> kept_[kMaxMembers + 1] = {};
};

}  // namespace darb
