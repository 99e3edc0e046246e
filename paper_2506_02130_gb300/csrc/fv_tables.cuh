// Places of the FFT axes' twiddle tables within a plan's table buffer (host only, plain C++).
#pragma once
#include <cstddef>
#include <map>
#include <utility>

namespace fv {

// Axes of one length share a table.  An axis with a compile-time length has its own tables behind the plain one, so it
// shares only with its like: the up axis of one channel can have the length that x or y of another has, and takes the
// general passes.
class TableMap {
public:
    // Offset of the table of an axis of length M; extra: elements behind the plain table (fixed axes).
    size_t place(int M, bool fixed, size_t extra)
    {
        const auto at = at_.emplace(std::make_pair(M, fixed), total_);
        if (at.second) total_ += M + (fixed ? extra : 0);
        return at.first->second;
    }
    // Whether the caller is to fill this table: true once per table.
    bool take(int M, bool fixed) { return at_.erase(std::make_pair(M, fixed)) != 0; }
    size_t total() const { return total_; }

private:
    std::map<std::pair<int, bool>, size_t> at_;
    size_t total_ = 0;
};

}  // namespace fv
