// How the cooperative FP64 kernels (persistent64.cu) share a lattice among blocks, warps and passes, and
// whether the device takes the launch.  Host code without CUDA headers, so that the rules can be checked on
// the CPU.
#pragma once

#include <algorithm>

namespace ovl {

constexpr int LW = 16;         // warps per block
constexpr int L_MAXPASS = 4;   // passes whose state fits shared memory (57 KB of half spinors + 37 KB each)

// Blocks (one per SM at most), passes over a block's warps, and the row split of a launch over V sites at
// `spw` sites per warp unsplit.  RS = 2 halves the units' FP64 instructions (74 against 129 of the Lanczos
// process's first phase) and doubles their number: better while it lowers the count of the busiest SM
// quarter by more than it adds in all.
struct Split {
    int rs, G, npass;
};
inline Split split_units(int V, int spw, int num_sms) {
    auto make = [&](int rs) {
        const int units = (V + spw / rs - 1) / (spw / rs);
        Split s;
        s.rs = rs;
        s.G = std::max(1, std::min(units, num_sms));
        s.npass = ((units + s.G - 1) / s.G + LW - 1) / LW;
        return s;
    };
    auto quarter = [&](const Split& s) {  // units of the busiest SM quarter
        const int units = (V + spw / s.rs - 1) / (spw / s.rs);
        return ((units + s.G - 1) / s.G + 3) / 4;
    };
    const Split one = make(1), two = make(2);
    return two.npass == 1 && 74 * quarter(two) < 129 * quarter(one) ? two : one;
}

// The launch's blocks wait on one another, so all of them have to be resident: `per_sm` of them fit an SM (0: the
// shared memory or the registers of one are not to be had), `cooperative` is the device's attribute.  Where
// they do not fit, the per-step kernels run.
inline bool split_fits(const Split& s, int num_sms, int per_sm, bool cooperative) {
    return s.npass <= L_MAXPASS && cooperative && (long long)per_sm * num_sms >= s.G;
}

}  // namespace ovl
