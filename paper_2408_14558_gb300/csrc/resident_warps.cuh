// The CTA size of a persistent kernel (host code only).
#pragma once

namespace spg {

// The number of warps per CTA, from `least` to `most`, that keeps most warps on an
// SM (of equal ones the largest; 0 where none fits); ctas(w) asks how many CTAs of
// w warps an SM holds.
template <typename Ctas>
int most_resident_warps(int least, int most, Ctas ctas) {
    int best = 0, resident = 0;
    for (int w = most; w >= least && w > 0; w--) {
        const int r = w * ctas(w);
        if (r > resident) {
            resident = r;
            best = w;
        }
    }
    return best;
}

}  // namespace spg
