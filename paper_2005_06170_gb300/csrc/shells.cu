// Host-side shell tables of the binning (see shells.h). No device code: the file is
// compiled by nvcc into the library and by a plain C++ compiler into a CPU test.
#include "shells.h"

#include <algorithm>
#include <cmath>

namespace pkmom {

int shell_tables(int nbins, double umin, double umax, std::vector<uint16_t> &bintab, std::vector<int> &thresh)
{
    const int nsq_max = static_cast<int>(std::floor(umax * umax)) + 1;
    bintab.assign(nsq_max + 1, 0xffff);
    for (int nsq = 1; nsq <= nsq_max; ++nsq) {
        const double u = std::sqrt(static_cast<double>(nsq));
        if (u < umin || u > umax) continue;
        double tb = std::floor(((u - umin) * nbins) / (umax - umin));
        if (tb > nbins - 1) tb = nbins - 1;
        bintab[nsq] = static_cast<uint16_t>(tb);
    }
    // shell b is the interval thresh[b] <= |n|^2 < thresh[b + 1] (bins are monotone in |n|^2)
    thresh.assign(nbins + 1, nsq_max + 1);
    int last = 0;
    for (int nsq = nsq_max; nsq >= 1; --nsq) {
        const int b = bintab[nsq];
        if (b == 0xffff) continue;
        if (!last) last = nsq;
        for (int k = b; k >= 0 && thresh[k] > nsq; --k) thresh[k] = nsq;
    }
    thresh[nbins] = last + 1;
    for (int k = nbins - 1; k >= 0; --k) thresh[k] = std::min(thresh[k], thresh[k + 1]);
    return nsq_max;
}

std::vector<uint32_t> bin_item_list(const std::vector<int> &thresh, int ng, int nbins)
{
    std::vector<uint32_t> work;
    for (int r = 0; r < ng; ++r) {
        const int k = r >> 1, i0 = (r & 1) ? ng - 1 - k : k;
        const int n0 = i0 < ng / 2 ? i0 : i0 - ng;
        for (int b = nbins - 1; b >= 0; --b)
            if (thresh[b + 1] > thresh[b] && thresh[b + 1] - 1 - n0 * n0 >= 0)
                work.push_back(static_cast<uint32_t>(i0) * nbins + b);
    }
    return work;
}

void mu_task_list(const std::vector<int> &thresh, int ng, int nbins, std::vector<uint32_t> &tasks,
                  std::vector<int> &range)
{
    tasks.clear();
    range.assign(2 * nbins, 0);
    for (int b = nbins - 1; b >= 0; --b) {
        range[2 * b] = range[2 * b + 1] = static_cast<int>(tasks.size() / 2);
        const int width = thresh[b + 1] - thresh[b];
        if (width <= 0) continue;
        int reach = static_cast<int>(std::sqrt(static_cast<double>(thresh[b + 1] - 1)));
        while (reach > 0 && reach * reach > thresh[b + 1] - 1) --reach;
        while ((reach + 1) * (reach + 1) <= thresh[b + 1] - 1) ++reach;
        reach = std::min(reach, ng / 2 - 1);
        const int slabs = std::max(1, std::min(64, static_cast<int>(1500.0 / (1.5707963267948966 * width))));
        for (int n0 = -reach; n0 <= reach; n0 += slabs) {
            tasks.push_back(static_cast<uint32_t>(b));
            tasks.push_back(static_cast<uint32_t>(n0 + ng / 2) |
                            static_cast<uint32_t>(std::min(slabs, reach - n0 + 1)) << 16);
        }
        range[2 * b + 1] = static_cast<int>(tasks.size() / 2);
    }
}

}  // namespace pkmom
