// deal.cu -- host side of the batches' balance: work items dealt to CTAs, longest
// first, each to the CTA with the least work so far.
#include <algorithm>
#include <functional>
#include <map>
#include <queue>
#include <utility>
#include <vector>

#include "host_internal.h"

namespace spfm_host {

void deal(const std::vector<int> &planes, int ctas, std::vector<int> &order, std::vector<int> &owner)
{
    const size_t n = planes.size();
    order.resize(n);
    owner.resize(n);
    if (n == 0) return;
    // longest first, by counting (neighbouring tiles stay together)
    const int most = *std::max_element(planes.begin(), planes.end());
    std::vector<size_t> at(most + 2, 0);
    for (int p : planes) ++at[most - p + 1];
    for (int k = 0; k <= most; ++k) at[k + 1] += at[k];
    for (size_t k = 0; k < n; ++k) order[at[most - planes[k]]++] = (int)k;
    // a long list in turn up to its last few rounds, the rest to the least loaded
    std::vector<long long> load(ctas, 0);
    const size_t turns = n > 64u * (size_t)ctas ? (n / ctas - 16) * ctas : 0;
    for (size_t k = 0; k < turns; ++k) {
        owner[k] = (int)(k % ctas);
        load[owner[k]] += planes[order[k]] + kItemStart;
    }
    using Cta = std::pair<long long, int>;
    std::priority_queue<Cta, std::vector<Cta>, std::greater<Cta>> least;
    for (int c = 0; c < ctas; ++c) least.push({load[c], c});
    for (size_t k = turns; k < n; ++k) {
        Cta t = least.top();
        least.pop();
        owner[k] = t.second;
        t.first += planes[order[k]] + kItemStart;
        least.push(t);
    }
}

long long deal_span(const std::vector<long long> &count, int ctas)
{
    // CTAs by their work so far: equal items raise the lowest level together
    std::map<long long, long long> level;
    level[0] = ctas;
    for (int p = (int)count.size() - 1; p > 0; --p)
        for (long long left = count[p]; left > 0;) {
            const auto low = level.begin();
            const long long work = low->first, m = std::min(left, low->second);
            if (m == low->second) level.erase(low);
            else low->second -= m;
            level[work + p + kItemStart] += m;
            left -= m;
        }
    return level.rbegin()->first;
}

}  // namespace spfm_host

extern "C" int spfm_debug_deal(int n, const int *planes, int ctas, int *owner, long long *span)
{
    if (n < 0 || ctas < 1 || (n > 0 && (!planes || !owner))) return -1;
    int most = 0;
    for (int i = 0; i < n; ++i) {
        if (planes[i] < 1) return -1;
        most = std::max(most, planes[i]);
    }
    std::vector<int> order, by_order;
    std::vector<long long> count(most + 1, 0);
    for (int i = 0; i < n; ++i) ++count[planes[i]];
    spfm_host::deal(std::vector<int>(planes, planes + n), ctas, order, by_order);
    for (int k = 0; k < n; ++k) owner[k] = -1;
    for (int k = 0; k < n; ++k) owner[order[k]] = by_order[k];
    if (span) *span = spfm_host::deal_span(count, ctas);
    return 0;
}
