// launch_shape.cu -- host-side choice of the z-chunk (planes per CTA) of a
// single-grid step launch.
//
// A launch is (tiles) xy tiles x (chunks) z-chunks of CTAs; each CTA marches
// its chunk plus one halo plane on each side.  The choice trades the halo
// planes that short chunks re-read against the imbalance of the last round of
// CTAs on the device's resident slots (SMs x CTAs per SM of that kernel):
//
// - Many rounds (16-plane chunks would fill four or more rounds of the
//   slots): chunks of 16 planes or more, about `target` CTAs (six rounds of
//   the kernel family's design occupancy).  A 512^3 sweep placed the optimum
//   there, and with many rounds the last one's imbalance is a small part of
//   the launch.
// - Few rounds: every chunk length from 4 to 64 planes is scored by the
//   makespan of a greedy dispatch of the CTAs, in launch order, to the slots:
//   a CTA takes (its planes + 1) units, and one that has to wait for a slot
//   2 units more (its start and the fill of its ring, which a CTA of the first
//   round overlaps with the launch before; both constants are a fit).  The
//   shortest makespan wins, ties to the longer chunk.  The launch order puts the
//   short last chunk of each column last.  The model takes a CTA's speed as
//   independent of the CTAs beside it on its SM, which holds for the streaming
//   kernels at three or four CTAs per SM; a kernel with fewer (none of this
//   family) would keep the rule of many rounds.
// - Less than a round at 4 planes: the shortest chunks that still fit one round,
//   since such a launch lasts as long as one CTA's march (FP32, contact faces, 13
//   groups, us a step: 32^3 4 planes 7.1, 1 (chosen) 4.9; 64^3 7.0 and 4.8; 96^3
//   4 planes 7.5, 3 (chosen) 7.1, 2 (more than a round) 9.7).
//
// Sweeps of 1 to 64 planes over 40 streaming launches (FP32 32^3 to 384^3, periodic,
// contact and mixed faces, TI, CF and stochastic rounding, 150 x 133 x 117; BF16
// 128^3 and 256^3): the choice ran 1.0 % above the best measured one on average
// and 10 % at worst (320^3 channel: 54 planes 59.6 us, 18 planes 54.1); at 320^3
// and 384^3 otherwise 3 to 5 %.
//
// TI_n has a rule of its own: its CTAs differ in work (those in the interface
// band compute the 13 couplings of each cell, a plane of them some 2 us; those
// in the bulk do not), so it wants many small CTAs.  About six rounds of
// the slots, chunks of 4 to 16 planes; where chunks of 4 leave slots empty, the
// shortest chunks that still fit one round.  Measured at two CTAs per SM (us a
// step, FP32 27-point, tilted plane, planes per CTA): 60^3 20: 34.3, 4: 10.1, 1
// (chosen): 7.0; 64^3 16: 28.9, 4: 8.9, 1 (chosen): 5.2; 96^3 16: 29.1, 4 (chosen):
// 12.7, 2: 14.0; 192^3 16: 65.9, 4 (chosen): 54.1, 2: 57.1; 256^3 16: 113.6, 9
// (chosen): 106.1, 6: 104.6; 320^3 16 (chosen): 178.2, 12: 171.7, 4: 183.0.
//
// The FP64 kernels (CF and TI global) are bound by the FP64 pipe, which the CTAs
// of an SM share: what counts is the work of the fullest SM, ceil(CTAs / SMs)
// CTAs, a plane of a CTA costing about 9 FP64 instructions a cell as it is read
// and 21 more as it is written (the halo planes are only read).  A CTA alone on
// its SM leaves the pipe idle a fifth of the time, two leave it 2 %.  Chunks of
// 1 to 64 planes, the least work, ties to the longer chunk.  Measured, us a step
// (planes per CTA; 13 groups but for the first): 128 x 32 x 32 7-point 2 (chosen)
// 10.9, 1: 11.7, 4 (the streaming rule) 17.4; 72^3 4 (chosen) 66, 2: 97; 96^3 6
// (chosen) 95, 12: 109, 2: 109; 100^3 10 (chosen) 153, 5: 219; 256^3 37 (chosen)
// 1632, 16: 1669.
#include <map>
#include <mutex>
#include <queue>
#include <tuple>
#include <vector>

#include "spfm_internal.h"

namespace spfm {

// makespan, in plane units, of `tiles` x ceil(nz / zc) CTAs dispatched in
// launch order to `slots` slots by a greedy scheduler (see above)
static long long dispatch_makespan(int tiles, int nz, int zc, int slots)
{
    constexpr long long h = 1, w = 2;
    const int chunks = (nz + zc - 1) / zc;
    const int last = nz - (chunks - 1) * zc;
    const long long d = zc + h, ds = last + h;
    const long long nfull = (long long)tiles * (last < zc ? chunks - 1 : chunks);
    const long long nshort = last < zc ? tiles : 0;
    // the equal CTAs first: r slots carry q + 1 of them, the others q, each
    // after the first on its slot having waited
    const long long q = nfull / slots, r = nfull % slots;
    auto load = [&](long long k) { return k == 0 ? 0 : k * d + (k - 1) * w; };
    long long span = load(q + (r > 0));
    if (nshort == 0) return span;
    // the short CTAs go to the slots that free first
    std::priority_queue<long long, std::vector<long long>, std::greater<long long>> free_at;
    for (long long i = 0; i < slots; ++i) free_at.push(load(i < r ? q + 1 : q));
    for (long long i = 0; i < nshort; ++i) {
        const long long t = free_at.top() + (nfull + i >= slots ? w : 0) + ds;
        free_at.pop();
        free_at.push(t);
        if (t > span) span = t;
    }
    return span;
}

static int model_zchunk(int tiles, int nz, int per_sm, int slots, int target)
{
    if (nz <= 4) return nz;
    const long long rounds16 = (long long)tiles * ((nz + 15) / 16);
    if (rounds16 >= 4LL * slots || per_sm < 3) {
        int chunks = (target + tiles - 1) / tiles;
        const int max_chunks = nz / 16 > 1 ? nz / 16 : 1;
        if (chunks > max_chunks) chunks = max_chunks;
        if (chunks < 1) chunks = 1;
        return (nz + chunks - 1) / chunks;
    }
    int best = 4;
    long long best_span = -1;
    const int hi = nz < 64 ? nz : 64;
    for (int zc = 4; zc <= hi; ++zc) {
        const long long span = dispatch_makespan(tiles, nz, zc, slots);
        if (best_span < 0 || span <= best_span) {
            best_span = span;
            best = zc;
        }
    }
    return best;
}

// the shortest chunks whose CTAs fit one round
static int one_round_zchunk(int tiles, int nz, int slots)
{
    const int chunks = slots / tiles < nz ? slots / tiles : nz;
    return (nz + chunks - 1) / chunks;
}

// planes per CTA of a TI_n launch (see above)
static int uneven_zchunk(int tiles, int nz, int slots)
{
    if ((long long)tiles * ((nz + 3) / 4) < slots) return one_round_zchunk(tiles, nz, slots);
    const long long zc = ((long long)tiles * nz + 6LL * slots - 1) / (6LL * slots);
    return zc < 4 ? 4 : (zc > 16 ? 16 : (int)zc);
}

// planes per CTA of an FP64 launch (see above)
static int fp64_zchunk(int tiles, int nz, int sms)
{
    int best = 1;
    long long best_work = -1;
    for (int zc = 1; zc <= (nz < 64 ? nz : 64); ++zc) {
        const long long ctas = (long long)tiles * ((nz + zc - 1) / zc);
        const long long n = (ctas + sms - 1) / sms, idle = n == 1 ? 20 : (n == 2 ? 2 : 0);
        const long long work = n * (100 + idle) * (9 * (zc + 2) + 21 * zc);
        if (best_work < 0 || work <= best_work) {
            best_work = work;
            best = zc;
        }
    }
    return best;
}

int choose_zchunk(int family, int tiles, int nz, int per_sm, int sms, int target)
{
    const int slots = per_sm * sms;
    if (family == kUneven) return uneven_zchunk(tiles, nz, slots);
    if (family == kFp64) return fp64_zchunk(tiles, nz, sms);
    if ((long long)tiles * ((nz + 3) / 4) <= slots) return one_round_zchunk(tiles, nz, slots);
    return model_zchunk(tiles, nz, per_sm, slots, target);
}

namespace {
std::mutex g_mu;
// (kernel, threads, device) -> resident CTAs per SM; (tiles, nz, slots, target or -family) -> z-chunk
std::map<std::tuple<const void *, int, int>, int> g_occ;
std::map<std::tuple<int, int, int, int>, int> g_zc;
}  // namespace

int pick_zchunk(const void *kern, int threads, int tiles, int nz, int target, int family)
{
    int dev = 0, sms = 152;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    std::lock_guard<std::mutex> lock(g_mu);
    const auto ok = std::make_tuple(kern, threads, dev);
    auto o = g_occ.find(ok);
    int per_sm;
    if (o != g_occ.end()) {
        per_sm = o->second;
    } else {
        per_sm = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, threads, 0) != cudaSuccess || per_sm < 1) {
            cudaGetLastError();   // the launch itself reports a kernel that cannot run
            per_sm = 1;
        }
        g_occ[ok] = per_sm;
    }
    const int slots = per_sm * sms;
    const auto zk = std::make_tuple(tiles, nz, slots, family == kStream ? target : -family);
    auto z = g_zc.find(zk);
    if (z != g_zc.end()) return z->second;
    if (g_zc.size() >= 4096) g_zc.clear();   // many grid shapes (a serving process): start over
    const int zc = choose_zchunk(family, tiles, nz, per_sm, sms, target);
    g_zc[zk] = zc;
    return zc;
}

}  // namespace spfm

extern "C" int spfm_debug_pick_zchunk(int tiles, int nz, int per_sm, int sms, int target)
{
    if (tiles < 1 || nz < 1 || per_sm < 1 || sms < 1 || target < 1) return -1;
    return spfm::model_zchunk(tiles, nz, per_sm, per_sm * sms, target);
}

extern "C" int spfm_debug_zchunk(int family, int tiles, int nz, int per_sm, int sms, int target)
{
    if (family < spfm::kStream || family > spfm::kFp64) return -1;
    if (tiles < 1 || nz < 1 || per_sm < 1 || sms < 1 || target < 1) return -1;
    return spfm::choose_zchunk(family, tiles, nz, per_sm, sms, target);
}
