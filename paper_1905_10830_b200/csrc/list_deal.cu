// SMs and blocks for the tensors of a list (tc_encode_many, tc_decode_many): which share of the device each of the kernels
// gets that work on a list at the same time.  No device code here.
#include <algorithm>
#include <cmath>

#include "tc_internal.h"

namespace {

constexpr int kOthersLeast = 8;                        // SMs of tensors with kernels of their own

// A block's set-up and first tile, us: basis, tensor memory, tables and first copies, and the tile through all stages, which work on two
// tiles and more at a time afterwards (13 with tiles of 2 us, 41 for three tiles of 8.6).
double first_us(const ListWork &w) { return 8.0 + std::max(5.0, 1.75 * w.tile_us); }

// Blocks that finish the tensor in `us`, or in the time of a first tile.
long long blocks_for(const ListWork &w, double us)
{
    const double more = std::min(std::max((us - first_us(w)) / w.tile_us, 0.0), 1e15);
    const long long each = 1 + (long long)more;
    return (w.tiles + each - 1) / each;
}

// us of one SM that the tensors take
double all_us(const std::vector<ListWork> &work)
{
    double us = 0.0;
    for (const ListWork &w : work) us += w.tile_us * (double)w.tiles;
    return us;
}

// The least time (to 1 %) from `us` on for which fits(us); it fits some time.
template <typename Fits>
double least_time(double us, Fits fits)
{
    if (fits(us)) return us;
    double least = us, most = 1.25 * us;
    while (!fits(most) && most < 1e12) { least = most; most *= 1.5; }
    while (most - least > 0.01 * least) {
        const double mid = 0.5 * (least + most);
        if (fits(mid)) most = mid; else least = mid;
    }
    return most;
}

}  // namespace

void deal_blocks(std::vector<ListWork> &work, int sms)
{
    const double us = least_time(std::max(13.0, all_us(work) / sms), [&](double t) {
        long long sum = 0;
        for (const ListWork &w : work) sum += blocks_for(w, t);
        return sum <= sms;
    });
    for (ListWork &w : work) w.blocks = (int)blocks_for(w, us);
}

int list_launches(size_t tensors, int sms)
{
    const int most = std::min(kListItems, std::max(sms, 1));
    return (int)((tensors + most - 1) / most);
}

int deal_list(const std::vector<std::vector<ListWork>> &classes, double others_us, int others, int sm_count, std::vector<int> &sms)
{
    sms.assign(classes.size(), 0);
    const int n_classes = (int)std::count_if(classes.begin(), classes.end(), [](const auto &c) { return !c.empty(); });
    if (n_classes == 0) return sm_count;
    if (n_classes == 1 && others == 0) {
        for (size_t j = 0; j < classes.size(); ++j) sms[j] = classes[j].empty() ? 0 : sm_count;
        return 0;
    }
    const int shared = std::max(n_classes, others > 0 ? sm_count - std::min(kOthersLeast, sm_count / 2) : sm_count);
    // Blocks of a class in its largest launch: launch r of R takes tensors r, r + R, ...; each has a part of the time.
    auto of_class = [&](const std::vector<ListWork> &c, double us) {
        const int launches = list_launches(c.size(), shared / n_classes);
        long long most = 0;
        for (int r = 0; r < launches; ++r) {
            long long sum = 0;
            for (size_t i = r; i < c.size(); i += launches) sum += blocks_for(c[i], us / launches);
            most = std::max(most, sum);
        }
        return most;
    };
    auto of_all = [&](double t) {
        double sum = 0.0;
        for (const auto &c : classes) sum += (double)of_class(c, t);
        return sum;
    };
    // All done at the same time.  Beside others the shared launches have up to a quarter of the SMs all the same, which they leave early:
    // entropy coders fill those, while a launch on few SMs that starts late ends late (six layers of 128x28x28 x 64 with a table per channel and three
    // of 256x14x14 x 32, decode: 127 us with 37 SMs, 161 with 6).
    double total = others_us;
    for (const auto &c : classes) total += all_us(c);
    double us = least_time(std::max(13.0, total / sm_count), [&](double t) {
        return of_all(t) + std::max(others > 0 ? std::ceil(others_us / t) : 0.0, (double)(sm_count - shared)) <= sm_count;
    });
    if (others > 0) us = std::min(us, least_time(std::max(13.0, 4.0 * (total - others_us) / sm_count), [&](double t) { return t >= us || of_all(t) <= sm_count / 4; }));
    int left = sm_count, largest = -1;
    for (size_t j = 0; j < classes.size(); ++j) {
        if (classes[j].empty()) continue;
        sms[j] = (int)of_class(classes[j], us);
        left -= sms[j];
        if (largest < 0 || sms[j] > sms[largest]) largest = (int)j;
    }
    if (others > 0) return std::max(1, left);
    sms[largest] += std::max(0, left);
    return 0;
}

// us of one SM that a tensor with kernels of its own takes a tile where there are many (`bits` of code a pixel), within a third of
// what 100 000 pixels took over 32 to 1024 channels: encodes on the tensor cores 6.0 with 32, 10.3 with 128, 24 with 320, 50 with 576, 96 with
// 960; decodes 17 with 320, 36 with 576, 70 with 960; the bit width adds 2 to 20 %, a table per channel a quarter.  fp32 kernels 8.2 with 24, 22 with
// 72, 104 with 200; exact ones 38 with 64, 130 with 128, 420 with 256, 1250 with 512.
extern "C" double tc_list_own_us(long long tiles, int c, int k, double bits, bool per_channel, bool tensor_cores, bool exact, bool encode)
{
    double us;
    if (exact) us = 0.0047 * c * k + 0.4 * k;
    else if (!tensor_cores) us = 4.0 + 0.1 * k + 0.0019 * c * k;
    else {
        us = encode ? 2.0 + k * (0.045 + 5.5e-5 * c) : k * (0.043 + 3e-5 * c);
        us = (us + 0.002 * bits) * (per_channel ? 1.25 : 1.0);
    }
    return us * (double)tiles;
}

// For the tests: `classes` lists of n_tensors[j] tensors each, one after the other in `tiles` and `tile_us`.
extern "C" int tc_deal_list(int classes, const int *n_tensors, const long long *tiles, const double *tile_us, double others_us, int others,
                            int sm_count, int *class_sms)
{
    std::vector<std::vector<ListWork>> work(classes);
    std::vector<int> sms;
    for (int j = 0, at = 0; j < classes; ++j)
        for (int i = 0; i < n_tensors[j]; ++i, ++at) work[j].push_back({tiles[at], tile_us[at], 0});
    const int rest = deal_list(work, others_us, others, sm_count, sms);
    std::copy(sms.begin(), sms.end(), class_sms);
    return rest;
}
