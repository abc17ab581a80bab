// Record slots of the overdamped runs (host code only).
//
// A launch leaves two doubles, the sums of R and R R(0), for every record and slot, and a
// second kernel adds a record's slots up.  How many slots a record has is the kernel's
// choice: one for 256 particles, one for 128, one a team of 8 or 16 (Hybrid Taus, the LCG),
// one a CTA or a using warp of it (Lagged Fibonacci).  The promise to callers is 16 bytes
// per record and 256 particles, or kRecordScratch where that is more: a kernel of more slots
// runs only while they fit it, and Lagged Fibonacci runs of more records are cut into
// launches.
#pragma once

#include <algorithm>
#include <cstdint>

namespace gb {

constexpr int64_t kRecordLimit = (int64_t)4 << 30;      // bytes, at one slot for 256 particles
constexpr int64_t kRecordScratch = (int64_t)256 << 20;

inline double record_bytes(int64_t n_rec, int64_t slots) { return 16.0 * (double)n_rec * (double)slots; }
inline int64_t record_blocks(int64_t n) { return (n + 255) / 256; }

// What ou_run refuses, whichever kernel would run: by the blocks of 256 particles (Lagged
// Fibonacci: at most five a SM of them, four at order 4).
inline bool records_refused(int64_t n_rec, int64_t blocks)
{
    return n_rec > 0x7fffffff || record_bytes(n_rec, blocks) > (double)kRecordLimit;
}
inline int64_t lfg_record_blocks(int64_t n, int sms, int order)
{
    return std::min<int64_t>((order == 4 ? 4 : 5) * (int64_t)sms, record_blocks(n));
}

// Whether `slots` slots a record of n particles are within the promise.
inline bool records_fit(int64_t n_rec, int64_t slots, int64_t n)
{
    return slots <= record_blocks(n) || record_bytes(n_rec, slots) <= (double)kRecordScratch;
}

// Lagged Fibonacci: particles of a CTA (even), its slots (a using warp's units are of `unit`
// particles), and the records of one launch.
constexpr int kOuWarps = 15;
inline int64_t lfg_share(int64_t n, int sms) { return ((n + sms - 1) / sms + 1) & ~(int64_t)1; }
inline int lfg_record_slots(int64_t share, int unit)
{
    return (int)std::min<int64_t>(kOuWarps, (share + unit - 1) / unit);
}
inline int64_t lfg_launch_records(int64_t n, int sms)
{
    return std::max<int64_t>(2, kRecordScratch / (16 * (int64_t)sms * lfg_record_slots(lfg_share(n, sms), 32)));
}

}  // namespace gb
