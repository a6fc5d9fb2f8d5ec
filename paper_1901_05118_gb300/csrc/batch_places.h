// Which launches of the batch engine are started beside each other: plain
// arithmetic, used by the engine and checked on the CPU.
//
// Places are those of the cooperative FP32 kernel's CTAs, per_sm to an SM; a CTA of an
// on-chip launch fills an SM (its registers do) and counts per_sm.  The hardware may spread
// a cooperative group's CTAs one to an SM, so an on-chip launch that the count lets start may still wait on the
// GPU until the group's launch ends.  (No two can block each other: a
// cooperative launch starts when all of its CTAs have a place, or waits without any.)  It then
// starts without a turn of the host.  Counting such SMs as taken made two
// mixed-precision requests of 96^3 beside a stream of 32^3 ones faster (1165 -> 1015 ms)
// at the stream's cost (200 -> 163 requests/s), and the burst of both never faster, up to a fifth slower.
#pragma once

namespace excmg {

struct SmPlaces {
    int sms;        // SMs of the GPU
    int per_sm;     // CTAs of the cooperative FP32 kernel per SM
    int resident;   // CTAs of on-chip launches under way
    int coop;       // CTAs of cooperative groups under way
};

inline int free_places(const SmPlaces& p) { return p.per_sm * (p.sms - p.resident) - p.coop; }

// Whether an on-chip launch of `ctas` CTAs starts.
inline bool on_chip_fits(const SmPlaces& p, int ctas) { return p.per_sm * ctas <= free_places(p); }

// CTAs that a cooperative group which asks for `want` starts with, 0 where it
// waits: a launch keeps its CTAs for up to 256 iterations, so with less than half of what it
// asks for (two SMs beside a 66^3 level) it would hold its members back for longer than the wait.
inline int coop_share(const SmPlaces& p, int want) {
    const int all = p.per_sm * p.sms, left = free_places(p);
    if (want > all) want = all;
    return left >= want ? want : 2 * left >= want ? left : 0;
}

}  // namespace excmg
