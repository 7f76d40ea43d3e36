// nd_schedule.h -- the time-sliced schedule of a size class with more replicas
// than resident CTAs (or clusters), in closed form.
#pragma once

#ifdef __CUDACC__
#define ND_HOST_DEVICE __host__ __device__ __forceinline__
#else
#define ND_HOST_DEVICE inline
#endif

namespace nd {

// A piece of one replica's trajectory run by one CTA or cluster.
struct Segment {
    int rep;                 // replica index
    int wait;                // wait until flags[rep] is kHandedOver before starting
    int signal;              // set flags[rep] to kHandedOver when done
    int pos;                 // the replica's position in its class
    long long step_begin;    // first time step (relative to the call's step0)
    long long nsteps;
};

// Replica-steps of a slot: B x n cut into nslots equal, contiguous ranges.  A
// slot touches at most slot_room replicas.
ND_HOST_DEVICE long long slot_share(int B, long long n, int nslots) { return (B * n + nslots - 1) / nslots; }
ND_HOST_DEVICE int slot_room(int B, int nslots) { return B / nslots + 2; }

// Segment k of a slot (all but rep), and how many it has.  Slot i runs the start
// of the replica it shares with slot i + 1 first (and signals it), then its
// whole replicas, then the end of the replica it shares with slot i - 1, after
// waiting for that signal: a wait is for the first segment of the slot before,
// which waits for nothing.  Every slot makes the same number of steps.
ND_HOST_DEVICE int slot_segment(int B, long long n, long long share, int slot, int k, Segment &g)
{
    const long long W = B * n, start = slot * share;
    if (start >= W) return 0;
    const long long end = start + share < W ? start + share : W;
    const int r0 = (int)(start / n), r1 = (int)((end - 1) / n);
    const long long o0 = start - r0 * n, o1 = end - r1 * n;   // steps of r0 before the slot's, of r1 up to its end
    if (r0 == r1) {
        g = Segment{0, o0 > 0, o1 < n, r0, o0, o1 - o0};
        return 1;
    }
    const int part = o1 < n, first = o0 > 0 ? r0 + 1 : r0, whole = r1 + 1 - part - first;
    if (k < part) g = Segment{0, 0, 1, r1, 0, o1};
    else if (k < part + whole) g = Segment{0, 0, 0, first + k - part, 0, n};
    else g = Segment{0, 1, 0, r0, o0, n - o0};
    return part + whole + (o0 > 0);
}

}  // namespace nd
