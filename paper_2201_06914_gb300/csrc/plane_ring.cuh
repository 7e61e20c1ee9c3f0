// What a thread of a marching block does in a ring of plane slots, and what it does once one of
// its bounded waits has given up.  Free of device code, so that the rules run on the host too
// (tests/test_plane_ring.py).
//
// Plane i of a march of n planes lies in slot i mod NS.  A slot's `full` barrier completes one
// phase (number i / NS) per plane: one arrival, made with the plane's byte count, and the bytes.
// An issuing thread starts the copies of plane i + LA before it computes plane i, after the block's
// readers have left the slot; the first LA planes are issued before the march.
//
// A thread whose wait gives up raises the error flag and neither waits nor issues from then on:
//   - a copy into a slot that was not seen empty could tear the plane another warp is reading;
//   - a second arrival at a `full` phase that is still pending is undefined;
//   - an issuing thread has waited for every earlier plane of a slot before it issues the next one,
//     so at most one phase of a slot is outstanding when it stops, and drain() may wait for that
//     phase by its parity.  With two outstanding the parity of the older one would pass for it.
#pragma once

#ifdef __CUDACC__
#define WP_RING_FN __host__ __device__ __forceinline__
#else
#define WP_RING_FN inline
#endif

namespace wp {

template <int NS, int LA>
struct PlaneRing {
    int issued = 0;   // planes issued when a wait of this thread gave up (0: none has)

    // Issuing threads, before plane i: plane i + LA into its slot.  empty(): waits until the readers
    // have left it (only called from the slot's second plane on).
    template <class Empty, class Raise, class Issue>
    WP_RING_FN void refill(int i, int n, Empty empty, Raise raise, Issue issue)
    {
        if (issued || i + LA >= n) return;
        if (i + LA >= NS && !empty()) {
            issued = i + LA;
            raise();
            return;
        }
        issue();
    }

    // Every thread, before it reads plane i.
    template <class Full, class Raise>
    WP_RING_FN void await(int i, int n, Full full, Raise raise)
    {
        if (issued || full()) return;
        issued = i + LA + 1 < n ? i + LA + 1 : n;
        raise();
    }

    // Issuing threads, after a march in which a wait gave up: the copies in flight land before the
    // block's memory is reused.  full(slot, parity): bounded wait.
    template <class Full>
    WP_RING_FN void drain(int n, Full full) const
    {
        const int m = issued ? issued : n;
        for (int s = 0; s < NS; s++) {
            const int planes = (m + NS - 1 - s) / NS;   // of this slot
            if (planes > 0) full(s, (unsigned)((planes - 1) & 1));
        }
    }
};

}  // namespace wp
