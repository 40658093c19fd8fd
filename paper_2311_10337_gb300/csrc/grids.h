// Grid sizes that depend on the device and are decided on the host.
#pragma once

#include <stdint.h>

namespace dgec {

// CTAs of the dendrogram's middle rounds: one for each 512 live edges, so that
// a thread has no chain of bids and loads one after another, but at most one
// an SM (a second CTA on some SMs makes every phase wait for those), and no
// more than the per-CTA counts have room for. 20,000 edges: 0.24 ms at one CTA
// per 4,096 edges, 0.154 so; 317,000 on 152 SMs: 0.49 ms, 0.51 with 192 CTAs, 0.45
// with 152.
inline int mid_ctas(int64_t live, int sms, int room) {
    int64_t g = (live + 511) / 512;
    if (g > sms) g = sms;
    if (g > room) g = room;
    return g > 1 ? (int)g : 1;
}

}  // namespace dgec
