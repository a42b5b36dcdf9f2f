// Walker update with several commits per round, 4 lanes per walker.
#include "walker_scan.cuh"

namespace mucal {

void walker_scan_4_fns(const void *(&fns)[kWalkerScanFns]) { walker_scan_fns_t<4>(fns); }

}  // namespace mucal
