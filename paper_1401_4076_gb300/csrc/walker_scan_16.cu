// Walker update with several commits per round, 16 lanes per walker.
#include "walker_scan.cuh"

namespace mucal {

void walker_scan_16_fns(const void *(&fns)[kWalkerScanFns]) { walker_scan_fns_t<16>(fns); }

}  // namespace mucal
