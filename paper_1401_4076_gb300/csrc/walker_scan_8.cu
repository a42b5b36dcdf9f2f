// Walker update with several commits per round, 8 lanes per walker.
#include "walker_scan.cuh"

namespace mucal {

void walker_scan_8_fns(const void *(&fns)[kWalkerScanFns]) { walker_scan_fns_t<8>(fns); }

}  // namespace mucal
