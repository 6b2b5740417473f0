// Instantiation of the threshold-table kernel of general boxes for words of
// 1 .. 8 sites of a colour.
#include "pa_boxtab.cuh"

namespace pa {

cudaError_t launch_boxtab_a(int S, const BoxShape& box, RunDev* runs, const Work* table, int nwork, int WR,
                             cudaStream_t st) {
  switch (S) {
    case 1: return launch_boxtab_s<1>(box, runs, table, nwork, WR, st);
    case 2: return launch_boxtab_s<2>(box, runs, table, nwork, WR, st);
    case 3: return launch_boxtab_s<3>(box, runs, table, nwork, WR, st);
    case 4: return launch_boxtab_s<4>(box, runs, table, nwork, WR, st);
    case 5: return launch_boxtab_s<5>(box, runs, table, nwork, WR, st);
    case 6: return launch_boxtab_s<6>(box, runs, table, nwork, WR, st);
    case 7: return launch_boxtab_s<7>(box, runs, table, nwork, WR, st);
    case 8: return launch_boxtab_s<8>(box, runs, table, nwork, WR, st);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace pa
