// Instantiation of the threshold-table kernel of general boxes for words of
// 9 .. 16 sites of a colour.
#include "pa_boxtab.cuh"

namespace pa {

cudaError_t launch_boxtab_b(int S, const BoxShape& box, RunDev* runs, const Work* table, int nwork, int WR,
                             cudaStream_t st) {
  switch (S) {
    case 9: return launch_boxtab_s<9>(box, runs, table, nwork, WR, st);
    case 10: return launch_boxtab_s<10>(box, runs, table, nwork, WR, st);
    case 11: return launch_boxtab_s<11>(box, runs, table, nwork, WR, st);
    case 12: return launch_boxtab_s<12>(box, runs, table, nwork, WR, st);
    case 13: return launch_boxtab_s<13>(box, runs, table, nwork, WR, st);
    case 14: return launch_boxtab_s<14>(box, runs, table, nwork, WR, st);
    case 15: return launch_boxtab_s<15>(box, runs, table, nwork, WR, st);
    case 16: return launch_boxtab_s<16>(box, runs, table, nwork, WR, st);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace pa
