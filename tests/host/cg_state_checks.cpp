// The end-of-solve rule of the conjugate gradients (cg_state.h): whatever a launch writes about the
// end, a thread of the same launch that reads it before and one that reads it after decide alike, and
// the launches after the last iteration all return.  Prints one line per check.
#include <cstdio>
#include <initializer_list>

#include "cg_state.h"

using namespace hdf;

int main() {
    int bad = 0;
    for (int end : {0, 1, 2, 3, 4, 7, 1000}) {
        // kernels of iteration it, in order: finish, step (may write the end), gemv, dir (may write it)
        for (int writer : {1, 3}) {
            int last = end == 0 ? 0 : kCgRunning;
            int undecided = 0, wrong = 0;
            for (int it = 1; it <= end + 9; ++it)
                for (int kernel = 0; kernel < 4; ++kernel) {
                    const bool early = cg_past_end(last, it);
                    if (it == end && kernel == writer && !early) last = it;
                    const bool late = cg_past_end(last, it);
                    undecided += early != late;
                    wrong += early != (it > end);
                }
            std::printf("%s end %d written by kernel %d\n", undecided || wrong ? "FAIL" : "ok", end, writer);
            bad += undecided + wrong;
        }
    }
    return bad ? 1 : 0;
}
