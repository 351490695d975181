// C entries over one block of svd.cu, for tests/test_svd_unit.py.
#include "svd.h"

using namespace spmps;

// launch_svd of a block of dim x other without any buffer.
extern "C" int svd_launch_empty(int dim, int other) {
    SvdPlan P;
    P.build({{dim, other}}, kSvdSmemDefault);
    return launch_svd(P, nullptr, nullptr, nullptr, nullptr);
}
