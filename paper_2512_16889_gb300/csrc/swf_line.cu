// Instances of the register line kernels (swf_line.cuh) for the lengths of one list and one
// precision: compiled once per list and precision (SWF_LINE_LIST, SWF_LINE_REAL) so that the
// units build in parallel.
#include "swf_line.cuh"
#include "swf_line_list.h"

#define SWF_CAT_(a, b, c) a##b##_##c
#define SWF_CAT(a, b, c) SWF_CAT_(a, b, c)

namespace swf {

#define X(n, r1, r2) {n, r1, r2, k_xline<SWF_LINE_REAL, r1, r2>, k_line<SWF_LINE_REAL, r1, r2>, \
                      k_f2_line<SWF_LINE_REAL, r1, r2>},
#define LIST_(l) SWF_LINES_##l(X)
#define LIST(l) LIST_(l)
static const LineEntry<SWF_LINE_REAL> entries[] = {LIST(SWF_LINE_LIST)};

// find_line<list>_<real>: the entry of n in this list, or null.
const LineEntry<SWF_LINE_REAL>* SWF_CAT(find_line, SWF_LINE_LIST, SWF_LINE_REAL)(int n) {
  for (const auto& e : entries)
    if (e.n == n) return &e;
  return nullptr;
}

}  // namespace swf
