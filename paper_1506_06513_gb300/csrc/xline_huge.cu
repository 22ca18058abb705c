// x lines of 576 to 1024 points (see xline.cuh; XLine<R, L, G>: nx = 2 R L).
#include "xline.cuh"

namespace flusi {

const XLineOps* xline_table_huge(int* n)
{
    static const XLineOps t[] = {
        XLineOf<XLine<24, 12, 2>>::all(),
        XLineOf<XLine<27, 12, 2>>::all(),
        XLineOf<XLine<24, 16, 2>>::all(),
        XLineOf<XLine<27, 16, 2>>::all(),
        XLineOf<XLine<27, 18, 1>>::all(),
        XLineOf<XLine<32, 16, 2>>::lines_only(),
    };
    *n = int(sizeof t / sizeof t[0]);
    return t;
}

}  // namespace flusi
