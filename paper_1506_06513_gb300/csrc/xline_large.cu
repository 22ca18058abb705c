// x lines of 324 to 512 points (see xline.cuh; XLine<R, L, G>: nx = 2 R L).
#include "xline.cuh"

namespace flusi {

const XLineOps* xline_table_large(int* n)
{
    static const XLineOps t[] = {
        XLineOf<XLine<18, 9, 3>>::all(),
        XLineOf<XLine<24, 8, 4>>::all(),
        XLineOf<XLine<27, 8, 4>>::all(),
        XLineOf<XLine<27, 9, 3>>::all(),
        XLineOf<XLine<16, 16, 2>>::lines_only(),
    };
    *n = int(sizeof t / sizeof t[0]);
    return t;
}

}  // namespace flusi
