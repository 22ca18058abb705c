// x lines of 16 to 128 points (see xline.cuh; XLine<R, L, G>: nx = 2 R L).
#include "xline.cuh"

namespace flusi {

const XLineOps* xline_table_small(int* n)
{
    static const XLineOps t[] = {
        XLineOf<XLine<4, 2, 16>>::all(),
        XLineOf<XLine<3, 3, 10>>::all(),
        XLineOf<XLine<3, 4, 8>>::all(),
        XLineOf<XLine<4, 4, 8>>::all(),
        XLineOf<XLine<6, 3, 10>>::all(),
        XLineOf<XLine<6, 4, 8>>::all(),
        XLineOf<XLine<9, 3, 10>>::all(),
        XLineOf<XLine<6, 6, 5>>::all(),
        XLineOf<XLine<9, 6, 5>>::all(),
        XLineOf<XLine<8, 4, 8>>::all(),
        XLineOf<XLine<12, 4, 8>>::lines_only(),
        XLineOf<XLine<8, 8, 4>>::all(),
    };
    *n = int(sizeof t / sizeof t[0]);
    return t;
}

}  // namespace flusi
