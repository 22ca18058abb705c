// x lines of 144 to 288 points (see xline.cuh; XLine<R, L, G>: nx = 2 R L).
#include "xline.cuh"

namespace flusi {

const XLineOps* xline_table_medium(int* n)
{
    static const XLineOps t[] = {
        XLineOf<XLine<12, 6, 5>>::all(),
        XLineOf<XLine<9, 9, 3>>::all(),
        XLineOf<XLine<12, 8, 4>>::all(),
        XLineOf<XLine<18, 6, 5>>::all(),
        XLineOf<XLine<12, 12, 2>>::all(),
        XLineOf<XLine<16, 8, 4>>::all(),
    };
    *n = int(sizeof t / sizeof t[0]);
    return t;
}

}  // namespace flusi
