"""Tiles of the two-pass y and z kernels (csrc/colfft.cuh), by their index
arithmetic alone (no GPU): every TMA box of every length, tile width and 2/3 rule
lands on a 128-byte boundary of shared memory, inside its buffer, and the blocks
fit a streaming multiprocessor's 227 KB.
"""
from device_code import program_output

SOURCE = r"""
#include <cstdio>
#include "colfft.cuh"
using namespace flusi;
template <class X> void check(int n, bool y)
{
    const size_t row = sizeof(float2) * X::C;
    printf("%d %d %d %d %zu %zu", n, (int)y, X::C, X::BUFS, sizeof(float2) * X::BUF, X::kSmem);
    const int part = n / X::CH;
    // box rows as the tensor maps have them (prepare_y, prepare_z)
    printf(" %zu %d", (size_t)part * row, forward_box_rows(part, row));
    for (int strict = 0; strict < 2; ++strict) {
        const int K = strict && n % 3 == 0 ? n / 3 - 1 : n / 3, bh = inverse_box_rows(n, K, row);
        printf(" %d %d %zu", K, bh, (size_t)((X::CH == 1 ? n : part) - K - 1) * row);
    }
    printf("\n");
}
int main()
{
#define ONE(n, R, L)                                                            \
    check<Col<R, L, col_tile(n, 256)>>(n, true);                                \
    check<Col<R, L, 16>>(n, true);                                              \
    check<Col<R, L, col_tile(n, 64)>>(n, false);                                \
    check<Col<R, L, (n) <= 512 ? 8 : col_tile(n, 64)>>(n, false);
    FLUSI_COL_LENGTHS(ONE)
    return 0;
}
"""


def test_boxes_land_on_128_byte_boundaries(tmp_path):
    lines = [tuple(map(int, l.split())) for l in program_output(SOURCE, tmp_path).splitlines()]
    assert len(lines) == 4 * 23
    for n, y, cols, bufs, buf, smem, part, fwd, *inv in lines:
        where = (n, "y" if y else "z", cols)
        row = 8 * cols
        # a row range and, at the end of the ring, the next buffer start aligned
        assert bufs == 1 or buf % 128 == 0, where
        assert part <= buf and bufs * buf <= smem <= 227 * 1024, where
        if fwd:
            boxes = part // row // fwd
            assert boxes * fwd * row == part and (boxes == 1 or fwd * row % 128 == 0), where
        for K, bh, upper in (inv[:3], inv[3:]):
            if bh:   # rows 0..K from the start, rows K..2K of the source from `upper`
                boxes = (K + 1) // bh
                assert boxes * bh == K + 1 and upper % 128 == 0 and (boxes == 1 or bh * row % 128 == 0), where
                assert upper + (K + 1) * row <= buf, where
