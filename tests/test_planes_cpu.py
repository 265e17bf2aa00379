"""Block, lane and padding arithmetic of the 3D updates along a plane's
elements, replayed on the host: every node of a plane is taken exactly once by
the two-node, the one-node and the even binary16 update, for rows with and
without ghost nodes and every block size the autotuner tries."""
import pytest


def pitch(n0, n1, ghost):
    """SX, SY of a 3D level (build_view)."""
    old = (-(-(n0 + 2 * ghost) // 32) * 32, n1 + 2 * ghost)
    sx = -(-(n0 + 2 * ghost) // 8) * 8
    lines = 1 if sx % 32 == 0 else 2 if sx % 16 == 0 else 4
    sy = -(-(n1 + 2 * ghost) // lines) * lines
    return (sx, sy) if sx * sy <= old[0] * old[1] else old


@pytest.mark.parametrize("n0,n1", [(4, 4), (5, 7), (32, 9), (33, 8), (63, 5), (65, 6), (81, 10),
                                   (160, 4), (161, 7), (193, 5), (257, 3)])
@pytest.mark.parametrize("ghost", [0, 1])
def test_every_node_once(n0, n1, ghost):
    sx, sy = pitch(n0, n1, ghost)
    assert sx >= n0 + 2 * ghost and sx % 8 == 0 and sx * sy % 32 == 0 or sx % 32 == 0
    for threads in (32, 64, 96, 128):
        for nodes, width in ((2, 1), (1, 1), (1, 2)):  # two rows; one node; two of a row
            row = sx // width
            last = (-(-n1 // nodes) - 1) * row + -(-n0 // width)
            blocks = -(-last // threads)
            seen = []
            for e in range(blocks * threads):
                y, x = e // row * nodes, e % row * width
                if x >= n0 or y >= n1:
                    continue
                seen += [(x + dx, y + dy) for dy in range(nodes) for dx in range(width)
                         if x + dx < n0 and y + dy < n1]
            assert len(seen) == n0 * n1 == len(set(seen))
