"""Where the FP32 path keeps a layer's partial sums, replayed on the CPU: the records that
tiles of side 32, 64 and 128 write, and those that the round's sums read, are the same set
of quarters of the 128 x 128 blocks, and a tile's record lies in the quarter it is in."""
import numpy as np
import pytest


def simt_record(T, bi, bj):
    S = 128 // T
    i, j, u, v = bi // S, bj // S, bi % S, bj % S
    place = (v & 1) | ((u & 1) << 1) | ((v & 2) << 1) | ((u & 2) << 2)
    return (j * (j + 1) // 2 + i) * (16 if S == 4 else 4) + place


def is_diagonal(k):
    root = int(np.sqrt(np.float32(8 * k + 9)) + np.float32(0.5))
    return root * root == 8 * k + 9


def records_read(sub, cnt):
    out = set()
    for k in range(cnt):
        for q in range(4):
            if is_diagonal(k) and q == 2:
                continue
            for e in range(sub):
                if not (sub == 4 and e == 2 and is_diagonal(k) and q != 1):
                    out.add((k * 4 + q) * sub + e)
    return out


def test_diagonal_blocks_are_squares():
    diagonal = {j * (j + 3) // 2 for j in range(512)}   # N up to 65536
    for k in list(range(2000)) + sorted(diagonal) + [d + e for d in sorted(diagonal) for e in (-1, 1) if d > 0]:
        assert is_diagonal(k) == (k in diagonal)


@pytest.mark.parametrize("np_", [128, 256, 384, 768, 1664])
@pytest.mark.parametrize("T", [32, 64, 128])
def test_records_written_are_the_records_read(T, np_):
    n, cnt = np_ // T, np_ // 128 * (np_ // 128 + 1) // 2
    sub = 4 if T == 32 else 1
    written = {}
    for bj in range(n):
        for bi in range(bj + 1):
            for g in range(4 if T == 128 else 1):
                r = simt_record(T, bi, bj) + g
                assert r not in written
                written[r] = (bi, bj, g)
    read = records_read(sub, cnt)
    if T == 128:   # a diagonal tile also writes its quarter below the diagonal, a zero
        written = {r: w for r, w in written.items() if not (w[0] == w[1] and w[2] == 2)}
    assert set(written) == read
    for r, (bi, bj, g) in written.items():
        block, quarter = r // (4 * sub), r // sub % 4
        row, col = bi * T + (g >> 1) * 64, bj * T + (g & 1) * 64
        assert block == (col // 128) * (col // 128 + 1) // 2 + row // 128
        assert quarter == (row // 64 % 2) * 2 + col // 64 % 2
