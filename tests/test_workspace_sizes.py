"""A workspace sized for a program's largest batch serves its shorter ones: neither size falls as rows are added (host only)."""

import pytest


@pytest.mark.parametrize("block", [128, 32, 0, -32])
@pytest.mark.parametrize("d,V", [(256, 1024), (640, 2056), (4096, 151936), (5120, 4096), (8192, 9224)])
@pytest.mark.parametrize("vocab_chunk", [0, 2048])
def test_workspace_sizes_do_not_fall_with_rows(d, V, block, vocab_chunk):
    import paper_2605_13907_b200 as ais
    params = ais.default_params(vocab_chunk=vocab_chunk)
    rows = list(range(0, 8192, 61)) + [int(8192 * 1.07 ** k) for k in range(70)]
    least = size = 0
    for T in rows:
        shape = ais.make_shape(T, d, V, 2, 4, block)
        m, n = ais.workspace_min_bytes(shape, params), ais.workspace_bytes(shape, params)
        assert least <= m <= n and size <= n, T
        least, size = m, n
