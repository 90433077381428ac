"""Samples per gridding chunk: four in launches that fit the chip at once,
eight in larger ones, launch by launch (eight pieces of a plan each). The
chunks of a piece's fullest lattice tile are counted again from the positions
of its samples and compared with what the plan reports; counts for four and
eight samples lie almost a factor of two apart."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

ROWS, COLS, TAPS = 32, 64, 4          # lattice cells of a tile, taps per axis


@pytest.fixture(scope="module")
def hr():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1604_07651_gb300 as hr
    return hr


def _most_chunks(plan, piece, length):
    """Most chunks of at most `length` consecutive samples of a trace that one tile holds."""
    theta, rho, w = plan.piece_samples(piece)
    m0, n0 = np.floor(theta).astype(int) - 1, np.floor(rho).astype(int) - 1
    tiles = {}
    for dm in (0, TAPS - 1):
        for dn in (0, TAPS - 1):
            for t, c in zip(*np.unique(((m0 + dm) // ROWS * 4096 + (n0 + dn) // COLS)[w != 0], return_counts=True)):
                tiles[t] = max(tiles.get(t, 0), c)
    most = 0
    for t in sorted(tiles, key=tiles.get)[-8:]:
        ti, tj = divmod(int(t), 4096)
        on = ((w != 0) & (m0 < (ti + 1) * ROWS) & (m0 + TAPS > ti * ROWS) & (n0 < (tj + 1) * COLS) & (n0 + TAPS > tj * COLS))
        edge = np.diff(np.pad(on, ((0, 0), (1, 1))).astype(np.int8), axis=1)
        runs = np.nonzero(edge == -1)[1] - np.nonzero(edge == 1)[1]
        most = max(most, int(np.sum(-(-runs // length))))
    return most


@pytest.mark.parametrize("Nt,Nx,nq,want", [
    (600, 600, 1, [4] * 3),
    (1024, 256, 3, [8] * 8 + [4]),
    (600, 600, 5, [8] * 15),
    (1024, 256, 8, [8] * 24),
])
def test_chunk_length_by_launch(hr, Nt, Nx, nq, want):
    plan = hr.Plan(Nt, Nx, Nt, Nx, 2.0 / (Nt - 1), 2.0 / (Nx - 1), 0.2, 0.7, n_qsplit=nq)
    pieces = plan.pieces()
    assert len(pieces) == len(want)
    for i in {0, len(want) // 2, len(want) - 2, len(want) - 1}:
        n = _most_chunks(plan, i, want[i])
        assert abs(pieces[i]["grid_max_tile_chunks"] - n) <= 0.02 * n, (i, n)
    plan.close()
