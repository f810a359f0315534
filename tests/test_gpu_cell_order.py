"""Scans and the stable cell order at the edges of their segments, tiles and passes."""
import numpy as np
import pytest

import chaingen
import oracle
import paper_1001_3764_gb300 as md

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    md.load()


# one pass (512 cells at most) and two; tiles of 1,024 and (above 131,072 atoms) 4,096; one, two and 31 scan segments
@pytest.mark.parametrize("n,M", [(1, 1), (31, 3), (1023, 8), (1024, 9), (8192, 30), (8193, 30), (32768, 8), (32769, 8), (1025, 16), (4097, 17), (131072, 8),
                                 (131073, 9), (200_001, 50), (1 << 20, 5), (1 << 20, 50)])
def test_static_binning_gives_the_stable_order(n, M):
    import torch
    L = 7.25
    x = np.random.default_rng(n + M).uniform(0.0, L, size=(n, 3))
    x[: n // 3] *= 0.3       # uneven cells
    want_cell_of, want_start, want_perm = oracle.bin_atoms(x, L, M)
    pos = torch.from_numpy(np.ascontiguousarray(x.T)).cuda()
    cell_of, perm = (torch.full((n,), -1, dtype=torch.int32, device="cuda") for _ in range(2))
    start = torch.full((M ** 3 + 1,), -1, dtype=torch.int32, device="cuda")
    md.md_bin_static(pos.data_ptr(), n, L, M, cell_of.data_ptr(), start.data_ptr(), perm.data_ptr(),
                     torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    assert np.array_equal(cell_of.cpu().numpy(), want_cell_of)
    assert np.array_equal(start.cpu().numpy(), want_start)
    assert np.array_equal(perm.cpu().numpy(), want_perm)


@pytest.mark.parametrize("L", [17.7, 18.8, 57.0])
def test_system_bins_over_one_and_more_scan_launches(L):
    """16, 17 and 51 cells per side: one segment, two, and more cells than a segment finds its prefix in alone."""
    m = chaingen.melt(12, seed=90, L=L)
    s = md.System(m)
    M = s.info["cells_per_side"]
    cell_of, start, perm = s.bins()
    want_cell_of, want_start, want_perm = oracle.bin_atoms(m["pos"], m["L"], M)
    assert np.array_equal(cell_of, want_cell_of)
    assert np.array_equal(start, want_start)
    assert np.array_equal(perm, want_perm)
    f_orc, _, _ = oracle.System(oracle.chain_topology(150), 12, m["L"], use_cells=False).forces(m["pos"])
    f = s.forces()
    assert np.linalg.norm(f - f_orc) <= 1e-5 * np.linalg.norm(f_orc)
    s.close()
