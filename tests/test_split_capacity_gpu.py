"""The split CG's largest systems: a CTA's rows, halo and copy buffers fill its
shared memory.  A strip of cameras (each coupled to the next two) takes 32 copy
buffers of 4,736 bytes, 80 bytes a halo camera, 80 a row for its record, 24 for
its sums and 48 a pass of 32 entries: 190 bytes a row, and 226 KB hold 420 rows on
each SM; the 4 bytes of a row's start must not take that away.  Whether the split
recurrence ran shows in its phase times (profile 2), which the standard one
leaves at zero."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows,split", [(300, True), (400, True), (416, True), (440, False)])
def test_rows_per_cta(rows, split):
    import torch

    from paper_2307_08383_gb300.build import build
    build()
    import paper_2307_08383_gb300 as B
    n = rows * torch.cuda.get_device_properties(0).multi_processor_count
    pairs = np.arange(n)[:, None] + np.arange(3)
    col = pairs[pairs < n].astype(np.int32)
    row_ptr = np.concatenate([[0], np.cumsum((pairs < n).sum(1))]).astype(np.int32)
    row = np.repeat(np.arange(n), np.diff(row_ptr))
    rng = np.random.default_rng(rows)
    val = rng.integers(-8, 9, (len(col), 6, 6)) / 16.0
    d = row_ptr[:-1]  # diagonal blocks
    val[d] = val[d] + val[d].transpose(0, 2, 1)
    val[d] += 24.0 * np.eye(6)
    b = rng.integers(-200, 201, (n, 6)) / 16.0
    g = B.Problem.from_rcs(row_ptr, col, val, b, precision=B.BA_FP32, pcg_rel_tol=1e-5, profile=2)
    info, conv = g.solve_rcs()
    assert conv
    x = g.step()[0].reshape(n, 6)
    assert (g.stats()["pcg_phase_us"][0] > 0) == split
    g.close()
    r = b.copy()
    np.subtract.at(r, row, np.einsum("kab,kb->ka", val, x[col]))
    off = row != col
    np.subtract.at(r, col[off], np.einsum("kba,kb->ka", val[off], x[row[off]]))
    assert np.linalg.norm(r) <= (1e-5 + 150 * 2.0 ** -24) * np.linalg.norm(b)
