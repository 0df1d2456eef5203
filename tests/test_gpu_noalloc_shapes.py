"""imrt_eval_csr_noalloc at the edges of its row tiles (32 rows, 64 beyond 524,288 voxels) and of its
loads (rounds of 192 entries, two in flight): dose and objective against FP64 sums of the same arrays."""
import ctypes

import numpy as np
import pytest

from paper_0908_4421_gb300 import _lib as L

pytestmark = pytest.mark.gpu


def _csr(rng, m, n, lengths):
    """Rows of the given lengths with random distinct ascending columns."""
    row_ptr = np.zeros(m + 1, np.int64)
    np.cumsum(lengths, out=row_ptr[1:])
    col = np.empty(int(row_ptr[-1]), np.int32)
    for j in np.flatnonzero(lengths):
        k = int(lengths[j])
        start = int(rng.integers(0, n - k + 1))
        col[row_ptr[j]:row_ptr[j + 1]] = np.arange(start, start + k)
    val = rng.uniform(0.01, 1.0, col.size).astype(np.float32)
    return row_ptr, col, val


@pytest.mark.parametrize("m,n,kind", [
    (1, 1, "one"), (31, 700, "ragged"), (32, 700, "ragged"), (33, 700, "ragged"), (257, 513, "edges"),
    (20001, 300, "ragged"), (70, 40, "empty"), (524289, 9, "short"),
])
def test_noalloc_row_tiles(m, n, kind):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    lib = L.load()
    rng = np.random.Generator(np.random.PCG64(m))
    if kind == "one":
        lengths = np.ones(m, np.int64)
    elif kind == "empty":
        lengths = np.zeros(m, np.int64)
    elif kind == "edges":  # around one and two rounds of 192 entries
        lengths = rng.choice([0, 1, 31, 32, 33, 191, 192, 193, 383, 384, 385, 513], m)
    else:
        lengths = np.where(rng.random(m) < 0.4, 0, rng.integers(0, n + 1, m))
    row_ptr, col, val = _csr(rng, m, n, lengths)
    x = rng.uniform(0.0, 2.0, n).astype(np.float32)
    mask = rng.integers(0, 256, m).astype(np.uint8)
    thr = np.array([[3.0, 5.0]] + [[np.nan, 1.0 + s] for s in range(7)], np.float32)
    w = np.array([[2.0, 3.0]] + [[0.0, 1.0 + s] for s in range(7)], np.float32)
    rows = np.repeat(np.arange(m), lengths)
    z64 = np.bincount(rows, val.astype(np.float64) * x[col].astype(np.float64), m)
    G64 = 0.0
    for s in range(8):
        sel = (mask >> s) & 1 == 1
        for k in range(2):
            if sel.sum() and w[s, k] != 0 and not np.isnan(thr[s, k]):
                e = np.maximum(0.0, (1 if k else -1) * (z64[sel] - float(thr[s, k])))
                G64 += float(w[s, k]) / int(sel.sum()) * float((e * e).sum())
    dev = [torch.from_numpy(a).cuda() for a in (row_ptr, col, val, mask, x)]
    z = torch.full((m,), -1.0, device="cuda")
    csr = L.imrt_csr(m, n, col.size, dev[0].data_ptr(), dev[1].data_ptr(), dev[2].data_ptr(), 1)
    G = ctypes.c_double(-1.0)
    for _ in range(2):  # the scratch is shared by all calls: the second sees what the first left
        L.check(lib.imrt_eval_csr_noalloc(ctypes.byref(csr), dev[3].data_ptr(), 8, thr.ctypes.data, w.ctypes.data,
                                          dev[4].data_ptr(), z.data_ptr(), ctypes.addressof(G), 0))
    got = z.cpu().numpy().astype(np.float64)
    # FP32: a lane adds at most ceil(len / 32) products, then 5 shuffle additions
    bound = (np.ceil(lengths / 32) + 6) * 2.0 ** -23 * z64
    assert np.all(np.abs(got - z64) <= bound)
    # the objective's terms are FP64 at the FP32 doses: dG = sum |r_j| |dz_j|, |r_j| <= 2 c e summed over terms
    slack = float(np.max(bound)) * 2 * float(w.sum()) * (float(np.max(z64, initial=0.0)) + 8.0) + 1e-9 * G64
    assert abs(G.value - G64) <= slack
    torch.cuda.synchronize()
