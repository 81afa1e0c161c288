"""Neighbour lists from elements on irregular connectivity: element sizes, unaligned element arrays,
repeated vertices, rows around the in-block list's length and far beyond it, node counts around a
block's size; overflow is refused exactly where the raw entries outgrow the slots."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def F():
    from paper_2408_02758_gb300 import ftle

    return ftle


def rows_of(n, el):
    rows = [set() for _ in range(n)]
    raw = np.zeros(n, dtype=np.int64)
    for e in el.tolist():
        for a in e:
            others = [b for b in e if b != a]
            rows[a].update(others)
            raw[a] += len(others)
    return [sorted(r) for r in rows], int(raw.max()) if n else 0


@pytest.mark.parametrize("v", [2, 3, 4])
@pytest.mark.parametrize("n", [1, 2, 127, 128, 129, 700])
@pytest.mark.parametrize("hub", [0, 31, 32, 33, 150])
def test_irregular_elements(F, v, n, hub):
    import torch

    rng = np.random.default_rng(1000 * v + 10 * n + hub)
    el = rng.integers(0, n, size=(3 * n, v))  # repeated vertices among them
    near = (np.arange(2 * n)[:, None] // 2 + np.arange(v)[None]) % n
    hubs = np.zeros((hub if n > hub else 0, v), dtype=np.int64)
    for k in range(hubs.shape[0]):
        hubs[k, 1:] = 1 + (k + np.arange(v - 1)) % (n - 1)
    el = np.concatenate([el, near, hubs]).astype(np.int32)
    el = el[rng.permutation(len(el))]
    rows, raw = rows_of(n, el)
    store = torch.empty(el.size + 1, dtype=torch.int32, device="cuda")
    for shift in (0, 1):  # 16-byte aligned, and not
        e = store[shift: shift + el.size].view(el.shape)
        e.copy_(torch.from_numpy(el))
        rp, ci = F.ftle_csr_from_elements(n, e, max(1, raw))
        assert rp.cpu().tolist() == [0] + np.cumsum([len(r) for r in rows]).tolist()
        assert ci.cpu().tolist() == [j for r in rows for j in r]
    if raw > 1:
        with pytest.raises(F.FTLEError) as err:
            F.ftle_csr_from_elements(n, e, raw - 1)
        assert err.value.status == F.FTLE_ERANGE
