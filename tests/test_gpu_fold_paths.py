"""The fold's launches against one another and against the state vector: one launch that folds
and scales (few elements), an element per thread, groups of four elements."""
import numpy as np
import pytest

import rqc_inputs as ri
from oracle import statevector

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def bits(x):
    return torch.tensor(np.asarray(x, dtype=np.uint64).view(np.int64), device="cuda")


def amplitudes(qfx, plan, x1s, items):
    ws = torch.empty(plan.workspace_bytes(items), dtype=torch.uint8, device="cuda")
    out = qfx.amplitudes(plan, bits(x1s), workspace=ws)
    qfx.sync()
    return out


@pytest.mark.parametrize("items", [1, 640])
def test_scale_ignores_entries_that_overflow(qfx, items):
    """Open sites whose last gate is diag(1e-25, 1e300): the second entry overflows FP32 and
    becomes NaN, the first ones need the site's scale (the product of two of them lies below
    FP32).  The amplitudes of the first entries are FP32-accurate whatever the others are."""
    c = ri.rqc(2, 2, 8, seed=4)
    plain = ri.rqc(2, 2, 8, seed=4)
    last = max(g.layer for g in c.gates)
    for grid, mat in ((c, np.diag([1e-25, 1e300])), (plain, np.eye(2))):
        for i, g in enumerate(grid.gates):
            if g.layer == last and g.q0 in (0, 3):
                grid.gates[i] = ri.Gate(g.layer, g.q0, -1, ri.U1, mat.astype(np.complex128))
    plan = qfx.Plan(qfx.Circuit(c), open_sites=[0, 1, 2, 3])
    got = amplitudes(qfx, plan, [0] * items, items).cpu().numpy()
    psi = statevector.amplitudes(plain)
    for j in range(16):
        x = sum(((j >> i) & 1) << q for i, q in enumerate(plan.open_sites))
        if x & 0b1001 == 0:
            want = 1e-50 * psi[x]
            assert np.all(np.abs(got[:, j] - want) <= 1e-5 * max(abs(want), 1e-50 * 2.0 ** -2)), (j, got[0, j], want)


@pytest.mark.parametrize("shape,n_batch", [((2, 2, 56), 160), ((1, 2, 64), 640)])
def test_more_events_than_one_stage_holds(qfx, shape, n_batch):
    """72 and 74 events a site, above the 64 that one stage in shared memory holds.  (2, 2, 56):
    one item of 2^14-element sites takes an element per thread; (1, 2, 64): one item of 256
    elements folds and scales in one launch; all items together take groups of four.  The same
    bits, and the state vector's amplitudes."""
    rows, cols, d = shape
    c = ri.rqc(rows, cols, d, seed=5)
    plan = qfx.Plan(qfx.Circuit(c), n_open=1)
    x1s = ri.random_bitstrings(rows * cols, n_batch, seed=6)
    many = amplitudes(qfx, plan, x1s, n_batch)
    one = torch.cat([amplitudes(qfx, plan, x1s[i:i + 1], 1) for i in range(0, n_batch, 53)])
    assert torch.equal(many[::53], one)
    psi = statevector.amplitudes(c)
    q = plan.open_sites[0]
    want = np.array([[psi[(int(x) & ~(1 << q)) | (j << q)] for j in range(2)] for x in x1s])
    err = np.abs(many.cpu().numpy() - want)
    assert np.all(err <= 1e-5 * np.maximum(np.abs(want), 2.0 ** (-rows * cols / 2)))
