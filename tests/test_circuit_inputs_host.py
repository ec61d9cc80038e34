"""What circuits accept and refuse as gate fields and matrices, and how rows of gate entries
become circuits (host only)."""
import enum

import numpy as np
import pytest

import paper_1905_00444_gb300 as qfx
import rqc_inputs as ri

torch = pytest.importorskip("torch")


def grid(**change):
    c = ri.rqc(3, 3, 8, seed=2)
    for name, value in change.items():
        setattr(c.gates[12], name, value(getattr(c.gates[12], name)))
    return c


@pytest.mark.parametrize("name", ["layer", "q0", "q1", "kind"])
@pytest.mark.parametrize("kind", [float, np.float64, np.float32, str, lambda v: v + 0.5, lambda v: None])
def test_fields_that_are_not_integers_are_refused(name, kind):
    with pytest.raises(TypeError):
        qfx.Circuit(grid(**{name: kind}))


@pytest.mark.parametrize("kind", [int, np.int64, np.int8, np.uint16, lambda v: enum.IntEnum("E", {"a": v}).a,
                                  lambda v: v + 2**32, lambda v: v - 2**70])
def test_integers_of_any_type_are_taken(kind):
    """Those beyond the ABI's 32 bits wrap, as its ctypes record has them."""
    want = qfx.Plan(qfx.Circuit(grid()), n_open=2).steps
    for name in ("layer", "q0", "kind"):
        assert qfx.Plan(qfx.Circuit(grid(**{name: kind})), n_open=2).steps == want


def test_matrices_of_torch_tensors():
    """Complex tensors, also ones that require gradients, as well as numpy arrays; a list has no
    shape and is refused."""
    c = ri.rqc(2, 2, 8, seed=3)
    for g in c.gates:
        g.mat = torch.from_numpy(np.asarray(g.mat)).requires_grad_(True)
    assert qfx.Plan(qfx.Circuit(c), n_open=1).steps == qfx.Plan(qfx.Circuit(ri.rqc(2, 2, 8, seed=3)), n_open=1).steps
    c.gates[0].mat = [[1, 0], [0, 1]]
    with pytest.raises(AttributeError):
        qfx.Circuit(c)


def test_entries_reach_the_abi_unchanged():
    c = ri.rqc(3, 3, 8, seed=2, two_qubit="fsim")
    table = qfx.qfx.gate_table(c.gates, [qfx.qfx._entries(g.mat) for g in c.gates])
    for row, g in zip(table, c.gates):
        flat = np.asarray(g.mat).reshape(-1)
        assert (row["layer"], row["q0"], row["q1"], row["kind"]) == (g.layer, g.q0, g.q1, g.kind)
        np.testing.assert_array_equal(row["mat"][:flat.size], flat)
        assert not row["mat"][flat.size:].any()


def rebuilt(circuit, rows):
    """The entries of every gate of the circuit that the autograd wrapper builds from `rows`."""
    from paper_1905_00444_gb300.autograd import _circuit_with
    c = _circuit_with(circuit, rows)
    if hasattr(c, "compile"):
        assert c.compile().n_gates == len(c.gates)
    return [np.asarray(g.mat).reshape(-1) for g in c.gates]


@pytest.mark.parametrize("shape", [(4,), (16,), (20,), (2, 2), (4, 1), (16, 1), (1, 4), (5, 1, 1)])
def test_rows_of_gate_entries(shape):
    """Rows of any shape whose first 4 elements are 4 values give a gate those values."""
    c = ri.rqc(3, 3, 8, seed=2)
    rows = ri.random_complex((len(c.gates),) + shape, seed=9).astype(np.complex128)
    for mat, row in zip(rebuilt(c, rows), rows):
        np.testing.assert_array_equal(mat, row[:4].reshape(-1))


@pytest.mark.parametrize("shape", [(3,), (4, 4), (2, 8), (1, 16), (1, 2), (2, 4)])
def test_rows_of_other_shapes_are_refused(shape):
    c = ri.rqc(3, 3, 8, seed=2)
    with pytest.raises(ValueError):
        rebuilt(c, np.ones((len(c.gates),) + shape, dtype=np.complex128))


def test_rows_of_general_gates():
    c = ri.rqc(3, 3, 8, seed=2, two_qubit="fsim")
    for shape in ((16,), (16, 1)):
        rows = ri.random_complex((len(c.gates),) + shape, seed=9).astype(np.complex128)
        for mat, row, g in zip(rebuilt(c, rows), rows, c.gates):
            np.testing.assert_array_equal(mat, row.reshape(-1)[:16 if g.q1 >= 0 else 4])
    for shape in ((4,), (20,), (4, 4)):
        with pytest.raises(ValueError):
            rebuilt(c, np.ones((len(c.gates),) + shape, dtype=np.complex128))
    c.gates = [g for g in c.gates if g.q1 >= 0]        # general gates only
    rows = ri.random_complex((len(c.gates), 4, 4), seed=9).astype(np.complex128)
    for mat, row in zip(rebuilt(c, rows), rows):
        np.testing.assert_array_equal(mat, row.reshape(-1))


def test_fewer_rows_than_gates():
    """The circuit has as many gates as there are rows; gates past them are not looked at."""
    c = ri.rqc(3, 3, 8, seed=2)
    n = len(c.gates) - 9
    c.gates.append(ri.rqc(3, 3, 8, seed=2, two_qubit="fsim").gates[9])
    assert len(rebuilt(c, np.ones((n, 4), dtype=np.complex128))) == n
    assert rebuilt(c, np.ones((0, 4), dtype=np.complex128)) == []
