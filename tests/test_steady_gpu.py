"""Mixed calls on networks created from 64-bit data take solvers with a fixed order of sums
(eig_steady.cu), those on 32-bit data the general ones: both against the oracle and each other
on data that 32 bits hold exactly; chains, a group, a tree, and a result applied to again."""
import numpy as np
import pytest

from oracle import cbc, metrics
from paper_2601_19650_gb300 import _cbc
from synth import make_problem

from test_parity_gpu import MIXED_BAR, _apply_batched, _check_against_oracle

pytestmark = pytest.mark.gpu


def _problem(narrow, wide, **over):
    """A problem on 32-bit values, as 64-bit data where `wide`."""
    p = make_problem(2 if "topo" not in over else 3, dtype=narrow, **over)
    for net in (p.state, p.op):
        net.tensors = [np.asarray(t).astype(narrow).astype(wide or narrow) for t in net.tensors]
    return p


PAIRS = [(np.float32, np.float64), (np.complex64, np.complex128)]


def _twice(p):
    """The operator applied to the state, and to that result."""
    st, op = p.state, p.op
    opt = _cbc.make_options(_cbc.CBC_PREC_MIXED)
    hs = _cbc.create_from_host(st.parent, st.phys, st.bond, st.tensors, "state")
    ho = _cbc.create_from_host(op.parent, op.phys, op.bond, op.tensors, "op")
    one = _cbc.cbc_apply(hs, ho, p.max_bond, p.tol, opt)
    two = _cbc.cbc_apply(one, ho, p.max_bond, p.tol, opt)
    cplx = np.iscomplexobj(st.tensors[0])
    res = [_cbc.fetch_network(h, _cbc.output_shape_fn(st.parent, st.phys), cplx) for h in (one, two)]
    for h in (hs, one, two):
        _cbc.ttn_destroy(h)
    _cbc.ttno_destroy(ho)
    return res


@pytest.mark.parametrize("narrow,wide", PAIRS)
@pytest.mark.parametrize("over", [
    dict(L=2, chi=4, D=2, max_bond=4, seed=1),
    dict(L=12, chi=16, D=4, max_bond=11, seed=2),
    dict(L=9, chi=8, D=3, max_bond=0, seed=3),
    dict(L=10, chi=64, D=8, max_bond=50, seed=4),      # cuts of up to 400
    dict(topo="binary", L=3, chi=12, D=3, max_bond=10, seed=5)])
def test_both_routes(over, narrow, wide):
    a, b = _problem(narrow, None, **over), _problem(narrow, wide, **over)
    ra, rb = _twice(a), _twice(b)
    ref = cbc.cbc(b.state.parent, b.state.tensors, b.op.tensors, b.max_bond, b.tol)
    for (got, bonds, ln) in (ra[0], rb[0]):
        assert list(bonds) == list(ref.out_bonds)
        assert metrics.rel_err(b.state.parent, got, ref.tensors, ln, 0.0) <= MIXED_BAR
    # the second application adds its own error to that of its input on either side
    assert list(ra[1][1]) == list(rb[1][1])
    assert metrics.rel_err(b.state.parent, ra[1][0], rb[1][0], ra[1][2], rb[1][2]) <= 4 * MIXED_BAR


@pytest.mark.parametrize("narrow,wide", PAIRS)
@pytest.mark.parametrize("count", [3, 9])
def test_group(count, narrow, wide):
    # both sides of the rule that gives the Cholesky one CTA per matrix (8 matrices)
    probs = [_problem(narrow, wide, L=9, chi=24, D=4, max_bond=20, seed=40 + j) for j in range(count)]
    res, _ = _apply_batched(probs, _cbc.CBC_PREC_MIXED)
    _check_against_oracle(probs, res, MIXED_BAR)


def test_group_of_both_types():
    probs = [_problem(np.complex64, np.complex128 if j % 2 else None, L=8, chi=16, D=4,
                      max_bond=12, seed=70 + j) for j in range(4)]
    res, _ = _apply_batched(probs, _cbc.CBC_PREC_MIXED)
    _check_against_oracle(probs, res, MIXED_BAR)
