"""A bounded wait that gives up in a kernel fails the call of the handle that ran it, and no other
handle's: the mark is set from the host (mgwr_inject_give_up), no wait runs out."""
import threading

import pytest

from paper_1608_05400_gb300 import inputs
from paper_1608_05400_gb300 import mgwr as G

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    G.load()


def _solver(precision, d=2, n=31, M=128):
    s = G.Solver(d, n, M, 1.0, 0.5)
    if precision != G.MGWR_FP64:
        s.set_precision(precision)
    s.set_rhs(inputs.random_field(n ** d, M, 3))
    return s


def _solve(s):
    return s.solve(1, 1, 1, tol=1e-8, max_cycles=40)


@pytest.mark.parametrize("precision", [G.MGWR_FP64, G.MGWR_MIXED, G.MGWR_MIXED_DD])
def test_a_mark_fails_its_own_handle_once(precision):
    with _solver(precision) as a, _solver(precision) as b:
        a.inject_give_up()
        _solve(b)
        with pytest.raises(G.MGWRError) as e:
            _solve(a)
        assert e.value.status == G.MGWR_E_CUDA and "gave up" in str(e.value)
        _solve(b)
        _solve(a)


def test_marks_of_handles_on_several_threads():
    handles = [_solver(G.MGWR_FP64) for _ in range(4)]
    for s in handles:
        _solve(s)
    handles[2].inject_give_up()
    status = [None] * 4

    def run(i):
        try:
            _solve(handles[i])
            status[i] = G.MGWR_OK
        except G.MGWRError as e:
            status[i] = e.status

    threads = [threading.Thread(target=run, args=(i,)) for i in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for s in handles:
        s.close()
    assert status == [G.MGWR_OK, G.MGWR_OK, G.MGWR_E_CUDA, G.MGWR_OK]


# every call that runs a half-sweep, a one-point solve or a defect reports it
@pytest.mark.parametrize("call", [
    lambda s, l: s.residual(), lambda s, l: s.defect(G.MGWR_H64, l),
    lambda s, l: s.coarsest(G.MGWR_H64), lambda s, l: s.smooth_defect(G.MGWR_H64, l),
    lambda s, l: s.smooth(G.MGWR_H64, l, G.MGWR_RED), lambda s, l: s.smooth_restrict(G.MGWR_H64, l),
    lambda s, l: s.cycle(G.MGWR_H64, 1, 1, 1)],
    ids=["residual", "defect", "coarsest", "smooth_defect", "smooth", "smooth_restrict", "cycle"])
def test_component_calls_report_a_mark(call):
    with _solver(G.MGWR_FP64) as s:
        l = s.num_levels() - 1
        call(s, l)
        s.inject_give_up()
        with pytest.raises(G.MGWRError) as e:
            call(s, l)
        assert e.value.status == G.MGWR_E_CUDA
        call(s, l)
