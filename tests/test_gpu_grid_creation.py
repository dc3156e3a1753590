"""Creating a grid whose levels are solved exactly times no smoothing sweeps:
it launches nothing that its solves do not."""
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [(26, 22, 18), (70, 21, 9)])
def test_no_sweeps_are_timed_where_none_run(n):
    import paper_1901_06427_gb300.binding as B
    before = B.lib().rbfib_launch_count()
    g = B.Grid(n)
    assert B.lib().rbfib_launch_count() == before
    g.close()
