"""How many BiCGSTAB iterations a captured graph holds, for every convergence-check interval a caller may ask for:
a whole number of graphs makes up the interval, and no graph is shorter than three iterations unless the interval is
(an interval of 7 ran as seven graphs of one iteration). CPU."""
import ctypes as C


def test_graphs_fill_the_interval():
    from paper_1712_08743_gb300 import _lib, build

    build.build()
    iters = _lib.load()._ZN4helm16bicg_graph_itersEi   # int helm::bicg_graph_iters(int)
    iters.restype, iters.argtypes = C.c_int, [C.c_int]
    for chunk in range(1, 1001):
        k = iters(chunk)
        assert chunk % k == 0 and (k >= 3 or k == chunk)
        assert k <= 5 or not any(chunk % q == 0 for q in (3, 4, 5))
    assert iters(10) == 5 and iters(7) == 7 and iters(22) == 11
