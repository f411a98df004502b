"""Products of one context from two host threads on one stream, on two streams,
and as replays of captured graphs beside them: every result is the lone
product's, bit for bit.  The small mesh takes the scratch of fe_small.h, the
large one the colour-ordered launches."""
import threading

import pytest

from paper_2208_07129_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SMALL, LARGE = (3, 3, 2), (5, 4, 4)      # below and above the small-mesh limit at p = 6
MODES = ["fp64", "df64", "fp32"]
RUNS = 50


@pytest.fixture(scope="module")
def fe():
    from paper_2208_07129_gb300 import build, fe as fe_mod
    build.build()
    fe_mod.lib()
    return fe_mod


class Case:
    """A context, two inputs and the results of their lone products."""

    def __init__(self, fe, n, bent, mode, nv=16):
        self.fe = fe
        self.ctx = fe.fe_setup(*n, 6, 8, vertices=inputs.perturbed_vertices(*n, seed=1) if bent else None)
        fe.fe_set_potential(self.ctx, inputs.coulomb_potential(fe.fe_quadrature_points(self.ctx)))
        fe.fe_set_mode(self.ctx, mode)
        dt = torch.float32 if mode == "fp32" else torch.float64
        self.X = [torch.from_numpy(inputs.random_block(fe.fe_num_dofs(self.ctx), nv, "normal", 5 + k)).to("cuda", dt)
                  for k in range(2)]
        self.want = [torch.empty_like(x) for x in self.X]
        for x, y in zip(self.X, self.want):
            fe.fe_apply(self.ctx, x, y)
        torch.cuda.synchronize()

    def blocks(self, k):
        return [torch.full_like(self.X[k], float("nan")) for _ in range(RUNS)]

    def check(self, Y):
        torch.cuda.synchronize()
        for k in range(2):
            assert all(torch.equal(y, self.want[k]) for y in Y[k])

    def capture(self, k, y, runs=1):
        s, g = torch.cuda.Stream(), torch.cuda.CUDAGraph()
        s.wait_stream(torch.cuda.current_stream())
        with torch.cuda.graph(g, stream=s):
            for _ in range(runs):
                self.fe.fe_apply(self.ctx, self.X[k], y)
        return g


@pytest.fixture
def case(fe, request):
    made = []

    def make(*args):
        made.append(Case(fe, *args))
        return made[-1]

    yield make
    torch.cuda.synchronize()
    for c in made:
        fe.fe_destroy(c.ctx)


@pytest.mark.parametrize("mode", MODES)
@pytest.mark.parametrize("bent", [False, True])
def test_two_threads_on_one_stream(case, mode, bent):
    c = case(SMALL, bent, mode)
    s = torch.cuda.Stream()
    Y = [c.blocks(k) for k in range(2)]
    torch.cuda.synchronize()
    gate = threading.Barrier(2)

    def work(k):
        gate.wait()
        for y in Y[k]:
            c.fe.fe_apply(c.ctx, c.X[k], y, stream=s)

    threads = [threading.Thread(target=work, args=(k,)) for k in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    c.check(Y)


@pytest.mark.parametrize("mode", MODES)
@pytest.mark.parametrize("bent", [False, True])
@pytest.mark.parametrize("n", [SMALL, LARGE])
def test_two_streams(case, mode, bent, n):
    c = case(n, bent, mode)
    streams = [torch.cuda.Stream() for _ in range(2)]
    Y = [c.blocks(k) for k in range(2)]
    torch.cuda.synchronize()
    for r in range(RUNS):
        for k in range(2):
            c.fe.fe_apply(c.ctx, c.X[k], Y[k][r], stream=streams[k])
    c.check(Y)


@pytest.mark.parametrize("mode", MODES)
def test_streams_that_come_and_go(case, mode):
    c = case(SMALL, False, mode)
    Y = [c.blocks(k) for k in range(2)]
    torch.cuda.synchronize()
    for r in range(RUNS):
        for k in range(2):
            c.fe.fe_apply(c.ctx, c.X[k], Y[k][r], stream=torch.cuda.Stream(priority=-(r & 1)))
    c.check(Y)


@pytest.mark.parametrize("mode", MODES)
@pytest.mark.parametrize("bent", [False, True])
def test_replays_beside_products(case, mode, bent):
    """Two graphs (two products each) on two streams, products on a third."""
    c = case(SMALL, bent, mode)
    G = [torch.full_like(x, float("nan")) for x in c.X]
    graphs = [c.capture(k, G[k], runs=2) for k in range(2)]
    Y = [c.blocks(k) for k in range(2)]
    streams = [torch.cuda.Stream() for _ in range(3)]
    torch.cuda.synchronize()
    for r in range(RUNS):
        for k in range(2):
            with torch.cuda.stream(streams[k]):
                graphs[k].replay()
            c.fe.fe_apply(c.ctx, c.X[k], Y[k][r], stream=streams[2])
    c.check(Y)
    c.check([[G[0]], [G[1]]])


@pytest.mark.parametrize("mode", MODES)
def test_more_captures_than_blocks(case, mode):
    """Captures past the last block run colour by colour; destroyed graphs give
    their blocks back."""
    c = case(SMALL, False, mode)
    for _ in range(3):
        Y = [torch.full_like(c.X[k & 1], float("nan")) for k in range(19)]
        graphs = [c.capture(k & 1, Y[k]) for k in range(19)]
        streams = [torch.cuda.Stream() for _ in range(19)]
        torch.cuda.synchronize()
        for _ in range(10):
            for g, s in zip(graphs, streams):
                with torch.cuda.stream(s):
                    g.replay()
        torch.cuda.synchronize()
        for k in range(19):
            assert torch.equal(Y[k], c.want[k & 1])
        del graphs


@pytest.mark.parametrize("mode", MODES)
def test_forked_capture(case, mode):
    """Parallel branches of one graph do not share a block."""
    c = case(SMALL, False, mode)
    Y = [torch.full_like(x, float("nan")) for x in c.X]
    a, b, g = torch.cuda.Stream(), torch.cuda.Stream(), torch.cuda.CUDAGraph()
    a.wait_stream(torch.cuda.current_stream())
    with torch.cuda.graph(g, stream=a):
        b.wait_stream(a)
        c.fe.fe_apply(c.ctx, c.X[0], Y[0], stream=a)
        c.fe.fe_apply(c.ctx, c.X[1], Y[1], stream=b)
        a.wait_stream(b)
    for _ in range(RUNS):
        g.replay()
    c.check([[Y[0]], [Y[1]]])
