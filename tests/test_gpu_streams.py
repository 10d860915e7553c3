"""GPU tests of FP64 products in flight at the same time (ExpPart, csrc/blk.cu): a product's fixed-point unit
comes from its own vector's exponents, whatever runs on other streams or in graphs."""
import pytest

torch = pytest.importorskip("torch")

from paper_0706_3293_gb300 import workloads as W

pytestmark = pytest.mark.gpu

N = 16


@pytest.fixture(scope="module")
def prob():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_0706_3293_gb300 import api
    b = api.Basis(N, 1, 0)
    bl = api.BondList.make(*W.ring_bonds(N, -1.0, -0.5))
    gen = torch.Generator("cuda").manual_seed(1)
    big = torch.rand(b.dim, dtype=torch.float64, device="cuda", generator=gen) - 0.5
    small = big * 2.0**-600                               # in the unit of big it is all zeros, big in its unit overflows
    ref = [api.matvec(b, bl, v).clone() for v in (big, small)]
    assert torch.equal(ref[1], ref[0] * 2.0**-600)
    torch.cuda.synchronize()
    return api, b, bl, (big, small), ref


def check(runs, ref):
    torch.cuda.synchronize()
    assert all(torch.equal(y, ref[k]) for k, ys in enumerate(runs) for y in ys)


def test_two_streams_with_many_products_queued(prob):
    api, b, bl, xs, ref = prob
    streams = [torch.cuda.Stream() for _ in xs]
    out = [[torch.empty_like(x) for _ in range(500)] for x in xs]
    torch.cuda.synchronize()
    for k, s in enumerate(streams):
        with torch.cuda.stream(s):
            torch.cuda._sleep(20_000_000)                 # both queues fill before either runs
            for y in out[k]:
                api.matvec(b, bl, xs[k], out=y)
    check(out, ref)


def test_more_streams_than_slots(prob):
    api, b, bl, xs, ref = prob
    b = api.Basis(N, 1, 0)
    streams = [torch.cuda.Stream() for _ in range(24)]
    out = [[torch.empty_like(x) for _ in range(12 * 8)] for x in xs]
    torch.cuda.synchronize()
    for rep in range(8):
        for j, s in enumerate(streams):
            with torch.cuda.stream(s):
                api.matvec(b, bl, xs[j % 2], out=out[j % 2][rep * 12 + j // 2])
    check(out, ref)


def test_graph_replays_beside_eager_products(prob):
    api, b, bl, xs, ref = prob
    graphs, gout = [], []
    for k, x in enumerate(xs):                            # two products a graph
        ys = [torch.empty_like(x) for _ in range(2)]
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            for y in ys:
                api.matvec(b, bl, x, out=y)
        graphs.append(g)
        gout.append(ys)
    eager = [[torch.empty_like(xs[1]) for _ in range(200)]]
    side = [torch.cuda.Stream() for _ in range(3)]
    torch.cuda.synchronize()
    for k, s in enumerate(side):
        with torch.cuda.stream(s):
            torch.cuda._sleep(20_000_000)
            if k < 2:
                for _ in range(100):
                    graphs[k].replay()
            else:
                for y in eager[0]:
                    api.matvec(b, bl, xs[1], out=y)
    check(gout, ref)
    check(eager, ref[1:])


def test_slots_come_back_with_their_graphs(prob):
    """Captures without end on one basis take no more device memory."""
    api, b, bl, xs, ref = prob
    y = torch.empty_like(xs[0])

    def captures(n):
        for _ in range(n):
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g):
                for _ in range(32):
                    api.matvec(b, bl, xs[0], out=y)
            g.replay()
            torch.cuda.synchronize()
            del g
    captures(20)
    torch.cuda.empty_cache()
    before = torch.cuda.mem_get_info()[0]
    captures(200)                                         # 200 x 32 slots of 2 KB would be 13 MB
    torch.cuda.empty_cache()
    assert before - torch.cuda.mem_get_info()[0] < 4 << 20
    assert torch.equal(y, ref[0])
