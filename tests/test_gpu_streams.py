"""One handle over several streams: its calls share a workspace and the counters by
which a launch's last block finishes a sum, so what it enqueues on one stream
comes before what it enqueues on the next.  Small whole numbers: every sum is
exact, and each call's result is compared."""
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def aunmf():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_1609_09154_gb300 import aunmf

    return aunmf


def ints(g, *shape):
    return torch.randint(-3, 4, shape, generator=g, device="cuda").float()


@pytest.mark.parametrize("order", [(0, 1), (0, 1, 2, 1), (0, 3, 1)])
def test_calls_that_follow_each_other_on_several_streams(aunmf, order):
    """Big and small Grams and losses in turn (grids of other sizes, no
    synchronisation between them), then each on one stream alone."""
    g = torch.Generator(device="cuda")
    g.manual_seed(1)
    streams = [torch.cuda.Stream() for _ in range(3)] + [torch.cuda.default_stream()]
    h = aunmf.Handle(stream=streams[0])
    Xs = [ints(g, r, k) for r, k in ((300000, 12), (700, 10), (5000, 17), (40000, 96))]
    Gs = [(X.double().T @ X.double()).float() for X in Xs]
    A, W, H = ints(g, 1500, 900), ints(g, 1500, 6), ints(g, 6, 900)
    L = 0.5 * ((A.double() - W.double() @ H.double()) ** 2).sum()
    torch.cuda.synchronize()
    for _ in range(4):
        got, losses = [], []
        for i in range(24):
            s = streams[order[i % len(order)]]
            h.set_stream(s)
            with torch.cuda.stream(s):
                got.append((h.gram_w(Xs[i % 4]), i % 4))
                losses.append(h.loss_fwd(A, W, H, "tf32")[0])
        torch.cuda.synchronize()
        assert all(torch.equal(G, Gs[j]) for G, j in got)
        assert all(float(x) == float(L) for x in losses)
    with torch.cuda.stream(streams[1]):
        h.set_stream(streams[1])
        assert all(torch.equal(h.gram_w(X), G) for X, G in zip(Xs, Gs))
    torch.cuda.synchronize()
    h.close()


def test_autograd_on_two_streams(aunmf):
    from paper_1609_09154_gb300.autograd import nmf_loss

    g = torch.Generator(device="cuda")
    g.manual_seed(2)
    A = ints(g, 3000, 2000)
    W, H = ints(g, 3000, 7).requires_grad_(), ints(g, 7, 2000).requires_grad_()
    D = (W.double() @ H.double() - A.double()).detach()
    dW, dH = (D @ H.double().T.detach()).float(), (W.double().T.detach() @ D).float()
    torch.cuda.synchronize()
    out = []
    for i in range(6):
        with torch.cuda.stream(torch.cuda.Stream()):
            out.append((nmf_loss(A, W, H, "tf32"), *torch.autograd.grad(nmf_loss(A, W, H), (W, H))))
    torch.cuda.synchronize()
    for loss, a, b in out:
        assert float(loss.detach()) == float(0.5 * (D ** 2).sum()) and torch.equal(a, dW) and torch.equal(b, dH)


def test_calls_captured_in_a_graph(aunmf):
    """A handle used on one stream, captured on another, then used on a third."""
    g = torch.Generator(device="cuda")
    g.manual_seed(3)
    X, Y = ints(g, 200000, 12), ints(g, 3000, 9)
    GX, GY = (X.double().T @ X.double()).float(), (Y.double().T @ Y.double()).float()
    h = aunmf.Handle()
    big = h.gram_w(X)  # the workspace, and work under way when the capture begins
    h.gram_w(Y)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        h.set_stream(torch.cuda.current_stream())
        G1 = h.gram_w(X)
        G2 = h.gram_w(Y)
    s = torch.cuda.Stream()
    h.set_stream(s)
    for _ in range(3):
        with torch.cuda.stream(s):
            G3 = h.gram_w(Y)
            G1.zero_()
            graph.replay()
            G4 = h.gram_w(X)
        torch.cuda.synchronize()
        assert torch.equal(G1, GX) and torch.equal(G2, GY) and torch.equal(G3, GY) and torch.equal(G4, GX)
    assert torch.equal(big, GX)
    h.set_stream(torch.cuda.current_stream())
    h.close()


def test_first_call_captured(aunmf):
    """A handle whose first call of all is captured: its counters start at 0 for the
    calls that follow, whether or not the graph has run."""
    g = torch.Generator(device="cuda")
    g.manual_seed(4)
    X, Y = ints(g, 1500, 10), ints(g, 900, 9)
    GX, GY = (X.double().T @ X.double()).float(), (Y.double().T @ Y.double()).float()
    h = aunmf.Handle()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, capture_error_mode="relaxed"):
        h.set_stream(torch.cuda.current_stream())
        G1 = h.gram_w(X)
    h.set_stream(torch.cuda.current_stream())
    assert torch.equal(h.gram_w(Y), GY)
    for _ in range(2):
        graph.replay()
        assert torch.equal(h.gram_w(Y), GY)
        assert torch.equal(G1, GX)
    h.close()
