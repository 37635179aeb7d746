"""The surrogate network beyond its accuracy at ordinary sizes: its state on creation."""
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def pkg():
    import paper_2210_07501_gb300 as p
    p.build()
    p.load()
    return p


@pytest.mark.parametrize("own_stream", [False, True])
def test_new_network_runs_on_the_parameters_it_reports(pkg, own_stream):
    """A network reads its weights from copies laid out for the kernels; on creation, too, they are those
    of the parameters: outputs before any set_params are bit for bit those after putting the
    reported parameters back.  Many networks in a row, on a stream that nothing else orders."""
    x = torch.randn((1, 12, 17, 33), device="cuda")
    y0, y1 = (torch.empty((1, 4, 17, 33), device="cuda") for _ in range(2))
    for seed in range(20):
        stream = torch.cuda.Stream() if own_stream else torch.cuda.current_stream()
        torch.cuda.synchronize()
        net = pkg.Cnn(17, 33, batch_max=1, seed=seed, stream=stream)
        net.forward(x, y0)
        net.set_params(net.get_params())
        net.forward(x, y1)
        torch.cuda.synchronize()
        assert float(y0.abs().max()) > 0 and torch.equal(y0, y1), seed
        net.close()
