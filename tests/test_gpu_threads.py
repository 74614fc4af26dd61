"""Calls of different sizes in threads of one process, each on its own stream: a
kernel's shared-memory limit is one setting of the process, so no call may leave
it below what another thread's launch needs.  Every call succeeds and gives the
bits that it gives alone."""
import threading

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1204_6367_gb300 import inputs  # noqa: E402


@pytest.fixture(scope="module")
def gd():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1204_6367_gb300 import build, gdrr
    build.build()
    gdrr.lib()
    return gdrr


def _filter(gd, nu, stream):
    geo = gd.fdk_geometry(900.0, 1400.0, nu, 2, 0.9, 1.1, (4, 4, 4), (1.0, 1.0, 1.0))
    g = torch.linspace(0.0, 3.0, 2 * nu, device="cuda").reshape(1, 2, nu)
    return lambda: gd.gdrr_fdk_filter(geo, g, stream=stream)


def _transport(gd, pool, stream):
    ctx = gd.Context(inputs.small_problem(), stream=stream)
    gd.gdrr_set_options(ctx, photon_pool=pool)
    return lambda: gd.gdrr_mc_project(ctx, 500, 3)[1]


def _estimator(gd, c, stream):
    net = gd.Cnn(1, 16, 16, c, stream=stream)
    x = torch.linspace(0.0, 1.0, 512, device="cuda").reshape(1, 2, 16, 16)
    y = torch.linspace(0.0, 1.0, 256, device="cuda").reshape(1, 1, 16, 16)

    def run():
        net.forward(x)
        net.backward(y)
        return torch.from_numpy(net.get_grads())
    return run


def _denoiser(gd, nu, stream):
    ctx = gd.Context(inputs.small_problem(), stream=stream)
    s = torch.linspace(10.0, 30.0, nu * 600, dtype=torch.float64, device="cuda").reshape(600, nu)
    return lambda: gd.gdrr_denoise_scatter(ctx, s, 1.0, 0.05, iters=2)


@pytest.mark.parametrize("make, sizes", [(_filter, (4096, 64)), (_transport, (3, 1)), (_estimator, (64, 32)),
                                         (_denoiser, (900, 820))])
def test_calls_of_other_sizes_in_other_threads(gd, make, sizes):
    streams = [torch.cuda.Stream() for _ in sizes]
    errors, start = [], threading.Barrier(len(sizes))

    def work(size, stream):
        try:
            with torch.cuda.stream(stream):
                run = make(gd, size, stream)
                first = run()
                stream.synchronize()
                start.wait()
                for _ in range(1500):
                    out = run()
                stream.synchronize()
                assert torch.equal(out, first)
        except BaseException as e:                          # reported by the test's own thread
            errors.append((size, repr(e)))
            start.abort()

    threads = [threading.Thread(target=work, args=a) for a in zip(sizes, streams)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors
