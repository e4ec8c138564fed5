"""How the library's kernels are launched, from a trace of the launches."""
import json

import pytest

from paper_1909_06374_gb300 import LC_FP32, LC_FP64, Plan, workloads

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _trace_once(call, tmp_path):
    path = tmp_path / "trace.json"
    torch.cuda.synchronize()
    with torch.profiler.profile(activities=[torch.profiler.ProfilerActivity.CUDA]) as prof:
        call()
        torch.cuda.synchronize()
    prof.export_chrome_trace(str(path))
    return json.loads(path.read_text())["traceEvents"]


def _trace(call, tmp_path):
    for _ in range(2):  # the first trace of a process may come without kernels
        events = _trace_once(call, tmp_path)
        if any(e.get("cat") == "kernel" for e in events):
            return events
    pytest.skip("no kernel activity records on this machine")


@pytest.mark.parametrize("prec", [LC_FP32, LC_FP64])
@pytest.mark.parametrize("curves,log2n", [(1, 10), (1, 14), (1, 16), (8, 16), (64, 14), (1, 20)])
def test_periodogram_of_a_few_curves_spreads_over_the_gpu(curves, log2n, prec, tmp_path):
    """At least a block per 256 pairs of bins or two blocks per SM, whichever is fewer."""
    with Plan([workloads.job(log2n, 0, seed=c, curve_id=c) for c in range(curves)], prec) as p:
        x = torch.rand(p.total, dtype=p.dtype, device="cuda")
        events = _trace(lambda: p.periodogram(x), tmp_path)
    grids = [e["args"]["grid"][0] for e in events if e.get("cat") == "kernel" and "k_periodogram" in e["name"]]
    assert len(grids) == 1
    pairs = curves << (log2n - 2)
    assert grids[0] >= min(pairs // 256, 2 * torch.cuda.get_device_properties(0).multi_processor_count)


@pytest.mark.parametrize("prec,curves,log2n,threads", [(LC_FP64, 1, 16, 128), (LC_FP64, 128, 16, 256),
                                                       (LC_FP64, 16, 18, 256), (LC_FP32, 1, 16, 128),
                                                       (LC_FP32, 8, 17, 256), (LC_FP32, 200, 13, 256),
                                                       (LC_FP32, 4, 19, 256)])
def test_batches_take_full_tiles(prec, curves, log2n, threads, tmp_path):
    """Tiles of few columns (128 threads) where full ones would leave most of
    the GPU idle, and only there."""
    with Plan([workloads.job(log2n, 0, seed=c, curve_id=c) for c in range(curves)], prec) as p:
        x = torch.rand(p.total, dtype=p.dtype, device="cuda")
        events = _trace(lambda: p.periodogram(x), tmp_path)
    blocks = {e["args"]["block"][0] for e in events if e.get("cat") == "kernel" and "k_fft_tile" in e["name"]}
    assert blocks == {threads}


@pytest.mark.parametrize("log2n,iters,calls,graphs", [(13, 8, 4, [8, 8, 2, 2]), (13, 10, 2, [10, 4]),
                                                      (13, 34, 2, [10, 10]), (8, 34, 3, [34, 34, 10]),
                                                      (8, 100, 1, [25])])
def test_graphs_of_several_iterations_where_they_repay(log2n, iters, calls, graphs, tmp_path):
    """A plan of few iterations replays a graph of one: the longer graph's
    instantiation costs more than it saves until enough have been run."""
    with Plan([workloads.job(log2n, iters, seed=3, curve_id=0)], LC_FP32) as warm:
        _trace(warm.generate, tmp_path)
    with Plan([workloads.job(log2n, iters, seed=3, curve_id=0)], LC_FP32) as p:
        p.setup()
        x = p.get_state()
        for want in graphs[:calls]:
            events = _trace_once(lambda: p.iterate(iters), tmp_path)
            got = sum(e.get("name", "").startswith("cudaGraphLaunch") for e in events)
            assert got == want
            p.set_state(x)
