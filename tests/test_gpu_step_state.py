"""What a step leaves behind beside its fields: where the state lies, and what is conserved."""
import numpy as np
import pytest
import torch

from paper_2512_16230_gb300 import workloads as W

from _harness import gpu_model

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _lib(lbm_lib):
    return lbm_lib


def _populations(m, n, seed, scale):
    w = m.lattice.query()["w"].reshape((-1,) + (1,) * len(n))
    return scale * w * (1.0 + np.random.default_rng(seed).uniform(-0.1, 0.1, size=(m.Q,) + tuple(reversed(n))))


# Captured in a CUDA graph on the model's stream, calls of an even number of steps together advance the state by
# as many steps at every replay. 64 x 48 and 20 x 256 run a call in one launch, 631 x 16 runs a launch per step.
@pytest.mark.parametrize("calls", [(20,), (21, 23), (20, 21, 21)])
@pytest.mark.parametrize("store", ["f32", "f16_dev"])
@pytest.mark.parametrize("eq", ["nse", "ncde"])
@pytest.mark.parametrize("name,n,one_launch", [("rD2Q17", (64, 48), True), ("rD2Q25", (20, 256), True),
                                               ("rD2Q13", (631, 16), False)])
def test_replayed_steps_advance_the_state(name, n, one_launch, eq, store, calls):
    spec = W.LATTICES[name]
    rates = np.random.default_rng(3).uniform(0.9, 1.5, spec.R)
    kw = dict(force=(0, 1, 3e-3, 1, 0.4)) if eq == "nse" else dict(u_const=(0.03, 0.06), nonlin=1.0)
    out = []
    for replayed in (False, True):
        stream = torch.cuda.Stream()
        with torch.cuda.stream(stream):
            m = gpu_model(spec, eq, n, rates, store=store, cs2_eq=0.55, **kw)
            m.set_populations(_populations(m, n, 16, 1.0 if eq == "nse" else 0.7))
        if replayed:
            before = m.counters()[1]
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph, stream=stream):
                for k in calls:
                    m.step(k)
            assert m.counters()[1] - before == (len(calls) if one_launch else sum(calls))
            with torch.cuda.stream(stream):
                graph.replay()
                graph.replay()
        else:
            for _ in range(2 * sum(calls)):
                m.step(1)
        out.append(m.get_populations())
        m.close()
    assert np.array_equal(out[0], out[1])
