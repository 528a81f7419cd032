"""What a step leaves behind beside its fields: where the state lies, and what is conserved."""
import numpy as np
import pytest
import torch

from paper_2512_16230_gb300 import workloads as W

from _harness import gpu_model, oracle_lattice

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


def _coefficient_drift(spec, s_high, s_orders):
    """Largest relative change of the mass in a step by rounding the operator of the higher rows to FP32: each of
    its coefficients by 2^-24 of itself, the diagonal 1 - s_high and, for an order k with a rate of its own,
    sum_ij w_i w_j |P_ij| |s_k - s_high|, P the W-orthogonal projector on the rows of that order."""
    lat = oracle_lattice(spec)
    total = abs(1.0 - s_high)
    for k, s in s_orders.items():
        B = lat.Hfull[[r for r, o in enumerate(lat.full_orders) if o == k]]
        P = B.T @ np.linalg.inv((B * lat.w) @ B.T) @ B
        total += abs(s - s_high) * float(lat.w @ np.abs(P) @ lat.w)
    return 2.0 ** -24 * total


# One rate per order >= 4 in FP32, with rates that FP32 does not hold: 1.05 is 4.8e-8 off, which the step must not
# multiply the mass by. One cell and two cells per thread, and batched.
@pytest.mark.parametrize("name,n,batched", [("rD3Q53", (32, 32, 32), False), ("rD3Q53", (48, 48, 48), False),
                                            ("rD3Q53", (32, 32, 32), True)])
def test_order_rates_conserve_mass(name, n, batched):
    from paper_2512_16230_gb300 import lbm
    spec, s_high, s_orders, steps = W.LATTICES[name], 1.05, {4: 1.1}, 200
    d, cells = len(n), int(np.prod(n))
    # a vortex of a tenth of the lattice speed, so that no two cells round alike
    x = [np.arange(k) * (2 * np.pi / k) for k in n]
    X = np.meshgrid(*reversed(x), indexing="ij")[::-1]
    u = np.zeros((d,) + tuple(reversed(n)))
    u[0], u[1] = 0.1 * np.sin(X[0]) * np.cos(X[1]), -0.1 * np.cos(X[0]) * np.sin(X[1])
    rho = 1.0 + np.random.default_rng(17).uniform(-0.01, 0.01, size=tuple(reversed(n)))
    m = gpu_model(spec, "nse", n, W.rates_nse(d, 0.01, spec.cs2[0], spec=spec), s_high=s_high, store="f32",
                  s_orders=s_orders)
    m.init_fields(rho, u)
    before = m.conserved_sums()[0]
    if batched:
        b = lbm.Batch()
        b.set_solo_threshold(0)
        b.add(m)
        b.step(steps)
        b.remove(m)
        b.close()
    else:
        m.step(steps)
    change = m.conserved_sums()[0] / before - 1.0
    m.close()
    # and some 40 roundings of 2^-24 per cell and step, independent of each other
    assert abs(change) <= steps * _coefficient_drift(spec, s_high, s_orders) + 40 * 2.0 ** -24 * np.sqrt(steps / cells)


# A uniform stream in FP32: on its own a rounding of the momentum to FP32 in a step, of a product with 1 / 0.6 that
# lies a third of a unit in the last place apart for neighbouring momenta, moves it by a third of 2^-24 at most.
@pytest.mark.parametrize("speed", [0.0387, 0.021])
@pytest.mark.parametrize("name,n", [("rD3Q45", (24, 20, 16)), ("rD3Q53-cubic", (24, 20, 16)), ("rD3Q45", (48, 44, 40))])
def test_uniform_stream_keeps_its_momentum(name, n, speed):
    spec, steps = W.LATTICES[name], 200
    rng = np.random.default_rng(18)
    rho = 1.0 + 1e-3 * rng.uniform(-1, 1, size=tuple(reversed(n)))
    u = 1e-3 * rng.uniform(-1, 1, size=(3,) + tuple(reversed(n)))
    u[0] += speed
    m = gpu_model(spec, "nse", n, W.rates_nse(3, 0.05, spec.cs2[0], spec=spec), store="f32")
    m.init_fields(rho, u)
    before = m.conserved_sums()[1]
    m.step(steps)
    change = m.conserved_sums()[1] / before - 1.0
    m.close()
    assert abs(change) <= steps * 2.0 ** -24 / 3


# The launches of a batch of a 64 x 48 and a 128 x 128 solve, 20 steps: one a step for both in one group, one a step for
# each with the larger one alone, and with both alone a single one for the smaller, whose steps run in one launch.
@pytest.mark.parametrize("threshold,launches", [(0, 20), (4000, 40), (3000, 21)])
def test_batch_counts_the_launches_it_issued(threshold, launches):
    from paper_2512_16230_gb300 import lbm
    spec = W.LATTICES["rD2Q17"]
    lat = lbm.Lattice(spec.kind, spec.c, spec.cs2, spec.free_w)
    models = [gpu_model(spec, "nse", n, W.rates_nse(2, 0.05, spec.cs2[0], spec=spec), lat=lat) for n in ((64, 48), (128, 128))]
    b = lbm.Batch()
    b.set_solo_threshold(threshold)
    for m in models:
        m.set_populations(_populations(m, m.n, 19, 1.0))
        b.add(m)
    b.step(20)
    counted = b.counters()["launches"]
    b.close()
    for m in models:
        m.close()
    assert counted == launches
