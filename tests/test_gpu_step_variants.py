"""The variants of the collide-stream step that a call is given by its grid, storage and rates: each one
gives bitwise the populations of the one-cell-per-thread kernels, at the sizes where its tiling ends."""
import numpy as np
import pytest

from paper_2512_16230_gb300 import workloads as W

from _harness import gpu_model, oracle_lattice

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _lib(lbm_lib):
    return lbm_lib


def _populations(spec, n, seed, eq):
    w = oracle_lattice(spec).w
    r = np.random.default_rng(seed).uniform(-0.1, 0.1, size=(len(w),) + tuple(reversed(n)))
    return w.reshape((-1,) + (1,) * len(n)) * (1.0 if eq == "nse" else 0.7) * (1.0 + r)


def _kwargs(eq, d, s_high):
    if eq == "nse":
        return dict(s_high=s_high, cs2_eq=0.55, force=(0, d - 1, 3e-3, 1, 0.4))
    return dict(s_high=s_high, cs2_eq=0.55, u_const=tuple(np.linspace(0.03, 0.06, d)), nonlin=1.0)


def _rates(spec):
    return np.random.default_rng(3).uniform(0.6, 1.9, spec.R)


# row-staged kernel: tiles of several rows that wrap in y and z within the tile, a last tile with fewer
# rows, one row of 8 cells per thread group
@pytest.mark.parametrize("s_high", [1.0, 1.3])
@pytest.mark.parametrize("eq", ["nse", "ncde"])
@pytest.mark.parametrize("name,n", [("rD2Q17", (8, 5000)), ("rD3Q33", (24, 47, 53)), ("rD3Q53", (40, 31, 37))])
def test_row_tiles_of_several_rows(name, n, eq, s_high):
    spec = W.LATTICES[name]
    f0 = _populations(spec, n, 5, eq)
    out = {}
    for mode in ("rows", "threads"):
        gm = gpu_model(spec, eq, n, _rates(spec), store="f16_dev", **_kwargs(eq, spec.d, s_high))
        gm.set_gather(mode)
        gm.set_populations(f0)
        gm.step(3)
        out[mode] = gm.get_populations()
        gm.close()
    assert np.array_equal(out["rows"], out["threads"])


def test_row_tiles_with_per_cell_rates_and_cross_diffusion():
    spec, n = W.LATTICES["rD2Q25"], (8, 5000)
    f0 = _populations(spec, n, 6, "ncde")
    psi = np.random.default_rng(7).uniform(-1, 1, size=(n[1], n[0]))
    out = {}
    for mode in ("rows", "threads"):
        gm = gpu_model(spec, "ncde", n, _rates(spec), store="bf16_dev", ncde_mode="rate", a1=-0.2, a2=0.02, psi=psi,
                       **_kwargs("ncde", 2, 1.0))
        gm.set_gather(mode)
        gm.set_populations(f0)
        gm.step(3)
        out[mode] = gm.get_populations()
        gm.close()
    assert np.array_equal(out["rows"], out["threads"])


def test_population_io_keeps_every_value():
    """set_populations followed by get_populations returns FP32 values unchanged, also those for which the
    widening takes the conversion instruction: zeros of both signs, subnormals, infinities and NaN."""
    spec = W.LATTICES["rD2Q9"]
    n = (37, 5)
    v = np.array([0.0, -0.0, 1e-45, -1e-40, 1.1754944e-38, 3.4028235e38, -1.0, 1.0 + 2.0 ** -23, np.inf, -np.inf, np.nan,
                  0.1], dtype=np.float32)
    f0 = np.resize(v, 9 * n[0] * n[1]).reshape(9, n[1], n[0]).astype(np.float64)
    gm = gpu_model(spec, "nse", n, np.ones(spec.R), store="f32")
    gm.set_populations(f0)
    g = gm.get_populations()
    gm.close()
    assert np.array_equal(g, f0, equal_nan=True)
    assert np.array_equal(np.signbit(g[f0 == 0]), np.signbit(f0[f0 == 0]))


def _batched(spec, eq, n, f0, steps, prepare=lambda m: None, **kw):
    """The same solve in the work-list kernel of a batch, which takes one cell per thread."""
    from paper_2512_16230_gb300 import lbm
    m = gpu_model(spec, eq, n, _rates(spec), **kw)
    prepare(m)
    m.set_populations(f0)
    b = lbm.Batch()
    b.set_solo_threshold(0)
    b.add(m)
    b.step(steps)
    out = m.get_populations()
    b.remove(m)
    b.close()
    m.close()
    return out


# just above the size from which two cells go to a thread: n_x even, n_x odd with an odd and an even cell count
PAIR_GRIDS = {2: [(322, 250), (287, 283), (283, 286)], 3: [(46, 43, 41), (45, 43, 43)]}


@pytest.mark.parametrize("store", ["f32", "bf16_dev"])
@pytest.mark.parametrize("s_high", [1.0, 1.3])
@pytest.mark.parametrize("eq", ["nse", "ncde"])
@pytest.mark.parametrize("name", ["rD2Q13", "rD2Q25", "rD3Q33", "rD3Q53"])
def test_two_cells_per_thread(name, eq, s_high, store):
    spec = W.LATTICES[name]
    for n in PAIR_GRIDS[spec.d]:
        f0 = _populations(spec, n, 8, eq)
        kw = dict(store=store, **_kwargs(eq, spec.d, s_high))
        m = gpu_model(spec, eq, n, _rates(spec), **kw)
        m.set_populations(f0)
        m.step(3)
        one = m.get_populations()
        m.close()
        assert np.array_equal(one, _batched(spec, eq, n, f0, 3, **kw)), n


def test_two_cells_per_thread_with_gradient_terms():
    """The density history of M2G on rD3Q27 and the cross diffusion of the NCDE, both read at neighbours."""
    for name, eq, n, extra in (("rD3Q27", "nse", (45, 43, 43), lambda m: m.set_m2g_anisotropy(1)),
                               ("rD3Q27", "nse", (46, 43, 41), lambda m: m.set_m2g_anisotropy(1)),
                               ("rD2Q21", "ncde", (287, 283), None), ("rD2Q21", "ncde", (322, 250), None)):
        spec = W.LATTICES[name]
        f0 = _populations(spec, n, 9, eq)
        kw = dict(store="f32", **_kwargs(eq, spec.d, 1.0))
        if extra is None:
            kw.update(ncde_mode="rate", a1=-0.2, a2=0.02,
                      psi=np.random.default_rng(7).uniform(-1, 1, size=tuple(reversed(n))))
        prepare = extra or (lambda m: None)
        m = gpu_model(spec, eq, n, _rates(spec), **kw)
        prepare(m)
        m.set_populations(f0)
        m.step(4)
        one = m.get_populations()
        m.close()
        assert np.array_equal(one, _batched(spec, eq, n, f0, 4, prepare, **kw)), (name, n)


# small 2D grids: a call of several steps runs in one launch on a cluster, calls of one step do not. Rows that
# do not divide by the CTAs, fewer rows than CTAs, the largest grid taken and the first one that is not
@pytest.mark.parametrize("store", ["f32", "f16_dev"])
@pytest.mark.parametrize("s_high", [1.0, 1.3])
@pytest.mark.parametrize("eq", ["nse", "ncde"])
@pytest.mark.parametrize("name,grids", [("rD2Q13", [(37, 29), (5, 3), (630, 16), (631, 16)]), ("rD2Q25", [(64, 48), (7, 6), (20, 256)])])
def test_steps_of_a_small_grid_in_one_launch(name, grids, eq, s_high, store):
    spec = W.LATTICES[name]
    for n in grids:
        f0 = _populations(spec, n, 10, eq)
        out = []
        for calls in ([1] * 7, [5, 2]):
            m = gpu_model(spec, eq, n, _rates(spec), store=store, **_kwargs(eq, 2, s_high))
            m.set_populations(f0)
            for k in calls:
                m.step(k)
            assert m.counters()[0] == 7
            out.append(m.get_populations())
            m.close()
        assert np.array_equal(out[0], out[1]), n


def test_steps_in_one_launch_with_per_cell_rates_and_cross_diffusion():
    spec, n = W.LATTICES["rD2Q17"], (41, 23)
    f0 = _populations(spec, n, 11, "ncde")
    psi = np.random.default_rng(7).uniform(-1, 1, size=(n[1], n[0]))
    out = []
    for calls in ([1] * 6, [6]):
        m = gpu_model(spec, "ncde", n, _rates(spec), store="f32", ncde_mode="rate", a1=-0.2, a2=0.02, psi=psi,
                      **_kwargs("ncde", 2, 1.0))
        m.set_populations(f0)
        for k in calls:
            m.step(k)
        out.append(m.get_populations())
        m.close()
    assert np.array_equal(out[0], out[1])


@pytest.mark.parametrize("s_high", [1.0, 1.3])
@pytest.mark.parametrize("eq", ["nse", "ncde"])
@pytest.mark.parametrize("name", ["rD2Q9", "rD2Q13", "rD2Q25"])
def test_fp64_small_grid_is_the_large_one_periodically(name, eq, s_high):
    """A small FP64 grid takes four threads per cell, a large one one thread: repeated periodically along x, the
    small solve is bitwise the large one (48 x 33 against 12 copies of it)."""
    spec, n, copies = W.LATTICES[name], (48, 33), 12
    f0 = _populations(spec, n, 12, eq)
    out = []
    for k in (1, copies):
        m = gpu_model(spec, eq, (n[0] * k, n[1]), _rates(spec), store="f64", **_kwargs(eq, 2, s_high))
        m.set_populations(np.tile(f0, (1, 1, k)))
        m.step(3)
        out.append(m.get_populations())
        m.close()
    assert np.array_equal(np.tile(out[0], (1, 1, copies)), out[1])


# one rate per order >= 4: two cells per thread against one (the batch), and FP64, whose blocks are the same
@pytest.mark.parametrize("store", ["f32", "f16_dev"])
@pytest.mark.parametrize("name,n", [("rD2Q25", (322, 250)), ("rD2Q17", (287, 283)), ("rD3Q27", (46, 43, 41)),
                                    ("rD3Q33", (45, 43, 43)), ("rD3Q53", (46, 43, 41)), ("rD3Q45", (45, 43, 43)),
                                    ("rD3Q53", (45, 43, 43))])
def test_order_rates_two_cells_per_thread(name, n, store):
    spec = W.LATTICES[name]
    f0 = _populations(spec, n, 13, "nse")
    kw = dict(store=store, s_orders={4: 0.8, 5: 1.35, 6: 1.6, 7: 0.9, 8: 1.25}, **_kwargs("nse", spec.d, 1.2))
    m = gpu_model(spec, "nse", n, _rates(spec), **kw)
    m.set_populations(f0)
    m.step(2)
    one = m.get_populations()
    m.close()
    assert np.array_equal(one, _batched(spec, "nse", n, f0, 2, **kw))
    if store == "f32":
        m = gpu_model(spec, "nse", n, _rates(spec), **dict(kw, store="f64"))
        m.set_populations(f0)
        m.step(2)
        ref = m.get_populations()
        m.close()
        # two roundings of the populations to FP32 and some 40 in sums of the collision, each 2^-24 of the largest
        assert np.abs(one - ref).max() <= 2 * 42 * 2.0 ** -24 * np.abs(ref).max()


# wide, many rows: the row-staged tcgen05 kernel is the default; one row fewer than it asks for: the CUDA cores
@pytest.mark.parametrize("fewer", [0, 1])
def test_order_rates_default_on_wide_rows(fewer):
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    spec, n = W.LATTICES["rD3Q53"], (240, sms - fewer, 64)
    rho, u = np.ones(tuple(reversed(n))), np.random.default_rng(14).uniform(-0.02, 0.02, size=(3,) + tuple(reversed(n)))
    out = []
    for mode in (None, 1 - fewer, fewer):
        m = gpu_model(spec, "nse", n, _rates(spec), store="f16_dev", s_high=1.2, s_orders={4: 0.8, 5: 1.35, 8: 1.25})
        if mode is not None:
            m.set_tensor_cores(mode)
        m.init_fields(rho, u)
        m.step(2)
        out.append(m.read_fields()[1])
        m.close()
    assert np.array_equal(out[0], out[1]) and not np.array_equal(out[0], out[2])


# 16-bit storage by default: two cells per thread from 80,000 cells, one below; the row-staged kernel's populations
@pytest.mark.parametrize("s_high", [1.0, 1.3])
@pytest.mark.parametrize("name,n", [("rD3Q53", (48, 42, 40)), ("rD3Q53", (48, 41, 40)), ("rD3Q45", (48, 42, 40))])
def test_default_of_16_bit_storage(name, n, s_high):
    spec = W.LATTICES[name]
    f0 = _populations(spec, n, 15, "nse")
    out = []
    for mode in ("auto", "rows"):
        gm = gpu_model(spec, "nse", n, _rates(spec), store="bf16_dev", **_kwargs("nse", 3, s_high))
        gm.set_gather(mode)
        gm.set_populations(f0)
        gm.step(3)
        out.append(gm.get_populations())
        gm.close()
    assert np.array_equal(out[0], out[1])


# The same for calls long enough to run in one launch, with the launches counted: the widest rows taken (512 cells, 8192
# populations a CTA) and the first ones not taken, and the shortest call of 64 x 48 and of 20 x 256 that is.
@pytest.mark.parametrize("store", ["f32", "f16_dev"])
@pytest.mark.parametrize("s_high", [1.0, 1.3])
@pytest.mark.parametrize("eq", ["nse", "ncde"])
@pytest.mark.parametrize("name,n,calls,launches", [
    ("rD2Q13", (37, 29), (20, 21), 2), ("rD2Q13", (5, 3), (20, 21), 2), ("rD2Q13", (512, 16), (20, 21), 2),
    ("rD2Q13", (513, 16), (20, 21), 41), ("rD2Q25", (327, 16), (20, 21), 2), ("rD2Q25", (328, 16), (20, 21), 41),
    ("rD2Q25", (7, 6), (20, 21), 2), ("rD2Q25", (64, 48), (12, 13), 13), ("rD2Q25", (20, 256), (18, 19), 19)])
def test_long_calls_on_a_small_grid_in_one_launch(name, n, calls, launches, eq, s_high, store):
    spec = W.LATTICES[name]
    f0 = _populations(spec, n, 10, eq)
    out = []
    for split in ([1] * sum(calls), calls):
        m = gpu_model(spec, eq, n, np.random.default_rng(3).uniform(0.9, 1.5, spec.R), store=store, **_kwargs(eq, 2, s_high))
        m.set_populations(f0)
        before = m.counters()[1]
        for k in split:
            m.step(k)
        assert m.counters()[1] - before == (sum(calls) if split is not calls else launches)
        out.append(m.get_populations())
        m.close()
    assert np.array_equal(out[0], out[1])


@pytest.mark.parametrize("store", ["f32", "bf16_dev"])
def test_long_call_in_one_launch_with_per_cell_rates_and_cross_diffusion(store):
    spec, n, steps = W.LATTICES["rD2Q17"], (41, 23), 21
    f0 = _populations(spec, n, 11, "ncde")
    psi = np.random.default_rng(7).uniform(-1, 1, size=(n[1], n[0]))
    out = []
    for calls in ([1] * steps, [steps]):
        m = gpu_model(spec, "ncde", n, _rates(spec), store=store, ncde_mode="rate", a1=-0.2, a2=0.02, psi=psi,
                      **_kwargs("ncde", 2, 1.0))
        m.set_populations(f0)
        before = m.counters()[1]
        for k in calls:
            m.step(k)
        assert m.counters()[1] - before == len(calls)
        out.append(m.get_populations())
        m.close()
    assert np.array_equal(out[0], out[1])
