"""The step-by-step convolution of float-class handles (what they run without room for block sums):
every pipeline shape, record tile and lag chunking, single and batched, against the FP64 handle, which
the parity tests compare with the oracle."""
import numpy as np
import pytest

from paper_2102_08756_gb300.synth import separable_history
from tests._errors import Worst, rel_l2

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CS, CP, RHO = 3464.0, 6000.0, 2670.0
DT = 0.3 * 100.0 / CP
TOL = {"fp32": 1e-5, "bf16x2": 1e-4, "bf16": 1e-2}


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()


def _make(n1, n3, n_cut, precision, kahan, side=1, stream=None):
    from paper_2102_08756_gb300.sbim import SBIM
    return SBIM(n1, n3, 100.0 * n1, 100.0 * n3, CS, CP, RHO, DT, n_cut, side, precision, kahan, stream=stream)


def _fields(n1, n3, steps, seed):
    h = separable_history(n1, n3, n1 * 100.0, n3 * 100.0, steps, DT, CS, seed=seed, spectrum="k2")
    return [(torch.from_numpy(h.u(m).astype(np.float32)).cuda(),
             torch.from_numpy(h.v(m).astype(np.float32)).cuda()) for m in range(steps)]


# whole records (256) and half records (512), both multiples of every tile
@pytest.mark.parametrize("grid,window", [((32, 32), 0.0), ((32, 32), 7.3), ((64, 48), 0.0)])
@pytest.mark.parametrize("variant,tile,lags", [(0, 128, 0), (1, 64, 0), (1, 128, 5), (1, 256, 0), (2, 64, 16),
                                               (2, 128, 0), (2, 256, 7), (3, 64, 0), (3, 128, 16),
                                               (3, 256, 0)])
@pytest.mark.parametrize("precision,kahan", [("fp32", 1), ("fp32", 0), ("bf16x2", 1), ("bf16", 0),
                                             ("bf16", 1)])
def test_launch_shapes(precision, kahan, variant, tile, lags, grid, window):
    n1, n3 = grid
    n_cut = 29
    g = _make(n1, n3, n_cut, precision, kahan, side=-1)
    ref = _make(n1, n3, n_cut, "fp64", 0, side=-1)
    g.set_time_blocks(False)
    g.set_conv_tile(tile)
    g.set_conv_config(variant, lags)
    for h in (g, ref):
        h.set_window(window)
    err = Worst()
    for m, (u, v) in enumerate(_fields(n1, n3, n_cut + 16, seed=variant + tile)):
        r = ref.step(u.double(), v.double()).cpu().numpy()
        err.update(rel_l2(g.step(u, v).double().cpu().numpy(), r))
        if m % 6 == 4:
            err.update(rel_l2(g.step_repeat(u, v).double().cpu().numpy(), r))
        if m % 6 == 5:
            t = g.step_host(u.cpu().numpy(), v.cpu().numpy())
            r = ref.step(u.double(), v.double()).cpu().numpy()
            err.update(rel_l2(t.astype(np.float64), r))
    assert not g.time_blocks()
    g.check()
    assert err.value < TOL[precision], err


@pytest.mark.parametrize("shape,lags,tile", [(1, 16, 128), (2, 64, 128), (3, 16, 64), (4, 64, 64),
                                             (5, 16, 128), (6, 1024, 128)])
@pytest.mark.parametrize("precision,kahan,members", [
    ("fp32", 1, "mixed"), ("bf16x2", 1, "mixed"), ("bf16", 0, "whole"), ("bf16", 0, "half")])
def test_batches(precision, kahan, members, shape, lags, tile):
    """Persistent CTAs (1-3) and one CTA per work item (4-6) over whole- and half-record members:
    bit-equal to the members stepped alone, and within the bound of the FP64 handle.  (Uncompensated
    sums of the whole- and the half-record kernels round differently, and a batch that holds both runs
    the latter: such members come in batches of their own.)"""
    from paper_2102_08756_gb300 import sbim as B
    whole, half = [(32, 32, 21), (48, 48, 40)], [(192, 32, 40), (24, 24, 3), (64, 6, 33)]
    members = {"mixed": whole + half, "whole": whole, "half": half}[members]
    n1, n3, cut = [list(x) for x in zip(*members)]
    k = len(members)
    stream = torch.cuda.Stream()
    err = Worst()
    with torch.cuda.stream(stream):
        b = B.sbim_batch_create(n1, n3, [100.0 * x for x in n1], [100.0 * x for x in n3], [CS] * k, [CP] * k,
                                [RHO] * k, [DT] * k, cut, [1] * k, B.PRECISION[precision], kahan,
                                stream.cuda_stream)
        B.sbim_set_time_blocks(B.sbim_batch_member(b, 1), False)   # one is enough
        B.sbim_batch_set_conv_config(b, shape, lags)
        B.sbim_batch_set_conv_tile(b, tile)
        assert not any(B.sbim_get_time_blocks(B.sbim_batch_member(b, i)) for i in range(k))
        alone = []
        for a, c, n in members:
            h = _make(a, c, n, precision, kahan, stream=stream)
            h.set_time_blocks(False)
            h.set_conv_tile(tile)
            h.set_conv_config((shape - 1) % 3 + 1, lags)
            alone.append(h)
        ref = [_make(a, c, n, "fp64", 0, stream=stream) for a, c, n in members]
        f = [_fields(a, c, 50, seed=i) for i, (a, c, _) in enumerate(members)]
        for m in range(50):
            tau = [torch.empty_like(x[m][0]) for x in f]
            B.sbim_batch_step(b, [x[m][0].data_ptr() for x in f], [x[m][1].data_ptr() for x in f],
                              [t.data_ptr() for t in tau])
            for i in range(k):
                u, v = f[i][m]
                assert torch.equal(tau[i], alone[i].step(u, v)), (m, i)
                r = ref[i].step(u.double(), v.double())
                stream.synchronize()
                err.update(rel_l2(tau[i].double().cpu().numpy(), r.cpu().numpy()))
        for i in range(k):
            B.sbim_check_device(B.sbim_batch_member(b, i))
        B.sbim_batch_destroy(b)
    assert err.value < TOL[precision], err


# the assembly by record (few chunks for the records) and by member (the same plane in more chunks),
# whole and half records; FP64 against itself
@pytest.mark.parametrize("precision,grid", [("fp32", (256, 256)), ("bf16x2", (256, 256)), ("bf16", (256, 256)),
                                            ("fp32", (384, 160)), ("fp64", (512, 512)), ("fp64", (1024, 250))])
@pytest.mark.parametrize("kahan", [0, 1])
def test_assembly_by_record_and_by_member(precision, grid, kahan):
    n1, n3 = grid
    n_cut = 14
    ref = _make(n1, n3, n_cut, "fp64", 0)
    ref.set_conv_config(1, 4)
    hs = []
    for lags in (0, 4):
        h = _make(n1, n3, n_cut, precision, kahan)
        h.set_time_blocks(False)
        h.set_conv_config(2, lags)
        hs.append(h)
    tol = TOL.get(precision, 1e-12)
    err = Worst()
    for u, v in _fields(n1, n3, 19, seed=5):
        r = ref.step(u.double(), v.double()).cpu().numpy()
        x = (u.double(), v.double()) if precision == "fp64" else (u, v)
        for h in hs:
            err.update(rel_l2(h.step(*x).double().cpu().numpy(), r))
    assert err.value < tol, err


def test_batched_assembly_by_record():
    from paper_2102_08756_gb300 import sbim as B
    n, n_cut = 256, 12
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        b = B.sbim_batch_create([n, 32], [n, 32], [100.0 * n, 3200.0], [100.0 * n, 3200.0], [CS] * 2, [CP] * 2,
                                [RHO] * 2, [DT] * 2, [n_cut, 7], [1, -1], 1, 1, stream.cuda_stream)
        B.sbim_set_time_blocks(B.sbim_batch_member(b, 0), False)
        B.sbim_batch_set_conv_config(b, 5, 1024)
        alone = [_make(n, n, n_cut, "fp32", 1, stream=stream), _make(32, 32, 7, "fp32", 1, side=-1, stream=stream)]
        for h in alone:
            h.set_time_blocks(False)
            h.set_conv_config(2, 1024)
        f = [_fields(n, n, 20, seed=1), _fields(32, 32, 20, seed=2)]
        for m in range(20):
            tau = [torch.empty_like(x[m][0]) for x in f]
            B.sbim_batch_step(b, [x[m][0].data_ptr() for x in f], [x[m][1].data_ptr() for x in f],
                              [t.data_ptr() for t in tau])
            for i in range(2):
                assert torch.equal(tau[i], alone[i].step(*f[i][m])), (m, i)
        B.sbim_batch_destroy(b)
