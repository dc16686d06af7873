"""The memory of the block sums (sbim_set_time_blocks): a handle is created without it, takes it at
its first step only where it leaves room, returns it on request, and steps to the same tractions
with it and without it."""
import numpy as np
import pytest

from paper_2102_08756_gb300.synth import separable_history
from tests._errors import Worst, rel_l2

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CS, CP, RHO = 3464.0, 6000.0, 2670.0
DT = 0.3 * 100.0 / CP
TOL = {"fp32": 1e-5, "bf16x2": 1e-4, "bf16": 1e-2}
MB, SPARE = 1 << 20, 256 << 20


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()


def _make(n, n_cut, precision="fp32", stream=None):
    from paper_2102_08756_gb300.sbim import SBIM
    return SBIM(n, n, 100.0 * n, 100.0 * n, CS, CP, RHO, DT, n_cut, 1, precision, precision != "bf16",
                stream=stream)


def _free():
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    return torch.cuda.mem_get_info()[0]


def _step(h, n):
    z = torch.zeros((3, n, n), device="cuda")
    return h.step(z, z)


def test_sums_are_taken_at_the_first_step_and_given_back():
    n, n_cut = 256, 1024
    h = _make(n, 16)          # what a first handle brings in with it
    _step(h, n)
    h.close()
    before = _free()
    h = _make(n, n_cut)
    ring = h.info()["hist_bytes"]
    created = before - _free()
    records = h.info()["n_slots"] // 4
    # the ring, at most n_cut / 16 lag chunks of partial sums, tables, spectra and FFT plans
    assert ring <= created < ring + 160 * records * n_cut // 16 + 32 * MB
    _step(h, n)
    assert h.time_blocks()
    extra = before - _free() - created
    assert 16 * records * n_cut <= extra < 32 * records * n_cut + 64 * MB
    h.set_time_blocks(False)
    assert not h.time_blocks() and abs(before - _free() - created) <= 4 * MB
    _step(h, n)
    h.set_time_blocks(True)
    assert h.time_blocks()
    h.check()


def test_handles_that_fit_without_block_sums_are_all_created():
    """Room for three handles and half the extra memory of one: each is created and stepped in
    turn, and none takes the memory that the next one needs."""
    n, n_cut = 512, 512
    h = _make(n, n_cut)
    _step(h, n)
    h.set_time_blocks(False)
    records, ring = h.info()["n_slots"] // 4, h.info()["hist_bytes"]
    h.close()
    free = _free()
    h = _make(n, n_cut)
    need = free - _free()
    h.close()
    fill = torch.empty(_free() - (3 * need + SPARE + 8 * records * n_cut) - 64 * MB, dtype=torch.uint8,
                       device="cuda")
    hs = []
    for _ in range(3):
        hs.append(_make(n, n_cut))
    for x in hs:
        _step(x, n)
        x.check()
    for x in hs:
        x.close()
    # created and stepped in turn: the first leaves the second its room
    del fill
    fill = torch.empty(_free() - (2 * need + SPARE + 8 * records * n_cut) - 64 * MB, dtype=torch.uint8,
                       device="cuda")
    a = _make(n, n_cut)
    _step(a, n)
    assert not a.time_blocks()
    b = _make(n, n_cut)
    _step(b, n)
    a.check()
    b.check()
    assert ring < need
    a.close()
    b.close()
    # and with the room back, the next decision takes them
    del fill
    _free()
    c = _make(n, n_cut)
    _step(c, n)
    assert c.time_blocks()
    c.close()


@pytest.mark.parametrize("precision", ["fp32", "bf16x2", "bf16"])
def test_forms_in_turn(precision):
    """Block sums on, off and on again in the middle of blocks, with repeats and rewinds."""
    n, n_cut = 48, 40
    h, ref = _make(n, n_cut, precision), _make(n, n_cut, "fp64")
    hist = separable_history(n, n, n * 100.0, n * 100.0, 120, DT, CS, seed=4, spectrum="k2")
    err = Worst()
    for m in range(120):
        u, v = [torch.from_numpy(x(m).astype(np.float32)).cuda() for x in (hist.u, hist.v)]
        if m % 23 == 11:
            h.set_time_blocks(m % 2)
        if m % 31 == 20 and m > 0:
            h.rewind()
            ref.rewind()
        r = ref.step(u.double(), v.double()).cpu().numpy()
        err.update(rel_l2(h.step(u, v).double().cpu().numpy(), r))
        if m % 5 == 2:
            err.update(rel_l2(h.step_repeat(u, v).double().cpu().numpy(), r))
    assert err.value < TOL[precision], err


def test_first_steps_under_capture():
    """A handle first stepped under stream capture allocates nothing there; the graph, a repeat in
    it, and direct steps with block sums then alternate on one history."""
    n, n_cut = 48, 24
    stream = torch.cuda.Stream()
    hist = separable_history(n, n, n * 100.0, n * 100.0, 90, DT, CS, seed=9, spectrum="k2")
    err = Worst()
    with torch.cuda.stream(stream):
        h, ref = _make(n, n_cut, stream=stream), _make(n, n_cut, "fp64", stream=stream)
        u, v, tau = [torch.zeros((3, n, n), device="cuda") for _ in range(3)]
        stream.synchronize()
        g = torch.cuda.CUDAGraph()
        g.capture_begin()
        h.step(u, v, tau)
        h.step_repeat(u, v, tau)
        g.capture_end()
        for m in range(90):
            u.copy_(torch.from_numpy(hist.u(m).astype(np.float32)))
            v.copy_(torch.from_numpy(hist.v(m).astype(np.float32)))
            if m % 7 < 4:
                g.replay()
            else:
                h.step(u, v, tau)
                assert h.time_blocks()
            r = ref.step(u.double(), v.double()).cpu().numpy()
            stream.synchronize()
            err.update(rel_l2(tau.double().cpu().numpy(), r))
    assert err.value < TOL["fp32"], err


def test_a_restored_run_goes_on_in_its_form():
    n, n_cut = 48, 40
    f = [(1e-3 * torch.randn((3, n, n), device="cuda"), torch.randn((3, n, n), device="cuda")) for _ in range(70)]

    def run(h, a, b):
        return [h.step(u, v) for u, v in f[a:b]]

    def same(x, y):
        return all(torch.equal(p, q) for p, q in zip(x, y))

    by_step, by_block = _make(n, n_cut), _make(n, n_cut)
    by_step.set_time_blocks(False)
    run(by_step, 0, 37)
    run(by_block, 0, 37)
    saved = by_step.save(), by_block.save()
    after = run(by_step, 37, 70), run(by_block, 37, 70)
    assert not same(*after)                       # the forms round differently
    h = _make(n, n_cut)
    for k in (0, 1, 0, 1):
        h.load(saved[k])
        assert same(run(h, 37, 70), after[k]) and h.time_blocks() == bool(k)
    # told to do without block sums, a handle does, and differs by rounding only
    h.set_time_blocks(False)
    h.load(saved[1])
    got = run(h, 37, 70)
    assert not h.time_blocks()
    err = Worst()
    for p, q in zip(got, after[1]):
        err.update(rel_l2(p.double().cpu().numpy(), q.double().cpu().numpy()))
    assert err.value < TOL["fp32"], err
