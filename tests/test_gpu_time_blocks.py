"""The time-blocked convolution (block sums over 16 steps, staggered over the
record tiles) against the FP64 handle, which convolves step by step: cutoffs
around the block length, chunk edges, both record layouts, every float-class
history; the state changes that make the block sums obsolete; and non-finite
values, which must enter and leave the tractions at the same steps."""
import numpy as np
import pytest

from paper_2102_08756_gb300.synth import separable_history
from tests._errors import Worst, rel_l2

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CS, CP, RHO = 3464.0, 6000.0, 2670.0
# the bounds of the parity tests: float storage and transforms, bf16 storage
TOL = {"fp32": 1e-5, "bf16x2": 1e-4, "bf16": 1e-2}


@pytest.fixture(scope="module", autouse=True)
def built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()


def _pair(n1, n3, n_cut, precision, side=1):
    from paper_2102_08756_gb300.sbim import SBIM
    dx = 100.0
    dt = 0.3 * dx / CP
    make = lambda p, k: SBIM(n1, n3, n1 * dx, n3 * dx, CS, CP, RHO, dt, n_cut, side, p, k)  # noqa: E731
    return make(precision, precision != "bf16"), make("fp64", False), dt


def _fields(n1, n3, dt, steps, seed):
    h = separable_history(n1, n3, n1 * 100.0, n3 * 100.0, steps, dt, CS, seed=seed, spectrum="k2")
    return [(torch.from_numpy(h.u(m).astype(np.float32)).cuda(),
             torch.from_numpy(h.v(m).astype(np.float32)).cuda()) for m in range(steps)]


# whole records; half records; 18 tiles, so a full group of 16 and a ragged one
@pytest.mark.parametrize("precision", ["fp32", "bf16x2", "bf16"])
@pytest.mark.parametrize("grid", [(32, 32), (64, 6), (176, 96)])
@pytest.mark.parametrize("n_cut,lags", [(1, 0), (2, 0), (15, 0), (16, 0), (17, 0), (31, 16), (33, 16),
                                        (50, 20), (70, 0)])
def test_block_sums_match_step_by_step(precision, grid, n_cut, lags):
    n1, n3 = grid
    g, ref, dt = _pair(n1, n3, n_cut, precision, side=-1)
    if lags:
        g.set_conv_config(2, lags)
    err = Worst()
    for u, v in _fields(n1, n3, dt, 90, seed=n1 + n_cut):
        t = g.step(u, v).double().cpu().numpy()
        r = ref.step(u.double(), v.double()).cpu().numpy()
        err.update(rel_l2(t, r))
    g.check()
    assert err.value < TOL[precision], err


@pytest.mark.parametrize("precision", ["fp32", "bf16"])
def test_changes_of_state_between_blocks(precision):
    """Reset, a new window, another chunking, several rewinds and a checkpoint of
    another handle, each in the middle of a block."""
    n1, n3, n_cut = 48, 32, 40
    g, ref, dt = _pair(n1, n3, n_cut, precision)
    donor, donor64, _ = _pair(n1, n3, n_cut, precision)
    f = _fields(n1, n3, dt, 60, seed=5)
    fd = _fields(n1, n3, dt, 60, seed=6)
    for u, v in fd[:29]:
        donor.step(u, v)
        donor64.step(u.double(), v.double())
    err = Worst()

    def steps(a, b):
        for u, v in f[a:b]:
            r = ref.step(u.double(), v.double()).cpu().numpy()
            err.update(rel_l2(g.step(u, v).double().cpu().numpy(), r))

    steps(0, 21)
    for h in (g, ref):
        h.set_window(5.0)
    steps(21, 25)
    for h in (g, ref):
        h.set_window(0.0)
    steps(25, 27)
    g.set_conv_config(1, 16)
    steps(27, 40)
    for h in (g, ref):
        for _ in range(9):
            h.rewind()
    steps(40, 55)
    for h in (g, ref):
        h.reset()
    steps(3, 30)
    g.load(donor.save())
    ref.load(donor64.save())
    steps(29, 50)
    assert err.value < TOL[precision], err


def test_non_finite_values_leave_with_their_last_lag():
    n1, n3, n_cut = 24, 16, 21
    g, ref, dt = _pair(n1, n3, n_cut, "fp32")
    f = _fields(n1, n3, dt, 60, seed=8)
    seen = 0
    for m, (u, v) in enumerate(f):
        if m == 9:
            u = u.clone()
            u[1, 3, 5] = float("nan")
        t = torch.isfinite(g.step(u, v))
        r = torch.isfinite(ref.step(u.double(), v.double()))
        assert torch.equal(t, r), m
        seen += int(not bool(r.all()))
    assert seen == n_cut


def _batch(members, n_cut, dt, stream):
    from paper_2102_08756_gb300 import sbim as B
    k = len(members)
    n1, n3 = [list(x) for x in zip(*members)]
    b = B.sbim_batch_create(n1, n3, [100.0 * x for x in n1], [100.0 * x for x in n3], [CS] * k, [CP] * k,
                            [RHO] * k, [dt] * k, [n_cut] * k, [1] * k, 1, 1, stream.cuda_stream)
    return B, b


def _batch_step(B, b, f):
    tau = [torch.empty_like(u) for u, _ in f]
    B.sbim_batch_step(b, [u.data_ptr() for u, _ in f], [v.data_ptr() for _, v in f],
                      [t.data_ptr() for t in tau])
    return tau


# whole and half records in one batch, in both orders, and each alone
@pytest.mark.parametrize("members", [[(32, 32), (64, 6), (48, 48)], [(64, 6), (32, 32)], [(64, 6)], [(32, 32)]])
def test_batches_of_mixed_layouts(members):
    from paper_2102_08756_gb300.sbim import SBIM
    n_cut, dt = 40, 0.3 * 100.0 / CP
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        B, b = _batch(members, n_cut, dt, stream)
        alone = [SBIM(n1, n3, n1 * 100.0, n3 * 100.0, CS, CP, RHO, dt, n_cut, 1, "fp32", True,
                      stream=stream) for n1, n3 in members]
        for h in alone:
            h.set_conv_config(2, 1024)
        f = [_fields(n1, n3, dt, 60, seed=k) for k, (n1, n3) in enumerate(members)]
        for m in range(60):
            tau = _batch_step(B, b, [x[m] for x in f])
            for k, h in enumerate(alone):
                assert torch.equal(tau[k], h.step(*f[k][m])), (m, k)
        B.sbim_batch_destroy(b)


def test_batch_members_restored_in_the_middle_of_a_run():
    """Every tile's sums are formed again in one step: both record layouts, 18 tiles in one member,
    members restored from the checkpoints of handles that went on alone; then a new window."""
    from paper_2102_08756_gb300.sbim import SBIM
    members, n_cut, dt = [(176, 96), (64, 6)], 45, 0.3 * 100.0 / CP
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        B, b = _batch(members, n_cut, dt, stream)
        alone = [SBIM(n1, n3, n1 * 100.0, n3 * 100.0, CS, CP, RHO, dt, n_cut, 1, "fp32", True,
                      stream=stream) for n1, n3 in members]
        f = [_fields(n1, n3, dt, 75, seed=k) for k, (n1, n3) in enumerate(members)]
        for k, h in enumerate(alone):
            h.set_conv_config(2, 1024)
            for m in range(53):
                h.step(*f[k][m])
            B.sbim_load(B.sbim_batch_member(b, k), h.save())
        for m in range(53, 75):
            tau = _batch_step(B, b, [x[m] for x in f])
            for k, h in enumerate(alone):
                assert torch.equal(tau[k], h.step(*f[k][m])), (m, k)
        B.sbim_batch_destroy(b)


def test_settings_that_change_nothing_keep_the_sums():
    """The same window, another pipeline shape or tile: no sums are formed again, the bits are those of
    a handle left alone."""
    n1, n3, n_cut = 48, 32, 40
    g, same, dt = _pair(n1, n3, n_cut, "fp32")[0], _pair(n1, n3, n_cut, "fp32")[0], 0.3 * 100.0 / CP
    for m, (u, v) in enumerate(_fields(n1, n3, dt, 60, seed=3)):
        if m % 7 == 3:
            g.set_window(0.0)
            g.set_conv_config(1 + m % 3, 0)
            g.set_conv_tile(64 if m % 2 else 128)
        assert torch.equal(g.step(u, v), same.step(u, v)), m


def test_member_with_its_own_chunking_between_batch_steps():
    """A batch keeps its copy of a member's chunking; the member, given a coarser one and
    stepped by itself, and the batch then alternate on the same sums buffer."""
    n1, n3, n_cut = 48, 32, 70
    stream = torch.cuda.Stream()
    err = Worst()
    with torch.cuda.stream(stream):
        _, ref, dt = _pair(n1, n3, n_cut, "fp32", side=1)
        B, b = _batch([(n1, n3)], n_cut, dt, stream)
        B.sbim_batch_set_conv_config(b, 2, 16)
        member = B.sbim_batch_member(b, 0)
        f = _fields(n1, n3, dt, 100, seed=9)
        for m, (u, v) in enumerate(f):
            if m == 75:
                B.sbim_set_conv_config(member, 2, 64)
            if m >= 75 and m % 3:
                tau = torch.empty_like(u)
                B.sbim_step(member, u.data_ptr(), v.data_ptr(), tau.data_ptr())
            else:
                tau = _batch_step(B, b, [(u, v)])[0]
            stream.synchronize()
            r = ref.step(u.double(), v.double()).cpu().numpy()
            err.update(rel_l2(tau.double().cpu().numpy(), r))
        B.sbim_batch_destroy(b)
    assert err.value < TOL["fp32"], err


# few lags and many; large planes with short BF16 histories (whole records: 384^2 convolves step by step)
@pytest.mark.parametrize("precision,grid,n_cut", [("fp32", (48, 32), 40), ("fp32", (48, 32), 90),
                                                  ("bf16", (48, 32), 40), ("bf16x2", (48, 32), 130),
                                                  ("bf16", (384, 384), 20), ("bf16x2", (512, 256), 24)])
def test_host_direct_and_repeated_steps_in_turn(precision, grid, n_cut):
    """Host-buffer, direct and repeated steps of one handle against the FP64 handle."""
    from paper_2102_08756_gb300 import sbim as B
    n1, n3 = grid
    g, ref, dt = _pair(n1, n3, n_cut, precision)
    err = Worst()
    for m, (u, v) in enumerate(_fields(n1, n3, dt, n_cut + 20, seed=3)):
        r = ref.step(u.double(), v.double()).cpu().numpy()
        if m % 5 in (0, 1, 3):
            t = torch.from_numpy(g.step_host(u.cpu().numpy(), v.cpu().numpy()))
        else:
            t = g.step(u, v)
        err.update(rel_l2(t.double().cpu().numpy(), r))
        if m % 5 in (1, 4):
            out = torch.empty_like(u)
            B.sbim_step_repeat(g.h, u.data_ptr(), v.data_ptr(), out.data_ptr())
            err.update(rel_l2(out.double().cpu().numpy(), r))
    g.check()
    assert err.value < TOL[precision], err


@pytest.mark.parametrize("n,n_cut", [(64, 1000), (128, 600)])
def test_sums_are_as_exact_as_step_by_step(n, n_cut):
    """White fields, whose error is the convolution's more than the transforms': over 32 steps with
    the whole history the block sums are no further from FP64 than sums compensated term by term."""
    g, ref, dt = _pair(n, n, n_cut, "fp32")
    by_step, _, _ = _pair(n, n, n_cut, "fp32")
    by_step.set_conv_config(0, 0)
    gen = torch.Generator(device="cuda").manual_seed(17)
    U = 1e-3 * torch.randn((4, 3 * n * n), generator=gen, device="cuda", dtype=torch.float64)
    t = torch.arange(n_cut + 40, device="cuda", dtype=torch.float64)
    w = 0.25 * np.pi / 100.0 * CS * dt * (0.05 + 0.95 * torch.rand((4, 8, 1), generator=gen, device="cuda",
                                                                    dtype=torch.float64))
    sig = torch.sin(w * t + 6.28 * torch.rand((4, 8, 1), generator=gen, device="cuda",
                                              dtype=torch.float64)).sum(1)
    zero = torch.zeros((3, n, n), device="cuda")
    hs = (g, by_step, ref)
    for h in hs:
        h.set_window(1e-6)
    err = [0.0, 0.0]
    for m in range(n_cut + 40):
        if m == n_cut + 4:
            for h in hs:
                h.set_window(0.0)
        u = (sig[:, m] @ U).reshape(3, n, n).float()
        r = ref.step(u.double(), zero.double())
        tau = [h.step(u, zero).double() for h in hs[:2]]
        if m >= n_cut + 8:
            for k in range(2):
                assert bool(torch.isfinite(tau[k]).all())
                err[k] += float((tau[k] - r).square().sum())
    assert err[0] <= err[1], err


# rewinds to before a block whose predecessor has no history in some chunk: the first blocks
# of a run (levels 0 .. 15, staggered over 18 tiles) and, with 16-lag chunks, the second chunk
# of a block at 32; then other displacements
@pytest.mark.parametrize("steps,back,lags", [(17, 2, 0), (17, 9, 0), (17, 17, 0), (2, 2, 0), (33, 23, 16),
                                             (33, 30, 0), (20, 6, 16)])
@pytest.mark.parametrize("precision", ["fp32", "bf16"])
def test_rewinds_to_before_the_first_blocks(precision, steps, back, lags):
    n1, n3 = 176, 96
    g, ref, dt = _pair(n1, n3, 48, precision)
    if lags:
        g.set_conv_config(2, lags)
    f = _fields(n1, n3, dt, 60, seed=31)
    other = _fields(n1, n3, dt, 60, seed=32)
    for u, v in f[:steps]:
        g.step(u, v)
        ref.step(u.double(), v.double())
    for h in (g, ref):
        for _ in range(back):
            h.rewind()
    err = Worst()
    for u, v in other[steps - back:46]:
        r = ref.step(u.double(), v.double()).cpu().numpy()
        err.update(rel_l2(g.step(u, v).double().cpu().numpy(), r))
    assert err.value < TOL[precision], err


def test_member_with_a_finer_chunking_leaves_the_batch_its_buffers():
    """A member given a finer chunking by itself needs larger buffers; the batch, and a graph
    captured before, go on with the arguments they hold."""
    n1, n3, n_cut = 48, 32, 90
    stream = torch.cuda.Stream()
    err = Worst()
    with torch.cuda.stream(stream):
        _, ref, dt = _pair(n1, n3, n_cut, "fp32", side=1)
        B, b = _batch([(n1, n3)], n_cut, dt, stream)
        member = B.sbim_batch_member(b, 0)
        ub, vb, tb = [torch.zeros((3, n3, n1), device="cuda") for _ in range(3)]
        B.sbim_batch_capture(b, [ub.data_ptr()], [vb.data_ptr()], [tb.data_ptr()])
        keep = []
        for m, (u, v) in enumerate(_fields(n1, n3, dt, 120, seed=12)):
            if m in (40, 95):
                B.sbim_set_conv_config(member, 2, 32 if m == 40 else 16)
                keep.append(torch.full((1 << 22,), float("nan"), device="cuda"))
            ub.copy_(u)
            vb.copy_(v)
            if m % 4 == 3 and m >= 40:
                tau = torch.empty_like(u)
                B.sbim_step(member, u.data_ptr(), v.data_ptr(), tau.data_ptr())
            elif m % 2:
                tau = _batch_step(B, b, [(u, v)])[0]
            else:
                B.sbim_batch_replay(b)
                tau = tb
            stream.synchronize()
            r = ref.step(u.double(), v.double()).cpu().numpy()
            err.update(rel_l2(tau.double().cpu().numpy(), r))
        B.sbim_batch_destroy(b)
    assert err.value < TOL["fp32"], err
