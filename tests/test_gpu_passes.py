"""The three-pass step kernel against the tile kernels, bit for bit (the
choice between them must not show in any field), and against the oracle.

Sizes sit at the edges of its decomposition: runs of 256 cells (one cell,
one short, one over), slots of several runs, planes smaller and larger than
a slot, lattices of one cell along an axis, several steps per launch and
across launches (16 at most in one)."""
from dataclasses import replace

import numpy as np
import pytest

from oracle import oracle as O
from tests.helpers import norm_err, random_populations, tensor_err

pytestmark = pytest.mark.gpu

TOL_FEW = 2e-6
SHAPES = [(1, 1, 2), (2, 1, 2), (1, 128, 2), (17, 5, 3), (16, 16, 2), (257, 1, 3), (7, 5, 6), (64, 3, 40), (33, 17, 11),
          (128, 64, 33), (141, 75, 9)]


@pytest.fixture(scope="module")
def L():
    from paper_1411_2181_gb300 import build
    build.build()
    from paper_1411_2181_gb300 import lbfe
    return lbfe


def params(L, shape, prec, adv, phase, **kw):
    Lx, Ly, Lz = shape
    return L.Params(Lx=Lx, Ly=Ly, Lz=Lz, R=2.0, Uw=0.03, G=3.1, eta_M=0.4, lambda_=1.3, eta_P=0.15, tau_P=6.0, L2=40.0,
                    visco_phase=phase, g=(1e-4, -3e-5, 2e-5), precision=prec, advection=adv, **kw)


def solver(L, ps, tune, states):
    s = L.Solver(ps)
    if tune is not None:
        s.tune(*tune)
    for k, (p, (f, C)) in enumerate(zip(s.params, states)):
        s.init(k, np.ones((2, p.Lz, p.Ly, p.Lx)))
        s.set_field(k, L.FIELD_F, f)
        s.set_field(k, L.FIELD_C, C)
    return s


def same(L, a, b, n=1):
    for k in range(n):
        for w in (L.FIELD_F, L.FIELD_C):
            assert np.array_equal(a.get_field(k, w), b.get_field(k, w)), (k, w)


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("prec", [0, 1, 2])
@pytest.mark.parametrize("adv", [0, 1])
def test_fields_are_the_tile_kernels(L, shape, prec, adv):
    phase = (sum(shape) + prec + adv) % 3
    p = params(L, shape, prec, adv, phase)
    st = [random_populations(shape, seed=sum(shape) + prec)]
    tile = solver(L, p, (8, 0, 0), st)
    passes = solver(L, p, (8, 0, L.STEP_PASSES), st)
    assert passes.launch_config()["kernel"] == L.STEP_PASSES
    for n in (1, 2, 3, 17):
        tile.step(n)
        passes.step(n)
        same(L, tile, passes)
    assert tile.check() == passes.check()
    tile.close()
    passes.close()


@pytest.mark.parametrize("shape", [(33, 17, 11), (141, 75, 9)])
def test_against_the_oracle(L, shape):
    p = params(L, shape, 0, 0, 2)
    f0, C0 = random_populations(shape, seed=4)
    s = solver(L, p, (8, 0, L.STEP_PASSES), [(f0, C0)])
    orc = O.Oracle(p.oracle_dict())
    orc.f[:] = f0
    orc.C[:] = C0
    s.step(3)
    orc.step(3)
    assert norm_err(s.get_field(0, L.FIELD_F), orc.f, 2) < TOL_FEW
    assert tensor_err(s.get_field(0, L.FIELD_C), orc.C) < TOL_FEW


@pytest.mark.parametrize("prec", [0, 2])
def test_batches_of_any_sizes_equal_solo_tile_runs(L, prec):
    """70 instances (two launches a step): the batch in passes, each member
    alone in tiles."""
    rng = np.random.default_rng(5)
    shapes = [(int(rng.integers(1, 40)), int(rng.integers(1, 30)), int(rng.integers(2, 20))) for _ in range(70)]
    ps = [params(L, sh, prec, 0, k % 3) for k, sh in enumerate(shapes)]
    st = [random_populations(sh, seed=k) for k, sh in enumerate(shapes)]
    batch = solver(L, ps, (8, 0, L.STEP_PASSES), st)
    for n in (1, 4, 18):
        batch.step(n)
    for k in (0, 13, 41, 63, 64, 69):
        solo = solver(L, ps[k], (8, 0, 0), [st[k]])
        solo.step(23)
        for w in (L.FIELD_F, L.FIELD_C):
            assert np.array_equal(batch.get_field(k, w), solo.get_field(0, w)), k
        solo.close()
    batch.close()


def test_field_queries_and_kernel_changes_between_steps(L):
    """The queries use the scratch the passes use; a handle may go from one
    kernel to the other and back at any step, with an odd number of steps."""
    shape = (33, 17, 11)
    p = params(L, shape, 1, 0, 1)
    st = [random_populations(shape, seed=8)]
    a, b = solver(L, p, (8, 0, 0), st), solver(L, p, (8, 0, L.STEP_PASSES), st)
    for k, tune in enumerate([None, (12, 0, 0), (8, 0, L.STEP_PASSES), (16, 3, 0), (8, 0, L.STEP_PASSES)]):
        if tune:
            b.tune(*tune)
        a.step(k + 1)
        b.step(k + 1)
        for w in (L.FIELD_RHO, L.FIELD_U):
            assert np.array_equal(a.get_field(0, w), b.get_field(0, w))
        same(L, a, b)
    with pytest.raises(L.LbfeError):
        b.tune(12, 0, L.STEP_PASSES)
    with pytest.raises(L.LbfeError):
        b.tune(8, 8, L.STEP_PASSES)


def test_captured_by_the_caller(L):
    """Steps captured into the caller's graph and replayed."""
    import torch
    shape = (33, 17, 11)
    p = params(L, shape, 2, 0, 1)
    st = [random_populations(shape, seed=9)]
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        a, b = solver(L, p, (8, 0, L.STEP_PASSES), st), solver(L, p, (8, 0, L.STEP_PASSES), st)
        a.step(12)
        b.step(2)
        g = torch.cuda.CUDAGraph()
        torch.cuda.synchronize()
        with torch.cuda.graph(g, stream=stream):
            b.step(2)
        for _ in range(5):
            g.replay()
        torch.cuda.synchronize()
        same(L, a, b)


def test_expired_waits_report_timeout(L):
    """Pass M left uncounted: the bounded waits of pass X expire, the kernel
    ends and the handle reports it; a new handle steps as before."""
    import time
    shape = (33, 17, 11)
    p = params(L, shape, 0, 0, 1)
    st = [random_populations(shape, seed=3)]
    s = solver(L, p, (8, 0, L.STEP_PASSES), st)
    s.test_inject(L.INJECT_LOST_COUNTS)
    t0 = time.time()
    s.step(1)
    assert s.check() == L.ERR_TIMEOUT
    assert time.time() - t0 < 30.0
    s.close()
    a, b = solver(L, p, (8, 0, L.STEP_PASSES), st), solver(L, p, (8, 0, 0), st)
    a.step(3)
    b.step(3)
    assert a.check() == L.OK
    same(L, a, b)


def test_two_handles_on_two_streams(L):
    """Launches that share the GPU (their blocks need not all be resident at
    once): each handle's fields are those of its own run."""
    import torch
    shapes = [(96, 64, 48), (64, 80, 56)]
    out = []
    for together in (True, False):
        hs = []
        for k, sh in enumerate(shapes):
            st = torch.cuda.Stream()
            with torch.cuda.stream(st):
                hs.append(solver(L, params(L, sh, 0, 0, 1), (8, 0, L.STEP_PASSES), [random_populations(sh, seed=k, amp=0.01)]))
        torch.cuda.synchronize()
        for _ in range(8):
            for s in hs:
                s.step(20)
                if not together:
                    torch.cuda.synchronize()
        assert all(s.check() == L.OK for s in hs)
        out.append([s.get_field(0, w) for s in hs for w in (L.FIELD_F, L.FIELD_C)])
        for s in hs:
            s.close()
    assert all(np.array_equal(a, b) for a, b in zip(*out))


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("shapes", [[(141, 75, 9)], [(256, 128, 12)], [(7, 5, 6), (256, 128, 12), (33, 17, 11)]])
def test_a_launch_stops_at_expired_waits(L, shapes, prec):
    """Waits expire with jobs handed over and copies of both stages issued
    (slots of one and of four runs, one and several steps, small and large
    lattices in a batch): the launch ends with a status, no job or copy is
    overwritten, and the blocks that take the shared memory over next, at
    once on the same stream, compute the right fields."""
    import time
    ps = [params(L, sh, prec, 0, 1) for sh in shapes]
    st = [random_populations(sh, seed=3, amp=0.01) for sh in shapes]
    ref = solver(L, ps, (8, 0, 0), st)
    ref.step(3)
    for steps in (1, 2, 5):
        s, nxt = (solver(L, ps, (8, 0, L.STEP_PASSES), st) for _ in range(2))
        s.test_inject(L.INJECT_LOST_COUNTS)
        t0 = time.time()
        s.step(steps)
        nxt.step(3)
        assert s.check() == L.ERR_TIMEOUT and time.time() - t0 < 30.0
        assert nxt.check() == L.OK
        same(L, nxt, ref, len(shapes))
        s.close()
        nxt.close()
    ref.close()


@pytest.mark.parametrize("prec", [0, 2])
def test_a_handle_steps_again_after_expired_waits(L, prec):
    """A launch that gave up leaves its counters as if every slot had been
    counted: the same handle, its hook undone and initialised again, steps in
    order, at once, with the tile kernel's bits (70 instances: two launches a
    step).  The status keeps telling of the expired wait."""
    import time
    rng = np.random.default_rng(11)
    shapes = [(141, 75, 9), (256, 64, 12)] + [(int(rng.integers(1, 40)), int(rng.integers(1, 30)), int(rng.integers(2, 20)))
                                              for _ in range(68)]
    ps = [params(L, sh, prec, 0, k % 3) for k, sh in enumerate(shapes)]
    st = [random_populations(sh, seed=k, amp=0.01) for k, sh in enumerate(shapes)]
    s, ref = solver(L, ps, (8, 0, L.STEP_PASSES), st), solver(L, ps, (8, 0, 0), st)
    for lost in (1, 3):
        s.test_inject(L.INJECT_LOST_COUNTS)
        s.step(lost)
        assert s.check() == L.ERR_TIMEOUT
        s.test_inject(0)
        for h in (s, ref):
            for k, (p, (f, C)) in enumerate(zip(ps, st)):
                h.init(k, np.ones((2, p.Lz, p.Ly, p.Lx)))
                h.set_field(k, L.FIELD_F, f)
                h.set_field(k, L.FIELD_C, C)
        t0 = time.time()
        for n in (1, 4, 18):
            s.step(n)
            ref.step(n)
        assert s.check() == L.ERR_TIMEOUT and time.time() - t0 < 0.5
        same(L, s, ref, len(shapes))
    s.close()
    ref.close()


def test_which_kernel_runs(L):
    """A handle tells which kernel its steps run on: the estimate's choice for
    new handles (small, ragged and FP16 boxes; the tile kernel on 192 x 96 x 80
    and 128 x 96 x 80), what lbfe_tune said for tuned ones, the tiles under the
    short-copies hook.  The default tile shape stays what it is."""
    for shape, prec, kern in [((32, 32, 32), 0, L.STEP_PASSES), ((32, 32, 32), 1, L.STEP_PASSES),
                              ((141, 75, 53), 0, L.STEP_PASSES), ((141, 75, 53), 2, L.STEP_PASSES),
                              ((100, 96, 80), 1, L.STEP_PASSES), ((192, 96, 80), 0, L.STEP_CELL),
                              ((192, 96, 80), 1, L.STEP_CELL), ((192, 96, 80), 2, L.STEP_CELL),
                              ((128, 96, 80), 0, L.STEP_CELL)]:
        s = L.Solver(params(L, shape, prec, 0, 1))
        assert s.step_variant(20) == kern, (shape, prec)
        assert s.launch_config()["kernel"] == L.STEP_CELL
        s.tune(8, 0, L.STEP_PASSES)
        assert s.step_variant(20) == s.step_variant(1) == s.launch_config()["kernel"] == L.STEP_PASSES
        s.test_inject(L.INJECT_SHORT_COPIES)
        assert s.step_variant(20) == L.STEP_CELL
        s.test_inject(0)
        s.tune(16, 0, L.STEP_CELL)
        assert s.step_variant(20) == s.step_variant(1) == L.STEP_CELL
        s.close()
    assert L._lib.lbfe_step_variant(None, 1) == -1


@pytest.mark.parametrize("prec", [0, 1, 2])
def test_default_tiles_are_the_passes(L, prec):
    """The shape a new handle steps a large lattice with (8 rows, 12 with
    2-byte storage, rows copied by TMA) against the passes, bit for bit."""
    shape = (192, 96, 80)
    p = params(L, shape, prec, 0, 1)
    st = [random_populations(shape, seed=2, amp=0.01)]
    a, b = solver(L, p, None, st), solver(L, p, (8, 0, L.STEP_PASSES), st)
    assert a.step_variant(5) == L.STEP_CELL
    a.step(5)
    b.step(5)
    same(L, a, b)


@pytest.mark.parametrize("prec,adv", [(0, 0), (2, 0), (0, 1)])
def test_the_steps_of_a_call_decide_too(L, prec, adv):
    """A launch of the passes has an end that nothing overlaps: 64^3 takes the
    tiles for a call of one step (38 us, passes 47) and the passes for twenty
    (32), 32^3 the passes for both.  A handle that goes from one to the other
    with every call has the bits of either."""
    small = L.Solver(params(L, (32, 32, 32), prec, adv, 1))
    assert small.step_variant(1) == small.step_variant(20) == L.STEP_PASSES
    shape = (50, 96, 80) if prec or adv else (64, 64, 64)
    p = params(L, shape, prec, adv, 1)
    st = [random_populations(shape, seed=6, amp=0.01)]
    s, tile, passes = solver(L, p, None, st), solver(L, p, (8, 0, 0), st), solver(L, p, (8, 0, L.STEP_PASSES), st)
    assert s.step_variant(1) == L.STEP_CELL and s.step_variant(20) == L.STEP_PASSES
    assert passes.step_variant(1) == L.STEP_PASSES
    for n in (1, 20, 1, 1, 17, 20, 1):
        for h in (s, tile, passes):
            h.step(n)
        same(L, s, tile)
        same(L, s, passes)
