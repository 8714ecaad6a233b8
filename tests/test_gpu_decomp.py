"""The x-split domain decomposition on the GPU: slabs held by one process
(one solver each, ghost columns exchanged through the C ABI's column
blocks) advance exactly as the undivided lattice, bit for bit, in FP32 and
with FP16 storage.  The multi-GPU transport (NCCL between ranks) is the
same exchange over torch.distributed; it is covered on the CPU with gloo
ranks (tests/test_decomp.py)."""
from dataclasses import replace

import numpy as np
import pytest

from paper_1411_2181_gb300 import configs, decomp

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    from paper_1411_2181_gb300 import build
    build.build()
    from paper_1411_2181_gb300 import lbfe
    return lbfe


@pytest.mark.parametrize("parts", [2, 3])
@pytest.mark.parametrize("prec", [0, 1])
def test_slabs_equal_the_undivided_lattice(L, parts, prec):
    p, rho, _ = configs.config1()
    p = replace(p, precision=prec)
    steps = 30
    whole = L.Solver(p)
    whole.init(0, rho)
    whole.step(steps)
    slabs = []
    for x0, nx in decomp.partition(p.Lx, parts):
        s = L.Solver(decomp.local_params(p, nx))
        s.init(0, decomp.slab_field(rho, x0, nx))
        slabs.append(decomp.Slab(x0, nx, decomp.CudaSlabStepper(s)))
    decomp.run(slabs, decomp.LocalRing(slabs), steps)
    f = np.concatenate([decomp.interior(s.stepper.s.get_field(0, L.FIELD_F)) for s in slabs], axis=-1)
    C = np.concatenate([decomp.interior(s.stepper.s.get_field(0, L.FIELD_C)) for s in slabs], axis=-1)
    assert np.array_equal(f, whole.get_field(0, L.FIELD_F))
    assert np.array_equal(C, whole.get_field(0, L.FIELD_C))
    for s in slabs:
        assert s.stepper.s.check() == L.OK


def test_column_blocks_round_trip(L):
    p, rho, _ = configs.config1()
    s = L.Solver(replace(p, precision=1))
    s.init(0, rho)
    s.step(3)
    import torch
    n = s.columns_bytes(0, 5)
    assert n == 5 * p.Ly * p.Lz * (38 * 2 + 6 * 4 + 8)
    t = torch.empty(n, dtype=torch.uint8, device="cuda")
    f0 = s.get_field(0, L.FIELD_F)
    s.get_columns(0, 7, 5, t.data_ptr())
    s.set_columns(0, 20, 5, t.data_ptr())
    f1 = s.get_field(0, L.FIELD_F)
    assert np.array_equal(f1[..., 20:25], f0[..., 7:12])
    assert np.array_equal(np.delete(f1, range(20, 25), axis=-1), np.delete(f0, range(20, 25), axis=-1))
    with pytest.raises(L.LbfeError):
        s.get_columns(0, p.Lx - 2, 5, t.data_ptr())


@pytest.mark.parametrize("prec", [0, 1, 2])
@pytest.mark.parametrize("x0,nx", [(0, 37), (1, 1), (3, 2), (5, 31), (36, 1)])
@pytest.mark.parametrize("shift", [0, 2, 1])
def test_column_blocks_against_the_fields(L, prec, x0, nx, shift):
    """Blocks of odd lattices, every unit width (whole runs, single columns,
    buffers at 16-, 2- and 1-byte boundaries): the block holds the stored
    columns, bit for bit the whole-lattice block's, and comes back intact."""
    import torch
    p, _, _ = configs.config1()
    p = replace(p, Lx=37, Ly=9, Lz=5, precision=prec)
    rho = 1.0 + np.random.default_rng(nx).uniform(-0.1, 0.1, (2, p.Lz, p.Ly, p.Lx))
    s = L.Solver(p)
    s.init(0, rho)
    s.step(2)
    eb = 4 if prec == 0 else 2

    def split(raw, n):
        cells = n * p.Ly * p.Lz
        f = raw[:38 * cells * eb].reshape(38, p.Lz, p.Ly, n, eb)
        c = raw[38 * cells * eb:38 * cells * eb + 24 * cells].reshape(6, p.Lz, p.Ly, n, 4)
        d = raw[38 * cells * eb + 24 * cells:].reshape(-1, p.Lz, p.Ly, n, 8)
        return f, c, d

    def get(x, n):
        buf = torch.zeros(s.columns_bytes(0, n) + 16, dtype=torch.uint8, device="cuda")
        s.get_columns(0, x, n, buf.data_ptr() + shift)
        torch.cuda.synchronize()
        assert not buf[:shift].any() and not buf[shift + s.columns_bytes(0, n):].any()
        return buf, buf.cpu().numpy()[shift:shift + s.columns_bytes(0, n)]

    _, whole = get(0, p.Lx)
    assert np.array_equal(split(whole, p.Lx)[1].copy().view(np.float32)[..., 0], s.get_field(0, L.FIELD_C))
    if prec == 0:
        assert np.array_equal(split(whole, p.Lx)[0].copy().view(np.float32)[..., 0].reshape(2, 19, p.Lz, p.Ly, p.Lx),
                              s.get_field(0, L.FIELD_F))
    buf, raw = get(x0, nx)
    for part, ref in zip(split(raw, nx), split(whole, p.Lx)):
        assert np.array_equal(part, ref[:, :, :, x0:x0 + nx])
    # the columns overwritten, then set back: nothing else moves
    junk = torch.full_like(buf, 60)
    s.set_columns(0, x0, nx, junk.data_ptr() + shift)
    for part, ref in zip(split(get(0, p.Lx)[1], p.Lx), split(whole, p.Lx)):
        keep = np.ones(p.Lx, bool)
        keep[x0:x0 + nx] = False
        assert np.array_equal(part[:, :, :, keep], ref[:, :, :, keep])
        assert (part[:, :, :, x0:x0 + nx] == 60).all()
    s.set_columns(0, x0, nx, buf.data_ptr() + shift)
    assert np.array_equal(get(0, p.Lx)[1], whole)
    s.close()


def test_column_blocks_through_pinned_host_memory(L):
    """A pinned host buffer takes the copy engine's path: same bytes."""
    import torch
    p, rho, _ = configs.config1()
    s = L.Solver(p)
    s.init(0, rho)
    s.step(2)
    n = s.columns_bytes(0, 3)
    dev = torch.empty(n, dtype=torch.uint8, device="cuda")
    host = torch.empty(n, dtype=torch.uint8).pin_memory()
    s.get_columns(0, 4, 3, dev.data_ptr())
    s.get_columns(0, 4, 3, host.data_ptr())
    torch.cuda.synchronize()
    assert torch.equal(dev.cpu(), host)
    s.close()


@pytest.mark.parametrize("nx", [80, 192])
def test_large_column_blocks_at_odd_addresses(L, nx):
    """Either side of the size where a block at an odd address goes to the
    copy engine (80 columns of 192 x 96 x 80 in FP16: 66 MB, of twice the depth
    132 MB; whole lattices 159 and 319 MB): the same bytes at any address, out
    and back."""
    import torch
    for Lz in (80, 160):
        p = L.Params(Lx=192, Ly=96, Lz=Lz, R=16.0, Uw=0.02, eta_M=0.5, precision=1)
        rho = 0.5 + np.random.default_rng(Lz).uniform(-0.1, 0.1, (2, Lz, 96, 192))
        s = L.Solver(p)
        s.init(0, rho)
        n = s.columns_bytes(0, nx)
        want = torch.empty(n, dtype=torch.uint8, device="cuda")
        s.get_columns(0, 0, nx, want.data_ptr())
        buf = torch.zeros(n + 16, dtype=torch.uint8, device="cuda")
        s.get_columns(0, 0, nx, buf.data_ptr() + 1)
        torch.cuda.synchronize()
        assert torch.equal(buf[1:1 + n], want) and not buf[:1].any() and not buf[1 + n:].any()
        s.step(1)
        s.set_columns(0, 0, nx, buf.data_ptr() + 1)
        back = torch.empty_like(want)
        s.get_columns(0, 0, nx, back.data_ptr())
        torch.cuda.synchronize()
        assert torch.equal(back, want)
        s.close()
