"""GPU parity of the direct forms (cdc_direct.cu, aeq_direct.cu), the kernels a plan
runs unless it picks a transform kernel: tile, block and batch edges, both layouts,
worst-case values, buffers at odd offsets.  Bit-exact against the CPU oracle."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2405_04253_gb300 as F  # noqa: E402


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def poison(shape):
    return torch.full(shape, 0x3C3C, dtype=torch.int16, device="cuda")


@pytest.mark.parametrize("n_pol", [1, 2])
@pytest.mark.parametrize("n,L,off", [(1, 31, 0), (255, 17, 1), (256, 31, 0), (257, 8, 3), (287, 31, 2), (1024, 1, 0),
                                     (1025, 2, 0), (4096 + 31, 19, 5), (256 * 400 + 9, 30, 0), (256 * 400, 13, 1)])
def test_cdc_tiles(orc, n, L, off, n_pol):
    """Frames around the 256-sample tile, one and four tiles an item (more than
    304 tiles), every tap-pair remainder, buffers off the 32-byte store's
    alignment; nothing outside the frame's output is written."""
    rng = np.random.default_rng(n + L)
    x = rng.integers(-16, 16, (n + off + 40, n_pol, 2)).astype(np.int8)
    taps = rng.integers(-32, 32, (L, 2)).astype(np.int8)
    taps[0] = -32
    out = poison((n + off + 40, n_pol, 2))
    xd = dev(x)
    F.cdc_run(F.Plan(), [F.Frame(xd[off:off + n], out[off:off + n], taps, n_pol=n_pol)])
    torch.cuda.synchronize()
    got = out.cpu().numpy()
    assert np.array_equal(got[off:off + n].astype(np.int32), orc.cdc(x[off:off + n], taps))
    assert (got[:off] == 0x3C3C).all() and (got[off + n:] == 0x3C3C).all()


@pytest.mark.parametrize("n,L,off", [(1, 5, 0), (2, 3, 1), (511, 17, 0), (512, 3, 2), (515, 31, 1), (4 * 512 * 80 + 7, 19, 0),
                                     (4 * 512 * 80, 15, 3)])
def test_chain_tiles(orc, n, L, off):
    """The chain's decimated tiles (256 symbols), both decimation phases."""
    rng = np.random.default_rng(7 * n + L)
    x = rng.integers(-16, 16, (n + off + 9, 2, 2)).astype(np.int8)
    taps = rng.integers(-32, 32, (L, 2)).astype(np.int8)
    plan = F.Plan(mu_shift=14, aeq_segment=512)
    nsym = F.chain_nsym(n, L)
    out = poison((nsym + 3, 4))
    F.cdc_aeq_run(plan, [F.Frame(dev(x)[off:off + n], out[:nsym], taps)])
    torch.cuda.synchronize()
    ref, _ = orc.chain(x[off:off + n], taps, orc.ChainParams(mu_shift=14, seg_len=512))
    got = out.cpu().numpy()
    assert np.array_equal(got[:nsym], ref) and (got[nsym:] == 0x3C3C).all()


@pytest.mark.parametrize("period", [1, 3])
@pytest.mark.parametrize("na,alpha", [(32, 2), (64, 4080)])
@pytest.mark.parametrize("lens", [[1, 15, 16, 17, 47, 48, 49], [127, 128, 129, 191, 192, 193, 383, 385], [2000] * 700])
def test_aeq_layouts(orc, lens, na, alpha, period):
    """Block and staged-batch edges; few items (several warps each) and many of
    equal length (a warp each)."""
    rng = np.random.default_rng(len(lens) + na + period)
    x = rng.integers(-16, 16, (sum(lens) + 1, 4)).astype(np.int8)
    T0 = orc.aeq_init_taps(16, 2048) + rng.integers(-(1 << 22), 1 << 22, (4, 4, 16)).astype(np.int32)
    xd, out = dev(x), poison((sum(lens), 4))
    st = dev(np.stack([T0] * len(lens)))
    plan = F.Plan(n_aeq=na, alpha_aeq=alpha, mu_shift=9, aeq_update_period=period)
    xs, outs = torch.split(xd[1:], lens), torch.split(out, lens)
    F.aeq_run(plan, [F.Frame(a, b, state=s) for a, b, s in zip(xs, outs, st)])
    torch.cuda.synchronize()
    at = 0
    got, Tg = out.cpu().numpy(), st.cpu().numpy()
    for k, n in enumerate(lens):
        if n < 2000 or k % 97 == 0:
            ref, Tr = orc.aeq(x[1 + at:1 + at + n], T0, na, alpha, mu_shift=9, rde_a=64, period=period)
            assert np.array_equal(got[at:at + n], ref), k
            assert np.array_equal(Tg[k], Tr), k
        at += n


@pytest.mark.parametrize("taps", [None, 8191, -8192])
@pytest.mark.parametrize("copies", [1, 700])
@pytest.mark.parametrize("na,alpha", [(32, 2), (64, 4080)])
@pytest.mark.parametrize("mu,a", [(30, 4096), (40, 1), (0, 4096), (63, 64), (62, 4096)])
def test_aeq_extremes(orc, na, alpha, mu, a, copies, taps):
    """Mixed taps, and every tap at an end of its range: saturated outputs and
    |e z| up to 2^46 (the third limb), every shift range, both layouts."""
    rng = np.random.default_rng(mu + na)
    x = np.full((700, 4), -16, dtype=np.int8)
    x[::3 if taps is None else 7] = 15
    W = rng.choice([-8192, 8191, -1, 0, 127, -128], size=(4, 4, 16)) if taps is None else np.full((4, 4, 16), taps)
    T0 = (W.astype(np.int64) << 16).astype(np.int32)
    plan = F.Plan(n_aeq=na, alpha_aeq=alpha, mu_shift=mu, rde_a=a)
    xd, out = dev(x), poison((copies, 700, 4))
    st = dev(np.stack([T0] * copies))
    F.aeq_run(plan, [F.Frame(xd, o, state=s) for o, s in zip(out, st)])
    torch.cuda.synchronize()
    ref, Tr = orc.aeq(x, T0, na, alpha, mu_shift=mu, rde_a=a)
    assert (out.cpu().numpy() == ref).all() and (st.cpu().numpy() == Tr).all()
    if taps is not None:
        assert np.abs(ref.astype(np.int64)).max() >= 32767


@pytest.mark.parametrize("fs", [1, 2])
def test_aeq_freq_sum_plans(orc, fs):
    """Guarded sums (2) give the per-pair results in direct form; wrapping sums
    (1) stay with the transforms."""
    rng = np.random.default_rng(fs)
    x = rng.integers(-16, 16, (3001, 4)).astype(np.int8)
    T0 = (rng.integers(-8192, 8192, (4, 4, 16)).astype(np.int64) << 16).astype(np.int32)
    st, out = dev(T0), poison((3001, 4))
    F.aeq_run(F.Plan(mu_shift=12, aeq_freq_sum=fs), [F.Frame(dev(x), out, state=st)])
    torch.cuda.synchronize()
    ref, Tr = orc.aeq(x, T0, 32, 2, mu_shift=12, rde_a=64, freq_sum=fs)
    assert np.array_equal(out.cpu().numpy(), ref) and np.array_equal(st.cpu().numpy(), Tr)


@pytest.mark.parametrize("copies", [1, 700])
@pytest.mark.parametrize("na,alpha", [(32, 2), (64, 4080)])
def test_aeq_state_beyond_range(orc, na, alpha, copies):
    """A state beyond the 30-bit range (inputs small enough that no transform
    wraps) is used as it is and clamped by the first update."""
    rng = np.random.default_rng(na + copies)
    x = rng.integers(-2, 3, (300, 4)).astype(np.int8)
    T0 = rng.integers(-(1 << 30), 1 << 30, (4, 4, 16)).astype(np.int32)
    plan = F.Plan(n_aeq=na, alpha_aeq=alpha, mu_shift=9)
    xd, out = dev(x), poison((copies, 300, 4))
    st = dev(np.stack([T0] * copies))
    F.aeq_run(plan, [F.Frame(xd, o, state=s) for o, s in zip(out, st)])
    torch.cuda.synchronize()
    ref, Tr = orc.aeq(x, T0, na, alpha, mu_shift=9, rde_a=64)
    assert (out.cpu().numpy() == ref).all() and (st.cpu().numpy() == Tr).all()


@pytest.mark.parametrize("pin", [True, False])
@pytest.mark.parametrize("op", ["cdc", "aeq"])
def test_host_buffers(orc, op, pin):
    """One-shot calls on host buffers of one frame: page-locked ones in place,
    pageable ones staged."""
    rng = np.random.default_rng(17)
    n = 5001
    x = rng.integers(-16, 16, (n, 2, 2)).astype(np.int8)
    taps = rng.integers(-32, 32, (17, 2)).astype(np.int8)
    xt, out = torch.from_numpy(x), torch.full((n, 2, 2) if op == "cdc" else (n, 4), 0x3C3C, dtype=torch.int16)
    if pin:
        xt, out = xt.pin_memory(), out.pin_memory()
    plan = F.Plan(mu_shift=9, aeq_segment=700, aeq_warmup=33)
    if op == "cdc":
        F.cdc_run(plan, [F.Frame(xt, out, taps)], host=True)
        assert np.array_equal(out.numpy().astype(np.int32), orc.cdc(x, taps))
        return
    T0 = orc.aeq_init_taps(16, 2048)
    st = dev(T0)
    F.aeq_run(plan, [F.Frame(xt.reshape(n, 4), out, state=st)], host=True)
    ref, Tr = orc.aeq_segmented(x.reshape(n, 4), T0, 32, 2, 9, 64, 700, 33, True, 1, 0)
    assert np.array_equal(out.numpy(), ref) and np.array_equal(st.cpu().numpy(), Tr)
