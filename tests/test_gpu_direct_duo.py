"""GPU parity of the direct AEQ's duo layout (many chains) at block and batch edges and
on segments.  Bit-exact against the CPU oracle."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2405_04253_gb300 as F  # noqa: E402

POISON = 0x3C3C


@pytest.mark.parametrize("period", [1, 3])
@pytest.mark.parametrize("na", [32, 64])
@pytest.mark.parametrize("n", [1, 15, 16, 17, 47, 48, 49, 383, 384, 385, 511, 512, 513])
def test_aeq_duo_edges(orc, n, na, period):
    """Frames around a block (16 symbols at N = 32, 48 at N = 64) and around the staged
    batch (512 and 384 symbols), so many of them that they run in the duo layout; every
    frame has its own symbols and taps."""
    count = 700
    rng = np.random.default_rng(n * 10 + na + period)
    plan = F.Plan(n_aeq=na, alpha_aeq=4080 if na == 64 else 2, mu_shift=9, aeq_update_period=period)
    assert plan.aeq_route(count, count * n, n) == "aeq_duo_kernel"
    x = rng.integers(-16, 16, (count, n, 4)).astype(np.int8)
    T0 = orc.aeq_init_taps(16, 2048) + rng.integers(-(1 << 22), 1 << 22, (count, 4, 4, 16)).astype(np.int32)
    xd, st = torch.from_numpy(x).cuda(), torch.from_numpy(T0).cuda()
    out = torch.full((count, n, 4), POISON, dtype=torch.int16, device="cuda")
    F.aeq_run(plan, [F.Frame(a, o, state=s) for a, o, s in zip(xd, out, st)])
    torch.cuda.synchronize()
    got, Tg = out.cpu().numpy(), st.cpu().numpy()
    for k in (0, 1, 349, count - 2, count - 1):
        ref, Tr = orc.aeq(x[k], T0[k], na, 4080 if na == 64 else 2, mu_shift=9, rde_a=64, period=period)
        assert np.array_equal(got[k], ref) and np.array_equal(Tg[k], Tr), k


@pytest.mark.parametrize("period", [1, 3])
@pytest.mark.parametrize("na", [32, 64])
@pytest.mark.parametrize("seg,warm", [(100, 60), (97, 1), (113, 0)])
def test_aeq_duo_segments(orc, seg, warm, na, period):
    """Segments with and without warm-up, enough of one frame for the duo layout, from
    a carried state; alone (parameter) and beside another frame (tables)."""
    n = 40_007
    rng = np.random.default_rng(seg + na)
    alpha = 4080 if na == 64 else 2
    plan = F.Plan(n_aeq=na, alpha_aeq=alpha, mu_shift=9, aeq_segment=seg, aeq_warmup=warm, aeq_update_period=period)
    runs = [min(n, k + seg) - max(0, k - warm) for k in range(0, n, seg)]
    assert plan.aeq_route(len(runs), sum(runs), max(runs)) == "aeq_duo_kernel"
    x = rng.integers(-16, 16, (n, 4)).astype(np.int8)
    T0 = orc.aeq_init_taps(16, 2048) + rng.integers(-(1 << 22), 1 << 22, (4, 4, 16)).astype(np.int32)
    ref, Tr = orc.aeq_segmented(x, T0, na, alpha, 9, 64, seg, warm, True, period, 0)
    for frames in (1, 2):
        st = torch.from_numpy(T0).cuda()
        outs = [torch.full((m, 4), POISON, dtype=torch.int16, device="cuda") for m in (n, 33)]
        xd = torch.from_numpy(x).cuda()
        F.aeq_run(plan, [F.Frame(xd, outs[0], state=st), F.Frame(xd[:33], outs[1])][:frames])
        torch.cuda.synchronize()
        assert np.array_equal(outs[0].cpu().numpy(), ref) and np.array_equal(st.cpu().numpy(), Tr)
