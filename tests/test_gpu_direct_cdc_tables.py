"""GPU parity of the direct CDC through work tables: calls and prepared batches of
several frames, on device and host buffers.  Bit-exact against the CPU oracle."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2405_04253_gb300 as F  # noqa: E402

POISON = 0x3C3C


def cdc_frames(rng, sizes, place):
    """Frames of mixed polarisations and taps with POISON around every output; their
    guarded outputs, and a function that returns what each should hold."""
    frames, guarded, args = [], [], []
    for n in sizes:
        npol, L = int(rng.integers(1, 3)), int(rng.integers(1, 32))
        x = rng.integers(-16, 16, (n, npol, 2)).astype(np.int8)
        taps = rng.integers(-32, 32, (L, 2)).astype(np.int8)
        g = place(torch.full((n + 2, npol, 2), POISON, dtype=torch.int16))
        frames.append(F.Frame(place(torch.from_numpy(x)), g[1:n + 1], taps, n_pol=npol))
        guarded.append(g)
        args.append((x, taps))
    return frames, guarded, args


def check_cdc(orc, guarded, args):
    for i, (g, (x, taps)) in enumerate(zip(guarded, args)):
        got = g.cpu().numpy()
        assert (got[0] == POISON).all() and (got[-1] == POISON).all(), i
        if x.shape[0]:
            assert np.array_equal(got[1:-1].astype(np.int32), orc.cdc(x, taps)), i


# 304 tiles of 256 samples (two per SM) is the line between items of one tile and of four
SIZES = {"one_tile_items": [1, 255, 256, 257, 0, 512, 9001, 3, 1025],
         "four_tile_items": [40_000, 1, 256 * 5, 0, 70_001, 1023, 1024, 1025, 257]}


@pytest.mark.parametrize("sizes", list(SIZES))
@pytest.mark.parametrize("via", ["call", "host_call", "batch", "graph", "stage"])
def test_cdc_tables_of_mixed_frames(orc, via, sizes):
    """The direct CDC over several frames: one and two polarisations in one launch,
    frames of less than a tile to many items, an empty one among them."""
    rng = np.random.default_rng(len(via) + len(sizes))
    host = via == "host_call"
    frames, guarded, args = cdc_frames(rng, SIZES[sizes], (lambda t: t) if host else (lambda t: t.cuda()))
    tiles = sum(-(-n // 256) for n in SIZES[sizes])
    n_sm = torch.cuda.get_device_properties(0).multi_processor_count
    assert (tiles <= 2 * n_sm) == (sizes == "one_tile_items")
    plan = F.Plan()
    assert plan.cdc_route() == "cdc_direct_kernel"
    if via in ("call", "host_call"):
        F.cdc_run(plan, frames, host=host)
    else:
        b = F.Batch(plan, frames, F.OP_CDC, use_graph=via == "graph")
        assert b.kernel_count() == 1
        for _ in range(2):
            b.launch_stage(0) if via == "stage" else b.launch()
    torch.cuda.synchronize()
    check_cdc(orc, guarded, args)


@pytest.mark.parametrize("sizes", [[5001], [77_777], *SIZES.values()], ids=["one", "one_long", *SIZES])
@pytest.mark.parametrize("graph", [False, True])
def test_cdc_batch_on_host_buffers(orc, graph, sizes):
    """A prepared CDC batch on page-locked host buffers, inputs read in place and
    through the input copy, switched on and off between launches."""
    rng = np.random.default_rng(len(sizes) + graph)
    frames, guarded, args = cdc_frames(rng, sizes, lambda t: t.pin_memory() if t.numel() else t)
    b = F.Batch(F.Plan(), frames, F.OP_CDC, use_graph=graph, host=True)
    for copy in (False, True, True, False):
        b.set_input_copy(copy)
        for g in guarded:
            g.fill_(POISON)
        b.launch()
        torch.cuda.synchronize()
        check_cdc(orc, guarded, args)


@pytest.mark.parametrize("step,L", [(32, 17), (40, 17), (34, 31), (64, 1)])
def test_cdc_step_and_extremes(orc, step, L):
    """The overlap-save step and worst-case magnitudes, one frame and two."""
    rng = np.random.default_rng(step + L)
    x = rng.integers(-16, 16, (4000, 2, 2)).astype(np.int8)
    x[:700] = -16
    taps = np.full((L, 2), -32, np.int8)
    taps[L // 2:] = 31
    ref = orc.cdc(x, taps, 64, 4080, step)
    for frames in (1, 2):
        outs = [torch.full((4000, 2, 2), POISON, dtype=torch.int16, device="cuda") for _ in range(frames)]
        xd = torch.from_numpy(x).cuda()
        F.cdc_run(F.Plan(cdc_step=step), [F.Frame(xd, o, taps) for o in outs])
        torch.cuda.synchronize()
        assert all(np.array_equal(o.cpu().numpy().astype(np.int32), ref) for o in outs)
