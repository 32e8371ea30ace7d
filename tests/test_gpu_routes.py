"""Which kernel a call, a prepared batch or a session runs, by the names the CUDA
profiler records: the launch rules, the plan settings that pick a kernel, and the
same rule for a frame passed as a parameter and through work tables."""
import re

import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2405_04253_gb300 as F  # noqa: E402


def kernels(fn, instance=False):
    """Names of the library's kernels that fn launches, in order of their start
    (instance: with their template arguments)."""
    from torch.profiler import ProfilerActivity, profile
    for _ in range(3):                       # the first session of a process may record nothing
        torch.cuda.synchronize()
        with profile(activities=[ProfilerActivity.CUDA]) as prof:
            fn()
            torch.cuda.synchronize()
        ev = sorted((e for e in prof.events() if "fnt::" in e.name), key=lambda e: e.time_range.start)
        if ev:
            pat = r"::(\w+(?:<[^(]*>)?)\(" if instance else r"::(\w+)[<(]"
            return [re.search(pat, e.name.replace("(anonymous namespace)::", "")).group(1) for e in ev]
    pytest.skip("the CUDA profiler records no kernels here")


def symbols(rng, n):
    return torch.from_numpy(rng.integers(-16, 16, (n, 4)).astype(np.int8)).cuda()


def aeq_frames(rng, lens):
    return [F.Frame(symbols(rng, n), torch.zeros((n, 4), dtype=torch.int16, device="cuda")) for n in lens]


def pdm_frame(rng, n, L=17, state=None):
    x = torch.from_numpy(rng.integers(-16, 16, (n, 2, 2)).astype(np.int8)).cuda()
    taps = rng.integers(-32, 32, (L, 2)).astype(np.int8)
    return F.Frame(x, torch.zeros((F.chain_nsym(n, L), 4), dtype=torch.int16, device="cuda"), taps, state)


def run_totals(n, seg, warm):
    """Runs of a frame of n symbols: how many, their symbols in all, the longest."""
    if seg <= 0 or seg >= n:
        return 1, n, n
    runs = [min(n, k + seg) - max(0, k - warm) for k in range(0, n, seg)]
    return len(runs), sum(runs), max(runs)


@pytest.mark.parametrize("period", [1, 3])
@pytest.mark.parametrize("na", [32, 64])
@pytest.mark.parametrize("kind", [0, 1, 2])
@pytest.mark.parametrize("lens", [[3000], [400] * 250, [400] * 700])
def test_aeq_route_names_the_kernel_that_runs(lens, kind, na, period):
    rng = np.random.default_rng(len(lens) + kind)
    plan = F.Plan(n_aeq=na, alpha_aeq=4080 if na == 64 else 2, mu_shift=9, aeq_update_period=period)
    plan.set_aeq_kernel(kind)
    fr = aeq_frames(rng, lens)
    want = plan.aeq_route(len(lens), sum(lens), max(lens))
    assert kernels(lambda: F.aeq_run(plan, fr)) == [want]
    if kind == 0:
        # few (chain, polarisation) items per SM take the split layout
        line = 3.5 if na == 64 else 2.8 if period > 1 else 4.0
        few = 2 * len(lens) < line * torch.cuda.get_device_properties(0).multi_processor_count
        assert want == ("aeq_split_kernel" if few else "aeq_duo_kernel")


@pytest.mark.parametrize("kind", [0, 1, 2])
@pytest.mark.parametrize("n", [5000, 400_000])
def test_cdc_route_names_the_kernel_that_runs(n, kind):
    rng = np.random.default_rng(n + kind)
    plan = F.Plan()
    plan.set_cdc_kernel(kind)
    x = torch.from_numpy(rng.integers(-16, 16, (n, 2, 2)).astype(np.int8)).cuda()
    fr = F.Frame(x, torch.zeros((n, 2, 2), dtype=torch.int16, device="cuda"), np.ones((17, 2), np.int8))
    items = 2 * -(-(-(-n // 48)) // 32)
    assert kernels(lambda: F.cdc_run(plan, [fr]))[-1] == plan.cdc_route(items)
    assert plan.cdc_route(items) == ["cdc_direct_kernel", "cdc_kernel", "cdc_split_kernel"][kind]


@pytest.mark.parametrize("na", [32, 64])
@pytest.mark.parametrize("n,seg,warm", [(30000, 512, 0), (30000, 512, 100), (30001, 512, 1 << 20),
                                        (30001, 512, (1 << 63) - 1), (2600, 512, 3000), (200_000, 250, 4000),
                                        (511, 512, 1 << 40)])
def test_one_frame_takes_the_layout_of_its_tables(n, seg, warm, na):
    """A frame passed as a parameter (a call on it alone, a batch of it) runs in the
    layout that its runs' lengths give, as it does through tables, also where the
    warm-up passes the frame's start or seg + warmup passes 64 bits."""
    rng = np.random.default_rng(n + seg)
    plan = F.Plan(n_aeq=na, alpha_aeq=4080 if na == 64 else 2, mu_shift=9, aeq_segment=seg, aeq_warmup=warm)
    f, g = aeq_frames(rng, [n, 1])
    want = plan.aeq_route(*run_totals(n, seg, warm))
    assert kernels(lambda: F.aeq_run(plan, [f])) == [want]
    got = f.out.clone()
    b = F.Batch(plan, [f], F.OP_AEQ, use_graph=False)
    assert kernels(b.launch) == [want]
    assert torch.equal(f.out, got)
    f.out.zero_()
    assert kernels(lambda: F.aeq_run(plan, [f, g])) == [want]
    assert torch.equal(f.out, got)


@pytest.mark.parametrize("n", [20_000, 66_000, 180_000, 400_000])
@pytest.mark.parametrize("chunks", [2, 16])
def test_pipeline_cuts_direct_batches_where_it_cuts_transform_ones(n, chunks):
    """set_pipeline: a batch that the transform CDC runs in chunks is cut in direct
    form too, with the same results."""
    rng = np.random.default_rng(n + chunks)
    counts, outs = [], []
    f = pdm_frame(rng, n)
    for kind in (0, 1):
        plan = F.Plan(mu_shift=9, aeq_segment=512)
        plan.set_cdc_kernel(kind)
        plan.set_pipeline(chunks)
        b = F.Batch(plan, [f], F.OP_CHAIN, use_graph=False)
        f.out.zero_()
        b.launch()
        torch.cuda.synchronize()
        counts.append(b.kernel_count())
        outs.append(f.out.clone())
    assert torch.equal(*outs)
    assert counts[1] == 2 or counts[0] > 2, counts


CDC_NAMES = ["cdc_direct_kernel", "cdc_kernel", "cdc_split_kernel"]


@pytest.mark.parametrize("chunks", [1, 4])
@pytest.mark.parametrize("lens", [[30_000], [9000, 0, 517, 40_000]])
@pytest.mark.parametrize("first", [0, 1, 2])
def test_prepared_batch_follows_the_cdc_kernel(lens, first, chunks):
    """set_cdc_kernel acts on the next launch of an existing batch (whole, by stage or
    captured by the caller), until the batch has recorded a graph of its own."""
    rng = np.random.default_rng(sum(lens) + first)
    plan = F.Plan(mu_shift=9, aeq_segment=512)
    plan.set_pipeline(chunks)
    frames = [pdm_frame(rng, n, L) for n, L in zip(lens, (17, 5, 31, 8))]
    F.cdc_aeq_run(plan, frames)
    torch.cuda.synchronize()
    want = [f.out.clone() for f in frames]
    plan.set_cdc_kernel(first)
    b = F.Batch(plan, frames, F.OP_CHAIN, use_graph=False)
    g = F.Batch(plan, frames, F.OP_CHAIN, use_graph=True)

    def check(names, kind):
        # (preparing the transform form also computes the tap spectra)
        assert {k for k in names if k.startswith("cdc")} - {"cdc_spectra_kernel"} == {CDC_NAMES[kind]}
        assert all(torch.equal(f.out, w) for f, w in zip(frames, want)), kind
        for f in frames:
            f.out.zero_()

    def stages():
        b.launch_stage(0)
        b.launch_stage(1)

    for kind in (first, 1, 0, 2, 0, 1):
        plan.set_cdc_kernel(kind)
        check(kernels(b.launch), kind)
        check(kernels(stages), kind)
    # the caller's capture, on a batch that was made in the other form
    plan.set_cdc_kernel(0 if first else 1)
    c = F.Batch(plan, frames, F.OP_CHAIN, use_graph=False)
    plan.set_cdc_kernel(first)
    graph, side = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    with torch.cuda.graph(graph, stream=side):
        c.launch(side)
    check(kernels(graph.replay), first)
    # a recorded graph stays as it is
    plan.set_cdc_kernel(2 - first)
    check(kernels(g.launch), 2 - first)
    plan.set_cdc_kernel(first)
    check(kernels(g.launch), 2 - first)


@pytest.mark.parametrize("graph", [False, True])
@pytest.mark.parametrize("op", [F.OP_CDC, F.OP_CHAIN])
def test_input_copy_in_both_forms_of_a_batch(op, graph):
    """Host inputs read in place or through the batch's copy, in the form the batch was
    made in and in the one it moved to."""
    rng = np.random.default_rng(op)
    plan = F.Plan(mu_shift=9)
    xs = [torch.from_numpy(rng.integers(-16, 16, (n, 2, 2)).astype(np.int8)).pin_memory() for n in (5000, 700)]
    taps = rng.integers(-32, 32, (17, 2)).astype(np.int8)
    shapes = [(x.shape[0], 2, 2) if op == F.OP_CDC else (F.chain_nsym(x.shape[0], 17), 4) for x in xs]
    outs = [torch.zeros(s, dtype=torch.int16).pin_memory() for s in shapes]
    dev = [F.Frame(x.cuda(), torch.zeros(s, dtype=torch.int16, device="cuda"), taps) for x, s in zip(xs, shapes)]
    (F.cdc_run if op == F.OP_CDC else F.cdc_aeq_run)(plan, dev)
    want = [f.out.cpu() for f in dev]
    b = F.Batch(plan, [F.Frame(x, o, taps) for x, o in zip(xs, outs)], op, use_graph=graph, host=True)
    for kind, copy in [(0, False), (1, False), (1, True), (0, True), (0, False), (1, False)]:
        plan.set_cdc_kernel(kind)
        b.set_input_copy(copy)
        for o in outs:
            o.zero_()
        b.launch()
        torch.cuda.synchronize()
        assert all(torch.equal(o, w) for o, w in zip(outs, want)), (kind, copy)


def test_transform_settings_act_on_the_kernel_that_has_them():
    """The tensor-core gradient and two-polarisation CDC items change the instance of
    the transform kernels that runs; the direct forms ignore them."""
    rng = np.random.default_rng(5)
    f = pdm_frame(rng, 30_000)

    def instances(kind, tensor, pols):
        plan = F.Plan(mu_shift=9, aeq_segment=512)
        plan.set_aeq_kernel(kind)
        plan.set_cdc_kernel(kind)
        plan.set_tensor_gradient(tensor)
        plan.set_cdc_items(pols)
        f.out.zero_()
        names = kernels(lambda: F.cdc_aeq_run(plan, [f]), instance=True)
        return names[-2:], f.out.clone()

    base, want = instances(1, False, 1)
    tensor, got = instances(1, True, 2)
    assert base[0] != tensor[0] and base[1] != tensor[1] and torch.equal(got, want)
    assert [n.split("<")[0] for n in base] == ["cdc_kernel", "aeq_kernel"] == [n.split("<")[0] for n in tensor]
    direct, got = instances(0, True, 2)
    assert direct == instances(0, False, 1)[0] and torch.equal(got, want)
    assert [n.split("<")[0] for n in direct] == ["cdc_direct_kernel", "aeq_split_kernel"]
