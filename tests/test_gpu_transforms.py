"""The transform kernels on the routes that the direct forms take by default: serving
sessions, the allocation-free call (its table path), full-size batches, pipelined
batches, and the settings and sums that only the transform kernels have."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2405_04253_gb300 as F  # noqa: E402
import synth  # noqa: E402

MU = 9


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def i16(shape):
    return torch.full(shape, 0x5A5A, dtype=torch.int16, device="cuda")


def plan_of(cdc, aeq, tensor=False, pols=0, warps=0, cap=0, **kw):
    p = F.Plan(mu_shift=MU, **kw)
    p.set_cdc_kernel(cdc)
    p.set_aeq_kernel(aeq)
    p.set_tensor_gradient(tensor)
    p.set_cdc_items(pols)
    p.set_launch(warps, warps)
    p.set_aeq_occupancy(cap)
    return p


# (CDC kernel, AEQ kernel): both transforms, and one stage of each form
KERNELS = [(1, 1), (2, 2), (0, 1), (2, 0)]


@pytest.mark.parametrize("cdc,aeq", KERNELS)
@pytest.mark.parametrize("kw,opts", [({}, {}), ({}, dict(tensor=True, pols=2)), (dict(aeq_update_period=3), {}),
                                     (dict(n_aeq=64, alpha_aeq=4080, aeq_segment=432), dict(tensor=True))])
def test_session_on_picked_kernels(orc, cdc, aeq, kw, opts):
    """Links with several frames in flight, chained on the device, on every pair of
    kernels, equal sequential oracle processing."""
    rng = np.random.default_rng(71)
    links = [rng.integers(-32, 32, (L, 2)).astype(np.int8) for L in (17, 5, 19)]
    frames = [(int(rng.integers(0, 3)), rng.integers(-16, 16, (int(rng.integers(500, 7000)), 2, 2)).astype(np.int8))
              for _ in range(11)]
    s = F.Session(plan_of(cdc, aeq, **opts, **kw), len(links), 1 << 30, 2)
    for link, taps in enumerate(links):
        s.set_link(link, taps)
    xs = [dev(x) for _, x in frames]
    outs = [i16((F.chain_nsym(x.shape[0], links[link].shape[0]), 4)) for link, x in frames]
    torch.cuda.synchronize()
    assert len(s.submit_many(F.Requests([link for link, _ in frames], xs, outs))) == len(frames)
    done = []
    while len(done) < len(frames):
        done += s.poll_array(timeout_us=1000000).tolist()
    assert all(c[2] == F.FNT_OK for c in done)
    prm = orc.ChainParams(mu_shift=MU, n_aeq=kw.get("n_aeq", 32), alpha_aeq=kw.get("alpha_aeq", 2),
                          seg_len=kw.get("aeq_segment", 0), period=kw.get("aeq_update_period", 1))
    T = {link: orc.aeq_init_taps(16, prm.w0) for link in range(len(links))}
    for i, (link, x) in enumerate(frames):
        ref, T[link] = orc.chain(x, links[link], prm, T0=T[link])
        assert np.array_equal(outs[i].cpu().numpy(), ref), i
    assert all(np.array_equal(s.get_link_state(link), T[link]) for link in T)
    s.close()


@pytest.mark.parametrize("cdc,aeq", KERNELS)
@pytest.mark.parametrize("kw", [{}, dict(aeq_segment=700, aeq_warmup=33), dict(n_aeq=64, alpha_aeq=4080, aeq_segment=500)])
def test_noalloc_through_its_tables(orc, cdc, aeq, kw):
    """The allocation-free call where it builds tables: more calls in a row than it has
    host copies of them, frames of other lengths and taps each, direct calls in between,
    carried state; each equals the oracle."""
    rng = np.random.default_rng(72)
    plan, direct = plan_of(cdc, aeq, **kw), plan_of(0, 0, **kw)
    prm = orc.ChainParams(mu_shift=MU, n_aeq=kw.get("n_aeq", 32), alpha_aeq=kw.get("alpha_aeq", 2),
                          seg_len=kw.get("aeq_segment", 0), warmup=kw.get("aeq_warmup", 0))
    T = orc.aeq_init_taps(16, prm.w0)
    st = dev(T)
    jobs = []
    for k in range(11):
        n, L = (1, 2, 3)[k] if k < 3 else int(rng.integers(300, 9000)), int(rng.choice([1, 5, 8, 17, 31]))
        x, taps = rng.integers(-16, 16, (n, 2, 2)).astype(np.int8), rng.integers(-32, 32, (L, 2)).astype(np.int8)
        jobs.append((x, taps, dev(x), i16((max(1, F.chain_nsym(n, L)), 4))))
    torch.cuda.synchronize()
    for k, (x, taps, xd, out) in enumerate(jobs):
        F.cdc_aeq_run_noalloc(direct if k % 5 == 4 else plan, F.Frame(xd, out, taps, st))
    torch.cuda.synchronize()
    for k, (x, taps, xd, out) in enumerate(jobs):
        nsym = F.chain_nsym(x.shape[0], taps.shape[0])
        if nsym:
            ref, T = orc.chain(x, taps, prm, T0=T)
            assert np.array_equal(out.cpu().numpy(), ref), k
        else:
            assert (out == 0x5A5A).all()
    assert np.array_equal(st.cpu().numpy(), T)


@pytest.mark.parametrize("cdc,aeq", KERNELS)
def test_noalloc_tables_at_their_limits(cdc, aeq):
    """The largest frame with the most CDC items and AEQ segments the tables hold, on
    transform kernels and on one stage of each form."""
    n = F.NOALLOC_MAX_SAMPLES
    f = synth.config2(n // 2)
    kw = dict(cdc_step=32, aeq_segment=256)
    nsym = F.chain_nsym(n, f.taps.shape[0])
    x, ref, out = dev(f.x), i16((nsym, 4)), i16((nsym, 4))
    init = dev(F.Plan().initial_state())
    st_ref, st = init.clone(), init.clone()
    F.cdc_aeq_run(plan_of(0, 0, **kw), [F.Frame(x, ref, f.taps, st_ref)])
    F.cdc_aeq_run_noalloc(plan_of(cdc, aeq, **kw), F.Frame(x, out, f.taps, st))
    torch.cuda.synchronize()
    assert torch.equal(out, ref) and torch.equal(st, st_ref)


@pytest.mark.parametrize("cap,warps", [(4, 4), (12, 4), (20, 2)])
@pytest.mark.parametrize("tensor", [False, True])
def test_occupancy_cap_of_the_warp_kernel(orc, cap, warps, tensor):
    """Capped and uncapped launches of AEQ kernel 1 give the same bits, the oracle's."""
    rng = np.random.default_rng(73)
    fr = [synth.random_frame(rng, n, 2, int(rng.choice([5, 17, 19]))) for n in [4096, 9000, 20000, 333, 60000]]
    got = []
    for c in (0, cap):
        outs = [i16((F.chain_nsym(f.x.shape[0], f.taps.shape[0]), 4)) for f in fr]
        F.cdc_aeq_run(plan_of(1, 1, tensor=tensor, warps=warps, cap=c),
                      [F.Frame(dev(f.x), o, f.taps) for f, o in zip(fr, outs)])
        torch.cuda.synchronize()
        got.append([o.cpu().numpy() for o in outs])
    assert all(np.array_equal(a, b) for a, b in zip(*got))
    ref, _ = orc.chain(fr[3].x, fr[3].taps, orc.ChainParams(mu_shift=MU))
    assert np.array_equal(got[1][3], ref)


@pytest.mark.parametrize("na,alpha", [(32, 2), (64, 4080)])
@pytest.mark.parametrize("taps", ["init", "random", "wrapping", "small"])
@pytest.mark.parametrize("mu,period,tensor", [(10, 1, False), (12, 3, True), (63, 1, False)])
def test_guarded_summation_of_the_warp_kernel(orc, na, alpha, taps, mu, period, tensor):
    """aeq_freq_sum = 2 on the kernel that sums: a plan that picks it, by either number."""
    rng = np.random.default_rng(na + len(taps))
    x = rng.integers(-16, 16, (1500, 4)).astype(np.int8)
    T0 = orc.aeq_init_taps(16, 2048)
    if taps == "random":
        T0 = T0 + rng.integers(-(1 << 22), 1 << 22, (4, 4, 16)).astype(np.int32)
    elif taps == "wrapping":
        x[::4] = -16
        T0 = (rng.choice([8191, 8000, -8192, 4000, 127], size=(4, 4, 16)).astype(np.int64) << 16).astype(np.int32)
    elif taps == "small":
        W = np.full((4, 4, 16), 0)
        W[[0, 1, 2, 3], [0, 1, 2, 3], 8], W[:, :, 7] = 20, 3
        T0 = (W << 16).astype(np.int32)
    ref, Tr = orc.aeq(x, T0, na, alpha, mu_shift=mu, rde_a=64, period=period)
    for kind in (1, 2):
        plan = F.Plan(n_aeq=na, alpha_aeq=alpha, mu_shift=mu, aeq_update_period=period, aeq_freq_sum=2)
        plan.set_aeq_kernel(kind)
        plan.set_tensor_gradient(tensor)
        assert plan.aeq_route(1, 1500, 1500) == "aeq_kernel"
        out, st = i16((1500, 4)), dev(T0)
        F.aeq_run(plan, [F.Frame(dev(x), out, state=st)])
        torch.cuda.synchronize()
        assert np.array_equal(out.cpu().numpy(), ref) and np.array_equal(st.cpu().numpy(), Tr), kind


@pytest.mark.parametrize("seg,cdc,aeq,opts", [(0, 1, 2, {}), (864, 1, 1, dict(pols=2, tensor=True)), (864, 2, 1, dict(pols=1))])
def test_full_size_stream(seg, cdc, aeq, opts):
    """The 2^21-sample stream on the transform kernels equals the direct forms, whole and
    pipelined: the CTA-per-chain kernel on the serial recurrence, the warp kernel on
    864-symbol segments (two-polarisation items with the tensor-core gradient too)."""
    f = synth.config2()
    kw = dict(n_aeq=64, alpha_aeq=4080, aeq_segment=seg)
    nsym = F.chain_nsym(f.x.shape[0], f.taps.shape[0])
    x, ref = dev(f.x), i16((nsym, 4))
    init = dev(F.Plan().initial_state())
    st_ref = init.clone()
    F.cdc_aeq_run(plan_of(0, 0, **kw), [F.Frame(x, ref, f.taps, st_ref)])
    plan = plan_of(cdc, aeq, **opts, **kw)
    runs = -(-nsym // seg) if seg else 1
    assert plan.aeq_route(runs, nsym, seg or nsym) == ("aeq_serial_kernel" if aeq == 2 else "aeq_kernel")
    for chunks in (1, 4):
        plan.set_pipeline(chunks)
        st, out = init.clone(), i16((nsym, 4))
        b = F.Batch(plan, [F.Frame(x, out, f.taps, st)], F.OP_CHAIN, use_graph=True)
        b.launch()
        torch.cuda.synchronize()
        assert torch.equal(out, ref) and torch.equal(st, st_ref), chunks


@pytest.mark.parametrize("chunks,graph,pols", [(4, True, 1), (3, False, 2), (1, False, 0), (5, True, 2)])
def test_pipelined_transform_batch(orc, chunks, graph, pols):
    """Many frames in chunks on the transform kernels, launched twice (the tap spectra
    are those of the batch's creation)."""
    rng = np.random.default_rng(74)
    fr = [(rng.integers(-16, 16, (int(2 ** rng.uniform(10, 14.5)), 2, 2)).astype(np.int8),
           rng.integers(-32, 32, (int(rng.choice([5, 9, 13, 17, 19])), 2)).astype(np.int8)) for _ in range(40)]
    plan = plan_of(1, 1, pols=pols)
    plan.set_pipeline(chunks)
    frames = [F.Frame(dev(x), i16((F.chain_nsym(x.shape[0], t.shape[0]), 4)), t) for x, t in fr]
    b = F.Batch(plan, frames, F.OP_CHAIN, use_graph=graph)
    b.launch()
    for f in frames:
        f.out.zero_()
    b.launch()
    torch.cuda.synchronize()
    assert (b.kernel_count() > 2) == (chunks > 1)
    got = [f.out.clone() for f in frames]
    F.cdc_aeq_run(plan_of(0, 0), frames)
    torch.cuda.synchronize()
    assert all(torch.equal(g, f.out) for g, f in zip(got, frames))
    for i in (0, 7, 39):
        ref, _ = orc.chain(*fr[i], orc.ChainParams(mu_shift=MU))
        assert np.array_equal(got[i].cpu().numpy(), ref)
