"""FP64 / FP32 sigma on the tensor cores (digits summed exactly in integers; three
BF16 planes for the FP32 alpha-beta products) at the sizes where its tiles end, with
the vectors that it leaves to the SIMT kernels, on two streams and under capture.
Sampled rows against the oracle: FP64 to 1e-12 and FP32 to 64 * 2^-24 of
(|H||c|)_I, the tolerances of the SIMT kernels that this path replaces."""
import numpy as np
import pytest

import oracle
from gpu_util import assert_sigma_close
from tbsci_inputs import selected_strings, synth_hamiltonian

pytestmark = pytest.mark.gpu
F32 = dict(rel=64 * 2.0 ** -24, norm_rel=1e-5)


@pytest.fixture(scope="module")
def tb():
    import paper_2503_10335_gb300 as tb
    return tb


@pytest.fixture(scope="module")
def ctx(tb):
    c = tb.Context(0)
    yield c
    c.close()


def _space(tb, ctx, n, na, nb, la, lb, seed, scale=0.3, ecore=0.25):
    h, eri, _ = synth_hamiltonian(n, seed=seed, scale=scale)
    asel = None if la is None else selected_strings(n, na, la, seed + 1)
    bsel = None if lb is None else selected_strings(n, nb, lb, seed + 2)
    sp = tb.Space(ctx, n, na, nb, h, eri, ecore, alpha=asel, beta=bsel)
    return sp, oracle.make_space(n, na, nb, asel, bsel), h, eri


def _check(s, osp, h, eri, C, rows, **kw):
    ref, bound = oracle.sigma(osp, h, eri, 0.25, C.reshape(C.shape[0], -1), rows=rows, with_bound=True)
    assert_sigma_close(s.reshape(C.shape[0], -1)[:, rows], ref, bound, **kw)


def _rows(ndet, seed, k=400):
    r = np.random.default_rng(seed)
    return np.unique(np.concatenate([r.choice(ndet, min(k, ndet), replace=False), np.arange(min(40, ndet)), np.arange(max(0, ndet - 40), ndet)]))


def _graded(sp, decades, rng):
    """Normal deviates that fall by `decades` per excitation, in both spins; and the sampled rows: any, and the most excited."""
    a, b = sp.strings()
    level = (np.bitwise_count(a >> np.uint64(sp.nalpha)).astype(int)[:, None] + np.bitwise_count(b >> np.uint64(sp.nbeta)).astype(int))
    C = rng.standard_normal((1, sp.la, sp.lb)) * 10.0 ** (-decades * level)
    top = np.argsort(level.reshape(-1), kind="stable")[-500:]
    return C / np.linalg.norm(C), np.unique(np.concatenate([_rows(sp.ndet, 11, 1500), top]))


@pytest.mark.parametrize("dtype", ["f64", "f32"])
@pytest.mark.parametrize("n,na,nb,la,lb,decades", [
    (11, 5, 5, None, None, 0.8),
    (11, 5, 5, None, None, 1.0),
    (11, 5, 5, None, None, 1.5),
    (16, 8, 8, 700, 650, 1.0),
    (16, 8, 8, 700, 650, 1.5),
    (16, 8, 8, 1500, 1400, 1.5),  # more CTAs than run at once
])
def test_small_elements_keep_their_accuracy(tb, ctx, n, na, nb, la, lb, decades, dtype):
    """Vectors that decay by orders of magnitude per excitation, as CI vectors do: every element
    is as close, relative to the terms of its own sum, as anywhere else."""
    import torch
    sp, osp, h, eri = _space(tb, ctx, n, na, nb, la, lb, seed=760 + n)
    C, rows = _graded(sp, decades, np.random.default_rng(n))
    Ct = torch.from_numpy(C).to(torch.float64 if dtype == "f64" else torch.float32).cuda()
    s = sp.sigma(Ct)
    assert torch.equal(s, sp.sigma(Ct))
    _check(s.double().cpu().numpy(), osp, h, eri, Ct.double().cpu().numpy(), rows, **({} if dtype == "f64" else F32))
    sp.close()


@pytest.mark.parametrize("dtype", ["f64", "f32"])
@pytest.mark.parametrize("decades", [0.0, 0.5])
def test_small_integrals_keep_their_accuracy(tb, ctx, decades, dtype):
    """Integrals that spread over five decades from orbital to orbital: elements whose links are
    all small are as close as the others."""
    import torch
    n = 11
    h, eri, _ = synth_hamiltonian(n, seed=768)
    g = 10.0 ** (-np.linspace(0, 1.25, n))
    h = h * g[:, None] * g[None, :]
    eri = eri * np.einsum("i,j,k,l->ijkl", g, g, g, g)
    sp = tb.Space(ctx, n, 5, 5, h, eri, 0.25)
    osp = oracle.make_space(n, 5, 5)
    C, rows = _graded(sp, decades, np.random.default_rng(12))
    Ct = torch.from_numpy(C).to(torch.float64 if dtype == "f64" else torch.float32).cuda()
    _check(sp.sigma(Ct).double().cpu().numpy(), osp, h, eri, Ct.double().cpu().numpy(), rows, **({} if dtype == "f64" else F32))
    sp.close()


def test_f32_takes_peaked_vectors(tb, ctx):
    """The trial vectors of a mixed solve: one element thousands of times the root mean square.
    They stay on the tensor cores (the bits are not those of a captured call, which is SIMT)."""
    import torch
    sp, osp, h, eri = _space(tb, ctx, 13, 6, 6, 1040, 1030, seed=733)
    C = 1e-4 * np.random.default_rng(8).standard_normal((1, sp.la, sp.lb))
    C[0, 0, 0] = 0.9
    assert np.abs(C).max() > 256 * np.sqrt((C ** 2).mean())
    Ct = torch.from_numpy(C).float().cuda()
    s, out = sp.sigma(Ct), torch.empty_like(Ct)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        sp.sigma(Ct, out)
    g.replay()
    assert not torch.equal(s, out)
    _check(s.double().cpu().numpy(), osp, h, eri, Ct.double().cpu().numpy(), _rows(sp.ndet, 13), **F32)
    sp.close()


@pytest.mark.parametrize("dtype", ["f64", "f32"])
@pytest.mark.parametrize("n,na,nb,la,lb,nvec", [
    (13, 6, 6, 1030, 1025, 2),    # one row past a 128-row tile's multiple of 6, one column past 64
    (16, 8, 8, 1100, 1087, 1),    # rows with all 64 alpha singles (65 terms), a column short of 17 tiles
    (16, 12, 5, 1024, 1024, 1),   # twelve alpha electrons: W beyond eight integrals; whole tiles
    (10, 5, 5, 154, 155, 1),      # 23,870 determinants: the small-space kernel, four column slices per CTA
    (10, 5, 5, 160, 150, 9),      # 24,000: this path, in two launches of eight and one vectors
    (12, 6, 4, 33, 495, 3),       # small-space kernel, few long rows
    (16, 8, 8, 390, 60, 2),       # 23,400: too much for shared memory in FP64
    (8, 4, 4, None, None, 1),     # small-space kernel, one slice per CTA
    (8, 4, 3, 40, 33, 4),         # a column past a slice
    (2, 1, 1, None, None, 1),     # 2 x 2
    (13, 6, 5, None, None, 1),    # a full space: every list at its longest
])
def test_exact_sigma_parity(tb, ctx, n, na, nb, la, lb, nvec, dtype):
    import torch
    sp, osp, h, eri = _space(tb, ctx, n, na, nb, la, lb, seed=700 + n + na)
    tdt = torch.float64 if dtype == "f64" else torch.float32
    rng = np.random.default_rng(n)
    # string weights over two decades, as in a correlated vector
    C = rng.standard_normal((nvec, sp.la, sp.lb)) * (10.0 ** -rng.uniform(0, 2, sp.la))[None, :, None]
    Ct = torch.from_numpy(C).to(tdt).cuda()
    tb.tbsci_trace_enable(ctx.handle, True)
    s = sp.sigma(Ct)
    torch.cuda.synchronize()
    tb.tbsci_trace_enable(ctx.handle, False)
    names = {k for k, _ in tb.tbsci_trace_read(ctx.handle)[0]}
    assert ("k_same_spin_ex" in names) == (sp.ndet >= 24000), names
    assert torch.equal(s, sp.sigma(Ct))  # integer sums: the same in every run
    _check(s.double().cpu().numpy(), osp, h, eri, Ct.double().cpu().numpy(), _rows(sp.ndet, n), **({} if dtype == "f64" else F32))
    sp.close()


@pytest.mark.parametrize("dtype", ["f64", "f32"])
def test_vectors_left_to_the_simt_kernels(tb, ctx, dtype):
    """Per vector of one call: ordinary, a single determinant (its largest entry a
    thousand times its root mean square), zero, extreme magnitudes, infinity, NaN. Each
    agrees with the oracle (or is non-finite exactly where the SIMT kernels are, on a
    captured stream), whatever the others are."""
    import torch
    sp, osp, h, eri = _space(tb, ctx, 13, 6, 6, 1040, 1030, seed=731)
    tdt = torch.float64 if dtype == "f64" else torch.float32
    rng = np.random.default_rng(3)
    C = rng.standard_normal((6, sp.la, sp.lb))
    C[1] = 0.0
    C[1, 5, 7] = 1.0
    C[2] = 0.0
    C[3] *= 1e-25 if dtype == "f32" else 1e-180
    C[4, 17, 3] = np.inf
    C[5, 400, 1000] = np.nan
    Ct = torch.from_numpy(C).to(tdt).cuda()
    s = sp.sigma(Ct)
    got = s.double().cpu().numpy().reshape(6, -1)
    Cr = Ct.double().cpu().numpy()
    rows = np.unique(np.concatenate([_rows(sp.ndet, 5), [5 * sp.lb + 7]]))
    for v in range(4):
        _check(got[v][None], osp, h, eri, Cr[v][None], rows, **({} if dtype == "f64" else F32))
    assert torch.equal(s[0:1], sp.sigma(Ct[0:1].contiguous()))
    out = torch.empty_like(Ct)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):  # a captured call takes the SIMT kernels
        sp.sigma(Ct, out)
    g.replay()
    torch.cuda.synchronize()
    simt = out.double().cpu().numpy().reshape(6, -1)
    assert np.array_equal(np.isnan(got), np.isnan(simt)) and np.array_equal(np.isinf(got), np.isinf(simt))
    _, bound = oracle.sigma(osp, h, eri, 0.25, Cr[0].reshape(1, -1), rows=rows, with_bound=True)
    assert_sigma_close(got[:1, rows], simt[:1, rows], bound, **({} if dtype == "f64" else F32))
    sp.close()


def test_two_streams_share_a_space(tb, ctx):
    """Calls on two streams share the digit planes: each result is what it is alone."""
    import torch
    sp, _, _, _ = _space(tb, ctx, 13, 6, 6, 1030, 1025, seed=741)
    C = torch.randn((6, sp.la, sp.lb), dtype=torch.float64, device="cuda")
    want = [sp.sigma(C[v:v + 1].contiguous()) for v in range(6)]
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    parts = [C[v:v + 1].contiguous() for v in range(6)]
    outs = [torch.empty_like(p) for p in parts]
    torch.cuda.synchronize()
    for v in range(6):
        sp.sigma(parts[v], outs[v], stream=streams[v % 2])
    torch.cuda.synchronize()
    for v in range(6):
        assert torch.equal(outs[v], want[v])
    sp.close()


def test_without_room_for_the_tables(tb):
    """A budget that holds the prepared space but not the digit tables: the SIMT
    kernels serve the call, nothing more is counted, and the result stands."""
    import torch
    ctx = tb.Context(0)
    sp, osp, h, eri = _space(tb, ctx, 13, 6, 6, 1030, 1025, seed=751)
    need = tb.tbsci_hbm_used(ctx.handle)
    C = np.random.default_rng(4).standard_normal((1, sp.la, sp.lb))
    full = sp.sigma(torch.from_numpy(C).cuda())
    assert tb.tbsci_hbm_used(ctx.handle) > need
    sp.close()
    ctx.close()
    ctx = tb.Context(0, hbm_budget=need + (1 << 20))
    sp, _, _, _ = _space(tb, ctx, 13, 6, 6, 1030, 1025, seed=751)
    s = sp.sigma(torch.from_numpy(C).cuda())
    assert tb.tbsci_hbm_used(ctx.handle) == need
    rows = _rows(sp.ndet, 6)
    _check(s.cpu().numpy(), osp, h, eri, C, rows)
    _check(full.cpu().numpy(), osp, h, eri, C, rows)
    sp.close()
    ctx.close()


@pytest.mark.parametrize("la,lb,k", [(1040, 1030, 1), (1040, 1030, 3), (4000, 4000, 200), (4100, 4100, 200)])
def test_towering_elements(tb, ctx, la, lb, k):
    """k elements ten thousand times the rest, in one row, one column and linked rows: more than
    256 times the root mean square, so kept out of the digits (the last case: past 2^24
    determinants, all SIMT). Rows linked to them and rows that are not agree with the oracle."""
    import torch
    sp, osp, h, eri = _space(tb, ctx, 16, 8, 8, la, lb, seed=771)
    rng = np.random.default_rng(k)
    C = 1e-4 * rng.standard_normal((1, sp.la, sp.lb))
    at = [(5, 7), (5, 8), (6, 7)][:k] + [(int(a), int(b)) for a, b in zip(rng.choice(sp.la, k), rng.choice(sp.lb, k))][3:]
    for a, b in at:
        C[0, a, b] = rng.choice([-1.0, 1.0])
    assert np.abs(C).max() > 256 * np.sqrt((C ** 2).mean())
    Ct = torch.from_numpy(C).cuda()
    s = sp.sigma(Ct)
    assert torch.equal(s, sp.sigma(Ct))
    near = [a * sp.lb + j for a, b in at[:2] for j in range(0, sp.lb, 29)] + [i * sp.lb + b for a, b in at[:2] for i in range(0, sp.la, 29)]
    rows = np.unique(np.concatenate([_rows(sp.ndet, 9), near, [a * sp.lb + b for a, b in at]]))
    _check(s.cpu().numpy(), osp, h, eri, C, rows)
    sp.close()


@pytest.mark.parametrize("kind", ["f64", "f32", "tf32", "pruned"])
def test_tables_make_room(tb, kind):
    """What a sigma keeps to be faster (digit tables, planes, class lists) gives way to what a
    later call cannot do without: under a budget that holds the space and the vectors of that
    call alone, the call runs, and the sigma after it agrees with the one before."""
    import torch

    def make(budget):
        ctx = tb.Context(0, hbm_budget=budget)
        sp, _, h, eri = _space(tb, ctx, 13, 6, 6, 640, 630, seed=781)
        pr = None
        if kind == "pruned":
            a, b = sp.strings()
            keep = (np.bitwise_count(a >> np.uint64(6)).astype(int)[:, None] + np.bitwise_count(b >> np.uint64(6))) <= 6
            pr = sp.prune(np.concatenate([[0], np.cumsum(keep.sum(1))]).astype(np.int64), np.nonzero(keep)[1].astype(np.int32))
        return ctx, sp, pr
    ctx, sp, pr = make(0)
    need = tb.tbsci_hbm_used(ctx.handle)
    nvec = 24  # the host call's buffers: 155 MB, more than any of the tables
    H = np.random.default_rng(9).standard_normal((nvec, sp.la, sp.lb))
    want = sp.sigma_host(H)
    if pr:
        pr.close()
    sp.close()
    ctx.close()
    extra = 1 << 16
    while pr:  # the space alone: under the smallest budget that it fits, there is no room for its lists
        try:
            ctx, sp, small = make(need // 2 + extra)
        except tb.B.TbsciError:
            extra += extra // 4
            continue
        need = tb.tbsci_hbm_used(ctx.handle)
        small.close()
        sp.close()
        ctx.close()
        break
    ctx, sp, pr = make(need + 2 * H.nbytes)
    before = tb.tbsci_hbm_used(ctx.handle)
    assert (before > need) == (kind == "pruned")
    dt = {"f64": (torch.float64, None), "pruned": (torch.float64, None), "f32": (torch.float32, None),
          "tf32": (torch.float32, tb.TBSCI_F32_TC_TF32)}[kind]
    c = torch.randn((1, pr.ndet) if pr else (1, sp.la, sp.lb), dtype=dt[0], device="cuda")
    sigma = (lambda: pr.sigma(c)) if pr else (lambda: sp.sigma(c, dtype=dt[1]))
    first = sigma()
    assert tb.tbsci_hbm_used(ctx.handle) > need
    got = sp.sigma_host(H)
    assert np.abs(got - want).max() <= 1e-11 * np.abs(want).max()
    again = sigma()
    assert torch.linalg.vector_norm(again - first) <= (1e-13 if dt[0] == torch.float64 else 2e-6) * torch.linalg.vector_norm(first)
    if pr:
        pr.close()
    sp.close()
    assert tb.tbsci_hbm_used(ctx.handle) <= 2 * H.nbytes  # the host call's buffers, which the context keeps
    ctx.close()


@pytest.mark.parametrize("dtype", ["f64", "f32"])
def test_failed_allocation_leaves_nothing_behind(tb, dtype):
    """A host call with more vectors than the device holds returns ENOMEM, after the tables were
    taken back for it in vain. The next sigma makes them again (the same kernels, the same
    bits), and so does the first one of a space prepared then."""
    import torch
    ctx = tb.Context(0)
    C = np.random.default_rng(15).standard_normal((1, 640, 630))
    c = torch.from_numpy(C).to(torch.float64 if dtype == "f64" else torch.float32).cuda()
    sp, _, _, _ = _space(tb, ctx, 13, 6, 6, 640, 630, seed=793)
    want = sp.sigma(c)
    torch.cuda.synchronize()
    with_tables = tb.tbsci_hbm_used(ctx.handle)
    huge = (1 << 41) // (16 * sp.ndet)  # 2 TB of vectors: refused before any is read
    out = np.empty(1)
    for _ in range(2):
        assert tb.B.load().tbsci_sigma_host(ctx.handle, sp.ham, sp.ta, sp.tb, tb.B._ptr(C), tb.B._ptr(out), huge) == tb.TBSCI_ENOMEM
        assert torch.equal(sp.sigma(c), want)
        assert tb.tbsci_hbm_used(ctx.handle) == with_tables
        torch.cuda.synchronize()
        sp.close()
        sp, _, _, _ = _space(tb, ctx, 13, 6, 6, 640, 630, seed=793)  # not evaluated before the second turn's call
    sp.close()
    ctx.close()


def test_tables_of_an_ended_context(tb):
    """A space that outlives its context keeps its tables out of what another context's failed
    allocation takes back."""
    import torch
    gone = tb.Context(0)
    sp, _, _, _ = _space(tb, gone, 13, 6, 6, 640, 630, seed=791)
    sp.sigma(torch.randn((1, sp.la, sp.lb), dtype=torch.float64, device="cuda"))
    torch.cuda.synchronize()
    sp._handles = []  # its handles are not used again
    gone.close()
    ctx = tb.Context(0)
    sp, osp, h, eri = _space(tb, ctx, 13, 6, 6, 640, 630, seed=792)
    C = np.random.default_rng(14).standard_normal((1, sp.la, sp.lb))
    c = torch.from_numpy(C).cuda()
    want = sp.sigma(c)
    torch.cuda.synchronize()
    out = np.empty(1)
    huge = (1 << 41) // (16 * sp.ndet)  # 2 TB of vectors, refused before any is read
    assert tb.B.load().tbsci_sigma_host(ctx.handle, sp.ham, sp.ta, sp.tb, tb.B._ptr(C), tb.B._ptr(out), huge) == tb.TBSCI_ENOMEM
    assert torch.equal(sp.sigma(c), want)  # the tables are made again
    sp.close()
    ctx.close()
