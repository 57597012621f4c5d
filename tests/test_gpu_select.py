"""Bitstring selection loop (Sec. III.B) and coefficient distributions (Fig. 3):
GPU string weights, weight thresholds and histograms against the oracle's
plain definitions on the same vectors, and a self-contained selection loop
(solve, weigh, select, solve again) whose energies approach the full-space
energy from above as the threshold is lowered."""
import numpy as np
import pytest

import oracle
from tbsci_inputs import selected_strings, synth_hamiltonian

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def tb():
    import paper_2503_10335_gb300 as tb
    return tb


@pytest.fixture(scope="module")
def ctx(tb):
    c = tb.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("n,na,nb,acnt,bcnt", [(8, 4, 4, None, None), (10, 5, 5, 120, 257), (12, 4, 6, None, 200)])
def test_string_weights_and_selection_match_the_oracle(tb, ctx, n, na, nb, acnt, bcnt):
    import torch
    h, eri, _ = synth_hamiltonian(n, seed=800 + n)
    asel = None if acnt is None else selected_strings(n, na, acnt, 801 + n)
    bsel = None if bcnt is None else selected_strings(n, nb, bcnt, 802 + n)
    sp = tb.Space(ctx, n, na, nb, h, eri, alpha=asel, beta=bsel)
    osp = oracle.make_space(n, na, nb, asel, bsel)
    rng = np.random.default_rng(n)
    C = rng.standard_normal((sp.la, sp.lb)) * 10.0 ** rng.uniform(-4, 0, (sp.la, sp.lb))
    Cd = torch.from_numpy(C).cuda()
    wa, wb = sp.string_weights(Cd)
    ra, rb = oracle.string_weights(C, sp.la, sp.lb)
    assert np.max(np.abs(wa - ra)) <= 1e-13 * ra.max() and np.max(np.abs(wb - rb)) <= 1e-13 * rb.max()
    for delta in (0.5, 0.05, 1e-3, 0.0):
        ka, kb = sp.select_by_weight(Cd, delta)
        for w, ref_w, strings, kept in ((ra, ra, osp.sa, ka), (rb, rb, osp.sb, kb)):
            want = set(int(x) for x in strings[oracle.select_by_weight(ref_w, delta)])
            got = set(int(x) for x in kept)
            thr = delta * ref_w.max()
            # strings whose weight is within rounding of the threshold may go either way
            border = set(int(strings[i]) for i in np.nonzero(np.abs(ref_w - thr) <= 1e-12 * max(thr, 1e-300))[0])
            assert (got ^ want) <= border
            assert np.all(np.diff(kept.astype(np.int64)) > 0)
    sp.close()


def test_coefficient_histogram_exact_counts(tb, ctx):
    import torch
    rng = np.random.default_rng(3)
    x = rng.standard_normal(1_000_003) * 10.0 ** rng.uniform(-9, 0, 1_000_003)
    x[:7] = 0.0
    c_hf = 0.7
    edges = (10.0 ** np.arange(-9, 1)) * c_hf
    got = tb.tbsci_coefficient_histogram(ctx.handle, torch.from_numpy(x).cuda(), edges)
    assert np.array_equal(got, oracle.coefficient_histogram(x, edges))
    assert got.sum() == len(x)
    with pytest.raises(tb.B.TbsciError):
        tb.tbsci_coefficient_histogram(ctx.handle, torch.from_numpy(x).cuda(), edges[::-1].copy())


def test_selection_loop_is_variational_and_matches_the_oracle(tb, ctx):
    """Solve the full norb-10 space (252 x 252 strings), select strings by weight
    at decreasing delta, solve each selected TPB space again: the energies fall
    monotonically towards the full-space energy and never below it, and each
    equals the oracle's solve of the same selected space. The Hamiltonian uses
    the recipe's two-electron scale 0.1: at the default 0.3 the ground state
    spreads its weight evenly over the strings and no threshold selects any."""
    import torch
    n, N = 10, 5
    h, eri, _ = synth_hamiltonian(n, seed=810, scale=0.1)
    full = tb.Space(ctx, n, N, N, h, eri)
    e_full, info, X = full.davidson(1, want_vectors=True)
    assert info["converged"]
    c0 = X[0].contiguous()
    last = None
    for delta in (1e-1, 1e-2, 1e-3):
        ka, kb = full.select_by_weight(c0, delta)
        sub = tb.Space(ctx, n, N, N, h, eri, alpha=ka, beta=kb)
        e_sub, i_sub = sub.davidson(1)
        assert i_sub["converged"]
        assert e_sub[0] >= e_full[0] - 1e-10
        if last is not None:
            assert e_sub[0] <= last + 1e-10
        last = e_sub[0]
        osp = oracle.make_space(n, N, N, ka, kb)
        assert osp.ndet < full.ndet
        e_ref = oracle.solve(osp, h, eri, 0.0, 1)[0][0]
        assert abs(e_sub[0] - e_ref) < 1e-8, (delta, e_sub, e_ref)
        sub.close()
    # the coefficient distribution of the full solution, relative to the largest coefficient
    ratios, counts = full.coefficient_histogram(c0, float(torch.max(torch.abs(c0))), lo=-10, hi=0)
    assert counts.sum() == full.ndet and counts[-1] == 1  # only c_HF itself has |c / c_HF| >= 1
    full.close()


def test_selection_argument_errors(tb, ctx):
    import torch
    h, eri, _ = synth_hamiltonian(6, seed=5)
    sp = tb.Space(ctx, 6, 3, 3, h, eri)
    z = torch.zeros((sp.la, sp.lb), dtype=torch.float64, device="cuda")
    for call in (lambda: sp.string_weights(z), lambda: sp.select_by_weight(z, 0.1),
                 lambda: sp.select_by_weight(torch.ones_like(z), -1.0)):
        with pytest.raises(tb.B.TbsciError) as err:
            call()
        assert err.value.status == tb.TBSCI_EINVAL
    sp.close()


@pytest.mark.parametrize("edges", [[0.5], [-1.0, -0.0, 1e-300, 1.0], [1.0, 2.0, 3.0], list(10.0 ** np.linspace(-12, 0, 255)),
                                   list(10.0 ** np.linspace(-12, 0, 256)), [1.0, np.inf]])
@pytest.mark.parametrize("n", [1, 255, 1025, 300001])
def test_histogram_bins_at_their_edges(tb, ctx, edges, n):
    """Values equal to an edge, one unit below it, zeros, infinities and NaN: the bin
    of x is the number of edges at or below |x| (none for NaN)."""
    import torch
    e = np.array(edges)
    r = np.random.default_rng(n)
    special = np.concatenate([np.abs(e), np.nextafter(np.abs(e), 0), [0.0, np.inf, np.nan, 5e-324, 1.7e308]])
    x = np.where(r.random(n) < 0.5, r.choice(special, n), 10.0 ** r.uniform(-14, 2, n)) * r.choice([-1.0, 1.0], n)
    got = tb.tbsci_coefficient_histogram(ctx.handle, torch.from_numpy(x).cuda(), e)
    a = np.abs(x)
    want = np.bincount(np.where(np.isnan(a), 0, np.searchsorted(e, a, side="right")), minlength=len(e) + 1)
    assert np.array_equal(got, want)
