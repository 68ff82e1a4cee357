"""GPU-vs-oracle parity, through the C ABI (via the thin binding), element by element."""
import copy
import os
import re

import numpy as np
import pytest
import torch

import __graft_entry__ as entry
import paper_2605_14292_b200 as akv
from oracle import alpha_oracle as O
from oracle import c_oracle as CO
from paper_2605_14292_b200 import synth

import akv_check as chk
import akv_split

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    entry.build()
    akv.load_library()


def dev(x):
    return akv.to_device(x, "cuda")


def tiled(ev, times):
    """The same events `times` over, as one call of more sequences."""
    big = copy.copy(ev)
    for name in ("K", "V", "pos", "p_ref"):
        x = getattr(ev, name)
        setattr(big, name, np.tile(x, (times,) + (1,) * (x.ndim - 1)))
    return big


def beyond_one_and_three_per_sm(events):
    """How often a call of so many events has to be repeated for more events than SMs, and for more than three per SM."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    return sms // events + 1, 3 * sms // events + 1


def same_bits(few, many, keys=None):
    """The results of a call against those of its events many times over."""
    for k in keys or few:
        x, y = np.ascontiguousarray(few[k]), np.ascontiguousarray(many[k])
        same = (y.view(np.uint8).reshape(-1, x.nbytes) == x.view(np.uint8).reshape(1, -1)).all(1)
        assert same.all(), f"{k}: {int((~same).sum())} of {same.size} copies differ"


def takes_forms(ev):
    """Shapes whose kernel (event_pool_kernel) has forms for one, three and four events per SM."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    return ev.dtype == synth.BF16 and ev.shape[-1] == 128 and 128 < ev.shape[3] <= 256 and 64 < ev.budget <= 128 and ev.n_events <= sms


def run_fused_once(ev, lam=None, flags=0, n_cand=None, p_ref=True, W=None, budgets=None):
    lam = ev.lam if lam is None else lam
    K, V, pos, q = dev(ev.K), dev(ev.V), dev(ev.pos), dev(ev.qstat)
    pref = dev(ev.p_ref) if p_ref else None
    nc = None if n_cand is None else dev(np.asarray(n_cand, dtype=np.int32))
    hb = None if budgets is None else dev(np.ascontiguousarray(budgets, dtype=np.int32))
    opts = akv.Options(lam=lam, eps=ev.eps, rope_base=ev.rope_base, future_window=W or ev.future_window, flags=flags,
                       head_budgets=hb)
    sel = akv.alpha_compress_event(K, V, pos, q, ev.budget, opts, p_ref=pref, n_cand=nc, want_scores=True)
    torch.cuda.synchronize()
    return dict(K=akv.to_host_bits(K), V=akv.to_host_bits(V), pos=pos.cpu().numpy(), idx=sel.idx_sorted.cpu().numpy(),
                order=sel.pick_order.cpu().numpy(), gain=sel.pick_gain.cpu().numpy(), scores=sel.scores.cpu().numpy(),
                n_kept=sel.n_kept.cpu().numpy(), status=sel.status.cpu().numpy())


def run_fused(ev, lam=None, flags=0, n_cand=None, p_ref=True, W=None, budgets=None):
    """The fused call on a copy of the events, as host arrays. Where the kernel's form depends on the number of events the call is also made with
    the same events so often that the other forms take them: the results are the same to the bit."""
    g = run_fused_once(ev, lam, flags, n_cand, p_ref, W, budgets)
    if takes_forms(ev):
        written = ("K", "V", "pos", "status") if flags & akv.FLAG_TEST_STARVE_WAIT else None
        for times in beyond_one_and_three_per_sm(ev.n_events):
            same_bits(g, run_fused_once(tiled(ev, times), lam, flags, None if n_cand is None else list(n_cand) * times, p_ref, W, budgets), written)
    return g


def check_all(ev, g, lam, events=None, n_cand=None, p_ref=True, W=None, threads=8, budgets=None):
    B, L, H, N, d = ev.shape
    W = W or ev.future_window
    E = B * L * H
    log = []
    ref = None
    if n_cand is None and p_ref and events is None:
        ref = CO.event_batch(ev.K, ev.V, ev.pos, ev.qstat, ev.p_ref, ev.budget, lam, W=W, base=ev.rope_base,
                             eps=ev.eps, threads=threads, want_rows=False, budgets=budgets)
    todo = range(E) if events is None else events
    for e in todo:
        b, l, h = e // (L * H), (e // H) % L, e % H
        n = N if n_cand is None else int(n_cand[b])
        k_e = ev.budget if budgets is None else int(budgets[l][h])
        chk.check_event(ev.K[b, l, h], ev.V[b, l, h], ev.pos[b, l, h], ev.qstat[l, h],
                        int(ev.p_ref[b]) if p_ref else None, k_e, lam,
                        g["scores"][b, l, h], g["order"][b, l, h], g["idx"][b, l, h],
                        g["K"][b, l, h], g["V"][b, l, h], g["pos"][b, l, h], W=W, base=ev.rope_base, eps=ev.eps,
                        ref_scores=None if ref is None else ref["scores"][b, l, h],
                        ref_order=None if ref is None else ref["order"][b, l, h], n=n, log=log)
        assert g["n_kept"][b, l, h] == min(k_e, n)
        assert g["status"][b, l, h] == (2 if n < k_e else 0)
    return log


# ------------------------------------------------------------------ small shapes: several tiles, ragged tails
@pytest.mark.parametrize("dtype", [synth.BF16, synth.F32])
@pytest.mark.parametrize("N,d,budget", [(100, 128, 37), (77, 64, 77), (192, 128, 64), (33, 16, 5), (130, 256, 40),
                                        (50, 8, 20), (96, 40, 31)])
@pytest.mark.parametrize("lam", [0.0, 0.5, 1.5])
def test_fused_event_small(dtype, N, d, budget, lam):
    ev = synth.make_c3(seed=N + d, B=2, L=2, H=3, N=N, budget=budget) if d == 128 else \
        synth.make_plain(2, 2, 3, N, d, budget, lam, dtype=dtype, seed=N + d)
    if d == 128 and dtype == synth.F32:
        ev = synth.make_plain(2, 2, 3, N, d, budget, lam, dtype=dtype, seed=N + d)
    g = run_fused(ev, lam=lam)
    check_all(ev, g, lam)


def test_lambda0_greedy_loop_equals_fast_path_equals_topk():
    ev = synth.make_plain(2, 3, 2, 150, 128, 50, 0.0, dtype=synth.BF16, seed=3)
    fast = run_fused(ev, lam=0.0)
    loop = run_fused(ev, lam=0.0, flags=akv.FLAG_FORCE_GREEDY)
    assert np.array_equal(fast["order"], loop["order"]) and np.array_equal(fast["idx"], loop["idx"])
    assert np.array_equal(fast["K"][..., :50, :], loop["K"][..., :50, :])
    # top-k of the GPU's own scores, ties to the lower index
    for b in range(2):
        for l in range(3):
            for h in range(2):
                s = fast["scores"][b, l, h].astype(np.float64)
                assert fast["order"][b, l, h].tolist() == O.topk_indices(s, 50).tolist()


def test_ragged_candidate_counts_and_short_events():
    ev = synth.make_plain(4, 2, 2, 120, 128, 40, 0.5, dtype=synth.BF16, seed=9)
    n_cand = [120, 41, 40, 17]          # last one is below the budget: keep all, status 2
    g = run_fused(ev, n_cand=n_cand)
    check_all(ev, g, 0.5, n_cand=n_cand)
    # rows beyond n_cand were never read as candidates: no index >= n_cand
    for b, n in enumerate(n_cand):
        kept = min(40, n)
        assert g["idx"][b, :, :, :kept].max() < n


def test_default_reference_position_and_future_window():
    ev = synth.make_plain(2, 2, 2, 90, 128, 30, 0.5, dtype=synth.BF16, seed=12)
    ev.pos[:] = (np.sort(np.random.default_rng(1).choice(5000, size=90, replace=False))).astype(np.int32)
    g = run_fused(ev, p_ref=False, W=4)
    check_all(ev, g, 0.5, p_ref=False, W=4)


def test_large_positions_keep_score_accuracy():
    ev = synth.make_plain(1, 2, 2, 64, 128, 16, 0.5, dtype=synth.BF16, seed=13)
    ev.pos[:] = (1_000_000 + np.arange(64) * 997).astype(np.int32)
    ev.p_ref[:] = 1_100_000
    g = run_fused(ev)
    check_all(ev, g, 0.5)


def test_repeat_runs_are_bit_identical():
    ev = synth.make_c3(seed=4, B=2, L=2, H=2, N=192, budget=64)
    a, b = run_fused(ev), run_fused(ev)
    for k in ("K", "V", "pos", "idx", "order", "scores", "gain"):
        assert np.array_equal(a[k], b[k]), k


def test_nonfinite_scores_are_flagged_and_never_preferred():
    ev = synth.make_plain(1, 1, 2, 64, 128, 20, 0.5, dtype=synth.F32, seed=14)
    ev.K[0, 0, 0, 5, 3] = np.inf
    ev.K[0, 0, 0, 9, 100] = np.nan
    g = run_fused(ev)
    assert g["status"][0, 0, 0] == 1 and g["status"][0, 0, 1] == 0
    assert not ({5, 9} & set(g["idx"][0, 0, 0].tolist()))
    assert len(set(g["idx"][0, 0, 0].tolist())) == 20


@pytest.mark.parametrize("d", [128, 256])
def test_resident_kernel_norms_are_summed_in_a_tree(d):
    """The second pick's value is -lambda x_0 r, with r the reciprocal norm of its row x: the first row is a unit vector, so the
    dot product is exact. Errors of r: half of the squared norm's, and one rounding each for root, division and product. In
    fp32 emulation the whole is 4.8e-8 (d = 128) and 5.0e-8 (d = 256) root mean square for sums of eight squares in a tree,
    9.3e-8 and 1.2e-7 for one chain of d squares."""
    ev = synth.make_plain(8, 32, 8, 2, d, 2, 1.0, dtype=synth.F32, seed=d)
    ev.K[...] = 0
    ev.V[..., 0, :] = 0
    ev.V[..., 0, 0] = 1
    ev.V[..., 1, 0] = np.abs(ev.V[..., 1, 0]) + 0.5
    x = ev.V[..., 1, :].astype(np.float64)
    want = -x[..., 0] / np.sqrt((x * x).sum(-1))
    g = run_fused(ev)
    assert np.all(g["order"] == [0, 1])
    err = g["gain"][..., 1] / want - 1
    assert np.sqrt(np.mean(err ** 2)) < 7e-8


@pytest.mark.parametrize("dtype,d,N,budget,lam", [(synth.BF16, 64, 256, 128, 0.5), (synth.BF16, 64, 256, 128, 2.0), (synth.BF16, 96, 192, 64, 2.0),
                                                  (synth.F32, 64, 256, 128, 2.0), (synth.F32, 40, 192, 64, 2.0), (synth.F32, 64, 430, 64, 4.0),
                                                  (synth.BF16, 64, 700, 300, 1.0), (synth.BF16, 16, 400, 70, 1.0)])
@pytest.mark.parametrize("close", [False, True])
def test_resident_kernel_with_a_pool_larger_than_its_triangle(dtype, d, N, budget, lam, close):
    """Rounds of active sets, their state beside the tiles or (N = 430) at the head of the K tile; a set too small for them
    (d = 16, N = 400) leaves the event to the CTA-wide loop. close: scores that differ in their last bits, one event's not at all."""
    for shape in ((2, 1, 2), (10, 4, 4)):        # one CTA per SM, and two
        ev = synth.make_plain(*shape, N, d, budget, lam, dtype=dtype, seed=N + d)
        if close:
            ev.qstat *= np.float32(1e-6)
            ev.K[0, 0, 0] = ev.K[0, 0, 0, :1]      # (not zero: the check's relative errors need a scale)
            ev.pos[0, 0, 0] = 5
            ev.V[..., N - N // 4:, :] = ev.V[..., :N // 4, :]
        g = run_fused(ev, n_cand=[N, N - 5] + [N] * (shape[0] - 2))
        check_all(ev, g, lam, n_cand=[N, N - 5] + [N] * (shape[0] - 2), events=range(4))


@pytest.mark.parametrize("mode", ["flat", "layer"])
def test_resident_kernel_rounds_on_shared_signatures(mode):
    ev = synth.make_plain(2, 2, 2, 256, 64, 128, 1.5, dtype=synth.BF16, seed=17)
    V = dev(ev.V)
    sig = akv.alpha_signature_flat(V) if mode == "flat" else akv.alpha_signature_layer(V)
    K, pos = dev(ev.K), dev(ev.pos)
    opts = akv.Options(lam=1.5, sig_mode=akv.SIG_FLAT if mode == "flat" else akv.SIG_PER_LAYER)
    sel = akv.alpha_compress_event(K, V, pos, dev(ev.qstat), 128, opts, p_ref=dev(ev.p_ref), flat_sig=sig, want_scores=True)
    torch.cuda.synchronize()
    Kn, Vn, pn = akv.to_host_bits(K), akv.to_host_bits(V), pos.cpu().numpy()
    for b in range(2):
        for l in range(2):
            ref = O.signatures_flat(ev.V[b]) if mode == "flat" else O.signatures_per_layer(ev.V[b, l])
            for h in range(2):
                chk.check_event(ev.K[b, l, h], ev.V[b, l, h], ev.pos[b, l, h], ev.qstat[l, h], int(ev.p_ref[b]), 128, 1.5,
                                sel.scores[b, l, h].cpu().numpy(), sel.pick_order[b, l, h].cpu().numpy(),
                                sel.idx_sorted[b, l, h].cpu().numpy(), Kn[b, l, h], Vn[b, l, h], pn[b, l, h], sig=ref)


# ------------------------------------------------------------------ stand-alone entry points
@pytest.mark.parametrize("dtype", [synth.BF16, synth.F32])
def test_score_select_compact_chain_equals_fused(dtype):
    ev = synth.make_c3(seed=21, B=2, L=2, H=2, N=160, budget=48) if dtype == synth.BF16 else \
        synth.make_plain(2, 2, 2, 160, 128, 48, 0.5, dtype=dtype, seed=21)
    fused = run_fused(ev)
    K, V, pos, q, pref = dev(ev.K), dev(ev.V), dev(ev.pos), dev(ev.qstat), dev(ev.p_ref)
    opts = akv.Options(lam=ev.lam)
    status = torch.full((2, 2, 2), -7, dtype=torch.int32, device="cuda")
    s = akv.alpha_score(K, q, pos=pos, p_ref=pref, opts=opts, status=status)
    # the stand-alone scorer and the fused kernel may round differently in the last place
    assert np.max(np.abs(s.cpu().numpy() - fused["scores"])) < 2e-6
    # fed the very same scores, the stand-alone selection must reproduce the fused one's picks
    sel = akv.alpha_select(dev(fused["scores"]), V, ev.budget, opts)
    akv.kv_compact(K, V, pos, sel.idx_sorted)
    torch.cuda.synchronize()
    assert np.array_equal(sel.pick_order.cpu().numpy(), fused["order"])
    assert np.array_equal(sel.idx_sorted.cpu().numpy(), fused["idx"])
    # (the gains themselves may differ in the last place: the two routes sum a row's products in different orders)
    assert np.max(np.abs(sel.pick_gain.cpu().numpy() - fused["gain"])) < 1e-6
    assert np.array_equal(akv.to_host_bits(K)[..., :48, :], fused["K"][..., :48, :])
    assert np.array_equal(akv.to_host_bits(V)[..., :48, :], fused["V"][..., :48, :])
    assert np.array_equal(pos.cpu().numpy()[..., :48], fused["pos"][..., :48])
    assert int(status.abs().max()) == 0


@pytest.mark.parametrize("N,page", [(5, 4), (256, 64), (257, 16), (1000, 128)])
def test_scores_of_a_paged_cache_are_the_dense_ones(N, page):
    """bf16, d = 128: the score kernel's two layouts, with a block table in no order, to the bit."""
    ev = synth.make_plain(2, 2, 3, N, 128, 2, 0.5, dtype=synth.BF16, seed=N)
    K, pos, q, pref = dev(ev.K), dev(ev.pos), dev(ev.qstat), dev(ev.p_ref)
    pps = -(-N // page)
    table = torch.randperm(2 * pps, device="cuda").to(torch.int32).view(2, pps)
    rows = torch.zeros((2, 2, 3, pps * page, 128), dtype=torch.bfloat16, device="cuda")
    rows[..., :N, :] = K
    pool = torch.zeros((2, 2 * pps, 3, page, 128), dtype=torch.bfloat16, device="cuda")
    pool[:, table.long().flatten()] = rows.view(2, 2, 3, pps, page, 128).permute(1, 0, 3, 2, 4, 5).reshape(2, 2 * pps, 3, page, 128)
    dense = akv.alpha_score(K, q, pos=pos, p_ref=pref)
    assert torch.equal(dense, akv.alpha_score(pool, q, pos=pos, p_ref=pref, layout=akv.Layout.paged(pool, table, N)))
    ref = O.triattention_score(ev.K[1, 1, 2], ev.pos[1, 1, 2], ev.qstat[1, 2], int(ev.p_ref[1]), 1, 10000.0)
    chk.check_scores(dense[1, 1, 2].cpu().numpy(), ref, chk.score_scale(ev.K[1, 1, 2], ev.qstat[1, 2], 128))


def test_score_only_broadcast_positions_and_rotated_cache():
    ev = synth.make_plain(2, 3, 2, 70, 128, 10, 0.5, dtype=synth.BF16, seed=22)
    K, q = dev(ev.K), dev(ev.qstat)
    pos1 = dev(np.arange(70, dtype=np.int32) * 3)
    s = akv.alpha_score(K, q, pos=pos1, p_ref=dev(np.array([400, 500], dtype=np.int32)),
                        opts=akv.Options(future_window=3)).cpu().numpy()
    s0 = akv.alpha_score(K, q, pos=None).cpu().numpy()
    for b in range(2):
        for l in range(3):
            for h in range(2):
                ref = O.triattention_score(ev.K[b, l, h], np.arange(70) * 3, ev.qstat[l, h], [400, 500][b], 3)
                chk.check_scores(s[b, l, h], ref, chk.score_scale(ev.K[b, l, h], ev.qstat[l, h], 128))
                ref0 = O.triattention_score(ev.K[b, l, h], None, ev.qstat[l, h], None)
                chk.check_scores(s0[b, l, h], ref0, chk.score_scale(ev.K[b, l, h], ev.qstat[l, h], 128))


def test_select_given_scores_matches_oracle_and_duplicate_pair_closed_form():
    P, d = 40, 128
    s, V, leaders = synth.make_duplicate_pairs(P, d, 0.01, seed=2, dtype=synth.BF16)
    lam = float(s[0] - 0.01 - s[2 * (P - 1)]) + 0.05
    sc = torch.tensor(s, dtype=torch.float32, device="cuda").reshape(1, 1, 1, -1).contiguous()
    Vd = dev(V.reshape(1, 1, 1, 2 * P, d))
    for b in (1, 7, P):
        sel = akv.alpha_select(sc, Vd, b, akv.Options(lam=lam))
        assert sel.idx_sorted.cpu().numpy().ravel().tolist() == leaders[:b].tolist()
    top = akv.alpha_select(sc, Vd, 6, akv.Options(lam=0.0)).idx_sorted.cpu().numpy().ravel().tolist()
    assert top == sorted(sorted(range(2 * P), key=lambda i: (-np.float32(s[i]), i))[:6])


def test_compact_in_place_aliasing_and_negative_tail():
    ev = synth.make_plain(2, 2, 2, 64, 128, 20, 0.5, dtype=synth.BF16, seed=23)
    K, V, pos = dev(ev.K), dev(ev.V), dev(ev.pos)
    idx = np.zeros((2, 2, 2, 20), dtype=np.int32)
    idx[...] = np.arange(1, 21)                 # every destination is another row's source
    idx[1, 1, 1] = np.r_[np.arange(5, 64, 4)[:15], -1, -1, -1, -1, -1]
    akv.kv_compact(K, V, pos, dev(idx))
    torch.cuda.synchronize()
    Kn, Vn, pn = akv.to_host_bits(K), akv.to_host_bits(V), pos.cpu().numpy()
    for b in range(2):
        for l in range(2):
            for h in range(2):
                ii = idx[b, l, h]
                ii = ii[ii >= 0]
                assert np.array_equal(Kn[b, l, h, :len(ii)], ev.K[b, l, h][ii])
                assert np.array_equal(Vn[b, l, h, :len(ii)], ev.V[b, l, h][ii])
                assert np.array_equal(pn[b, l, h, :len(ii)], ev.pos[b, l, h][ii])
                assert np.array_equal(Kn[b, l, h, 21:], ev.K[b, l, h, 21:])     # untouched beyond the moved range


def test_flat_signature_eq1_and_selection_with_it():
    ev = synth.make_plain(2, 3, 2, 80, 128, 25, 0.7, dtype=synth.BF16, seed=24)
    V = dev(ev.V)
    sig = akv.alpha_signature_flat(V).cpu().numpy()
    for b in range(2):
        ref = O.signatures_flat(ev.V[b])
        assert np.max(np.abs(sig[b] - ref)) < 2e-7
    K, pos, q, pref = dev(ev.K), dev(ev.pos), dev(ev.qstat), dev(ev.p_ref)
    opts = akv.Options(lam=0.7, sig_mode=akv.SIG_FLAT)
    sel = akv.alpha_compress_event(K, V, pos, q, 25, opts, p_ref=pref, flat_sig=dev(sig), want_scores=True)
    torch.cuda.synchronize()
    Kn, Vn, pn = akv.to_host_bits(K), akv.to_host_bits(V), pos.cpu().numpy()
    for b in range(2):
        ref_sig = O.signatures_flat(ev.V[b])
        for l in range(3):
            for h in range(2):
                chk.check_event(ev.K[b, l, h], ev.V[b, l, h], ev.pos[b, l, h], ev.qstat[l, h], int(ev.p_ref[b]), 25, 0.7,
                                sel.scores[b, l, h].cpu().numpy(), sel.pick_order[b, l, h].cpu().numpy(),
                                sel.idx_sorted[b, l, h].cpu().numpy(), Kn[b, l, h], Vn[b, l, h], pn[b, l, h], sig=ref_sig)


def test_three_launch_path_for_events_that_do_not_fit_on_chip():
    """fp32 with N = 600 exceeds shared memory: score -> select -> compact with scratch scores."""
    ev = synth.make_plain(1, 2, 2, 600, 128, 50, 0.5, dtype=synth.F32, seed=25)
    K, V, pos, q, pref = dev(ev.K), dev(ev.V), dev(ev.pos), dev(ev.qstat), dev(ev.p_ref)
    sel = akv.alpha_compress_event(K, V, pos, q, 50, akv.Options(lam=0.5), p_ref=pref, want_scores=False)
    torch.cuda.synchronize()
    g = dict(K=akv.to_host_bits(K), V=akv.to_host_bits(V), pos=pos.cpu().numpy(), idx=sel.idx_sorted.cpu().numpy(),
             order=sel.pick_order.cpu().numpy(), n_kept=sel.n_kept.cpu().numpy(), status=sel.status.cpu().numpy())
    g["scores"] = akv.alpha_score(dev(ev.K), q, pos=dev(ev.pos), p_ref=pref).cpu().numpy()
    check_all(ev, g, 0.5)


def test_invalid_arguments_launch_nothing():
    ev = synth.make_plain(1, 1, 1, 32, 128, 8, 0.5, dtype=synth.BF16, seed=26)
    K, V, pos, q = dev(ev.K), dev(ev.V), dev(ev.pos), dev(ev.qstat)
    before = akv.launch_count()
    with pytest.raises(akv.AkvError) as e:
        akv.alpha_compress_event(K, V, pos, q, 33)
    assert e.value.code == 3
    with pytest.raises(akv.AkvError) as e:
        akv.alpha_compress_event(K, V, pos, q, 8, akv.Options(lam=-1.0))
    assert e.value.code == 1
    with pytest.raises(akv.AkvError) as e:
        akv.alpha_compress_event(K.view(torch.int16)[..., 1:].view(torch.bfloat16) if False else K, V, pos, q, 8,
                                 akv.Options(sig_mode=akv.SIG_FLAT))
    assert e.value.code == 1
    Kodd = torch.empty(32 * 128 + 8, dtype=torch.bfloat16, device="cuda")[4:4 + 32 * 128].view(1, 1, 1, 32, 128)
    with pytest.raises(akv.AkvError) as e:
        akv.alpha_score(Kodd, q)
    assert e.value.code == 4
    assert akv.launch_count() == before
    assert np.array_equal(akv.to_host_bits(K), ev.K)


# ------------------------------------------------------------------ events longer than the 128-row K tile
@pytest.mark.parametrize("N,budget", [(129, 48), (144, 64), (250, 33), (256, 64)])
def test_k_rows_beyond_the_tile_arrive_in_freed_slots(N, budget):
    """bf16, d = 128, budget <= 64: the kernel holds 128 K rows at a time; rows from 128 on are scored from
    the slots of the first rows. Ragged counts put the boundary inside, at and just after the tile."""
    ev = synth.make_c3(seed=N, B=4, L=2, H=2, N=N, budget=budget)
    g = run_fused(ev)
    check_all(ev, g, ev.lam)
    n_cand = [N, min(N, 129), 128, min(N, 131)]
    g = run_fused(ev, n_cand=n_cand)
    check_all(ev, g, ev.lam, n_cand=n_cand)


def in_pairs(ev, seed):
    """Rows in pairs of one value row, their keys and positions equal in every second pair (equal scores): the best candidate
    raises the maximum of the next one again and again. The first third at irregular positions, like kept rows."""
    rng = np.random.default_rng(seed)
    B, L, H, N, _ = ev.shape
    gaps = rng.integers(1, 30, size=(B, L, H, N // 3)).cumsum(-1)
    ev.pos[..., :N // 3] = gaps
    ev.pos[..., N // 3:] += 30 * N
    ev.p_ref[:] = 32 * N
    odd = np.arange(1, N, 2)
    ev.V[..., odd, :] = ev.V[..., odd - 1, :]
    ev.K[..., odd[::2], :] = ev.K[..., odd[::2] - 1, :]
    ev.pos[..., odd[::2]] = ev.pos[..., odd[::2] - 1]
    return ev


@pytest.mark.parametrize("N,budget,lam", [(129, 20, 0.5), (144, 64, 1.0), (160, 128, 0.5), (192, 64, 0.0), (250, 33, 1.0), (255, 65, 0.0),
                                          (256, 64, 0.5), (256, 128, 0.5), (256, 128, 2.0), (192, 70, 0.5), (193, 71, 1.0), (256, 96, 0.5)])
def test_events_with_an_sm_each_and_several_to_an_sm(N, budget, lam):
    """bf16, d = 128, budgets beyond 64: calls of no more events than SMs take the form of eight warps, others those of four, three or four (more
    than three per SM, budgets of at most 96) of them to an SM; smaller budgets one kernel. All against the oracle, with all candidates, ragged
    counts and when their waits run out."""
    few = in_pairs(synth.make_plain(2, 1, 3, N, 128, budget, lam, dtype=synth.BF16, seed=N + budget), N)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    for times in (1, sms // 6 + 1, 3 * sms // 6 + 1):
        ev, events = few, range(6)
        if times > 1:
            ev, events = synth.make_plain(2 * times, 1, 3, 1, 128, 1, lam, dtype=synth.BF16, seed=0), (0, 4, 6 * times - 1)
            ev.qstat, ev.budget = few.qstat, budget
            for name in ("K", "V", "pos", "p_ref"):
                setattr(ev, name, np.tile(getattr(few, name), (times,) + (1,) * (getattr(few, name).ndim - 1)))
        check_all(ev, run_fused(ev), lam, events=events)
        n_cand = [N - 1, N // 2 + 1] * (len(ev.p_ref) // 2)
        check_all(ev, run_fused(ev, n_cand=n_cand), lam, events=events, n_cand=n_cand)
        g = run_fused(ev, flags=akv.FLAG_TEST_STARVE_WAIT)
        assert np.all(g["status"] == 3) and np.array_equal(g["K"], ev.K) and np.array_equal(g["V"], ev.V) and np.array_equal(g["pos"], ev.pos)


@pytest.mark.parametrize("N,budget,lam", [(100, 40, 0.5), (128, 128, 0.5), (129, 20, 0.5), (160, 64, 1.0), (192, 64, 0.0), (192, 64, 0.5), (256, 64, 2.0),
                                          (129, 100, 0.5), (144, 70, 1.0), (176, 96, 0.5), (193, 90, 0.5), (208, 128, 1.0), (224, 96, 1.0), (225, 65, 0.0),
                                          (240, 80, 0.5), (241, 96, 2.0), (256, 96, 1.0), (256, 128, 0.0), (256, 128, 0.5), (256, 128, 2.0)])
@pytest.mark.parametrize("regular", [True, False])
def test_an_event_has_the_same_bits_in_every_call(N, budget, lam, regular):
    """bf16, d = 128: scores, picks, gains and kept rows of an event do not depend on how many other events the call has."""
    ev = synth.make_c3(seed=N, B=2, L=1, H=3, N=N, budget=budget)
    if not regular:
        ev = in_pairs(ev, N)
    few = run_fused_once(ev, lam=lam)
    check_all(ev, few, lam)
    for times in beyond_one_and_three_per_sm(6):
        same_bits(few, run_fused_once(tiled(ev, times), lam=lam))
    for n_cand in ([N, N // 2], [N - 17, N - 1]):
        few = run_fused_once(ev, lam=lam, n_cand=n_cand)
        for times in beyond_one_and_three_per_sm(6):
            same_bits(few, run_fused_once(tiled(ev, times), lam=lam, n_cand=n_cand * times))


@pytest.mark.parametrize("N,budget,lam", [(100, 40, 0.5), (192, 64, 0.5), (193, 90, 0.25), (256, 128, 0.5), (256, 128, 1.5)])
@pytest.mark.parametrize("twice", [True, False])
def test_an_event_has_the_same_bits_in_every_call_with_a_shared_matrix(N, budget, lam, twice):
    ev = _duplicated_rows(N, lam, B=1, L=2, H=3, N=N // 2 * 2, budget=budget) if twice else synth.make_c3(seed=N, B=1, L=2, H=3, N=N, budget=budget)

    def run(e, page=0):
        K, V, pos, lay = dev(e.K), dev(e.V), dev(e.pos), None
        sig = akv.alpha_signature_flat(V)
        gram = akv.alpha_gram_shared(sig, akv.Layout.dense(V), akv.Options(sig_mode=akv.SIG_FLAT))
        if page:
            B, L, H, n, d = e.shape
            pps = -(-n // page)
            table = torch.randperm(B * pps, device="cuda").to(torch.int32).view(B, pps)
            pools = torch.zeros((2, L, B * pps, H, page, d), dtype=torch.bfloat16, device="cuda")
            for pool, x in zip(pools, (K, V)):
                rows = torch.zeros((B, L, H, pps * page, d), dtype=torch.bfloat16, device="cuda")
                rows[..., :n, :] = x
                pool[:, table.long().flatten()] = rows.view(B, L, H, pps, page, d).permute(1, 0, 3, 2, 4, 5).reshape(L, B * pps, H, page, d)
            K, V, lay = pools[0], pools[1], akv.Layout.paged(pools[0], table, n)
        sel = akv.alpha_compress_event(K, V, pos, dev(e.qstat), budget, akv.Options(lam=lam, sig_mode=akv.SIG_FLAT, shared_gram=gram), p_ref=dev(e.p_ref),
                                       flat_sig=sig, want_scores=True, layout=lay)
        if page:
            K, V = (x[:, table.long().flatten()].view(L, B, pps, H, page, d).permute(1, 0, 3, 2, 4, 5).reshape(B, L, H, pps * page, d)[..., :n, :].contiguous()
                    for x in (K, V))
        return dict(K=akv.to_host_bits(K), V=akv.to_host_bits(V), pos=pos.cpu().numpy(), idx=sel.idx_sorted.cpu().numpy(), order=sel.pick_order.cpu().numpy(),
                    gain=sel.pick_gain.cpu().numpy(), scores=sel.scores.cpu().numpy(), n_kept=sel.n_kept.cpu().numpy(), status=sel.status.cpu().numpy())

    few = run(ev)
    assert few["status"].max() == 0
    for times in beyond_one_and_three_per_sm(6):
        same_bits(few, run(tiled(ev, times)))
        for page in (64, 8):
            same_bits(few, run(tiled(ev, times), page))


@pytest.mark.parametrize("page,N,budget", [(16, 256, 128), (16, 250, 64), (16, 241, 100), (8, 128, 40), (8, 130, 64), (8, 256, 128), (256, 131, 70),
                                           (16, 256, 96), (8, 256, 96), (64, 193, 71), (32, 225, 90), (16, 241, 65)])
def test_pages_on_both_sides_of_those_whose_offsets_are_kept(page, N, budget):
    """Up to sixteen pages of an event have their offsets on chip: one less, as many and one more, in no order, for events with an
    SM each and several to an SM (four, budgets of at most 96: with late K rows from 193 rows on and V rows in registers from 71 kept ones
    on); against the same rows in a dense cache, to the bit."""
    for B in (1, 40, 120):
        ev = synth.make_plain(B, 2, 2, N, 128, budget, 0.5, dtype=synth.BF16, seed=N + page)
        plain = run_fused_once(ev)
        pps = -(-N // page)
        table = torch.randperm(B * pps, device="cuda").to(torch.int32).view(B, pps)
        pools = []
        for x in (dev(ev.K), dev(ev.V)):
            rows = torch.zeros((B, 2, 2, pps * page, 128), dtype=torch.bfloat16, device="cuda")
            rows[..., :N, :] = x
            pool = torch.zeros((2, B * pps, 2, page, 128), dtype=torch.bfloat16, device="cuda")
            pool[:, table.long().flatten()] = rows.view(B, 2, 2, pps, page, 128).permute(1, 0, 3, 2, 4, 5).reshape(2, B * pps, 2, page, 128)
            pools.append(pool)
        pos, lay = dev(ev.pos), akv.Layout.paged(pools[0], table, N)
        sel = akv.alpha_compress_event(pools[0], pools[1], pos, dev(ev.qstat), budget, akv.Options(lam=0.5), p_ref=dev(ev.p_ref), layout=lay)
        assert np.array_equal(sel.pick_order.cpu().numpy(), plain["order"]) and np.array_equal(sel.pick_gain.cpu().numpy(), plain["gain"])
        assert np.array_equal(pos.cpu().numpy(), plain["pos"])
        for pool, name in zip(pools, "KV"):
            rows = pool[:, table.long().flatten()].view(2, B, pps, 2, page, 128).permute(1, 0, 3, 2, 4, 5).reshape(B, 2, 2, pps * page, 128)
            assert np.array_equal(akv.to_host_bits(rows[..., :N, :].contiguous()), plain[name]), name


@pytest.mark.parametrize("N,budget,lam", [(192, 64, 0.5), (193, 71, 0.5), (224, 96, 1.0), (256, 96, 0.5), (256, 128, 0.5), (256, 128, 0.0)])
def test_rows_that_lie_apart_and_selection_alone_in_every_form(N, budget, lam):
    """With an SM for each event, and with three and four of them to an SM: a cache whose rows are 136 elements apart, and alpha_select on scores
    given, as in the fused call on contiguous rows, to the bit."""
    ev = synth.make_c3(seed=N + budget, B=2, L=1, H=3, N=N, budget=budget)
    few = run_fused_once(ev, lam=lam)
    for times in (1,) + beyond_one_and_three_per_sm(6):
        e = tiled(ev, times)
        K, V = (torch.empty(e.shape[:-1] + (136,), dtype=torch.bfloat16, device="cuda")[..., :128].copy_(dev(x)) for x in (e.K, e.V))
        pos, opts = dev(e.pos), akv.Options(lam=lam)
        scores = dev(np.ascontiguousarray(np.tile(few["scores"], (times, 1, 1, 1))))
        sel = akv.alpha_select(scores, V, budget, opts, layout=akv.Layout.dense(V))
        same_bits({k: few[k] for k in ("idx", "order", "gain", "n_kept", "status")},
                  dict(idx=sel.idx_sorted.cpu().numpy(), order=sel.pick_order.cpu().numpy(), gain=sel.pick_gain.cpu().numpy(),
                       n_kept=sel.n_kept.cpu().numpy(), status=sel.status.cpu().numpy()))
        sel = akv.alpha_compress_event(K, V, pos, dev(e.qstat), budget, opts, p_ref=dev(e.p_ref), layout=akv.Layout.dense(K), want_scores=True)
        same_bits(few, dict(K=akv.to_host_bits(K.contiguous()), V=akv.to_host_bits(V.contiguous()), pos=pos.cpu().numpy(), idx=sel.idx_sorted.cpu().numpy(),
                            order=sel.pick_order.cpu().numpy(), gain=sel.pick_gain.cpu().numpy(), scores=sel.scores.cpu().numpy(),
                            n_kept=sel.n_kept.cpu().numpy(), status=sel.status.cpu().numpy()))


@pytest.mark.parametrize("shift", [28, 29, 30])
@pytest.mark.parametrize("N,budget", [(100, 40), (192, 64), (256, 128), (256, 140)])
def test_one_page_that_could_hold_far_more_slots_than_the_event_has(N, budget, shift):
    """A whole sequence in one page, whose size is stated as up to 2^30 slots; against the same rows in a dense cache, to the bit."""
    for B in (2, 80):
        ev = synth.make_plain(B, 2, 2, N, 128, budget, 0.5, dtype=synth.BF16, seed=N)
        plain = run_fused(ev)
        table = torch.randperm(B, device="cuda").to(torch.int32).view(B, 1)
        pools = [torch.empty((2, B, 2, N, 128), dtype=torch.bfloat16, device="cuda") for _ in "KV"]
        for pool, x in zip(pools, (dev(ev.K), dev(ev.V))):
            pool[:, table.long().flatten()] = x.transpose(0, 1)
        sl, sp, sh, sn, _ = pools[0].stride()
        lay = akv.Layout(B, 2, 2, N, 128, synth.BF16, (0, sl, 0, 0), 1 << shift, table, (sp, sh, sn))
        pos = dev(ev.pos)
        sel = akv.alpha_compress_event(pools[0], pools[1], pos, dev(ev.qstat), budget, akv.Options(lam=0.5), p_ref=dev(ev.p_ref), layout=lay)
        assert np.array_equal(sel.pick_order.cpu().numpy(), plain["order"]) and np.array_equal(sel.pick_gain.cpu().numpy(), plain["gain"])
        assert np.array_equal(pos.cpu().numpy(), plain["pos"])
        for pool, name in zip(pools, "KV"):
            assert np.array_equal(akv.to_host_bits(pool[:, table.long().flatten()].transpose(0, 1).contiguous()), plain[name]), name


@pytest.mark.parametrize("N,budget", [(2, 2), (3, 2), (33, 33), (64, 40), (128, 128), (129, 90), (192, 64), (256, 100)])
@pytest.mark.parametrize("lam", [0.5, 2.0])
def test_resident_kernel_picks_in_pairs(N, budget, lam):
    """Algorithm 1 two picks at a time: rows that come in pairs, down to the smallest sets and to all rows kept."""
    ev = in_pairs(synth.make_plain(1, 2, 2, N, 64, budget, lam, dtype=synth.F32, seed=N), N)
    check_all(ev, run_fused(ev), lam)


@pytest.mark.parametrize("page,pages_per_seq", [(64, 4), (32, 6), (256, 1)])
def test_paged_event_longer_than_the_tile(page, pages_per_seq):
    """Paged cache (page sizes are powers of two), budget 64: K pages are copied whole, a 256-slot page in two
    pieces around row 128."""
    c5 = synth.make_c5(seed=page, B=3, L=2, H=2, page=page, pages_per_seq=pages_per_seq, budget=64, rounds=1)
    L, H, N, d, b = c5.L, c5.H, c5.N, c5.d, c5.budget
    pool_K, pool_V = dev(c5.pool_K), dev(c5.pool_V)
    table, pos, q = dev(c5.block_table), dev(c5.pos), dev(c5.qstat)
    lay = akv.Layout.paged(pool_K, table)
    hostK = synth.paged_gather_dense(c5.pool_K, c5.block_table)
    hostV = synth.paged_gather_dense(c5.pool_V, c5.block_table)
    sel = akv.alpha_compress_event(pool_K, pool_V, pos, q, b, akv.Options(lam=c5.lam), layout=lay, want_scores=True)
    torch.cuda.synchronize()
    idx, order, sc = sel.idx_sorted.cpu().numpy(), sel.pick_order.cpu().numpy(), sel.scores.cpu().numpy()
    posn = pos.cpu().numpy()
    for bb in range(c5.B):
        pages = c5.block_table[bb].tolist()
        for l in range(L):
            for h in range(H):
                Kn = akv.to_host_bits(pool_K[l, pages, h]).reshape(N, d)
                Vn = akv.to_host_bits(pool_V[l, pages, h]).reshape(N, d)
                chk.check_event(hostK[bb, l, h], hostV[bb, l, h], c5.pos[bb, l, h], c5.qstat[l, h], None, b, c5.lam,
                                sc[bb, l, h], order[bb, l, h], idx[bb, l, h], Kn, Vn, posn[bb, l, h], log=[])


@pytest.mark.parametrize("maker", ["c3_192", "c2_256", "f32_96"])
def test_pool_pruning_changes_no_pick(maker):
    """The pool that Algorithm 1 runs over is pruned exactly: with pruning switched off (every candidate in the
    pool, which takes the kernels' large-pool routes) the picks, their order and the compacted rows are the same."""
    if maker == "c3_192":
        ev = synth.make_c3(seed=21, B=2, L=2, H=2, N=192, budget=64)
    elif maker == "c2_256":
        ev = synth.make_c2(seed=22, B=1, L=2, H=2)
    else:
        ev = synth.make_plain(2, 2, 2, 96, 64, 30, 0.5, dtype=synth.F32, seed=23)
    pruned = run_fused(ev)
    full = run_fused(ev, flags=akv.FLAG_NO_PRUNE)
    for k in ("order", "idx", "K", "V", "pos", "n_kept", "status"):
        assert np.array_equal(pruned[k], full[k]), k
    check_all(ev, full, ev.lam)


def test_reference_position_behind_some_keys():
    """Keys ahead of the reference position have negative distances; the fast kernel measures distances from
    the last key and turns the query statistic by the difference. Positions are sparse and large."""
    ev = synth.make_c3(seed=31, B=3, L=2, H=2, N=192, budget=64)
    rng = np.random.default_rng(31)
    ev.pos[:] = np.sort(rng.choice(3_000_000, size=192, replace=False)).astype(np.int32)
    ev.p_ref[:] = np.array([ev.pos[0, 0, 0, 100], ev.pos[0, 0, 0, 0] - 5, ev.pos[0, 0, 0, -1]], dtype=ev.p_ref.dtype)
    g = run_fused(ev)
    check_all(ev, g, ev.lam)


@pytest.mark.parametrize("N,budget", [(192, 64), (256, 128), (256, 140), (1000, 100)])
def test_a_selection_that_gives_up_lists_no_row(N, budget):
    """With the starve flag alpha_select issues no product: its waits run out, it reports status 3 and lists no row, and the
    compaction behind it (the three launches of the static variant) leaves the cache alone."""
    ev = synth.make_plain(1, 2, 2, N, 128, budget, 0.5, dtype=synth.BF16, seed=N)
    K, V, pos, q, pref = dev(ev.K), dev(ev.V), dev(ev.pos), dev(ev.qstat), dev(ev.p_ref)
    opts = akv.Options(lam=0.5, flags=akv.FLAG_TEST_STARVE_WAIT)
    s = akv.alpha_score(K, q, pos=pos, p_ref=pref, opts=opts)
    sel = akv.alpha_select(s, V, budget, opts, layout=akv.Layout.dense(V))
    assert bool((sel.status == 3).all()) and bool((sel.idx_sorted == -1).all()) and bool((sel.n_kept == 0).all())
    sel = akv.alpha_compress_event_static(K, V, pos, q, budget, opts, p_ref=pref)
    assert bool((sel.status == 3).all())
    for x, name in ((akv.to_host_bits(K), "K"), (akv.to_host_bits(V), "V"), (pos.cpu().numpy(), "pos")):
        assert np.array_equal(x, getattr(ev, name))


# ------------------------------------------------------------------ per-layer signatures, per-head budgets (Section 6)
@pytest.mark.parametrize("dtype,N,d", [(synth.BF16, 80, 128), (synth.F32, 600, 64)])
def test_per_layer_signature_mode(dtype, N, d):
    """Signatures averaged over the heads of one layer: the reduction, and the event that selects with it
    (resident kernel for the small shape, three launches for the large one)."""
    ev = synth.make_plain(2, 3, 2, N, d, 25, 0.7, dtype=dtype, seed=27)
    V = dev(ev.V)
    sig = akv.alpha_signature_layer(V).cpu().numpy()
    assert sig.shape == (2, 3, N, d)
    for b in range(2):
        for l in range(3):
            assert np.max(np.abs(sig[b, l] - O.signatures_per_layer(ev.V[b, l]))) < 2e-7
    K, pos, q, pref = dev(ev.K), dev(ev.pos), dev(ev.qstat), dev(ev.p_ref)
    opts = akv.Options(lam=0.7, sig_mode=akv.SIG_PER_LAYER)
    sel = akv.alpha_compress_event(K, V, pos, q, 25, opts, p_ref=pref, flat_sig=dev(sig), want_scores=True)
    torch.cuda.synchronize()
    Kn, Vn, pn = akv.to_host_bits(K), akv.to_host_bits(V), pos.cpu().numpy()
    for b in range(2):
        for l in range(3):
            ref_sig = O.signatures_per_layer(ev.V[b, l])
            for h in range(2):
                chk.check_event(ev.K[b, l, h], ev.V[b, l, h], ev.pos[b, l, h], ev.qstat[l, h], int(ev.p_ref[b]), 25, 0.7,
                                sel.scores[b, l, h].cpu().numpy(), sel.pick_order[b, l, h].cpu().numpy(),
                                sel.idx_sorted[b, l, h].cpu().numpy(), Kn[b, l, h], Vn[b, l, h], pn[b, l, h], sig=ref_sig)


@pytest.mark.parametrize("maker", ["c3_192", "c3_256", "c2_256", "f32_96", "f32_600"])
def test_per_head_budgets(maker):
    """A budget per (layer, head): every kernel family keeps budgets[l, h] rows per event, pads its index rows
    to the largest budget with -1 and reports the kept count; uniform budgets equal the scalar call."""
    if maker == "c3_192":
        ev = synth.make_c3(seed=41, B=2, L=3, H=2, N=192, budget=64)
    elif maker == "c3_256":
        ev = synth.make_c3(seed=45, B=2, L=3, H=2, N=256, budget=96)
    elif maker == "c2_256":
        ev = synth.make_c2(seed=42, B=2, L=3, H=2)
    elif maker == "f32_96":
        ev = synth.make_plain(2, 3, 2, 96, 64, 30, 0.5, dtype=synth.F32, seed=43)
    else:
        ev = synth.make_plain(2, 3, 2, 600, 128, 50, 0.5, dtype=synth.F32, seed=44)
    kmax = ev.budget
    rng = np.random.default_rng(7)
    budgets = rng.integers(1, kmax + 1, size=(3, 2)).astype(np.int32)
    budgets[0, 0], budgets[2, 1] = kmax, 1
    g = run_fused(ev, budgets=budgets)
    check_all(ev, g, ev.lam, budgets=budgets)
    assert int(g["n_kept"].sum()) == 2 * int(budgets.sum())
    scalar = run_fused(ev)
    uniform = run_fused(ev, budgets=np.full((3, 2), kmax, dtype=np.int32))
    for k in ("order", "idx", "K", "V", "pos", "n_kept", "status"):
        assert np.array_equal(scalar[k], uniform[k]), k


# ------------------------------------------------------------------ bounded waits, workspace query, large grids
@pytest.mark.parametrize("maker", ["tri_192", "tri_96", "tc_256"])
def test_bounded_wait_runs_out_and_reports_status_3(maker):
    """With the starve flag no K row is requested and the waits poll only a few times: every wait of the fused
    tensor-memory kernels runs out with nothing in flight, each event reports status 3, tensor memory is given
    back (the next, normal call runs) and K, V and positions are left as they were."""
    if maker == "tri_192":
        ev = synth.make_c3(seed=51, B=2, L=2, H=2, N=192, budget=64)
    elif maker == "tri_96":
        ev = synth.make_c3(seed=52, B=2, L=2, H=2, N=96, budget=40)
    else:
        ev = synth.make_c2(seed=53, B=2, L=2, H=2)
    g = run_fused(ev, flags=akv.FLAG_TEST_STARVE_WAIT)
    assert np.all(g["status"] == 3)
    assert np.array_equal(g["K"], ev.K) and np.array_equal(g["V"], ev.V) and np.array_equal(g["pos"], ev.pos)
    good = run_fused(ev)
    check_all(ev, good, ev.lam)


@pytest.mark.parametrize("dtype,N,d,budget", [(synth.F32, 192, 128, 64), (synth.F32, 40, 72, 40), (synth.BF16, 256, 64, 128)])
@pytest.mark.parametrize("lam", [0.0, 0.5])
def test_resident_waits_run_out_and_report_status_3(dtype, N, d, budget, lam):
    """The same of the kernel whose K and V tiles stay in shared memory, with and without the penalty: nothing is requested,
    its two waits run out, the cache is left alone and the next call is a normal one."""
    ev = synth.make_plain(2, 2, 2, N, d, budget, lam, dtype=dtype, seed=N + d)
    g = run_fused(ev, flags=akv.FLAG_TEST_STARVE_WAIT)
    assert np.all(g["status"] == 3)
    assert np.array_equal(g["K"], ev.K) and np.array_equal(g["V"], ev.V) and np.array_equal(g["pos"], ev.pos)
    check_all(ev, run_fused(ev), lam)
    # rows apart: their copies are awaited in another way, beside the same two waits
    K, V = torch.zeros((2, 2, 2, 2, N, d + 8), dtype=torch.float32 if dtype == synth.F32 else torch.bfloat16, device="cuda")[..., :d]
    pos = dev(ev.pos)
    K.copy_(dev(ev.K)); V.copy_(dev(ev.V))
    sel = akv.alpha_compress_event(K, V, pos, dev(ev.qstat), budget, akv.Options(lam=lam, flags=akv.FLAG_TEST_STARVE_WAIT), p_ref=dev(ev.p_ref))
    assert bool((sel.status == 3).all())
    assert np.array_equal(akv.to_host_bits(K), ev.K) and np.array_equal(akv.to_host_bits(V), ev.V) and np.array_equal(pos.cpu().numpy(), ev.pos)


def test_workspace_query_matches_the_route():
    bf = akv.Layout(2, 2, 2, 192, 128, akv.api.AKV_BF16, (2 * 2 * 192 * 128, 2 * 192 * 128, 192 * 128, 128))
    assert akv.workspace_bytes(bf, 64) == 0                                  # on chip, one launch
    f32_small = akv.Layout(1, 1, 1, 192, 128, akv.api.AKV_F32, (192 * 128,) * 3 + (128,))
    assert akv.workspace_bytes(f32_small, 64) == 0                           # tiles resident in shared memory
    f32_big = akv.Layout(1, 2, 2, 600, 128, akv.api.AKV_F32, (4 * 600 * 128, 2 * 600 * 128, 600 * 128, 128))
    assert akv.workspace_bytes(f32_big, 50) == 1 * 2 * 2 * 600 * 4          # the scores between the launches
    bf_big = akv.Layout(1, 2, 2, 4096, 128, akv.api.AKV_BF16, (4 * 4096 * 128, 2 * 4096 * 128, 4096 * 128, 128))
    assert akv.workspace_bytes(bf_big, 128) == 0                             # streaming kernel, scores stay on chip


def test_score_with_more_events_than_a_grid_dimension_holds():
    """70 000 events: the event index is folded into grid.x, which has room for them."""
    B, N, d = 70_000, 8, 8
    rng = np.random.default_rng(61)
    K = rng.standard_normal((B, 1, 1, N, d)).astype(np.float32)
    q = rng.standard_normal((1, 1, d)).astype(np.float32)
    s = akv.alpha_score(dev(K), dev(q), pos=dev(np.arange(N, dtype=np.int32)),
                        p_ref=dev(np.full(B, N, dtype=np.int32))).cpu().numpy()
    for b in (0, 1, 65_535, 65_536, B - 1):
        ref = O.triattention_score(K[b, 0, 0], np.arange(N), q[0, 0], N)
        chk.check_scores(s[b, 0, 0], ref, chk.score_scale(K[b, 0, 0], q[0, 0], d))


# ------------------------------------------------------------------ large pools: the streaming one-launch kernel
@pytest.mark.parametrize("N,budget,lam", [(257, 40, 0.5), (300, 128, 0.0), (1000, 64, 0.5), (1000, 100, 1.5), (2050, 128, 1.0), (5041, 128, 1.0),
                                          (5042, 128, 1.0), (9000, 128, 1.0)])
def test_large_pool_stream_kernel(N, budget, lam):
    """bf16, d = 128, N > 256: K streams through a ring, scores stay on chip, pool rows of V only (up to N = 5120 in the
    prefill kernel, beyond in the stream kernel). Ragged candidate counts put the end of an event inside a ring stage, at
    its edge, and below the budget."""
    ev = synth.make_c3(seed=N, B=4, L=1, H=2, N=N, budget=budget)
    before = akv.launch_count()
    g = run_fused(ev, lam=lam)
    assert akv.launch_count() == before + 1                                   # one launch for the whole event
    check_all(ev, g, lam)
    n_cand = [N, N - 63, 64 * (N // 64), budget - 3]
    g = run_fused(ev, lam=lam, n_cand=n_cand)
    check_all(ev, g, lam, n_cand=n_cand)


def test_large_pool_stream_kernel_variants():
    """The prefill kernel: no pruning (the pool outgrows the active set), the greedy
    loop forced at lambda = 0, per-head budgets, irregular positions with the default reference position, every
    row scored from scratch, and the bounded waits running out."""
    ev = synth.make_c3(seed=71, B=2, L=2, H=2, N=900, budget=48)
    base = run_fused(ev)
    check_all(ev, base, ev.lam)
    full = run_fused(ev, flags=akv.FLAG_NO_PRUNE)
    for k in ("order", "idx", "K", "V", "pos"):
        assert np.array_equal(base[k], full[k]), k
    fast, loop = run_fused(ev, lam=0.0), run_fused(ev, lam=0.0, flags=akv.FLAG_FORCE_GREEDY)
    assert np.array_equal(fast["order"], loop["order"]) and np.array_equal(fast["K"], loop["K"])
    check_all(ev, fast, 0.0)
    budgets = np.array([[48, 1], [17, 30]], dtype=np.int32)
    check_all(ev, run_fused(ev, budgets=budgets), ev.lam, budgets=budgets)
    fresh = run_fused(ev, flags=akv.FLAG_NO_CHAIN)
    assert np.max(np.abs(fresh["scores"] - base["scores"])) < 2e-6
    check_all(ev, fresh, ev.lam)
    ev.pos[:] = np.sort(np.random.default_rng(72).choice(200_000, size=900, replace=False)).astype(np.int32)
    g = run_fused(ev, p_ref=False)
    check_all(ev, g, ev.lam, p_ref=False)
    starved = run_fused(ev, flags=akv.FLAG_TEST_STARVE_WAIT)
    assert np.all(starved["status"] == 3)
    assert np.array_equal(starved["K"], ev.K) and np.array_equal(starved["V"], ev.V) and np.array_equal(starved["pos"], ev.pos)


@pytest.mark.parametrize("N,budget", [(700, 128), (1500, 128)])
def test_large_pool_active_set_bound_reached(N, budget):
    """Every V row exists twice and the penalty is strong: the prefill kernel's loop over the best-scored rows reaches its
    bound and goes on with further active sets."""
    ev = synth.make_plain(2, 1, 2, N, 128, budget, 2.0, dtype=synth.BF16, seed=N)
    ev.V[..., N // 2:, :] = ev.V[..., :N // 2, :]
    check_all(ev, run_fused(ev), ev.lam)


@pytest.mark.parametrize("N,budget,scale,twice", [(257, 128, 1.0, False), (700, 128, 0.4, True), (701, 100, 0.05, True), (1500, 128, 0.25, True),
                                                  (5120, 128, 0.3, True), (5121, 128, 1.0, False), (1000, 1, 1.0, False), (300, 128, 1e-9, True)])
def test_prefill_sized_pool_beyond_the_active_set(N, budget, scale, twice):
    """Two events per SM, an active set of 192 rows. Statistics scaled down (scores then differ less than the penalty) and
    every V row twice send the picks beyond it, to one or many more rounds with further active sets, also where more than
    192 scores are equal."""
    ev = synth.make_plain(2, 1, 2, N, 128, budget, 0.5, dtype=synth.BF16, seed=N + budget)
    ev.qstat[...] *= scale
    if twice:
        ev.V[..., N - N // 2:, :] = ev.V[..., :N // 2, :]
    if N == 701:
        ev.K[0, 0, 0] = ev.K[0, 0, 0, :1]      # one event whose scores are all equal
        ev.pos[0, 0, 0] = 5
    before = akv.launch_count()
    g = run_fused(ev)
    assert akv.launch_count() == before + 1
    check_all(ev, g, ev.lam)
    K, V, pos = dev(ev.K), dev(ev.V), dev(ev.pos)
    s = akv.alpha_score(K, dev(ev.qstat), pos=pos, p_ref=dev(ev.p_ref), opts=akv.Options(lam=0.5))
    sel = akv.alpha_select(s, V, budget, akv.Options(lam=0.5), layout=akv.Layout.dense(V))      # selection by itself
    sn, order = s.cpu().numpy(), sel.pick_order.cpu().numpy()
    for b in range(2):
        for h in range(2):
            rep = O.replay_pick_order(sn[b, 0, h].astype(np.float64), O.signatures_per_head(ev.V[b, 0, h], ev.eps), 0.5,
                                      order[b, 0, h].astype(np.int64), chk.MARGIN_TOL)
            assert rep.ok, rep.log[:3]


@pytest.mark.parametrize("L,H,N", [(1, 4, 1023), (1, 4, 1024), (1, 4, 1025), (1, 37, 1601), (2, 19, 2048), (5, 15, 2047), (5, 15, 2113), (4, 15, 3072),
                                   (1, 3, 5120), (5, 15, 3008), (4, 37, 4096)])
def test_scoring_shared_by_several_ctas(L, H, N):
    """Few long events: several CTAs share an event's scoring (four from N = 1024, two from 2048, by the number of events). The
    same events in a call of more than any chip's multiprocessors are scored by one CTA each: every output is the same to the
    bit, also with irregular positions, candidates that end within one CTA's share, and a wait that runs out."""
    ev = synth.make_plain(1, L, H, N, 128, 40, 0.5, dtype=synth.BF16, seed=N + H)
    times = 512 // (L * H)
    many = synth.make_plain(times, 1, 1, 1, 128, 1, 0.5, dtype=synth.BF16, seed=0)
    for irregular in (False, True):
        if irregular:
            ev.pos[:] = np.sort(np.random.default_rng(N).choice(100_000, size=N, replace=False)).astype(np.int32)
        for name in ("K", "V", "pos", "p_ref"):
            setattr(many, name, np.repeat(getattr(ev, name), times, axis=0))
        many.qstat, many.budget = ev.qstat, ev.budget
        for n in (N, N - 70, 513, 30):
            a = run_fused(ev, n_cand=[n], p_ref=not irregular)
            b = run_fused(many, n_cand=[n] * times, p_ref=not irregular)
            for k, x in a.items():
                x, y = (x[..., :n], b[k][..., :n]) if k == "scores" else (x, b[k])
                assert np.array_equal(x[0], y[0]) and np.array_equal(x[0], y[-1]), (k, n, irregular)
    starved = run_fused(ev, flags=akv.FLAG_TEST_STARVE_WAIT)
    assert np.all(starved["status"] == 3)
    assert np.array_equal(starved["K"], ev.K) and np.array_equal(starved["V"], ev.V) and np.array_equal(starved["pos"], ev.pos)


@pytest.mark.parametrize("L,H,N", [(1, 4, 1100), (1, 37, 4096), (2, 19, 4096), (1, 111, 3000), (4, 37, 4096)])
def test_first_cta_learns_that_another_gave_up(L, H, N):
    """With the starve flag the first CTA of a cluster has its rows and scores them; only the others' waits run out. That reaches
    it through its shared memory: the event reports status 3, writes nothing, and the next call is a normal one."""
    ev = synth.make_plain(1, L, H, N, 128, 40, 0.5, dtype=synth.BF16, seed=N + H)
    for lam in (0.5, 0.0):
        assert akv_split.prefill_split(L * H, N, torch.cuda.get_device_properties(0).multi_processor_count, topk=lam == 0.0) > 1
        starved = run_fused(ev, lam=lam, flags=akv.FLAG_TEST_STARVE_WAIT)
        assert np.all(starved["status"] == 3)
        # (scores of the first CTA's rows are there, in eights of stages; no others)
        assert np.all(starved["scores"][..., :512] != 0.0) and np.all(starved["scores"][..., -1] == 0.0)
        for k in ("K", "V", "pos"):
            assert np.array_equal(starved[k], getattr(ev, k)), k
    good = run_fused(ev)
    check_all(ev, good, 0.5, events=[0, L * H - 1])


@pytest.mark.parametrize("rest,N,budget", [(1, 3009, 17), (40, 3072, 128), (70, 3100, 64)])
def test_last_events_of_a_topk_call_in_a_launch_of_their_own(rest, N, budget):
    """Top-k over many long events: the few beyond the full waves share their scoring and come in a second launch, which ends after
    the first; every event as in a small call, to the bit, also when captured and replayed."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    E, base = 2 * sms + rest, 7
    assert akv_split.prefill_tail(E, N, sms, topk=True) == rest and akv_split.prefill_tail(E, N, sms, topk=False) == 0
    ev = synth.make_plain(1, 1, base, N, 128, budget, 0.0, dtype=synth.BF16, seed=N)
    small = run_fused(ev)
    check_all(ev, small, 0.0, events=[0, base - 1])
    which = torch.arange(E, device="cuda") % base
    K0, V0, pos0, q = (dev(x).index_select(dim, which) for x, dim in ((ev.K, 2), (ev.V, 2), (ev.pos, 2), (ev.qstat, 1)))
    K, V, pos = K0.clone(), V0.clone(), pos0.clone()
    opts, pref = akv.Options(lam=0.0), dev(ev.p_ref)
    before = akv.launch_count()
    sel = akv.alpha_compress_event(K, V, pos, q, budget, opts, p_ref=pref)
    idx = sel.idx_sorted.clone()          # (the next thing on the stream)
    assert akv.launch_count() == before + 2

    def same():
        for got, want in ((K.view(torch.int16), small["K"].view(np.int16)), (V.view(torch.int16), small["V"].view(np.int16)), (pos, small["pos"]),
                          (sel.pick_order, small["order"]), (sel.pick_gain, small["gain"]), (idx, small["idx"]), (sel.status, small["status"])):
            assert torch.equal(got, torch.from_numpy(want).cuda().index_select(2, which))

    same()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        K.copy_(K0); V.copy_(V0); pos.copy_(pos0)
        akv.alpha_compress_event(K, V, pos, q, budget, opts, p_ref=pref, out=sel)
        idx.copy_(sel.idx_sorted)
    for _ in range(2):
        sel.pick_order.zero_(); idx.zero_()
        graph.replay()
        same()


@pytest.mark.parametrize("rest", [1, 40])
@pytest.mark.parametrize("kind", ["starved", "budgets", "pages"])
def test_kinds_of_topk_call_whose_last_events_have_a_launch_of_their_own(kind, rest):
    """Waits that run out (the second launch's CTAs leave early, and still only behind the first launch), a budget per head, pages in any
    order: both launches look them up for their own events."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    E, base, N, budget, page = 2 * sms + rest, 7, 3072, 64, 64
    assert akv_split.prefill_tail(E, N, sms, topk=True) == rest
    ev = synth.make_plain(1, 1, base, N, 128, budget, 0.0, dtype=synth.BF16, seed=rest)
    few = (np.arange(base, dtype=np.int32) * 9 + 5) % budget + 1
    small = run_fused_once(ev, budgets=few[None] if kind == "budgets" else None)
    which = torch.arange(E, device="cuda") % base
    K, V, pos, q = (dev(x).index_select(dim, which) for x, dim in ((ev.K, 2), (ev.V, 2), (ev.pos, 2), (ev.qstat, 1)))
    opts, lay = akv.Options(lam=0.0), None
    if kind == "starved":
        opts.flags = akv.FLAG_TEST_STARVE_WAIT
    elif kind == "budgets":
        opts.head_budgets = torch.from_numpy(few).cuda()[which][None].contiguous()
    else:
        table = torch.randperm(N // page, device="cuda").to(torch.int32)[None]
        place = table.long().flatten().argsort()
        K, V = (x.view(1, E, N // page, page, 128)[:, :, place].transpose(1, 2).contiguous() for x in (K, V))
        lay = akv.Layout.paged(K, table, N)
    K0, V0, pos0, before = K.clone(), V.clone(), pos.clone(), akv.launch_count()
    sel = akv.alpha_compress_event(K, V, pos, q, budget, opts, p_ref=dev(ev.p_ref), layout=lay)
    status, Kc, Vc = sel.status.clone(), K.clone(), V.clone()      # (the next things on the stream)
    assert akv.launch_count() == before + 2
    if kind == "starved":
        assert bool((status == 3).all()) and torch.equal(Kc, K0) and torch.equal(Vc, V0) and torch.equal(pos, pos0)
        return
    if kind == "pages":
        Kc, Vc = (x[:, table.long().flatten()].transpose(1, 2).reshape(1, 1, E, N, 128) for x in (Kc, Vc))
    for got, want in ((Kc.view(torch.int16), small["K"].view(np.int16)), (Vc.view(torch.int16), small["V"].view(np.int16)), (pos, small["pos"]),
                      (sel.pick_order, small["order"]), (sel.pick_gain, small["gain"]), (sel.idx_sorted, small["idx"]), (status, small["status"]),
                      (sel.n_kept, small["n_kept"])):
        assert torch.equal(got, torch.from_numpy(want).cuda().index_select(2, which))


@pytest.mark.parametrize("L,H,N,lam", [(2, 2, 1100, 0.0), (2, 2, 1100, 0.5), (2, 19, 2048, 0.0), (2, 19, 2113, 0.5), (5, 15, 3072, 0.0), (5, 15, 2048, 0.5)])
def test_shared_scoring_of_all_kinds_of_call(L, H, N, lam):
    """Four or two CTAs per event, with and without the penalty: budgets per head, a non-finite key in every CTA's part and pages in
    any order, against the same events in a call that takes one CTA each, to the bit, and a few events against the oracle."""
    ev = synth.make_plain(1, L, H, N, 128, 40, lam, dtype=synth.BF16, seed=N + H)
    rng = np.random.default_rng(N)
    times = 512 // (L * H)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    split = akv_split.prefill_split(L * H, N, sms, topk=lam == 0.0)
    assert split > 1 and akv_split.prefill_split(L * H * times, N, sms, topk=lam == 0.0) == 1
    many = synth.make_plain(times, 1, 1, 1, 128, 1, lam, dtype=synth.BF16, seed=0)
    many.qstat, many.budget = ev.qstat, ev.budget

    def both(**kw):
        for name in ("K", "V", "pos", "p_ref"):
            setattr(many, name, np.repeat(getattr(ev, name), times, axis=0))
        a, b = run_fused(ev, lam=lam, **kw), run_fused(many, lam=lam, **kw)
        for k, x in a.items():
            assert np.array_equal(x[0], b[k][-1], equal_nan=x.dtype == np.float32), k
        return a

    check_all(ev, both(), lam, events=[0, L * H - 1])
    budgets = rng.integers(1, 41, size=(L, H)).astype(np.int32)
    budgets[0, 0], budgets[-1, -1] = 40, 1
    check_all(ev, both(budgets=budgets), lam, events=[0, L * H - 1], budgets=budgets)
    # the same rows in pages
    K, V, pos, q, pref = (dev(x) for x in (ev.K, ev.V, ev.pos, ev.qstat, ev.p_ref))
    plain = run_fused(ev, lam=lam)
    for page in (64, 16):
        pps = -(-N // page)
        table = torch.as_tensor(rng.permutation(pps), device="cuda").to(torch.int32).view(1, pps)
        pools = torch.zeros((2, L, pps, H, page, 128), dtype=torch.bfloat16, device="cuda")
        for x, pool in zip((K, V), pools):
            rows = torch.zeros((L, H, pps * page, 128), dtype=torch.bfloat16, device="cuda")
            rows[:, :, :N] = x[0]
            pool[:, table[0].long()] = rows.view(L, H, pps, page, 128).permute(0, 2, 1, 3, 4)
        p = pos.clone()
        sel = akv.alpha_compress_event(pools[0], pools[1], p, q, 40, akv.Options(lam=lam), p_ref=pref, layout=akv.Layout.paged(pools[0], table, N), want_scores=True)
        for k, x in (("order", sel.pick_order), ("idx", sel.idx_sorted), ("gain", sel.pick_gain), ("scores", sel.scores), ("pos", p)):
            assert np.array_equal(x.cpu().numpy(), plain[k]), (k, page)
        for name, pool in zip(("K", "V"), pools):
            rows = pool[:, table[0].long()].permute(0, 2, 1, 3, 4).reshape(L, H, pps * page, 128)[:, :, :N]
            assert np.array_equal(akv.to_host_bits(rows.contiguous()), plain[name][0]), (name, page)
    # a key without a finite score in every CTA's part
    share = 64 * akv_split.split_share((N + 63) // 64, split)
    bad = [c * share + 5 for c in range(split) if c * share + 5 < N]
    assert len(bad) > 1
    ev.K[..., bad, 3] = 0x7F80 if ev.K.dtype == np.uint16 else np.inf
    g = both()
    assert np.all(g["status"] == 1) and not set(bad) & set(g["idx"].ravel().tolist())


@pytest.mark.parametrize("N,budget", [(129, 65), (130, 128), (160, 97), (161, 128), (193, 71), (224, 100), (225, 96), (255, 128), (256, 127)])
@pytest.mark.parametrize("lam", [0.0, 0.5])
def test_kept_slots_in_order_at_the_edges_of_words(N, budget, lam):
    """The 256-row kernel orders kept slots by bits in eight words: event sizes and budgets at and beside the words' edges."""
    ev = synth.make_plain(2, 1, 2, N, 128, budget, lam, dtype=synth.BF16, seed=N + budget)
    check_all(ev, run_fused(ev), lam)
    n_cand = [N, budget + 1]
    check_all(ev, run_fused(ev, n_cand=n_cand), lam, n_cand=n_cand)


@pytest.mark.parametrize("dtype,N,d,page", [(synth.F32, 1, 128, 0), (synth.F32, 63, 128, 0), (synth.F32, 65, 128, 0), (synth.F32, 130, 128, 0),
                                            (synth.F32, 200, 64, 0), (synth.BF16, 256, 64, 0), (synth.F32, 70, 128, 1), (synth.F32, 70, 128, 16),
                                            (synth.BF16, 90, 72, 32), (synth.F32, 192, 128, 64), (synth.F32, 71, 128, 2), (synth.BF16, 200, 64, 4),
                                            (synth.BF16, 200, 64, 8), (synth.F32, 65, 256, 0), (synth.BF16, 250, 8, 0), (synth.BF16, 250, 8, 64)])
@pytest.mark.parametrize("padded", [False, True])
def test_resident_tiles_by_bulk_copies(dtype, N, d, page, padded):
    """The resident kernel's tiles arrive in copies of 32 KB, whole pages or single rows (padded: rows that do not lie one
    behind the other), by bulk copies from 1 KB on, below by all threads: sizes at and beside a copy's end, candidates that end
    inside one, pages in any order."""
    ev = synth.make_plain(2, 1, 2, N, d, max(1, N // 3), 0.5, dtype=dtype, seed=N + d)
    width = d + (8 if padded else 0)
    rng = np.random.default_rng(N)

    def place(x):   # -> the tensor that holds the rows, and the view the call takes
        t = torch.zeros((2, 1, 2, N, width), dtype=torch.float32 if dtype == synth.F32 else torch.bfloat16, device="cuda")
        t[..., :d] = dev(x)
        if not page:
            return t[..., :d]
        pps = -(-N // page)
        pool = torch.zeros((1, 2 * pps, 2, page, width), dtype=t.dtype, device="cuda")
        rows = torch.zeros((2, 1, 2, pps * page, width), dtype=t.dtype, device="cuda")
        rows[:, :, :, :N] = t
        for b in range(2):
            pool[0, torch.as_tensor(table[b], device="cuda").long()] = rows[b, 0].view(2, pps, page, width).permute(1, 0, 2, 3)
        return pool[..., :d]

    table = rng.permutation(2 * (-(-N // page) if page else 1)).reshape(2, -1).astype(np.int32)
    K, V, pos = place(ev.K), place(ev.V), dev(ev.pos)
    lay = akv.Layout.paged(K, dev(table), N) if page else akv.Layout.dense(K)
    n_cand = [N, max(1, N - 5)]
    sel = akv.alpha_compress_event(K, V, pos, dev(ev.qstat), ev.budget, akv.Options(lam=0.5), p_ref=dev(ev.p_ref), n_cand=dev(np.asarray(n_cand, dtype=np.int32)),
                                   layout=lay, want_scores=True)
    plain = run_fused(ev, n_cand=n_cand)
    check_all(ev, plain, 0.5, n_cand=n_cand)
    assert np.array_equal(sel.pick_order.cpu().numpy(), plain["order"]) and np.array_equal(sel.idx_sorted.cpu().numpy(), plain["idx"])
    for b in range(2):
        assert np.array_equal(sel.scores.cpu().numpy()[b, ..., :n_cand[b]], plain["scores"][b, ..., :n_cand[b]])
    assert np.array_equal(pos.cpu().numpy(), plain["pos"])


def _takes_stream_kernel(N, budget):
    """bf16, d = 128, per-head signatures: what the prefill kernel's limits leave"""
    text = open(os.path.join(os.path.dirname(akv.__file__), "csrc", "akv_event_prefill.cuh")).read()
    limit = {k: int(re.search(r"constexpr int %s = (\d+);" % k, text).group(1)) for k in ("kPfMaxN", "kPfMaxBudget")}
    return N > 256 and (N > limit["kPfMaxN"] or budget > limit["kPfMaxBudget"])


@pytest.mark.parametrize("N,budget,lam", [(300, 129, 0.5), (900, 200, 1.0), (1500, 150, 0.0), (5041, 129, 1.0), (5042, 140, 1.0), (5121, 64, 0.5)])
@pytest.mark.parametrize("twice", [False, True])
def test_stream_kernel(N, budget, lam, twice):
    """Budgets above 128 and N above 5120, rings of eight and of four stages. twice: every V row twice, so that the loop over the
    active set reaches its bound and the route over the whole pool follows (the one within the operand tile, or plain dot
    products where the pool outgrows it)."""
    assert _takes_stream_kernel(N, budget)
    ev = synth.make_plain(4, 1, 2, N, 128, budget, 2 * lam if twice else lam, dtype=synth.BF16, seed=N + budget)
    if twice:
        ev.V[..., N - N // 2:, :] = ev.V[..., :N // 2, :]
    before = akv.launch_count()
    g = run_fused(ev)
    assert akv.launch_count() == before + 1
    check_all(ev, g, ev.lam)
    n_cand = [N, N - 63, 64 * (N // 64), budget - 3]
    check_all(ev, run_fused(ev, n_cand=n_cand), ev.lam, n_cand=n_cand)


def test_stream_kernel_variants():
    """No pruning, the loop forced at lambda = 0, per-head budgets, scores taken afresh, irregular positions with the default
    reference position, close and equal scores, starved waits."""
    N, budget = 900, 140
    assert _takes_stream_kernel(N, budget)
    ev = synth.make_c3(seed=75, B=2, L=2, H=2, N=N, budget=budget)
    base = run_fused(ev)
    check_all(ev, base, ev.lam)
    full = run_fused(ev, flags=akv.FLAG_NO_PRUNE)
    for k in ("order", "idx", "K", "V", "pos"):
        assert np.array_equal(base[k], full[k]), k
    fast, loop = run_fused(ev, lam=0.0), run_fused(ev, lam=0.0, flags=akv.FLAG_FORCE_GREEDY)
    assert np.array_equal(fast["order"], loop["order"]) and np.array_equal(fast["K"], loop["K"])
    budgets = np.array([[140, 1], [17, 130]], dtype=np.int32)
    check_all(ev, run_fused(ev, budgets=budgets), ev.lam, budgets=budgets)
    fresh = run_fused(ev, flags=akv.FLAG_NO_CHAIN)
    assert np.max(np.abs(fresh["scores"] - base["scores"])) < 2e-6
    for width in (0.0, 1e-3):
        close = _close_scores(N, budget, 0.5, width, seed=76)
        check_all(close, run_fused(close), 0.5)
    ev.pos[:] = np.sort(np.random.default_rng(77).choice(200_000, size=N, replace=False)).astype(np.int32)
    check_all(ev, run_fused(ev, p_ref=False), ev.lam, p_ref=False)
    starved = run_fused(ev, flags=akv.FLAG_TEST_STARVE_WAIT)
    assert np.all(starved["status"] == 3)
    assert np.array_equal(starved["K"], ev.K) and np.array_equal(starved["V"], ev.V) and np.array_equal(starved["pos"], ev.pos)


@pytest.mark.parametrize("budget,lam,twice", [(150, 0.5, False), (150, 1.5, True), (100, 1.5, True)])
def test_paged_large_pools(budget, lam, twice):
    """A paged cache of N = 576 in the stream kernel (150 kept) and in the prefill kernel beyond its first active set (100
    kept, every V row twice), under budgets per head."""
    c5 = synth.make_c5(seed=78, B=2, L=2, H=2, page=64, pages_per_seq=9, budget=budget, rounds=1)
    L, H, N, d = c5.L, c5.H, c5.N, c5.d
    assert _takes_stream_kernel(N, budget) == (budget > 128)
    if twice:
        for bb in range(c5.B):
            pages = c5.block_table[bb]
            c5.pool_V[:, pages[5:]] = c5.pool_V[:, pages[:4]]
    hostK = synth.paged_gather_dense(c5.pool_K, c5.block_table)
    hostV = synth.paged_gather_dense(c5.pool_V, c5.block_table)
    pool_K, pool_V = dev(c5.pool_K), dev(c5.pool_V)
    pos = dev(c5.pos)
    budgets = np.array([[budget, 60], [budget - 1, 90]], dtype=np.int32)
    sel = akv.alpha_compress_event(pool_K, pool_V, pos, dev(c5.qstat), budget, akv.Options(lam=lam, head_budgets=dev(budgets)),
                                   layout=akv.Layout.paged(pool_K, dev(c5.block_table)), want_scores=True)
    torch.cuda.synchronize()
    idx, order, sc, posn = (x.cpu().numpy() for x in (sel.idx_sorted, sel.pick_order, sel.scores, pos))
    for bb in range(c5.B):
        pages = c5.block_table[bb].tolist()
        for l in range(L):
            for h in range(H):
                Kn = akv.to_host_bits(pool_K[l, pages, h]).reshape(N, d)
                Vn = akv.to_host_bits(pool_V[l, pages, h]).reshape(N, d)
                chk.check_event(hostK[bb, l, h], hostV[bb, l, h], c5.pos[bb, l, h], c5.qstat[l, h], None, int(budgets[l, h]), lam,
                                sc[bb, l, h], order[bb, l, h], idx[bb, l, h], Kn, Vn, posn[bb, l, h], log=[])


def test_large_pool_stream_kernel_paged():
    c5 = synth.make_c5(seed=73, B=2, L=2, H=2, page=64, pages_per_seq=9, budget=100, rounds=1)   # N = 576
    L, H, N, d, b = c5.L, c5.H, c5.N, c5.d, c5.budget
    pool_K, pool_V = dev(c5.pool_K), dev(c5.pool_V)
    table, pos, q = dev(c5.block_table), dev(c5.pos), dev(c5.qstat)
    lay = akv.Layout.paged(pool_K, table)
    hostK = synth.paged_gather_dense(c5.pool_K, c5.block_table)
    hostV = synth.paged_gather_dense(c5.pool_V, c5.block_table)
    sel = akv.alpha_compress_event(pool_K, pool_V, pos, q, b, akv.Options(lam=c5.lam), layout=lay, want_scores=True)
    torch.cuda.synchronize()
    idx, order, sc = sel.idx_sorted.cpu().numpy(), sel.pick_order.cpu().numpy(), sel.scores.cpu().numpy()
    posn = pos.cpu().numpy()
    for bb in range(c5.B):
        pages = c5.block_table[bb].tolist()
        for l in range(L):
            for h in range(H):
                Kn = akv.to_host_bits(pool_K[l, pages, h]).reshape(N, d)
                Vn = akv.to_host_bits(pool_V[l, pages, h]).reshape(N, d)
                chk.check_event(hostK[bb, l, h], hostV[bb, l, h], c5.pos[bb, l, h], c5.qstat[l, h], None, b, c5.lam,
                                sc[bb, l, h], order[bb, l, h], idx[bb, l, h], Kn, Vn, posn[bb, l, h], log=[])


def test_chained_and_fresh_scores_agree_on_the_tensor_memory_kernels():
    for ev in (synth.make_c3(seed=81, B=2, L=2, H=2, N=192, budget=64), synth.make_c2(seed=82, B=1, L=2, H=2)):
        a, b = run_fused(ev), run_fused(ev, flags=akv.FLAG_NO_CHAIN)
        scale = np.abs(a["scores"]).max()
        assert np.max(np.abs(a["scores"] - b["scores"])) < 1e-6 * max(scale, 1.0)
        check_all(ev, b, ev.lam)


@pytest.mark.parametrize("N,budget,chain", [(128, 64, 8), (192, 64, 12), (256, 64, 16), (256, 128, 8), (256, 140, 8), (1000, 64, 8), (4096, 128, 8), (6000, 128, 8)])
def test_error_of_carried_rotations(N, budget, chain):
    """Scores of evenly spaced rows against float64, 2-norm over 2-norm. Fresh rotations leave 1.0e-7 (sums of 128 products of numbers that are
    right to 2^-25). A step of a chain adds the turn's error, the same one at every step: its sine and cosine are rounded twice, to
    2^-25 each, 4.3e-8 together. That is for rms of 0 .. chain - 1 steps. (With 2 pi / 2^37 off by 1.2e-6 a step added 8e-8.)"""
    ev = synth.make_plain(2, 2, 4, N, 128, budget, 0.5, dtype=synth.BF16, seed=N + budget)
    s = run_fused_once(ev)["scores"].astype(np.float64)
    ref = np.stack([[[O.triattention_score(ev.K[b, l, h], ev.pos[b, l, h], ev.qstat[l, h], int(ev.p_ref[b])) for h in range(4)] for l in range(2)]
                    for b in range(2)])
    bound = np.hypot(1.05e-7, 4.3e-8 * np.sqrt(np.mean(np.arange(chain) ** 2.0)))
    assert np.linalg.norm(s - ref) <= bound * np.linalg.norm(ref)


# ------------------------------------------------------------------ shared signatures with one cosine matrix per sequence
@pytest.mark.parametrize("L,H", [(1, 1), (1, 31), (4, 8), (3, 11), (9, 7), (1, 64), (5, 13)])
@pytest.mark.parametrize("dtype", [synth.BF16, synth.F32])
def test_signatures_over_any_number_of_pairs(dtype, L, H):
    """Rows requested four at a time from 32 (layer, head) pairs on, and a remainder one by one. fp32 sums of unit-scale rows:
    a unit row is within 1e-6 of the float64 one."""
    ev = synth.make_plain(2, L, H, 37, 64, 5, 0.5, dtype=dtype, seed=L * H)
    V = dev(ev.V)
    flat, layer = akv.alpha_signature_flat(V).cpu().numpy(), akv.alpha_signature_layer(V).cpu().numpy()
    for b in range(2):
        assert np.max(np.abs(flat[b] - O.signatures_flat(ev.V[b]))) < 1e-6
        for l in range(L):
            assert np.max(np.abs(layer[b, l] - O.signatures_per_layer(ev.V[b, l]))) < 1e-6


@pytest.mark.parametrize("mode", ["flat", "layer"])
@pytest.mark.parametrize("N", [96, 256, 300])
def test_shared_cosine_matrix(mode, N):
    """Algorithm 1's cosine matrix of the shared signatures, once per sequence (Eq. 1) or per sequence and layer:
    three-part bf16 split on the tensor cores against the float64 product, with a ragged candidate count."""
    ev = synth.make_plain(2, 2, 3, N, 128, 16, 0.5, dtype=synth.BF16, seed=90 + N)
    V = dev(ev.V)
    n_cand = np.array([N, N - 37], dtype=np.int32)
    nc = dev(n_cand)
    lay = akv.Layout.dense(V)
    if mode == "flat":
        opts = akv.Options(sig_mode=akv.SIG_FLAT)
        sig = akv.alpha_signature_flat(V, n_cand=nc)
    else:
        opts = akv.Options(sig_mode=akv.SIG_PER_LAYER)
        sig = akv.alpha_signature_layer(V, n_cand=nc)
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    gram = akv.alpha_gram_shared(sig, lay, opts, n_cand=nc, status=status).cpu().numpy()
    assert int(status.item()) == 0
    for b in range(2):
        n = int(n_cand[b])
        groups = [None] if mode == "flat" else range(2)
        for l in groups:
            ref_sig = O.signatures_flat(ev.V[b][:, :, :n]) if l is None else O.signatures_per_layer(ev.V[b, l][:, :n])
            got = gram[b][:n, :n] if l is None else gram[b, l][:n, :n]
            assert np.max(np.abs(got - ref_sig @ ref_sig.T)) < 5e-7
            rest = gram[b][n:] if l is None else gram[b, l][n:]
            assert np.all(rest == 0)                                  # rows beyond the candidates are left alone


@pytest.mark.parametrize("mode,N,budget", [("flat", 256, 128), ("flat", 192, 64), ("layer", 256, 100), ("flat", 130, 20), ("flat", 8, 3),
                                           ("layer", 31, 31), ("flat", 32, 17), ("flat", 33, 8)])
def test_fused_event_with_shared_cosine_matrix(mode, N, budget):
    """Shared signatures in the fused path: signature pass, one cosine matrix per sequence (and layer), then every
    event of the sequence in ONE launch that reads its cosines from that matrix. Checked against the oracle with
    the float64 signatures, and against the general route (dot products of signature rows pick by pick)."""
    ev = synth.make_c3(seed=95 + N, B=2, L=3, H=2, N=N, budget=budget)
    lam = 0.7
    K, V, pos, q, pref = dev(ev.K), dev(ev.V), dev(ev.pos), dev(ev.qstat), dev(ev.p_ref)
    lay = akv.Layout.dense(V)
    smode = akv.SIG_FLAT if mode == "flat" else akv.SIG_PER_LAYER
    sig = akv.alpha_signature_flat(V) if mode == "flat" else akv.alpha_signature_layer(V)
    gram = akv.alpha_gram_shared(sig, lay, akv.Options(sig_mode=smode))
    K2, V2, pos2 = K.clone(), V.clone(), pos.clone()
    before = akv.launch_count()
    sel = akv.alpha_compress_event(K, V, pos, q, budget, akv.Options(lam=lam, sig_mode=smode, shared_gram=gram), p_ref=pref,
                                   flat_sig=sig, want_scores=True)
    assert akv.launch_count() == before + 1
    ref = akv.alpha_compress_event(K2, V2, pos2, q, budget, akv.Options(lam=lam, sig_mode=smode), p_ref=pref, flat_sig=sig)
    torch.cuda.synchronize()
    Kn, Vn, pn = akv.to_host_bits(K), akv.to_host_bits(V), pos.cpu().numpy()
    n_same = 0
    for b in range(2):
        for l in range(3):
            ref_sig = O.signatures_flat(ev.V[b]) if mode == "flat" else O.signatures_per_layer(ev.V[b, l])
            for h in range(2):
                chk.check_event(ev.K[b, l, h], ev.V[b, l, h], ev.pos[b, l, h], ev.qstat[l, h], int(ev.p_ref[b]), budget, lam,
                                sel.scores[b, l, h].cpu().numpy(), sel.pick_order[b, l, h].cpu().numpy(),
                                sel.idx_sorted[b, l, h].cpu().numpy(), Kn[b, l, h], Vn[b, l, h], pn[b, l, h], sig=ref_sig)
                n_same += int(torch.equal(sel.pick_order[b, l, h], ref.pick_order[b, l, h]))
    assert n_same >= 11                                               # the two routes round differently: near-ties may differ
    assert int(sel.status.abs().max()) == 0 and int(sel.n_kept.min()) == budget


@pytest.mark.parametrize("N,budget", [(256, 128), (193, 90)])
def test_shared_cosine_matrix_with_four_events_to_an_sm(N, budget):
    """The same of a call of more than three events per SM."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    B, lam = sms // 2 + 1, 0.5
    ev = synth.make_c3(seed=N, B=B, L=2, H=3, N=N, budget=budget)
    K, V, pos = dev(ev.K), dev(ev.V), dev(ev.pos)
    sig = akv.alpha_signature_flat(V)
    gram = akv.alpha_gram_shared(sig, akv.Layout.dense(V), akv.Options(sig_mode=akv.SIG_FLAT))
    sel = akv.alpha_compress_event(K, V, pos, dev(ev.qstat), budget, akv.Options(lam=lam, sig_mode=akv.SIG_FLAT, shared_gram=gram), p_ref=dev(ev.p_ref),
                                   flat_sig=sig, want_scores=True)
    Kn, Vn, pn = akv.to_host_bits(K), akv.to_host_bits(V), pos.cpu().numpy()
    for b, l, h in ((0, 0, 0), (B // 2, 1, 1), (B - 1, 1, 2)):
        chk.check_event(ev.K[b, l, h], ev.V[b, l, h], ev.pos[b, l, h], ev.qstat[l, h], int(ev.p_ref[b]), budget, lam,
                        sel.scores[b, l, h].cpu().numpy(), sel.pick_order[b, l, h].cpu().numpy(), sel.idx_sorted[b, l, h].cpu().numpy(),
                        Kn[b, l, h], Vn[b, l, h], pn[b, l, h], sig=O.signatures_flat(ev.V[b]))
    assert int(sel.status.abs().max()) == 0 and int(sel.n_kept.min()) == budget


def _duplicated_rows(seed, lam, B=2, L=2, H=2, N=256, budget=128):
    """Every V row occurs twice (rows j and j + N/2 are bit-identical): once a row is picked its twin is
    penalised by lambda, so the picks must go far down the score order, beyond any active set."""
    ev = synth.make_plain(B, L, H, N, 128, budget, lam, dtype=synth.BF16, seed=seed)
    ev.V[..., N // 2:, :] = ev.V[..., :N // 2, :]
    return ev


@pytest.mark.parametrize("lam,budget,active", [(2.0, 128, 180), (1.5, 128, 180), (1.0, 96, 158)])
def test_active_set_bound_reached_and_the_loop_continues_over_the_whole_pool(lam, budget, active):
    """N = 256 with duplicated V rows: the one-warp loop over the best-scored rows reaches its bound;
    the picks made stand, the rest are taken over the whole pool. Every pick is checked against the oracle."""
    ev = _duplicated_rows(33, lam, budget=budget)
    if budget < 128:
        ev.qstat *= 0.05         # (scores that differ by less than the penalty)
    g = run_fused(ev, lam=lam)
    log = check_all(ev, g, lam)
    # the picks did go deep: some kept row's score rank lies beyond the rows an active set holds at most
    s = g["scores"][0, 0, 0]
    rank = np.argsort(np.argsort(-s))
    assert rank[g["idx"][0, 0, 0]].max() > active
    print("duplicated rows, lambda", lam, "near-tie divergences:", log)


@pytest.mark.parametrize("N,budget,lam", [(256, 64, 2.0), (192, 64, 1.0), (194, 3, 4.0), (128, 128, 2.0)])
def test_small_event_kernel_with_more_than_127_pool_rows(N, budget, lam):
    """Strong penalties leave a pool that outgrows the 127 rows of the small kernel's triangle: the loop runs over the
    best-scored ones, and with every V row twice it reaches its bound and is finished over the whole pool."""
    ev = _duplicated_rows(35, lam, N=N, budget=budget)
    check_all(ev, run_fused(ev, lam=lam), lam)
    plain = synth.make_plain(2, 2, 2, N, 128, budget, lam, dtype=synth.BF16, seed=N + budget)
    check_all(plain, run_fused(plain, lam=lam), lam)


def _close_scores(N, budget, lam, width, seed, B=2, L=1, H=2):
    """Scores of 0.3 + width * N(0, 1): the statistic looks at two coordinates, one constant in all keys, and every key
    sits at the reference position. width = 0: all scores equal."""
    ev = synth.make_plain(B, L, H, N, 128, budget, lam, dtype=synth.BF16, seed=seed)
    rng = np.random.default_rng(seed)
    ev.qstat[...] = 0
    ev.qstat[..., 0], ev.qstat[..., 1] = np.sqrt(128.0), np.sqrt(128.0) / 256
    ev.K[..., 0] = synth.f32_to_bf16_bits(np.float32(0.3))
    ev.K[..., 1] = synth.f32_to_bf16_bits((256 * width * rng.standard_normal(ev.K.shape[:-1])).astype(np.float32))
    ev.pos[...] = 7
    ev.p_ref[...] = 7
    return ev


@pytest.mark.parametrize("lam", [0.5, 1.0])
@pytest.mark.parametrize("width", [0.0, 1e-3, 3e-3])
@pytest.mark.parametrize("N,budget", [(192, 64), (128, 128), (256, 128), (256, 96), (300, 128), (1000, 64), (5120, 128)])
def test_scores_close_together(N, budget, width, lam):
    """The best-scored rows that an active set holds are then told apart by the last bits of their scores, or by their slots."""
    ev = _close_scores(N, budget, lam, width, seed=N)
    check_all(ev, run_fused(ev), lam)


@pytest.mark.parametrize("N,budget", [(192, 64), (256, 128), (256, 96), (1000, 128)])
def test_zero_cache_and_non_finite_scores(N, budget):
    """A zero-filled cache keeps its lowest slots; so does one whose scores are all NaN, with status 1."""
    ev = synth.make_plain(1, 2, 2, N, 128, budget, 0.5, dtype=synth.BF16, seed=N)
    nan = synth.make_plain(1, 2, 2, N, 128, budget, 0.5, dtype=synth.BF16, seed=N)
    ev.K[...], ev.V[...] = 0, 0
    nan.K[..., 3] = synth.f32_to_bf16_bits(np.float32(np.nan))
    for e, status in ((ev, 0), (nan, 1)):
        g = run_fused(e)
        assert np.all(g["status"] == status)
        assert np.array_equal(g["order"], np.broadcast_to(np.arange(budget), g["order"].shape))
        assert np.array_equal(g["idx"], g["order"])
        for k in ("K", "V", "pos"):
            assert np.array_equal(g[k], getattr(e, k))


@pytest.mark.parametrize("lam", [0.0, 0.5])
@pytest.mark.parametrize("N,budget", [(192, 64), (256, 128), (250, 90), (256, 140), (1000, 100), (1000, 140), (5200, 100)])
def test_a_few_non_finite_scores_on_the_tensor_memory_kernels(N, budget, lam):
    """Flagged and never preferred: with the rows of infinite and NaN scores out of the candidates the result is the same."""
    ev = synth.make_plain(1, 1, 2, N, 128, budget, lam, dtype=synth.BF16, seed=N + budget)
    bad = [0, 5, 9, N // 2, N - 1]
    ev.K[0, 0, 0, bad[:3], 3] = synth.f32_to_bf16_bits(np.float32(np.inf))
    ev.K[0, 0, 0, bad[3:], 100] = synth.f32_to_bf16_bits(np.float32(np.nan))
    g = run_fused(ev)
    assert g["status"][0, 0].tolist() == [1, 0]
    order = g["order"][0, 0, 0].astype(np.int64)
    assert not set(bad) & set(order.tolist()) and len(set(order.tolist())) == budget
    good = np.setdiff1d(np.arange(N), bad)
    with np.errstate(invalid="ignore"):
        s = O.triattention_score(ev.K[0, 0, 0], ev.pos[0, 0, 0], ev.qstat[0, 0], int(ev.p_ref[0]))
    rep = O.replay_pick_order(s[good], O.signatures_per_head(ev.V[0, 0, 0][good], ev.eps), lam, np.searchsorted(good, order), chk.MARGIN_TOL)
    assert rep.ok, rep.log[:3]


@pytest.mark.parametrize("dtype,N,budget", [(synth.BF16, 192, 64), (synth.BF16, 256, 128), (synth.BF16, 256, 96), (synth.BF16, 256, 140), (synth.BF16, 1000, 128),
                                            (synth.BF16, 1000, 140), (synth.F32, 128, 64), (synth.F32, 128, 128)])
def test_zero_value_rows_with_eps_zero(dtype, N, budget):
    """eps = 0 and zero value rows: their reciprocal norm is infinite, their cosine counts as 0 (the oracle's with a tiny eps).
    In one event every value row is zero: no penalty, and the kept rows are the top-k."""
    ev = synth.make_plain(2, 1, 2, N, 128, budget, 0.5, dtype=dtype, seed=N + budget)
    ev.V[:, :, :, 3::7] = 0
    ev.V[0, 0, 0] = 0
    ev.eps = 0.0
    g = run_fused(ev)
    ev.eps = 1e-30
    check_all(ev, g, ev.lam)
    assert g["order"][0, 0, 0].tolist() == O.topk_indices(g["scores"][0, 0, 0].astype(np.float64), budget).tolist()


@pytest.mark.parametrize("N,budget", [(192, 64), (256, 128)])
def test_topk_order_with_equal_scores(N, budget):
    """lambda = 0 with every key row four times at one position: equal scores go to the lower slot, in the picks made and
    at the edge of the kept set (the pool of rows that reach the boundary score is then larger than the budget)."""
    ev = synth.make_plain(1, 2, 2, N, 128, budget, 0.0, dtype=synth.BF16, seed=N)
    ev.K[...] = np.repeat(ev.K[..., ::4, :], 4, axis=-2)
    ev.pos[...] = 7
    g = run_fused(ev, lam=0.0)
    check_all(ev, g, 0.0)
    for l in range(2):
        for h in range(2):
            assert g["order"][0, l, h].tolist() == O.topk_indices(g["scores"][0, l, h].astype(np.float64), budget).tolist()


def test_active_set_bound_reached_with_a_shared_cosine_matrix():
    """The same with Eq. 1 signatures and one cosine matrix per sequence (one layer, one head: the flat signature
    is the head's own), so the continuation reads its cosines from that matrix."""
    lam = 1.5
    ev = _duplicated_rows(34, lam, B=2, L=1, H=1)
    K, V, pos, q, pref = dev(ev.K), dev(ev.V), dev(ev.pos), dev(ev.qstat), dev(ev.p_ref)
    sig = akv.alpha_signature_flat(V)
    gram = akv.alpha_gram_shared(sig, akv.Layout.dense(V), akv.Options(sig_mode=akv.SIG_FLAT))
    sel = akv.alpha_compress_event(K, V, pos, q, ev.budget, akv.Options(lam=lam, sig_mode=akv.SIG_FLAT, shared_gram=gram),
                                   p_ref=pref, flat_sig=sig, want_scores=True)
    torch.cuda.synchronize()
    Kn, Vn, pn = akv.to_host_bits(K), akv.to_host_bits(V), pos.cpu().numpy()
    for b in range(2):
        chk.check_event(ev.K[b, 0, 0], ev.V[b, 0, 0], ev.pos[b, 0, 0], ev.qstat[0, 0], int(ev.p_ref[b]), ev.budget, lam,
                        sel.scores[b, 0, 0].cpu().numpy(), sel.pick_order[b, 0, 0].cpu().numpy(),
                        sel.idx_sorted[b, 0, 0].cpu().numpy(), Kn[b, 0, 0], Vn[b, 0, 0], pn[b, 0, 0],
                        sig=O.signatures_flat(ev.V[b]))
    assert int(sel.status.abs().max()) == 0 and int(sel.n_kept.min()) == ev.budget


# ------------------------------------------------------------------ grouped-query statistics
@pytest.mark.parametrize("N,budget,G", [(192, 64, 7), (256, 128, 4), (256, 96, 3), (256, 140, 2), (700, 60, 8)])
def test_mean_of_grouped_statistics_on_the_tensor_memory_kernels(N, budget, G):
    """The mean over a KV head's query heads is the score of their mean statistic, so these calls take the kernels of
    ungrouped ones (one for each of the four shapes)."""
    ev = synth.make_plain(2, 2, 3, N, 128, budget, 0.5, dtype=synth.BF16, seed=N + G)
    Q = np.random.default_rng(G).standard_normal((2, 3 * G, 128)).astype(np.float32)

    def run(e):
        K, V, pos = dev(e.K), dev(e.V), dev(e.pos)
        sel = akv.alpha_compress_event(K, V, pos, dev(Q), budget, akv.Options(lam=0.5, gqa_group=G), p_ref=dev(e.p_ref), want_scores=True)
        return dict(K=akv.to_host_bits(K), V=akv.to_host_bits(V), pos=pos.cpu().numpy(), scores=sel.scores.cpu().numpy(), order=sel.pick_order.cpu().numpy(),
                    idx=sel.idx_sorted.cpu().numpy(), gain=sel.pick_gain.cpu().numpy())

    g = run(ev)
    if takes_forms(ev):
        for times in beyond_one_and_three_per_sm(ev.n_events):
            same_bits(g, run(tiled(ev, times)))
    for b in range(2):
        for l in range(2):
            for h in range(3):
                q = Q[l, h * G:(h + 1) * G].astype(np.float64).mean(0)
                chk.check_event(ev.K[b, l, h], ev.V[b, l, h], ev.pos[b, l, h], q, int(ev.p_ref[b]), budget, 0.5,
                                g["scores"][b, l, h], g["order"][b, l, h], g["idx"][b, l, h], g["K"][b, l, h], g["V"][b, l, h], g["pos"][b, l, h])


@pytest.mark.parametrize("B", [1, 40, 120])
@pytest.mark.parametrize("N,budget", [(192, 64), (256, 128), (256, 96), (256, 140), (700, 60), (5200, 60)])
def test_grouped_statistics_are_scored_with_fresh_rotations(N, budget, B):
    """The scores of grouped calls keep the general kernels' precision: no rotation is carried from row to row."""
    ev = synth.make_plain(B if N <= 256 else 1, 2, 2, N, 128, budget, 0.5, dtype=synth.BF16, seed=N)
    Q = np.random.default_rng(N).standard_normal((2, 2 * 4, 128)).astype(np.float32)
    s = []
    for flags in (0, akv.FLAG_NO_CHAIN):
        sel = akv.alpha_compress_event(dev(ev.K), dev(ev.V), dev(ev.pos), dev(Q), budget, akv.Options(lam=0.5, gqa_group=4, flags=flags),
                                       p_ref=dev(ev.p_ref), want_scores=True)
        s.append(sel.scores.cpu().numpy())
    assert np.array_equal(s[0], s[1])


@pytest.mark.parametrize("reduce", ["mean", "max"])
@pytest.mark.parametrize("dtype,N,d", [(synth.BF16, 150, 128), (synth.F32, 600, 64)])
def test_grouped_query_statistics(reduce, dtype, N, d):
    """Several query statistics per KV head: scores are the mean or the maximum over the group (stand-alone scorer),
    and the fused call selects with them (resident kernel for the small shape, three launches for the large one)."""
    G = 4
    ev = synth.make_plain(2, 2, 2, N, d, 30, 0.5, dtype=dtype, seed=101)
    rng = np.random.default_rng(102)
    Q = rng.standard_normal((2, 2 * G, d)).astype(np.float32)            # [L, H * G, d]
    K, V, pos, pref = dev(ev.K), dev(ev.V), dev(ev.pos), dev(ev.p_ref)
    opts = akv.Options(lam=0.5, gqa_group=G, gqa_reduce=akv.GQA_MAX if reduce == "max" else akv.GQA_MEAN)
    s = akv.alpha_score(K, dev(Q), pos=pos, p_ref=pref, opts=opts).cpu().numpy()
    sel = akv.alpha_compress_event(K, V, pos, dev(Q), 30, opts, p_ref=pref, want_scores=True)
    torch.cuda.synchronize()
    Kn, Vn, pn = akv.to_host_bits(K), akv.to_host_bits(V), pos.cpu().numpy()
    for b in range(2):
        for l in range(2):
            for h in range(2):
                qs = Q[l, h * G:(h + 1) * G]
                ref = O.triattention_score_group(ev.K[b, l, h], ev.pos[b, l, h], qs, int(ev.p_ref[b]), reduce=reduce)
                scale = max(chk.score_scale(ev.K[b, l, h], q, d).max() for q in qs) * np.ones(N)
                chk.check_scores(s[b, l, h], ref, scale)
                chk.check_event(ev.K[b, l, h], ev.V[b, l, h], ev.pos[b, l, h], qs[0], int(ev.p_ref[b]), 30, 0.5,
                                None, sel.pick_order[b, l, h].cpu().numpy(), sel.idx_sorted[b, l, h].cpu().numpy(),
                                Kn[b, l, h], Vn[b, l, h], pn[b, l, h], ref_scores=ref)
                assert np.max(np.abs(sel.scores[b, l, h].cpu().numpy() - ref)) < 1e-5 * scale.max()



def test_report_worst_score_error():
    """Printed for the record (run last in this file): the worst score error of everything checked so far."""
    print("worst |err|/|s| where |s| >= 0.1 scale: %.3e; worst |err|/scale: %.3e; scores checked: %d"
          % (chk.WORST["rel_to_score"], chk.WORST["rel_to_scale"], chk.WORST["n"]))
    assert chk.WORST["rel_to_score"] <= chk.SCORE_RTOL
