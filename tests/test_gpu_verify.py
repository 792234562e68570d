"""GPU parity of dsbd_verify_step / dsbd_select_width against the oracle (through the C ABI)."""
import numpy as np
import pytest
import torch

import oracle
import paper_2409_16560_b200 as dsbd
from paper_2409_16560_b200 import binding, inputs
from parity_util import check_exempt, compare_verify, run_gpu_verify, to_host_f32

pytestmark = pytest.mark.gpu


def _oracle(forest, params, zp, zq, rp, rq, threads=8):
    return oracle.verify_step(forest, params, zp, zq, rp.astype(np.float64), rq.astype(np.float64),
                              threads=threads)


def _both(data, steps, thresh=None):
    f, prm = data["forest"], dict(data["params"])
    if thresh is not None:
        prm["thresh"] = thresh
    zp_h, zq_h = to_host_f32(data["logits_p"]), to_host_f32(data["logits_q"])
    rp_h, rq_h = to_host_f32(data["root_logp"]), to_host_f32(data["root_logq"])
    exempt = decisions = 0
    for step in steps:
        prm["step"] = step
        gpu, status = run_gpu_verify(f, prm, data["logits_p"], data["logits_q"], data["root_logp"],
                                     data["root_logq"])
        assert status == 0
        ref = _oracle(f, prm, zp_h, zq_h, rp_h, rq_h)
        e, d = compare_verify(ref, gpu, f)
        exempt += e
        decisions += d
    check_exempt(exempt, decisions)
    return exempt, decisions


@pytest.mark.parametrize("name,steps", [("C1", range(40)), ("C2", range(40)), ("C3", range(6)),
                                        ("C4", range(3)), ("C6", range(6))])
def test_configs_full_size(name, steps):
    data = inputs.generate(inputs.config(name), "cuda", parts=("verify",))
    _both(data, steps)


@pytest.mark.parametrize("thresh,wmin", [(0.9, 1), (0.3, 1), (0.7, 8)])
def test_other_width_settings(thresh, wmin):
    data = inputs.generate(inputs.config("C3", R=2, V=5000), "cuda", parts=("verify",))
    data["params"]["W_min_r"] = None
    data["params"]["W_min"] = wmin
    _both(data, range(8), thresh=thresh)


@pytest.mark.parametrize("top_k,top_p", [(0, 1.0), (10, 0.8)])
def test_c5_all_requests(top_k, top_p):
    """The large configuration at full size, as the benchmark launches it: all 64 requests of
    three decode steps against the oracle, unwarped and with the warping of the paper's
    experiments (top-k 10 / top-p 0.8 on the joints)."""
    spec = inputs.config("C5")
    data = inputs.generate(spec, "cuda", parts=("verify",), draft_top_k=top_k, draft_top_p=top_p)
    data["params"].update(top_k=top_k, top_p=top_p)
    f, prm = data["forest"], dict(data["params"])
    zp_h, zq_h = to_host_f32(data["logits_p"]), to_host_f32(data["logits_q"])
    rp_h, rq_h = to_host_f32(data["root_logp"]), to_host_f32(data["root_logq"])
    exempt = decisions = 0
    for step in range(3):
        prm["step"] = step
        gpu, status = run_gpu_verify(f, prm, data["logits_p"], data["logits_q"], data["root_logp"],
                                     data["root_logq"])
        assert status == 0
        assert np.all(gpu["req_error"] == 0)
        assert np.all((gpu["l_last"] >= 1) & (gpu["l_last"] <= f["max_depth"] + 1))
        assert np.all(gpu["out_width"] >= 1)
        ref = _oracle(f, prm, zp_h, zq_h, rp_h, rq_h, threads=16)
        e, d = compare_verify(ref, gpu, f)
        exempt += e
        decisions += d
    check_exempt(exempt, decisions)


def _random_problem(rng, R, V, gamma, max_w, stride_pad=0, ninf_frac=0.0, tree="chain", min_w=1):
    widths = rng.integers(1, max_w + 1, size=R)
    if isinstance(tree, str):
        tree = inputs._chain(gamma) if tree == "chain" else inputs._binary(gamma)
    spec = dict(R=R, W=(min_w, max_w), tree=tree, prefix=(1, 1))
    forest, widths, _ = inputs.build_forest(spec, rng)
    N, B = forest["N"], forest["B"]
    stride = V + stride_pad
    zp = rng.normal(0, 2.5, size=(N, stride)).astype(np.float32)
    zq = (zp + rng.normal(0, 1.0, size=(N, stride))).astype(np.float32)
    if ninf_frac > 0:
        mask = rng.uniform(size=(1, stride)) < ninf_frac      # the same vocabulary entries for p and q
        zp[np.broadcast_to(mask, zp.shape)] = -np.inf
        zq[np.broadcast_to(mask, zq.shape)] = -np.inf
    tok = np.zeros(N, np.int32)
    for n in range(N):
        p = forest["parent"][n]
        if p >= 0:
            z = zq[p, :V].astype(np.float64)
            pr = np.exp(z - z.max()); pr /= pr.sum()
            tok[n] = rng.choice(V, p=pr)
    forest["token"] = tok
    rp = rng.normal(0, 1, B).astype(np.float32)
    rq = (rp + rng.normal(0, 0.5, B)).astype(np.float32)
    prm = dict(V=V, temperature=0.9, thresh=0.6, W_min=1, W_max=max_w, W_nom=max_w, seed=5, step=0,
               W_min_r=np.minimum(2, widths).astype(np.int32))
    return forest, prm, zp, zq, rp, rq, stride


@pytest.mark.parametrize("V,pad,ninf,tree", [(1023, 0, 0.0, "chain"), (1025, 3, 0.0, "chain"),
                                             (4097, 0, 0.0, "binary"), (777, 1, 0.2, "chain"),
                                             (3000, 0, 0.3, "binary"), (5, 0, 0.0, "chain")])
def test_ragged_vocab_unaligned_rows_masked_entries(V, pad, ninf, tree):
    rng = np.random.default_rng(V)
    exempt = decisions = 0
    for trial in range(6):
        forest, prm, zp, zq, rp, rq, stride = _random_problem(rng, R=5, V=V, gamma=3, max_w=4,
                                                              stride_pad=pad, ninf_frac=ninf, tree=tree)
        prm["step"] = trial
        dz = lambda a: torch.as_tensor(a).cuda()
        gpu, status = run_gpu_verify(forest, prm, dz(zp), dz(zq), dz(rp), dz(rq), row_stride=stride)
        assert status == 0
        ref = oracle.verify_step(forest, prm, zp, zq, rp.astype(np.float64), rq.astype(np.float64),
                                 row_stride=stride)
        e, d = compare_verify(ref, gpu, forest)
        exempt += e
        decisions += d
    check_exempt(exempt, decisions)


@pytest.mark.parametrize("R,V,max_w,gamma", [(700, 300, 3, 2), (3, 2500, 64, 1), (40, 9000, 16, 3)])
def test_many_requests_and_widest_layers(R, V, max_w, gamma):
    """More requests than resident clusters (several waves, small clusters), and the limit of
    64 beams / 64 live drafts per layer."""
    rng = np.random.default_rng(R + V)
    forest, prm, zp, zq, rp, rq, stride = _random_problem(rng, R=R, V=V, gamma=gamma, max_w=max_w)
    if max_w == 64:
        prm["W_min_r"] = None
        prm["W_min"] = 1
    dz = lambda a: torch.as_tensor(a).cuda()
    exempt = decisions = 0
    for step in range(2):
        prm["step"] = step
        gpu, status = run_gpu_verify(forest, prm, dz(zp), dz(zq), dz(rp), dz(rq))
        assert status == 0
        ref = oracle.verify_step(forest, prm, zp, zq, rp.astype(np.float64), rq.astype(np.float64), threads=8)
        e, d = compare_verify(ref, gpu, forest)
        exempt += e
        decisions += d
    check_exempt(exempt, decisions)


def test_peaky_distributions_use_the_exact_fallback():
    """When the histogram bin that a residual threshold falls into holds a heavy cell its
    bracket is too wide, and that residual mass is recomputed exactly by a pass over the rows.
    The path must be exercised and stay in parity."""
    rng = np.random.default_rng(11)
    exempt = decisions = fallbacks = respass = 0
    for trial in range(3):
        # a small vocabulary: every cell is heavy compared with the bracket tolerance, so any
        # threshold that shares its bin with a cell needs the exact evaluation
        forest, prm, zp, zq, rp, rq, stride = _random_problem(rng, R=200, V=64, gamma=3, max_w=6)
        prm["step"] = trial
        dz = lambda a: torch.as_tensor(a).cuda()
        gpu, status = run_gpu_verify(forest, prm, dz(zp), dz(zq), dz(rp), dz(rq))
        assert status == 0
        ref = oracle.verify_step(forest, prm, zp, zq, rp.astype(np.float64), rq.astype(np.float64))
        e, d = compare_verify(ref, gpu, forest)
        exempt += e; decisions += d
        st = gpu["req_stats"].reshape(-1, 8)
        assert np.array_equal(st[:, 0], np.minimum(ref["l_last"], forest["max_depth"]))   # layers verified
        assert st[:, 1].sum() == (ref["trace_kind"] == oracle.TR_ACCEPT).sum()            # accept tests
        acc = ref["trace_kind"] == oracle.TR_ACCEPT
        near_ref = int((np.abs(ref["trace_u"][acc] - np.minimum(ref["trace_a"][acc], 1.0)) < 1e-5).sum())
        assert abs(int(st[:, 4].sum()) - near_ref) <= 1                                    # near ties (the band's edge may differ)
        fallbacks += int(st[:, 2].sum()); respass += int(st[:, 3].sum())
    check_exempt(exempt, decisions)
    assert fallbacks > 0


def test_flat_tail_of_tiny_cells():
    """Rows whose vocabulary is a few heavy tokens plus a flat tail of about 10^5 cells of
    probability 1e-9 .. 1e-8 each (a per-cell mass near 2^-31): the tail as a whole carries
    1e-4 .. 1e-3 of the mass, far more than the 1e-5 tie band, so a histogram that rounded such
    cells to a coarse fixed-point unit would bias every residual mass.  Statuses, widths and
    tokens must still match the oracle."""
    rng = np.random.default_rng(21)
    V, R = 120000, 6
    forest, prm, _, _, rp, rq, stride = _random_problem(rng, R=R, V=64, gamma=3, max_w=4)
    N = forest["N"]
    zp = (-5.0 + 0.4 * rng.standard_normal((N, V))).astype(np.float32)
    heavy = rng.integers(0, V, size=(N, 40))
    for n in range(N):
        zp[n, heavy[n]] = rng.normal(11.0, 1.5, size=40)
    zq = (zp + 0.5 * rng.standard_normal((N, V))).astype(np.float32)
    tok = np.zeros(N, np.int32)
    for n in range(N):
        par = forest["parent"][n]
        if par >= 0:
            tok[n] = heavy[par, rng.integers(0, 40)]
    forest["token"] = tok
    prm = dict(prm, V=V, temperature=1.0)
    dz = lambda a: torch.as_tensor(a).cuda()
    exempt = decisions = 0
    for step in range(4):
        prm["step"] = step
        gpu, status = run_gpu_verify(forest, prm, dz(zp), dz(zq), dz(rp), dz(rq))
        assert status == 0
        ref = oracle.verify_step(forest, prm, zp, zq, rp.astype(np.float64), rq.astype(np.float64), threads=8)
        e, d = compare_verify(ref, gpu, forest)
        exempt += e; decisions += d
    check_exempt(exempt, decisions)
    # the tail is real mass: about 120000 cells of e^-5 against heavy cells of about e^11
    tail = np.exp(zp[0].astype(np.float64)); tail[heavy[0]] = 0.0
    assert tail.sum() / np.exp(zp[0].astype(np.float64)).sum() > 2e-5


def test_proportional_rows_overflow_is_detected():
    """Both models give the same next-token distribution in every row, so all cells of a row have
    the same ratio p_beam / q_beam (the ratio of the two beam weights) and land in one histogram
    bin: more mass than one 32-bit word of the histogram can hold.  The kernel must notice the
    wrapped word and compute that layer's residual masses by exact passes instead."""
    rng = np.random.default_rng(22)
    V = 100000
    forest, prm, _, _, rp, rq, stride = _random_problem(rng, R=4, V=64, gamma=2, max_w=4)
    N = forest["N"]
    zp = rng.normal(0.0, 1.0, size=(N, V)).astype(np.float32)
    zq = zp.copy()
    tok = np.zeros(N, np.int32)
    for n in range(N):
        if forest["parent"][n] >= 0:
            tok[n] = rng.integers(0, V)
    forest["token"] = tok
    rq = (rp + rng.normal(0, 1.0, len(rp))).astype(np.float32)       # beam weights differ between the models
    prm = dict(prm, V=V, temperature=1.0, thresh=0.3)
    dz = lambda a: torch.as_tensor(a).cuda()
    exempt = decisions = exact = wrapped = 0
    for step in range(3):
        prm["step"] = step
        gpu, status = run_gpu_verify(forest, prm, dz(zp), dz(zq), dz(rp), dz(rq))
        assert status == 0
        ref = oracle.verify_step(forest, prm, zp, zq, rp.astype(np.float64), rq.astype(np.float64), threads=8)
        e, d = compare_verify(ref, gpu, forest)
        exempt += e; decisions += d
        st = gpu["req_stats"].reshape(-1, 8)
        exact += int(st[:, 2].sum())
        wrapped += int(st[:, 6].sum())
    check_exempt(exempt, decisions)
    assert exact > 0 and wrapped > 0


@pytest.mark.parametrize("name,steps", [("C1", range(30)), ("C2", range(30)), ("C3", range(4)), ("C4", range(3)),
                                        ("C6", range(4))])
def test_configs_with_the_papers_warping(name, steps):
    """top-k 10 / top-p 0.8 on the joint distributions, the setting of the paper's experiments."""
    data = inputs.generate(inputs.config(name), "cuda", parts=("verify",), draft_top_k=10, draft_top_p=0.8)
    data["params"].update(top_k=10, top_p=0.8)
    _both(data, steps)


@pytest.mark.parametrize("top_k,top_p", [(1, 1.0), (3, 0.5), (64, 1.0), (64, 0.95), (7, 0.05)])
def test_warping_edge_settings(top_k, top_p):
    rng = np.random.default_rng(top_k)
    exempt = decisions = 0
    for trial in range(4):
        forest, prm, zp, zq, rp, rq, stride = _random_problem(rng, R=6, V=2100, gamma=3, max_w=5,
                                                              tree="binary" if trial % 2 else "chain")
        # make some drafts land inside the warped support: the best tokens of the small model
        best = np.argsort(-zq[:, :2100], axis=1)[:, :3]
        for n in range(forest["N"]):
            if forest["parent"][n] >= 0 and rng.uniform() < 0.7:
                forest["token"][n] = best[forest["parent"][n], rng.integers(0, 3)]
        prm.update(top_k=top_k, top_p=top_p, step=trial)
        dz = lambda a: torch.as_tensor(a).cuda()
        gpu, status = run_gpu_verify(forest, prm, dz(zp), dz(zq), dz(rp), dz(rq))
        # drafts outside the support of the warped q_beam (events of probability zero for a real
        # drafter) are accepted when p' has mass there and rejected otherwise; a rejection that
        # leaves no residual mass keeps p' -- neither side may report an error
        assert status == 0
        ref = oracle.verify_step(forest, prm, zp, zq, rp.astype(np.float64), rq.astype(np.float64))
        assert not ref["error"].any()
        e, d = compare_verify(ref, gpu, forest)
        exempt += e; decisions += d
    check_exempt(exempt, decisions)


@pytest.mark.parametrize("V,top_k", [(1000, 10), (2432, 50), (3000, 64)])
def test_top_k_near_the_number_of_tiles(V, top_k):
    """Fewer tiles than kept cells: every tile is taken and the threshold is found by bisection over
    counts that all threads of a half must read alike (a thread that read the next sweep's count took
    another branch, and its half waited for it for good).  Every repetition must
    give the first one's results."""
    rng = np.random.default_rng(V)
    forest, prm, zp, zq, rp, rq, _ = _random_problem(rng, R=61, V=V, gamma=2, max_w=8)
    prm.update(top_k=top_k, top_p=0.95, temperature=0.6, step=1)
    dev = [torch.as_tensor(x).cuda() for x in (zp, zq, rp, rq)]
    gpu, status = run_gpu_verify(forest, prm, *dev)
    assert status == 0
    for _ in range(40):
        again, status = run_gpu_verify(forest, prm, *dev)
        assert status == 0
        for k in ("out_width", "out_token", "out_parent", "node_status", "layer_width"):
            assert np.array_equal(again[k], gpu[k]), k
    ref = _oracle(forest, prm, zp, zq, rp, rq)
    check_exempt(*compare_verify(ref, gpu, forest))


@pytest.mark.parametrize("beams,gamma,V", [(15, 16, 512), (16, 15, 513), (16, 15, 1500), (6, 42, 700)])
def test_requests_around_the_node_cache_and_half_tiles(beams, gamma, V):
    """255, 256 and 258 nodes in a request (up to 256 are kept in every CTA's shared memory), at
    vocabularies where the histogram pass takes half tiles (one row tile, its second half empty, with one
    token, ragged) and where it takes whole ones; completion draws at every run position."""
    rng = np.random.default_rng(V)
    forest, prm, zp, zq, rp, rq, _ = _random_problem(rng, R=3, V=V, gamma=gamma, max_w=beams, min_w=beams)
    assert forest["N"] == 3 * beams * (gamma + 1)
    forest["draft_rank"] = rng.integers(0, 4, forest["N"]).astype(np.int32)
    dev = [torch.as_tensor(x).cuda() for x in (zp, zq, rp, rq)]
    exempt = decisions = 0
    for step in range(20):
        prm.update(step=step, thresh=0.3 + 0.03 * step)
        gpu, status = run_gpu_verify(forest, prm, *dev)
        assert status == 0
        e, d = compare_verify(_oracle(forest, prm, zp, zq, rp, rq), gpu, forest)
        exempt += e
        decisions += d
    check_exempt(exempt, decisions)


@pytest.mark.parametrize("V,beams,W_min,W_max", [(1, 3, 3, 3), (1000, 2, 2, 8), (1025, 5, 8, 8), (4097, 6, 4, 4),
                                                 (9000, 40, 3, 3), (33000, 4, 4, 9), (50257, 3, 3, 3)])
def test_layers_of_known_width(V, beams, W_min, W_max):
    """Layers whose width does not depend on the residual masses (at most W_min drafts, or W_min = W_max): no rejection,
    a rejection with none, three, four and many drafts behind it (passes on demand up to two or three, else the
    histogram), several rejections in a row, accepts between them; clusters of 1 to 16 CTAs, whole and half tiles, vocabularies of
    one token, one more than a tile and rows that are not aligned."""
    rng = np.random.default_rng(V + beams)
    forest, prm, zp, zq, rp, rq, _ = _random_problem(rng, R=4, V=V, gamma=3, max_w=beams, min_w=beams)
    zp = (zp + rng.normal(0, 1.0, zp.shape)).astype(np.float32)
    prm.update(W_min_r=None, W_min=W_min, W_max=W_max)
    dev = [torch.as_tensor(x).cuda() for x in (zp, zq, rp, rq)]
    exempt = decisions = on_demand = 0
    n0 = np.concatenate([forest["beam_node_off"][forest["req_beam_off"][:-1]], [forest["N"]]])
    for step in range(12):
        prm["step"] = step
        gpu, status = run_gpu_verify(forest, prm, *dev)
        assert status == 0
        e, d = compare_verify(_oracle(forest, prm, zp, zq, rp, rq), gpu, forest)
        exempt += e
        decisions += d
        # a pass takes a rejection, and the rows are looked into by layers that make one or build a histogram
        st = gpu["req_stats"].reshape(-1, 8)
        rejected = np.array([(gpu["node_status"][a:b] == binding.NODE_REJECTED).sum() for a, b in zip(n0[:-1], n0[1:])])
        assert np.all(st[:, 7] <= rejected)
        assert np.all(st[rejected == 0][:, [5, 7]] == 0)
        on_demand += int(st[:, 7].sum())
    check_exempt(exempt, decisions)
    if beams <= W_min:
        assert on_demand > 0


@pytest.mark.parametrize("V,beams,seeds", [(128256, 2, 3), (50257, 2, 2), (1025, 2, 1)])
def test_draws_behind_a_layer_of_known_width_are_those_of_a_histogram(V, beams, seeds):
    """One layer of two drafts whose two beams are wanted: W_min = 2 says so beforehand (no histogram is built), a
    threshold that every tail reaches says so afterwards.  The sums that a residual draw searches are the same numbers either
    way (run position 2: those of the histogram pass; 3: the cells at s as one float), so every output is, bit for bit."""
    R, steps = 64, 400
    forest, _, _ = inputs.build_forest(dict(R=R, W=beams, tree=inputs._chain(1), prefix=(1, 1)), np.random.default_rng(V))
    f = dsbd.Forest(forest, "cuda")
    off = dsbd.default_out_off(forest, dict(W_max=beams, W_nom=beams))
    drawn = 0
    for seed in range(seeds):
        gen = torch.Generator(device="cuda").manual_seed(1000 * V + seed)
        zq = 2.0 * torch.randn(forest["N"], V, generator=gen, device="cuda")
        zp = zq + 0.8 * torch.randn(forest["N"], V, generator=gen, device="cuda")
        rp, rq = (torch.randn(forest["B"], generator=gen, device="cuda") for _ in range(2))
        parent = torch.as_tensor(forest["parent"], device="cuda").long()
        drafts = torch.nonzero(parent >= 0).squeeze(1)
        f.dev["token"][drafts] = torch.multinomial(torch.softmax(zq[parent[drafts]], dim=1), 1, generator=gen).squeeze(1).to(torch.int32)
        known = dict(V=V, temperature=1.0, thresh=0.7, W_min=beams, W_max=beams, W_nom=beams, seed=seed, step=0, top_k=0, top_p=1.0)
        outs = [dsbd.alloc_verify_out(f, off, "cuda") for _ in range(2)]
        ws = torch.empty(dsbd.verify_workspace(f, known), dtype=torch.uint8, device="cuda")
        status = torch.zeros(1, dtype=torch.int32, device="cuda")
        moved = torch.zeros((), dtype=torch.int64, device="cuda")
        n_drawn = torch.zeros((), dtype=torch.int64, device="cuda")
        for step in range(steps):
            for out, prm in zip(outs, (known, dict(known, W_min=1, thresh=1e-9))):
                for name in ("out_token", "out_parent", "out_node", "out_root_beam", "out_source", "out_logp", "out_logq"):
                    out[name].zero_()
                dsbd.verify_step(f, dict(prm, step=step), zp, zq, rp, rq, out, workspace=ws, status=status)
            for name in outs[0]:
                if name != "req_stats":
                    moved += (outs[0][name] != outs[1][name]).sum()
            n_drawn += (outs[0]["out_source"] == binding.SRC_RESIDUAL).sum()
        assert int(status) == 0 and int(outs[0]["req_error"].abs().sum()) == 0
        assert int(moved) == 0, "%d outputs differ" % int(moved)
        drawn += int(n_drawn)
    assert drawn > 0.1 * R * steps * seeds


@pytest.mark.parametrize("beams,sigma", [(2, 0.38), (3, 0.5), (4, 0.7)])
def test_words_of_a_layer_of_few_drafts_do_not_wrap(beams, sigma):
    """100 requests: two CTAs add the whole layer to their histograms.  Two models sigma nats apart over a flat vocabulary put
    0.4 / sigma of their mass per nat next to ratio 1, which is 0.9e-4 to 1.1e-4 for each CTA in a bin of ln(beams) / 4096 nats.
    A bin has 20 cells or more, so the fullest of 4096 holds up to twice that: below the 2^-12 = 2.4e-4 at which a word wraps.
    Of the 0.05 of the mass beyond the last edge, ratio `beams`, each of 2 x 256 words holds 1e-4 or less."""
    V, R = 128256, 100
    forest, _, _ = inputs.build_forest(dict(R=R, W=beams, tree=inputs._chain(1), prefix=(1, 1)), np.random.default_rng(R))
    gen = torch.Generator(device="cuda").manual_seed(V + beams)
    zp = 0.3 * torch.randn(forest["N"], V, generator=gen, device="cuda")
    zq = zp + sigma * torch.randn(forest["N"], V, generator=gen, device="cuda")
    rp = rq = torch.zeros(forest["B"], device="cuda")
    prm = dict(V=V, temperature=1.0, thresh=0.7, W_min=1, W_max=beams, W_nom=beams, seed=5, step=0, top_k=0, top_p=1.0)
    gpu, status = run_gpu_verify(forest, prm, zp, zq, rp, rq)
    assert status == 0
    assert int(gpu["req_stats"].reshape(R, -1)[:, 6].sum()) == 0
    e, d = compare_verify(_oracle(forest, prm, *(to_host_f32(x) for x in (zp, zq, rp, rq))), gpu, forest)
    check_exempt(e, d)


@pytest.mark.parametrize("V,R", [(128256, 16), (5001, 2)])
def test_inputs_written_right_before_the_call(V, R):
    """Kernels of a call are in place before the work ahead of it in the stream ends: whatever that work writes (logits, tokens, root
    scores), calls one behind the other see the values of their turn, as they do one at a time."""
    rng = np.random.default_rng(V)
    forest, prm, zp, zq, rp, rq, _ = _random_problem(rng, R=R, V=V, gamma=2, max_w=3, min_w=3)
    prm.update(W_min_r=None, W_min=2)
    f, n = dsbd.Forest(forest, "cuda"), 3
    first = [torch.as_tensor(x).cuda() for x in (zp, zq, rp, rq)] + [f.dev["token"].clone()]
    gen = torch.Generator(device="cuda").manual_seed(V)
    sets = [first] + [[x + torch.randn(x.shape, generator=gen, device="cuda") for x in first[:4]] +
                      [torch.randint(0, V, first[4].shape, generator=gen, device="cuda").to(torch.int32)] for _ in range(n - 1)]
    live = [x.clone() for x in first[:4]] + [f.dev["token"]]
    ws = torch.empty(dsbd.verify_workspace(f, prm), dtype=torch.uint8, device="cuda")
    off = dsbd.default_out_off(forest, prm)

    def call(k, status):
        for dst, src in zip(live, sets[k % n]):
            dst.copy_(src)
        out = dsbd.alloc_verify_out(f, off, "cuda")
        dsbd.verify_step(f, dict(prm, step=k), *live[:4], out, workspace=ws, status=status)
        return out

    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    alone = []
    for k in range(24):
        alone.append(call(k, status))
        torch.cuda.synchronize()
    behind = [call(k, status) for k in range(24)]
    torch.cuda.synchronize()
    assert int(status) == 0
    for k in range(24):
        for name in alone[k]:
            assert torch.equal(alone[k][name], behind[k][name]), (k, name)


@pytest.mark.parametrize("R,pattern,W,passes", [(160, "RRRA", 1, 0), (160, "ARRA", 2, 2), (160, "AARR", 3, 2), (160, "RARA", 1, 0),
                                                (4, "RRRA", 1, 3), (4, "RRRR", 1, 4), (4, "RARR", 2, 2), (4, "RRRRA", 1, 0),
                                                (4, "AAAA", 4, 0), (4, "AARR", 1, 0)])
def test_passes_on_demand_are_few(R, pattern, W, passes):
    """One layer of known width whose drafts are accepted (A: far more likely under the large model) or rejected (R: impossible
    under it) by construction.  A rejection behind a rejection takes a pass, and so does the first; one behind an accept has the
    residual mass already.  With more than two drafts (three, where a warp has at most two tiles: 4 requests here) behind the
    first rejection the layer takes the histogram instead; it ends with W accepts."""
    V, m = 16400, len(pattern)
    forest, _, _ = inputs.build_forest(dict(R=R, W=m, tree=inputs._chain(1), prefix=(1, 1)), np.random.default_rng(1))
    rng = np.random.default_rng(V + R)
    zq = rng.normal(0, 1.5, size=(forest["N"], V)).astype(np.float32)
    zp = (zq + rng.normal(0, 1.0, size=zq.shape)).astype(np.float32)
    token = np.zeros(forest["N"], np.int32)
    drafts = np.nonzero(forest["parent"] >= 0)[0]
    for i, n in enumerate(drafts):
        row, token[n] = forest["parent"][n], rng.integers(0, V)
        accept = pattern[i % m] == "A"
        zp[row, token[n]] = 9.0 if accept else -60.0
        zq[row, token[n]] = -20.0 if accept else 1.0
    forest["token"] = token
    rp = rq = np.zeros(forest["B"], np.float32)
    prm = dict(V=V, temperature=1.0, thresh=0.7, W_min=W, W_max=W, W_nom=W, seed=3, step=0, top_k=0, top_p=1.0)
    gpu, status = run_gpu_verify(forest, prm, *(torch.as_tensor(x).cuda() for x in (zp, zq, rp, rq)))
    assert status == 0
    e, d = compare_verify(_oracle(forest, prm, zp, zq, rp, rq), gpu, forest)
    check_exempt(e, d)
    seen = {"A": binding.NODE_ACCEPTED, "R": binding.NODE_REJECTED}
    want = [seen[c] for c in pattern]
    stop = [i for i in range(m) if pattern[:i + 1].count("A") == W]
    if stop:
        want[stop[0] + 1:] = [binding.NODE_CUT] * (m - 1 - stop[0])
    assert np.array_equal(gpu["node_status"][drafts].reshape(R, m), np.tile(want, (R, 1)))
    assert np.all(gpu["req_stats"].reshape(R, -1)[:, 7] == passes)


@pytest.mark.parametrize("V", [2000, 40000])
def test_histograms_with_a_layer_of_known_width_between(V):
    """A layer with a histogram, one that needs none, another with one: drafts that widen again behind a chain."""
    rng = np.random.default_rng(V)
    forest, prm, zp, zq, rp, rq, _ = _random_problem(rng, R=4, V=V, gamma=4, max_w=5, min_w=5,
                                                     tree=[-1, 0, 1, 2, 2, 2, 3, 4, 4, 5, 5, 5])
    zq = (zp + rng.normal(0, 0.4, zp.shape)).astype(np.float32)      # most drafts are accepted
    prm.update(W_min_r=None, W_min=2)
    dev = [torch.as_tensor(x).cuda() for x in (zp, zq, rp, rq)]
    depth = np.zeros(forest["N"], np.int64)
    for n, par in enumerate(forest["parent"]):
        depth[n] = 0 if par < 0 else depth[par] + 1
    n0 = np.concatenate([forest["beam_node_off"][forest["req_beam_off"][:-1]], [forest["N"]]])
    tested = (binding.NODE_ACCEPTED, binding.NODE_REJECTED, binding.NODE_CUT)
    exempt = decisions = between = 0
    for step in range(16):
        prm.update(step=step, thresh=0.7 + 0.015 * step)
        gpu, status = run_gpu_verify(forest, prm, *dev)
        assert status == 0
        e, d = compare_verify(_oracle(forest, prm, zp, zq, rp, rq), gpu, forest)
        exempt += e
        decisions += d
        for r in np.nonzero(gpu["l_last"] >= 3)[0]:
            d, st = depth[n0[r]:n0[r + 1]], gpu["node_status"][n0[r]:n0[r + 1]]
            drafts = [int((np.isin(st, tested) & (d == l)).sum()) for l in (1, 2, 3)]
            between += drafts[0] > 2 and drafts[1] <= 2 and drafts[2] > 2      # W_min = 2
    check_exempt(exempt, decisions)
    assert between > 0


@pytest.mark.parametrize("V", [1000, 2000, 4000, 8000, 32000])
def test_every_cluster_size(V):
    """8 rows of 1, 2, 4, 8 and 32 tiles: clusters of 1, 2, 4, 8 and 16 CTAs, whose slices of the merged
    histogram the chain of 8 rejections looks into; scores tempered so that the ratios reach far bins."""
    rng = np.random.default_rng(V)
    forest, prm, zp, zq, rp, rq, _ = _random_problem(rng, R=1, V=V, gamma=3, max_w=8, min_w=8)
    zp = (zp + rng.normal(0, 2.0, zp.shape)).astype(np.float32)
    dev = [torch.as_tensor(x).cuda() for x in (zp, zq, rp, rq)]
    exempt = decisions = 0
    for step in range(10):
        prm.update(step=step, thresh=0.2 + 0.06 * step)
        gpu, status = run_gpu_verify(forest, prm, *dev)
        assert status == 0
        e, d = compare_verify(_oracle(forest, prm, zp, zq, rp, rq), gpu, forest)
        exempt += e
        decisions += d
    check_exempt(exempt, decisions)


@pytest.mark.parametrize("R", [9, 14, 18, 36, 80])
def test_as_many_clusters_as_the_device_holds(R):
    """6 rows of 16 tiles: clusters of 16 CTAs as long as all requests' fit at once, then of 8, 4 and 2."""
    rng = np.random.default_rng(R)
    forest, prm, zp, zq, rp, rq, _ = _random_problem(rng, R=R, V=16384, gamma=1, max_w=6, min_w=6)
    dev = [torch.as_tensor(x).cuda() for x in (zp, zq, rp, rq)]
    gpu, status = run_gpu_verify(forest, prm, *dev)
    assert status == 0
    check_exempt(*compare_verify(_oracle(forest, prm, zp, zq, rp, rq), gpu, forest))


@pytest.mark.parametrize("V,beams", [(524288, 2), (524289, 2), (600001, 3), (1050000, 1), (20000, 13), (4000, 64)])
def test_draws_over_pieces_and_shares(V, beams):
    """A draw from p_beam searches its row's tile masses 512 at a time: 512, 513, 586 and 1026 tiles.  A residual draw searches 256
    shares of the layer's tiles first: shares of 4, 5 and 7 tiles, of one (13 x 20 = 260 tiles: two), of one (64 x 4)."""
    rng = np.random.default_rng(V + beams)
    forest, prm, zp, zq, rp, rq, _ = _random_problem(rng, R=1, V=V, gamma=2 if V < 100000 else 1, max_w=beams, min_w=beams)
    zp = (zp + rng.normal(0, 2.0, zp.shape)).astype(np.float32)
    dev = [torch.as_tensor(x).cuda() for x in (zp, zq, rp, rq)]
    exempt = decisions = 0
    for step in range(4):
        prm.update(step=step, thresh=0.3, W_min=min(2, beams), W_min_r=None)
        gpu, status = run_gpu_verify(forest, prm, *dev)
        assert status == 0
        e, d = compare_verify(_oracle(forest, prm, zp, zq, rp, rq), gpu, forest)
        exempt += e
        decisions += d
    check_exempt(exempt, decisions)


@pytest.mark.parametrize("beams,V,top_k,top_p", [(64, 72000, 10, 0.8), (64, 72000, 64, 0.9), (36, 121900, 1, 1.0)])
def test_warped_layers_with_more_tiles_than_the_bound_cache(beams, V, top_k, top_p):
    """64 x 71 = 4544 tile bounds, more than are kept in shared memory (4368), and 36 x 120 = 4320, just fewer."""
    rng = np.random.default_rng(V + top_k)
    forest, prm, zp, zq, rp, rq, _ = _random_problem(rng, R=1, V=V, gamma=1, max_w=beams, min_w=beams)
    prm.update(top_k=top_k, top_p=top_p)
    dev = [torch.as_tensor(x).cuda() for x in (zp, zq, rp, rq)]
    exempt = decisions = 0
    for step in range(2):
        prm["step"] = step
        gpu, status = run_gpu_verify(forest, prm, *dev)
        assert status == 0
        e, d = compare_verify(_oracle(forest, prm, zp, zq, rp, rq), gpu, forest)
        exempt += e
        decisions += d
    check_exempt(exempt, decisions)


def test_roots_only_forest_goes_straight_to_the_extra_layer():
    rng = np.random.default_rng(3)
    V, B = 2000, 3
    forest = dict(R=1, B=B, N=B, max_depth=0, req_beam_off=np.array([0, B], np.int32),
                  beam_node_off=np.arange(B + 1, dtype=np.int32), parent=np.full(B, -1, np.int32),
                  token=np.zeros(B, np.int32))
    zp = rng.normal(0, 2, size=(B, V)).astype(np.float32)
    zq = rng.normal(0, 2, size=(B, V)).astype(np.float32)
    rp = rng.normal(0, 1, B).astype(np.float32)
    prm = dict(V=V, thresh=0.7, W_min=1, W_max=4, W_nom=4, seed=9)
    exempt = decisions = 0
    for step in range(20):
        prm["step"] = step
        dz = lambda a: torch.as_tensor(a).cuda()
        gpu, status = run_gpu_verify(forest, prm, dz(zp), dz(zq), dz(rp), dz(rp))
        assert status == 0 and gpu["l_last"][0] == 1 and gpu["out_width"][0] == 4
        ref = oracle.verify_step(forest, prm, zp, zq, rp.astype(np.float64), rp.astype(np.float64))
        e, d = compare_verify(ref, gpu, forest)
        exempt += e; decisions += d
    check_exempt(exempt, decisions)


def test_draft_rank_order_and_equal_models():
    rng = np.random.default_rng(4)
    forest, prm, zp, zq, rp, rq, stride = _random_problem(rng, R=3, V=500, gamma=3, max_w=4, tree="binary")
    # a draw order that disagrees with the node numbering
    forest["draft_rank"] = rng.permutation(forest["N"]).astype(np.int32)
    dz = lambda a: torch.as_tensor(a).cuda()
    gpu, status = run_gpu_verify(forest, prm, dz(zp), dz(zq), dz(rp), dz(rq))
    ref = oracle.verify_step(forest, prm, zp, zq, rp.astype(np.float64), rq.astype(np.float64))
    assert status == 0
    compare_verify(ref, gpu, forest)
    # p == q: every draft up to the width is accepted
    prm2 = dict(prm, W_min_r=None, W_min=1, W_max=64, W_nom=2)
    gpu, status = run_gpu_verify(forest, prm2, dz(zp), dz(zp), dz(rp), dz(rp))
    ref = oracle.verify_step(forest, prm2, zp, zp, rp.astype(np.float64), rp.astype(np.float64))
    assert status == 0 and np.all(gpu["l_last"] == forest["max_depth"] + 1)
    compare_verify(ref, gpu, forest)
    assert not np.any(gpu["node_status"] == dsbd.binding.NODE_REJECTED)


def test_bad_token_is_reported_not_trapped():
    rng = np.random.default_rng(6)
    forest, prm, zp, zq, rp, rq, stride = _random_problem(rng, R=2, V=300, gamma=2, max_w=2)
    forest["token"][forest["N"] - 1] = 300
    dz = lambda a: torch.as_tensor(a).cuda()
    gpu, status = run_gpu_verify(forest, prm, dz(zp), dz(zq), dz(rp), dz(rq))
    assert status == 1          # DSBD_DEV_BAD_TOKEN


def test_host_side_errors():
    rng = np.random.default_rng(7)
    forest, prm, zp, zq, rp, rq, stride = _random_problem(rng, R=1, V=64, gamma=1, max_w=2)
    f = dsbd.Forest(forest, "cuda")
    out = dsbd.alloc_verify_out(f, oracle.default_out_off(forest, prm), "cuda")
    dz = lambda a: torch.as_tensor(a).cuda()
    prm_dev = dict(prm, W_min_r=None)
    small = torch.empty(256, dtype=torch.uint8, device="cuda")
    with pytest.raises(dsbd.DsbdError) as e:
        dsbd.verify_step(f, prm_dev, dz(zp), dz(zq), dz(rp), dz(rq), out, workspace=small)
    assert e.value.code == -3
    with pytest.raises(dsbd.DsbdError) as e:
        dsbd.verify_step(f, dict(prm_dev, temperature=0.0), dz(zp), dz(zq), dz(rp), dz(rq), out)
    assert e.value.code == -1


def test_width_parameters_are_validated():
    """A zero-initialised W_max / W_nom, or a cap below the minimum width, is refused on the host;
    per-request widths, which only the device sees, are reported per request and the request
    is not verified."""
    rng = np.random.default_rng(12)
    forest, prm, zp, zq, rp, rq, stride = _random_problem(rng, R=3, V=200, gamma=2, max_w=3)
    f = dsbd.Forest(forest, "cuda")
    out = dsbd.alloc_verify_out(f, oracle.default_out_off(forest, prm), "cuda")
    dz = lambda a: torch.as_tensor(a).cuda()
    base = dict(prm, W_min_r=None, W_min=2, W_max=3, W_nom=3)
    for bad in (dict(W_max=0), dict(W_nom=0), dict(W_min=0), dict(W_min=3, W_max=2)):
        with pytest.raises(dsbd.DsbdError) as e:
            dsbd.verify_step(f, dict(base, **bad), dz(zp), dz(zq), dz(rp), dz(rq), out)
        assert e.value.code == -1, bad
    wmax_r = torch.tensor([3, 0, 3], dtype=torch.int32, device="cuda")
    status = dsbd.verify_step(f, dict(base, W_max_r=wmax_r), dz(zp), dz(zq), dz(rp), dz(rq), out)
    torch.cuda.synchronize()
    assert int(status.item()) == 6                     # DSBD_DEV_BAD_PARAM
    assert out["req_error"].cpu().tolist() == [0, 6, 0]
    assert "width" in dsbd.status_string(6)


def test_select_width_rejects_a_malformed_live_list():
    """Node ids outside the forest and offsets beyond the list are reported, never used as
    addresses; well-formed requests of the same call still get their width."""
    rng = np.random.default_rng(13)
    forest, prm, zp, zq, rp, rq, stride = _random_problem(rng, R=3, V=700, gamma=2, max_w=4)
    prm = dict(prm, W_min_r=None)
    rbo, bno = forest["req_beam_off"], forest["beam_node_off"]
    live = [bno[rbo[r]:rbo[r + 1]].copy() for r in range(forest["R"])]
    live_off = np.concatenate([[0], np.cumsum([len(x) for x in live])]).astype(np.int32)
    m = np.array([len(x) for x in live], np.int32)
    sp = rng.normal(0, 1, forest["N"]).astype(np.float32)
    f = dsbd.Forest(forest, "cuda")
    dz = lambda a: torch.as_tensor(a).cuda()
    good = np.concatenate(live).astype(np.int32)
    w_ref, _, _ = oracle.select_width(forest, prm, zp, zq, sp.astype(np.float64), sp.astype(np.float64),
                                      live_off, good, m)
    for bad_id in (forest["N"], -1, 1 << 30):
        nodes = good.copy()
        nodes[live_off[1]] = bad_id                    # first live parent of request 1
        width, _, _, status = dsbd.select_width(f, prm, dz(zp), dz(zq), dz(sp), dz(sp), dz(live_off),
                                                dz(nodes), dz(m), out_stride=8)
        torch.cuda.synchronize()
        assert int(status.item()) == 4                 # DSBD_DEV_BAD_FOREST
        w = width.cpu().numpy()
        assert w[0] == w_ref[0] and w[2] == w_ref[2]
    off = live_off.copy()
    off[-1] = 1 << 20                                  # a list far longer than the forest
    _, _, _, status = dsbd.select_width(f, prm, dz(zp), dz(zq), dz(sp), dz(sp), dz(off), dz(good), dz(m),
                                        out_stride=8)
    torch.cuda.synchronize()
    assert int(status.item()) == 4


@pytest.mark.parametrize("top_k,top_p", [(0, 1.0), (10, 0.8), (40, 1.0)])
def test_select_width_matches_oracle(top_k, top_p):
    rng = np.random.default_rng(8)
    forest, prm, zp, zq, rp, rq, stride = _random_problem(rng, R=4, V=3000, gamma=2, max_w=5)
    prm = dict(prm, W_min_r=None, top_k=top_k, top_p=top_p)
    rbo, bno = forest["req_beam_off"], forest["beam_node_off"]
    live = [bno[rbo[r]:rbo[r + 1]] for r in range(forest["R"])]      # the roots
    live_off = np.concatenate([[0], np.cumsum([len(x) for x in live])]).astype(np.int32)
    live_nodes = np.concatenate(live).astype(np.int32)
    m = np.array([len(x) for x in live], np.int32)
    sp = rng.normal(0, 1, forest["N"]).astype(np.float32)
    sq = rng.normal(0, 1, forest["N"]).astype(np.float32)
    f = dsbd.Forest(forest, "cuda")
    dz = lambda a: torch.as_tensor(a).cuda()
    width, alpha, tail, status = dsbd.select_width(f, prm, dz(zp), dz(zq), dz(sp), dz(sq), dz(live_off),
                                                   dz(live_nodes), dz(m), out_stride=8)
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    w_ref, a_ref, t_ref = oracle.select_width(forest, prm, zp, zq, sp.astype(np.float64),
                                              sq.astype(np.float64), live_off, live_nodes, m)
    assert np.array_equal(width.cpu().numpy(), w_ref)
    for r in range(forest["R"]):
        assert np.abs(alpha[r, :m[r]].cpu().numpy() - a_ref[r, :m[r]]).max() < 2e-5
        assert np.abs(tail[r, :m[r] + 1].cpu().numpy() - t_ref[r, :m[r] + 1]).max() < 2e-5


@pytest.mark.parametrize("value", [float(np.finfo(np.float32).min), -1e30, -1e15, -1e9, -np.inf])
@pytest.mark.parametrize("top_k", [0, 10])
def test_tiles_masked_with_huge_values(top_k, value):
    """A row with whole tiles at the mask's value: value / tau times log2(e) is beyond the type's range or rounded by
    far more than one, and the tile has no mass.  (Kept cells: more than tiles that hold some in half of the requests.)"""
    V = 5000
    rng = np.random.default_rng(top_k)
    forest, prm, zp, zq, rp, rq, _ = _random_problem(rng, R=4, V=V, gamma=3, max_w=4)
    zp[:, 1024:3072] = zq[:, 1024:3072] = value
    for n in range(forest["N"]):
        if 1024 <= forest["token"][n] < 3072:
            forest["token"][n] += 2048 if forest["token"][n] + 2048 < V else -1024
    prm.update(temperature=1.0, top_k=top_k, top_p=0.9 if top_k else 1.0)
    dev = [torch.as_tensor(x).cuda() for x in (zp, zq, rp, rq)]
    gpu, status = run_gpu_verify(forest, prm, *dev)
    assert status == 0
    check_exempt(*compare_verify(_oracle(forest, prm, zp, zq, rp, rq), gpu, forest))


def _masked_tiles(rng, n_rows, V, keep, value):
    """Two models' logits in which all but `keep` of the 1024-token tiles are masked with `value`."""
    zp = rng.normal(0, 2.5, size=(n_rows, V)).astype(np.float32)
    zq = (zp + rng.normal(0, 1.0, size=(n_rows, V))).astype(np.float32)
    tile = np.arange(V) // 1024
    masked = ~np.isin(tile, rng.choice(tile[-1] + 1, size=keep, replace=False))
    zp[:, masked] = value
    zq[:, masked] = value
    return zp, zq, np.flatnonzero(~masked)


@pytest.mark.parametrize("value", [-np.inf, float(np.finfo(np.float32).min), -1e30, -1e9, -1e4])
@pytest.mark.parametrize("V,top_k,extra", [(32000, 10, 0), (32000, 10, 2), (32000, 20, 1), (128256, 50, 2)])
def test_top_k_with_masked_tiles(V, top_k, extra, value):
    """k to k + 2 tiles hold the live vocabulary, the others are masked: the cut lies at the k-th largest tile bound
    whatever the distance to the next one.  (Temperature 1.5 keeps the scaled mask finite.)"""
    rng = np.random.default_rng(V + top_k + extra)
    forest, prm, _, _, rp, rq, _ = _random_problem(rng, R=3, V=8, gamma=2, max_w=1)
    zp, zq, live = _masked_tiles(rng, forest["N"], V, top_k + extra, value)
    for n in range(forest["N"]):
        par = forest["parent"][n]
        if par >= 0:                               # a token that the small model is likely to draft
            forest["token"][n] = live[np.argsort(-zq[par, live])[rng.integers(0, 8)]]
    prm.update(V=V, top_k=top_k, top_p=0.95, temperature=1.5)
    dev = [torch.as_tensor(x).cuda() for x in (zp, zq, rp, rq)]
    exempt = decisions = 0
    for step in range(3):
        prm["step"] = step
        gpu, status = run_gpu_verify(forest, prm, *dev)
        assert status == 0
        e, d = compare_verify(_oracle(forest, prm, zp, zq, rp, rq), gpu, forest)
        exempt += e
        decisions += d
    check_exempt(exempt, decisions)


def test_residual_next_to_a_dominant_cell():
    """One rejection; the residual is 12 cells of 2^-25 (of the heaviest cell) that share their lane with a cell of mass
    0.53, and the residuals of that cell and of one of 0.47 elsewhere, a quarter of it.  Each small cell is a quarter
    of the heavy one's last bit; a sum that holds both has none of them.  The heavy cells' masses are floats, their residuals
    (0.56 and 1 of their last bits) therefore 0 or 1 times 2^-24 and 0 to 2 times 2^-25: the small cells' share of
    1.9e-7 is at least 0.61, less 3 sigma of 512 draws 0.545."""
    R, V, u = 512, 512, 2.0 ** -23
    small = [it * 128 + c for it in (1, 2, 3) for c in range(4)]         # lane 0's cells, behind the heaviest
    zp = np.full((2, V), -np.inf, np.float32)
    zp[0, 0], zp[0, 4] = 0.0, np.log(0.875)
    zq = zp.copy()
    zp[0, small] = np.log(u / 4)
    zq[0, 500] = np.log(4 * u)                                           # the draft: outside the support of p
    zp[1], zq[1] = 0.0, 0.0
    N = 2 * R
    forest = dict(R=R, B=R, N=N, max_depth=1, req_beam_off=np.arange(R + 1, dtype=np.int32),
                  beam_node_off=(2 * np.arange(R + 1)).astype(np.int32), token=np.full(N, 500, np.int32),
                  parent=np.stack([np.full(R, -1), 2 * np.arange(R)], 1).reshape(-1).astype(np.int32))
    prm = dict(V=V, temperature=1.0, thresh=0.5, W_min=1, W_max=1, W_nom=1, seed=3, step=0)
    dev = [torch.as_tensor(np.tile(z, (R, 1))).cuda() for z in (zp, zq)]
    zero = torch.zeros(R, device="cuda")
    gpu, status = run_gpu_verify(forest, prm, *dev, zero, zero)
    assert status == 0 and (gpu["req_error"] == 0).all()
    assert (gpu["out_source"] == 1).all() and (gpu["l_last"] == 1).all()
    share = np.isin(gpu["out_token"], small).mean()
    assert share > 0.545, share


def test_a_node_with_a_malformed_parent_is_not_accepted():
    """A parent at or behind its own node is reported; the node stays unreached, its descendants are pruned."""
    rng = np.random.default_rng(2)
    forest, prm, zp, zq, rp, rq, _ = _random_problem(rng, R=1, V=600, gamma=4, max_w=3, min_w=3)
    prm.update(W_min=1, W_min_r=None, thresh=0.3)
    lo = int(forest["beam_node_off"][1])
    forest["parent"] = forest["parent"].copy()
    forest["parent"][lo + 1] = lo + 3
    dev = [torch.as_tensor(x).cuda() for x in (zp, zq, rp, rq)]
    f = dsbd.Forest(dict(forest, parent=np.where(forest["parent"] == lo + 3, lo, forest["parent"])), "cuda")
    f.dev["parent"] = torch.as_tensor(forest["parent"]).cuda()
    prm_dev = dict(prm)
    out = dsbd.alloc_verify_out(f, oracle.default_out_off(forest, prm), "cuda")
    status = dsbd.verify_step(f, prm_dev, *dev, out)
    assert int(status.item()) == 4
    got = out["node_status"].cpu().numpy()[lo:lo + 5]
    assert got[0] == 1 and got[1] == 0 and got[2] == 4, got


def test_draft_ranks_up_to_the_type_s_largest():
    """Equal ranks go by node id, whatever their value."""
    rng = np.random.default_rng(9)
    forest, prm, zp, zq, rp, rq, _ = _random_problem(rng, R=4, V=900, gamma=3, max_w=8, min_w=8)
    big = np.iinfo(np.int32).max
    forest["draft_rank"] = rng.choice([big, big, big - 1, 0, np.iinfo(np.int32).min], forest["N"]).astype(np.int32)
    dev = [torch.as_tensor(x).cuda() for x in (zp, zq, rp, rq)]
    exempt = decisions = 0
    for step in range(10):
        prm["step"] = step
        gpu, status = run_gpu_verify(forest, prm, *dev)
        assert status == 0
        e, d = compare_verify(_oracle(forest, prm, zp, zq, rp, rq), gpu, forest)
        exempt += e
        decisions += d
    check_exempt(exempt, decisions)


def _tampered(depth, beams, request, **arrays):
    """Three requests of `beams` chains of `depth` drafts; the call on the forest as it is, and on one whose device arrays differ
    (name = function of the array and of the first tree of `request`).  Returns the forest and both outputs with their status."""
    rng = np.random.default_rng(depth * beams)
    forest, prm, zp, zq, rp, rq, _ = _random_problem(rng, R=3, V=600, gamma=depth, max_w=beams, min_w=beams)
    prm.update(W_min=1, W_min_r=None, thresh=0.3)
    dev = [torch.as_tensor(x).cuda() for x in (zp, zq, rp, rq)]
    res = []
    for change in (False, True):
        f = dsbd.Forest(forest, "cuda")
        if change:
            for name, fn in arrays.items():
                x = forest[name].copy()
                fn(x, int(forest["req_beam_off"][request]))
                f.dev[name] = torch.as_tensor(x).cuda()
        out = dsbd.alloc_verify_out(f, oracle.default_out_off(forest, prm), "cuda")
        status = dsbd.verify_step(f, dict(prm), *dev, out)
        res.append(({k: v.cpu().numpy() for k, v in out.items()}, int(status.item())))
    return forest, prm, res


# nodes of a request: kept in shared memory (up to 256), scores by the writer's threads (up to 1024), by its trees' threads
REQUEST_SIZES = [(3, 6), (3, 64), (9, 30), (17, 64)]


def _others_unchanged(forest, prm, request, good, bad):
    out_off, bno, rbo = oracle.default_out_off(forest, prm), forest["beam_node_off"], forest["req_beam_off"]
    for r in set(range(forest["R"])) - {request}:
        w = good["out_width"][r]
        assert bad["out_width"][r] == w and bad["req_error"][r] == 0 and bad["l_last"][r] == good["l_last"][r]
        s, n = slice(out_off[r], out_off[r] + w), slice(bno[rbo[r]], bno[rbo[r + 1]])
        for k in ("out_parent", "out_node", "out_token", "out_root_beam", "out_source", "out_logp"):
            assert np.array_equal(good[k][s], bad[k][s]), (r, k)
        assert np.array_equal(good["node_status"][n], bad["node_status"][n])


@pytest.mark.parametrize("depth,beams", REQUEST_SIZES)
@pytest.mark.parametrize("tree,value", [(2, "empty"), (-1, "empty"), (1, 1 << 30), (1, -5), (-1, 1 << 30), (1, "next request")])
def test_tree_offsets_that_contradict_the_forest(depth, beams, tree, value):
    """A tree without nodes (inside, or the last one), a root far outside the forest, before it or in the next request: reported, the
    request is not verified, and the others are what they are without it."""
    def change(off, b0):
        t = b0 + (tree if tree > 0 else beams + tree)
        off[t] = {"empty": off[t + 1], "next request": off[b0 + beams] + 2}.get(value, value)
    forest, prm, ((good, ok), (bad, status)) = _tampered(depth, beams, 1, beam_node_off=change)
    assert ok == 0 and status == 4 and bad["req_error"].tolist() == [0, 4, 0]         # DSBD_DEV_BAD_FOREST
    assert bad["out_width"][1] == 0
    _others_unchanged(forest, prm, 1, good, bad)


@pytest.mark.parametrize("first,last", [(-1, None), (None, 1 << 30), (None, 0)])
def test_request_offsets_that_contradict_the_forest(first, last):
    """Requests whose trees lie outside the forest or end before they begin."""
    def change(off, b0):
        off[0 if first is not None else 3] = first if first is not None else last
    r = 0 if first is not None else 2
    forest, prm, ((good, ok), (bad, status)) = _tampered(3, 6, r, req_beam_off=change)
    assert ok == 0 and status == 4 and bad["req_error"][r] == 4 and bad["out_width"][r] == 0
    _others_unchanged(forest, prm, r, good, bad)


@pytest.mark.parametrize("depth,beams", REQUEST_SIZES)
def test_a_second_root_inside_a_tree(depth, beams):
    """A node behind its tree's first one that names no parent: reported, it stays unreached and no draft behind it is tested; the other
    requests are what they are without it."""
    n = (beams + 1) * (depth + 1) + 1                    # request 1, second tree, layer 1

    def change(parent, b0):
        parent[n] = -1
    forest, prm, ((good, ok), (bad, status)) = _tampered(depth, beams, 1, parent=change)
    bno = forest["beam_node_off"]
    assert n == bno[forest["req_beam_off"][1] + 1] + 1 and forest["parent"][n + 1] == n
    assert ok == 0 and status == 4 and bad["req_error"].tolist() == [0, 0, 0]
    assert bad["node_status"][n] == 0 and bad["node_status"][n + 1] in (0, 4)        # unreached, pruned
    assert not np.any(np.isin(bad["node_status"][n:bno[forest["req_beam_off"][1] + 2]], (1, 2, 3)))
    assert bad["out_width"][1] >= 1
    _others_unchanged(forest, prm, 1, good, bad)


@pytest.mark.parametrize("top_k", [0, 10])
def test_cluster_sizes_are_the_largest_of_which_all_requests_fit(top_k):
    """6 rows of 16 tiles: 16 CTAs to a request up to as many requests as the device says it holds such clusters, from one more on 8, and
    so on down to 1; fewer tiles, smaller clusters.  Clusters stay inside a GPC and two CTAs fit an SM."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count

    def asked(R, rows, V):
        arrays = dict(req_beam_off=None, beam_node_off=None, parent=None, token=None)
        f = dsbd.Forest.from_device(R, R, R, 1, {k: torch.zeros(4, dtype=torch.int32, device="cuda") for k in arrays}, 1, rows, rows)
        return dsbd.verify_cluster_ctas(f, dict(V=V, W_min=1, W_max=1, W_nom=1, top_k=top_k))

    R = 1
    for ctas in (16, 8, 4, 2):
        got, resident = asked(R, 6, 16384)
        assert got == ctas and sms // 2 < resident * ctas <= 2 * sms
        assert asked(resident, 6, 16384) == (ctas, resident)
        R = resident + 1
    assert asked(R, 6, 16384)[0] == 1
    assert [asked(1, rows, 16384)[0] for rows in (5, 4, 3, 2, 1)] == [8, 8, 4, 4, 2] and asked(1, 1, 15000)[0] == 1


def test_an_extra_layer_whose_support_does_not_fit():
    """300 tiles of equal bounds, more than the search for a support keeps: reported, no beam is drawn, and the width of the layer that was
    reached is told as for any other."""
    V, W = 300 * 1024, 2
    forest = dict(R=1, B=W, N=W, max_depth=0, req_beam_off=np.array([0, W], np.int32), beam_node_off=np.arange(W + 1, dtype=np.int32),
                  parent=np.full(W, -1, np.int32), token=np.zeros(W, np.int32))
    prm = dict(V=V, temperature=1.0, thresh=0.5, W_min=W, W_max=W, W_nom=5, seed=1, step=0, top_k=10, top_p=1.0)
    z, zero = torch.zeros(W, V, device="cuda"), torch.zeros(W, device="cuda")
    gpu, status = run_gpu_verify(forest, prm, z, z, zero, zero)
    assert status == 3 and gpu["req_error"][0] == 3                      # DSBD_DEV_CAPACITY
    assert gpu["l_last"][0] == 1 and gpu["out_width"][0] == 0
    assert gpu["layer_width"][0].tolist() == [5]


@pytest.mark.parametrize("V", [524289, 525312, 600001, 1050000])
def test_draws_from_the_last_of_a_row_s_tile_masses(V):
    """A draw from p_beam searches its row's tile masses 512 at a time: here most of each row's mass lies behind the first (second) 512, in
    one token, one tile, 74 and two tiles there."""
    rng = np.random.default_rng(V + 1)
    forest, prm, zp, zq, rp, rq, _ = _random_problem(rng, R=2, V=V, gamma=1, max_w=2, min_w=2)
    last = (V - 1) // (512 * 1024) * (512 * 1024)
    for z in (zp, zq):
        z[:, last:] += np.log(20.0 * V / (V - last)).astype(np.float32)
    dev = [torch.as_tensor(x).cuda() for x in (zp, zq, rp, rq)]
    exempt = decisions = behind = 0
    for step in range(8):
        prm.update(step=step, thresh=0.3, W_min=2, W_min_r=None, W_nom=8)
        gpu, status = run_gpu_verify(forest, prm, *dev)
        assert status == 0
        e, d = compare_verify(_oracle(forest, prm, zp, zq, rp, rq), gpu, forest)
        exempt += e
        decisions += d
        out_off = oracle.default_out_off(forest, prm)
        for r in range(2):
            s = slice(out_off[r], out_off[r] + gpu["out_width"][r])
            behind += int(((gpu["out_token"][s] >= last) & (gpu["out_source"][s] >= 2)).sum())        # fills, extra draws
    check_exempt(exempt, decisions)
    assert behind > 0
