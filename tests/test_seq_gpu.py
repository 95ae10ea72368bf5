"""The one-launch pass (a cluster per sequence) against the streaming kernel.

Windows of at most 16 positions of small and medium problems are taken by one
kernel with a thread-block cluster per sequence; wider windows by the
streaming kernel and its second pass.  The uniforms depend on (sequence,
position, iteration) only, so the same rows in a wider window (K = 17, its
last position never present) must give the same decisions, bit for bit, and
signals equal up to the rounding of 32-bit sums added in another order.
Both are compared with the oracle elsewhere (test_gpu_parity).
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

# Each logarithm, sum and quotient of a signal is good to a few units of 2^-24
# of values up to ln V < 12: 16 such units.  C adds three terms of at most 1.
SIGNAL_TOL = 16 * 12 * 2.0 ** -24


@pytest.fixture(scope="module")
def cmsd():
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2508_15371_gb300 import cmsd as c
    c.lib()
    return c


def _inputs(B, K, V, dtype, bonus, masked, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    Kt = K + 1 if bonus else K
    z = 1.5 * torch.randn((B, Kt, V), generator=g, device="cuda")
    at = torch.randint(0, V, (B, Kt, 1), generator=g, device="cuda")
    z.scatter_add_(2, at, 8.0 * torch.rand((B, Kt, 1), generator=g, device="cuda"))
    t = z + torch.randn((B, Kt, V), generator=g, device="cuda")
    if masked:
        off = torch.rand((V,), generator=g, device="cuda") < 0.4
        off[:2] = False
        z[:, :, off] = -float("inf")
        t[:, :, off] = -float("inf")
    dt = torch.float32 if dtype == "f32" else torch.bfloat16
    e = torch.rand((B, K, V), generator=g, device="cuda").clamp_(1e-9, 1 - 1e-7)
    z = z.to(dt)
    tok = (z[:, :K].float() - torch.log(-torch.log(e))).argmax(dim=2).to(torch.int32)
    return z[:, :K].contiguous(), t.to(dt), tok


def _widen(x, extra):
    """The same rows with `extra` more (of zeros) at the end of each window."""
    pad = torch.zeros((x.shape[0], extra) + tuple(x.shape[2:]), dtype=x.dtype, device=x.device)
    return torch.cat([x, pad], dim=1).contiguous()


def _same(narrow, wide, k_row, bonus):
    K = narrow["out_tokens"].shape[1] - (1 if bonus else 0)
    for b, kb in enumerate(k_row.tolist()):
        assert int(narrow["n_accept"][b]) == int(wide["n_accept"][b])
        assert torch.equal(narrow["out_tokens"][b], wide["out_tokens"][b, :K + (1 if bonus else 0)]), (b, kb)
        if "accept" in narrow:
            assert torch.equal(narrow["accept"][b], wide["accept"][b, :K])
        if "k_next" in narrow:
            assert int(narrow["k_next"][b]) == int(wide["k_next"][b])
        for n in ("H", "margin", "conf", "lse"):
            if n in narrow and kb:
                d = (narrow[n][b, :kb] - wide[n][b, :kb]).abs().max().item()
                assert d <= SIGNAL_TOL, (n, b, d)
        if "argmax" in narrow and kb:
            assert torch.equal(narrow["argmax"][b, :kb], wide["argmax"][b, :kb])


def _in_one_launch(cmsd, d, t, tok, p, k_row, cluster, threads):
    """The fused pass by the one-launch kernel, whatever the rule says."""
    call = cmsd.FusedCall(d, t, tok, p, seed=9, iteration=3, k_row=k_row, signals=True)
    rc = cmsd.lib().cmsd_test_confidence_verify_cluster(
        *call._head, 9, 3, *call._tail, torch.cuda.current_stream().cuda_stream, cluster, threads)
    assert rc == cmsd.OK
    return call.out


# Sizes: no whole vector, one group, lines and pieces that end inside a row,
# draws of one and of two blocks of groups per lane set (B=32) and by bounds
# (B=64).  Which cluster sizes they take depends on the rule; every size is
# asked for below.
SHAPES = [(1, 1, 2), (3, 2, 33), (2, 16, 1000), (1, 4, 32000), (5, 7, 4099), (8, 8, 32128), (40, 3, 8193),
          (70, 5, 6400), (150, 2, 4096), (700, 1, 2048), (2, 8, 128256),
          (32, 2, 64128), (32, 2, 128256), (64, 2, 128255)]


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
@pytest.mark.parametrize("rule", ["paper", "sampled"])
@pytest.mark.parametrize("B,K,V", SHAPES)
def test_one_launch_equals_streaming(cmsd, B, K, V, rule, dtype):
    es = 4 if dtype == "f32" else 2
    for bonus in ([False, True] if (V * es) % 16 == 0 else [False]):
        d, t, tok = _inputs(B, K, V, dtype, bonus, masked=V >= 1000 and B % 2 == 0, seed=V + B)
        rng = np.random.default_rng(V)
        k_row = torch.from_numpy(rng.integers(0, K + 1, B).astype(np.int32)).cuda()
        k_row[0] = K
        W = 17 - K
        p = cmsd.params(K, rule, bonus=bonus, tau_base=-0.5)
        pw = cmsd.params(K, rule, bonus=bonus, tau_base=-0.5)     # the same draft-length bounds
        d2, tok2 = _widen(d, W), _widen(tok[:, :, None], W)[:, :, 0].contiguous()
        t2 = _widen(t, W)
        full = torch.full((B,), K, dtype=torch.int32, device="cuda")
        for kr in (k_row, None):
            a = cmsd.confidence_verify(d, t, tok, k_row=kr, p=p, seed=9, iteration=3)
            b = cmsd.confidence_verify(d2, t2, tok2, k_row=full if kr is None else kr, p=pw, seed=9, iteration=3)
            _same(a, b, full if kr is None else kr, bonus)
            code = cmsd.F32 if dtype == "f32" else cmsd.BF16
            if cmsd.launch_plan(cmsd.FUSED, B, K, V, code, p, kr is not None)[1] == 0:
                _same(_in_one_launch(cmsd, d, t, tok, p, kr, 1, 256), b, full if kr is None else kr, bonus)
        kr = k_row
        sig = cmsd.confidence(d, k_row=kr, p=p)
        sig2 = cmsd.confidence(d2, k_row=kr, p=pw)
        for i, kb in enumerate(kr.tolist()):
            assert int(sig["k_next"][i]) == int(sig2["k_next"][i])
            assert torch.equal(sig["argmax"][i, :kb], sig2["argmax"][i, :kb])
        conf = sig["conf"].nan_to_num(0.5).clamp(0, 1)
        lse = sig["lse"].nan_to_num(0.0)
        a = cmsd.verify(d, t, tok, conf, draft_lse=lse, k_row=kr, p=p, seed=9, iteration=4)
        b = cmsd.verify(d2, t2, tok2, _widen(conf[:, :, None], W)[:, :, 0].contiguous(),
                        draft_lse=_widen(lse[:, :, None], W)[:, :, 0].contiguous(), k_row=kr, p=pw, seed=9, iteration=4)
        _same(a, b, kr, bonus)


@pytest.mark.parametrize("threads", [256, 512])
@pytest.mark.parametrize("cluster", [1, 2, 3, 4, 5, 6, 7, 8, 9, 10, 12, 16])
def test_every_cluster_size_equals_streaming(cmsd, cluster, threads):
    """The fused pass by the one-launch kernel with each cluster size, on
    windows of odd and of aligned rows, against the streaming kernel."""
    for B, K, V, dtype, rule, bonus in ((3, 5, 4099, "bf16", "sampled", False), (2, 16, 20008, "bf16", "paper", True),
                                        (2, 3, 32001, "f32", "paper", False), (2, 7, 65536, "f32", "sampled", True),
                                        (1, 4, 128256, "bf16", "sampled", True)):
        d, t, tok = _inputs(B, K, V, dtype, bonus, masked=B == 2, seed=V + cluster)
        p = cmsd.params(K, rule, bonus=bonus, tau_base=-0.5)
        k_row = torch.tensor([K, max(0, K - 3), 0][:B], dtype=torch.int32, device="cuda")
        full = torch.full((B,), K, dtype=torch.int32, device="cuda")
        W = 17 - K
        d2, t2, tok2 = _widen(d, W), _widen(t, W), _widen(tok[:, :, None], W)[:, :, 0].contiguous()
        for kr in (None, k_row):
            a = _in_one_launch(cmsd, d, t, tok, p, kr, cluster, threads)
            wide = cmsd.confidence_verify(d2, t2, tok2, k_row=full if kr is None else kr, p=p, seed=9, iteration=3)
            _same(a, wide, full if kr is None else kr, bonus)


def test_cluster_sizes_that_are_refused(cmsd):
    d, t, tok = _inputs(1, 17, 1024, "bf16", False, False, seed=1)
    for K, cluster, threads in ((17, 1, 256), (4, 11, 256), (4, 0, 256), (4, 17, 512), (4, 2, 128)):
        call = cmsd.FusedCall(d[:, :K].contiguous(), t[:, :K].contiguous(), tok[:, :K].contiguous(),
                              cmsd.params(K, "sampled"))
        rc = cmsd.lib().cmsd_test_confidence_verify_cluster(
            *call._head, 0, 0, *call._tail, torch.cuda.current_stream().cuda_stream, cluster, threads)
        assert rc == cmsd.EDTYPE, (K, cluster, threads)


def test_launch_plan_is_what_runs(cmsd):
    """The plan against the library's own events: a second interval is longer
    than the microsecond or two between events around nothing only where a
    second kernel ran."""
    p = cmsd.params(8, "sampled")
    assert cmsd.launch_plan(cmsd.FUSED, 4, 8, 4096, cmsd.BF16, p)[0] == 1
    for K, rule, launches in ((8, "sampled", 1), (17, "sampled", 2), (17, "paper", 1)):
        p = cmsd.params(K, rule)
        n, nc, th = cmsd.launch_plan(cmsd.FUSED, 4, K, 128256, cmsd.BF16, p)
        assert (n, nc > 0, th in (256, 512)) == (launches, K <= 16, True)
        d, t, tok = _inputs(4, K, 128256, "bf16", False, False, seed=K)
        cmsd.confidence_verify(d, t, tok, p=p)
        torch.cuda.synchronize()
        cmsd.profile_start(20)
        for i in range(20):
            cmsd.confidence_verify(d, t, tok, p=p, iteration=i)
        _, second = cmsd.profile_stop(20)
        assert (np.median(second) > 0.0035) == (launches == 2), (K, rule, np.median(second))


def test_device_errors_are_reported(cmsd):
    """Out-of-range tokens and windows are clamped and set their bits."""
    d, t, tok = _inputs(3, 4, 4096, "bf16", False, False, 1)
    p = cmsd.params(4, "sampled")
    ws = cmsd.workspace(3, 4, 4096)
    cmsd.workspace_errors(ws)
    cmsd.confidence_verify(d, t, tok, p=p, ws=ws)
    assert cmsd.workspace_errors(ws) == 0
    tok[1, 2] = 4096
    cmsd.confidence_verify(d, t, tok, p=p, ws=ws)
    assert cmsd.workspace_errors(ws) == 1
    tok[1, 2] = 0
    cmsd.confidence_verify(d, t, tok, p=p, ws=ws, k_row=torch.tensor([4, -1, 5], dtype=torch.int32, device="cuda"))
    assert cmsd.workspace_errors(ws) == 2


@pytest.mark.parametrize("noise,bonus", [(1.0, False), (0.0, False), (1.0, True)])
def test_rows_beyond_every_share(cmsd, noise, bonus):
    """Rows whose share fits no CTA's shared memory take the race over every
    group (noise 0: target equal to drafter, whose empty residual is the
    target's argmax)."""
    from parity_util import bonus_view, compare, gpu_fused, oracle_fused
    from paper_2508_15371_gb300 import workloads as W
    B, K, V = 2, 2, 3_100_000
    rng = np.random.default_rng(3)
    d = rng.normal(0, 1.0, (B, K + 1, V)).astype(np.float32)
    t = d + np.float32(noise) * rng.normal(0, 1.0, d.shape).astype(np.float32) if noise else d.copy()
    t[:, :, 77] += 9.0 if noise else 0.0
    Kt = K + 1 if bonus else K
    tok = rng.integers(0, V, (B, K)).astype(np.int32)
    w = W.Workload(name="wide", B=B, K=K, V=V, dtype="bf16", draft=W.f32_to_bf16_bits(d[:, :K]),
                   target=W.f32_to_bf16_bits(t[:, :Kt]), tokens=tok, seed=5)
    p = cmsd.params(K, "sampled", bonus=bonus, tau_base=30.0 if bonus else -5.0)
    g = gpu_fused(cmsd, torch, w, p, iteration=2)
    compare(w, g, oracle_fused(w, p, iteration=2))
    assert (g["n_accept"] == K).any() if bonus else (g["n_accept"] < K).any()


def _tie_pairs(V, es, most, seed):
    """(lower, upper) entries for rows 0, 1, ... of a tensor of V-entry rows: two
    that one lane of a piece reads in both of its ways, singly and in a
    16-byte vector.

    A piece starts at a whole 128-byte line from its row's start and ends at
    one, or at V; its unaligned tail goes to the lanes 31, 30, ..., its
    unaligned head to the lanes 0, 1, ....  The lanes of the vectors depend on
    the starting line modulo four, so four starts stand for all.  `most`
    candidates for each of the rows' places off 16-byte boundaries, those at
    the row's end always among them.
    """
    rng = np.random.default_rng(seed)
    vec, line = 16 // es, 128 // es
    classes = []
    for mis in range(vec):
        ends, rest = [], []
        for end in list(range(line, V, line)) + [V]:
            for back in range(1, (end + mis) % vec + 1):
                lane = 32 - back
                for f in range(4):
                    va = f * line + (-(f * line + mis)) % vec        # the piece's first whole vector
                    j = (end - (end + mis) % vec - vec - va) // vec  # and its last one, from there
                    j -= (j - lane) % 32
                    for t in (j, j - 32):
                        if t >= 0:
                            (ends if end == V else rest).append((va + t * vec + int(rng.integers(0, vec)), end - back))
        for start in range(0, V - 33 * vec, line):
            for lane in range(-(start + mis) % vec):
                va = start + (-(start + mis)) % vec
                rest.append((start + lane, va + lane * vec + int(rng.integers(0, vec))))
        rest = [rest[k] for k in rng.permutation(len(rest))[:max(0, most - len(ends))]]
        classes.append(ends + rest or [(V // 2, V - 1)])
    n = vec * max(len(c) for c in classes)
    return [classes[r * V % vec][r // vec % len(classes[r * V % vec])] for r in range(n)]


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
@pytest.mark.parametrize("V,most", [(129, 60), (257, 60), (4099, 800), (32001, 400)])
def test_ties_off_vector_boundaries_take_the_lowest_index(cmsd, V, most, dtype):
    """A maximum at two entries of a row, one read by itself and one in a
    vector of the same lane: the argmax, and the PAPER rule's correction, is
    the lower of the two.  Batches of several sizes, so that rows are cut into
    pieces of several lengths."""
    es = 4 if dtype == "f32" else 2
    pairs = _tie_pairs(V, es, most, seed=V + es)
    n = len(pairs)
    # rows 0 .. n - 1 of the tensor; a batch is a run of rows that starts on a
    # 16-byte boundary (every 8th row), so a row keeps its place off them
    g = torch.Generator(device="cuda").manual_seed(V)
    dt = torch.float32 if dtype == "f32" else torch.bfloat16
    z = (4.0 * torch.rand((n, V), generator=g, device="cuda") - 4.0).to(dt)
    rows = torch.arange(n, device="cuda")
    low, high = torch.tensor(pairs, device="cuda").T
    assert (low >= 0).all() and (low < high).all() and (high < V).all()
    z[rows, low] = 9.0
    z[rows, high] = 9.0
    want = low.to(torch.int32)
    p = cmsd.params(1, "paper", beta_rank=0, tau_base=0.0, gamma=0.0)      # accepts the maximum alone
    sizes, at = [8, 32, 64, 152, 1], 0
    while at < n:
        B = min(sizes[0], n - at)
        sizes = sizes[1:] + sizes[:1]
        x = z[at:at + B].view(B, 1, V)
        tok = ((want[at:at + B] + 1) % V).view(B, 1)
        tok = torch.where(x[:, 0].gather(1, tok.long()) == 9.0, (tok + 1) % V, tok)
        a = cmsd.confidence(x)
        f = cmsd.confidence_verify(x, x, tok, p=p)
        v = cmsd.verify(x, x, tok, a["conf"], p=p)
        for name, got in (("confidence", a["argmax"]), ("fused", f["argmax"]), ("fused token", f["out_tokens"]),
                          ("verify token", v["out_tokens"])):
            bad = (got[:, 0] != want[at:at + B]).nonzero()[:, 0]
            assert len(bad) == 0, (name, B, [(pairs[at + int(k)], int(got[int(k), 0])) for k in bad[:4]])
        at += (B + 7) // 8 * 8


@pytest.mark.parametrize("dtype,rule,bonus", [("bf16", "sampled", False), ("bf16", "paper", True), ("f32", "paper", False),
                                              ("f32", "sampled", True)])
@pytest.mark.parametrize("V", [1003, 2048, 8000])
def test_short_rows_in_large_batches_equal_small_ones(cmsd, V, dtype, rule, bonus):
    """Rows that the streaming kernel's slices cross the ends of take its
    variant of 768 threads and two vectors a stage; the same sequences alone
    take whole pieces and 512 threads.  The draws depend on (sequence,
    position, iteration), so decisions are the same and signals differ by the
    rounding of sums in another order."""
    if bonus and (V * (4 if dtype == "f32" else 2)) % 16:
        bonus = False
    B, K, few = 170, 17, 5
    d, t, tok = _inputs(B, K, V, dtype, bonus, masked=V == 2048, seed=V)
    p = cmsd.params(K, rule, bonus=bonus, tau_base=-0.5)
    code = cmsd.F32 if dtype == "f32" else cmsd.BF16
    rng = np.random.default_rng(V)
    k_row = torch.from_numpy(rng.integers(0, K + 1, B).astype(np.int32)).cuda()
    k_row[0], k_row[1] = K, 0
    small = [x[:few].contiguous() for x in (d, t, tok, k_row)]
    for ragged in (False, True):
        assert cmsd.launch_plan(cmsd.FUSED, few, K, V, code, p, ragged)[1:] == (0, 512)
        if not ragged:
            assert cmsd.launch_plan(cmsd.FUSED, B, K, V, code, p, ragged)[1:] == (0, 768)
        a = cmsd.confidence_verify(d, t, tok, k_row=k_row if ragged else None, p=p, seed=9, iteration=3)
        b = cmsd.confidence_verify(*small[:3], k_row=small[3] if ragged else None, p=p, seed=9, iteration=3)
        a = {n: x[:few] for n, x in a.items()}
        kr = small[3] if ragged else torch.full((few,), K, dtype=torch.int32)
        _same(a, b, kr, bonus)
        big, one = cmsd.confidence(d, k_row=k_row if ragged else None, p=p), cmsd.confidence(
            small[0], k_row=small[3] if ragged else None, p=p)
        for i, kb in enumerate(kr.tolist()):
            assert int(big["k_next"][i]) == int(one["k_next"][i])
            assert torch.equal(big["argmax"][i, :kb], one["argmax"][i, :kb])
        conf, lse = big["conf"].nan_to_num(0.5).clamp(0, 1), big["lse"].nan_to_num(0.0)
        a = cmsd.verify(d, t, tok, conf, draft_lse=lse, k_row=k_row if ragged else None, p=p, seed=9, iteration=4)
        b = cmsd.verify(*small[:3], conf[:few].contiguous(), draft_lse=lse[:few].contiguous(),
                        k_row=small[3] if ragged else None, p=p, seed=9, iteration=4)
        _same({n: x[:few] for n, x in a.items()}, b, kr, bonus)
