"""The C-ABI library without a GPU: it loads, exports every symbol the headers
declare, computes Philox on the host like the oracle, and rejects bad
arguments on the host before touching CUDA."""
import ctypes
import os
import re

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PKG = os.path.join(ROOT, "paper_2508_15371_gb300")


def _built(name):
    path = os.path.join(PKG, name)
    if not os.path.exists(path):
        from paper_2508_15371_gb300 import build
        build.build()
    return path


def _declared(header):
    src = open(os.path.join(ROOT, "include", header)).read()
    src = re.sub(r"/\*.*?\*/", "", src, flags=re.S)
    return sorted(set(re.findall(r"\b(cmsd_\w+)\s*\(", src)))


@pytest.mark.parametrize("header,lib", [("cmsd.h", "libcmsd.so"), ("cmsd_workload.h", "libcmsd_workload.so")])
def test_library_exports_every_declared_symbol(header, lib):
    L = ctypes.CDLL(_built(lib))
    names = _declared(header)
    assert names
    for n in names:
        assert hasattr(L, n), f"{lib} does not export {n}"


def test_no_load_is_multicast_to_a_cluster():
    # every rank of a multi-GPU program loads this one library, and a bulk load
    # that writes several CTAs' shared memory is unsafe there
    csrc = os.path.join(PKG, "csrc")
    for f in sorted(os.listdir(csrc)):
        code = re.sub(r"//[^\n]*", "", open(os.path.join(csrc, f)).read())
        assert "multicast::cluster" not in code, f


@pytest.fixture(scope="module")
def cmsd():
    _built("libcmsd.so")
    from paper_2508_15371_gb300 import cmsd as c
    c.lib()
    return c


def test_host_philox_matches_oracle(cmsd):
    from oracle import philox
    rng = np.random.default_rng(3)
    for _ in range(300):
        seed = int(rng.integers(0, 2 ** 63))
        c = [int(x) for x in rng.integers(0, 2 ** 32, 4)]
        want = philox.philox4x32_10(c, philox.seed_key(seed))
        for wd in range(4):
            assert cmsd.philox_u32(seed, *c, wd) == want[wd]


def test_params_default(cmsd):
    p = cmsd.params(8, "paper")
    assert (p.k_min, p.k_max, p.beta_rank, p.tau_sign, p.rule) == (1, 8, 3, 1, 0)
    assert abs(p.tau_base - 0.1) < 1e-7 and abs(sum(p.lam) - 1) < 1e-6
    s = cmsd.params(16, "sampled")
    assert (s.k_max, s.beta_rank, s.rule) == (16, 0, 1)


def _call_conf(cmsd, draft=8192, B=2, K=4, V=100, dtype=1, p=None):
    p = p if p is not None else cmsd.params(K)
    L = cmsd.lib()
    return L.cmsd_confidence(ctypes.c_void_p(draft) if draft else None, B, K, V, dtype, None,
                             ctypes.byref(p) if p is not False else None,
                             None, None, None, None, None, None, None, 0, None)


def test_argument_errors_rejected_on_host(cmsd):
    assert _call_conf(cmsd, B=0) == cmsd.OK                 # empty call: nothing to do
    assert _call_conf(cmsd, K=0) == cmsd.OK
    assert _call_conf(cmsd, V=1) == cmsd.EINVAL
    assert _call_conf(cmsd, B=-1) == cmsd.EINVAL
    assert _call_conf(cmsd, K=2000) == cmsd.EINVAL
    assert _call_conf(cmsd, dtype=7) == cmsd.EDTYPE
    assert _call_conf(cmsd, draft=0) == cmsd.EINVAL
    assert _call_conf(cmsd, draft=8200) == cmsd.EALIGN
    assert _call_conf(cmsd, p=False) == cmsd.EINVAL
    assert _call_conf(cmsd, B=1 << 20, K=1024, V=1 << 20) == cmsd.EINVAL   # B*K*V >= 2^46
    for bad in (dict(k_min=0), dict(k_min=5, k_max=4), dict(lam=(0.5, 0.5, 0.5)),
                dict(lam=(1.2, -0.1, -0.1)), dict(beta_sig=0.0), dict(alpha=0.0),
                dict(alpha=1.5), dict(beta_rank=-1), dict(tau_sign=0), dict(tau_base=float("inf"))):
        assert _call_conf(cmsd, p=cmsd.params(4, **bad)) == cmsd.EINVAL, bad


def test_verify_argument_errors(cmsd):
    L = cmsd.lib()
    p = cmsd.params(4, "sampled")
    a = ctypes.c_void_p(4096)
    # sampled rule needs draft_lse
    rc = L.cmsd_verify(a, a, a, None, 2, 4, 100, 1, ctypes.byref(p), a, None, 0, 0, a, a, None,
                       None, 0, None)
    assert rc == cmsd.EINVAL
    p.rule = 5
    rc = L.cmsd_verify(a, a, a, None, 2, 4, 100, 1, ctypes.byref(p), a, a, 0, 0, a, a, None,
                       None, 0, None)
    assert rc == cmsd.EDTYPE
    q = cmsd.params(4, "paper")
    rc = L.cmsd_confidence_verify(a, ctypes.c_void_p(4100), a, None, 2, 4, 100, 1, ctypes.byref(q), 0, 0,
                                  None, None, None, None, None, None, a, a, None, None, 0, None)
    assert rc == cmsd.EALIGN
    rc = L.cmsd_confidence_verify(a, a, a, None, 2, 4, 100, 1, ctypes.byref(q), 0, 0,
                                  None, None, None, None, None, None, None, a, None, None, 0, None)
    assert rc == cmsd.EINVAL          # n_accept is required
    assert L.cmsd_strerror(cmsd.ENOWS).decode().startswith("workspace")


def test_product_path_fails_loudly_without_library(tmp_path, monkeypatch):
    from paper_2508_15371_gb300 import cmsd as c
    monkeypatch.setattr(c, "LIB_PATH", str(tmp_path / "missing.so"))
    monkeypatch.setattr(c, "_lib", None)
    with pytest.raises(c.CmsdError):
        c.lib()


def test_ablation_presets(cmsd):
    # the variants of the ablation (Sec. IV, Table III) as parameter sets
    full = cmsd.params(16, "sampled")
    assert (full.k_fixed, full.bonus) == (0, 0)
    fk = cmsd.params(16, "sampled", preset="fixed_k")
    assert fk.k_fixed == 16 and abs(fk.gamma - 1.0) < 1e-7
    ft = cmsd.params(16, "sampled", preset="fixed_tau")
    assert ft.k_fixed == 0 and ft.gamma == 0.0
    fkt = cmsd.params(16, "sampled", preset="fixed_k_tau")
    assert fkt.k_fixed == 16 and fkt.gamma == 0.0
    for name, j in (("entropy_only", 0), ("margin_only", 1), ("softmax_only", 2)):
        q = cmsd.params(16, "paper", preset=name)
        assert list(q.lam) == [1.0 if k == j else 0.0 for k in range(3)]
    p = cmsd.Params()
    assert cmsd.lib().cmsd_params_preset(ctypes.byref(p), 8, 0, 99) == cmsd.EINVAL


def test_bonus_and_fixed_k_argument_checks(cmsd):
    # k_fixed outside [k_min, k_max] and a bonus row with rows that are not a
    # whole number of 16-byte vectors are refused on the host
    L = cmsd.lib()
    a = ctypes.c_void_p(1 << 20)
    bad_k = cmsd.params(8, "paper", k_fixed=9)
    rc = L.cmsd_confidence_verify(a, a, a, None, 2, 8, 4096, cmsd.BF16, ctypes.byref(bad_k), 0, 0,
                                  None, None, None, None, None, None, a, a, None, None, 0, None)
    assert rc == cmsd.EINVAL
    odd = cmsd.params(8, "paper", bonus=1)
    rc = L.cmsd_confidence_verify(a, a, a, None, 2, 8, 4097, cmsd.BF16, ctypes.byref(odd), 0, 0,
                                  None, None, None, None, None, None, a, a, None, None, 0, None)
    assert rc == cmsd.EINVAL


def test_lmhead_refuses_tensors_of_another_device(cmsd, monkeypatch):
    import torch

    class OnDevice:
        """What lmhead_confidence asks of a tensor before it launches."""
        is_cuda = True

        def __init__(self, shape, index):
            self.shape, self.device, self._index = shape, torch.device("cuda", index), index

        def is_contiguous(self):
            return True

        def element_size(self):
            return 2

        def get_device(self):
            return self._index

    monkeypatch.setattr(torch.cuda, "current_device", lambda: 0)
    for dh, dw in ((1, 1), (0, 1), (1, 0)):
        with pytest.raises(cmsd.CmsdError, match="current device"):
            cmsd.lmhead_confidence(OnDevice((4, 64), dh), OnDevice((100, 64), dw))


CONF, VERIFY, FUSED = 0, 1, 2


def _choose(cmsd, resident, call, B, K, V, dtype=1, rule=1, bonus=0, ragged=0, sms=152):
    """(CTAs per sequence, threads) of the one-launch kernel, (0, 0) for the
    streaming kernel, on a device of sms SMs with these resident clusters [2, 17]."""
    table = np.ascontiguousarray(resident, np.int32)
    nc, th = ctypes.c_int32(-1), ctypes.c_int32(-1)
    rc = cmsd.lib().cmsd_test_choose(call, B, K, V, dtype, rule, bonus, ragged, sms, table.ctypes.data,
                                     ctypes.byref(nc), ctypes.byref(th))
    assert rc == cmsd.OK
    assert th.value in ((256, 512) if nc.value else (512, 768))
    return (nc.value, th.value) if nc.value else (0, 0)


def _stream_threads(cmsd, call, B, K, V, dtype=1, rule=1, ragged=0):
    table = np.zeros((2, 17), np.int32)               # no cluster fits: the streaming kernel
    nc, th = ctypes.c_int32(-1), ctypes.c_int32(-1)
    assert cmsd.lib().cmsd_test_choose(call, B, K, V, dtype, rule, 0, ragged, 152, table.ctypes.data, ctypes.byref(nc),
                                       ctypes.byref(th)) == cmsd.OK and nc.value == 0
    return th.value


def test_choice_of_kernel_where_one_cluster_fits(cmsd):
    # a small partition of a device: one cluster of each size at a time, or of
    # the large sizes only one and of the small ones as many as there is room
    one = np.ones((2, 17), np.int32)
    room = np.stack([16 // np.maximum(1, np.arange(17)), 8 // np.maximum(1, np.arange(17))])
    for resident in (one, room, np.minimum(room, 2)):
        for call in (CONF, VERIFY, FUSED):
            for rule in (0, 1):
                for B, K, V in ((1, 4, 32000), (1, 16, 128256), (2, 8, 128256), (16, 8, 32001), (300, 2, 8000)):
                    for dtype in (0, 1):
                        for ragged in (0, 1):
                            nc, th = _choose(cmsd, resident, call, B, K, V, dtype, rule, 0, ragged)
                            assert (nc, th) == (0, 0) or resident[1 if th == 512 else 0][nc] >= 1
    assert _choose(cmsd, np.zeros((2, 17)), FUSED, 1, 4, 32000) == (0, 0)
    assert _choose(cmsd, one, FUSED, 1, 17, 32000) == (0, 0)


def test_choice_of_kernel_counts_the_devices_own_sms(cmsd):
    # clusters as 16 SMs hold them: 25 CTAs of 256 threads share these SMs, and
    # the streaming kernel is faster; on 152 SMs each would have one to itself
    n = np.maximum(1, np.arange(17))
    resident = np.stack([32 // n, 16 // n])
    assert _choose(cmsd, resident, VERIFY, 5, 2, 128256, rule=0, sms=152) == (5, 256)
    assert _choose(cmsd, resident, VERIFY, 5, 2, 128256, rule=0, sms=16) == (0, 0)


def test_launch_plan_argument_errors_and_empty_calls(cmsd):
    p = cmsd.params(8, "sampled")
    for call in (CONF, VERIFY, FUSED):
        assert cmsd.launch_plan(call, 0, 8, 32000, cmsd.BF16, p) == (0, 0, 0)
    for bad in (dict(call=3), dict(call=-1), dict(V=1), dict(K=2000), dict(p=cmsd.params(8, k_min=0)),
                dict(V=4097, p=cmsd.params(8, bonus=1))):
        kw = dict(call=FUSED, B=0, K=8, V=32000, dtype=cmsd.BF16, p=p)
        kw.update(bad)
        with pytest.raises(cmsd.CmsdError):
            cmsd.launch_plan(**kw)


# Clusters of 1 .. 16 CTAs that a GB300 of 152 SMs holds at once, of 256 and of 512 threads.
GB300 = np.array([[0, 304, 152, 97, 74, 58, 46, 38, 36, 30, 28, 0, 23, 0, 0, 0, 14],
                  [0, 152, 76, 46, 36, 28, 23, 15, 15, 15, 13, 0, 8, 0, 0, 0, 7]])


@pytest.mark.parametrize("call,K,V,rule,bonus", [(VERIFY, 12, 32001, 1, 0), (VERIFY, 12, 32001, 0, 0),
                                                 (VERIFY, 8, 128256, 1, 0), (FUSED, 8, 128256, 1, 0),
                                                 (FUSED, 8, 32128, 0, 0), (FUSED, 4, 32001, 1, 0),
                                                 (FUSED, 8, 64128, 1, 1), (CONF, 8, 32001, 0, 0)])
def test_ragged_windows_get_a_place_each(cmsd, call, K, V, rule, bonus):
    # windows given by k_row may all be full: a cluster without a place would
    # then run after the others, in twice the time
    for B in range(1, 201):
        nc, th = _choose(cmsd, GB300, call, B, K, V, 1, rule, bonus, ragged=1)
        assert nc < 2 or B <= GB300[1 if th == 512 else 0][nc], (B, nc, th)


def test_choice_of_kernel_off_vector_boundaries(cmsd):
    # cluster_race takes half the share off 16-byte boundaries that it takes on
    # them: 16 CTAs of 256 threads race a row of 152064 entries, not one of 152063
    assert 152064 > 4 * 16 * 256 * 8
    assert _choose(cmsd, GB300, VERIFY, 10, 1, 152064) == (16, 256)
    assert _choose(cmsd, GB300, VERIFY, 10, 1, 152063) == (10, 512)


def _draw(cmsd, B, V, dtype, rule, bonus, resident):
    table = np.ascontiguousarray(resident, np.int32)
    n = ctypes.c_int32(-9)
    assert cmsd.lib().cmsd_test_draw(B, V, dtype, rule, bonus, table.ctypes.data, ctypes.byref(n)) == cmsd.OK
    return n.value


def test_choice_of_the_second_kernel(cmsd):
    # the sides measured on a GB300: (B, V, dtype, rule, bonus) -> CTAs per sequence, 0 the staged draw
    bf16, f32 = [74, 148, 304], [36, 148, 304]
    for args, resident, want in [
            ((40, 128256, 1, 1, 0), bf16, 0), ((100, 128256, 1, 1, 0), bf16, 0), ((100, 32000, 1, 1, 0), bf16, 4),
            ((40, 128255, 0, 1, 0), f32, 0), ((80, 128256, 0, 1, 0), f32, 4), ((180, 128255, 0, 1, 0), f32, 4),
            ((180, 128255, 1, 1, 0), bf16, 0), ((180, 128256, 1, 1, 0), bf16, 4), ((300, 128255, 1, 1, 0), bf16, 4),
            ((300, 128256, 1, 1, 0), bf16, 2), ((180, 32000, 1, 1, 0), bf16, 2), ((600, 152063, 1, 1, 0), bf16, 2),
            ((130, 128256, 1, 1, 1), bf16, 4), ((152, 128256, 1, 1, 1), bf16, 2), ((450, 128256, 1, 0, 1), bf16, 4),
            ((450, 32000, 1, 0, 1), bf16, 2)]:
        assert _draw(cmsd, *args, resident) == want, args
    # rows whose shares do not fit: no staged draw, no half row per CTA, no cluster at all
    assert _draw(cmsd, 8, 1_000_000, 1, 1, 0, [0, 148, 304]) == 4
    assert _draw(cmsd, 600, 1_500_000, 1, 1, 0, [0, 148, 0]) == 4
    assert _draw(cmsd, 600, 3_100_000, 1, 1, 0, [0, 0, 0]) == -1


def test_choice_of_kernel_counts_the_draws_share(cmsd):
    # one CTA a sequence would take a whole long row's draw (B=167 K=1 V=128255
    # f32 verify: 93.0 us, streamed 44.8; B=240 K=1 V=152063 fused: 72.3, 49.9)
    for args in ((VERIFY, 167, 1, 128255, 0), (VERIFY, 155, 1, 152063, 1), (FUSED, 240, 1, 152063, 1),
                 (FUSED, 300, 2, 128255, 0), (FUSED, 400, 2, 64127, 1)):
        assert _choose(cmsd, GB300, *args) == (0, 0), args
    assert _choose(cmsd, GB300, FUSED, 64, 8, 128256) == (4, 256)


def test_choice_of_kernel_prices_ragged_streaming(cmsd):
    # (B=310 K=1 V=8000 PAPER, windows of 0 and 1: 11.5 us streamed, 6.6 in one
    # launch; B=155 K=2 V=32001 PAPER verify 9.7, 7.0)
    assert _choose(cmsd, GB300, FUSED, 310, 1, 8000, 1, 0, 0, ragged=1) == (1, 256)
    assert _choose(cmsd, GB300, VERIFY, 155, 2, 32001, 1, 0, 0, ragged=1)[0] > 0
    # (B=32 K=16 V=32000 f32 sampled, windows of a third on average 19.5 us
    # streamed, 17.0 by eights; spread over 0..K 26.8, 24.7; full 35.2, 29.1)
    assert _choose(cmsd, GB300, FUSED, 32, 16, 32000, 0, 1, 0, ragged=1) == (8, 256)


def test_short_rows_crossed_by_slices_take_more_warps(cmsd):
    # 2432 warps of 512 threads per SM: 2400 and 1190 rows in whole pieces, 816,
    # 2880 and 7200 not
    for B, K, want in ((100, 24, 512), (70, 17, 512), (48, 17, 768), (180, 16, 768), (300, 24, 768)):
        for call, rule in ((FUSED, 0), (FUSED, 1), (CONF, 0), (VERIFY, 0), (VERIFY, 1)):
            assert _stream_threads(cmsd, call, B, K, 8000, rule=rule) == want, (B, K, call, rule)
        assert _stream_threads(cmsd, FUSED, B, K, 128256) == 512                    # long rows
        assert _stream_threads(cmsd, FUSED, 2 * B, K, 8000, ragged=1) == want       # half full on average
    assert _stream_threads(cmsd, CONF, 300, 24, 32000) == 512 and _stream_threads(cmsd, FUSED, 300, 24, 32000) == 768
    assert _stream_threads(cmsd, FUSED, 300, 24, 8000, dtype=0) == 768
    assert _stream_threads(cmsd, FUSED, 300, 24, 32000, dtype=0) == 512
    assert _stream_threads(cmsd, FUSED, 1 << 20, 1024, 8000) == 768
