"""The rule that chooses between the two forms of the two-slice hop (staged links, or
direction by direction), as the launcher and the block plan call it. No GPU."""
import ctypes as C

import pytest

FP64, FP32, FP16, BF16 = 0, 1, 2, 3
ANY = 100000  # fields enough for any number of waves


@pytest.fixture(scope="module")
def rule():
    from paper_1811_08488_gb300 import build
    lib = C.CDLL(build.build())
    f = getattr(lib, "_ZN3dwf16hop_staged_sitesEi8dwf_preciiiixi")  # dwf::hop_staged_sites
    f.restype = C.c_int
    f.argtypes = [C.c_int] * 6 + [C.c_longlong, C.c_int]
    return lambda Ls, p, dag, pre, nd, n, fields=1, sms=152: f(Ls, p, dag, pre, nd, n, fields, sms)


def sites_per_cta(Ls):
    return 4 * (32 // (Ls // 2))


@pytest.mark.parametrize("p", [FP64, FP32, FP16, BF16])
@pytest.mark.parametrize("dag,pre", [(0, 0), (0, 1), (1, 0)])
def test_few_lanes_per_link_are_not_staged(rule, p, dag, pre):
    for Ls in (2, 4, 3, 7, 9):
        staged = Ls == 4 and p in (FP16, BF16) and pre  # two lanes with M_phi on load
        assert rule(Ls, p, dag, pre, 4096, 4096, ANY) == (4096 if staged else 0)
        assert rule(Ls, p, dag, pre, 2048, 4096, ANY) == 0
    if p == FP64:
        assert rule(12, p, dag, pre, 4096, 4096, ANY) == 0


@pytest.mark.parametrize("p", [FP32, FP16, BF16])
@pytest.mark.parametrize("Ls", [6, 8, 12, 14, 16, 24, 32])
def test_all_sites(rule, p, Ls):
    n = 10 * sites_per_cta(Ls) - 1  # ten CTAs, the last partly filled
    for dag, pre in ((0, 0), (0, 1), (1, 0)):
        waves = 2
        if p != FP32:
            waves = 0 if pre or Ls >= 8 else None
        elif Ls >= (24 if pre else 12):
            waves = 0
        for sms in (100, 152):
            fields = -(-max(waves or 0, 0) * 4 * sms // 10) or 1
            if waves is None:
                assert rule(Ls, p, dag, pre, n, n, ANY, sms) == 0
                continue
            assert rule(Ls, p, dag, pre, n, n, fields, sms) == n
            if waves:
                assert rule(Ls, p, dag, pre, n, n, fields - 1, sms) == 0
    assert rule(Ls, p, 0, 1, 0, n, ANY) == 0  # no site has its neighbours


@pytest.mark.parametrize("p,pre,waves", [(FP16, 1, 3), (BF16, 1, 3), (FP32, 0, 24)])
@pytest.mark.parametrize("Ls", [6, 12, 16])
def test_some_sites(rule, p, pre, waves, Ls):
    per = sites_per_cta(Ls)
    dense, n = 5 * per + 1, 9 * per  # six CTAs, the last one reaching into the others
    for sms in (100, 152):
        fields = -(-waves * 4 * sms // 6)
        assert rule(Ls, p, 0, pre, dense, n, fields, sms) == 6 * per
        assert rule(Ls, p, 0, pre, dense, n, fields - 1, sms) == 0
        assert rule(Ls, p, 1, 0, dense, n, ANY, sms) == 0  # adjoint hops: all or none
        assert rule(Ls, p, 0, 1 - pre, dense, n, ANY, sms) == 0
    # rounded up to whole CTAs, never past the sites that there are
    assert rule(Ls, p, 0, pre, 8 * per + 1, 9 * per - 1, ANY) == 9 * per - 1
