"""Host logic of the autotuner around the automatic choice (no GPU): whether that
choice is the series, and that a shape tuned with it is not handed to a chain
without it."""
import pytest

from paper_2210_06874_gb300 import autotune, hmc

BASE = dict(L=6, Nt=32, beta=4.0, precision=hmc.PREC_MIXED)
# same lattice and delta, but no series: 3 |delta kappa| > 4, mass preconditioning, a
# cluster mode of the tensor-core tiles
WITHOUT = [dict(kappa=11.0), dict(hb_inner=2, hb_gamma=0.5), dict(cluster_mode=1),
           dict(cluster_mode=2)]


def test_series_feasible():
    assert autotune.series_feasible(hmc.Params(**BASE))
    for kw in WITHOUT + [dict(L=28)]:
        assert not autotune.series_feasible(hmc.Params(**{**BASE, **kw})), kw


@pytest.mark.parametrize("kw", WITHOUT)
def test_cached_shape_is_not_shared(monkeypatch, kw):
    """tune() and tune_ru() with the automatic shape in their caches for BASE must
    measure again for a chain without the series (here: reach the device)."""
    class Measured(Exception):
        pass

    def measure(*_):
        raise Measured
    monkeypatch.setattr(autotune.torch.cuda, "current_device", measure)
    a, b = hmc.Params(**BASE), hmc.Params(**BASE, **kw)
    monkeypatch.setattr(autotune, "_cache", {})
    monkeypatch.setattr(autotune, "_ru_cache", {})
    for f, cache, value in ((autotune.tune, autotune._cache, ((0, 0, 0, 0), 1e-5)),
                            (autotune.tune_ru, autotune._ru_cache, 0.01)):
        keys = []

        class Spy(dict):
            def __contains__(self, key):
                keys.append(key)
                return super().__contains__(key)
        spy = Spy(cache)
        monkeypatch.setattr(autotune, "_cache" if f is autotune.tune else "_ru_cache", spy)
        with pytest.raises(Measured):
            f(a)
        spy[keys[-1]] = value
        assert f(a).operand_mode == 0          # served from the cache
        with pytest.raises(Measured):
            f(b)
