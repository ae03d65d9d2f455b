"""Fixed launch tiles against the rules by shape: a fixed tile can be given back, a
saved one put back changes nothing, and the recorded tiles leave the rules alone."""
import pytest

import paper_1003_1898_gb300 as P
from paper_1003_1898_gb300 import build, tune


@pytest.fixture(scope="module")
def lib():
    build.build()
    yield P.lib()
    tune.load_and_apply()


def test_tiles_saved_and_restored_leave_the_shape_rules(lib):
    # A saved tile put back is a no-op, also when none was fixed; 0, 0, 0 gives a
    # fixed one back.
    slots = [(g, 0) for g in P.GEN_NAMES if g != "ranlux"] + [("ranlux", p) for p in (24, 48, 97, 223, 389, 120, 240, 408)]
    for gen, lux in slots:
        P.prng_set_tile(gen, lux, *tune.BY_SHAPE)
        saved = P.prng_get_tile(gen, lux)
        assert saved == tune.BY_SHAPE
        other = tune.tiles_for(gen, lux)[1]
        P.prng_set_tile(gen, lux, *other)
        assert P.prng_get_tile(gen, lux) == other
        fixed = P.prng_get_tile(gen, lux)
        P.prng_set_tile(gen, lux, *fixed)
        assert P.prng_get_tile(gen, lux) == other
        P.prng_set_tile(gen, lux, *saved)
        assert P.prng_get_tile(gen, lux) == tune.BY_SHAPE
        for bad in ((0, 0, 1), (0, 48, 0), (128, 0, 0)):
            with pytest.raises(P.PrngError) as e:
                P.prng_set_tile(gen, lux, *bad)
            assert e.value.code == -7
            assert P.prng_get_tile(gen, lux) == tune.BY_SHAPE


def test_recorded_tiles_leave_the_shape_rules(lib):
    # Applying the recorded tiles fixes one only where fills have no rule by shape;
    # a cache that names fixed tiles is honoured.
    for key, v in tune.load().items():
        gen = key.split("_")[0]
        assert (tuple(v["tile"]) == tune.BY_SHAPE) == (gen in tune.SHAPE_RULES), key
    try:
        tune.apply({"xor128": {"tile": [128, 64, 1]}, "ranlux_p223": {"tile": [64, 96, 1]}})
        assert P.prng_get_tile("xor128") == (128, 64, 1) and P.prng_get_tile("ranlux", 223) == (64, 96, 1)
    finally:
        tune.load_and_apply()
    assert P.prng_get_tile("xor128") == tune.BY_SHAPE and P.prng_get_tile("ranlux", 223) == tune.BY_SHAPE
