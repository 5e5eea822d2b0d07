"""bench.py labels its kernels by what the timed solves ran, not by the grid's size."""
import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.mark.parametrize("n,route,ctas", [
    ({"single": 0, "two": 2000, "chip": 0}, "two", 152),
    ({"single": 1, "two": 999, "chip": 0}, "two", 152),         # an odd last step
    ({"single": 0, "two": 0, "chip": 250}, "chip", 152),
    ({"single": 16, "two": 0, "chip": 9}, "chip", 152),
    ({"single": 4000, "two": 0, "chip": 0}, "single", 76),
])
def test_route_and_codec_ctas(n, route, ctas):
    sys.path.insert(0, ROOT)
    import bench
    base = {"single": 7, "two": 3, "chip": 5}
    got = bench.route_of(base, {k: base[k] + v for k, v in n.items()})
    assert got == route and bench.codec_ctas(got, 152) == ctas
    for codec in ("time", "space") if route == "single" else ("time",):
        kind, name = bench.DOMINANT[route, codec]
        assert kind in bench.BYTES_PER_NODE and name
