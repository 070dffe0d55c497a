"""The choice of planes per chunk (csrc/waves.h) against its own cost model counted out wave by wave: full
chunks fill whole waves, the tiles' last, shorter chunks the free slots of the last one and then as
many waves as they need, however many tiles there are."""
import ctypes
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2211_15634_gb300", "csrc")


@pytest.fixture(scope="module")
def chunk(tmp_path_factory):
    d = tmp_path_factory.mktemp("waves")
    src, lib = d / "w.cpp", d / "libw.so"
    src.write_text('#include "waves.h"\n'
                   'extern "C" int chunk(long long nz, long long tiles, int sms, int per_sm, double extra, double one,'
                   ' double later, int least, int most) {\n'
                   '    return psd::wave_chunk_of(nz, tiles, sms, per_sm, psd::WaveCost{extra, one, later, least, most});\n}\n')
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, str(src), "-o", str(lib)], check=True)
    fn = ctypes.CDLL(str(lib)).chunk
    fn.argtypes = [ctypes.c_longlong] * 2 + [ctypes.c_int] * 2 + [ctypes.c_double] * 3 + [ctypes.c_int] * 2
    return fn


def cost(c, nz, tiles, sms, per_sm, extra, one, later):
    """The planes that the slots are held for, wave by wave."""
    def wave(q):  # a wave of q CTAs
        per = -(-q // sms)
        return one + (1.0 - one) * (per - 1) / (per_sm - 1)

    slots, (n, rem) = sms * per_sm, divmod(nz, c)
    total, left, waves = 0.0, tiles * n, 0
    while left >= slots:
        total, left, waves = total + c + extra, left - slots, waves + 1
    short = tiles if rem else 0
    if short <= (slots - left if left else 0):  # they end within the last wave
        total += wave(left + short) * (rem + extra) + wave(left) * (c - rem) if short else wave(left) * (c + extra) if left else 0.0
        short = 0
    elif left:
        total, short = total + (c + extra if short else wave(left) * (c + extra)), max(0, short - (slots - left))
    while short > 0:
        q = min(short, slots)
        total, short = total + (1.0 if q == slots else wave(q)) * (rem + extra), short - q
    return total * (1.0 - later if waves else 1.0)


@pytest.mark.parametrize("nz,tiles", [(3, 4000), (4, 2000), (5, 1995), (10, 1677), (7, 460), (48, 300), (126, 16), (61, 700),
                                      (17, 3000), (200, 90), (256, 130), (33, 457), (100, 456)])
@pytest.mark.parametrize("per_sm,extra,one,later,least,most", [(2, 2.0, 0.6, 0.0, 2, 64), (3, 0.5, 0.6, 0.05, 3, 40),
                                                               (5, 2.0, 0.6, 0.2, 3, 12)])
def test_choice_is_the_cheapest(chunk, nz, tiles, per_sm, extra, one, later, least, most):
    sms = 152
    got = chunk(nz, tiles, sms, per_sm, extra, one, later, least, most)
    if tiles * -(-nz // least) <= sms:
        assert got == least
        return
    costs = {c: cost(c, nz, tiles, sms, per_sm, extra, one, later) for c in range(least, min(most, nz) + 1)}
    assert costs[got] <= min(costs.values()) * (1 + 1e-9), (got, costs)
