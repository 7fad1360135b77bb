"""Host rules that shape a launch, called in the built library by their C++
names: no GPU needed."""
import ctypes

import pytest


@pytest.fixture(scope="module")
def so():
    from paper_2503_10302_gb300 import build, pcomp
    build.build()
    return pcomp.lib()


def _chunks(so, H, Gc, tpb, pref):
    f = getattr(so, "_ZN2pc10apt_chunksEiiii")   # pc::apt_chunks(int, int, int, int)
    f.restype, f.argtypes = ctypes.c_int, [ctypes.c_int] * 4
    return f(H, Gc, tpb, pref)


@pytest.mark.parametrize("tpb", [64, 128, 256, 320, 384, 448, 512])
@pytest.mark.parametrize("Gc", range(1, 9))
def test_thread_chunks_are_applied_where_they_fit(so, Gc, tpb):
    """A requested number of thread chunks holds for whole warps and at least
    one replica group per chunk; otherwise, and for 0, the rule's own choice
    does, which fits too."""
    for H in (4, 32, 500, 2048):
        own = _chunks(so, H, Gc, tpb, 0)
        assert own in (1, 2, 4, 8) and own <= Gc and tpb % (32 * own) == 0
        for pref in (1, 2, 4, 8):
            fits = pref <= Gc and tpb % (32 * pref) == 0
            assert _chunks(so, H, Gc, tpb, pref) == (pref if fits else own)
