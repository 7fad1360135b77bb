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


def test_persistent_anneal_starts_no_cta_without_a_run(so):
    """Items come chunk by chunk, R runs each: a grid of at most R CTAs takes
    only first chunks to begin with, whatever the GPU holds at a time."""
    f = getattr(so, "_ZN2pc8sqa_gridEiii")   # pc::sqa_grid(int, int, int)
    f.restype, f.argtypes = ctypes.c_int, [ctypes.c_int] * 3
    for resident in (1, 152, 304, 3648):
        for R in (1, 2, 151, 153, 200, 304, 456, 4000, 100000):
            for chunks in (1, 2, 24):
                assert f(resident, R, R * chunks) == min(resident, R)


def test_small_graphs_with_cluster_moves_stay_on_one_cta(so):
    """Two labels on two CTAs: always without cluster moves, with them from 8
    warps beyond the first of each colour class per attempt on (32 colours of
    32 vertices: none)."""
    f = getattr(so, "_ZN2pc15gapt_split_paysEiii")   # pc::gapt_split_pays(int, int, int)
    f.restype, f.argtypes = ctypes.c_bool, [ctypes.c_int] * 3
    for more in (0, 1, 4, 7, 8, 30, 127):
        for spp in (1, 2, 4, 10, 2 ** 31 - 1):
            assert f(more, spp, 0)
            assert f(more, spp, 1) == (more * spp >= 8)


def test_the_largest_cta_stages_swap_tables(so):
    """64 replicas of a 16^3 lattice with cluster moves and 32 temperatures fit
    a CTA's 232,448 bytes with 64 swap-table entries per pair, not with 256: the
    shorter length is the last one a schedule needs."""
    f = getattr(so, "_ZN2pc14apt_smem_bytesEiiiiiii")   # pc::apt_smem_bytes(N, groups, mode, icm, T, n_bins, entries)
    f.restype, f.argtypes = ctypes.c_size_t, [ctypes.c_int] * 7
    assert f(4096, 8, 0, 1, 32, 0, 64) == 226448 <= 232448 < f(4096, 8, 0, 1, 32, 0, 256)
    assert max(f(n, g, 0, i, t, 0, 64) for n in (8, 1728, 4096) for g in range(1, 9) for i in (0, 1)
               for t in (1, 9, 32)) == 226448
