"""How projections are cut: the choice is made on the host from sizes and from how many clusters the device holds, so it is
checked without one, with the counts of a B200."""
import ctypes

import pytest

import paper_2512_20687_b200 as ph
from paper_2512_20687_b200 import build

B200_CLUSTERS = (0, 148, 74, 45, 33, 26, 22, 15, 15)        # resident at a time, of 1 to 8 CTAs
RING, QUAD, MAX_STAGES = 208 * 1024, 32 * 16 * 4, 12


def cut(B, K, N, gated=False, clusters=B200_CLUSTERS):
    build.build_library()
    out = (ctypes.c_int32 * 4)()
    ph.load().photon_internal_projection_cut((ctypes.c_int32 * 9)(*clusters), B, K, N, int(gated), out)
    return tuple(out)


@pytest.mark.parametrize("gated", [False, True])
def test_every_cut_is_one_the_kernel_can_run(gated):
    for B in (1, 16, 17, 32, 33, 64, 65, 128, 129, 300, 600, 1204, 2048):
        x_rows = 128 if B > 64 else 64 if B > 32 else 32 if B > 16 else 16
        quarters = max(1, x_rows // 32)
        for K in (64, 128, 192, 256, 704, 1024, 2048, 2816, 4096, 5632, 8192, 12224, 16384):
            for N in (64, 128, 192, 256, 320, 512, 1024, 1472, 2048, 3072, 4096, 4736, 8192, 11264):
                if gated and N % 128:
                    continue
                nt, ks, stages, mma_warps = cut(B, K, N, gated)
                what = (B, K, N, nt, ks, stages)
                assert nt in (64, 128, 256) and N % nt == 0 and not (gated and nt != 128), what
                groups = nt // 16
                assert 1 <= ks <= min(8, groups) and K // 64 >= ks, what                # every CTA has columns to finish and a block of K
                # each MMA warp comes back to a stage after one phase of its barriers, not two
                assert mma_warps == (2 if nt == 64 else 1) and stages % mma_warps == 0, what
                blocks = 2 if nt <= 128 else 1
                assert 2 <= stages <= MAX_STAGES and stages * blocks * (x_rows + nt) * 128 <= RING, what
                # an MMA reads 128 rows from the last x block
                assert (stages * blocks - 1) * x_rows * 128 + 128 * 128 <= RING, what
                # staging and receive areas of the exchange, side by side in the ring, for the widest share
                first = [groups * r // ks for r in range(ks + 1)]
                own = [b - a for a, b in zip(first, first[1:])]
                receive = (groups - groups // ks) * quarters * QUAD
                for o in own:
                    assert o >= 1 and (groups - o) * quarters * QUAD <= receive, what
                    assert ks == 1 or receive + (ks - 1) * o * quarters * QUAD <= RING, what


# Cuts that count as one wave where the clusters do not fit at once, or that pay for their exchange in every wave.
@pytest.mark.parametrize("B,K,N", [(300, 4096, 4096), (300, 2816, 1024), (300, 5632, 2048), (200, 2048, 1472), (640, 2048, 8192),
                                   (512, 2048, 11264), (1600, 8192, 2048), (1204, 4096, 4096), (1600, 2048, 3072)])
def test_a_split_does_not_cost_another_wave(B, K, N):
    nt, ks, _, _ = cut(B, K, N)
    tiles = N // nt * -(-B // 128)
    assert ks == 1 or tiles <= B200_CLUSTERS[ks], (nt, ks, tiles)


def test_clusters_that_the_device_does_not_hold_are_not_taken():
    for K, N in ((8192, 2048), (16384, 256), (5632, 2048)):
        assert cut(64, K, N, clusters=(0, 148, 74, 0, 0, 0, 0, 0, 0))[1] <= 2
        assert cut(64, K, N, clusters=(0, 148, 0, 0, 0, 0, 0, 0, 0))[1] == 1


def pair_cut(B, K, N, out_major, residual=False, gated=False, clusters=B200_CLUSTERS):
    build.build_library()
    out = (ctypes.c_int32 * 8)()
    ph.load().photon_internal_pair_cut((ctypes.c_int32 * 9)(*clusters), B, K, N, int(out_major), int(residual), int(gated), out)
    return tuple(out)


@pytest.mark.parametrize("out_major", [False, True])
def test_every_cut_for_pairs_covers_the_output_and_fits_the_ring(out_major):
    pairs = B200_CLUSTERS[2]
    for B in (1, 129, 256, 257, 300, 900, 1204, 2048, 4099, 16384):
        for K in (64, 256, 1024, 5632):
            for N in (64, 128, 448, 1024, 1408, 2048, 2112, 3072, 11264):
                _, nt, m_tiles, n_tiles, whole, pieces, stages, stage_bytes = pair_cut(B, K, N, out_major)
                what = (B, K, N, nt, whole, pieces)
                assert nt in (128, 192, 256) and m_tiles == -(-B // 256) and n_tiles == -(-N // nt), what
                tiles = m_tiles * n_tiles
                assert pieces == whole + 2 * (tiles - whole), what
                # halves are the last, partly filled round, and then fit one round
                assert whole == tiles or (whole == tiles // pairs * pairs and pieces - whole <= pairs), what
                # x rows and the weight columns that a stage's copies bring: N-major weights come 64 columns at a time
                columns = nt // 2 if out_major else -(-(nt // 2) // 64) * 64
                assert stage_bytes == (128 + columns) * 128 and stage_bytes % 1024 == 0, what
                assert 2 <= stages <= 8 and stages * stage_bytes <= 196 * 1024, what


def test_pairs_are_taken_for_many_rows_only_and_where_the_device_holds_them():
    for K, N in ((2048, 3072), (2048, 2048), (1024, 3072), (5632, 2048), (2048, 11264)):
        assert pair_cut(16384, K, N, True)[0] and not pair_cut(128, K, N, True)[0]
        assert not pair_cut(16384, K, N, True, clusters=(0, 148, 0, 0, 0, 0, 0, 0, 0))[0]


@pytest.mark.parametrize("B,K,N,residual", [(1600, 2048, 8192, False), (1540, 2048, 8192, False), (3334, 4096, 4096, True), (4737, 64, 2048, False)])
def test_pairs_are_taken_from_more_than_two_waves_on(B, K, N, residual):
    for out_major in (False, True):
        assert pair_cut(B, K, N, out_major, residual)[0]
