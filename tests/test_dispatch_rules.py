"""The choice between the attention kernels, as the library's own functions make it (no GPU needed: 148 SMs are assumed without
one).  The cases stand on both sides of a rule's line, at sizes where the other kernel was measured to be slower in a step."""
import ctypes

import pytest


@pytest.fixture(scope="module")
def lib():
    from paper_2506_12035_b200 import build
    return ctypes.CDLL(build.build())


@pytest.mark.parametrize("n,S,dh,items,want", [
    # one item per SM or fewer: mma.sync with four query warps at head_dim 80 only
    (36, 2048, 64, 64, True), (48, 1088, 64, 144, True), (64, 1088, 64, 148, True), (41, 320, 64, 148, False),
    (64, 1088, 80, 144, False), (56, 640, 80, 96, False), (48, 1088, 80, 144, True), (65, 1088, 80, 144, True),
    # more items: the streams fill one another's gaps
    (48, 1088, 64, 149, True), (41, 1088, 64, 1024, True), (49, 320, 64, 2048, True), (64, 1088, 80, 149, True),
    (41, 320, 64, 2048, False), (32, 2048, 64, 2048, False)])
def test_streams_or_mma_sync(lib, n, S, dh, items, want):
    wins = lib._ZN6marche24attention_tc_stream_winsEiiiii
    wins.restype = ctypes.c_bool
    assert wins(n, S, dh, items, 48) is want
    assert wins(n, S, dh, items, 0) is (n > 0)                      # min_rows 0: wherever the caller asks for them


@pytest.mark.parametrize("n,S,dh,items,want", [
    (24, 128, 64, 512, True), (24, 128, 64, 576, False), (8, 100, 64, 592, False),       # two tiles, up to 32 rows
    (24, 64, 64, 592, True), (24, 192, 64, 592, True), (40, 128, 64, 2048, True),
    (8, 164, 80, 256, True), (8, 164, 80, 288, False), (24, 164, 80, 288, True), (8, 320, 80, 288, True)])
def test_keys_split_or_not(lib, n, S, dh, items, want):
    wins = lib._ZN6marche20attention_split_winsEiiii
    wins.restype = ctypes.c_bool
    assert wins(n, S, dh, items) is want


@pytest.mark.parametrize("n,S,dh,items,cs", [(64, 320, 80, 64, 1), (64, 320, 80, 32, 1), (64, 320, 80, 16, 4), (64, 320, 64, 64, 2), (48, 320, 80, 64, 2),
                                             (64, 448, 80, 64, 2)])
def test_ctas_per_item_of_the_split(lib, n, S, dh, items, cs):
    got_cs, got_nk = ctypes.c_int(), ctypes.c_int()
    plan = lib._ZN6marche20attention_split_planEiiiiPiS0_
    plan.restype = ctypes.c_bool
    assert plan(n, S, dh, items, ctypes.byref(got_cs), ctypes.byref(got_nk)) and got_cs.value == cs


@pytest.mark.parametrize("n,n_new,S,dh,items,want", [
    (0, 0, 320, 64, 8, False), (8, 33, 320, 64, 8, False), (300, 33, 1088, 64, 1024, False), (400, 1, 2048, 64, 2048, False),
    # one item per SM or fewer: the sequence has to be long enough for the launch to pay
    (16, 1, 128, 64, 128, False), (16, 1, 129, 64, 128, True), (64, 17, 192, 64, 16, False), (64, 17, 193, 64, 16, True),
    (16, 1, 100, 80, 128, False), (48, 1, 192, 80, 64, True), (96, 17, 192, 80, 32, False), (96, 16, 192, 80, 32, True),
    (100, 4, 320, 64, 128, False), (100, 4, 1088, 64, 128, False), (150, 20, 320, 64, 32, True), (97, 20, 128, 80, 16, True),
    # up to two per SM
    (41, 4, 192, 64, 288, False), (41, 4, 256, 64, 288, True), (16, 2, 192, 64, 288, True), (64, 9, 256, 64, 288, False),
    (64, 9, 320, 64, 288, True), (64, 18, 1088, 64, 288, False), (100, 9, 640, 64, 256, False), (100, 9, 1088, 64, 256, True),
    (151, 9, 320, 64, 256, False), (151, 9, 640, 64, 256, True), (320, 2, 320, 64, 192, True), (41, 9, 192, 80, 256, False),
    (56, 9, 128, 80, 256, True), (80, 26, 128, 80, 256, True), (24, 3, 128, 80, 256, True), (24, 3, 64, 80, 256, False),
    (16, 3, 640, 80, 256, True), (16, 3, 1088, 80, 256, False), (64, 20, 640, 64, 288, True), (64, 20, 320, 64, 288, False),
    # more: the plain kernel has to be far from the scoring one
    (64, 9, 1088, 64, 1024, False), (41, 5, 320, 80, 2048, False), (72, 10, 320, 64, 2048, True), (72, 24, 320, 64, 2048, False),
    (116, 24, 1088, 64, 1024, True), (320, 2, 320, 64, 2048, True), (320, 32, 320, 80, 2048, True)])
def test_scores_in_a_launch_of_their_own(lib, n, n_new, S, dh, items, want):
    wins = lib._ZN6marche21attention_scores_winsEiiiii
    wins.restype = ctypes.c_bool
    assert wins(n, n_new, S, dh, items) is want


@pytest.mark.parametrize("M,N,K,norm,want", [
    # with the LayerNorm: as many CTAs as run at once, a third more of 16 warps
    (16, 2304, 768, 1, True), (16, 3072, 768, 1, True), (16, 3840, 1280, 1, True), (1, 5120, 1280, 1, True), (16, 4608, 1536, 1, True),
    (16, 6144, 2048, 1, True), (16, 4992, 1664, 1, False), (16, 5760, 1920, 1, False), (1, 7168, 1792, 1, False), (16, 8192, 2048, 1, False),
    (16, 4096, 2048, 1, True),
    # without
    (16, 4608, 1536, 0, True), (16, 4864, 1536, 0, False), (1, 5120, 1280, 0, False), (1, 8192, 1024, 0, False), (8, 2560, 4096, 0, False),
    (8, 2048, 2048, 0, True), (9, 2048, 2048, 0, False), (16, 1024, 2048, 0, True), (16, 4608, 2048, 0, True), (16, 1280, 5120, 0, True),
    (1, 1536, 6144, 0, False), (16, 2048, 6144, 0, True), (16, 1024, 6144, 0, True),
    # two groups of rows, three
    (32, 768, 768, 0, True), (32, 3072, 1024, 1, False), (33, 768, 768, 0, False), (24, 1280, 2560, 0, False), (17, 1152, 1152, 0, False),
    (24, 1280, 768, 0, True), (32, 1024, 2048, 0, True)])
def test_projections_of_a_handful_of_rows(lib, M, N, K, norm, want):
    wins = lib._ZN6marche13gemm_few_winsEiiib
    wins.restype = ctypes.c_bool
    assert wins(M, N, K, ctypes.c_bool(norm)) is want


@pytest.mark.parametrize("n,S,dh,items,want", [
    # one unit per CTA; one round of four for two of three
    (116, 1088, 64, 148, 1), (116, 1088, 64, 149, 3), (80, 100, 80, 144, 1), (80, 129, 80, 144, 3), (64, 100, 64, 444, 3), (64, 100, 64, 445, 4),
    (320, 320, 64, 192, 4), (64, 100, 64, 593, 3), (320, 320, 80, 192, 3),
    # two rounds for three over long sequences
    (116, 511, 64, 1024, 3), (116, 512, 64, 1024, 4), (200, 1088, 64, 448, 4), (128, 2048, 64, 889, 4), (128, 2048, 64, 888, 3), (128, 2048, 64, 1185, 3),
    # three rounds for four, seven for ten: behind a short last tile
    (151, 1088, 64, 800, 4), (161, 1088, 64, 800, 3), (160, 1088, 64, 800, 4), (256, 1088, 64, 800, 3), (151, 895, 64, 800, 3), (151, 1088, 64, 2048, 4),
    (23, 1088, 64, 1600, 3), (151, 1088, 64, 1024, 3)])
def test_streams_per_cta(lib, n, S, dh, items, want):
    streams = lib._ZN6marche20attention_tc_streamsEiiii
    assert streams(n, S, dh, items) == want


@pytest.mark.parametrize("streams", [3, 4])
@pytest.mark.parametrize("items,n_qt", [(444, 1), (448, 1), (592, 1), (888, 1), (1184, 1), (2048, 1), (300, 3), (448, 2), (1024, 2), (2048, 2), (149, 9), (2048, 3),
                                        (512, 149)])
def test_units_are_dealt_once_and_evenly(lib, streams, items, n_qt):
    """Every unit to one CTA, as many to each but for one; no stream of many units gets tiles of one kind only.  Items of one tile
    stay in the CTAs' order, the last turn's on the first CTAs, up to two turns of the streams."""
    grid, units = 148, items * n_qt
    deal, turn = lib._ZN6marche21attention_tc_rotationEliiiPi, ctypes.c_int()
    rotate = deal(ctypes.c_long(units), n_qt, grid, streams, ctypes.byref(turn))
    if n_qt == 1:
        assert (rotate, turn.value) == ((0, 0) if units <= 2 * streams * grid else (1, 0))
    taken, kinds = set(), {}
    for k in range((units + grid - 1) // grid):
        for cta in range(grid):
            i = k * grid + (cta + k * rotate + k // streams * turn.value) % grid
            if i < units:
                assert i not in taken
                taken.add(i)
                kinds.setdefault((cta, k % streams), []).append(i % n_qt)
    assert len(taken) == units
    if 1 < n_qt < 9 and units >= 3 * streams * grid:
        assert all(len(set(v)) > 1 for v in kinds.values())
