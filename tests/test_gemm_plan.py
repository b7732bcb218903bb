"""CPU tests of the GEMM's launch plan (Sec. 4.2, Eq. 7): the kernel, tile shape and split of K that qvla_w4a4_linear's GEMM
takes for M > 128 tokens, read through qvla_debug_gemm_plan (host logic only, no GPU).

The plan is a launch-time estimate fitted to GB300 measurements; these tests pin the decisions the measurements justified and
the rules around them:
  * the backbone's down projection (816 x 16384 -> 2048) runs CTA pairs on whole 128-token tiles, the weights in TMEM (26.2 us
    against 38.0 for the token-major kernel's CTA pairs with K in 2 work units);
  * few tiles of many k-blocks split: 256 x 16384 -> 2048 into 4 units;
  * from K = 768 every launch takes that kernel; below, the estimates weigh it against the token-major kernel;
  * gated layers never split (their epilogue pairs gate and up rows of one accumulator);
  * without the workspace room for the partials every launch runs whole tiles, and with it a split stays within that room;
  * a unit keeps at least 8 k-blocks, and a split is taken only where it is estimated 10% faster;
  * launches whose tiles already fill the SMs run whole tiles."""

import random

import pytest

from paper_2605_28803_gb300 import qvla as Q

SMS = 152  # GB300


def plan(M, K, N, gated=False, room=True, sms=SMS):
    return Q.qvla_debug_gemm_plan(M, K, N, gated=gated, num_sms=sms, split_room=room)


def test_down_projection_runs_whole_tiles_of_128_tokens():
    assert plan(816, 16384, 2048) == ("tmem 128x256", 1)


def test_few_tiles_split_in_four():
    assert plan(256, 16384, 2048) == ("tmem 128x256", 4)
    assert plan(150, 16384, 2048) == ("tmem 96x256", 4)  # a ragged token tile


def test_ragged_shapes_of_the_split_tests():
    # the shapes tests/test_gpu_split_k.py runs bit-identical against whole tiles
    assert plan(300, 16384, 2000) == ("tmem 160x256", 4)
    assert plan(700, 16384, 1904) == ("tmem 192x256", 2)
    assert plan(256, 14080, 2048) == ("tmem 128x256", 4)  # 110 k-blocks: units of 27 and 28
    assert plan(400, 14080, 2048) == ("tmem 128x256", 2)  # units of 55
    assert plan(129, 16384, 16) == ("tmem 160x256", 4)  # one tile


def test_gated_layers_never_split():
    # the backbone's gate/up projection: 2 x 16384 weight rows
    assert plan(816, 2048, 32768, gated=True) == ("tmem 192x256", 1)
    for M in (129, 256, 816):
        assert plan(M, 16384, 2048, gated=True)[1] == 1


@pytest.mark.parametrize("M,K,N", [(816, 16384, 2048), (256, 16384, 2048), (300, 16384, 2000), (700, 16384, 1904)])
def test_no_room_means_whole_tiles(M, K, N):
    assert plan(M, K, N, room=False)[1] == 1


def test_units_keep_eight_k_blocks():
    # K = 2048 has 16 k-blocks and could run units of 8, K = 4096 in 2 or 4, but the estimates gain less than 10%
    assert plan(816, 2048, 2048)[1] == 1
    assert plan(256, 2048, 2048)[1] == 1
    assert plan(150, 4096, 2048)[1] == 1
    for K in range(128, 16385, 128):
        for M in (129, 150, 300, 700):
            assert plan(M, K, 512)[1] == 1 or K // 128 // plan(M, K, 512)[1] >= 8


def test_full_waves_run_whole_tiles():
    for M, K, N in [(3200, 16384, 2048), (8192, 16384, 2048), (8192, 2048, 16384), (3200, 1024, 4096)]:
        assert plan(M, K, N)[1] == 1


def test_from_k_768_the_weights_are_in_tmem():
    rng = random.Random(1)
    for _ in range(300):
        M, N = rng.randint(129, 4096), 16 * rng.randint(1, 1024)
        assert plan(M, 128 * rng.randint(6, 128), N)[0].startswith("tmem ")
        assert not plan(M, 128 * rng.randint(1, 5), N)[0].startswith("pair ")


def test_few_k_blocks_go_by_the_estimates():
    assert plan(1600, 384, 1024) == ("single 128x128", 1)
    assert plan(1500, 128, 4112) == ("single 128x256", 1)
    assert plan(485, 384, 19968) == ("tmem 128x256", 1)
    assert plan(131, 384, 21760) == ("tmem 160x256", 1)


def test_a_split_stays_within_the_workspace_room():
    # the room: 4 partials of every output with rows and weight rows padded to 256, a count a 128 x 128 tile; a tile of w
    # tokens x 256 weight rows takes two counts
    rng = random.Random(2)
    split = 0
    for _ in range(2000):
        M, K, N = rng.randint(129, 1200), 128 * rng.randint(16, 128), 16 * rng.randint(1, 256)
        shape, parts = plan(M, K, N)
        if parts == 1:
            continue
        split += 1
        w = int(shape.split()[1].split("x")[0])
        tiles = -(-M // w) * -(-N // 256)
        assert tiles * parts * 2 * 128 * w <= 4 * (-(-M // 256) * 256) * (-(-N // 256) * 256)
        assert 2 * tiles <= -(-M // 128) * -(-N // 128)
    assert split > 100


def test_fewer_sms_change_the_plan_not_its_rules():
    assert plan(816, 16384, 2048, sms=76) == ("tmem 96x256", 1)
    for M, K, N in [(816, 16384, 2048), (256, 16384, 2048), (150, 16384, 2048)]:
        for sms in (76, 132, 152, 160):
            shape, parts = plan(M, K, N, sms=sms)
            assert parts in (1, 2, 4)
            assert 16384 // 128 // parts >= 8


def test_plan_refuses_bad_arguments():
    for args in [(128, 1024, 1024), (816, 1000, 1024), (816, 1024, 1000), (816, 1024, 1024 + 128)]:
        gated = args == (816, 1024, 1024 + 128)
        with pytest.raises(Q.QvlaError) as e:
            plan(*args, gated=gated)
        assert e.value.status == 1
    with pytest.raises(Q.QvlaError):
        plan(816, 1024, 1024, sms=1)
