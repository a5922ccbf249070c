"""Who decodes a group: the rules of the decoder's launch, asked without a GPU."""
import pytest

from paper_2112_04291_b200 import binding, build

N = 1 << 26                        # entries, more than the L2 holds


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()


def _route(mode=0, streams=8, n=N, group_log2=14, owned=13, mean=0, keys=None, words=None, bulk=True):
    keys = mean if keys is None else keys
    return binding.debug_decoder_route(mode, streams, n, group_log2, owned, mean, keys, -(-keys * 15 // 32) if words is None else words, bulk)


@pytest.mark.parametrize("mode", [0, 1, 2, 3])
def test_groups_of_few_keys_go_to_a_warp_and_unlike_large_ones_to_the_block(mode):
    assert _route(mode, keys=248) == "warp" and _route(mode, keys=249) == "block"
    assert _route(mode, streams=1, n=1 << 24, keys=1024) == "warp" and _route(mode, streams=1, n=1 << 24, owned=7, keys=257) == "block"
    assert _route(mode, group_log2=16, keys=10) == "wide block" and _route(mode, streams=1, group_log2=17, keys=10) == "wide block"


@pytest.mark.parametrize("mode,line", [(0, 400), (1, 400), (2, 256), (3, 400)])
def test_ranks_from_a_mean_on(mode, line):
    assert _route(mode, mean=line) == "four warps by ranks" and _route(mode, mean=line - 1) == "warp"
    assert _route(mode, mean=line, owned=4) == ("four warps" if mode == 0 else "four warps by ranks")
    assert _route(mode, mean=line - 1, owned=8) == ("two warps" if mode != 2 else "four warps by ranks")


def test_aggregation_over_the_slice_from_a_mean_on():
    assert _route(mean=999) == "four warps by ranks" and _route(mean=1000) == "block over the slice"


def test_groups_wider_than_the_slice_stay_with_teams():
    for mean in (1000, 1500, 1800):
        assert _route(group_log2=15, mean=mean, words=mean // 2) == "four warps by ranks", mean
    assert _route(group_log2=15, mean=1000, owned=4) == "four warps"


def test_no_slice_early_where_it_moves_in_words():
    for mean in (1000, 1500, 2000):
        assert _route(mean=mean, bulk=False) == "four warps by ranks", mean
    for streams in (1, 3):
        assert _route(streams=streams, owned=7, keys=1535, bulk=False) == "block"
        assert _route(streams=streams, owned=7, keys=1536, bulk=False) == _route(streams=streams, owned=7, keys=768) == "block over the slice"


def test_one_stream_over_a_vector_that_the_l2_holds():
    for n, line in ((8_000_000, 1536), (15_000_000, 1536), (15_000_001, 900), (20_000_000, 900), (20_000_001, 768)):
        assert _route(streams=1, n=n, owned=7, keys=line - 1) == "block", n
        assert _route(streams=1, n=n, owned=7, keys=line) == "block over the slice", n
        assert _route(streams=2, n=n, owned=7, keys=768) == "block over the slice", n


@pytest.mark.parametrize("mode", [0, 1, 2, 3])
def test_teams_of_four_take_what_their_memory_holds(mode):
    # a team's memory: 4 x 6144 bytes.  Ranks: 6 bytes a word of the bit map, 8 an entry, the blobs and 7 words; the table: 8 KiB, 6 bytes an
    # entry (even numbers of entries in both), the blobs and 3 words
    for group_log2, words in ((14, 1000), (11, 900), (8, 700)):
        most = (24576 - 6 * (1 << group_log2) // 32 - 4 * (words + 7)) // 16 * 2
        by_ranks = dict(mode=mode, group_log2=group_log2, mean=999 if mode == 0 else 1200, words=words)
        assert _route(keys=most, **by_ranks) == "four warps by ranks" and _route(keys=most + 1, **by_ranks).startswith("block")
    if mode == 0:
        most = (24576 - 8192 - 4 * (1000 + 3)) // 12 * 2
        assert _route(owned=4, mean=999, keys=most, words=1000) == "four warps" and _route(owned=4, mean=999, keys=most + 1, words=1000).startswith("block")


def test_update_over_the_slice_of_g_from_a_mean_on():
    for streams, line in ((2, 1400), (3, 1600), (4, 1800), (5, 2000), (8, 2000)):
        assert _route(2, streams, mean=line - 1, words=900) == "four warps by ranks" and _route(2, streams, mean=line, words=900) == "block", streams
        assert _route(2, streams, mean=line, words=900, bulk=False) == _route(3, streams, mean=line, words=900) == "four warps by ranks", streams
    assert _route(2, 2, group_log2=15, mean=1500, words=900) == "four warps by ranks"


def test_two_entries_a_lane_in_flight_only_where_memory_is_the_bound():
    two = "warp, two in flight"
    assert _route(streams=1, n=1 << 28, owned=55, keys=164) == two
    assert _route(streams=1, n=1 << 28, owned=55, keys=511) == two and _route(streams=1, n=1 << 28, owned=55, keys=512) == "warp"
    assert _route(streams=1, n=(1 << 25) + 1, group_log2=12, owned=28, keys=100) == two
    assert _route(streams=1, n=1 << 25, group_log2=12, owned=28, keys=100) == "warp"
    assert _route(streams=1, n=1 << 26, owned=16, keys=100) == "warp"


def test_no_teams_of_two_in_the_update_in_one_launch():
    for owned, mean in ((8, 200), (8, 255), (13, 150)):
        assert _route(2, owned=owned, mean=mean, keys=2 * mean, words=900 if owned == 13 else 100) == "four warps by ranks", owned
        assert _route(3, owned=owned, mean=mean, keys=2 * mean, words=900 if owned == 13 else 100) == "two warps", owned
