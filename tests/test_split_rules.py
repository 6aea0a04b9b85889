"""The rules that split work over a cluster's CTAs (csrc/split.h), on the CPU."""

from _split import rules, tiles


def test_a_sequences_shares_do_not_depend_on_the_launch_bound():
    """A chunked prefill's cluster is sized by the caller's bound of the context; the CTAs that
    a sequence uses are those of its own length, whatever the (larger) bound."""
    R = rules()
    for sms in (148, 152):
        for pairs in (1, 9, 18, 19, 37, 38, 39, 75, 76, 77, 152, 1000):
            for own in (1, 2, 5, 9, 10, 11, 12, 23, 24, 25, 47, 48, 400):
                alone = R.prefill_cluster(pairs, own, sms)
                for bound in (own, own + 1, 10, 12, 24, 48, 256, 1 << 20):
                    if bound >= own:
                        assert R.prefill_shares(own, R.prefill_cluster(pairs, bound, sms)) == alone


def test_prefill_clusters_fit_the_sms_and_every_size_occurs():
    R = rules()
    seen = set()
    for pairs in range(1, 200):
        for tiles in range(1, 80):
            n = R.prefill_cluster(pairs, tiles, 152)
            seen.add(n)
            assert n == 1 or (pairs * n <= 152 and tiles >= 10 and tiles // n >= 3)
    assert seen == {1, 2, 4, 8}


def test_backward_splits_keep_work_for_the_heaviest_tiles_ctas():
    R = rules()
    seen = set()
    for B, hq, hkv in ((1, 1, 1), (1, 8, 1), (2, 16, 2), (1, 32, 8), (8, 12, 12), (4, 16, 16)):
        for S in (1, 100, 129, 300, 528, 1000, 1921, 4096):
            for causal in (0, 1):
                n = R.backward_split(B, hq, hkv, S, causal, 152)
                seen.add(n)
                assert n == 1 or hq // hkv * tiles(S) >= 2 * n
    assert seen == {1, 2, 4, 8}
    assert R.backward_split(1, 12, 12, 1024, 1, 152) == 1   # measured: two CTAs a key tile are slower
