"""The rules that split work over a cluster's CTAs (csrc/split.h), on the CPU."""

from _split import rules


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
