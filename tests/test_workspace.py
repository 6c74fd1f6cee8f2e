"""Workspace of a 256^3 member (no GPU needed): its fields, the partial sums of
the narrowest update tile, its counts, and one set of moment sums for each of
the 32 CTAs that its statistics pass has at most; 4 KB for the rest (run state,
moments, shells, alignment)."""
import paper_2506_23712_gb300.ens as E
from paper_2506_23712_gb300 import build as B


def test_moment_partials_follow_the_statistics_pass():
    B.build()
    h = E.hist_spec(qr_bins=16, tail_bins=32)
    small = E.Member(N=16, nu=0.02, k_lo=1, k_hi=2).c()
    big = E.Member(N=256, nu=0.02, k_lo=1, k_hi=2).c()
    per_member = E.ens_query([small, big, big], h) - E.ens_query([small, big], h)
    N, kc = 256, 85
    NK, NZp = 2 * kc + 1, 96
    fields = 8 * (2 * 3 * NK * NK * NZp + 8 * NK * N * NZp + 8 * N * N * NZp)
    partials = 4 * 8 * (NK * NZp // 8)
    counts = 8 * E.ens_counts_len(h)
    assert 0 <= per_member - fields - partials - counts <= 32 * E.ENS_NMOM * 8 + 4096
