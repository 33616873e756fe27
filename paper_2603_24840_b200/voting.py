"""ctypes binding of the test-time rank-weighted vote (marshalling only)."""
from . import binding as B


def arrol_rank_vote(ctx: B.Context, score, answer, P: int, G: int, weight, winner, winner_weight, stream=None):
    B._check(B.load_library().arrol_rank_vote(ctx.handle, B._ptr(score), B._ptr(answer), int(P), int(G), B._ptr(weight),
                                              B._ptr(winner), B._ptr(winner_weight), B._stream(stream)), "arrol_rank_vote")
