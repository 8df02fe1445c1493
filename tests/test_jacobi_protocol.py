"""The cooperative Jacobi kernel ends whichever way its waits end.

Its three roles meet at two named barriers per iteration (all of them at
barrier 1, compute and exchange at barrier 2) and the exchange warp's verdict
travels through shared memory; a role that leaves one barrier early would
strand the others, because the barriers count a fixed number of threads.  That
cannot be provoked on a GPU, so the roles are replayed here step by step in
every order the barriers allow, with the statements on the verdict that the
kernel has."""
import os

import pytest

SOURCE = os.path.join(os.path.dirname(__file__), "..", "paper_2011_03602_gb300", "csrc", "jacobi.cu")


class Flag:
    """One flag, stored in every iteration: what the roles must not share."""

    def __init__(self, iters):
        self.ok = True

    def store(self, it, ok):
        self.ok = ok

    def compute_leaves(self, it):
        return not self.ok

    def residual_leaves(self, it):
        return it > 0 and not self.ok


class FailedAt:
    """The kernel's verdict: the iteration that failed, stored then only."""

    STATEMENTS = ("if (lane == 0) failed_at = a.iters;", "if (!ok && lane == 0) failed_at = it;",
                  "if (failed_at == it) {", "if (failed_at < it) return;")

    def __init__(self, iters):
        self.at = iters

    def store(self, it, ok):
        if not ok:
            self.at = it

    def compute_leaves(self, it):
        return self.at == it

    def residual_leaves(self, it):
        return self.at < it


def compute(iters, verdict):
    for it in range(iters):
        yield "b1"
        yield "b2"
        if verdict.compute_leaves(it):
            if it + 1 < iters:
                yield "b1"
            return


def exchange(iters, verdict, fails_at):
    for it in range(iters):
        yield "b1"
        yield "step"  # the wait
        verdict.store(it, it != fails_at)
        yield "b2"
        if it == fails_at:
            if it + 1 < iters:
                yield "b1"
            return


def residual(iters, verdict):
    for it in range(iters):
        yield "b1"
        yield "step"  # anything may happen between the barrier and the read
        if verdict.residual_leaves(it):
            return


NEEDS = {"b1": {0, 1, 2}, "b2": {0, 1}}


def replay(choices, iters, kind, fails_at):
    """Where the roles are after the given choices, and who may go on."""
    verdict = kind(iters)
    roles = [compute(iters, verdict), exchange(iters, verdict, fails_at), residual(iters, verdict)]
    at = [next(r) for r in roles]

    def ready():
        out = [(i,) for i in range(3) if at[i] == "step"]
        for bar, need in NEEDS.items():
            if all(at[i] == bar for i in need):
                out.append(tuple(sorted(need)))
        return out

    for c in choices:
        for i in c:  # a barrier releases every role; what each does next is a choice of its own
            at[i] = next(roles[i], "end")
    return at, ready()


def stuck_orders(iters, kind, fails_at):
    """Orders after which some role waits for one that has left."""
    bad, todo = [], [()]
    while todo:
        path = todo.pop()
        at, go = replay(path, iters, kind, fails_at)
        if not go and any(x != "end" for x in at):
            bad.append(path)
        todo += [path + (g,) for g in go]
    return bad


def test_model_finds_the_race_of_a_flag():
    assert stuck_orders(3, Flag, 1)


@pytest.mark.parametrize("iters", [1, 2, 3, 4])
def test_kernel_ends_in_every_order(iters):
    with open(SOURCE) as f:
        text = f.read()
    kernel = text[text.index("jacobi_fused_kernel(FusedArgs a)"):text.index("size_t fused_words_bytes")]
    for statement in FailedAt.STATEMENTS:
        assert kernel.count(statement) == 1, statement
    assert kernel.count("failed_at") == len(FailedAt.STATEMENTS) + 3  # the declaration and the comment
    for fails_at in [None] + list(range(iters)):
        assert not stuck_orders(iters, FailedAt, fails_at), fails_at
