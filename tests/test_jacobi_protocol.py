"""The cooperative Jacobi kernel ends whichever way its waits end.

Its three roles meet at two named barriers per iteration (all of them at
barrier 1, compute and exchange at barrier 2) and the exchange warp's verdict
travels through shared memory; a role that leaves one barrier early would
strand the others, because the barriers count a fixed number of threads.  That
cannot be provoked on a GPU, so the roles are replayed here step by step in
every order the barriers allow, with the number of verdict slots and the slots'
indices as the kernel has them."""
import os
import re

import pytest

SOURCE = os.path.join(os.path.dirname(__file__), "..", "paper_2011_03602_gb300", "csrc", "jacobi.cu")


def verdict_slots():
    """(slots, accesses): the declaration of ok_s and what indexes it."""
    with open(SOURCE) as f:
        text = f.read()
    kernel = text[text.index("jacobi_fused_kernel(FusedArgs a)"):text.index("size_t fused_words_bytes")]
    decl = re.search(r"__shared__ int ok_s(?:\[(\d+)\])?;", kernel)
    assert decl, "ok_s not found"
    return int(decl.group(1) or 1), re.findall(r"ok_s\[([^\]]*)\][ ;)]", kernel.replace(decl.group(0), ""))


def compute(iters, slots, ok):
    for it in range(iters):
        yield "b1"
        yield "b2"
        if not ok[it % slots]:
            if it + 1 < iters:
                yield "b1"
            return


def exchange(iters, slots, ok, fails_at):
    for it in range(iters):
        yield "b1"
        yield "step"  # the wait
        ok[it % slots] = it != fails_at
        yield "b2"
        if it == fails_at:
            if it + 1 < iters:
                yield "b1"
            return


def residual(iters, slots, ok):
    for it in range(iters):
        yield "b1"
        yield "step"  # anything may happen between the barrier and the read
        if it > 0 and not ok[(it - 1) % slots]:
            return


NEEDS = {"b1": {0, 1, 2}, "b2": {0, 1}}


def replay(choices, iters, slots, fails_at):
    """The state after the given choices: (positions, ended, who may go on)."""
    ok = [True] * slots
    roles = [compute(iters, slots, ok), exchange(iters, slots, ok, fails_at), residual(iters, slots, ok)]
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


def stuck_orders(iters, slots, fails_at):
    """Orders after which some role waits for one that has left."""
    bad, todo = [], [()]
    while todo:
        path = todo.pop()
        at, go = replay(path, iters, slots, fails_at)
        if not go and any(x != "end" for x in at):
            bad.append(path)
        todo += [path + (g,) for g in go]
    return bad


def test_model_finds_the_race_of_a_single_slot():
    assert stuck_orders(3, 1, 1)


@pytest.mark.parametrize("iters", [1, 2, 3, 4])
def test_kernel_ends_in_every_order(iters):
    slots, index = verdict_slots()
    assert slots == 1 or sorted(set(index)) == ["(it - 1) & 1", "it & 1"]
    for fails_at in [None] + list(range(iters)):
        assert not stuck_orders(iters, slots, fails_at), fails_at
