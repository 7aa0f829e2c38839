"""The iterate exchange of k_cluster_solve, every interleaving of its warps on a small
cluster: a wait names a barrier's phase by its parity alone, so no warp may reach its
wait for sweep g after the barrier has completed the phase of sweep g + 2 (it would
wait for a phase that nobody completes).  Warps of slots with an antenna hold each
other back by their stores; a slot without one stores nothing and must not wait."""
import os
import re

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1003_5575_gb300", "csrc",
                   "cluster_solve_kernels.cuh")


def lost_waits(warps, sweeps, idle_waits):
    """Waits that can be overtaken.  warps: (CTA, slot has an antenna) of each warp, the
    first of a CTA its expect_tx thread; a sweep of a warp is: expect, send, wait, and
    the last one meets its CTA's warps before the send."""
    n_cta = 1 + max(c for c, _ in warps)
    senders = [w for w, (_, live) in enumerate(warps) if live]
    first = [next(w for w, (c, _) in enumerate(warps) if c == cta) for cta in range(n_cta)]

    def completed(state, cta, b):
        """Phases of barrier b of the CTA that are complete: expected, and every store arrived."""
        n = 0
        for g in range(b, sweeps, 2):
            if state[first[cta]] <= 3 * g or any(state[w] < 3 * g + 2 for w in senders):
                break
            n += 1
        return n

    start = tuple(0 for _ in warps)          # 3 g + (0: to expect, 1: to send, 2: to wait)
    seen, todo, lost = {start}, [start], set()
    while todo:
        state = todo.pop()
        for w, (cta, live) in enumerate(warps):
            g, stage = divmod(state[w], 3)
            if g == sweeps:
                continue
            if stage == 1 and g == sweeps - 1 and any(state[v] < 3 * g + 1 for v, (c, _) in enumerate(warps) if c == cta):
                continue                     # the last sweep's CTA barrier
            if stage == 2 and (live or idle_waits):
                n = completed(state, cta, g & 1)
                if n >= g // 2 + 2:
                    lost.add((w, g))
                if n % 2 != (g // 2 + 1) % 2:
                    continue                 # the parity test says: not yet
            after = state[:w] + (state[w] + 1,) + state[w + 1:]
            if after not in seen:
                seen.add(after)
                todo.append(after)
    return lost


WARPS = [(0, True), (0, False), (1, True), (1, True)]


def test_a_waiting_idle_slot_can_be_overtaken():
    assert {w for w, _ in lost_waits(WARPS, 5, idle_waits=True)} == {1}


def test_no_wait_of_the_kernel_can_be_overtaken():
    body = open(SRC).read().split("k_cluster_solve(ClusterSolveArgs a)")[1].split("struct ClusterAlsArgs")[0]
    guards = re.findall(r"(if \(live\) )?cluster_wait\(", body)
    assert guards and lost_waits(WARPS, 5, idle_waits=not all(guards)) == set()


def test_models_written_beside_the_prep_launch_are_not_read_as_constants():
    """k_cluster_prep is resident while the launch before it writes the model matrices:
    neither a read-only pointer nor the non-coherent load may be used for them."""
    body = open(SRC).read().split("k_cluster_prep(")[1].split("\n}\n")[0]
    assert re.search(r"const float2\* Mblk,", body) and not re.search(r"__ldg\(M4", body)
