"""The context's launch count holds what ran: an iteration's six launches and, of the graph's
conditional update blocks, those that a slot asked for."""
import pytest

from paper_1112_5280_gb300 import lqcd, synth

pytestmark = pytest.mark.gpu

CHUNK = 8
ITERATION = 6  # five steps, and the finisher of the fourth
UPDATE = 10    # seven steps, three of them with a finisher
FINISH = 3     # the odd half and the full residual of a finished slot


def _steps(systems, use_graph):
    """The launches of each engine step and each system's reliable updates."""
    ctx = lqcd.Context(0)
    eng = lqcd.Engine(ctx, lqcd.solve_opts(sloppy_prec="f32", use_graph=use_graph, chunk=CHUNK), max_slots=4)
    objs, ids = [], []
    for k, (dims, kappa, tol) in enumerate(systems):
        g = ctx.gauge(dims, synth.random_links(dims, 0.5, seed=3 + k))
        src = ctx.field(dims, data=synth.gaussian_spinor(dims, seed=7 + k))
        objs.append((g, src, ctx.field(dims)))
        ids.append(eng.submit(g, src, kappa, tol))
    counts, done, active = [], [], len(ids)
    while active:
        before = ctx.launches
        active = eng.step()
        finished = eng.completed()
        done += finished
        counts.append(ctx.launches - before - FINISH * len(finished))
    updates = [eng.result(i, o[2])["reliable_updates"] for i, o in zip(ids, objs)]
    eng.close()
    ctx.close()
    return counts, updates


@pytest.mark.parametrize("systems", [[((6, 4, 4, 8), 0.15, 1e-11)],
                                     [((6, 4, 4, 8), 0.15, 1e-11), ((4, 4, 4, 8), 0.12, 1e-9)]])
def test_launch_count(systems):
    counts, updates = _steps(systems, use_graph=1)
    direct, direct_updates = _steps(systems, use_graph=0)
    assert updates == direct_updates and len(counts) == len(direct)
    # issued one by one: the update block after every fourth iteration, needed or not
    assert all(n == CHUNK * ITERATION + 2 * UPDATE for n in direct)
    blocks = [(n - CHUNK * ITERATION) / UPDATE for n in counts]
    assert all(b in (0, 1, 2) for b in blocks)
    # the first update of a solve runs when it is submitted; slots may share a block
    assert max(updates) - 1 <= sum(blocks) <= sum(u - 1 for u in updates)
    assert sum(blocks) < 2 * len(blocks)
