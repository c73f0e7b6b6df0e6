"""Early-stop checks inside the multi-step launch or between launches, chosen by the check
period and the items per CTA: both sides of each line against the checks between launches,
and the cuts and spins of both against the adjacency on the host."""
import numpy as np
import pytest

from paper_2603_25762_gb300 import qhap, synth

pytestmark = pytest.mark.gpu


# hifi-region at full size has 57 row tiles: 57, 228 and 456 items of 128 replicas, one to
# three per CTA on 152 SMs.  The lines lie at 128, 30 and 22 steps per check.
@pytest.mark.parametrize("R,check_every,inside", [(128, 128, True), (128, 129, False),
                                                  (512, 30, True), (512, 31, False),
                                                  (1024, 22, True), (1024, 23, False)])
def test_check_placement(R, check_every, inside):
    import torch

    if torch.cuda.get_device_properties(0).multi_processor_count != 152:
        pytest.skip("items per CTA differ")
    ctx = qhap.Context(0)
    g = ctx.build_graph(synth.hifi_region(1002), mode=qhap.MODE_READ)
    kw = dict(replicas=R, steps=2 * check_every + 9, precision=qhap.PREC_BF16, seed=4,
              check_every=check_every, patience=3, step_kernel="multistep-stream-tile")
    sol = ctx.solve(g, check_mode=0, **kw)
    ref = ctx.solve(g, check_mode=1, **kw)
    fewer = sol.timing()["n_step_launches"] < ref.timing()["n_step_launches"]
    assert fewer == inside
    assert np.array_equal(sol.cuts(), ref.cuts())
    spins = sol.spins(g.n_nodes)
    assert np.array_equal(spins, ref.spins(g.n_nodes))
    bo, _ = g.blocks()
    rp, col, w = g.edges()
    row = np.repeat(np.arange(g.n_nodes), np.diff(rp))
    for b in range(g.n_blocks):
        e = bo[row] == b
        cut = ((spins[row[e]] != spins[col[e]]) * w[e]).sum() / 2
        blk = sol.block(b)
        assert cut == blk["best_cut"] == sol.cuts()[b].max()
        assert blk["best_replica"] == int(np.argmax(sol.cuts()[b]))
    assert np.array_equal(spins == 0, bo < 0)
    for s in (sol, ref):
        s.free()
    g.free()
    ctx.close()


@pytest.mark.parametrize("n", [1, 10])
def test_launches_end_with_the_last_block(n):
    """Checks between launches: the host is one period ahead of the device, so one period
    follows the one in which the last block stopped."""
    ctx = qhap.Context(0)
    fr = synth.tiny_reads(1001) if n == 1 else synth.batched_blocks(1004, n_blocks=n, n_min=20,
                                                                    n_max=400)
    g = ctx.build_graph(fr, mode=qhap.MODE_READ)
    sol = ctx.solve(g, replicas=128, steps=3000, precision=qhap.PREC_BF16, seed=2, check_every=40,
                    patience=3, check_mode=1, step_kernel="multistep-stream-tile")
    run = max(sol.block(b)["steps_run"] for b in range(g.n_blocks))
    assert run < 3000 - 80
    assert sol.timing()["n_step_launches"] == run // 40 + 1
    _, trace = sol.check_trace()
    assert np.isfinite(trace[: run // 40]).any(axis=1).all()
    assert np.isnan(trace[run // 40:]).all()
    sol.free()
    g.free()
    ctx.close()
