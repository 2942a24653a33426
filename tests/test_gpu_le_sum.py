"""The emitted-radiance gradient of LRB-3 with known masks: a sum over all paths by the blocks of two
passes.  Against the FP64 sum of the paths' own terms (delta_total over Le, from path_dbg)."""
import pytest
import torch

from paper_2609_32920_gb300 import inputs as I
from paper_2609_32920_gb300 import lt

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scene", ["box", "slab_in_box", "slab"])
@pytest.mark.parametrize("n", [1, 300, (1 << 17) + 5, 1 << 20])
# the sum is added to the array by the kernel that adds up the albedo copies (scatter 0), or by the last
# block of pass 3
@pytest.mark.parametrize("attached,scatter", [(0, 0), (1, 0), (0, 2), (1, 2)])
def test_sum_is_rounded_once(scene, n, attached, scatter):
    sc = {"box": lambda: I.box_scene(64, heightmap=16), "slab_in_box": lambda: I.slab_in_box(64, n=24),
          "slab": lambda: I.slab_scene(64, n=24)}[scene]()
    S = lt.Scene(sc)
    Le = S.Le.double()
    state = S.new_lrb3_state(n)
    for seed in range(4):
        dI = torch.tensor(I.smooth_adjoint(S.W, S.H, seed), dtype=torch.float32, device="cuda")
        kw = dict(seed=seed, n_paths=n, max_depth=6, attached=attached)
        S.primal(S.opts(lrb3_state=state, **kw))
        dbg = torch.zeros((n, 4), device="cuda")
        o = S.opts(lrb3_state=state, lrb3_mask_ready=1, dbg_out=dbg, scatter=scatter, **kw)
        got = S.backward_lrb3(o, dI)[1]
        terms = dbg[:, :3].double() / Le
        ref, mass = terms.sum(0), terms.abs().sum(0)
        # one rounding of the result, and each lane's FP32 sum of its few terms: at most 2^-24 per add
        # of the lane's own mass, independent over the lanes, so far below 2^-25 of the whole (in small
        # calls, where a lane has one term, its division by Le)
        tol = 2.0 ** -24 * (ref.abs() + (1.0 if n < 1000 else 0.5) * mass)
        assert ((got.double() - ref).abs() <= tol).all()
        g = S.new_grads()
        g[1].copy_(got)
        S.backward_lrb3(o, dI, grads=g, accumulate=True)
        assert torch.allclose(g[1], 2 * got, rtol=3e-7, atol=float(2.0 ** -22 * mass.max()))
    S.sync_status()
