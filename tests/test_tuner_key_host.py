"""Two grids that the library gives different default shapes or kernels do not
share a tuned launch shape."""
import problems as pb
from paper_2108_12240_gb300 import autotune


def test_key_tells_grids_apart():
    g = pb.torus_3d(nroot=(4, 3, 2))
    others = [pb.torus_3d(), g.with_(c2p="nk"), g.with_(recon="minmod"), pb.torus_3d(nroot=(4, 3, 2), nblock=(8, 8, 8))]
    keys = {autotune.key_of(x, "fp64") for x in [g, *others]} | {autotune.key_of(g, "mixed")}
    assert len(keys) == len(others) + 2
    assert autotune.key_of(pb.torus_3d(nroot=(4, 3, 2)), "fp64") == autotune.key_of(g, "fp64")
