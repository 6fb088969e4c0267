"""Work memory of the 3-D kernels: a slot holds the 19 cubes of a patch with its
ghosts and little more (the new record is built where gathered cubes were),
and a run of 16-cell patches on a grid of less than three patches per SM holds
less device memory than the two lattices of the uncompressed run."""
import numpy as np
import pytest

from paper_2302_09883_gb300 import Sim3, inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("P,store", [(16, "bf16"), (16, "f32"), (32, "bf16"), (32, "f32")])
def test_a_slot_is_its_cubes(P, store):
    # two patches against one: a slot, and per patch an arena share of 64 KB, a
    # ring and a table entry, twice, and the sums
    one, two = (Sim3(n * P, P, P, P, 3, 1e-6, store=store, tau=0.8, arena_factor=0.01).resident_bytes() for n in (1, 2))
    ring = 4 * (30 * (P + 1) ** 2 + 12 * (P + 1))
    slot = two - one - 2 * (65536 + 8 + ring) - 19 * 8
    cubes = 19 * 4 * (P + 3) ** 3
    assert cubes <= slot <= 1.03 * cubes


@pytest.mark.parametrize("store", ["bf16", "f32"])
def test_small_patches_hold_less_than_two_lattices(store):
    n = (176, 80, 112)
    g = Sim3(*n, 16, 3, 1e-5, store=store, tau=0.8)
    g.init_macro(inputs.shear_wave_3d(*n, seed=1))
    g.step(2)
    g.sync()
    assert g.resident_bytes() < 2 * 19 * 4 * np.prod(n)
