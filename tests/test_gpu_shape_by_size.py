"""Launch shapes taken by size (no shape set): the rule, and the same counts on every side of its lines."""
import numpy as np
import pytest
import torch

import rs_inputs as ri
from gpu_helpers import rs

LARGE2, LARGE3, SMALL2, SMALL4 = (128, 8, 512, 2), (128, 8, 512, 3), (128, 4, 512, 2), (128, 4, 256, 4)


def _pick(masses, n, rows, n0, sms=152):
    import paper_0905_2453_gb300 as m
    return m.rs_launch_config_by_size(masses, n, rows, n0, sms)


@pytest.mark.parametrize("masses", [False, True])
def test_rule(masses):
    """Few lenses take many small CTAs, many lenses large ones, and the three-CTA build is not taken where an SM gets
    a single one (row blocks and maps of about 1e5 rays)."""
    for n0, rows in ((2048, 40), (4096, 24), (8192, 16), (16384, 8), (288, 288), (1024, 64), (1, 1), (7, 3)):
        for n in (100, 1000, 3000, 60000, 10 ** 7):
            assert _pick(masses, n, rows, n0) != LARGE3, (n, rows, n0)
    assert all(_pick(masses, n, 4096, 4096) == SMALL4 for n in (0, 1, 100, 500))
    assert all(_pick(masses, n, 4096, 4096) == LARGE3 for n in (2000, 10 ** 4, 10 ** 8))
    assert _pick(masses, 10 ** 5, 256, 256) == SMALL2          # not one small CTA per SM
    assert _pick(masses, 10 ** 5, 512, 512) == LARGE2          # two large CTAs on the fullest SM
    assert _pick(masses, 10 ** 5, 640, 640) == SMALL4          # 480 large CTAs: four on some, three on most
    assert _pick(masses, 10 ** 5, 2 ** 31, 1) in (LARGE2, LARGE3, SMALL2, SMALL4)


def test_rule_rejects_bad_sizes():
    import paper_0905_2453_gb300 as m
    for bad in ((-1, 4, 4, 152), (4, -1, 4, 152), (4, 4, -1, 152), (4, 4, 4, 0)):
        with pytest.raises(m.RSError):
            m.rs_launch_config_by_size(False, *bad)


@pytest.mark.gpu
@pytest.mark.parametrize("mass", ["equal", "salpeter"])
def test_counts_do_not_depend_on_the_shape_taken(mass):
    m = rs()
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    seen = set()
    for n, side in ((100, 300), (700, 200), (1300, 200), (1300, 512), (1300, 640), (2500, 2048), (7000, 512)):
        spec = ri.disc_field("by-size", n, 0.5, 0.1, 0.2, side, 64, seed=n, mass=mass)
        masses = mass != "equal"
        f = m.Field.from_spec(spec)
        try:
            for rows in ((0, side), (side // 3, side // 3 + 21)):
                shape = m.rs_launch_config_by_size(masses, n, rows[1] - rows[0], side, sms)
                seen.add(shape)
                out = []
                for setting in (None, LARGE2):
                    if setting:
                        m.rs_set_launch_config(masses, *setting)
                    else:
                        m.rs_unset_launch_config(masses)
                    c = torch.zeros((64, 64), dtype=torch.int32, device="cuda")
                    o = torch.zeros(1, dtype=torch.int64, device="cuda")
                    f.shoot(spec.grid, spec.window, c, o, rows=rows)
                    out.append((c.cpu().numpy(), int(o.item())))
                assert np.array_equal(out[0][0], out[1][0]) and out[0][1] == out[1][1], (n, side, rows, shape)
        finally:
            f.close()
    if sms == 152:
        assert seen == {LARGE2, LARGE3, SMALL2, SMALL4}


@pytest.mark.gpu
@pytest.mark.parametrize("fields", [[(1300, 200, "equal")], [(100, 300, "equal"), (5000, 150, "salpeter")],
                                    [(100, 300, "salpeter"), (700, 260, "equal"), (900, 0, "equal"), (3000, 37, "equal")],
                                    [(700, 300, "salpeter")] * 5])
def test_batches_of_few_fields(fields):
    """Batches whose items do not fill the SMs (fewer items than CTAs, a field without rays) give the plain counts."""
    m = rs()
    specs = [ri.disc_field("few", n, 0.5, 0.0, 0.2, side or 16, 48, seed=n + k, mass=mass)
             for k, (n, side, mass) in enumerate(fields)]
    grids = [s.grid if side else m.RayGrid(s.grid.origin, s.grid.spacing, (0, 5)) for s, (_, side, _) in zip(specs, fields)]
    fs = [m.Field.from_spec(s) for s in specs]
    try:
        b = m.Batch(fs, grids, [s.window for s in specs])
        try:
            b.launch()
            b.launch()  # the plan zeroes its counts
            torch.cuda.synchronize()
            for k, (f, s) in enumerate(zip(fs, specs)):
                c = torch.zeros((48, 48), dtype=torch.int32, device="cuda")
                o = torch.zeros(1, dtype=torch.int64, device="cuda")
                if grids[k].n[0]:
                    f.shoot(grids[k], s.window, c, o)
                assert torch.equal(b.counts[k], c) and int(b.out_of_window[k].item()) == int(o.item()), k
        finally:
            b.close()
    finally:
        for f in fs:
            f.close()
