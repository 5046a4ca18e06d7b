"""The autotuner times the passes that a handle's scheme runs, its cache keeps their shapes apart, and a handle reports
the shape that ran."""
import numpy as np
import pytest

from paper_1712_05145_gb300 import synthetic

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("grid,kwargs", [((32, 32, 32), {}), ((64, 48, 32), {"pass_mode": 2}), ((512, 64, 4), {}), ((512, 16, 4), {})],
                         ids=["planes", "rows", "clusters", "rows of unsplit planes"])
def test_each_scheme_keeps_its_own_shape(grid, kwargs, tmp_path, monkeypatch):
    from paper_1712_05145_gb300 import hom
    path = tmp_path / "tune.txt"
    monkeypatch.setenv("HOM_TUNE_CACHE", str(path))
    ms = synthetic.voronoi(grid, seed=12, n_grains=8)
    schemes = [hom.HOM_CG, hom.HOM_BICGSTAB, hom.HOM_BASIC]
    out = {}
    for turn in range(2):
        for k, scheme in enumerate(schemes):
            H = hom.Homogenization(ms, scheme=scheme, autotune=1, **kwargs)
            info = H.solve(0, 1e-5)
            assert all(i["status"] == 0 for i in info), info
            got = (hom.hom_launch_config(H.h), hom.hom_zpass_config(H.h), hom.hom_ypass_config(H.h), H.effective(0))
            H.close()
            assert len(path.read_text().splitlines()) == (k + 1 if turn == 0 else 3)
            if turn == 0:
                out[scheme] = got
            else:
                assert got[:3] == out[scheme][:3] and np.array_equal(got[3], out[scheme][3])
    keys = [line.split("|")[0] for line in path.read_text().splitlines()]
    assert len(set(keys)) == 3


def test_the_reported_z_tile_is_that_of_the_last_step():
    """FP64 steps of 32^3: 544 columns, tiles of 64 with six CTAs each are 54 CTAs a load.  One load takes the narrowest
    tile of 64-byte runs that holds 256 values (8 columns of 32), six loads have a CTA for every place as they are."""
    torch = pytest.importorskip("torch")
    from paper_1712_05145_gb300 import hom
    H = hom.Homogenization(synthetic.centred_sphere(32), precision=hom.HOM_FP64)
    assert hom.hom_zpass_config(H.h) == (1, 6)
    out = torch.empty((6, 6, 32, 32, 32), dtype=torch.float64, device="cuda")
    for n, lg in ((1, 3), (6, 6), (1, 3)):
        hom.hom_ls_apply(H.h, n, None, np.eye(6)[:n], out)
        assert hom.hom_zpass_config(H.h) == (1, lg)
    H.close()
