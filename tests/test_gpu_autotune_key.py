"""What the cache of autotuned CTAs per SM is keyed by: a step's band tiles and
the batch's other groups beside the group's own work, and the way it is timed."""
import pytest

import lbm_workloads as W

pytestmark = pytest.mark.gpu


def tune(path, monkeypatch, cfgs):
    import paper_2307_16766_gb300 as lbm
    monkeypatch.setenv("LBM_AUTOTUNE_CACHE", str(path))
    B = lbm.Batch(cfgs)
    for r, c in enumerate(cfgs):
        B[r].init_fields(*W.uniform(c["nx"], c["ny"]))
    B.step(1)
    B.close()
    return path.read_text().splitlines()


def runs(sides, n=2, lattice="D2Q37"):
    return [W.run(lattice, 60, 48, 0.8, storage="f32", sides=sides, schemes=("cbc_relax",) * 4)] * n


def test_entries_of_a_bulk_only_timing_are_not_taken(tmp_path, monkeypatch):
    import torch
    path = tmp_path / "tune.txt"
    name = torch.cuda.get_device_name().replace(" ", "_")
    old = ["%s %d %d %d 1" % (name, lat, st, b) for lat in range(3) for st in range(3) for b in range(16)]
    path.write_text("\n".join(old) + "\n")
    assert len(tune(path, monkeypatch, runs(("cbc",) * 4))) == len(old) + 1


def test_band_tiles_and_other_groups_have_entries_of_their_own(tmp_path, monkeypatch):
    path = tmp_path / "tune.txt"
    assert len(tune(path, monkeypatch, runs(("periodic",) * 4))) == 1
    assert len(tune(path, monkeypatch, runs(("cbc",) * 4))) == 2               # the same bulk work, and tiles
    assert len(tune(path, monkeypatch, runs(("cbc",) * 4) + runs(("cbc",) * 4, 1, "D2Q9"))) == 4
    assert len(tune(path, monkeypatch, runs(("cbc",) * 4))) == 4               # known
    assert len(tune(path, monkeypatch, runs(("periodic",) * 4))) == 4
