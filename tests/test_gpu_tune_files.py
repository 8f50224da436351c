"""A saved launch configuration names the same kernel whatever the variants' order in the library: per mode and number in
the file, the Gaussians staged per batch and the resident CTAs that the registers allow for."""
import pytest

from paper_2507_15683_gb300 import synth

pytestmark = pytest.mark.gpu

KERNELS = {0: [(256, 5), (128, 5), (256, 4), (64, 5)], 2: [(128, 4), (64, 4), (128, 3), (64, 3)]}


@pytest.mark.parametrize("mode", sorted(KERNELS))
def test_numbers_in_a_file(gsr, tmp_path, mode):
    S = gsr.Scene(synth.aerial_scene(5, 200, extent=(0.0, 20.0, 0.0, 20.0), n_clusters=2))
    cams = [synth.camera(64, 48, 50.0)]
    path = str(tmp_path / "launch.txt")
    gsr.gs_scene_set_launch(S.handle, mode, cams, 1, 0, 8)
    gsr.gs_tune_save(S.handle, path)
    line = [l for l in open(path) if l.split("|")[1:2] == [str(mode)]][0]
    for v, kernel in enumerate(KERNELS[mode]):
        with open(path, "w") as f:
            f.write("|".join(line.split("|")[:3]) + "|%d 0 8\n" % v)
        assert gsr.gs_tune_load(S.handle, path) == 1
        got = gsr.gs_scene_get_launch(S.handle, mode, cams)
        assert (got["batch"], got["min_blocks"]) == kernel
        gsr.gs_tune_save(S.handle, path)
        assert [l for l in open(path) if l.split("|")[1:2] == [str(mode)]][0].split("|")[3].split()[0] == str(v)
    S.close()
