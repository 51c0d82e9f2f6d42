"""Which problems AUTO gives to the separable path (planning only: its scratch is another than the
direct kernels')."""
import dataclasses

import pytest

import paper_2103_09686_gb300 as dm


def _separable(p):
    return dm.dmcr_workspace_size(p) != dm.dmcr_workspace_size(dataclasses.replace(p, path=dm.DMCR_PATH_DIRECT))


# measured (loss and gradient, us): 833 direct, 3232 separable; 2551, 3695; 1040, 1356; 1054, 1078 (its descriptor
# 349, 438); 298, 341; 438, 441 (154, 195)
@pytest.mark.parametrize("shape,window,levels,phases", [((2, 512, 512), (1, 20, 20), 1, 1), ((4, 512, 512), (2, 20, 20), 1, 1),
                                                        ((3, 300, 300), (1, 30, 30), 1, 1), ((4, 256, 256), (1, 30, 30), 2, 1),
                                                        ((100, 120), (20, 20), 1, 5), ((96, 96), (12, 12), 1, 8)])
def test_thin_volumes_and_many_phases_stay_direct(shape, window, levels, phases):
    assert not _separable(dm.Params(shape=shape, window=window, levels=levels, phases=phases))


# 22455 direct, 1224 separable; 7903, 395; 1345, 885; 5756, 435; 394, 273; 575, 511; 36290, 754; 1634, 127
@pytest.mark.parametrize("shape,window,levels,phases", [((512, 2, 512), (20, 1, 20), 1, 1), ((256, 3, 256), (24, 1, 24), 1, 1),
                                                        ((2, 1024, 64), (1, 100, 20), 1, 1), ((16, 256, 256), (8, 16, 16), 1, 1),
                                                        ((256, 256), (8, 8), 1, 4), ((256, 256), (8, 8), 1, 5),
                                                        ((512, 512, 4), (20, 20, 2), 1, 1), ((512, 512), (64, 64), 3, 1)])
def test_where_the_transforms_are_faster(shape, window, levels, phases):
    assert _separable(dm.Params(shape=shape, window=window, levels=levels, phases=phases))
