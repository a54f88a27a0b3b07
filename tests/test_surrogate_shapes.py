"""sg.conv3d_fwd_to sizes its result from the caller's volume shape while the kernel writes one value per
voxel of x: shapes that do not belong together are refused on the host, before anything is launched."""
import pytest
import torch

from paper_1909_08406_gb300 import sg

NATURAL = (1, 8, 16, 64, 16)


def _call(x_shape, natural, df, dt, add_shape=None, z_shape=None):
    x = torch.zeros(x_shape, dtype=torch.bfloat16)
    w = torch.zeros((32, 27, 16), dtype=torch.bfloat16)
    add = None if add_shape is None else torch.zeros(add_shape, dtype=torch.bfloat16)
    z = None if z_shape is None else torch.zeros(z_shape)
    return sg.conv3d_fwd_to(x, w, None, sg.ACT_NONE, False, natural, df, dt, add=add, z_out=z)


@pytest.mark.parametrize("natural,df", [((1, 8, 8, 64, 16), 1), ((1, 4, 16, 64, 16), 1), ((2, 8, 16, 64, 16), 1),
                                        (NATURAL, 2), ((1, 8, 16, 32, 16), 1)])
def test_volume_shape_must_be_that_of_x(natural, df):
    with pytest.raises(RuntimeError, match="natural"):
        _call(NATURAL, natural, df, 1)


def test_extents_that_the_spacing_does_not_divide():
    with pytest.raises(RuntimeError, match="natural"):
        _call((4, 4, 8, 64, 16), (1, 9, 17, 64, 16), 2, 1)


@pytest.mark.parametrize("df,dt", [(1, 1), (1, 2), (4, 2)])
def test_added_tensor_and_kept_values_must_have_their_layouts_shape(df, dt):
    x_shape = sg.relabelled_shape(NATURAL, df)
    y_shape = sg.relabelled_shape(NATURAL, dt)[:-1] + (32,)
    with pytest.raises(RuntimeError, match="add"):
        _call(x_shape, NATURAL, df, dt, add_shape=y_shape[:-1] + (16,))
    with pytest.raises(RuntimeError, match="add"):
        _call(x_shape, NATURAL, df, dt, add_shape=(y_shape[0], y_shape[1] - 1) + y_shape[2:])
    with pytest.raises(RuntimeError, match="z_out"):
        _call(x_shape, NATURAL, df, dt, z_shape=x_shape)
