"""Plane-major arrays of a single element: planes have their pitch whatever the (free)
stride of the element axis, also inside larger planes (validated on the host only)."""
import pytest
import torch

from paper_1504_01023_gb300 import api


@pytest.mark.parametrize("et", [api.TET, api.PRISM])
@pytest.mark.parametrize("pitch", [1, 4, 256])
def test_plane_strides_of_one_element(et, pitch):
    ns = api.NS[et]
    quad = api.QUAD_TET4 if et == api.TET else api.QUAD_PRISM6

    def planes(k):
        return torch.zeros(k, pitch, dtype=torch.float64)[:, :1]

    a = api.make_args(et, planes(3 * ns), planes(20), api.GENERIC, quad, api.PER_ELEMENT, api.FP64, api.SOA)
    o = api.make_out(planes(ns * ns), planes(ns), None, api.SOA)
    assert a.n_elem == 1 and a.coords_stride == pitch and a.coefs_stride == pitch and o.stride == pitch
    with pytest.raises(AssertionError):        # one pitch for both outputs
        api.make_out(planes(ns * ns), torch.zeros(ns, pitch + 3, dtype=torch.float64)[:, :1], None, api.SOA)
