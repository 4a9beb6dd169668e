"""Which stencils run the streamed kernel: all of an automatic map but one aligned
step of radius 1, and the widest windows on whole tiles that fill a wave of SMs.  No GPU."""
import pytest

from paper_2309_01906_gb300 import binding as hb


@pytest.mark.parametrize("ny,nx,r,T,kernel", [
    (4096, 4096, 1, 1, "stencil_tile"), (4096, 4095, 1, 1, "stencil_stream"), (4096, 4096, 1, 2, "stencil_stream"),
    # whole tiles, a wave of them and a little less
    (768, 768, 4, 4, "stencil_tile"), (1024, 1024, 4, 2, "stencil_tile"), (8000, 128, 4, 3, "stencil_tile"),
    (1024, 1024, 3, 8, "stencil_tile"), (8000, 128, 3, 8, "stencil_tile"),
    # other windows, ragged tiles, less than three quarters of a wave, more than one
    (1024, 1024, 3, 7, "stencil_stream"), (1024, 1024, 3, 2, "stencil_stream"), (8000, 128, 4, 5, "stencil_stream"),
    (1000, 1000, 4, 2, "stencil_stream"), (537, 1004, 4, 4, "stencil_stream"), (5187, 124, 4, 3, "stencil_stream"),
    (768, 768, 4, 2, "stencil_stream"), (512, 512, 4, 4, "stencil_stream"), (1024, 1024, 4, 4, "stencil_stream"),
    (16384, 16384, 4, 2, "stencil_stream"), (1024, 1022, 4, 2, "stencil_stream"),
    (64, 64, 4, 6, "stencil_tile"),       # no streamed kernel
])
def test_route(ny, nx, r, T, kernel):
    st = hb.Stencil(ny, nx, r, [0.0] * (2 * r + 1) ** 2, T)
    assert st.describe()["kernel"] == kernel
    st.close()
    if kernel == "stencil_stream":        # an explicit tile is always tiled
        st = hb.Stencil(ny, nx, r, [0.0] * (2 * r + 1) ** 2, T, tile=(16, 64))
        assert st.describe()["kernel"] == "stencil_tile"
        st.close()
