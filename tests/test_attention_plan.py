"""The plan of an attention launch with fewer slices than SMs, and the form of a fused
step, are the ones that were measured to be the shorter.  Without a GPU (148 SMs, no
clusters are assumed): whole slices against the work split, and an argmax grid against the
argmax in the attention grid."""
import pytest


@pytest.mark.parametrize("slices,T,D,prefix,plan", [
    (80, 64, 128, 3000, 0),      # 31.3 us whole, 33.5 split
    (100, 64, 128, 3000, 0),     # 32.8, 39.0
    (80, 100, 128, 3000, 0),     # 32.0, 36.1
    (100, 32, 64, 3000, 0),      # 20.5, 22.6
    (20, 64, 128, 1500, 0),      # 16.3, 16.2
    (20, 64, 128, 3000, 1),      # 27.1, 19.5
    (20, 32, 64, 8000, 1),       # 43.6, 18.4
    (80, 64, 128, 8000, 1),      # 69.0, 63.1
    (80, 32, 64, 8000, 1),       # 44.5, 34.6
    (140, 64, 128, 8000, 0),     # 89.1, 99.0
    (148, 64, 128, 8000, 0),     # a slice for every SM
])
def test_whole_slices_or_the_work_split(slices, T, D, prefix, plan):
    torch = pytest.importorskip("torch")
    if torch.cuda.is_available():
        pytest.skip("the device's clusters take part in the plan")
    from paper_2405_18628_gb300 import build, ppd
    build.build()
    assert ppd.ppd_attention_plan(1, 1, slices, T, D, prefix + T) == plan
    assert ppd.ppd_attention_plan(1, 1, slices, T, D, prefix + T, workspace=False) == 0


@pytest.mark.parametrize("L,B,H,T,D,prefix,ratio,form", [
    # slices in whole rounds of SMs: no narrow argmax grid
    (4, 1, 37, 64, 128, 2048, 1000, 2),     # 106.3 us with an argmax grid, 104.2 without (608 slices)
    (4, 1, 37, 64, 128, 2048, 150, 2),      # 107.3, 104.2
    (4, 1, 37, 64, 128, 2048, 64, 1),       # 107.3, 116.0
    (4, 1, 37, 64, 128, 2048, 20, 1),       # 111.2, 197.9
    (4, 8, 37, 128, 128, 4096, 64, 1),      # 360.5, 399.2 (1216 slices)
    # fewer slices than SMs
    (1, 1, 32, 64, 128, 2048, 1000, 1),     # 17.2, 25.1
    (1, 1, 100, 32, 64, 2048, 300, 1),      # 19.2, 22.8
])
def test_argmax_grid_or_in_the_attention_grid(L, B, H, T, D, prefix, ratio, form):
    torch = pytest.importorskip("torch")
    if torch.cuda.is_available():
        pytest.skip("148 SMs assumed")
    from paper_2405_18628_gb300 import build, ppd
    build.build()
    V = 4 * L * B * H * (prefix + 2 * T) * D // ratio // (4 * B * T)
    assert ppd.ppd_verify_step_form(L, B, H, T, D, V, prefix + T) == form
