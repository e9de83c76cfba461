"""The plan of an attention launch with fewer slices than SMs is the one that was measured
to be the shorter.  Without a GPU (148 SMs, no clusters are assumed): whole slices against
the work split."""
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
