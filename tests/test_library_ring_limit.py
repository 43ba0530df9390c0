"""Delay rings beyond the 32-bit index range are refused before the library touches the GPU (no GPU
needed): 2^31 values, counted as levels x (1 or 2 for traces) x variables x subdomain faces x face
nodes.
"""
import pytest

from paper_2603_28710_gb300 import adg


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2603_28710_gb300 import build
    build.build()


@pytest.mark.parametrize("flux,at_np,n", [("std", 1, (64, 64, 552)), ("at", 1, (64, 64, 528)),
                                          ("at_trace", 1, (64, 64, 264))])
def test_rings_beyond_the_index_range_are_rejected(flux, at_np, n):
    # every element a subdomain: 3 faces of 4 nodes per element, 16 (std) or 17 levels
    levels = 16 if flux == "std" else 17
    assert levels * (2 if flux == "at_trace" else 1) * 5 * 3 * n[0] * n[1] * n[2] * 4 >= 2 ** 31
    with pytest.raises(adg.AdgError) as e:
        adg.Solver(dim=3, n_elem=n, degree=1, dt=1e-4, P=n, flux=flux, at_np=at_np, precision="fp32",
                   delay_mode="random", random_delay_max=15)
    assert e.value.status == 2 and "ring" in str(e.value)
