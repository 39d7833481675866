"""The y passes on survey rows (Fields::rows), which replace the plane kernel at 256^3 and wherever
BPS_FUSED_YZ=0 keeps the three passes, on small grids: the running moments, which read the whole
field after the survey sums and so need a dense inverse y pass, and 96^3, whose rows are looked up
with a radix that does not divide a word."""
import pytest

from tests import test_gpu_parity, test_gpu_posterior
from tests.helpers import Problem

pytestmark = pytest.mark.gpu


def test_moments_of_a_survey_with_empty_lines(monkeypatch):
    monkeypatch.setenv("BPS_FUSED_YZ", "0")
    pb = Problem(32, n_sub=2, n_bins=8)
    assert (pb.R.max(axis=(0, 3)) == 0).any()
    test_gpu_posterior.test_running_moments_match_the_oracle_chain()


@pytest.mark.parametrize("f_sky", [0.15, 0.6])
def test_gradient_at_96(monkeypatch, f_sky):
    import torch
    test_gpu_parity.test_gradient_three_passes_with_line_supports(torch, monkeypatch, 96, 2, f_sky)
