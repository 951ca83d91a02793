"""The launches that bench.py claims for the paths of an A-application."""
import pytest

import bench


def per_step(prec, n_t, modes, n_det=1024, chunk=1024):
    p = bench.apply_path(prec, n_t, modes)
    return p["kernels"], bench.launches_per_iteration(n_det, chunk, bench.CIRC_FUSED_LAUNCHES, p["map_out"],
                                                      bench.CG_FUSED_LAUNCHES, p["filter"], p["flush"])


# map copy in, forward, filter (three launches with correlated noise), inverse, the flush
# that writes the map; 3 of the circulant apply and 2 of the step
@pytest.mark.parametrize("prec,n_t,modes,chunk,kernels,a", [
    ("f32", 1 << 20, 0, 1024, "k_pair_", 5), ("bf16", 1 << 13, 0, 1024, "k_pair_", 5),
    ("f32", 1 << 18, 3, 1024, "k_pair_", 7), ("f32", 1 << 20, 0, 512, "k_pair_", 1 + 2 * 4),
    # FP64: no flush, the accumulator copied out
    ("f64", 1 << 18, 0, 1024, "k_pair_", 5), ("f64", 1 << 20, 0, 256, "k_pair_", 2 + 4 * 3),
    # outside the register FFTs: forward, filter and inverse a chunk, map in and out
    ("f32", 1 << 12, 0, 1024, "k_tod_", 5), ("f64", 1 << 21, 0, 1024, "k_tod_", 5)])
def test_launches(prec, n_t, modes, chunk, kernels, a):
    assert per_step(prec, n_t, modes, chunk=chunk) == (kernels, a + 3 + 2)
