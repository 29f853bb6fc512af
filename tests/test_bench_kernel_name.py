"""The roofline line's kernel name: one kernel, with an issued rate, only where the
assignment's filter is never tried."""
import bench


def test_assignment_kernel_claims_no_more_than_the_sizes_say():
    for t in (1, 819, 2944):
        name, one = bench.assignment_kernel(t)
        assert one and name == "tc_gemm_kernel<256, kSplit, TcEpiArgmax8>"
    for t in (2945, 13107):
        name, one = bench.assignment_kernel(t)
        assert not one and "TcEpiFilter" in name and "TcEpiArgmax8" in name
