"""Bytes that the bench counts for the operator as qdd_apply_D runs it."""
import bench


def test_apply_bytes_per_site():
    """FP32 spinor results leave the operator as FP64 in the host layout: 96 bytes more than in their own storage."""
    for prec, more in (("f64", 0), ("df64", 0), ("f32", 96), ("h16", 96), ("f16", 0), ("bf16", 0)):
        for rows3 in (True, False):
            assert bench.apply_bytes_per_site(prec, rows3) == bench.op_bytes_per_site(prec, rows3) + more
