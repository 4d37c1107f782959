"""bench.py counts a product's bytes in the form that the solve reads the matrix in:
rows by their diagonals only where it is told that they are laid out so."""
import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_bytes_of_both_forms():
    sys.path.insert(0, ROOT)
    import bench
    from paper_2302_04180_gb300 import gen
    prof = {"k1_spmv_dot": [10, 1.0], "k3_spmv_dot2": [10, 1.0]}
    for A in (gen.poisson3d(12), gen.random_csr(1001, 9, 3)):
        assert bench._roofline(A, prof)["alg_bytes_per_launch"] == 12 * A.nnz + 32 * A.n + 8
        # 4 bytes per row and 8 per 32 rows instead of 4 per nonzero and 8 per row
        words = 4 * A.n + 8 * ((A.n + 31) // 32)
        laid = bench._roofline(A, prof, diagonals=True)["alg_bytes_per_launch"]
        assert laid == 8 * A.nnz + words + 24 * A.n
