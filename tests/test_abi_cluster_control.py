"""The cluster control and query check their arguments on the host."""


def test_cluster_control_validates_on_the_host():
    from paper_2405_16406_gb300 import build
    build.build()
    from paper_2405_16406_gb300 import spinq as S
    for bad in (-1, 9, 1000):
        assert S.spinq_gemm_cluster(bad) == -1
    assert S.spinq_gemm_cluster(5) == 0
    assert S.spinq_gemm_cluster(0) == 5
    for M, N, K in ((0, 256, 128), (16, 100, 128), (16, 256, 100), (16, 256, 0), (-1, 256, 128), (16, 256, 65664)):
        assert S.spinq_w4a4_gemm_cluster_plan(M, N, K) == -1
