"""bench.py's count of what a launch moves follows the kernels that ran."""


def test_implementation_bytes_follow_the_kernels_that_ran():
    import bench
    n, px, c, nv = 1000, 500, 8, 400
    step = ("clear", "depth", "accumulate", "normalize", "bwd_prepass", "bwd_points", "bwd_reduce")
    grads, records = 4 * c + 12, px * 48
    visible = nv * (4 + 12 + c * 2 + grads)  # mask, xyz, tau -> gradients

    def got(kernel, *more):
        return bench.implementation_bytes(kernel, n, px, c, 2, 2, nv, ran=step + more)

    # without a seed pass the clear writes counts and sums, and the accumulate pass adds every member
    assert got("clear") == px * (8 + 4 + 32) and got("clear", "seed") == px * 8
    assert got("accumulate", "seed") == n * 5 + nv * 12 + px * 8
    assert got("accumulate") == got("accumulate", "seed") + nv * 16 + 2 * px * 36
    # the zero gradients: in the index-order pass by mask, in the binned one by bit, or ahead of it
    assert got("bwd_points") == visible + records + (n - nv) * (4 + grads)
    assert got("bwd_points", "bwd_bin") == visible + records + nv * 4 + 125 + (n - nv) * grads
    assert got("bwd_points", "bwd_bin", "bwd_zero") == visible + records + nv * 4
    assert got("bwd_zero", "bwd_bin", "bwd_zero") == n * grads
    assert got("bwd_bin", "bwd_bin") == n * 4 + 250 + nv * 8
