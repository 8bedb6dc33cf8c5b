"""Re-timing of the kernel variants in whole programs (host logic, no GPU): the
sliced remote product is tried in the deferred ordering even when other variants
win alone by less than deferring saves."""
import pytest

pytest.importorskip("torch")


class _Part:
    def __init__(self, refused=()):
        self.now, self.refused = {}, refused

    def set_op_variant(self, op, variant, param):
        from paper_2203_02530_gb300 import spmv
        if (op, variant, param) in self.refused:
            raise spmv.SpmvError(spmv.EINVAL, "refused")
        self.now[op] = (variant, param)


def _run(refused=()):
    from paper_2203_02530_gb300 import search, spmv
    L, R = spmv.OP_LOCAL, spmv.OP_REMOTE
    # alone: three WARP geometries win the remote product by 0.1 us
    times = {(L, spmv.VARIANT_SELL16, 107): 159.4, (L, spmv.VARIANT_SELL, 107): 175.8,
             (R, spmv.VARIANT_WARP, 0): 5.5, (R, spmv.VARIANT_WARP, 1): 5.5, (R, spmv.VARIANT_WARP, 2): 5.6,
             (R, spmv.VARIANT_SELL, 107): 5.6, (R, spmv.VARIANT_SELL, 9): 6.0}
    tuned = {"local": (spmv.VARIANT_SELL16, 107), "remote": (spmv.VARIANT_WARP, 0)}
    part = _Part(refused)
    programs = {"strict": ([0, 1, 2, 3], [0, 0, 0, 0]), "relaxed": ([0, 2, 1, 3], [0, 0, 1, 0]),
                "relaxed+defer": ([0, 2, 1, 3], [0, 0, 1, 0])}

    def evaluator(mode):
        def evaluate(order, smap):
            assert (order, smap) == programs[mode]
            deferred = "defer" in mode and part.now[R][0] == spmv.VARIANT_SELL
            return times[(L,) + part.now[L]] + times[(R,) + part.now[R]] + 6.0 - (4.0 if deferred else 0.0)
        return evaluate

    got, table = search.variants_in_context(part, times, tuned, programs, {m: evaluator(m) for m in programs})
    return spmv, part, got, table


def test_deferrable_remote_product_is_tried_and_kept():
    spmv, part, (t, mode, local, remote), table = _run()
    assert (mode, local, remote) == ("relaxed+defer", (spmv.VARIANT_SELL16, 107), (spmv.VARIANT_SELL, 107))
    assert t == pytest.approx(159.4 + 5.6 + 2.0)
    assert part.now == {spmv.OP_LOCAL: local, spmv.OP_REMOTE: remote}
    assert (local, (spmv.VARIANT_WARP, 0)) in table   # the tuned pair is among them


def test_refused_pairs_are_left_out():
    from paper_2203_02530_gb300 import spmv
    _, part, (t, mode, local, remote), table = _run(refused={(spmv.OP_REMOTE, spmv.VARIANT_SELL, 107)})
    assert remote == (spmv.VARIANT_WARP, 0)
    assert all(rv != (spmv.VARIANT_SELL, 107) for _, rv in table)
