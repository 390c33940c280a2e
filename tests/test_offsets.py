"""The offsets of a batch may be any sequence of whole numbers; a contiguous numpy int64 array is passed as it lies."""
import numpy as np


class Column:
    """Looks like a numpy array in part, as a data frame's column does, whose flags are of its own kind."""
    ndim, dtype, flags = 1, "int64", object()

    def __init__(self, values):
        self.values = values

    def __iter__(self):
        return iter(self.values)

    def __len__(self):
        return len(self.values)


def test_offsets_of_any_sequence():
    import paper_1408_6729_gb300 as bsps
    from paper_1408_6729_gb300 import build
    build.build()
    tune, off = bsps.bsps_tune_default(), [0, 300, 5000, 70_000]
    want = bsps.bsps_batch_bucket_base(off, tune)
    for form in (Column(off), tuple(off), np.array(off), np.array(off, np.int32), np.array(off, ">i8"),
                 np.repeat(np.array(off, np.int64), 2)[::2], np.array(off, np.float64), [np.int64(v) for v in off]):
        assert bsps.bsps_batch_bucket_base(form, tune) == want
