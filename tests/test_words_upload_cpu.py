"""Argument errors of the word upload, without a GPU."""
import paper_1805_01450_gb300 as q


def test_arguments():
    L = q.lib()
    assert L.qvx_words_upload(None, 0, None, None) == q.QVX_OK
    assert L.qvx_words_upload(None, 1, None, None) == q.QVX_EINVAL
    assert L.qvx_words_upload(None, -1, None, None) == q.QVX_EINVAL
