"""What a launch of the on-chip steps does when, read from its source."""
import os

from paper_1611_00907_gb300 import _lib


def test_the_state_is_stored_behind_the_last_wait():
    path = os.path.join(os.path.dirname(os.path.abspath(_lib.__file__)), "csrc",
                        "resident_impl.cuh")
    text = open(path).read()
    body = text[text.index("resident_kernel(const ResidentArgs"):]
    waited = body.index("if (__syncthreads_or(!ok)) return false;")
    for store in ("aa_write_index(", "store_rho_whole("):
        assert store not in body[:waited] and store in body[waited:]
