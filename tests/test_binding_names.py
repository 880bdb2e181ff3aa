"""A refused call is reported under the name of the call that was made.  No GPU needed: the library refuses a null
handle before it touches a device."""
import numpy as np
import pytest


@pytest.mark.parametrize("name", ["ann_surrogate_load", "ann_surrogate_load_rows"])
def test_refused_loads_name_the_call(name):
    from paper_2108_08919_gb300 import binding, build

    build.build()
    with pytest.raises(binding.AnnError, match=rf"^{name}: "):
        getattr(binding, name)(None, None, np.zeros((5, 8), dtype=np.float32))
