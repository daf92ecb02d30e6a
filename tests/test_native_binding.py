"""The native part of the Python binding marshals arguments like the C ABI expects them (no GPU: calls that are refused)."""
import os
import sysconfig

import pytest

from paper_2105_13890_b200 import build, eoq

build.build_lib()


class Memory:
    """Stands in for a tensor."""

    def __init__(self, address, n=64):
        self.address, self.n = address, n

    def data_ptr(self):
        return self.address

    def numel(self):
        return self.n

    def element_size(self):
        return 1


def test_statuses_and_argument_errors():
    d, m, n = eoq.conv_desc(1, 8, 8, 16, 16, 3, 3, 1, 1), Memory(1 << 12), eoq.native()
    # without a handle every call is refused before it looks at memory
    assert n.conv_fwd_dev(0, d, m, None, m, m, m, None, 1, m, m, m, 0) == eoq.EOQ_ERR_BAD_ARG
    assert eoq.eoq_conv_dgrad(0, d, m, m, m, m, m, None, None, m, stream=0, check=False) == eoq.EOQ_ERR_BAD_ARG
    assert eoq.eoq_conv_wgrad_dev(0, d, m, m, m, None, m, m, m, stream=0, check=False) == eoq.EOQ_ERR_BAD_ARG
    assert eoq.eoq_err_prescale_dev(0, m, m, None, None, 64, m, m, m, stream=0, check=False) == eoq.EOQ_ERR_BAD_ARG
    assert eoq.eoq_quantize(0, eoq.EOQ_SQ, m, True, None, 64, m, m, stream=0, check=False) == eoq.EOQ_ERR_BAD_ARG
    assert eoq.eoq_update_dev(0, [m, m], [m, m], [m, m], 1, -6, 0, 1 << 63, m, stream=0, check=False) == eoq.EOQ_ERR_BAD_ARG
    assert eoq.eoq_weight_prep(0, [d], [m], [m], stream=0, check=False) == eoq.EOQ_ERR_BAD_ARG
    with pytest.raises(eoq.EoqError):
        eoq.eoq_weight_prep(0, [d], [m], [m], stream=0)
    with pytest.raises(AttributeError):
        eoq.eoq_conv_dgrad(0, d, object(), m, m, m, m, stream=0)
    with pytest.raises(TypeError):
        eoq.eoq_conv_dgrad(0, m, m, m, m, m, m, stream=0)
    with pytest.raises(ValueError):
        eoq.eoq_update_dev(0, [m, m], [m], [m, m], 1, -6, 0, 1, m, stream=0)


def test_module_is_the_one_of_this_interpreter(tmp_path, monkeypatch):
    """A module built for another interpreter, however new, neither counts as built nor is loaded."""
    tag = sysconfig.get_config_var("EXT_SUFFIX")
    assert "cpython" in tag and os.path.basename(build.BIND) == "_eoqbind" + tag
    assert eoq.BIND_PATH == build.BIND and os.path.samefile(eoq.native().__file__, build.BIND)
    # one for another interpreter lies beside the library (newer than the sources): this one's is built all the same
    os.symlink(build.LIB, tmp_path / "libeoq.so")
    other = tmp_path / "_eoqbind.so"
    other.write_bytes(b"built for another interpreter")
    monkeypatch.setattr(build, "HERE", str(tmp_path))
    monkeypatch.setattr(build, "BIND", str(tmp_path / os.path.basename(build.BIND)))
    assert build.build_bind() == build.BIND and os.path.getsize(build.BIND) > 1000
    assert other.read_bytes() == b"built for another interpreter"
