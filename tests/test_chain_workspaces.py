"""A training step's workspaces are no larger than the calls that use them ask for."""
import pytest

from paper_2105_13890_b200 import eoq, workloads
from paper_2105_13890_b200.chain import ChainedStep

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name,batch", [("resnet20", 4), ("resnet18", 2)])
def test_projection_workspace_fits_projections(name, batch):
    """The projections' stream back-propagates errors of projections only."""
    small = name == "resnet20"
    wl = workloads.resnet20(batch) if small else workloads.resnet18(batch)
    st = ChainedStep(wl, eoq.eoq_create(0), classes=10 if small else 1000, pool=None if small else (3, 2, 1))
    need = [eoq.eoq_workspace_size(blk.proj.desc, eoq.EOQ_PASS_DGRAD) for blk in st.blocks if blk.proj]
    assert len(need) == (2 if small else 3)
    assert st.workspace_sides[st.branch].numel() == max(need) < st.workspace.numel()
    assert all(t.numel() == st.workspace.numel() for t in st.workspace_sides[:st.branch])
