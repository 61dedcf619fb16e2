// Steps of a state that changes buffers, for the closure.
#pragma once

namespace rslb {

// nsteps steps: step(cur) advances the state from buffer cur into buffer cur ^ 1 and
// leaves it in cur when it fails.  The state starts in buffer 0 and is there again
// on return, after a failure too: back() copies buffer 1 to 0.  Returns the
// first error, or ok.
template <typename E, typename Step, typename Back>
E swap_steps(int nsteps, E ok, Step step, Back back) {
  E e = ok;
  int cur = 0;
  for (int n = 0; n < nsteps && e == ok; ++n) {
    e = step(cur);
    if (e == ok) cur ^= 1;
  }
  if (cur) {
    const E b = back();
    if (e == ok) e = b;
  }
  return e;
}

}  // namespace rslb
