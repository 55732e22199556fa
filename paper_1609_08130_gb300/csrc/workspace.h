// workspace.h -- workspaces that grow with the number of columns of a call.
#pragma once

namespace rss {

// Make a set of buffers hold `want` (columns, or groups of columns).  `have`
// says what they hold and is 0 while `replace` frees and allocates, so an
// allocation that throws leaves a set that the next call makes anew instead of
// one that is taken for whole.
template <typename Replace> void regrow(int &have, int want, Replace &&replace) {
  if (have >= want) return;
  have = 0;
  replace();
  have = want;
}

}  // namespace rss
